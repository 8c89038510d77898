"""The spectral radius that the persistent solve reports is the power estimate
s.K^7 s / s.K^6 s, formed here in FP64 from the scene's own matrix.

Tolerance: FP32 steps give their coefficients to about 1e-6, and the last
moment used is at least 1e-3 of the first (smaller ones are not used), so the
ratio is good to about 1e-3; FP64 scenes stay inside the same bound.
"""
import pytest

from paper_2503_16037_gb300 import scenes
from paper_2503_16037_gb300 import tursca as T

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SCENES = [lambda: scenes.make_plain(), lambda: scenes.make_random(21, 19, 9, seed=5, S=2, R=2, M=2048),
          lambda: scenes.make_plume(nx=48, ny=48, nz=32), lambda: scenes.make_cloud(32, 32, 40)]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2503_16037_gb300 import build
    build.build()


@pytest.mark.parametrize("precision", [T.FP32_REFINE, T.FP64])
@pytest.mark.parametrize("maker", SCENES)
def test_rho_is_estimated(maker, precision):
    rn = T.Runner(maker(), precision)
    rn.set_medium(*rn.fields("cuda"))
    rn.assemble()
    rn.solve(rtol=1e-10)
    assert rn.info.solver == T.SOLVER_BICGSTAB
    n = rn.stats.n_nodes
    rp = torch.from_numpy(rn.get(T.F_ROW_PTR, n + 1, torch.int32)).cuda().long()
    col = torch.from_numpy(rn.get(T.F_COL, rn.stats.nnz, torch.int32)).cuda().long()
    val = torch.from_numpy(rn.get(T.F_VAL, rn.stats.nnz, rn.dtype)).cuda().double()
    s = torch.from_numpy(rn.get(T.F_S, n, rn.dtype)).cuda().double()
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), rp[1:] - rp[:-1])
    m, y = [], s
    for _ in range(8):
        m.append(float(s @ y / (s @ s)))
        y = torch.zeros_like(s).index_add_(0, rows, val * y[col])
    j = max(i for i in range(7) if m[i] >= 1e-3)
    assert rn.info.rho_est == pytest.approx(m[j + 1] / m[j], rel=1e-3)
    rn.close()
