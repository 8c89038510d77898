"""The automatic solve's paths on the GPU: the persistent launch (one to all
warps on a group, values in shared memory, in L2 and streamed) and the passes
over larger grids, each against the system that the scene assembled.

Tolerance: the true residual ||s - x + K x||, formed here in FP64 from the
scene's own matrix, may exceed the requested rtol only by the rounding of the
solver's residual: FP32 pairs carry 48 bits, so a row of up to 128 terms is
off by less than 128 * 2^-48 = 5e-13 of its sum of magnitudes, which is at
most 2 max|x| against ||s||; 1e-12 * ||x|| / ||s|| bounds it.
"""
import pytest

from paper_2503_16037_gb300 import scenes
from paper_2503_16037_gb300 import tursca as T

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# one group; all warps on few groups; ragged strips; rows shorter than a
# group; two warps per group with streamed values; past the share of L2; passes
SHAPES = [((5, 5, 1), 1), ((8, 8, 8), 1), ((21, 19, 9), 2), ((16, 16, 16), 2), ((45, 37, 29), 2), ((130, 61, 12), 2),
          ((96, 96, 32), 2), ((130, 125, 36), 2)]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2503_16037_gb300 import build
    build.build()


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("shape,R", SHAPES)
def test_automatic_solve_meets_the_tolerance(shape, R, fp64):
    nx, ny, nz = shape
    if fp64 and nx * ny * nz > 300000:
        pytest.skip("the FP64 passes are those of every larger grid: nothing new in this shape")
    sc = scenes.make_random(nx, ny, nz, seed=nx + nz, S=2, R=R, M=2048)
    rn = T.Runner(sc, T.FP64 if fp64 else T.FP32_REFINE)
    mu_a, mu_s = rn.fields("cuda")
    rn.set_medium(mu_a, mu_s)
    rn.assemble()
    rtol = 1e-9
    rn.solve(rtol=rtol)
    st = rn.stats
    n = st.n_nodes
    rp = torch.from_numpy(rn.get(T.F_ROW_PTR, n + 1, torch.int32)).cuda().long()
    col = torch.from_numpy(rn.get(T.F_COL, st.nnz, torch.int32)).cuda().long()
    val = torch.from_numpy(rn.get(T.F_VAL, st.nnz, rn.dtype)).cuda().double()
    s = torch.from_numpy(rn.get(T.F_S, n, rn.dtype)).cuda().double()
    x = torch.from_numpy(rn.get(T.F_X, n, torch.float64)).cuda()
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), rp[1:] - rp[:-1])
    kx = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, rows, val * x[col])
    rel = float((s - x + kx).norm() / s.norm())
    assert rel <= rtol + 1e-12 * float(x.norm() / s.norm())
    assert rn.info.rel_resid64 <= rtol


# 14 and 16 layers of 8 groups: 114 groups is where a block takes a whole group
@pytest.mark.parametrize("nz", [13, 15])
def test_assembly_with_and_without_split_groups(nz):
    from oracle import oracle as O

    sc = scenes.make_random(32, 31, nz, seed=nz, S=2, R=1, M=1024)
    r = O.run(sc)
    rn = T.Runner(sc, T.FP64)
    mu_a, mu_s = rn.fields("cuda")
    rn.set_medium(mu_a, mu_s)
    rn.assemble()
    rn.solve(rtol=1e-13)
    st = rn.stats
    s = rn.get(T.F_S, st.n_nodes, torch.float64)
    x = rn.get(T.F_X, st.n_nodes, torch.float64)
    # the bounds of the FP64 parity tests
    assert abs(s - r["s"]).max() <= 1e-11 * r["s"].max()
    assert abs(x - r["x"]).max() <= 1e-10 * abs(r["x"]).max()
