"""The automatic solve on the GPU takes the driver that its plan names: the
persistent launch where there is one (and only that), else the passes; the
adjoint over K^T likewise, and over a scene that runs in rounds its gradient is
that of the passes with a block per group.

Tolerance of the gradient: the adjoint solves to 1e-9; its FP32 sums, in the
order in which atomics arrive, of a few thousand terms are good to a few
thousand 2^-24 of their magnitudes in the worst case and to 1e-5 of the largest
entry with much to spare.
"""
import pytest

from paper_2503_16037_gb300 import scenes
from paper_2503_16037_gb300 import tursca as T

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2503_16037_gb300 import build
    build.build()


def counts(rn):
    return {k: v[0] for k, v in T.tursca_profile_read(rn.handle).items()}


def solved(shape, R, precision=T.FP32_REFINE, group_warps=0):
    sc = scenes.make_random(*shape, seed=3, S=1, R=R, M=1024)
    rn = T.Runner(sc, precision)
    if group_warps:
        T.tursca_set_option(rn.handle, T.OPT_GROUP_WARPS, group_warps)
    T.tursca_profile_enable(rn.handle, True)
    rn.run(*rn.fields("cuda"))
    return rn, counts(rn)


@pytest.mark.parametrize("shape,R,precision", [((5, 5, 1), 1, T.FP32_REFINE), ((8, 8, 8), 1, T.FP64),
                                               ((21, 19, 9), 2, T.FP32_REFINE), ((45, 37, 29), 2, T.FP32_REFINE),
                                               ((64, 64, 32), 2, T.FP64), ((96, 96, 32), 2, T.FP32_REFINE)])
def test_the_persistent_solve_runs(shape, R, precision):
    rn, c = solved(shape, R, precision)
    passes = c["spmv"] + c["cheb"] + c["gmres_prod"] + c["resid64"]
    assert c["persist"] == 2 * rn.info.iters - rn.info.refinements and passes == 0
    rn.adjoint(torch.ones_like(rn.rad))
    c = counts(rn)
    assert c["persist"] > 0 and c["spmv"] + c["cheb"] + c["gmres_prod"] + c["resid64"] == 0
    rn.close()


@pytest.mark.parametrize("shape,precision", [((130, 125, 36), T.FP32_REFINE), ((96, 96, 32), T.FP64),
                                             ((512, 8, 40), T.FP32_REFINE)])
def test_the_passes_run_where_there_is_no_plan(shape, precision):
    rn, c = solved(shape, 2, precision)
    assert c["persist"] == 0 and c["spmv"] + c["gmres_prod"] > 0 and c["resid64"] > 0
    rn.close()


@pytest.mark.parametrize("shape,forward", [((130, 125, 36), "rounds"), ((104, 104, 34), "persistent")])
def test_gradient_over_rounds_of_the_transpose(shape, forward):
    grads = []
    for w in (0, 6):  # rounds; a block per group
        rn, c = solved(shape, 2, T.FP32_REFINE, w)
        dJ = torch.linspace(0.5, 1.5, rn.rad.numel(), device="cuda", dtype=rn.dtype).reshape(rn.rad.shape)
        grads.append(rn.adjoint(dJ).double())
        assert (c["persist"] > 0) == (forward == "persistent" and w == 0) and counts(rn)["persist"] == 0
        rn.close()
    assert float(grads[1].abs().max()) > 0.0
    assert float((grads[0] - grads[1]).abs().max()) <= 1e-5 * float(grads[1].abs().max())


def test_csr_solve_in_a_graph():
    """The one launch of the CSR solve is captured like the launches before it."""
    n, row = 5000, 30
    g = torch.Generator().manual_seed(1)
    col = torch.randint(0, n, (n * row,), generator=g).int().cuda()
    val = (torch.rand(n * row, generator=g) / (2 * row)).cuda()
    ptr = (torch.arange(n + 1, dtype=torch.int32) * row).cuda()
    s = torch.rand(n, generator=g).cuda()
    x, y = (torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(2))
    T.tursca_csr_solve_noalloc(ptr, col, val, n, s, x, 10, 3, None, torch.cuda.current_stream().cuda_stream)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        T.tursca_csr_solve_noalloc(ptr, col, val, n, s, y, 10, 3, None, torch.cuda.current_stream().cuda_stream)
    s.mul_(2.0)
    graph.replay()
    torch.cuda.synchronize()
    assert float((y - 2.0 * x).abs().max()) <= 1e-13 * float(y.abs().max())
