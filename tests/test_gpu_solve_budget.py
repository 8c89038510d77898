"""What max_iter buys the automatic solve and what it reports, on every driver
it has: a BiCGStab step counts once, although it applies K twice (as a GMRES
step does), and a residual evaluation counts once."""
import pytest

from paper_2503_16037_gb300 import scenes
from paper_2503_16037_gb300 import tursca as T

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2503_16037_gb300 import build
    build.build()


def assembled(sc, precision, group_warps=0):
    rn = T.Runner(sc, precision)
    if group_warps:  # the solve runs pass by pass
        T.tursca_set_option(rn.handle, T.OPT_GROUP_WARPS, group_warps)
    rn.set_medium(*rn.fields("cuda"))
    rn.assemble()
    T.tursca_profile_enable(rn.handle, True)
    return rn


@pytest.mark.parametrize("precision,group_warps,counter", [(T.FP32_REFINE, 0, "persist"), (T.FP64, 0, "persist"),
                                                           (T.FP64, 8, "gmres_prod")])
def test_a_bicgstab_step_counts_once(precision, group_warps, counter):
    rn = assembled(scenes.make_random(21, 19, 9, seed=5, S=2, R=2, M=2048), precision, group_warps)
    rtol = 1e-12 if precision == T.FP64 else 1e-10
    rn.solve(rtol=rtol)
    info = rn.info
    products = T.tursca_profile_read(rn.handle)[counter][0]
    assert info.iters > info.refinements > 0
    steps = info.iters - info.refinements
    if counter == "persist":  # every product of the solve, the residuals' included
        assert products == 2 * steps + info.refinements
    else:  # the steps' products, of the one step that is queued ahead per refinement too
        assert 2 * steps <= products <= 2 * (steps + info.refinements)
    # that many steps suffice, half of them do not
    rn.solve(rtol=rtol, max_iter=info.iters)
    assert rn.info.rel_resid64 <= rtol
    with pytest.raises(T.TurscaError) as e:
        rn.solve(rtol=rtol, max_iter=info.iters // 2)
    assert e.value.status == T.E_NOT_CONVERGED
