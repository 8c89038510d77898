"""What max_iter buys the automatic solve and what it reports, on every driver
it has: a BiCGStab step counts once, although it applies K twice (as a GMRES
step does), and a residual evaluation counts once."""
import ctypes as C

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


@pytest.mark.parametrize("precision", [T.FP32_REFINE, T.FP64])
def test_a_solve_that_gives_up_goes_on_with_what_is_left(precision):
    """A tolerance below the residual's rounding: the persistent solve gives up
    after two refinements that gain nothing and the passes go on, from its x
    and with the rest of max_iter.  Every step applies K once or twice, so
    twice the reported steps covers every product that ran."""
    sc = scenes.make_random(16, 15, 9, seed=2, S=2, R=2, M=1024)
    rn = assembled(sc, precision)

    def solve(max_iter):
        info = T.tursca_solve_info()
        status = T.lib().tursca_solve_with(rn.handle, T.SOLVER_AUTO, C.c_double(1e-18), max_iter, C.byref(info))
        p = {k: v[0] for k, v in T.tursca_profile_read(rn.handle).items()}
        assert status == T.E_NOT_CONVERGED
        return info, p

    info, p = solve(400)
    assert p["persist"] > 0 and p["resid64"] > 0  # both ran
    passes = p["spmv"] + p["cheb"] + p["resid64"]
    assert 2 * info.iters >= p["persist"] + 2 * passes + p["gmres_prod"]
    assert info.iters <= 401  # a step and its residual may end a step late
    # the FP32 pairs' and FP64's floor is below 1e-12 of ||x|| (||x|| < 8 ||s|| here: K's rows sum to less than 0.9)
    assert info.rel_resid64 <= 1e-11
    # a budget that the persistent part nearly uses up: the passes get the rest
    budget = (p["persist"] + 1) // 2 + info.refinements + 6
    info, q = solve(budget)
    assert q["persist"] == p["persist"]
    assert q["spmv"] + q["cheb"] + q["resid64"] + q["gmres_prod"] // 2 <= budget - q["persist"] // 2 + 2
    assert info.iters <= budget + 1 and info.rel_resid64 <= 1e-11
    rn.close()


def test_images_stay_untouched_when_the_solve_fails():
    sc = scenes.make_random(16, 15, 9, seed=2, S=2, R=2, M=1024)
    rn = T.Runner(sc, T.FP32_REFINE)
    mu_a, mu_s = rn.fields("cuda")
    rn.run(mu_a, mu_s)
    before = rn.rad.clone()
    with pytest.raises(T.TurscaError) as e:
        rn.run(2.0 * mu_a, mu_s, rtol=1e-18, max_iter=200)
    assert e.value.status == T.E_NOT_CONVERGED
    assert torch.equal(before, rn.rad)
    rn.close()
