"""Refined n <= 4 solves report values that are not finite (LQT_ENONFINITE),
whichever pass they first appear in: an initial state that is not finite, and a
first trajectory that overflows while S, v and K stay finite.  One tile and
several, a time-invariant model and one that changes with the step."""
import numpy as np
import pytest

from paper_2104_03186_gb300 import inputs

pytestmark = pytest.mark.gpu


def _status(prob, **kw):
    import torch

    from paper_2104_03186_gb300 import lqt

    P = lqt.Problem.from_inputs(prob, **kw)
    out = P.allocate_outputs()
    opts = lqt.options(lqt.LQT_REFINE_ON)
    ws = torch.empty(lqt.lqt_workspace_bytes(P, opts), dtype=torch.uint8, device="cuda")
    lqt.lqt_solve(P, out, ws, opts=opts)
    return lqt.lqt_workspace_status(ws), out


def _model(kind, T):
    if kind == "vehicle":
        return inputs.vehicle(T, seed=1)
    n, m = kind
    return inputs.random_problem(n, m, p=n, T=T, seed=T + n)


MODELS = ["vehicle", (1, 1), (2, 1), (3, 2), (4, 2)]


@pytest.mark.parametrize("T", [1, 100, 1024, 1025, 20000])
@pytest.mark.parametrize("model", MODELS, ids=str)
def test_initial_state_not_finite(model, T):
    from paper_2104_03186_gb300 import lqt

    prob = _model(model, T)
    assert _status(prob)[0] == lqt.LQT_OK
    for bad in (np.nan, np.inf):
        prob.x0[-1] = bad
        assert _status(prob)[0] == lqt.LQT_ENONFINITE


@pytest.mark.parametrize("T", [100, 1025])
def test_initial_state_not_finite_fp64(T):
    from paper_2104_03186_gb300 import lqt

    prob = inputs.vehicle(T, seed=1)
    assert _status(prob, dtype=np.float64)[0] == lqt.LQT_OK
    prob.x0[0] = np.nan
    assert _status(prob, dtype=np.float64)[0] == lqt.LQT_ENONFINITE


@pytest.mark.parametrize("T", [200, 5000])
@pytest.mark.parametrize("varying", [False, True])
def test_trajectory_that_overflows(T, varying):
    """A state that nothing observes or controls grows from 1e37 by a factor of
    100: S does not see it, every product of F is finite, and x overflows."""
    import torch

    from paper_2104_03186_gb300 import lqt

    prob = inputs.vehicle(T, seed=2)
    F, L, H, HT, XT = (np.array(getattr(prob, f)) for f in ("F", "L", "H", "HT", "XT"))
    F[:, 3, :], F[:, :, 3], F[:, 3, 3] = 0.0, 0.0, 100.0 ** (1.0 / T)
    L[:, 3, :] = 0.0
    H[:, :, 3] = 0.0
    HT[:, 3] = 0.0
    if varying:
        F = np.repeat(F, T, axis=0)
    prob.F, prob.L, prob.H, prob.HT, prob.XT = F, L, H, HT, XT
    prob.x0[3] = 1e37
    st, out = _status(prob)
    assert st == lqt.LQT_ENONFINITE
    for f in ("S", "v", "K"):
        assert bool(torch.isfinite(out[f]).all()), f
