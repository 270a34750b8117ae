"""n >= 8: a control weight U_k that is not positive definite is reported also where
only a problem's first chunk sees it (include/lqt.h: LQT_ENOTSPD or, from the lane
groups and teams, LQT_ESINGULAR): one chunk, several, a time-invariant U and one
that changes with the step, whatever the terminal cost adds to L^T S L + U."""
import numpy as np
import pytest

from paper_2104_03186_gb300 import inputs

pytestmark = pytest.mark.gpu


def _problem(n, T, varying, bad):
    """Small stage costs and a large terminal one, so that every L^T S L + U is
    positive definite, with U = I but for the steps in `bad` (U = -I / 10)."""
    prob = inputs.random_problem(n, n // 2, p=n, T=T, seed=n + T, time_varying=False, with_c=False)
    prob.F = np.eye(n)[None]
    prob.L = np.eye(n, n // 2)[None]
    prob.H, prob.X = np.eye(n)[None], 1e-3 * np.eye(n)[None]
    prob.HT, prob.XT, prob.rT = np.eye(n), 1e6 * np.eye(n), np.zeros(n)
    U = np.repeat(np.eye(n // 2)[None], T, axis=0)
    U[bad] = -0.1 * np.eye(n // 2)
    prob.U = U if varying else U[:1]
    return prob


def _status(prob, dtype):
    import torch

    from paper_2104_03186_gb300 import lqt

    P = lqt.Problem.from_inputs(prob, dtype=dtype)
    out = P.allocate_outputs()
    if dtype == np.float32:
        ws = torch.empty(lqt.lqt_batch_workspace_bytes([P], [out]), dtype=torch.uint8,
                         device="cuda")
        lqt.lqt_solve_batched([P], [out], ws)
    else:
        ws = lqt.workspace_for(P, opts=lqt.LQT_REFINE_OFF)
        lqt.lqt_solve(P, out, ws, opts=lqt.LQT_REFINE_OFF)
    return lqt.lqt_workspace_status(ws)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n", [8, 16, 32])
def test_control_weight_not_positive_definite(n, dtype):
    from paper_2104_03186_gb300 import lqt

    refused = (lqt.LQT_ENOTSPD, lqt.LQT_ESINGULAR)
    for T in (1, 3, 9):
        assert _status(_problem(n, T, False, []), dtype) == lqt.LQT_OK
        assert _status(_problem(n, T, True, []), dtype) == lqt.LQT_OK
        assert _status(_problem(n, T, False, slice(None)), dtype) in refused
        # the first step lies in the first chunk, whatever its length
        assert _status(_problem(n, T, True, [0]), dtype) in refused
