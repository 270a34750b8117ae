"""n <= 4, a time-varying cost with more outputs than are kept in registers (p > 4):
the rows of H come by 16-byte loads where they are aligned, entry by entry
otherwise, with the same bits; one tile and several, against the oracle."""
import numpy as np
import pytest

from gpu_util import FP32_TOL, FP64_TOL, compare, oracle_solve
from paper_2104_03186_gb300 import inputs

pytestmark = pytest.mark.gpu


def _odd(t):
    """A contiguous copy of t that starts one element past 16 bytes."""
    import torch

    buf = torch.empty(t.numel() + 8, dtype=t.dtype, device=t.device)
    view = buf[1:1 + t.numel()].view(t.shape)
    view.copy_(t)
    return view


@pytest.mark.parametrize("n,m,dtype", [(4, 2, np.float32), (3, 2, np.float32), (4, 2, np.float64)])
@pytest.mark.parametrize("p", [5, 6, 8])
@pytest.mark.parametrize("T", [1, 100, 1025])
def test_many_outputs(n, m, dtype, p, T):
    import torch

    from paper_2104_03186_gb300 import lqt

    prob = inputs.random_problem(n, m, p=p, T=T, seed=p + T).rounded_to(dtype)
    P = lqt.Problem.from_inputs(prob, dtype=dtype)
    Q = lqt.Problem(P.n, P.m, P.p, P.pT, P.T, P.dtype, {k: _odd(a) for k, a in P.arrays.items()})
    a, b = lqt.solve(P, opts=lqt.LQT_REFINE_ON), lqt.solve(Q, opts=lqt.LQT_REFINE_ON)
    for k in a:
        assert torch.equal(a[k], b[k]), k
    compare({k: v.double().cpu().numpy() for k, v in a.items()}, oracle_solve(prob),
            FP32_TOL if dtype == np.float32 else FP64_TOL)
