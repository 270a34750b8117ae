"""The vector form of the refined n <= 4 solve's second pass is as accurate as the
outputs allow: x* and u* of a time-varying FP32 problem are sums of at most n + 4
terms of their own size, each rounded to 2^-24, so their relative error against
64 bits, in the root mean square over a long horizon, stays below (n + 4) 2^-24.
(Forming v_k from F^T w - K^T (L^T w), which cancels, is off by 1.4 to 2.3 times
that.)"""
import numpy as np
import pytest

from gpu_util import gpu_solve, oracle_solve
from paper_2104_03186_gb300 import inputs
from paper_2104_03186_gb300.accuracy import rel_fro

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1000, 10000])
@pytest.mark.parametrize("n,m,p", [(1, 1, 2), (2, 1, 2), (3, 1, 2), (4, 2, 1), (4, 2, 3)])
def test_refined_errors_are_a_few_roundings(n, m, p, T):
    bound = (n + 4) * 2.0 ** -24
    for seed in range(3):
        prob = inputs.random_problem(n, m, p=p, T=T, seed=10 * seed + n).rounded_to(np.float32)
        got, ref = gpu_solve(prob), oracle_solve(prob)
        errs = {k: rel_fro(got[k], ref[k]) for k in ("x", "u")}
        assert max(errs.values()) <= bound, (errs, bound)
