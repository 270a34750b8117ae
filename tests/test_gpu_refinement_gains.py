"""The n <= 4 refinement does not lose accuracy: x* and u* of a refined solve of a
time-varying FP32 problem are no further from 64 bits than those of the unrefined
one, whose iterate it starts from, and the rounding of the sum (2^-24).  (A second
pass that forms v_k from F^T w - K^T (L^T w), which cancels, fails this at n = 1, 2
and for the shorter horizons at n = 4.)"""
import numpy as np
import pytest

from gpu_util import gpu_solve, oracle_solve
from paper_2104_03186_gb300 import inputs
from paper_2104_03186_gb300.accuracy import rel_fro

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [100, 1000, 10000])
@pytest.mark.parametrize("n,m,p", [(1, 1, 2), (2, 1, 2), (3, 1, 2), (4, 2, 1), (4, 2, 3)])
def test_refined_solve_no_further_off_than_the_plain_one(n, m, p, T):
    for seed in range(3):
        prob = inputs.random_problem(n, m, p=p, T=T, seed=10 * seed + n).rounded_to(np.float32)
        ref = oracle_solve(prob)
        plain, refined = gpu_solve(prob, refine=0), gpu_solve(prob, refine=1)
        for k in ("x", "u"):
            assert rel_fro(refined[k], ref[k]) <= rel_fro(plain[k], ref[k]) + 2.0 ** -24, (k, seed)
