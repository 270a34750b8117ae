"""FULL refinement at n >= 8: the correction walks take the Newton-corrected S and K
with the chunk maps and G^-1 of the first pass (lqt_chain.cuh says why that is
enough).  The ill-conditioned precision study, several chunks, every step checked,
the chunks' first and last ones with the others: x* and u* are one rounding of
2^-24 each, and the first pass's error (1e-5 at most) times the relative error of
those maps (1e-3 at most) adds 1e-8."""
import numpy as np
import pytest

from gpu_util import compare, gpu_solve, oracle_solve
from paper_2104_03186_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 16, 32])
@pytest.mark.parametrize("T", [257, 4096])
def test_full_refinement_walks_across_chunks(n, T):
    from paper_2104_03186_gb300 import lqt

    prob = inputs.precision_study(T=T, seed=n, n=n, m=n // 2).rounded_to(np.float32)
    assert lqt.lqt_plan(lqt.Problem.from_inputs(prob), lqt.LQT_REFINE_FULL)["tiles"] > 1
    compare(gpu_solve(prob, refine=lqt.LQT_REFINE_FULL), oracle_solve(prob), 2 * 2.0 ** -24,
            names=("x", "u"), step_tol=4 * 2.0 ** -24)
