"""The launch modes of lqt_solve_batched as they are: the automatic mode is the
per-level launches, bit for bit; the cooperative launch, in a call whose sizes run
side by side, takes a size of many waves of chunks beside a small one."""
import numpy as np
import pytest

from gpu_util import FP32_TOL, compare, oracle_solve
from paper_2104_03186_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture
def restore_plan():
    from paper_2104_03186_gb300 import lqt

    yield
    lqt.lqt_batch_set_tuning([], "auto")
    lqt.apply_tuned_plans()


def test_auto_is_per_level_and_persistent_takes_many_waves(restore_plan):
    import torch

    from paper_2104_03186_gb300 import lqt

    # 65 536 chunks at n = 8, 128 at n = 16
    table = [(8, 4096, 4), (16, 4096, 64)]
    one = {n: inputs.diag_tracking(n, T=T, seed=1900 + n).rounded_to(np.float32)
           for n, T in ((8, 4096), (16, 300))}
    P = {n: lqt.Problem.from_inputs(p) for n, p in one.items()}
    Ps = [P[8]] * 64 + [P[16]] * 2
    outs = {}
    for mode in ("auto", "per_level", "persistent"):
        lqt.lqt_batch_set_tuning(table, mode)
        outs[mode] = lqt.solve_batched(Ps)
    for a, b in zip(outs["auto"], outs["per_level"]):
        for k in a:
            assert torch.equal(a[k], b[k]), k
    for i in (0, 63, 64, 65):
        compare({k: v.double().cpu().numpy() for k, v in outs["persistent"][i].items()},
                oracle_solve(one[Ps[i].n]), FP32_TOL)
