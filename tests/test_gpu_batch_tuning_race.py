"""lqt_batch_set_tuning from another thread while batches and warm solves run: a
call cuts its problems once, so a workspace that is too small for the cut it took
is refused (LQT_ENOMEM) and nothing is written past the one it was given."""
import threading

import numpy as np
import pytest

from gpu_util import FP32_TOL, compare, oracle_solve
from paper_2104_03186_gb300 import inputs

pytestmark = pytest.mark.gpu

GUARD = 32 << 20
COARSE, FINE = [(8, 4096, 64)], [(8, 4096, 4)]  # chunk lengths: short chunks take more workspace


@pytest.mark.parametrize("warm", [False, True])
def test_workspace_checked_on_the_cut_that_runs(warm):
    import torch

    from paper_2104_03186_gb300 import lqt

    # enough steps that the table's lengths differ (a small batch caps them)
    one = inputs.diag_tracking(8, T=4096, seed=3).rounded_to(np.float32)
    P = lqt.Problem.from_inputs(one)
    Ps = [P] * 64
    stop = threading.Event()
    toggler = None
    try:
        lqt.lqt_batch_set_tuning(COARSE, "per_level")
        known = lqt.solve_batched(Ps)
        outs = [dict(P.allocate_outputs(), S=k["S"], K=k["K"]) for k in known] if warm else \
            [P.allocate_outputs() for _ in Ps]
        size = lqt.lqt_warm_workspace_bytes if warm else lqt.lqt_batch_workspace_bytes
        solve = lqt.lqt_solve_warm if warm else lqt.lqt_solve_batched
        small = size(Ps, outs)
        lqt.lqt_batch_set_tuning(FINE, "per_level")
        assert size(Ps, outs) > small
        with pytest.raises(lqt.LQTError) as e:
            solve(Ps, outs, torch.empty(small, dtype=torch.uint8, device="cuda"))
        assert e.value.status == lqt.LQT_ENOMEM
        buf = torch.full((small + GUARD,), 0x5A, dtype=torch.uint8, device="cuda")

        def toggle():
            while not stop.is_set():
                lqt.lqt_batch_set_tuning(FINE, "per_level")
                lqt.lqt_batch_set_tuning(COARSE, "per_level")

        toggler = threading.Thread(target=toggle)
        toggler.start()
        for _ in range(200):
            try:
                solve(Ps, outs, buf[:small])
            except lqt.LQTError as err:
                assert err.status == lqt.LQT_ENOMEM
        stop.set()
        toggler.join()
        torch.cuda.synchronize()
        assert bool((buf[small:] == 0x5A).all())
        lqt.lqt_batch_set_tuning(COARSE, "per_level")
        solve(Ps, outs, buf[:small])
        assert lqt.lqt_workspace_status(buf) == lqt.LQT_OK
        ref = oracle_solve(one)
        for o in (outs[0], outs[-1]):
            compare({k: v.double().cpu().numpy() for k, v in o.items()}, ref, FP32_TOL)
    finally:
        stop.set()
        if toggler is not None:
            toggler.join()
        lqt.lqt_batch_set_tuning([], "auto")
        lqt.apply_tuned_plans()
