"""lqt_set_single_tile_chunk from another thread while host and condensed solves run:
a call lays its buffer out with the sizes it checked, or refuses it (LQT_ENOMEM),
and nothing is written past it."""
import threading

import numpy as np
import pytest

from gpu_util import FP32_TOL, compare, oracle_solve
from paper_2104_03186_gb300 import inputs

pytestmark = pytest.mark.gpu

GUARD = 32 << 20


@pytest.mark.parametrize("kind", ["host", "condensed", "reduced"])
def test_buffer_checked_with_the_sizes_used(kind):
    import torch

    from paper_2104_03186_gb300 import lqt

    B = {"host": 1, "condensed": 2, "reduced": 8}[kind]
    prob = inputs.vehicle(4096 if kind == "host" else 4096 * B, seed=1).rounded_to(np.float32)
    P = lqt.Problem.from_inputs(prob, pin=kind == "host")
    out = P.allocate_outputs(pin=kind == "host")
    size = (lambda: lqt.lqt_host_solve_bytes(P)) if kind == "host" else \
        (lambda: lqt.lqt_condensed_workspace_bytes(P, B))
    stop = threading.Event()
    toggler = None
    before = lqt.lqt_set_single_tile_chunk(16)
    try:
        small = size()
        lqt.lqt_set_single_tile_chunk(0)
        assert size() > small
        buf = torch.full((small + GUARD,), 0x5A, dtype=torch.uint8, device="cuda")

        def solve():
            if kind == "host":
                return lqt.lqt_solve_host(P, out, buf[:small])
            lqt.lqt_solve_condensed(P, B, out, buf[:small])
            return lqt.LQT_OK

        with pytest.raises(lqt.LQTError) as e:
            solve()
        assert e.value.status == lqt.LQT_ENOMEM

        def toggle():
            while not stop.is_set():
                lqt.lqt_set_single_tile_chunk(0)
                lqt.lqt_set_single_tile_chunk(16)

        toggler = threading.Thread(target=toggle)
        toggler.start()
        for _ in range(200):
            try:
                assert solve() == lqt.LQT_OK
            except lqt.LQTError as err:
                assert err.status == lqt.LQT_ENOMEM
        stop.set()
        toggler.join()
        torch.cuda.synchronize()
        assert bool((buf[small:] == 0x5A).all())
        lqt.lqt_set_single_tile_chunk(16)
        assert solve() == lqt.LQT_OK
        torch.cuda.synchronize()
        compare({k: v.double().cpu().numpy() for k, v in out.items()}, oracle_solve(prob),
                FP32_TOL)
    finally:
        stop.set()
        if toggler is not None:
            toggler.join()
        lqt.lqt_set_single_tile_chunk(before)
