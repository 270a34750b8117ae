"""Edges of the team kernels (n = 8, 16, 32), of the vector walks of their
refinement, and of the n <= 4 second pass: horizons around chunk and tile
lengths, numbers of outputs around the staged ones, and arrays that do not
start on 16 bytes (which must not change a bit of the result)."""
import numpy as np
import pytest

from gpu_util import FP32_TOL, FP64_TOL, compare, gpu_solve, oracle_solve
from paper_2104_03186_gb300 import inputs

pytestmark = pytest.mark.gpu


def _problem(n, p, T, seed, pT=None):
    return inputs.random_problem(n, n // 2, p=p, T=T, seed=seed, pT=pT)


@pytest.mark.parametrize("n", [8, 16, 32])
@pytest.mark.parametrize("T", [1, 3, 4, 9, 33, 258])
def test_team_kernels_short_horizons(n, T):
    """One chunk, chunks of unequal length, empty chunks; general H of p = n
    outputs; the refined solve, the plain one and FP64."""
    prob = _problem(n, n, T, seed=100 * n + T)
    ref32 = oracle_solve(prob.rounded_to(np.float32))
    for refine in (0, 1):
        compare(gpu_solve(prob.rounded_to(np.float32), refine=refine), ref32, FP32_TOL)
    ref = oracle_solve(prob)
    for refine in (0, 1):
        compare(gpu_solve(prob, dtype=np.float64, refine=refine), ref, FP64_TOL)


@pytest.mark.parametrize("n", [8, 16, 32])
@pytest.mark.parametrize("p", ["1", "n-1", "n+1", "2n"])
def test_team_kernels_output_counts(n, p):
    """p below and above the staged limit (p <= n), with a terminal cost of
    another size."""
    p = {"1": 1, "n-1": n - 1, "n+1": n + 1, "2n": 2 * n}[p]
    prob = _problem(n, p, 70, seed=7 * n + p, pT=2 * n).rounded_to(np.float32)
    compare(gpu_solve(prob), oracle_solve(prob), FP32_TOL)


@pytest.mark.parametrize("p", [1, 3, 4, 5])
@pytest.mark.parametrize("T", [1, 2, 511, 512, 513, 1024, 1025, 1537])
def test_small_second_pass(p, T):
    """One tile and several, a last tile of one chunk, references read four at a
    time (p <= 4) and one by one."""
    prob = inputs.random_problem(4, 2, p=p, T=T, seed=T + p).rounded_to(np.float32)
    compare(gpu_solve(prob), oracle_solve(prob), FP32_TOL)


@pytest.mark.parametrize("n,m", [(1, 1), (2, 1), (2, 2), (3, 1), (3, 2), (4, 1), (4, 4)])
def test_small_second_pass_other_sizes(n, m):
    prob = inputs.random_problem(n, m, p=2, T=1100, seed=10 * n + m).rounded_to(np.float32)
    compare(gpu_solve(prob), oracle_solve(prob), FP32_TOL)


def test_small_second_pass_fp64():
    prob = inputs.random_problem(4, 2, p=3, T=700, seed=5)
    compare(gpu_solve(prob, dtype=np.float64, refine=1), oracle_solve(prob), FP64_TOL)


def _odd(t):
    """A contiguous copy of t that starts one element past 16 bytes."""
    import torch

    buf = torch.empty(t.numel() + 8, dtype=t.dtype, device=t.device)
    view = buf[1:1 + t.numel()].view(t.shape)
    view.copy_(t)
    return view


@pytest.mark.parametrize("n,dtype", [(4, np.float32), (8, np.float32), (16, np.float32),
                                     (32, np.float32), (4, np.float64), (16, np.float64)])
def test_unaligned_arrays_give_the_same_bits(n, dtype):
    """Inputs that start one element past a 16-byte boundary (and, where the
    batched solve takes them, outputs) use the element-wise loads and stores."""
    import torch

    from paper_2104_03186_gb300 import lqt

    prob = _problem(n, 3 if n == 4 else n, 600 if n == 4 else 90, seed=n).rounded_to(dtype)
    P = lqt.Problem.from_inputs(prob, dtype=dtype)
    Q = lqt.Problem(P.n, P.m, P.p, P.pT, P.T, P.dtype, {k: _odd(a) for k, a in P.arrays.items()})
    a, b = lqt.solve(P, opts=lqt.LQT_REFINE_ON), lqt.solve(Q, opts=lqt.LQT_REFINE_ON)
    for k in a:
        assert torch.equal(a[k], b[k]), k
    if dtype == np.float32:
        a, b = P.allocate_outputs(), {k: _odd(t) for k, t in P.allocate_outputs().items()}
        ws = torch.empty(lqt.lqt_batch_workspace_bytes([P], [a]), dtype=torch.uint8, device="cuda")
        lqt.lqt_solve_batched([P], [a], ws)
        lqt.lqt_solve_batched([Q], [b], ws)
        assert lqt.lqt_workspace_status(ws) == lqt.LQT_OK
        for k in a:
            assert torch.equal(a[k], b[k]), k


def test_static_solve_in_the_least_workspace():
    """A refined n = 16 problem whose usual workspace exceeds the library's
    scratch array runs in the least one (the correction as a full pass)."""
    from paper_2104_03186_gb300 import lqt

    prob = inputs.diag_tracking(16, T=45000, seed=3).rounded_to(np.float32)
    P = lqt.Problem.from_inputs(prob)
    assert lqt.lqt_workspace_bytes(P) > lqt.LQT_STATIC_SCRATCH_BYTES
    out = P.allocate_outputs()
    assert lqt.lqt_solve_static(P, out) == lqt.LQT_OK
    compare({k: v.double().cpu().numpy() for k, v in out.items()}, oracle_solve(prob), FP32_TOL)


def test_batch_and_warm_sizes_side_by_side():
    """Every size in one call, forked and joined, twice on one stream and then on
    another: the same bits as the problems of each size by themselves."""
    import torch

    from paper_2104_03186_gb300 import lqt

    probs = [inputs.diag_tracking(n, T=T, seed=50 + n + T).rounded_to(np.float32)
             for n in (4, 8, 16, 32) for T in (257, 40)]
    Ps = [lqt.Problem.from_inputs(p) for p in probs]
    alone = []
    for n in (4, 8, 16, 32):
        alone += lqt.solve_batched([P for P in Ps if P.n == n])
    for stream in (None, None, torch.cuda.Stream()):
        if stream is not None:
            stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream or torch.cuda.current_stream()):
            got = lqt.solve_batched(Ps)
            warm = lqt.solve_warm(Ps, got)
        torch.cuda.synchronize()
        for a, b, w, p in zip(alone, got, warm, probs):
            for k in a:
                assert torch.equal(a[k], b[k]), (p.n, p.T, k)
            compare({k: v.double().cpu().numpy() for k, v in w.items()}, oracle_solve(p),
                    FP32_TOL, names=("v", "x", "u"))


def test_first_forked_call_of_a_thread_may_be_captured():
    """A new thread's first batch and warm calls inside a capture; then the same
    from a second thread, which takes over the first one's streams, with an
    eager call made while a capture holds some of them."""
    import threading

    import torch

    from paper_2104_03186_gb300 import lqt

    probs = [inputs.diag_tracking(n, T=600, seed=n).rounded_to(np.float32) for n in (4, 8, 16)]
    Ps = [lqt.Problem.from_inputs(p) for p in probs]
    want = lqt.solve_batched(Ps)
    warm = lqt.solve_warm(Ps, want)
    torch.cuda.synchronize()
    errors = []

    def run(eager_inside):
        try:
            outs = [P.allocate_outputs() for P in Ps]
            other = [P.allocate_outputs() for P in Ps]
            wout = [dict(P.allocate_outputs(), S=w["S"], K=w["K"]) for P, w in zip(Ps, want)]
            nb = lqt.lqt_batch_workspace_bytes(Ps, outs)
            ws, ws2 = (torch.zeros(nb, dtype=torch.uint8, device="cuda") for _ in range(2))
            wws = torch.zeros(lqt.lqt_warm_workspace_bytes(Ps, wout), dtype=torch.uint8,
                              device="cuda")
            side, side2 = torch.cuda.Stream(), torch.cuda.Stream()
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            mode = "thread_local" if not eager_inside else "relaxed"
            with torch.cuda.graph(graph, stream=side, capture_error_mode=mode):
                lqt.lqt_solve_batched(Ps, outs, ws, side)
                for _ in range(5 if eager_inside else 0):
                    lqt.lqt_solve_batched(Ps, other, ws2, side2)
                lqt.lqt_solve_warm(Ps, wout, wws, side)
            graph.replay()
            torch.cuda.synchronize()
            for o, e, a in zip(outs, want, other):
                for k in e:
                    assert torch.equal(o[k], e[k]), k
                    assert not eager_inside or torch.equal(a[k], e[k]), k
            for o, e in zip(wout, warm):
                for k in ("v", "x", "u"):
                    assert torch.equal(o[k], e[k]), k
        except BaseException as e:  # noqa: BLE001 - reported by the test's own thread
            errors.append(e)

    for eager_inside in (False, True):
        th = threading.Thread(target=run, args=(eager_inside,))
        th.start()
        th.join()
        assert not errors, errors
