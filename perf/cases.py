"""The work a user of the LQT solver has it do, as cases to be timed.

Each case is one call of the public binding (``paper_2104_03186_gb300.lqt``) on
device-resident inputs, with the outputs and the workspace allocated once, as a
control loop or a server keeps them.  The kinds:

* ``vehicle``  one 2-D constant-velocity tracking problem (n = 4, m = 2,
  time-invariant model), from a 100-step MPC horizon to a million steps;
* ``general``  one problem whose F, c, L, U, H, r, X all change with the step,
  FP32 (refined, the default) or FP64;
* ``study``    one ill-conditioned n = 32, m = 16 problem (cond(X_k) = 1e6);
* ``batch``    a ragged batch of independent problems, n in {4, 8, 16};
* ``serving``  what a server has in hand at one time: a few dozen requests,
  n in {4, 8, 16, 32}, T log-uniform;
* ``warm``     requests whose S_k and K_k are known from an earlier solve;
* ``unicycle`` ten linearise-and-solve passes of the nonlinear tracker.

``exact`` solves the same problems with torch in 64 bits.
"""
import math

import numpy as np
import torch

from paper_2104_03186_gb300 import inputs, lqt

DEV = "cuda"
FIELDS = ("F", "c", "L", "U", "H", "r", "X", "HT", "rT", "XT", "x0")


def listed():
    return [
        # a short horizon solved inside a control loop: launches and latency
        {"name": "vehicle_100", "kind": "vehicle", "T": 100},
        # the single-problem configuration of the tracking benchmark
        {"name": "vehicle_1000", "kind": "vehicle", "T": 1000},
        # a long offline trajectory, an odd length
        {"name": "vehicle_31415", "kind": "vehicle", "T": 31415},
        # the headline: a million steps
        {"name": "vehicle_1000000", "kind": "vehicle", "T": 1000000},
        # a time-varying model with offsets and p = 3 outputs
        {"name": "general_n4_100003", "kind": "general", "n": 4, "p": 3, "T": 100003,
         "dtype": "f32"},
        # the same in FP64, for users who need 1e-11
        {"name": "general_n4_f64_30011", "kind": "general", "n": 4, "p": 3, "T": 30011,
         "dtype": "f64"},
        # a larger state, everything time-varying, refined
        {"name": "general_n16_10007", "kind": "general", "n": 16, "p": 16, "T": 10007,
         "dtype": "f32"},
        # the precision study: ill-conditioned costs at n = 32
        {"name": "study_n32_65536", "kind": "study", "T": 65536},
        # the ragged batch of the benchmark: many independent problems at once
        {"name": "batch_4096", "kind": "batch", "count": 4096, "t_min": 64, "t_max": 4096,
         "mix": 7},
        # one batch of the serving loop
        {"name": "serving_48", "kind": "serving", "count": 48, "mix": 1},
        # warm-started requests of the serving loop
        {"name": "warm_24", "kind": "warm", "count": 24, "mix": 2},
        # the nonlinear experiment: ten passes along a race track
        {"name": "unicycle_100000", "kind": "unicycle", "T": 100000, "passes": 10},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["vehicle", "vehicle", "general", "general", "study", "batch", "serving",
                       "warm", "unicycle"])
    if kind == "vehicle":
        return {"kind": kind, "T": _log_int(rng, 100, 1000000)}
    if kind == "general":
        n = rng.choice([4, 4, 8, 16])
        dtype = "f64" if n == 4 and rng.random() < 0.3 else "f32"
        top = 30000 if dtype == "f64" else {4: 100000, 8: 20000, 16: 10000}[n]
        return {"kind": kind, "n": n, "p": rng.randint(1, n + 1), "T": _log_int(rng, 300, top),
                "dtype": dtype}
    if kind == "study":
        return {"kind": kind, "T": _log_int(rng, 1000, 65536)}
    if kind == "batch":
        t_max = _log_int(rng, 128, 4096)
        return {"kind": kind, "count": _log_int(rng, 256, 4096), "t_min": t_max // 64 + 1,
                "t_max": t_max, "mix": rng.randrange(1000)}
    if kind == "serving":
        return {"kind": kind, "count": _log_int(rng, 4, 256), "mix": rng.randrange(1000)}
    if kind == "warm":
        return {"kind": kind, "count": _log_int(rng, 1, 64), "mix": rng.randrange(1000)}
    return {"kind": "unicycle", "T": _log_int(rng, 1000, 100000), "passes": 10}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _stable(g, n, count, dtype):
    """I + 0.05 N(0, 1), scaled down to a spectral radius of at most 1.05 (the
    radius is taken as ||F^1024||^(1/1024), by repeated squaring)."""
    F = 0.05 * torch.randn((count, n, n), generator=g, device=DEV, dtype=dtype)
    F.diagonal(dim1=1, dim2=2).add_(1.0)
    for lo in range(0, count, 1 << 19):
        part = F[lo:lo + (1 << 19)]
        G, logn = part.clone(), torch.zeros(len(part), device=DEV, dtype=torch.float64)
        for i in range(11):
            s = G.flatten(1).norm(dim=1).clamp_min(1e-30)
            logn += s.double().log() / (1 << i)
            G /= s[:, None, None]
            if i < 10:
                G = G @ G
        part *= (1.05 / logn.exp()).clamp_max(1.0).to(dtype)[:, None, None]
    return F


def _orthogonal(g, n, count):
    """Products of n random reflections per matrix."""
    Q = torch.eye(n, device=DEV, dtype=torch.float64).repeat(count, 1, 1)
    for _ in range(n):
        v = torch.randn((count, n, 1), generator=g, device=DEV, dtype=torch.float64)
        v /= v.norm(dim=1, keepdim=True)
        Q -= 2.0 * v @ (v.mT @ Q)
    return Q


def _spread_spd(g, n, count, cond):
    """Symmetric matrices with log-uniform eigenvalues from 1/cond to 1."""
    V = _orthogonal(g, n, count)
    e = torch.rand((count, n), generator=g, device=DEV, dtype=torch.float64)
    lo, hi = e.amin(1, keepdim=True), e.amax(1, keepdim=True)
    lam = 10.0 ** (-math.log10(cond) * (1.0 - (e - lo) / (hi - lo)))
    X = (V * lam[:, None, :]) @ V.mT
    return 0.5 * (X + X.mT)


def _single(case, seed):
    """The arrays of a one-problem case (the problem's element type), and its T."""
    kind, T = case["kind"], case["T"]
    if kind in ("vehicle", "unicycle"):
        prob = inputs.vehicle(T, seed) if kind == "vehicle" else inputs.unicycle_track(T, seed)
        return {f: torch.from_numpy(getattr(prob, f)).to(DEV).float()
                for f in FIELDS if getattr(prob, f) is not None}
    g = _generator(seed)
    f64 = torch.float64

    def normal(*shape):
        return torch.randn(shape, generator=g, device=DEV, dtype=f64)

    if kind == "study":
        n, m = 32, 16
        F = 0.99 * _orthogonal(g, n, T)
        for _ in range(2):
            F += 0.01 / n * normal(T, n, 1) @ normal(T, 1, n)
        a = {"F": F, "L": normal(T, n, m) / math.sqrt(n),
             "U": 1e-3 * torch.eye(m, device=DEV, dtype=f64)[None],
             "H": torch.eye(n, device=DEV, dtype=f64)[None], "r": normal(T, n),
             "X": _spread_spd(g, n, T, 1e6), "HT": torch.eye(n, device=DEV, dtype=f64),
             "rT": normal(n), "XT": _spread_spd(g, n, 1, 1e6)[0], "x0": normal(n)}
        return {k: v.float().contiguous() for k, v in a.items()}
    n, p = case["n"], case["p"]
    m = n // 2
    B, D, E = normal(T, p, p), normal(T, m, m), normal(n, n)
    a = {"F": _stable(g, n, T, f64), "c": 0.1 * normal(T, n), "L": normal(T, n, m) / math.sqrt(n),
         "U": 0.1 * torch.eye(m, device=DEV, dtype=f64) + 0.1 / m * D @ D.mT,
         "H": normal(T, p, n) / math.sqrt(n), "r": normal(T, p), "X": B @ B.mT / p,
         "HT": normal(n, n) / math.sqrt(n), "rT": normal(n), "XT": E @ E.mT / n, "x0": normal(n)}
    return {k: v.to(f64 if case["dtype"] == "f64" else torch.float32).contiguous()
            for k, v in a.items()}


def _requests(case):
    """(n, T) of each problem of a many-problem case, drawn from its mix."""
    rng = np.random.default_rng(case["mix"])
    count = case["count"]
    if case["kind"] == "batch":
        ns = rng.choice([4, 8, 16], size=count)
        Ts = rng.integers(case["t_min"], case["t_max"] + 1, size=count)
    else:
        ns = rng.choice([4, 8, 16, 32] if case["kind"] == "serving" else [8, 16, 32], size=count)
        Ts = np.rint(np.exp(rng.uniform(math.log(32), math.log(2048), size=count))).astype(int)
    return [(int(n), int(T)) for n, T in zip(ns, Ts)]


def _many(case, seed):
    """Per state size n: the T of its problems and their arrays, packed one
    problem after another (diagonal tracking: H = I, diagonal X_k, U = 0.1 I)."""
    g = _generator(seed)
    found = {}
    for n, T in _requests(case):
        found.setdefault(n, []).append(T)
    packs = {}
    for n in sorted(found):
        Ts = found[n]
        m, total, count = n // 2, sum(Ts), len(Ts)

        def normal(*shape):
            return torch.randn(shape, generator=g, device=DEV)

        def diagonal(k):
            return torch.diag_embed(torch.rand((k, n), generator=g, device=DEV) * 1.5 + 0.5)

        packs[n] = Ts, {
            "F": _stable(g, n, total, torch.float32), "L": normal(total, n, m) / math.sqrt(n),
            "U": 0.1 * torch.eye(m, device=DEV)[None], "H": torch.eye(n, device=DEV)[None],
            "r": normal(total, n), "X": diagonal(total), "HT": torch.eye(n, device=DEV),
            "rT": normal(count, n), "XT": diagonal(count), "x0": normal(count, n)}
    return packs


# ---------------------------------------------------------------------------
# the framework
# ---------------------------------------------------------------------------

def _outputs(n, m, steps, ends, dtype):
    rows = {"S": (steps + ends, n, n), "v": (steps + ends, n), "K": (steps, m, n),
            "x": (steps + ends, n), "u": (steps, m)}
    return {k: torch.empty(s, dtype=dtype, device=DEV) for k, s in rows.items()}


def _problems(n, Ts, a, out):
    """A Problem and its output views for each problem of a pack."""
    probs, outs = [], []
    at = 0
    for i, T in enumerate(Ts):
        mine = {f: a[f] if f in ("U", "H", "HT") else a[f][i] if f in ("rT", "XT", "x0")
                else a[f][at:at + T] for f in a}
        probs.append(lqt.Problem(n, n // 2, n, n, T, lqt.LQT_F32, mine))
        outs.append({f: out[f][at:at + T] if f in ("K", "u") else out[f][at + i:at + i + T + 1]
                     for f in out})
        at += T
    return probs, outs


def _descriptors(probs, outs):
    arr = (lqt.lqt_batch_item * len(probs))()
    for i, (p, o) in enumerate(zip(probs, outs)):
        arr[i].problem = p.struct
        arr[i].solution = lqt.solution_struct(o, p)
    return np.frombuffer(arr, dtype=lqt.BATCH_ITEM).copy()


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serving", "warm"):
        packs = _many(case, seed)
        outs, probs, views = {}, [], []
        for n, (Ts, a) in packs.items():
            outs[n] = _outputs(n, n // 2, sum(Ts), len(Ts), torch.float32)
            P, o = _problems(n, Ts, a, outs[n])
            probs += P
            views += o
        items = _descriptors(probs, views)
        size = lqt.lqt_batch_workspace_bytes_array(items)
        if kind == "warm":
            # the earlier solve whose S and K the warm requests reuse
            first = torch.empty(size, dtype=torch.uint8, device=DEV)
            lqt.lqt_solve_batched_array(items, first)
            size = lqt.lqt_warm_workspace_bytes_array(items)
        ws = torch.empty(size, dtype=torch.uint8, device=DEV)
        return {"kind": kind, "items": items, "out": outs, "ws": ws, "keep": packs}
    a = _single(case, seed)
    n, m, p, pT = a["F"].shape[-1], a["L"].shape[-1], a["H"].shape[-2], a["HT"].shape[0]
    f64 = a["F"].dtype == torch.float64
    P = lqt.Problem(n, m, p, pT, case["T"], lqt.LQT_F64 if f64 else lqt.LQT_F32, a)
    state = {"kind": kind, "problem": P, "out": P.allocate_outputs()}
    if kind == "unicycle":
        state["nl"] = lqt.nonlinear(case["passes"])
        size = lqt.lqt_nonlinear_workspace_bytes(P, state["nl"])
    else:
        size = lqt.lqt_workspace_bytes(P)
    state["ws"] = torch.empty(size, dtype=torch.uint8, device=DEV)
    return state


def run(state):
    kind = state["kind"]
    if kind in ("batch", "serving"):
        lqt.lqt_solve_batched_array(state["items"], state["ws"])
        return {"n%d_%s" % (n, f): o[f] for n, o in state["out"].items() for f in o}
    if kind == "warm":
        lqt.lqt_solve_warm_array(state["items"], state["ws"])
        return {"n%d_%s" % (n, f): o[f] for n, o in state["out"].items() for f in ("v", "x", "u")}
    if kind == "unicycle":
        lqt.lqt_solve_nonlinear(state["problem"], state["nl"], state["out"], state["ws"])
    else:
        lqt.lqt_solve(state["problem"], state["out"], state["ws"])
    return state["out"]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _step_flops(n, m, p, general_h):
    """One Riccati step with its gains and one rollout step."""
    cost = 2 * p * p * n + 2 * p * n * n if general_h else 0
    gains = 2 * n * n * m + 2 * n * n * n + 2 * n * m * m + 2 * n * n * m + m ** 3 // 3 \
        + 2 * m * m * (n + 1)
    return cost + gains + 2 * n * n * n + 2 * n * n * m + 8 * n * n + 8 * n * m


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serving", "warm"):
        size = {"bytes": 0, "flops": 0}
        for n, T in _requests(case):
            m = n // 2
            read = n * n + n * m + n * n + n  # F, L, X, r
            # warm requests bring S and K and ask for v, x, u
            size["bytes"] += 4 * T * (read + n * n + n * m + 2 * n + m)
            size["flops"] += T * (8 * n * n + 12 * n * m + 2 * n * m * (n + m) if kind == "warm"
                                  else _step_flops(n, m, n, False))
        return size
    T = case["T"]
    if kind == "general":
        n, p, es = case["n"], case["p"], 8 if case["dtype"] == "f64" else 4
        m = n // 2
        read = n * n + n + n * m + m * m + p * n + p + p * p
    elif kind == "study":
        n, m, p, es, read = 32, 16, 32, 4, 32 * 32 + 32 * 16 + 32 + 32 * 32
    elif kind == "unicycle":
        n, m, p, es, read = 4, 2, 3, 4, 3 + 9
    else:
        n, m, p, es, read = 4, 2, 2, 4, 2
    written = n * n + n + m * n + n + m
    # time-invariant H^T X H is formed once (vehicle); H = I needs no products (study)
    flops = _step_flops(n, m, p, kind in ("general", "unicycle"))
    return {"bytes": int(es * T * (read + written)), "flops": int(T * flops * case.get("passes", 1))}


# ---------------------------------------------------------------------------
# 64 bits
# ---------------------------------------------------------------------------

class _Lanes:
    """Stretches [lo, lo + length) of the packed steps, longest first, walked
    side by side in 64 bits."""

    def __init__(self, a, lo, length):
        order = sorted(range(len(lo)), key=lambda i: -length[i])
        self.order = torch.tensor(order, device=DEV)
        self.a = a
        self.n, self.m = a["F"].shape[-1], a["L"].shape[-1]
        self.lo = torch.tensor([lo[i] for i in order], device=DEV)
        self.len = torch.tensor([length[i] for i in order], device=DEV)
        lens = [length[i] for i in order]
        self.top = lens[0] if lens else 0
        # lanes still walking at the j-th step
        self.active = np.searchsorted(-np.asarray(lens), -np.arange(self.top), side="left").tolist()

    def at(self, f, idx):
        x = self.a.get(f)
        if x is None:
            return None
        return x.double().expand((len(idx),) + x.shape[1:]) if x.shape[0] == 1 else x[idx].double()

    def step(self, idx):
        F, L, U = (self.at(f, idx) for f in ("F", "L", "U"))
        H, X = self.at("H", idx), self.at("X", idx)
        c, r = self.at("c", idx), self.at("r", idx)
        c = (torch.zeros((len(idx), self.n), device=DEV, dtype=torch.float64) if c is None else c)
        HX = H.mT @ X
        q = torch.zeros_like(c)[..., None] if r is None else HX @ r[..., None]
        return F, c[..., None], L, U, HX @ H, q

    def fold(self):
        """The conditional value element (A, b, C, eta, J) of each stretch."""
        C0, n = len(self.lo), self.n
        eye = torch.eye(n, device=DEV, dtype=torch.float64)
        A = eye.repeat(C0, 1, 1)
        C, J = torch.zeros_like(A), torch.zeros_like(A)
        b = torch.zeros((C0, n, 1), device=DEV, dtype=torch.float64)
        e = torch.zeros_like(b)
        for j in range(self.top):
            k = self.active[j]
            F, c, L, U, Q, q = self.step((self.lo + self.len - 1 - j)[:k])
            C1 = L @ torch.linalg.solve_ex(U, L.mT)[0]
            A2, b2, C2, e2, J2 = A[:k], b[:k], C[:k], e[:k], J[:k]
            rhs = torch.cat([F, c + C1 @ e2, C1], dim=2)
            Z = torch.linalg.solve_ex(eye + C1 @ J2, rhs)[0]
            X1, x2, X3 = Z[..., :n], Z[..., n:n + 1], Z[..., n + 1:]
            Jn = F.mT @ (J2 @ X1) + Q
            Cn = A2 @ X3 @ A2.mT + C2
            e[:k] = X1.mT @ (e2 - J2 @ c) + q
            b[:k] = A2 @ x2 + b2
            A[:k] = A2 @ X1
            C[:k] = 0.5 * (Cn + Cn.mT)
            J[:k] = 0.5 * (Jn + Jn.mT)
        return A, b, C, e, J

    def riccati(self, S, v, put):
        """From (S, v) at each stretch's end: put(idx, lanes, S, v, K) per
        step; returns the feedforward per step and each stretch's closed loop."""
        steps = int((self.lo + self.len).max())
        d = torch.zeros((steps, self.m, 1), device=DEV, dtype=torch.float64)
        Phi = torch.eye(self.n, device=DEV, dtype=torch.float64).repeat(len(self.lo), 1, 1)
        gam = torch.zeros((len(self.lo), self.n, 1), device=DEV, dtype=torch.float64)
        S, v = S.clone(), v.clone()
        for j in range(self.top):
            k = self.active[j]
            idx = (self.lo + self.len - 1 - j)[:k]
            F, c, L, U, Q, q = self.step(idx)
            SL, SF = S[:k] @ L, S[:k] @ F
            w = v[:k] - S[:k] @ c
            K = torch.linalg.solve_ex(U + L.mT @ SL, torch.cat([L.mT @ SF, L.mT @ w], dim=2))[0]
            K, dk = K[..., :self.n], K[..., self.n:]
            Ft = F - L @ K
            Sn = F.mT @ (SF - SL @ K) + Q
            S[:k] = 0.5 * (Sn + Sn.mT)
            v[:k] = Ft.mT @ w + q
            d[idx] = dk
            gam[:k] += Phi[:k] @ (c + L @ dk)
            Phi[:k] = Phi[:k] @ Ft
            put(idx, self.order[:k], S[:k], v[:k, :, 0], K)
        return d, Phi, gam

    def roll(self, x, K, d, put):
        x = x.clone()
        for j in range(self.top):
            k = self.active[j]
            idx = (self.lo + j)[:k]
            F, c, L = self.at("F", idx), self.at("c", idx), self.at("L", idx)
            u = d[idx] - K[idx] @ x[:k]
            put(idx, self.order[:k], x[:k, :, 0], u[..., 0])
            x[:k] = F @ x[:k] + L @ u + (0.0 if c is None else c[..., None])
        return x


def _terminal(a):
    HT, XT = a["HT"].double(), a["XT"].double()
    HX = HT.mT @ XT
    rT = a.get("rT")
    q = HX @ rT.double()[..., None] if rT is not None else torch.zeros_like(a["x0"]).double()[..., None]
    return HX @ HT, q


def _one64(a, T):
    """One problem, in about sqrt(T) stretches."""
    n, m = a["F"].shape[-1], a["L"].shape[-1]
    B = max(1, int(math.ceil(math.sqrt(T))))
    lo = list(range(0, T, B))
    lanes = _Lanes(a, lo, [min(B, T - s) for s in lo])
    ST, vT = _terminal(a)
    el = [t.cpu().numpy() for t in lanes.fold()]
    S, v = ST.cpu().numpy(), vT.cpu().numpy()
    ends = []
    for i in reversed(range(len(lo))):
        ends.append((S, v))
        A, b, C, e, J = (t[i] for t in el)
        X1 = np.linalg.solve(np.eye(n) + C @ S, A)
        S, v = A.T @ (S @ X1) + J, X1.T @ (v - S @ b) + e
        S = 0.5 * (S + S.T)
    ends.reverse()

    def dev(xs):
        return torch.from_numpy(np.stack(xs)).to(DEV)

    out = _outputs(n, m, T, 1, torch.float64)

    def put(idx, _, S, v, K):
        out["S"][idx], out["v"][idx], out["K"][idx] = S, v, K

    d, Phi, gam = lanes.riccati(dev([s for s, _ in ends]), dev([v for _, v in ends]), put)
    out["S"][T], out["v"][T] = ST, vT[:, 0]
    Phi, gam = Phi.cpu().numpy(), gam.cpu().numpy()
    x, starts = a["x0"].double().cpu().numpy()[:, None], []
    for i in range(len(lo)):
        starts.append(x)
        x = Phi[i] @ x + gam[i]

    def put_x(idx, _, x, u):
        out["x"][idx], out["u"][idx] = x, u

    last = lanes.roll(dev(starts), out["K"], d, put_x)
    out["x"][T] = last[-1, :, 0]
    return out


def _pack64(Ts, a):
    """The problems of one state size, side by side."""
    n, m, count = a["F"].shape[-1], a["L"].shape[-1], len(Ts)
    lo = np.concatenate([[0], np.cumsum(Ts)[:-1]]).tolist()
    lanes = _Lanes(a, lo, Ts)
    out = _outputs(n, m, sum(Ts), count, torch.float64)
    ST, vT = _terminal(a)
    end = torch.tensor(np.cumsum(Ts) + np.arange(count), device=DEV)
    out["S"][end], out["v"][end] = ST, vT[..., 0]

    def put(idx, lane, S, v, K):
        out["S"][idx + lane], out["v"][idx + lane], out["K"][idx] = S, v, K

    d, _, _ = lanes.riccati(ST[lanes.order], vT[lanes.order], put)

    def put_x(idx, lane, x, u):
        out["x"][idx + lane], out["u"][idx] = x, u

    x0 = a["x0"].double()[..., None]
    out["x"][end[lanes.order]] = lanes.roll(x0[lanes.order], out["K"], d, put_x)[..., 0]
    return out


def _linearised(a, x, u, dt=0.1):
    """The unicycle's Taylor expansion about the nominal (x, u)."""
    T = len(u)
    th, s = x[:T, 2], x[:T, 3]
    F = torch.eye(4, device=DEV, dtype=torch.float64).repeat(T, 1, 1)
    F[:, 0, 2], F[:, 0, 3] = -s * th.sin() * dt, th.cos() * dt
    F[:, 1, 2], F[:, 1, 3] = s * th.cos() * dt, th.sin() * dt
    L = torch.zeros((1, 4, 2), device=DEV, dtype=torch.float64)
    L[0, 2, 1] = L[0, 3, 0] = dt
    f = x[:T].clone()
    f[:, 0] += s * th.cos() * dt
    f[:, 1] += s * th.sin() * dt
    f[:, 2] += u[:, 1] * dt
    f[:, 3] += u[:, 0] * dt
    c = f - (F @ x[:T, :, None])[..., 0] - (L @ u[..., None])[..., 0]
    return {**a, "F": F, "L": L, "c": c}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serving", "warm"):
        want = ("v", "x", "u") if kind == "warm" else ("S", "v", "K", "x", "u")
        found = {}
        for n, (Ts, a) in _many(case, seed).items():
            out = _pack64(Ts, a)
            found.update({"n%d_%s" % (n, f): out[f] for f in want})
        return found
    a, T = _single(case, seed), case["T"]
    if kind != "unicycle":
        return _one64(a, T)
    x = a["x0"].double().repeat(T + 1, 1)
    u = torch.zeros((T, 2), device=DEV, dtype=torch.float64)
    out = None
    for _ in range(case["passes"]):
        out = _one64(_linearised(a, x, u), T)
        x, u = out["x"], out["u"]
    return out
