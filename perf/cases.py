"""The work that users of this package have it do, as cases that can be timed and compared.

Kinds (field "kind" of a case):

  prob        one click probability: torontonian() on a prepared state
  batch       many click probabilities of uneven size in one torontonian_batch() call
  sample      chain-rule samples: sample(), with forced click positions, free, or postselected on a click count
  subset_sum  the signed subset sum of an explicit matrix: subset_sum()
  build       a state from (U, r, eta) with its covariance read back: build_state(want_V=True)
  from_v      a state from a covariance and one block of its Sigma^-1: state_from_V(), sigma_inv_block()

A program keeps its Context (and with it the workspaces) and the states it asks about; what it
has anew for each call is the click pattern, the seed or the matrix.
"""
import math

import numpy as np
import torch

import gbs_inputs as gi
import paper_1810_00900_gb300 as gbs


def listed():
    return [
        # The smallest calls: one pattern of a small chip, where launches and waits are the cost.
        {"name": "prob_small", "kind": "prob", "M": 8, "N": 6, "r": 0.5, "eta": 1.0, "prec": "auto"},
        # An ordinary certified probability of a lossy 100-mode state.
        {"name": "prob_mid", "kind": "prob", "M": 100, "N": 13, "r": 0.7, "eta": 0.6, "prec": "auto"},
        # The benchmark's single large pattern, certified: 2^24 subset determinants that cancel by 1e25.
        {"name": "prob_large_certified", "kind": "prob", "M": 200, "N": 24, "r": 0.8, "eta": 1.0, "prec": "auto"},
        # As many subsets in FP64, on a bright state (13 dB) where FP64 carries the cancellation.
        {"name": "prob_large_fp64", "kind": "prob", "M": 26, "N": 24, "r": 1.5, "eta": 0.95, "prec": "fp64"},
        # Many users' requests of uneven size in one call, certified.
        {"name": "batch_certified", "kind": "batch", "requests": 256, "states": 6, "M": 100, "N_lo": 8, "N_hi": 20,
         "r": 0.8, "eta": 0.7, "prec": "auto"},
        # A distribution over patterns of a small bright chip in FP64 (verification, likelihoods).
        {"name": "batch_fp64", "kind": "batch", "requests": 1500, "states": 4, "M": 17, "N_lo": 5, "N_hi": 17,
         "r": 1.4, "eta": 0.9, "prec": "fp64"},
        # The paper's forced-outcome chain (uniform click positions), several trajectories together.
        {"name": "sample_forced", "kind": "sample", "M": 200, "n": 24, "N_post": 17, "forced": True, "graph": False,
         "r": 0.7, "eta": 1.0, "attempts": 1},
        # Free sampling of a small chip: many short steps.
        {"name": "sample_free", "kind": "sample", "M": 30, "n": 64, "N_post": 0, "forced": False, "graph": False,
         "r": 0.6, "eta": 0.8, "attempts": 1},
        # Dense-subgraph search: samples of a graph state postselected on a click count.
        {"name": "sample_graph", "kind": "sample", "M": 100, "n": 8, "N_post": 9, "forced": False, "graph": True,
         "r": 0.0, "eta": 1.0, "attempts": 12},
        # An explicit Hermitian matrix in the complex basis, FP64 (the defaults of subset_sum).
        {"name": "subset_sum_complex", "kind": "subset_sum", "n": 19, "r": 1.4, "eta": 0.9, "basis": "complex",
         "prec": "fp64"},
        # A state built from its factors, covariance read back.
        {"name": "build_covariance", "kind": "build", "M": 333, "r": 0.7, "eta": 0.8},
        # A state given by its covariance (dense inversion), and a block of the inverse.
        {"name": "from_covariance", "kind": "from_v", "M": 120, "N": 16, "r": 0.8, "eta": 0.7},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["prob", "prob", "prob", "batch", "batch", "sample", "sample", "subset_sum", "build", "from_v"])
    eta = round(rng.uniform(0.5, 1.0), 3)
    if kind == "prob" and rng.random() < 0.5:  # certified, dim states of any size
        N = rng.randint(4, 23)
        return {"kind": kind, "M": log_int(max(8, N), 300), "N": N, "r": round(rng.uniform(0.4, 1.0), 3), "eta": eta,
                "prec": "auto"}
    if kind == "prob":  # FP64, bright states
        N = rng.randint(6, 24)
        return {"kind": kind, "M": N + rng.randint(0, 2), "N": N, "r": round(rng.uniform(1.3, 1.6), 3),
                "eta": round(rng.uniform(0.85, 1.0), 3), "prec": "fp64"}
    if kind == "batch" and rng.random() < 0.5:
        lo = rng.randint(4, 10)
        return {"kind": kind, "requests": log_int(8, 300), "states": rng.randint(1, 6), "M": log_int(24, 150),
                "N_lo": lo, "N_hi": rng.randint(lo, 19), "r": round(rng.uniform(0.5, 1.0), 3), "eta": eta, "prec": "auto"}
    if kind == "batch":
        M = rng.randint(12, 17)
        return {"kind": kind, "requests": log_int(16, 1500), "states": rng.randint(1, 4), "M": M,
                "N_lo": rng.randint(M // 3, M - 1), "N_hi": M, "r": round(rng.uniform(1.3, 1.5), 3),
                "eta": round(rng.uniform(0.85, 1.0), 3), "prec": "fp64"}
    if kind == "sample" and rng.random() < 0.5:
        M = log_int(40, 220)
        return {"kind": kind, "M": M, "n": log_int(1, 24), "N_post": rng.randint(4, 16), "forced": True, "graph": False,
                "r": round(rng.uniform(0.4, 0.9), 3), "eta": eta, "attempts": 1}
    if kind == "sample":
        return {"kind": kind, "M": rng.randint(12, 36), "n": log_int(2, 64), "N_post": 0, "forced": False,
                "graph": False, "r": round(rng.uniform(0.3, 0.6), 3), "eta": eta, "attempts": 1}
    if kind == "subset_sum":
        return {"kind": kind, "n": rng.randint(6, 19), "r": round(rng.uniform(1.3, 1.5), 3),
                "eta": round(rng.uniform(0.85, 1.0), 3), "basis": rng.choice(["complex", "real"]), "prec": "fp64"}
    if kind == "build":
        return {"kind": kind, "M": log_int(20, 400), "r": round(rng.uniform(0.3, 1.0), 3), "eta": eta}
    M = log_int(10, 150)
    return {"kind": kind, "M": M, "N": rng.randint(2, min(M, 20)), "r": round(rng.uniform(0.3, 1.0), 3), "eta": eta}


# ------------------------------------------------------------------ inputs --

def _requests(case, seed):
    """(states' parameters, state index per request, patterns) of a prob or batch case."""
    n_states = case.get("states", 1)
    params = []
    for i in range(n_states):
        # the modes' squeezing around the stated value, as fabricated chips have it
        r = case["r"] * gi.uniform_range(seed + 101 * i, "squeezing", case["M"], 0.95, 1.05)
        params.append(gi.StateParams(gi.haar_unitary(case["M"], seed + 101 * i), r, case["eta"]))
    if case["kind"] == "prob":
        return params, [0], [gi.random_modes(case["M"], case["N"], seed)]
    rng = np.random.default_rng(seed)
    sizes = rng.integers(case["N_lo"], case["N_hi"] + 1, case["requests"])
    which = rng.integers(0, n_states, case["requests"])
    patterns = [np.sort(rng.choice(case["M"], int(s), replace=False)).astype(np.int32) for s in sizes]
    return params, [int(w) for w in which], patterns


def _matrix(case, seed):
    """Sigma^-1 of a bright n-mode state: the explicit matrix of a subset_sum case."""
    p = gi.uniform_squeezed_state(case["n"], case["r"], seed, case["eta"])
    h, _ = _click_block(p, np.arange(case["n"]), np.float64)
    if case["basis"] == "real":
        return h
    # per mode, (a, a^+) = q (x, p) with q = [[1, i], [1, -i]] / sqrt 2: q h q^+ blockwise
    q = np.kron(np.eye(case["n"]), np.array([[1, 1j], [1, -1j]]) / math.sqrt(2.0))
    return q @ h @ q.conj().T


def _covariance(p):
    a = 0.5 * (p.U * np.cosh(2 * p.r)) @ p.U.conj().T
    b = 0.5 * (p.U * np.sinh(2 * p.r)) @ p.U.T
    v = np.block([[a, b], [b.conj(), a.conj()]])
    return p.eta * v + (1.0 - p.eta) * 0.5 * np.eye(2 * p.M)


def _state_params(case, seed):
    r = case["r"] * gi.uniform_range(seed, "squeezing", case["M"], 0.8, 1.2)
    return gi.StateParams(gi.haar_unitary(case["M"], seed), r, case["eta"])


def prepare(case, seed):
    ctx = gbs.Context(0)
    kind = case["kind"]
    state = {"case": case, "ctx": ctx}
    if kind in ("prob", "batch"):
        params, which, patterns = _requests(case, seed)
        built = [gbs.build_state(ctx, p.U, p.r, p.eta) for p in params]
        state.update(states=[built[w] for w in which], patterns=patterns)
    elif kind == "sample":
        if case["graph"]:
            p = gi.graph_state(gi.planted_graph(case["M"], seed), 2.0 * case["N_post"], case["eta"])
        else:
            p = _state_params(case, seed)
        clicks = None
        if case["forced"]:
            clicks = gbs.draw_click_positions(case["M"], case["N_post"], seed, case["n"])
        state.update(st=gbs.build_state(ctx, p.U, p.r, p.eta), seed=seed, clicks=clicks)
    elif kind == "subset_sum":
        state.update(G=_matrix(case, seed))
    elif kind == "build":
        state.update(p=_state_params(case, seed))
    else:
        state.update(V=_covariance(_state_params(case, seed)), modes=gi.random_modes(case["M"], case["N"], seed))
    return state


def _prob_outputs(probs):
    out = {k: np.array([getattr(q, k) for q in probs]) for k in ("p", "tor_value", "abs_sum", "kappa", "err_bound",
                                                                  "logdet_sigma")}
    out["prec"] = np.array([gbs.PREC[q.prec] for q in probs], dtype=np.int64)
    return out


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "prob":
        return _prob_outputs([gbs.torontonian(ctx, state["states"][0], state["patterns"][0], case["prec"])])
    if kind == "batch":
        probs, status = gbs.torontonian_batch(ctx, state["states"], state["patterns"], case["prec"], check=False,
                                              return_status=True)
        return {**_prob_outputs(probs), "status": int(status)}
    if kind == "sample":
        patterns, p0, _, status = gbs.sample(ctx, state["st"], case["n"], state["seed"], case["N_post"],
                                             case["attempts"], forced_clicks=state["clicks"], want_p0=True)
        return {"patterns": patterns, "p0": p0, "status": int(status)}
    if kind == "subset_sum":
        inc, exc, tor, total = gbs.subset_sum(ctx, state["G"], case["basis"], case["prec"])
        return {"inc": inc, "exc": exc, "tor": tor, "abs_sum": total}
    if kind == "build":
        p = state["p"]
        st, V = gbs.build_state(ctx, p.U, p.r, p.eta, want_V=True)
        out = {"V": V, "logdet": st.logdet_sigma}
        st.free()
        return out
    st = gbs.state_from_V(ctx, state["V"])
    out = {"block": gbs.sigma_inv_block(ctx, st, state["modes"]), "logdet": st.logdet_sigma}
    st.free()
    return out


# -------------------------------------------------------------------- work --

def _tree_flops(n):
    """Subset tree over n modes: a rank-2 update of 2t rows per include child with t modes left
    (8 t^2 flops), one inverse square root and one addition per subset."""
    return sum(2.0 ** (n - 1 - t) * 8.0 * t * t for t in range(n)) + 2.0 * 2.0 ** n


def work(case):
    kind = case["kind"]
    if kind == "prob":
        M, N = case["M"], case["N"]
        return {"bytes": 16 * M * N + 16 * M + 64, "flops": _tree_flops(N) + 8 * M * N * (N + 1)}
    if kind == "batch":
        sizes = range(case["N_lo"], case["N_hi"] + 1)
        one = sum(_tree_flops(N) + 8 * case["M"] * N * (N + 1) for N in sizes) / len(sizes)
        return {"bytes": case["states"] * 16 * case["M"] ** 2 + case["requests"] * 64, "flops": case["requests"] * one}
    if kind == "sample":
        M, n = case["M"], case["n"]
        # clicks spread evenly over the chain; a step's tree is over the clicks so far
        N = case["N_post"] if case["N_post"] else min(20, max(1, int(M * 0.3)))
        trees = sum(_tree_flops(max(1, (N * k) // M)) for k in range(M))
        cond = sum(4.0 * (2 * k + 2 * N) ** 2 for k in range(M)) / 2
        return {"bytes": n * (32 * M * M + 9 * M), "flops": n * (trees + cond)}
    if kind == "subset_sum":
        c = 4 if case["basis"] == "complex" else 1
        return {"bytes": (16 if c == 4 else 8) * 4 * case["n"] ** 2 + 80, "flops": c * _tree_flops(case["n"])}
    M = case["M"]
    if kind == "build":
        return {"bytes": 16 * M * M + 64 * M * M, "flops": 8.0 * M ** 3}
    return {"bytes": 64 * M * M + 64 * case["N"] ** 2, "flops": 4 * 2.0 * (2 * M) ** 3}


# ------------------------------------------------------------------- exact --

def _click_block(p, modes, dt):
    """(Sigma^-1)_S in the real x/p basis and log det Sigma, in numpy's type dt."""
    u = p.U[np.asarray(modes)]
    x, y = u.real.astype(dt), u.imag.astype(dt)
    e = np.exp(2 * p.r.astype(dt))
    eta = dt(p.eta)
    dp, dm = (eta * e + 2 - eta) / 2, (eta / e + 2 - eta) / 2
    al, be = (1 / dp + 1 / dm) / 2, (1 / dp - 1 / dm) / 2
    ar, ai = (x * al) @ x.T + (y * al) @ y.T, (y * al) @ x.T - (x * al) @ y.T
    br, bi = (x * be) @ x.T - (y * be) @ y.T, (x * be) @ y.T + (y * be) @ x.T
    n = len(modes)
    h = np.zeros((2 * n, 2 * n), dtype=dt)
    h[0::2, 0::2], h[1::2, 0::2] = ar + br, ai + bi
    h[0::2, 1::2], h[1::2, 1::2] = bi - ai, ar - br
    return h, np.sum(np.log(dp) + np.log(dm))


class _Pair:
    """A tensor as an unevaluated sum of two float64 tensors: 64-bit arithmetic alone loses what the
    alternating sum cancels, so the sum is carried with twice the digits."""

    def __init__(self, hi, lo=None):
        self.hi, self.lo = hi, torch.zeros_like(hi) if lo is None else lo

    def __getitem__(self, k):
        return _Pair(self.hi[k], self.lo[k])

    @staticmethod
    def norm(s, e):
        h = s + e
        return _Pair(h, e - (h - s))

    def __add__(self, o):
        s = self.hi + o.hi
        b = s - self.hi
        return _Pair.norm(s, (self.hi - (s - b)) + (o.hi - b) + (self.lo + o.lo))

    def __neg__(self):
        return _Pair(-self.hi, -self.lo)

    def __sub__(self, o):
        return self + (-o)

    @staticmethod
    def split(a):
        t = 134217729.0 * a
        h = t - (t - a)
        return h, a - h

    def __mul__(self, o):
        p = self.hi * o.hi
        a, b = _Pair.split(self.hi)
        c, d = _Pair.split(o.hi)
        e = ((a * c - p) + a * d + b * c) + b * d
        return _Pair.norm(p, e + (self.hi * o.lo + self.lo * o.hi))

    def rsqrt(self):
        x = _Pair(1.0 / torch.sqrt(self.hi))
        half = _Pair(torch.full_like(self.hi, 0.5))
        one = _Pair(torch.ones_like(self.hi))
        for _ in range(2):
            x = x + half * (x * (one - self * (x * x)))
        return x


def _cat(a, b):
    return _Pair(torch.cat([a.hi, b.hi], 1), torch.cat([a.lo, b.lo], 1))


def _tor(blocks):
    """(Tor, sum of the terms' magnitudes) of equally large real x/p blocks [T, 2n, 2n] (numpy)."""
    dev = "cuda"
    hi = blocks.astype(np.float64)
    lo = (blocks - hi).astype(np.float64)
    c = _Pair(torch.tensor(hi, device=dev)[:, None], torch.tensor(lo, device=dev)[:, None])
    n = blocks.shape[1] // 2
    s = _Pair(torch.ones(blocks.shape[0], 1, dtype=torch.float64, device=dev))
    sign = torch.ones(1, 1, dtype=torch.float64, device=dev)
    for _ in range(n):
        a, b, d = c[:, :, 0, 0], c[:, :, 1, 0], c[:, :, 1, 1]
        g = (a * d - b * b).rsqrt()
        inv = g * g
        kaa, kab, kbb = (d * inv)[:, :, None], (-(b * inv))[:, :, None], (a * inv)[:, :, None]
        u0, u1, rest = c[:, :, 2:, 0], c[:, :, 2:, 1], c[:, :, 2:, 2:]
        l0, l1 = u0 * kaa + u1 * kab, u0 * kab + u1 * kbb
        upd = rest - l0[:, :, :, None] * u0[:, :, None, :] - l1[:, :, :, None] * u1[:, :, None, :]
        c = _cat(rest, upd)
        s = _cat(s, s * g)
        sign = torch.cat([-sign, sign], 1)
    t = _Pair(s.hi * sign, s.lo * sign)
    m = s
    while t.hi.shape[1] > 1:  # pairwise
        t, m = t[:, 0::2] + t[:, 1::2], m[:, 0::2] + m[:, 1::2]
    return (t.hi + t.lo)[:, 0].cpu().numpy(), (m.hi + m.lo)[:, 0].cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("prob", "batch"):
        top = case["N"] if kind == "prob" else case["N_hi"]
        # dim states of many clicks cancel more than twice 64 bits carry; the largest trees take too long
        if top > (13 if case["prec"] == "auto" else 24) or (kind == "batch" and top > 17):
            return None
        params, which, patterns = _requests(case, seed)
        n = len(patterns)
        tor, mag, ld = np.zeros(n), np.zeros(n), np.zeros(n)
        groups = {}
        for i, pat in enumerate(patterns):
            groups.setdefault(len(pat), []).append(i)
        for size, idx in groups.items():
            step = max(1, (1 << 21) >> size)
            for k in range(0, len(idx), step):
                part = idx[k:k + step]
                blocks = [_click_block(params[which[i]], patterns[i], np.longdouble) for i in part]
                tor[part], mag[part] = _tor(np.stack([b for b, _ in blocks]))
                ld[part] = [float(v) for _, v in blocks]
        out = {"p": tor * np.exp(-0.5 * ld), "tor_value": tor, "abs_sum": mag, "kappa": mag / np.abs(tor),
               "err_bound": None, "logdet_sigma": ld, "prec": None}
        if case["prec"] == "auto":  # the rung taken says which magnitudes it sums (FP64P: of groups of four terms)
            out["abs_sum"] = out["kappa"] = None
        if kind == "batch":
            out["status"] = None
        return out
    if kind == "sample":
        return None
    if kind == "subset_sum":
        if case["n"] > 20:
            return None
        p = gi.uniform_squeezed_state(case["n"], case["r"], seed, case["eta"])
        h, _ = _click_block(p, np.arange(case["n"]), np.longdouble)
        tor, mag = _tor(h[None])
        return {"inc": None, "exc": None, "tor": np.array([tor[0], 0.0, 0.0]), "abs_sum": float(mag[0])}
    p = _state_params(case, seed)
    e = np.exp(2 * p.r)
    logdet = float(np.sum(np.log((p.eta * e + 2 - p.eta) / 2) + np.log((p.eta / e + 2 - p.eta) / 2)))
    if kind == "build":
        return {"V": _covariance(p), "logdet": logdet}
    modes = gi.random_modes(case["M"], case["N"], seed)
    inv = np.linalg.inv(_covariance(p) + 0.5 * np.eye(2 * case["M"]))
    # per mode (a, a^+), the layout of sigma_inv_block
    rows = np.stack([modes, modes + case["M"]], 1).reshape(-1)
    return {"block": inv[np.ix_(rows, rows)], "logdet": logdet}
