"""The calls whose speed is followed: what a user of this library runs, through its public entry points.

A case is one call of one kind:

  amplitude  speedup_amplitude: every level of one bisection run of one instance (host in, host out)
  nd         speedup_amplitude_nd: the same for a system of several coordinates
  batch      speedup_amplitude_batch: an amplitude matrix on an endpoint grid, (T, s) per instance
  proposal   speedup_amplitude_proposal: paths drawn through the learned proposal's network
  train      speedup_train_proposal: plain paths, then Adam steps of the proposal's network
  spectrum   speedup_evolution_spectrum: band of the evolution operator and its lowest energies

Sizes are those of workloads.py, of the benchmark and of the tests, with sample counts that do not divide
evenly into blocks, work items or waves.
"""
from __future__ import annotations

import math
from fractions import Fraction
from functools import lru_cache

import numpy as np
import torch

import paper_1105_0542_gb300 as su

FIELDS = ("amp", "log_amp", "err", "rel_err", "err_naive", "ess", "max_share")


# ------------------------------------------------------------------ potentials of several coordinates

def _radial(d):
    """(x.x)/2 + (x.x)^2/24, the anharmonic oscillator of the paper's Sec. 3.3 in d coordinates."""
    V = {}
    for i in range(d):
        e = [0] * d
        e[i] = 2
        V[tuple(e)] = 0.5
        e[i] = 4
        V[tuple(e)] = 1 / 24
        for j in range(i + 1, d):
            e = [0] * d
            e[i] = e[j] = 2
            V[tuple(e)] = 1 / 12
    return V


SYSTEMS = {
    "aho2": (_radial(2), (0.0, 0.0), (1.0, 0.5)),
    "aho3": (_radial(3), (0.0, 0.0, 0.0), (1.0, 0.5, -0.5)),
    # two coupled particles in the plane
    "two": ({(2, 0, 0, 0): 0.5, (0, 2, 0, 0): 0.5, (0, 0, 2, 0): 0.5, (0, 0, 0, 2): 0.5, (2, 0, 2, 0): 0.1,
             (1, 0, 1, 0): -0.2, (0, 1, 0, 1): -0.2, (0, 2, 0, 2): 0.1},
            (0.3, 0.0, -0.3, 0.1), (0.2, 0.4, -0.1, -0.2)),
}

# the general potential: a trap with a Gaussian bump and a sech^2 dip
MIXED = dict(poly=(0.0, 0.0, 0.5), gauss=[(1.5, 2.0, 0.3)], sech=[(-1.0, 2.0, 0.0)])

# monomials of W_p: of the collapsed tables by formula, of the programs as generated
ND_TERMS = {("aho2", 4): 28, ("aho2", 5): 41, ("aho2", 6): 56, ("aho2", 7): 75, ("aho2", 8): 100, ("aho2", 9): 130,
            ("aho2", 10): 165, ("aho3", 4): 68, ("aho3", 5): 110, ("aho3", 6): 168, ("aho3", 7): 252,
            ("aho3", 8): 375, ("two", 3): 31, ("two", 4): 55, ("two", 5): 87, ("two", 6): 131}
GENERAL_TERMS = {4: 15, 5: 30, 6: 58, 7: 105, 8: 193, 9: 338, 10: 585, 11: 985, 12: 1629}


def _terms(case):
    p, kind, model = case["p"], case["kind"], case["model"]
    if kind == "nd":
        return ND_TERMS[(model, p)]
    if model == "general":
        return GENERAL_TERMS[p]
    if model == "mpt":
        return p * (p + 1)
    if model == "ho":
        return 2 * p
    return sum(max(0, 2 + math.ceil((p - 3 * j) / 2)) for j in range(p))


# ------------------------------------------------------------------ the cases

def _amplitude(name, model, g, a, b, T, p, s, n_mc, n_blocks, precision):
    c = dict(kind="amplitude", model=model, g=g, a=a, b=b, T=T, p=p, s=s, n_mc=n_mc, n_blocks=n_blocks,
             precision=precision)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest call: one short-time-action estimate of a few slices, as a user tries the library or scans
        # endpoints one at a time; latency of plan, launches and the copy back
        _amplitude("one_p4_s4", "aho", 1.0, 0.0, 1.0, 1.0, 4, 4, 100_000, 10, "fp64"),
        # a point of the convergence sweep at its middle level, double precision: the main use of the library
        _amplitude("sweep_p10_s10", "aho", 10.0, 0.0, 1.0, 1.0, 10, 10, 400_003, 100, "fp64"),
        # the sweep's highest compiled level in single precision
        _amplitude("sweep_p18_s10_f32", "aho", 10.0, 0.0, 1.0, 1.0, 18, 10, 3_000_001, 100, "fp32"),
        # the Poeschl-Teller convergence run of the paper's Fig. 2, double precision
        _amplitude("poschl_p10_s10", "mpt", 1.0, -0.5, 0.5, 1.0, 10, 10, 200_003, 100, "fp64"),
        # the double well, tunnelling from well to well, many samples in single precision
        _amplitude("well_p12_s6_f32", "dw", 1.0, -1.0, 1.0, 1.0, 12, 6, 20_000_000, 64, "fp32"),
        # a potential without a table: W_p from the derivatives of V at every slice
        _amplitude("general_p10_s6", "general", 1.0, -0.5, 0.7, 0.25, 10, 6, 200_001, 64, "fp64"),
        # the amplitude matrix for diagonalising the evolution operator, uneven instances in one launch
        dict(name="matrix_48_f32", kind="batch", model="aho", g=1.0, side=48, p=10, n_mc=100_000, n_blocks=16,
             s_lo=4, s_hi=8, precision="fp32"),
        # two coordinates, double precision, deep bisection
        dict(name="aho2_p10_s10", kind="nd", model="aho2", p=10, s=10, T=1.0, n_mc=100_003, n_blocks=64,
             precision="fp64"),
        # three coordinates, single precision
        dict(name="aho3_p8_s8_f32", kind="nd", model="aho3", p=8, s=8, T=1.0, n_mc=300_001, n_blocks=64,
             precision="fp32"),
        # inference of the learned proposal where the bridge is a poor one
        dict(name="proposal_s6", kind="proposal", model="ho", g=2.0, a=0.0, b=0.5, T=2.0, p=4, s=6, n_mc=1_000_003,
             n_blocks=50),
        # training of its network: plain paths, minibatches, forward, backward, Adam
        dict(name="train_512x200", kind="train", model="ho", g=2.0, a=0.0, b=0.5, T=2.0, p=4, s=6, n_train=200_000,
             steps=200, batch=512),
        # the energies of Fig. 3's anharmonic oscillator on its grid
        dict(name="spectrum_16385", kind="spectrum", model="aho", g=48.0, p=21, t=0.02, L=8.0, n=16385, nev=10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["amplitude"] * 5 + ["nd", "nd", "batch", "proposal", "train", "spectrum"])
    if kind == "amplitude":
        model = rng.choice(["aho", "aho", "aho", "dw", "mpt", "general"])
        precision = "fp64" if model == "general" else rng.choice(["fp64", "fp32"])
        T = 0.25 if model == "general" else rng.choice([0.25, 0.5, 1.0])
        g, a, b = {"aho": (rng.uniform(0.5, 10.0), 0.0, rng.uniform(0.2, 1.2)), "dw": (1.0, -1.0, 1.0),
                   "mpt": (rng.uniform(0.8, 1.5), -0.5, rng.uniform(0.2, 0.8)),
                   "general": (1.0, -0.5, 0.7)}[model]
        s = rng.randint(2, 8 if model == "general" else 10)
        p = rng.randint(4, 11) if model == "general" else rng.randint(1, 18) if model == "aho" else rng.randint(1, 12)
        # a budget of slice actions by what one of them costs on each path
        cost = {"general": 8e8, "fp64": 2e9, "fp32": 4e10}["general" if model == "general" else precision]
        cost /= max(1.0, (p * (p + 1) if model == "mpt" else GENERAL_TERMS.get(p, 1) if model == "general" else
                          2 * p) / (60.0 if model == "mpt" else 20.0))
        most = max(20_000, min(20_000_000, int(0.3 * cost / (2 << s))))
        return _amplitude("", model, g, a, b, T, p, s, _log_int(rng, 10_000, most) | 1, rng.choice([10, 64, 100]),
                          precision)
    if kind == "nd":
        model = rng.choice(list(SYSTEMS))
        precision = rng.choice(["fp64", "fp32"])
        p = rng.randint(4, {"aho2": 10, "aho3": 8, "two": 6}[model])
        s = rng.randint(3, 9)
        most = int((3e10 if precision == "fp64" else 2e11) / ND_TERMS[(model, p)] / (2 << s))
        return dict(kind="nd", model=model, p=p, s=s, T=rng.choice([0.5, 1.0]), precision=precision,
                    n_mc=_log_int(rng, 5_000, max(10_000, min(2_000_000, most))) | 1, n_blocks=rng.choice([16, 64]))
    if kind == "batch":
        lo = rng.randint(4, 5)
        precision = rng.choice(["fp32", "fp32", "fp64"])
        return dict(kind="batch", model="aho", g=rng.uniform(0.5, 2.0), s_lo=lo, s_hi=rng.randint(lo + 1, 8),
                    side=rng.randint(5, 15 if precision == "fp64" else 47), p=rng.randint(4, 12),
                    n_mc=_log_int(rng, 5_000, 20_000 if precision == "fp64" else 100_000) | 1,
                    n_blocks=rng.choice([8, 16]), precision=precision)
    if kind == "proposal":
        return dict(kind="proposal", model="ho", g=rng.uniform(1.0, 2.0), a=0.0, b=rng.uniform(0.2, 0.8),
                    T=rng.uniform(1.0, 2.0), p=4, s=rng.randint(3, 6),
                    n_mc=_log_int(rng, 50_000, 1_000_000) | 1, n_blocks=50)
    if kind == "train":
        return dict(kind="train", model="ho", g=rng.uniform(1.0, 2.0), a=0.0, b=0.5, T=rng.uniform(1.0, 2.0), p=4, s=6,
                    n_train=_log_int(rng, 50_000, 200_000), steps=rng.randint(50, 200), batch=32 * rng.randint(4, 16))
    return dict(kind="spectrum", model="aho", g=rng.uniform(4.0, 48.0), p=rng.randint(8, 21), t=0.02, L=8.0,
                n=2 * _log_int(rng, 1000, 7000) + 1, nev=rng.randint(2, 10))


def _params(case, g=None):
    g = case["g"] if g is None else g
    model = case["model"]
    if model == "general":
        return su.general_params(**MIXED)
    return {"aho": (1.0, g), "dw": (g,), "mpt": (g, 1.0), "ho": (g,)}[model]


def _network(seed, scale=0.05):
    """A network whose proposal leans off the bridge a little: hidden layers U(+-1/sqrt(fan-in)), a small output
    layer."""
    rng = np.random.default_rng(seed)
    theta = []
    for o, i in ((128, 6), (128, 128), (128, 128)):
        bound = 1.0 / math.sqrt(i)
        theta += [rng.uniform(-bound, bound, o * i), rng.uniform(-bound, bound, o)]
    theta += [rng.normal(0.0, scale / math.sqrt(128), 2 * 128), np.zeros(2)]
    return np.concatenate(theta).astype(np.float32)


def _instances(case, seed):
    """The grid's (a, b, T, s), every depth and time equally often, in an order of the seed's."""
    grid = np.linspace(-3.0, 3.0, case["side"])
    rng = np.random.default_rng(seed)
    n = case["side"] ** 2
    depth = case["s_lo"] + np.arange(n) % (case["s_hi"] - case["s_lo"] + 1)
    times = np.array([0.25, 0.5, 1.0, 2.0])[(np.arange(n) // 7) % 4]
    order = rng.permutation(n)
    return [(float(grid[k // case["side"]]), float(grid[k % case["side"]]), float(times[order[k]]),
             int(depth[order[k]])) for k in range(n)]


def prepare(case, seed):
    st = dict(case=case, seed=int(seed))
    if case["kind"] == "batch":
        st["instances"] = _instances(case, seed)
    elif case["kind"] == "proposal":
        st["proposal"] = su.Proposal(_network(seed))
    elif case["kind"] == "train":
        # an untrained proposal is the bridge: a zero output layer
        st["theta"] = _network(seed, 0.0)
    elif case["kind"] == "spectrum":
        st["g"] = case["g"] * (1.0 + 1e-3 * (seed % 1000))
    return st


def _kind_of(case):
    return np.float32 if case.get("precision", "fp32") == "fp32" else np.float64


def _levels(case, levels):
    """One array per result, over the levels; single-precision paths give single-precision results."""
    return {f: np.array([r[f] for r in levels], dtype=_kind_of(case)) for f in FIELDS}


def run(st):
    case, seed = st["case"], st["seed"]
    kind = case["kind"]
    if kind == "amplitude":
        return _levels(case, su.speedup_amplitude(case["model"], _params(case), case["a"], case["b"], case["T"],
                                                  case["p"], case["s"], case["n_mc"], seed,
                                                  precision=case["precision"], n_blocks=case["n_blocks"]))
    if kind == "nd":
        V, a, b = SYSTEMS[case["model"]]
        return _levels(case, su.speedup_amplitude_nd(V, a, b, case["T"], case["p"], case["s"], case["n_mc"], seed,
                                                     precision=case["precision"], n_blocks=case["n_blocks"]))
    if kind == "batch":
        return _levels(case, su.speedup_amplitude_batch(case["model"], _params(case), case["p"], st["instances"],
                                                        case["n_mc"], seed, precision=case["precision"],
                                                        n_blocks=case["n_blocks"]))
    if kind == "proposal":
        return _levels(case, su.speedup_amplitude_proposal(case["model"], _params(case), case["a"], case["b"],
                                                           case["T"], case["p"], case["s"], case["n_mc"], seed,
                                                           st["proposal"], n_blocks=case["n_blocks"]))
    if kind == "train":
        theta, losses = su.speedup_train_proposal(case["model"], _params(case), case["a"], case["b"], case["T"],
                                                  case["p"], case["s"], seed, st["theta"], n_train=case["n_train"],
                                                  steps=case["steps"], batch_paths=case["batch"], lr=1e-3)
        return {"theta": theta, "losses": losses.astype(np.float32)}
    # the residual norms that come with the energies are rounding noise (1e-13): they tell that the solver converged
    E, R, info = su.speedup_evolution_spectrum(case["model"], _params(case, st["g"]), case["p"], case["t"], case["L"],
                                               case["n"], case["nev"])
    return {"energies": np.array(E), "converged": int(info["converged"])}


def work(case):
    """Operations of the estimator: 2 per table or program entry and 8 more per slice action (every level's slices:
    2^(s+1) - 2 per sample); 33 792 multiply-adds of the network per midpoint, three times that in training; of the
    spectrum 30 products of the band with a block of 16 vectors.  Bytes: the results, the training paths, the band."""
    kind = case["kind"]
    if kind in ("amplitude", "nd"):
        return {"flops": float(case["n_mc"]) * ((2 << case["s"]) - 2) * (2 * _terms(case) + 8),
                "bytes": 56.0 * (case["s"] + 1)}
    if kind == "batch":
        n = case["side"] ** 2
        depths = range(case["s_lo"], case["s_hi"] + 1)
        mean = sum(2.0 ** s for s in depths) / len(depths)
        return {"flops": n * float(case["n_mc"]) * mean * (2 * _terms(case) + 8), "bytes": 88.0 * n}
    mids = (1 << case["s"]) - 1 if "s" in case else 0
    if kind == "proposal":
        return {"flops": float(case["n_mc"]) * mids * 2 * 33792, "bytes": 4.0 * 34178 + 56 * (case["s"] + 1)}
    if kind == "train":
        return {"flops": 6.0 * 33792 * case["steps"] * case["batch"] * mids,
                "bytes": 8.0 * 34178 + 4.0 * case["n_train"] * (mids + 2)}
    w = math.sqrt(80.0 * case["t"]) / (2 * case["L"] / (case["n"] - 1))
    return {"flops": 30 * 2.0 * 16 * case["n"] * (2 * w + 1), "bytes": 8.0 * case["n"] * (w + 1)}


# ------------------------------------------------------------------ the same in 64 bits

def _add(acc, poly, f=1):
    for m, v in poly.items():
        v = acc.get(m, 0) + f * v
        if v:
            acc[m] = v
        else:
            acc.pop(m, None)


def _mul(a, b):
    out = {}
    for m, v in a.items():
        _add(out, {tuple(x + y for x, y in zip(m, n)): v * w for n, w in b.items()})
    return out


class _Ring:
    """Polynomials in z_1..z_d as {exponents: coefficient} with the derivative along each coordinate: z = x, or (one
    coordinate) z = tanh(x), where d/dx z^i = i (z^(i-1) - z^(i+1))."""

    def __init__(self, d, tanh=False):
        self.d, self.tanh = d, tanh

    def der(self, poly, i):
        out = {}
        for m, v in poly.items():
            if m[i]:
                for step, f in ((-1, 1), (1, -1)) if self.tanh else ((-1, 1),):
                    e = list(m)
                    e[i] += step
                    _add(out, {tuple(e): f * m[i] * v})
        return out


def _shift(poly, d, i):
    """xb_i times a polynomial of (z, xb)."""
    return {m[:d + i] + (m[d + i] + 1,) + m[d + i + 1:]: v for m, v in poly.items()}


class _Full(_Ring):
    """The same over (z_1..z_d, xb_1..xb_d): der(., i) for i >= d is d/dxb."""

    def der(self, poly, i):
        if i < self.d:
            return super().der(poly, i)
        out = {}
        for m, v in poly.items():
            if m[i]:
                e = list(m)
                e[i] -= 1
                _add(out, {tuple(e): m[i] * v})
        return out


@lru_cache(maxsize=64)
def _w(vkey, d, tanh, p):
    """W_{m,k} (m < p) from the paper's recursion: 8 (m+k+1) W_mk = lap W_{m-1,k} + lapb W_{m,k+1} - sums of gradient
    products; W_mm = (xb.grad)^(2m) V / (2m+1)!."""
    R = _Full(d, tanh)
    V = {tuple(e) + (0,) * d: Fraction(c) for e, c in vkey if c}
    W, G, H = {}, {}, {}
    grad = lambda f: [R.der(f, i) for i in range(d)]                # noqa: E731
    gradb = lambda f: [R.der(f, d + i) for i in range(d)]           # noqa: E731

    def keep(m, k, f):
        W[m, k], G[m, k], H[m, k] = f, grad(f), gradb(f)

    diag = V
    for m in range(p):
        if m:
            for _ in range(2):
                nxt = {}
                for i in range(d):
                    _add(nxt, _shift(R.der(diag, i), d, i))
                diag = nxt
        keep(m, m, {e: v / math.factorial(2 * m + 1) for e, v in diag.items()})
        for k in range(m - 1, -1, -1):
            acc = {}
            for i in range(d):
                _add(acc, R.der(H[m, k + 1][i], d + i))
                if (m - 1, k) in G:
                    _add(acc, R.der(G[m - 1, k][i], i))
            for l in range(0, m - 1):
                for r in range(max(0, k - m + l + 2), min(k, l) + 1):
                    for i in range(d):
                        _add(acc, _mul(G[l, r][i], G[m - l - 2, k - r][i]), -1)
                        if l:
                            _add(acc, _mul(H[l, r][i], H[m - l - 1, k - r + 1][i]), -1)
            keep(m, k, {e: v / (8 * (m + k + 1)) for e, v in acc.items()})
    return W


def _collapsed(vkey, d, tanh, p, eps):
    out = {}
    for (m, k), poly in _w(vkey, d, tanh, p).items():
        _add(out, poly, Fraction(eps) ** (m - k))
    return {e: float(v) for e, v in out.items() if v}


def _potential(case):
    """(the potential as ((exponents, coefficient), ...), its coordinates, whether in tanh)."""
    g = case.get("g")
    if case["kind"] == "nd":
        V = SYSTEMS[case["model"]][0]
        return tuple(sorted(V.items())), len(next(iter(V))), False
    f = Fraction(g)
    V = {"aho": {(2,): Fraction(1, 2), (4,): f / 24}, "dw": {(0,): f, (2,): -2 * f, (4,): f}, "ho": {(2,): f * f / 2},
         "mpt": {(0,): -f, (2,): f}}[case["model"]]
    return tuple(sorted(V.items())), 1, case["model"] == "mpt"


def _philox(call, sample, seed):
    """Philox4x32-10 words for the counters (call, 0, sample lo, sample hi) as four int64 tensors."""
    M = 0xFFFFFFFF
    c0, c1 = torch.broadcast_tensors(call[None, :], sample[:, None])
    c0, c2 = c0.clone(), c1 & M
    c3, c1 = c1 >> 32, torch.zeros_like(c0)
    k0, k1 = seed & M, (seed >> 32) & M
    for _ in range(10):
        a, b = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((b >> 32) & M) ^ c1 ^ k0, b & M, ((a >> 32) & M) ^ c3 ^ k1, a & M
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c0, c1, c2, c3


def _pair(u1, u2):
    R = torch.sqrt(-2.0 * torch.log(u1))
    return R * torch.cos(2 * math.pi * u2), R * torch.sin(2 * math.pi * u2)


def _normals(lo, hi, count, seed, precision, dev):
    """The first `count` normals of the samples lo..hi-1, from 53-bit uniforms, or from 24-bit ones."""
    smp = torch.arange(lo, hi, device=dev, dtype=torch.int64)
    if precision == "fp64":
        w = _philox(torch.arange((count + 1) // 2, device=dev, dtype=torch.int64), smp, seed)
        u = [((x << 21) | (y >> 11)).double().add_(0.5).mul_(2.0 ** -53) for x, y in ((w[0], w[1]), (w[2], w[3]))]
        return torch.stack(_pair(*u), dim=2).reshape(hi - lo, -1)[:, :count]
    w = _philox(torch.arange(count // 4 + 1, device=dev, dtype=torch.int64), smp, seed)
    # (k + 1/2) 2^-24 as the single-precision number it is
    u = [((x >> 8).double() + 0.5).float().double() * 2.0 ** -24 for x in w]
    z = torch.stack(_pair(u[0], u[1]) + _pair(u[2], u[3]), dim=2).reshape(hi - lo, -1)
    return z[:, 1:count + 1]


def _log_weights(tables, d, tanh, q, s):
    """w_n = -eps_n sum_k W on the level-n subpath of the paths q (samples, 2^s + 1, d)."""
    cols = []
    for n in range(1, s + 1):
        eps, tab = tables[n]
        sub = q[:, ::1 << (s - n)]
        x, xb = 0.5 * (sub[:, 1:] + sub[:, :-1]), 0.5 * (sub[:, 1:] - sub[:, :-1])
        z = [torch.tanh(x[..., i]) if tanh else x[..., i] for i in range(d)] + [xb[..., i] for i in range(d)]
        cols.append(-eps * _evaluate(tab, z, 0).sum(1))
    return torch.stack(cols, 1)


def _evaluate(tab, z, i):
    """The polynomial {exponents: coefficient} at z, Horner in z_i, recursively."""
    if i == len(z):
        return tab.get((), 0.0)
    by = {}
    for m, v in tab.items():
        by.setdefault(m[0], {})[m[1:]] = v
    acc, at = None, 0
    for e in sorted(by, reverse=True):
        v = _evaluate(by[e], z, i + 1)
        if acc is None:
            acc = v
        else:
            for _ in range(at - e):
                acc = acc * z[i]
            acc = acc + v
        at = e
    for _ in range(at):
        acc = acc * z[i]
    return acc


def _estimate(w, w0, laf, n_blocks):
    """The results of every level from the per-sample log-weights (n, s)."""
    n, nb = w.shape[0], n_blocks
    rows = [dict(amp=math.exp(laf + w0), log_amp=laf + w0, err=0.0, rel_err=0.0, err_naive=0.0, ess=float(n),
                 max_share=1.0 / n)]
    for lev in range(w.shape[1]):
        x = w[:, lev]
        top = float(x.max())
        e = torch.exp(x - top)
        S, Q = float(e.sum()), float((e * e).sum())
        mean = S / n
        mu = np.array([float(e[b * n // nb:(b + 1) * n // nb].mean()) for b in range(nb)])
        err = float(mu.std(ddof=1)) / math.sqrt(nb)
        scale = math.exp(laf + top)
        rows.append(dict(amp=scale * mean, log_amp=laf + top + math.log(mean), err=scale * err, rel_err=err / mean,
                         err_naive=scale * math.sqrt(max(Q / n - mean * mean, 0.0) / (n - 1)), ess=S * S / Q,
                         max_share=1.0 / S))
    return rows


def _gelu(v):
    return 0.5 * v * (1.0 + torch.erf(v / math.sqrt(2.0)))


def _leaning_path(case, theta, q, z, s, T):
    """Fills the paths q through the proposal's network; the log density ratios of levels 1..s."""
    dev, n = q.device, q.shape[0]
    layers, at = [], 0
    for o, i in ((128, 6), (128, 128), (128, 128), (2, 128)):
        Wt = torch.tensor(theta[at:at + o * i], dtype=torch.float64, device=dev).reshape(o, i)
        at += o * i
        layers.append((Wt, torch.tensor(theta[at:at + o], dtype=torch.float64, device=dev)))
        at += o
    ratio, out = torch.zeros(n, dtype=torch.float64, device=dev), []
    for lev in range(1, s + 1):
        h, m = 1 << (s - lev), 1 << (lev - 1)
        ql, qr = q[:, 0:-1:2 * h, 0], q[:, 2 * h::2 * h, 0]
        f = torch.empty(n, m, 6, dtype=torch.float64, device=dev)
        for c, v in enumerate((case["a"], case["b"], T, lev / s, ql, qr)):
            f[..., c] = v
        for k, (Wt, bias) in enumerate(layers):
            f = torch.nn.functional.linear(f, Wt, bias)
            f = _gelu(f) if k < 3 else f
        zl = z[:, m - 1:2 * m - 1]
        t = f[..., 0] + torch.exp(f[..., 1]) * zl
        q[:, h::2 * h, 0] = 0.5 * (ql + qr) + math.sqrt(T / 2 ** (lev + 1)) * t
        ratio = ratio + (0.5 * zl * zl - 0.5 * t * t + f[..., 1]).sum(1)
        out.append(ratio)
    return torch.stack(out, 1)


def _exact_paths(case, seed):
    nd = case["kind"] == "nd"
    vkey, d, tanh = _potential(case)
    a, b = SYSTEMS[case["model"]][1:] if nd else ((case["a"],), (case["b"],))
    T, p, s, n = case["T"], case["p"], case["s"], case["n_mc"]
    precision = case.get("precision", "fp32")
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    tables = {k: (T / 2 ** k, _collapsed(vkey, d, tanh, p, Fraction(T) / 2 ** k)) for k in range(s + 1)}
    theta = _network(seed) if case["kind"] == "proposal" else None
    N, w = 1 << s, []
    chunk = max(1, (1 << 25 if theta is None else 1 << 21) // (N * d))
    for lo in range(0, n, chunk):
        hi = min(n, lo + chunk)
        z = _normals(lo, hi, (N - 1) * d, seed, precision, dev)
        q = torch.empty(hi - lo, N + 1, d, dtype=torch.float64, device=dev)
        q[:, 0], q[:, N] = torch.tensor(a, dtype=q.dtype, device=dev), torch.tensor(b, dtype=q.dtype, device=dev)
        ratio = 0.0
        if theta is not None:
            ratio = _leaning_path(case, theta, q, z, s, T)
        else:
            z = z.reshape(hi - lo, N - 1, d)
            for lev in range(1, s + 1):
                h, m = 1 << (s - lev), 1 << (lev - 1)
                mid = 0.5 * (q[:, 0:-1:2 * h] + q[:, 2 * h::2 * h])
                q[:, h::2 * h] = mid + math.sqrt(T / 2 ** (lev + 1)) * z[:, m - 1:2 * m - 1]
        w.append(_log_weights(tables, d, tanh, q, s) + ratio)
    ends = torch.tensor([a, b], dtype=torch.float64).reshape(1, 2, d)
    x, xb = 0.5 * (ends[:, 1] + ends[:, 0]), 0.5 * (ends[:, 1] - ends[:, 0])
    zs = [torch.tanh(x[:, i]) if tanh else x[:, i] for i in range(d)] + [xb[:, i] for i in range(d)]
    w0 = -T * float(_evaluate(tables[0][1], zs, 0))
    laf = sum(-0.5 * math.log(2 * math.pi * T) - (v - u) ** 2 / (2 * T) for u, v in zip(a, b))
    return {f: np.array([r[f] for r in _estimate(torch.cat(w), w0, laf, case["n_blocks"])]) for f in FIELDS}


def exact(case, seed):
    """Sampled cases: the same Philox stream, paths, W and estimator in torch, double precision throughout.  The
    spectrum: the Hamiltonian in 300 of 400 harmonic-oscillator states."""
    kind = case["kind"]
    if kind == "spectrum":
        g = case["g"] * (1.0 + 1e-3 * (seed % 1000))
        m, omega = 400, 3.0
        q = np.diag(np.sqrt(np.arange(1, m) / (2 * omega)), 1)
        q = q + q.T
        q2 = q @ q
        kin = np.diag(omega * (np.arange(m) + 0.5)) - 0.5 * omega ** 2 * q2
        Hm = (kin + 0.5 * q2 + g / 24 * (q2 @ q2))[:300, :300]
        return {"energies": np.linalg.eigvalsh(Hm)[:case["nev"]], "converged": None}
    if kind in ("batch", "train") or case["model"] == "general":
        return None
    normals = case["n_mc"] * (1 << case["s"])
    if kind == "nd" and normals * _terms(case) > 5e10:
        return None
    if normals * (16 if kind == "proposal" else 1) > 1.5e9:
        return None
    return _exact_paths(case, seed)
