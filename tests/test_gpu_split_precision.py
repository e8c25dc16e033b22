"""The samplers that evaluate the small entries of W_p in single precision
against the whole program in double (kernel="generic"): the split does run,
is no further from extended precision than the whole program, and leaves the
paths beyond its reach to the whole program."""
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1105_0542_gb300 as su  # noqa: E402
from oracle import general_v as gv  # noqa: E402

pytestmark = pytest.mark.gpu
LD = np.longdouble
QUARTIC = dict(poly=(0.1, 0.0, 0.5, 0.0, 0.2))
NARROW = dict(poly=(0.1, 0.0, 0.5), gauss=[(0.3, 30.0, 0.1)])
MORSE = dict(poly=(4.0,), expo=[(-8.0, 1.0, 0.3), (4.0, 2.0, 0.3)])


def _general(V, a, b, T, p, s, n, sample0=0, seed=77, **kw):
    out = torch.zeros((n, s), dtype=torch.float64, device="cuda")
    par = su.general_params(V.get("poly", ()), V.get("gauss", ()), V.get("sech", ()), V.get("expo", ()))
    su.speedup_logweights("general", par, a, b, T, p, s, sample0, n, seed, out, precision="fp64", **kw)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _extended(f):
    hi = float(f)
    return LD(hi) + LD(float(Fraction(f) - Fraction(hi)))


def _paths(a, b, T, s, n, seed, d=1):
    """The samples' paths in extended precision from the library's normals."""
    N = 1 << s
    z = torch.zeros((n, (N - 1) * d), dtype=torch.float64, device="cuda")
    su.speedup_normals(seed, 0, 0, n, (N - 1) * d, z)
    torch.cuda.synchronize()
    z = z.cpu().numpy().astype(LD).reshape(n, N - 1, d)
    q = np.empty((n, N + 1, d), dtype=LD)
    q[:, 0], q[:, N] = np.asarray(a, dtype=LD), np.asarray(b, dtype=LD)
    for lev in range(1, s + 1):
        h, m = 1 << (s - lev), 1 << (lev - 1)
        q[:, h::2 * h] = (q[:, 0:-1:2 * h] + q[:, 2 * h::2 * h]) / 2 + np.sqrt(LD(T) / 2 ** (lev + 1)) * z[:, m - 1:2 * m - 1]
    return q


def _derivatives(V, x, J):
    out = np.zeros((J + 1,) + x.shape, dtype=LD)
    a = V["poly"]
    for j in range(min(J, len(a) - 1) + 1):
        for i in range(len(a) - 1, j - 1, -1):
            out[j] = out[j] * x + LD(a[i]) * np.prod([LD(i - r) for r in range(j)])
    for A, beta, c in V.get("gauss", ()):
        u = x - LD(c)
        d0, d1 = np.zeros_like(x), LD(A) * np.exp(-LD(beta) * u * u)
        for n in range(J + 1):
            out[n] += d1
            d0, d1 = d1, -2 * LD(beta) * (u * d1 + n * d0)
    return out


def _general_top(V, a, b, T, p, s, n, seed):
    """The top level's log-weights in extended precision."""
    q = _paths((a,), (b,), T, s, n, seed)[..., 0]
    x, xb2 = (q[:, 1:] + q[:, :-1]) / 2, ((q[:, 1:] - q[:, :-1]) / 2) ** 2
    eps = Fraction(T) / 2 ** s
    U = _derivatives(V, x, 2 * p - 2)
    tot = np.zeros_like(x)
    for (m, k), poly in gv.coefficients(p).items():
        for mono, c in poly.items():
            t = _extended(c * eps ** (m - k)) * xb2 ** k
            for j, e in enumerate(mono):
                for _ in range(e):
                    t = t * U[j]
            tot = tot + t
    return (-_extended(eps) * tot.sum(1)).astype(np.float64), tot


@pytest.mark.parametrize("V,p,s", [(QUARTIC, 5, 8), (NARROW, 6, 9)], ids=["quartic", "narrow"])
def test_general_split_is_no_further_off_than_the_whole_program(V, p, s):
    """Root mean square distance of the finest level's weights from extended
    precision.  The single-precision part is below 2^-33 of the weight, and its
    roundings a few 2^-24 of that: the distance is that of the sum over the
    slices, by segments in both programs.  Half as much again for the 200
    samples' own scatter (5 %) and the segments' different lengths."""
    a, b, T, n, seed = -0.4, 0.6, 0.2, 200, 77
    ref, _ = _general_top(V, a, b, T, p, s, n, seed)
    w = {k: _general(V, a, b, T, p, s, 20_000, seed=seed, kernel=k)[:n, -1] for k in ("auto", "generic")}
    assert np.any(w["auto"] != w["generic"])   # two programs
    rms = {k: np.sqrt(np.mean((v - ref) ** 2)) for k, v in w.items()}
    assert rms["auto"] <= 1.5 * rms["generic"]


@pytest.mark.parametrize("V,p,s,n", [(QUARTIC, 12, 1, 777), (QUARTIC, 4, 10, 130), (NARROW, 8, 9, 300), (MORSE, 10, 4, 1001)],
                         ids=["two-slices", "p4", "narrow", "exponentials"])
def test_general_split_matches_the_whole_program(V, p, s, n):
    """Two slices, the smallest program that splits, a feature narrower than
    the bridge, exponentials; a partial last item.  A few 2^-50 of a weight
    (the guard's 2^-30 in single precision, 2^-24 of it a few times over, and
    the sums of up to 1024 slices)."""
    w = {k: _general(V, -0.4, 0.6, 0.2, p, s, n, kernel=k) for k in ("auto", "generic")}
    assert np.any(w["auto"][:, -1] != w["generic"][:, -1])
    assert np.all(np.abs(w["auto"] - w["generic"]) <= 2.0 ** -48 * np.maximum(1.0, np.abs(w["generic"])))


# samples of seed 1234 whose first normal is -6.17, -6.43: q_{N/2} some 3 sqrt(T) from the endpoints
FAR = [492790794, 2573160571]


def test_general_path_beyond_the_split_is_weighed_by_the_whole_program():
    """The single-precision entries of such a path in the exponentials of a
    Morse potential pass 2^-30 of the weight (they are a hundred times their
    typical sum): the weight is the whole program's, bit for bit, while its
    neighbours' are the split's."""
    a, b, T, p, s, n = 0.0, 0.6, 0.2, 8, 6, 12_000
    for f in FAR:
        w = {k: _general(MORSE, a, b, T, p, s, n, sample0=f - 100, seed=1234, kernel=k) for k in ("auto", "generic")}
        same = w["auto"] == w["generic"]
        assert same[100, 2] and same[100, 3]
        assert not same[:, 3].all()
        assert np.all(np.abs(w["auto"] - w["generic"]) <= 2.0 ** -50 * np.maximum(1.0, np.abs(w["generic"])))


def test_general_split_far_from_the_origin():
    """Features about 1000: both programs take the offsets from the same
    points, so they differ by what they do near the origin -- the guard's
    2^-30 in single precision, a few 2^-24 of it, and the sums' own rounding."""
    V = dict(poly=(0.0,), gauss=[(1.5, 2.0, 1000.3)], sech=[(-1.0, 2.0, 1000.0)])
    w = {k: _general(V, 999.5, 1000.7, 0.25, 8, 7, 20_000, kernel=k) for k in ("auto", "generic")}
    assert np.any(w["auto"][:, -1] != w["generic"][:, -1])
    assert np.all(np.abs(w["auto"] - w["generic"]) <= 2.0 ** -50 * np.maximum(1.0, np.abs(w["generic"])))


@pytest.mark.parametrize("s,n", [(6, 12_000), (4, 3000)])
def test_general_weights_do_not_depend_on_the_sample_count(s, n):
    """A run in parts by sample0, and one sample of it, have the run's weights
    bit for bit; so has the top level without the others."""
    args = (MORSE, 0.0, 0.6, 0.2, 10, s)
    w = _general(*args, n, sample0=FAR[0] - 100, seed=1234)
    g = _general(*args, n, sample0=FAR[0] - 100, seed=1234, kernel="generic")
    assert np.any(w != g)   # the split ran
    for lo, hi in ((0, 90), (90, n // 2), (n // 2, n), (100, 101)):
        assert np.array_equal(_general(*args, hi - lo, sample0=FAR[0] - 100 + lo, seed=1234), w[lo:hi])
    par = su.general_params(MORSE["poly"], (), (), MORSE["expo"])
    run = [su.speedup_amplitude("general", par, 0.0, 0.6, 0.2, 10, s, n, 1234, sample0=FAR[0] - 100, n_blocks=8, hierarchy=h)
           for h in (True, False)]
    assert run[0][s]["amp"] == run[1][s]["amp"] and run[0][s]["err"] == run[1][s]["err"]


@pytest.mark.parametrize("V,p,e", [(QUARTIC, 7, -8), (QUARTIC, 5, -12), (NARROW, 7, 12), (MORSE, 10, -4), (MORSE, 10, 40)],
                         ids=["quartic-8", "quartic-12", "narrow+12", "morse-4", "morse+40"])
def test_general_split_in_other_units(V, p, e):
    """Lengths in units of 2^e (times of 4^e, energies of 4^-e): the weights
    are those of e = 0, whatever of the derivatives a float's range holds.
    What the split's guard lets through, and both programs' sums of 512 slices,
    are a few 2^-50 of a weight."""
    u = 2.0 ** e
    U = dict(poly=tuple(c * u ** -(i + 2) for i, c in enumerate(V["poly"])),
             gauss=[(A / u ** 2, beta / u ** 2, c * u) for A, beta, c in V.get("gauss", ())],
             expo=[(E / u ** 2, kappa / u, x * u) for E, kappa, x in V.get("expo", ())])
    n = {5: 6510, 7: 1825, 10: 500}[p]
    w = _general(U, -0.4 * u, 0.6 * u, 0.2 * u * u, p, 9, n)
    g = _general(V, -0.4, 0.6, 0.2, p, 9, n, kernel="generic")
    assert np.all(np.abs(w - g) <= 2.0 ** -48 * np.maximum(1.0, np.abs(g)))


AHO2 = {(2, 0): 0.5, (4, 0): 1 / 24, (2, 2): 1 / 12, (0, 2): 0.5, (0, 4): 1 / 24}
AHO3 = {(2, 0, 0): 0.5, (0, 2, 0): 0.5, (0, 0, 2): 0.5, (4, 0, 0): 1 / 24, (0, 4, 0): 1 / 24, (0, 0, 4): 1 / 24,
        (2, 2, 0): 1 / 12, (2, 0, 2): 1 / 12, (0, 2, 2): 1 / 12}
TWO = {(2, 0, 0, 0): 0.5, (0, 2, 0, 0): 0.5, (0, 0, 2, 0): 0.5, (0, 0, 0, 2): 0.5, (2, 0, 2, 0): 0.1, (1, 0, 1, 0): -0.2,
       (0, 1, 0, 1): -0.2, (0, 2, 0, 2): 0.1}
ENDS = {1: ((0.2,), (-0.4,)), 2: ((0.0, 0.0), (1.0, 0.5)), 3: ((0.0, 0.0, 0.0), (1.0, 0.5, -0.5)),
        4: ((0.3, 0.0, -0.3, 0.1), (0.2, 0.4, -0.1, -0.2))}


def _nd(V, T, p, s, n, sample0=0, seed=1234, u=1.0, **kw):
    out = torch.zeros((n, s), dtype=torch.float64, device="cuda")
    a, b = ENDS[len(next(iter(V)))]
    su.speedup_logweights_nd({m: c * u ** -(sum(m) + 2) for m, c in V.items()}, tuple(x * u for x in a),
                             tuple(x * u for x in b), T * u * u, p, s, sample0, n, seed, out, precision="fp64", **kw)
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("V,T,p,s", [({(3,): 0.1, (2,): 0.5}, 0.5, 9, 6), (AHO2, 1.0, 10, 7), (AHO3, 1.0, 8, 5), (TWO, 1.0, 6, 6)],
                         ids=["1", "2", "3", "4"])
def test_nd_split_matches_the_whole_program(V, T, p, s):
    """One to four coordinates at levels that split: a few 2^-50 of a weight
    between the two programs (the guard's 2^-27 in single precision, 2^-24 of
    it a few times over, and the sums)."""
    w = {k: _nd(V, T, p, s, 1111, kernel=k) for k in ("auto", "generic")}
    assert np.any(w["auto"][:, -1] != w["generic"][:, -1])
    assert np.all(np.abs(w["auto"] - w["generic"]) <= 2.0 ** -48 * np.maximum(1.0, np.abs(w["generic"])))


@pytest.mark.parametrize("p", [7, 10])
def test_nd_level_beyond_the_split_is_weighed_by_the_whole_program(p):
    """A sample of seed 1234 inside 2.4 sqrt(T) of the endpoints whose slices'
    single-precision parts pass 2^-27 on level 9 alone: its weight there is the
    whole program's, bit for bit, while the neighbours' are the split's."""
    at = 227961
    same = _nd(AHO2, 0.5, p, 9, 100, sample0=at - 50) == _nd(AHO2, 0.5, p, 9, 100, sample0=at - 50, kernel="generic")
    assert same[50, 8] and not same[:, 8].all() and not same[50].all()


@pytest.mark.parametrize("V,p,e", [(AHO2, 8, 12), (AHO2, 8, 24), (AHO3, 8, 12), (TWO, 6, 18), (TWO, 6, 36), (AHO2, 8, -12), (TWO, 6, -40)])
def test_nd_split_in_other_units(V, p, e):
    """Lengths in units of 2^e: the weights are those of e = 0, whatever of the
    table's entries a float's range holds."""
    w = _nd(V, 0.5, p, 6, 1000, u=2.0 ** e)
    g = _nd(V, 0.5, p, 6, 1000, kernel="generic")
    assert np.all(np.abs(w - g) <= 2.0 ** -48 * np.maximum(1.0, np.abs(g)))
