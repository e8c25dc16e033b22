"""The double-precision sampler in fixed point against the oracle and against
the double sampler (kernel="generic") on the same samples, at the edges of its
plan: one slice pair to N = 1024, segments shorter and as long as the register
segment, table shapes that are compiled in and not, odd sample counts, levels
that stay in double, and paths that leave the planned range of q.

Tolerances: per-sample weights as in test_gpu_parity (1e-12 of the weight, or
Horner's bound of the absolute terms); estimates 1e-13, far above the rounding
of sums of a few hundred weights that each carry a few 1e-16."""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_1105_0542_gb300 as su  # noqa: E402
from oracle import mc  # noqa: E402
from tests.test_gpu_parity import U64, _excess, _gpu_w  # noqa: E402

pytestmark = pytest.mark.gpu
THREADS = os.cpu_count() or 1

# samples of seed 1234 whose first normal is -6.17, -6.43, 6.22: q_{N/2} beyond Q = 2.9 sqrt(T) + max(|a|, |b|)
FAR = [492790794, 2573160571, 2383927765]

CASES = [("ho", [1.0], 0.0, 1.0, 1.0, 4, s, 129, s0) for s, s0 in ((1, 0), (2, 0), (3, FAR[0]), (4, FAR[1] - 7))]
CASES += [("aho", [1.0, 1.0], -0.3, 0.4, 0.5, p, s, 257, s0)
          for p, s, s0 in ((1, 5, 0), (4, 1, FAR[1] - 100), (7, 6, 0), (10, 4, FAR[2] - 128), (18, 10, FAR[0] - 3),
                           (21, 7, FAR[1] - 255))]
CASES += [("mpt", [1.5, 1.2], -0.4, 0.6, 0.5, p, s, 130, s0) for p, s, s0 in ((1, 3, 0), (4, 6, FAR[0] - 64), (10, 9, 0), (12, 5, FAR[2]))]
CASES += [("dw", [1.0], -1.0, 1.0, 1.0, 12, 8, 100, 0), ("poly", [0.1, 0.0, 0.5, 0.0, 0.1, 0.0, 0.02], 0.2, 0.0, 0.3, 5, 7, 64, 0)]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}-p{c[5]}-s{c[6]}-at{c[8]}" for c in CASES])
def test_fixed_point_weights_match_oracle_and_double_sampler(case):
    model, params, a, b, T, p, s, n, s0 = case
    wg = _gpu_w(model, params, a, b, T, p, s, n, 1234, s0, precision="fp64")
    wd = _gpu_w(model, params, a, b, T, p, s, n, 1234, s0, precision="fp64", kernel="generic")
    o = mc.Oracle(model, params, p)
    wo, _ = o.logweights(a, b, T, s, 1234, n, sample0=s0, bits=53, threads=THREADS)
    wabs = o.logweights_abs(a, b, T, s, 1234, n, sample0=s0, bits=53)
    assert _excess(wg, wo, wabs, 1e-12, U64) <= 1.0
    assert _excess(wg, wd, wabs, 1e-12, U64) <= 1.0
    if s >= 7:
        assert np.any(wg != wd)   # two samplers, not one


@pytest.mark.parametrize("kw", [dict(), dict(hierarchy=False), dict(rounds=3), dict(n_blocks=7), dict(sample0=FAR[0] - 500)],
                         ids=["default", "top", "rounds", "blocks", "far"])
@pytest.mark.parametrize("s,p", [(1, 4), (4, 4), (6, 9), (9, 20)])
def test_fixed_point_estimates_match_double_sampler(s, p, kw):
    args = ("aho", [1.0, 2.0], 0.1, 0.6, 0.5, p, s, 1333, 1234)
    r = su.speedup_amplitude(*args, precision="fp64", **kw)
    g = su.speedup_amplitude(*args, precision="fp64", kernel="generic", **kw)
    for x, y in zip(r, g):
        if x["level"] in ((0, s) if kw.get("hierarchy") is False else range(s + 1)):
            assert x["n"] == y["n"]
            assert x["amp"] == pytest.approx(y["amp"], rel=1e-13)
            assert x["err"] == pytest.approx(y["err"], rel=1e-10, abs=1e-300)
