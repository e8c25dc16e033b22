"""speedup_amplitude_noalloc at the edge of its scratch: the fixed-point
sampler's images do not cost a call that the double sampler has room for."""
import math

import pytest

torch = pytest.importorskip("torch")

import paper_1105_0542_gb300 as su  # noqa: E402

pytestmark = pytest.mark.gpu


def _up(n):
    return (n + 255) // 256 * 256


def test_the_largest_call_of_the_double_sampler_is_accepted():
    """Tables, tuples of each 128 samples and each block, and the flag word
    fill the 8 MB: one item more is refused whatever the sampler."""
    p, s = 18, 10
    terms = sum(max(0, 2 + math.ceil((p - 3 * j) / 2)) for j in range(p))
    items = 0
    while _up(8 * s * terms) + _up(32 * s * (items + 1)) + _up(32 * s) + 256 <= 8 << 20:
        items += 1
    args = ("aho", [1.0, 10.0], 0.0, 1.0, 1.0, p, s)
    kw = dict(precision="fp64", n_blocks=1, rounds=1)
    for kernel in ("generic", "auto"):
        with pytest.raises(su.SpeedupError) as e:
            su.speedup_amplitude_noalloc(*args, 128 * items + 1, 5, kernel=kernel, **kw)
        assert e.value.code == -6
    g = su.speedup_amplitude_noalloc(*args, 128 * items, 5, kernel="generic", **kw)
    r = su.speedup_amplitude_noalloc(*args, 128 * items, 5, **kw)
    for lev in range(s + 1):
        assert r[lev]["n"] == 128 * items
        assert r[lev]["amp"] == pytest.approx(g[lev]["amp"], rel=1e-13)
