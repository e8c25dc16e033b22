"""What su_autotune stores belongs to the kernel that a plan runs: a shape timed
on another kernel does not take the split of a general potential or the
fixed-point sampler away, nor lend them its rounds."""
import pytest

torch = pytest.importorskip("torch")

import paper_1105_0542_gb300 as su  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _clear():
    su.su_autotune_clear()
    yield
    su.su_autotune_clear()


def _weights(model, params, a, b, T, p, s, n=500):
    out = torch.zeros((n, s), dtype=torch.float64, device="cuda")
    su.speedup_logweights(model, params, a, b, T, p, s, 0, n, 3, out, precision="fp64")
    torch.cuda.synchronize()
    return out.cpu().numpy()


def test_general_autotune_times_the_split():
    """Twenty explicit shapes run the whole program; the automatic one splits,
    and is the fastest of all (2.5 times on these levels)."""
    par = su.general_params((0.0, 0.0, 0.5), [(1.5, 2.0, 0.3)], [(-1.0, 2.0, 0.0)])
    args = ("general", par, -0.5, 0.7, 0.25, 10, 6)
    before = _weights(*args)
    best, all_ = su.su_autotune(*args, 20_000, 3, n_blocks=20)
    assert len(all_) == 24
    assert best["ms"] == min(t["ms"] for t in all_[:4]) < min(t["ms"] for t in all_[4:])
    pl = su.Plan(*args, 20_000, 3, n_blocks=20)
    assert pl.su_plan_shape() == (best["seg_log2"], best["rounds"])
    assert (_weights(*args) == before).all()


@pytest.mark.parametrize("p,s", [(1, 10), (2, 6), (4, 8), (7, 5), (12, 8), (12, 10)])
def test_a_shape_stored_for_the_double_sampler_leaves_the_fixed_point_sampler_on(p, s):
    """At T = 60 no plan in fixed point exists; its tuning is the double
    sampler's and does not reach the calls at T = 1/4."""
    args = ("aho", [1.0, 10.0], 0.0, 1.0)
    before = _weights(*args, 0.25, p, s)
    out = torch.zeros((500, s), dtype=torch.float64, device="cuda")
    su.speedup_logweights(*args, 0.25, p, s, 0, 500, 3, out, precision="fp64", kernel="generic")
    torch.cuda.synchronize()
    assert (out.cpu().numpy() != before).any()   # the fixed-point sampler runs
    best, _ = su.su_autotune(*args, 60.0, p, s, 50_000, 3, precision="fp64", n_blocks=20)
    assert (_weights(*args, 0.25, p, s) == before).all()
    pl = su.Plan(*args, 0.25, p, s, 50_000, 3, precision="fp64", n_blocks=20)
    assert pl.su_plan_shape() == (min(s, 4), 1)
    own, _ = su.su_autotune(*args, 0.25, p, s, 50_000, 3, precision="fp64", n_blocks=20)
    pl = su.Plan(*args, 0.25, p, s, 50_000, 3, precision="fp64", n_blocks=20)
    assert pl.su_plan_shape() == (own["seg_log2"], own["rounds"])
