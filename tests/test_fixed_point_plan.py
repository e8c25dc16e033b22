"""The fixed-point sampler's plan (csrc/fx_plan.cpp) on the host, at tables and
ranges whose scales are at or past a double's: it ends, and every level that it
takes has a scale that the kernel's conversions hold and a finite residue."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1105_0542_gb300", "csrc")
SRC = r"""
#include <cmath>
#include <cstdio>
#include <vector>
#include "sampler.h"
// ring a b T alpha S ncol len.. factor: the table of every level is factor 8^-k
int main() {
    using namespace su;
    static SamplerParams P{};
    double T, factor;
    if (std::scanf("%d %lf %lf %lf %lf %d %d", &P.ring, &P.a, &P.b, &T, &P.alpha, &P.S, &P.ncol) != 7) return 1;
    for (int j = 0; j < P.ncol; ++j) {
        if (std::scanf("%d", &P.len[j]) != 1) return 1;
        P.M += P.len[j];
    }
    if (std::scanf("%lf", &factor) != 1) return 1;
    P.levels = P.S;
    P.F = P.S < 4 ? P.S : 4;
    std::vector<double> t((size_t)P.S * P.M);
    for (size_t k = 0; k < t.size(); ++k) t[k] = std::ldexp(factor, -3 * (int)(k % P.M));
    std::vector<int64_t> head;
    std::vector<float> tail;
    fx_plan(P, T, t.data(), head, tail);
    std::printf("%d\n", P.fx.on);
    for (int d = 0; d < P.S; ++d) std::printf("%d %d %.17g\n", P.fx.lv[d].ok, P.fx.lv[d].e, P.fx.lv[d].res);
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("fxplan")
    (d / "plan.cpp").write_text(SRC)
    exe = str(d / "plan")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", "/usr/local/cuda/include", str(d / "plan.cpp"),
                    os.path.join(CSRC, "fx_plan.cpp"), "-o", exe], check=True)

    def run(ring, a, b, T, alpha, s, lens, factor):
        line = " ".join(str(v) for v in (ring, a, b, T, alpha, s, len(lens), *lens, factor))
        out = subprocess.run([exe], input=line, capture_output=True, text=True, timeout=60, check=True).stdout.split("\n")
        return int(out[0]), [(int(k), int(e), float(r)) for k, e, r in (x.split() for x in out[1:] if x)]

    return run


EVEN, TANH2 = 0, 2


@pytest.mark.parametrize("ring", [EVEN, TANH2])
@pytest.mark.parametrize("a,T,factor", [
    (0.3, 0.5, 0.0), (0.3, 0.5, 1e-60), (0.3, 0.5, 1e-200), (0.3, 0.5, 1e-295), (0.3, 0.5, 1e-305), (0.3, 0.5, 5e-324),
    (0.3, 0.5, 1e60), (0.3, 0.5, 1e280), (0.3, 0.5, 1e308), (1e40, 0.5, 1.0), (1e100, 0.5, 1.0), (1e154, 0.5, 1.0),
    (1e308, 0.5, 1.0), (0.0, 1e-320, 1.0), (0.0, 1e-200, 1.0), (0.0, 1e300, 1.0), (1e-200, 1e-200, 1e-200)])
def test_plan_ends_with_scales_that_a_double_holds(plan, ring, a, T, factor):
    on, levels = plan(ring, a, -a, T, 1.0, 10, (6, 4, 3, 1), factor)
    assert on == levels[0][0]
    for ok, e, res in levels:
        if ok:
            assert -900 <= e <= 900 and abs(res) < float("inf")


def test_plan_takes_ordinary_tables(plan):
    on, levels = plan(EVEN, 0.0, 0.5, 0.25, 1.0, 10, (6, 4, 3, 1), 1e-3)
    assert on and sum(ok for ok, _, _ in levels) >= 5


INDEX = r"""
#include <cmath>
#include <cstdio>
#include "fixed_point.cuh"
using namespace su;
// the node of tanh^2 for sums of two points, as the sampler finds it, from the plan's limbs
int main() {
    double step;
    long long us;
    while (std::scanf("%lf %lld", &step, &us) == 2) {
        const fx::Limbs l = fx::limbs((int64_t)std::nearbyint((long double)step * std::ldexp(1.0L, 64 + 53 - 63)));
        std::printf("%lld\n", (long long)(fx::mul(fx::magnitude((int64_t)us), l) >> 53));
    }
}
"""


def test_every_sum_of_two_points_has_a_node(tmp_path):
    """Sums that leave 64 bits wrap: also the most negative one finds a node
    of those in reach, 0..int(step)."""
    (tmp_path / "index.cpp").write_text(INDEX)
    exe = str(tmp_path / "index")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, str(tmp_path / "index.cpp"), "-o", exe], check=True)
    steps = (1e-12, 1e-7, 2.0 ** -22, 0.3, 1.0, 5.999999, 150.25, 383.999)
    sums = (-2 ** 63, -2 ** 63 + 1, -2 ** 62, -2 ** 32, -1, 0, 1, 2 ** 32 - 1, 2 ** 62, 2 ** 63 - 1)
    pairs = [(step, us) for step in steps for us in sums]
    out = subprocess.run([exe], input="\n".join(f"{a!r} {b}" for a, b in pairs), capture_output=True, text=True,
                         check=True).stdout.split()
    assert len(out) == len(pairs)
    for (step, us), k in zip(pairs, out):
        assert 0 <= int(k) <= int(step), (step, us)
