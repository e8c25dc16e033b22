// The split of a general potential's monomial program (host): which entries of
// each level need double precision.
//
// The size of an entry is its root mean square over the bridge: its monomial of
// the potential's derivatives averaged over the bridge's times and positions, its
// power of vs^2 from a step's second moment.  The smallest entries whose sum
// stays below 2^-33 of the level's weight go to single precision (their error
// there is a few 2^-24); of every node the double part takes the leading powers
// up to the last large one, and with it the node's ancestors.
#include <algorithm>
#include <cmath>

#include "sampler.h"

namespace su {

void general_moments(const GeneralEffective &G, const GeneralPotential &V, double a, double b, double T,
                     std::vector<double> &ms) {
    const size_t nn = G.depth.size();
    constexpr int times = 8, half = 8;   // 7 times, 17 positions to 6 standard deviations
    constexpr double dg = 6.0 / half;
    ms.assign(nn, 0.0);
    std::vector<double> D((size_t)G.J + 1), stk((size_t)G.J + 3 * G.p + 2, 1.0);
    for (int k = 1; k < times; ++k) {
        const double u = (double)k / times, mean = a + (b - a) * u, sd = std::sqrt(T * u * (1 - u));
        for (int g = -half; g <= half; ++g) {
            const double wgt = std::exp(-0.5 * g * g * dg * dg) * (dg / std::sqrt(2 * 3.14159265358979323846)) / (times - 1);
            general_derivatives(V, mean + sd * g * dg, G.J, D.data());
            for (size_t t = 0; t < nn; ++t) {
                double mu = 1.0;
                if (t) {
                    mu = stk[(size_t)G.depth[t] - 1] * D[(size_t)G.sym[t]];
                    stk[(size_t)G.depth[t]] = mu;
                }
                ms[t] += wgt * mu * mu;
            }
        }
    }
    for (double &v : ms) v = std::sqrt(v);
}

double general_split(const GeneralEffective &G, const std::vector<double> &ms, double a, double b, double T, int n,
                     const double *table, std::vector<int> &head) {
    const double N = std::ldexp(1.0, n), eps = T / N, s2 = eps + (b - a) * (b - a) / (N * N);
    std::vector<double> my((size_t)G.K, 1.0);
    for (int k = 1; k < G.K; ++k) my[(size_t)k] = my[(size_t)k - 1] * s2 * std::sqrt((4.0 * k - 1) * (4.0 * k - 3));
    const size_t nn = G.depth.size();
    std::vector<double> size(G.entry_k.size());
    double all = 0;
    for (size_t t = 0; t < nn; ++t)
        for (int k = 0; k < G.count[t]; ++k) {
            const size_t e = (size_t)G.first[t] + (size_t)k;
            all += size[e] = std::fabs(table[e]) * ms[t] * my[(size_t)k];
        }
    if (!std::isfinite(all)) {   // sizes beyond a double: nothing to split by
        head.assign(G.count.begin(), G.count.end());
        return 0;
    }
    // the smallest entries up to the sum: whole octaves, then the last one's in order
    const double most = 0x1p-33 * std::min(1.0, N * all) / N;
    constexpr int kOctaves = 400;
    auto octave = [](double v) { return v > 0 ? std::max(0, std::min(kOctaves - 1, std::ilogb(v) + 300)) : 0; };
    std::vector<double> sum(kOctaves, 0.0);
    for (double v : size) sum[(size_t)octave(v)] += v;
    double rest = 0;
    int oct = 0;
    while (oct < kOctaves && rest + sum[(size_t)oct] <= most) rest += sum[(size_t)oct++];
    std::vector<double> last;
    for (double v : size)
        if (octave(v) == oct) last.push_back(v);
    std::sort(last.begin(), last.end());
    double least = 0;   // of the large ones
    for (double v : last) {
        least = v;
        if (rest + v > most) break;
        rest += v;
    }
    head.assign(nn, 0);
    for (size_t t = 0; t < nn; ++t)
        for (int k = 0; k < G.count[t]; ++k) {
            const double v = size[(size_t)G.first[t] + (size_t)k];
            const int o = octave(v);
            if (o > oct || (o == oct && v >= least)) head[t] = k + 1;
        }
    return N * most;
}

}  // namespace su
