// The split of a general potential's monomial program (host): which entries of
// each level need double precision.
//
// The size of an entry is its root mean square over the bridge: its monomial of
// the potential's derivatives averaged over the bridge's times and positions, its
// power of vs^2 from a step's second moment.  The smallest entries whose sum
// stays below 2^-33 of the level's weight go to single precision (their error
// there is a few 2^-24); of every node the double part takes the leading powers
// up to the last large one, and with it the node's ancestors.  (These are typical
// sizes; what a path has is summed by the kernel, and limited there.)
//
// The choice depends on the estimator alone, not on how many samples a call has,
// so that a run's parts have the run's weights.  It takes 0.02 ms (p = 4) to 0.2 ms
// (p = 12, eight levels) of the host.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "sampler.h"

namespace su {

namespace {

constexpr int kTimes = 8, kPts = 16;   // 7 times, 16 positions to 6 standard deviations
constexpr double kStep = 12.0 / kPts;
constexpr int kOctaves = 400;

// Root mean squares over the bridge of the program's monomials (ms) and of the
// derivatives (ds), the positions of successive times shifted against each other.
void moments(const GeneralEffective &G, const GeneralPotential &V, double a, double b, double T, std::vector<double> &ms,
             std::vector<double> &ds) {
    const size_t nn = G.depth.size();
    const int J = G.J;
    ms.assign(nn, 0.0);
    ds.assign((size_t)J + 1, 0.0);
    using Row = double[kPts];
    std::vector<double> buf((size_t)(2 * J + 3 + G.J + 3 * G.p + 2) * kPts);
    Row *D = reinterpret_cast<Row *>(buf.data()), *t = D + J + 1, *stk = t + J + 2;
    for (int k = 1; k < kTimes; ++k) {
        const double u = (double)k / kTimes, mean = a + (b - a) * u, sd = std::sqrt(T * u * (1 - u));
        Row x, wgt;
        for (int i = 0; i < kPts; ++i) {
            const double g = kStep * (i - 0.5 * (kPts - 1) + (k - 0.5 * kTimes) / kTimes);
            x[i] = mean + sd * g;
            wgt[i] = std::exp(-0.5 * g * g) * (kStep / std::sqrt(2 * 3.14159265358979323846)) / (kTimes - 1);
        }
        for (int j = 0; j <= J; ++j)
            for (int i = 0; i < kPts; ++i) D[j][i] = 0.0;
        double der[9];
        std::copy(V.a, V.a + 9, der);
        for (int j = 0; j <= std::min(J, 8); ++j) {   // der: the coefficients of the j-th derivative
            for (int q = 8 - j; q >= 0; --q)
                for (int i = 0; i < kPts; ++i) D[j][i] = D[j][i] * x[i] + der[q];
            for (int q = 0; q < 8 - j; ++q) der[q] = der[q + 1] * (q + 1);
            der[8 - j] = 0.0;
        }
        for (int f = 0; f < V.ng; ++f) {
            // (d/dx)^n A e^{-beta u^2}: D_{n+1} = -2 beta (u D_n + n D_{n-1})
            const double A = V.gauss[f][0], beta = V.gauss[f][1], c = V.gauss[f][2];
            Row y, d0, d1;
            for (int i = 0; i < kPts; ++i) {
                const double v = x[i] - c;
                y[i] = -2.0 * beta * v;
                d0[i] = 0.0;
                d1[i] = A * std::exp(-beta * v * v);
            }
            for (int n = 0; n <= J; ++n)
                for (int i = 0; i < kPts; ++i) {
                    D[n][i] += d1[i];
                    const double d2 = y[i] * d1[i] - 2.0 * beta * n * d0[i];
                    d0[i] = d1[i];
                    d1[i] = d2;
                }
        }
        for (int f = 0; f < V.ns; ++f) {
            // Taylor coefficients of tanh, (n+1) t_{n+1} = -sum_k t_k t_{n-k}; sech^2 = tanh'
            const double alpha = V.sech[f][1], d = V.sech[f][2];
            for (int i = 0; i < kPts; ++i) {
                const double w = alpha * (x[i] - d), ch = std::cosh(w);
                t[0][i] = std::tanh(w);
                t[1][i] = 1.0 / (ch * ch);
            }
            double sc = V.sech[f][0];   // B alpha^n (n+1)!
            for (int n = 0; n <= J; ++n) {
                if (n) {
                    Row acc = {};
                    for (int q = 0; q < (n + 1) / 2; ++q)
                        for (int i = 0; i < kPts; ++i) acc[i] += t[q][i] * t[n - q][i];
                    const double even = n & 1 ? 0.0 : 1.0;
                    for (int i = 0; i < kPts; ++i)
                        t[n + 1][i] = (2.0 * acc[i] + even * (t[n / 2][i] * t[n / 2][i])) * (-1.0 / (n + 1));
                }
                sc *= (double)(n + 1);
                for (int i = 0; i < kPts; ++i) D[n][i] += sc * t[n + 1][i];
                sc *= alpha;
            }
        }
        for (int f = 0; f < V.ne; ++f) {
            Row e;
            for (int i = 0; i < kPts; ++i) e[i] = V.expo[f][0] * std::exp(-V.expo[f][1] * (x[i] - V.expo[f][2]));
            for (int n = 0; n <= J; ++n)
                for (int i = 0; i < kPts; ++i) {
                    D[n][i] += e[i];
                    e[i] *= -V.expo[f][1];
                }
        }
        for (int j = 0; j <= J; ++j)
            for (int i = 0; i < kPts; ++i) ds[(size_t)j] += wgt[i] * (D[j][i] * D[j][i]);
        for (int i = 0; i < kPts; ++i) {
            stk[0][i] = 1.0;
            ms[0] += wgt[i];
        }
        for (size_t q = 1; q < nn; ++q) {
            const double *up = stk[G.depth[q] - 1], *s = D[G.sym[q]];
            double *mu = stk[G.depth[q]], sum[4] = {};
            for (int i = 0; i < kPts; i += 4)
                for (int r = 0; r < 4; ++r) {
                    const double m = up[i + r] * s[i + r];
                    mu[i + r] = m;
                    sum[r] += wgt[i + r] * (m * m);
                }
            ms[q] += (sum[0] + sum[1]) + (sum[2] + sum[3]);
        }
    }
    for (double &v : ms) v = std::sqrt(v);
    for (double &v : ds) v = std::sqrt(v);
}

}  // namespace

bool general_split(const GeneralEffective &G, const GeneralPotential &V, double a, double b, double T, int S, int levels,
                   const double *tables, GeneralSplit &gs, GeneralImages &im) {
    const size_t nn = G.depth.size(), M = G.entry_k.size();
    // the potential's parameters as floats, far enough inside their range
    bool floats = true;
    auto param = [&](double v) { floats = floats && (v == 0.0 || (std::fabs(v) >= 0x1p-100 && std::fabs(v) <= 0x1p100)); };
    for (double v : V.a) param(v);
    for (int f = 0; f < V.ng; ++f) param(V.gauss[f][0]), param(V.gauss[f][1]);
    for (int f = 0; f < V.ns; ++f) param(V.sech[f][0]), param(V.sech[f][1]);
    for (int f = 0; f < V.ne; ++f) param(V.expo[f][0]), param(V.expo[f][1]);
    if (!floats) return false;
    // sizes in units in which the path is about one across (lengths 2^unit, energies
    // 4^-unit), so that their squares are doubles: deg = the power of 2^-unit of a monomial
    const int unit = std::ilogb(std::sqrt(T));
    GeneralPotential U = V;
    for (int i = 0; i <= 8; ++i) U.a[i] = std::ldexp(U.a[i], unit * (i + 2));
    for (int f = 0; f < V.ng; ++f) {
        U.gauss[f][0] = std::ldexp(U.gauss[f][0], 2 * unit);
        U.gauss[f][1] = std::ldexp(U.gauss[f][1], 2 * unit);
        U.gauss[f][2] = std::ldexp(U.gauss[f][2], -unit);
    }
    for (auto fam : {U.sech, U.expo})
        for (int f = 0; f < (fam == U.sech ? V.ns : V.ne); ++f) {
            fam[f][0] = std::ldexp(fam[f][0], 2 * unit);
            fam[f][1] = std::ldexp(fam[f][1], unit);
            fam[f][2] = std::ldexp(fam[f][2], -unit);
        }
    std::vector<int> deg(nn, 0), sdeg((size_t)G.J + 3 * G.p + 2, 0);
    for (size_t t = 1; t < nn; ++t) deg[t] = sdeg[(size_t)G.depth[t]] = sdeg[(size_t)G.depth[t] - 1] + G.sym[t] + 2;
    std::vector<double> ms, ds, fact(nn, 1.0), fs((size_t)G.J + 1, 1.0), stk((size_t)G.J + 3 * G.p + 2, 1.0);
    moments(G, U, std::ldexp(a, -unit), std::ldexp(b, -unit), std::ldexp(T, -2 * unit), ms, ds);
    for (int j = 2; j <= G.J; ++j) fs[(size_t)j] = fs[(size_t)j - 1] * j;
    for (size_t t = 1; t < nn; ++t) {
        fact[t] = stk[(size_t)G.depth[t] - 1] * fs[(size_t)G.sym[t]];
        stk[(size_t)G.depth[t]] = fact[t];
    }
    // the kernel's monomials (of derivatives over j!), and the smallest and largest
    // factor or partial product on the way to each, in typical size
    const bool near = std::abs(unit) * (2 * G.K + *std::max_element(deg.begin(), deg.end())) < 500;   // no power of the unit overflows
    std::vector<double> mono(nn, 1.0), mu(nn, 1.0), lo(nn, 1.0), hi(nn, 1.0), slo(stk.size(), 1.0), shi(stk.size(), 1.0);
    for (size_t t = 1; t < nn; ++t) {
        const size_t at = (size_t)G.depth[t];
        const double u = std::ldexp(ds[(size_t)G.sym[t]] / fs[(size_t)G.sym[t]], -unit * (G.sym[t] + 2));
        mono[t] = std::ldexp(ms[t], -unit * deg[t]);
        mu[t] = mono[t] / fact[t];
        lo[t] = slo[at] = std::min(slo[at - 1], std::min(u, mu[t]));
        hi[t] = shi[at] = std::max(shi[at - 1], std::max(u, mu[t]));
    }
    im.tail.assign((size_t)S * M, 0.0f);
    std::vector<double> size(M), my((size_t)G.K, 1.0), yk(my);
    std::vector<int> head(nn), bin(M);
    std::vector<size_t> path((size_t)kGenMaxDepth + 1, 0);
    std::vector<char> keep(nn), single(M);
    bool any = false;
    for (int d = 0; d < levels; ++d) {
        const double *table = tables + (size_t)d * M;
        const double N = std::ldexp(1.0, S - d), step = std::ldexp(b - a, -unit) / N;
        const double s2 = std::ldexp(T, -2 * unit) / N + step * step;
        for (int k = 1; k < G.K; ++k) my[(size_t)k] = my[(size_t)k - 1] * s2 * std::sqrt((4.0 * k - 1) * (4.0 * k - 3));
        for (int k = 0; k < G.K; ++k) yk[(size_t)k] = std::ldexp(my[(size_t)k], 2 * unit * k);
        double all = 0;
        for (size_t t = 0; t < nn; ++t)
            for (int k = 0; k < G.count[t]; ++k) {
                const size_t e = (size_t)G.first[t] + (size_t)k;
                const double v = std::fabs(table[e]);
                size[e] = near ? v * mono[t] * yk[(size_t)k] : std::ldexp(v, unit * (2 * k - deg[t])) * ms[t] * my[(size_t)k];
                all += size[e];
            }
        if (!std::isfinite(all)) continue;   // sizes beyond a double: nothing to split by
        // the smallest entries up to the sum: whole octaves (powers of two, down to
        // 2^-300), then sixty-fourths of the next one
        const double most = 0x1p-33 * std::min(1.0, N * all) / N;
        double sum[kOctaves] = {}, part[64] = {};
        for (size_t e = 0; e < M; ++e) {
            int64_t bits;
            std::memcpy(&bits, &size[e], 8);
            bin[e] = std::max(0, std::min(64 * kOctaves - 1, (int)(bits >> 46) - 64 * (1023 - 300)));
            sum[bin[e] / 64] += size[e];
        }
        double rest = 0;
        int oct = 0, sub = 0;
        while (oct < kOctaves && rest + sum[oct] <= most) rest += sum[oct++];
        for (size_t e = 0; e < M; ++e)
            if (bin[e] / 64 == oct) part[bin[e] % 64] += size[e];
        while (sub < 64 && rest + part[sub] <= most) rest += part[sub++];
        const int first = 64 * oct + sub;   // of the large ones
        // Entries whose factors or partial products a float's range does not hold (units
        // in which the potential's derivatives or the step are far from one) are large ones
        // too, or are left out where they do not count: what falls below 2^-126 is lost, in
        // all as much as a float's rounding of the others may be.
        const double none = 0x1p-24 * most / (double)M;
        double lost = 0;
        auto in_floats = [&](size_t t, int k, size_t e) {
            const double c = std::fabs(table[e]) * fact[t], cy = c * yk[(size_t)k];
            if (!(std::max(c, std::max(cy, hi[t])) <= 0x1p100)) return false;
            if (std::min(lo[t], std::min(c, cy)) >= 0x1p-102) return true;   // a float's rounding of the entry at most
            const double less = std::min(size[e], 0x1p-126 * std::max(mu[t] * std::max(1.0, yk[(size_t)k]), mu[t] / lo[t] * cy));
            if (!(lost + less <= 0x1p-24 * most)) return false;
            lost += less;
            return true;
        };
        int total = 0;
        for (size_t t = 0; t < nn; ++t) {
            head[t] = 0;
            for (int k = 0; k < G.count[t]; ++k) {
                const size_t e = (size_t)G.first[t] + (size_t)k;
                single[e] = bin[e] < first && in_floats(t, k, e);
                if (!single[e] && (bin[e] >= first || size[e] > none)) head[t] = k + 1;
            }
            total += head[t];
        }
        // worth it where the double part is short: at 51 % of 1629 entries the level takes
        // a fifth less than as a whole, between 52 and 60 % of 341 more
        const bool fits = total > 0 && 25 * total <= 13 * (int)M;
        if (!fits) continue;
        for (size_t t = 0; t < nn; ++t)
            for (int k = head[t]; k < G.count[t]; ++k) {
                const size_t e = (size_t)G.first[t] + (size_t)k;
                if (single[e]) im.tail[(size_t)d * M + e] = (float)(table[e] * fact[t]);
            }
        // the nodes with entries and their ancestors, in order
        std::fill(keep.begin(), keep.end(), 0);
        for (size_t t = 0; t < nn; ++t) {
            path[(size_t)G.depth[t]] = t;
            if (head[t])
                for (int q = 0; q <= G.depth[t]; ++q) keep[path[(size_t)q]] = 1;
        }
        gs.h0[d] = (int)im.hnodes.size();
        gs.hc[d] = (int)im.hcoef.size();
        for (size_t t = 0; t < nn; ++t) {
            if (!keep[t] && t) continue;
            im.hnodes.push_back({(unsigned char)G.depth[t], (unsigned char)G.sym[t], (unsigned short)head[t],
                                 (int)im.hcoef.size() - gs.hc[d]});
            for (int k = 0; k < head[t]; ++k) im.hcoef.push_back(table[(size_t)G.first[t] + (size_t)k]);
            if (t) gs.hj[d] = std::max(gs.hj[d], G.sym[t]);
        }
        gs.hn[d] = (int)im.hnodes.size() - gs.h0[d];
        any = true;
    }
    gs.on = any;
    gs.n_nodes = (int)nn;
    return any;
}

}  // namespace su
