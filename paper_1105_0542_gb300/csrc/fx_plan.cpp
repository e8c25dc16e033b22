// Ranges and scales of the fixed-point sampler (host).
//
// Units.  Path points are q 2^62 / Q with Q = max(|a|, |b|) + 2.9 sqrt(T): a
// bridge leaves [-Q, Q] with probability below 2 exp(-2 2.9^2) = 1e-7 per
// path, and such a path is taken again in double.  The ring variable is
// z = (us / 2Q)^2 in [0, 1), and the second one y = (vs / V)^2 with
// V = 2Q 2^-ky just above 5.6 to 6.6 sqrt(eps) plus the mean step (probability
// below 5e-8 that one of the level's steps is larger).
//
// With the level's entries C_ij = T_ij (2Q)^(2i) V^(2j), |sum| bounds of every
// partial Horner sum follow, and from them
//   E      such that the cut-off of the last products, half a unit of 2^-E per
//          slice, stays below 2^-55 of the level's weight (a double's own
//          rounding is 2^-53 of it);
//   heads  the leading entries of each column that are too large for single
//          precision.  The others sum to at most 2^25 / sqrt(N) units (root mean
//          square over the bridge): what rounding an entry to float costs adds
//          up over the N slices, to at most sqrt(N)/2 units.
// A level whose integer sums would not fit 64 bits at that E is evaluated in
// double (the coarsest levels of high p, where eps is large).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "fixed_point.cuh"
#include "sampler.h"

namespace su {

// the largest integer of a chain, with room for the products' constants
static constexpr double kFxMax = 0x1.8p62;
// ranges for which every scale below is a normal double: path points at most
// 1e100 and at least 1e-100 across, weights in units of 2^-900 to 2^900 (the
// conversion of the sums puts the unit into a double's exponent)
static constexpr double kFxLeast = 1e-100;
static constexpr int kFxUnits = 900;

void fx_plan(SamplerParams &P, double T, const double *tables, std::vector<int64_t> &head, std::vector<float> &tail) {
    FxParams &X = P.fx;
    std::memset(&X, 0, sizeof X);
    head.clear();
    tail.clear();
    const int S = P.S, M = P.M;
    if (S < 1 || P.wf_on || P.generic || P.tab_global || (P.ring != RING_EVEN && P.ring != RING_TANH2) || P.F != std::min(S, 4)) return;
    // Q of eight bits: its powers in the entries' scales are exact
    int qe;
    const double qm = std::frexp(std::max(std::fabs(P.a), std::fabs(P.b)) + 2.9 * std::sqrt(T), &qe);
    const double Q = std::ldexp(std::ceil(qm * 256), qe - 8);
    if (!(Q >= kFxLeast && Q <= 1 / kFxLeast)) return;
    const bool th = P.ring == RING_TANH2;
    X.q_unit = std::ldexp(Q, -62);
    if (th) {
        // alpha x = alpha us / 2 in units of 2^-53 node steps, cut by 2^64
        const long double step = std::fabs((long double)P.alpha) * Q * fx::kTanhSteps;
        if (!(step < fx::kTanhNodes)) return;
        const fx::Limbs l = fx::limbs((int64_t)std::nearbyint(step * std::ldexp(1.0L, 64 + 53 - 63)));
        X.ah = l.h;
        X.al = l.l;
        X.nodes = (int)step + 1;
    }
    X.qlim = (1 << 30) - (1 << 20);
    X.qa = (int64_t)std::nearbyint((long double)P.a / X.q_unit);
    X.qb = (int64_t)std::nearbyint((long double)P.b / X.q_unit);
    for (int n = 1; n <= S; ++n) {
        // product of a normal (units 2^-kZScale) with sg, cut by 2^64 and shifted left by shl
        long double sg = std::sqrt((long double)T / std::ldexp(1.0L, n + 1)) / X.q_unit * std::ldexp(1.0L, 64 - fx::kZScale);
        while (sg >= 0x1p62L) {
            sg *= 0.5L;
            ++X.shl[n];
        }
        const fx::Limbs l = fx::limbs((int64_t)std::nearbyint(sg));
        X.sgh[n] = l.h;
        X.sgl[n] = l.l;
    }
    int len_max = 1;
    for (int j = 0; j < P.ncol; ++j) len_max = std::max(len_max, P.len[j]);
    std::vector<std::vector<int64_t>> rows((size_t)S);
    tail.assign((size_t)S * M, 0.0f);
    const double qs = 4.0 * Q * Q, zs = th ? 1.0 : qs;   // scales of vs^2 and z
    // root mean squares of z^i, averaged over the times of the bridge
    std::vector<double> mz((size_t)len_max, 0.0);
    for (int k = 1; k < 16; ++k) {
        const double u = k / 16.0, mean = P.a + (P.b - P.a) * u, sd = std::sqrt(T * u * (1 - u));
        for (int g = -24; g <= 24; ++g) {
            const double x = mean + sd * g * 0.25;
            const double t = th ? std::tanh(P.alpha * x) : x / Q, z = std::min(1.0, t * t);
            double wgt = std::exp(-0.5 * g * g * 0.0625) * (0.25 / std::sqrt(2 * 3.14159265358979323846)) / 15;
            for (int i = 0; i < len_max; ++i, wgt *= z * z) mz[i] += wgt;
        }
    }
    for (double &v : mz) v = std::sqrt(v);
    std::vector<double> C((size_t)M);
    std::vector<int> col((size_t)M), row((size_t)M);
    for (int j = 0, at = 0; j < P.ncol; ++j)
        for (int i = 0; i < P.len[j]; ++i, ++at) {
            col[at] = j;
            row[at] = i;
        }
    for (int d = 0; d < P.levels; ++d) {
        const int n = S - d;
        const double *t = tables + (size_t)d * M;
        const double eps = T / std::ldexp(1.0, n), step = std::fabs(P.b - P.a) / std::ldexp(1.0, n);
        // N steps beyond reach standard deviations: probability N e^(-reach^2 / 2) / reach < 5e-8
        const double reach = std::sqrt(29.6 + 2 * n * 0.69314718055994531);
        FxLevel &L = X.lv[d];
        L.ky = std::max(0, std::min(24, (int)std::floor(std::log2(2.0 * Q / (reach * std::sqrt(eps) + step)))));
        L.vlim = (int)std::min((int64_t)0x7fffffff, (((int64_t)1 << 31) >> L.ky) - 1);
        const double ys = qs * std::ldexp(1.0, -2 * L.ky);
        // root mean squares of y^j: a step's second moment and the Gaussian factor (4j - 1)!!
        const double yt = (eps + step * step) / ys;
        std::vector<double> my((size_t)P.ncol, 1.0);
        for (int j = 1; j < P.ncol; ++j)
            my[j] = std::min(1.0, my[j - 1] * yt * std::sqrt((4.0 * j - 1) * (4.0 * j - 3)));
        double typ = 0, most = 0;
        bool finite = true;
        for (int k = 0; k < M; ++k) {
            C[k] = t[k];
            for (int i = 0; i < row[k]; ++i) C[k] *= zs;
            for (int j = 0; j < col[k]; ++j) C[k] *= ys;
            typ += std::fabs(C[k]) * mz[row[k]] * my[col[k]];
            most = std::max(most, std::fabs(C[k]));
            finite = finite && std::isfinite(C[k]);
        }
        if (!finite || !std::isfinite(typ)) continue;
        const double N = std::ldexp(1.0, n);
        const double ns = (d <= P.F && n > 0) ? std::min(4.0, std::ldexp(1.0, P.F - d)) : 1.0;   // slices per 64-bit sum
        const double tol = 0x1p-55 * std::min(1.0, N * typ);
        // W_p = 0 on the whole path: any scale will do
        const double units = tol > 0 ? std::ceil(std::log2(0.5 * std::sqrt(N) / tol)) : most > 0 ? kFxUnits + 1 : 60;
        if (!(std::fabs(units) <= kFxUnits)) continue;
        const int E = (int)units;
        const double scale = std::ldexp(1.0, E);
        // entries beyond each column's heads, root mean square
        auto rest = [&](const int *h, int j) {
            double s = 0;
            for (int k = 0; k < M; ++k)
                if (col[k] == j && row[k] >= (j < kFxCols ? h[j] : 0))
                    s += std::fabs(C[k]) * mz[row[k]] * my[j];
            return s * scale;
        };
        // grow the heads of the column with the largest rest until it fits
        int h[kFxCols] = {1};
        bool fits = true;
        for (;;) {
            double sum = 0, top = -1;
            int at = -1;
            for (int j = 0; j < P.ncol; ++j) {
                const double x = rest(h, j);
                sum += x;
                if (x > top) {
                    top = x;
                    at = j;
                }
            }
            if (sum <= 0x1p25 / std::sqrt(N)) break;
            fits = at < kFxCols;
            if (!fits) break;
            ++h[at];
        }
        int nc = 1;
        for (int j = 1; j < kFxCols; ++j)
            if (h[j]) nc = j + 1;
        for (int j = 0; j < nc; ++j) h[j] = std::max(h[j], 1);
        double all = 0;
        for (int k = 0; k < M; ++k) all += std::fabs(C[k]) * scale;
        fits = fits && all * ns < kFxMax;
        for (int j = 0; j < nc; ++j)
            for (int i = 0; i < h[j]; ++i) {
                // the chain of column j from entry i up, with the columns above it where the chain ends
                double s = 0;
                for (int k = 0; k < M; ++k)
                    if ((col[k] == j && row[k] >= i && row[k] < h[j]) || (i == 0 && col[k] > j && col[k] < nc && row[k] < h[col[k]]))
                        s += std::fabs(C[k]) * scale;
                fits = fits && std::ldexp(s, i + j) < kFxMax;
            }
        if (!fits) continue;
        L.ok = 1;
        L.nc = nc;
        L.e = E;
        // Entry i of column j in units of 2^-E / 2^(i + j): a product with z or y (below 2^63) halves.  Stored in the order of use: last column first, top entry first.  Every entry
        // that a product is added to takes the product's constant.
        for (int j = nc - 1; j >= 0; --j) {
            L.h[j] = h[j];
            const int off = (int)(std::find(col.begin(), col.end(), j) - col.begin());
            for (int i = h[j] - 1; i >= 0; --i) {
                int64_t v = i < P.len[j] ? (int64_t)std::nearbyint(std::ldexp(C[off + i] * scale, i + j)) : 0;
                if (i == 0 && j == 0) L.res = (C[off] * scale - (double)v) / scale;
                if (i < h[j] - 1) v -= fx::kBias;
                if (i == 0 && j < nc - 1) v -= fx::kBias;
                rows[d].push_back(v);
            }
        }
        for (int k = 0; k < M; ++k)
            if (col[k] >= nc || row[k] >= h[col[k]]) tail[(size_t)d * M + k] = (float)(C[k] * scale);
    }
    for (const auto &v : rows) X.hrow = std::max(X.hrow, (int)v.size());
    head.assign((size_t)S * X.hrow, 0);
    for (int d = 0; d < S; ++d) std::copy(rows[d].begin(), rows[d].end(), head.begin() + (size_t)d * X.hrow);
    // levels in double have at most as many slices in all as the finest one
    X.on = X.lv[0].ok;
}

}  // namespace su
