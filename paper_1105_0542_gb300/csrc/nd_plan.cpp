// The evaluation program of a several-coordinates plan and, for double
// precision, its split into a double and a single-precision part (host).
//
// Program.  W is evaluated by nested Horner: the 2d variables in a fixed order
// z_0..z_{2d-1}, a polynomial in z_k whose coefficients are polynomials in
// z_{k+1}, and so on.  One word per polynomial, depth first, highest power
// first: its number of coefficients (zero: the zero polynomial) and whether it
// has a factor z_k; where the powers of a depth keep their parity inside every
// polynomial (W of an even potential) the Horner variable of that depth is
// z_k^2.  The innermost coefficients are the table's entries in program order.
// Every variable sits at a known depth of a nest of loops, so its registers are
// named in the code: no entry is looked up by symbol and no partial product is
// stored.
//
// Split (double).  Entries whose root mean square over the bridge is small are
// left to single precision: what rounding them to floats costs, 2^-25 of their
// sum, adds up over the N slices to 2^-55 of the level's typical weight.  The
// others form a program of their own, evaluated in double.  These are typical
// sizes: what a path's slices have is summed by the kernel, and a level on which
// that passes 2^-27 of max(1, |w|) is weighed by the whole program in double.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "sampler.h"

namespace su {

namespace {

using Mono = std::vector<unsigned char>;

struct Item {
    const unsigned char *e;   // exponents in program order
    int entry;
};

// items[lo, hi) sorted by exponents, highest first, equal before depth k
void emit(const std::vector<Item> &it, size_t lo, size_t hi, int k, int nv, unsigned sq, NdProgram &G) {
    if (lo == hi) {
        G.words.push_back(0);
        return;
    }
    const int top = it[lo].e[k];
    const int step = (sq >> k) & 1 ? 2 : 1, e0 = step == 2 ? top & 1 : 0;
    G.words.push_back((uint32_t)((top - e0) / step + 1) | (e0 ? kNdOdd : 0u));
    size_t at = lo;
    for (int e = top; e >= e0; e -= step) {
        size_t end = at;
        while (end < hi && it[end].e[k] == e) ++end;
        if (k == nv - 1)
            G.slot.push_back(end > at ? it[at].entry : -1);
        else
            emit(it, at, end, k + 1, nv, sq, G);
        at = end;
    }
}

}  // namespace

void nd_order(const std::vector<Mono> &mono, int nv, int *order) {
    // greedily the variable that splits the monomials into the fewest groups
    std::vector<int> group(mono.size(), 0), key(mono.size()), uniq;
    std::vector<bool> used((size_t)nv, false);
    auto split = [&](int v) {
        for (size_t i = 0; i < mono.size(); ++i) key[i] = group[i] * 256 + mono[i][(size_t)v];
        uniq = key;
        std::sort(uniq.begin(), uniq.end());
        uniq.erase(std::unique(uniq.begin(), uniq.end()), uniq.end());
        return uniq.size();
    };
    for (int k = 0; k < nv; ++k) {
        int best = -1;
        size_t least = 0;
        for (int v = 0; v < nv; ++v) {
            if (used[(size_t)v]) continue;
            const size_t n = split(v);
            if (best < 0 || n < least) {
                best = v;
                least = n;
            }
        }
        order[k] = best;
        used[(size_t)best] = true;
        split(best);
        for (size_t i = 0; i < mono.size(); ++i)
            group[i] = (int)(std::lower_bound(uniq.begin(), uniq.end(), key[i]) - uniq.begin());
    }
}

void nd_program(const std::vector<Mono> &mono, const std::vector<int> &pick, int nv, const int *order, NdProgram &G) {
    std::vector<Mono> e(pick.size(), Mono((size_t)nv));
    std::vector<Item> it;
    for (size_t i = 0; i < pick.size(); ++i) {
        for (int k = 0; k < nv; ++k) e[i][k] = mono[(size_t)pick[i]][(size_t)order[k]];
        it.push_back({e[i].data(), pick[i]});
    }
    std::sort(it.begin(), it.end(), [&](const Item &a, const Item &b) {
        for (int k = 0; k < nv; ++k)
            if (a.e[k] != b.e[k]) return a.e[k] > b.e[k];
        return false;
    });
    // depths whose powers keep their parity inside every polynomial
    G.sq = 0;
    for (int k = 0; k < nv; ++k) {
        bool even = true;
        for (size_t i = 1; i < it.size(); ++i) {
            bool same = true;
            for (int j = 0; j < k; ++j) same = same && it[i].e[j] == it[i - 1].e[j];
            if (same && ((it[i].e[k] ^ it[i - 1].e[k]) & 1)) even = false;
        }
        if (even) G.sq |= 1u << k;
    }
    G.words.clear();
    G.slot.clear();
    emit(it, 0, it.size(), 0, nv, G.sq, G);
}

// root mean squares of x_c^e (averaged over the bridge's times), e = 0..top
static std::vector<double> moments(double a, double b, double T, int top) {
    std::vector<double> m((size_t)top + 1, 0.0);
    for (int k = 1; k < 16; ++k) {
        const double u = k / 16.0, mean = a + (b - a) * u, sd = std::sqrt(T * u * (1 - u));
        for (int g = -24; g <= 24; ++g) {
            const double x = mean + sd * g * 0.25;
            double w = std::exp(-0.5 * g * g * 0.0625) * (0.25 / std::sqrt(2 * 3.14159265358979323846)) / 15;
            for (int e = 0; e <= top; ++e, w *= x * x) m[(size_t)e] += w;
        }
    }
    for (double &v : m) v = std::sqrt(v);
    return m;
}

void nd_split(const std::vector<Mono> &mono, int D, const double *a, const double *b, double T, int n,
              const double *table, std::vector<char> &part) {
    const size_t M = mono.size();
    const double N = std::ldexp(1.0, n);
    // in units in which the path is about one across (lengths 2^unit)
    const int unit = std::ilogb(std::sqrt(T));
    const double Tu = std::ldexp(T, -2 * unit), eps = Tu / N;
    std::vector<std::vector<double>> mx((size_t)D), mb((size_t)D);
    for (int c = 0; c < D; ++c) {
        int tx = 1, tb = 1;
        for (const Mono &m : mono) {
            tx = std::max(tx, (int)m[(size_t)c]);
            tb = std::max(tb, (int)m[(size_t)(D + c)]);
        }
        const double au = std::ldexp(a[c], -unit), bu = std::ldexp(b[c], -unit);
        mx[c] = moments(au, bu, Tu, tx);
        const double s2 = 0.25 * (eps + (bu - au) * (bu - au) / (N * N));
        mb[c].assign((size_t)tb + 1, 1.0);
        for (int f = 1; f <= tb; ++f) mb[c][f] = mb[c][f - 1] * std::sqrt(s2 * (2.0 * f - 1));   // E g^2f = (2f - 1)!!
    }
    // the kernel's variables (2 x, 2 xb) in typical size: their powers above one, and
    // whether their squares are floats
    std::vector<double> big[2 * kNdMaxDim];
    bool square[2 * kNdMaxDim];
    for (int v = 0; v < 2 * D; ++v) {
        const std::vector<double> &m = v < D ? mx[(size_t)v] : mb[(size_t)(v - D)];
        const double z = std::ldexp(m[1], unit + 1);
        square[v] = z >= 0x1p-60 && z <= 0x1p60;
        big[v].assign(m.size(), 1.0);
        for (size_t e = 1; e < m.size(); ++e) big[v][e] = big[v][e - 1] * std::max(1.0, z);
    }
    std::vector<std::pair<double, int>> r(M);
    std::vector<double> hi(M, 1.0);
    std::vector<char> floats(M, 1);
    std::vector<int> deg(M, 0);
    double all = 0;
    for (size_t i = 0; i < M; ++i) {
        double v = 1.0;
        for (int c = 0; c < D; ++c) {
            const size_t x = mono[i][(size_t)c], xb = mono[i][(size_t)(D + c)];
            v *= mx[c][x] * mb[c][xb];
            hi[i] *= big[c][x] * big[D + c][xb];
            deg[i] += (int)(x + xb);
            if ((x && !square[c]) || (xb && !square[D + c])) floats[i] = 0;
        }
        v *= unit ? std::ldexp(std::fabs(table[i]), unit * deg[i]) : std::fabs(table[i]);
        r[i] = {v, (int)i};
        all += v;
    }
    part.assign(M, kNdDouble);
    if (!std::isfinite(all)) return;
    std::sort(r.begin(), r.end());
    // N 2^-25 rest <= 2^-55 min(1, N all)
    const double most = 0x1p-30 * std::min(1.0, N * all) / N;
    double rest = 0;
    size_t k = 0;
    for (; k < M && rest + r[k].first <= most; ++k) rest += r[k].first;
    // Of these, what a float's range does not hold stays in double (a partial product
    // below 2^-126 loses at most that times the factors to come), or does not count:
    // less than a float's rounding of the others.
    const double none = 0x1p-24 * most / (double)M;
    for (size_t q = 0; q < k; ++q) {
        const size_t i = (size_t)r[q].second;
        const double c = std::ldexp(std::fabs(table[i]), -deg[i]);
        if (floats[i] && std::max(1.0, c) * hi[i] <= 0x1p100 && 0x1p-126 * hi[i] <= none)
            part[i] = kNdFloat;
        else if (r[q].first <= none)
            part[i] = kNdNone;
    }
}

}  // namespace su
