#pragma once
// 64-bit fixed-point arithmetic for the double-precision sampler (sm_103a).
//
// On this part one double multiply-add holds the SM's FP64 pipe for sixteen
// cycles per warp (2 lanes a cycle), while 32-bit integer and single-precision
// instructions issue at up to four warps a cycle.  Everything whose range is
// known before the launch is therefore kept in 64-bit integers: a product is
// three 32-bit multiplies and three adds, and a sum two adds, with an absolute
// error a few bits below that of the double it takes the place of.
//
// The functions are host and device code: the tests run them on the CPU.
#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define SU_FX_FN __host__ __device__ __forceinline__
#else
#define SU_FX_FN inline
#endif

namespace su {
namespace fx {

SU_FX_FN int32_t hi32(int64_t x) { return (int32_t)(x >> 32); }
SU_FX_FN uint32_t lo32(int64_t x) { return (uint32_t)x; }

SU_FX_FN int32_t mulhi(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
    return __mulhi(a, b);
#else
    return (int32_t)(((int64_t)a * b) >> 32);
#endif
}
SU_FX_FN uint32_t umulhi(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
SU_FX_FN int clz64(uint64_t x) {   // x != 0
#ifdef __CUDA_ARCH__
    return __clzll((long long)x);
#else
    return __builtin_clzll(x);
#endif
}
SU_FX_FN int32_t round_int(float x) {
#ifdef __CUDA_ARCH__
    return __float2int_rn(x);
#else
    return (int32_t)std::nearbyintf(x);
#endif
}
SU_FX_FN float rsqrt_seed(float x) {
#ifdef __CUDA_ARCH__
    return rsqrtf(x);
#else
    return 1.0f / std::sqrt(x);
#endif
}

// A factor as two signed limbs, x = h 2^32 + l with l in [-2^31, 2^31): both
// halves then go through signed multiplies.
struct Limbs {
    int32_t h, l;
};
SU_FX_FN Limbs limbs(int64_t x) {
    const uint32_t l = lo32(x);
    return Limbs{(int32_t)(hi32(x) + (int32_t)(l >> 31)), (int32_t)l};
}

// x f / 2^64 + add + kBias for 0 <= f < 2^63 (as limbs) and |x| < 2^63.  The
// partial products below 2^64 are cut off, which lowers the result by one unit
// on average (in (-3, 0]): kBias is one unit less than the 2^30 that makes the
// cross terms, in [-2^30, 2^31 + 2^30), one unsigned word.  The callers'
// constants carry -kBias, so that the sum costs nothing.
constexpr int64_t kBias = (1LL << 30) - 1;
SU_FX_FN int64_t mul_add(int64_t x, Limbs f, int64_t add) {
    const uint32_t s = umulhi(lo32(x), (uint32_t)f.h) + (uint32_t)mulhi(hi32(x), f.l) + (1u << 30);
    return (int64_t)hi32(x) * f.h + add + (int64_t)(uint64_t)s;
}
SU_FX_FN int64_t mul(int64_t x, Limbs f) { return mul_add(x, f, -kBias); }

// x^2 / 2^64 for |x| < 2^63 (given as limbs), low by less than 2 units
SU_FX_FN int64_t square(Limbs x) {
    const int32_t t = mulhi(x.h, x.l);
    return (int64_t)x.h * x.h + (int64_t)t * 2;
}

// x 2^scale as a double (round to nearest, ties away from zero)
SU_FX_FN double to_double(int64_t x, int scale) {
    const uint64_t sign = (uint64_t)x & 0x8000000000000000ULL;
    const uint64_t n = x < 0 ? 0 - (uint64_t)x : (uint64_t)x;
    const int lz = clz64(n | 1);
    const uint64_t nn = n << lz;                       // leading one at bit 63
    const uint64_t t = (nn >> 11) + ((nn >> 10) & 1);  // 53 bits, 2^53 after a carry
    const uint64_t u = n ? (((uint64_t)(1086 + scale - lz) << 52) + t - (1ULL << 52)) | sign : 0;
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double d;
    std::memcpy(&d, &u, 8);
    return d;
#endif
}

// ---------------------------------------------------------------------------
// z = tanh^2(y), 0 <= y < kTanhNodes / kTanhSteps, in units of 2^-62, from y in
// units of 2^-53 steps of 1/64: in the step [i, i + 1) / 64 the Taylor polynomial
// of degree 7 about its middle (the next term is at most 2^-58, at the ends of
// the steps near y = 0), rewritten in f = 64 y - i in [0, 1).  Entries 0..4 are integers
// in units of 2^-62, entry 5 (below 2^-30) in units of 2^-60, entries 6 and 7
// (below 2^-36) single precision in units of 2^-60.
constexpr int kTanhSteps = 64, kTanhNodes = 384;
struct TanhNode {
    int64_t c[5];
    int32_t c5;
    float f6, f7;
    uint32_t pad;
};
struct TanhTable {
    TanhNode n[kTanhNodes];
};

// a b / 2^120
constexpr unsigned __int128 mul120(unsigned __int128 a, unsigned __int128 b) {
    const unsigned __int128 m = ((unsigned __int128)1 << 60) - 1;
    const unsigned __int128 ah = a >> 60, al = a & m, bh = b >> 60, bl = b & m;   // al bl / 2^120 is dropped
    return ah * bh + ((ah * bl) >> 60) + ((al * bh) >> 60);
}
constexpr TanhTable make_tanh_table() {
    TanhTable T{};
    unsigned __int128 e = (unsigned __int128)1 << 120, term = e;   // exp(-1/64)
    for (int k = 1; k < 20; ++k) {
        term = term / (64 * k);
        if (k & 1)
            e -= term;
        else
            e += term;
    }
    const unsigned __int128 r = mul120(e, e);
    const __int128 one = (__int128)1 << 62;
    for (int i = 0; i < kTanhNodes; ++i, e = mul120(e, r)) {
        // at y = (i + 1/2) / 64: e = exp(-2 y), a[n] the Taylor coefficients of tanh in units of 2^-62
        const unsigned __int128 num = ((unsigned __int128)1 << 120) - e;
        __int128 a[9] = {};
        a[0] = (__int128)((num << 4) / (uint64_t)((((unsigned __int128)1 << 120) + e) >> 58));
        for (int n = 0; n < 8; ++n) {
            __int128 s = n == 0 ? one << 62 : 0;
            for (int k = 0; k <= n; ++k) s -= a[k] * a[n - k];
            a[n + 1] = ((s + ((__int128)1 << 61)) >> 62) / (n + 1);
        }
        // tanh^2 = 1 - tanh': in powers of (f - 1/2), units of 2^-104
        __int128 b[8] = {};
        for (int n = 0; n < 8; ++n) b[n] = ((n == 0 ? one - a[1] : -(n + 1) * a[n + 1]) * ((__int128)1 << 42)) >> (6 * n);
        __int128 p[8] = {};
        for (int k = 0; k < 8; ++k) {
            __int128 binom = 1, s = 0;
            for (int n = k; n < 8; ++n) {
                const __int128 v = (b[n] * binom) >> (n - k);
                s += ((n - k) & 1) ? -v : v;
                binom = binom * (n + 1) / (n + 1 - k);
            }
            p[k] = s;
        }
        // entry k is multiplied by f (below 2^62) k times, each product a quarter: stored times 4^k
        TanhNode &o = T.n[i];
        for (int k = 0; k < 5; ++k)
            o.c[k] = (int64_t)((p[k] + ((__int128)1 << (41 - 2 * k))) >> (42 - 2 * k)) - (k < 4 ? kBias : 0);
        o.c5 = (int32_t)((p[5] + ((__int128)1 << 43)) >> 44);
        o.f6 = (float)(double)(int64_t)(p[6] >> 30) * 0x1p-14f;
        o.f7 = (float)(double)(int64_t)(p[7] >> 30) * 0x1p-14f;
    }
    return T;
}

#ifdef __CUDACC__
static __device__ const TanhTable g_tanh = make_tanh_table();
// the first n nodes into shared memory
__device__ __forceinline__ void tanh_load(TanhNode *t, int n, int tid, int nthreads) {
    const uint2 *s = reinterpret_cast<const uint2 *>(&g_tanh);
    uint2 *d = reinterpret_cast<uint2 *>(t);
    for (int i = tid; i < n * (int)(sizeof(TanhNode) / 8); i += nthreads) d[i] = s[i];
}
#endif

// |x| for the node index: a sum of two points that has left 64 bits may be
// -2^63, whose magnitude is taken as zero (such a path is weighed again)
SU_FX_FN int64_t magnitude(int64_t x) { return (x < 0 ? 0 - (uint64_t)x : (uint64_t)x) & 0x7FFFFFFFFFFFFFFFULL; }

SU_FX_FN int64_t tanh2(int64_t w, const TanhNode *__restrict__ t) {
    const TanhNode &n = t[(int)(w >> 53)];
    const int64_t f = (int64_t)(((uint64_t)w << 11) >> 2);         // units 2^-62
    const Limbs fl = limbs(f);
    const float ff = (float)hi32(f) * 0x1p-30f;
    const int32_t g5 = n.c5 + round_int(ff * fmaf(ff, n.f7, n.f6));
    int64_t g = n.c[4] + (int64_t)mulhi(g5, hi32(f)) * 4096;       // 2^-60 f -> 2^-62 / 4^4
    g = mul_add(g, fl, n.c[3]);
    g = mul_add(g, fl, n.c[2]);
    g = mul_add(g, fl, n.c[1]);
    return mul_add(g, fl, n.c[0]);
}

// ---------------------------------------------------------------------------
// Box-Muller in fixed point: z0 = R cos(theta), z1 = R sin(theta),
// R = sqrt(-2 ln u1), theta = 2 pi u2 (Sec. 4.1, both branches) for the 53-bit
// uniforms u1 = (a + 1/2) 2^-53, u2 = (b + 1/2) 2^-53, as integers in units of
// 2^-57 (|z| < 8.66).
//
//  * -2 ln u1 by the table-driven logarithm (P. T. P. Tang, "Table-driven
//    implementation of the logarithm function in IEEE floating-point
//    arithmetic", ACM TOMS 16, 1990): u1 = m 2^-k, m in [3/4, 3/2), the
//    node c_j = 3/4 + j/1024 nearest to m, r = m inv_j - 1 (inv_j the 32-bit
//    number nearest 1/c_j: exact in 96 bits, |r| < 2^-10.5), and
//      -2 ln u1 = [2 k ln 2 + 2 ln inv_j'] - 2 r + r^2 (1 + G),
//      G = -2 r/3 + r^2 (1/2 - 2 r/5 + r^2/3),
//    ln inv_j' that of the rounded inv_j; the bracket in units of 2^-56, the
//    r^2 part of G in single precision (below 2^-43 of the result).  At the
//    node c = 1 with k = 0 the bracket is zero and the sum stays in units of
//    2^-72, so that it keeps its relative accuracy as u1 goes to 1.
//  * the square root of the even-shifted integer: a single-precision seed and
//    two corrections d/(2s) of the exact integer remainders d = v - s^2.
//  * theta = o pi/4 + phi (odd octants reflected), phi = a_i + d with the 512
//    nodes a_i = pi (i + 1/2)/2048 and |d| <= pi/4096:
//      cos phi = cos d (cos a_i - sin a_i tan d), sin phi likewise,
//    and cos d goes into R: R - R (d^2/2 - d^4/24).
// Root mean square error 8e-18, largest 2e-16 (near u1 = 1, where the slope of
// the square root is large); the table-driven double routines that this
// replaces had 1e-16 and 19 double operations per pair, 304 cycles of the
// FP64 pipe per warp.
struct TrigNode {
    int64_t c, s;                 // cos a_i, sin a_i in units of 2^-62
};
constexpr int kLogNodes = 769;    // c_j = 3/4 + j/1024
constexpr int kTrigNodes = 512;
struct alignas(16) Tables {
    TrigNode tr[kTrigNodes];
    int64_t l2[kLogNodes + 1];    // 2 ln of the rounded inv, units 2^-56
    uint32_t inv[kLogNodes + 3];  // 2^31 / c_j, rounded
};
static_assert(sizeof(Tables) % 16 == 0, "copied in 16-byte pieces");
constexpr int kZScale = 57;       // normals in units of 2^-57

// The node values by their series in integers (units of 2^-62; the same on
// every host): sin and cos by Taylor, ln y = 2 artanh((y - 1)/(y + 1)).
constexpr int64_t q62(__int128 x) { return (int64_t)((x + ((__int128)1 << 61)) >> 62); }
constexpr Tables make_tables() {
    Tables t{};
    for (int i = 0; i < kTrigNodes; ++i) {
        // pi (2 i + 1) / 4096, from pi 2^61
        const int64_t a = (int64_t)((((__int128)0x6487ED5110B4611ALL * (2 * i + 1)) + (1 << 10)) >> 11);
        const int64_t a2 = q62((__int128)a * a);
        int64_t c = (int64_t)1 << 62, s = a, tc = c, ts = a;
        for (int k = 1; k <= 12; ++k) {
            tc = -q62((__int128)tc * a2) / ((2 * k - 1) * (2 * k));
            ts = -q62((__int128)ts * a2) / ((2 * k) * (2 * k + 1));
            c += tc;
            s += ts;
        }
        t.tr[i].c = c;
        t.tr[i].s = s;
    }
    for (int j = 0; j < kLogNodes; ++j) {
        // 2^31 / (3/4 + j/1024) = 2^41 / (768 + j)
        const int64_t inv = ((int64_t)1 << 42) / (768 + j);
        const int64_t y = (inv + 1) >> 1, one = (int64_t)1 << 31;
        const int64_t u = (int64_t)((__int128)(y - one) * ((__int128)1 << 62) / (y + one));
        const int64_t u2 = q62((__int128)u * u);
        int64_t pw = u, sum = u;
        for (int k = 1; k <= 13; ++k) {
            pw = q62((__int128)pw * u2);
            sum += pw / (2 * k + 1);
        }
        t.inv[j] = (uint32_t)y;
        t.l2[j] = (sum + 8) >> 4;   // 4 artanh, units 2^-56
    }
    return t;
}

#ifdef __CUDACC__
static __device__ const Tables g_tables = make_tables();
// the node tables into shared memory (16-byte aligned)
__device__ __forceinline__ void tables_load(Tables *t, int tid, int nthreads) {
    const uint4 *s = reinterpret_cast<const uint4 *>(&g_tables);
    uint4 *d = reinterpret_cast<uint4 *>(t);
    for (int i = tid; i < (int)(sizeof(Tables) / 16); i += nthreads) d[i] = s[i];
}
#endif

SU_FX_FN void normals(uint64_t a, uint64_t b, const Tables *__restrict__ t, int64_t &z0, int64_t &z1) {
    // ---- v = -2 ln u1 = vq 2^-sc
    // u1 = w 2^-54, rounded to a double (to even) where the half takes a 54th bit
    const uint64_t w = 2 * a + ((a >> 52) ? 2 * (a & 1) : 1);
    const int lz = clz64(w);
    const uint64_t x = w << lz;                       // u1 = x 2^-64 2^-(lz - 10)
    const bool low = x < (3ULL << 62);                // m = 2 x 2^-64 in [1, 3/2), else x 2^-64 in [3/4, 1)
    const int j = low ? 256 + (int)((x - (1ULL << 63) + (1ULL << 52)) >> 53)
                      : (int)((x - (3ULL << 62) + (1ULL << 53)) >> 54);
    const uint32_t inv = t->inv[j];
    const uint64_t p0 = (uint64_t)(uint32_t)x * inv;
    const uint64_t p1 = (uint64_t)(uint32_t)(x >> 32) * inv + (p0 >> 32);   // x inv = p1 2^32 + lo32(p0)
    // r 2^73 = (x inv - 2^95) >> 22, or with m = 2 x: (x inv - 2^94) >> 21
    const uint64_t pd = p1 - (low ? 1ULL << 62 : 1ULL << 63);
    const int64_t r1 = (int64_t)((pd << 10) | ((uint32_t)p0 >> 22));
    const int64_t r2 = (int64_t)((pd << 11) | ((uint32_t)p0 >> 21));
    const int64_t r = low ? r2 : r1;
    const Limbs rl = limbs(r);
    const int64_t rr = square(rl);                    // r^2, units 2^-82
    const float rf = (float)rl.h * 0x1p-41f;
    const float gf = fmaf(fmaf(rf, 1.0f / 3.0f, -0.4f), rf, 0.5f);
    const int32_t G = (int32_t)(((int64_t)rl.h * -1431655765) >> 30) + round_int(rf * rf * gf * 0x1p42f);   // units 2^-42
    const int64_t poly = -r + (rr >> 10) + (((int64_t)hi32(rr) * G) >> 20);           // units 2^-72
    const int k = lz - 10 + (low ? 1 : 0);
    const int64_t base = (int64_t)k * 99893036290645747LL + t->l2[j];                    // 2 ln 2 in units of 2^-56
    const bool fine = base == 0;
    int64_t vq = fine ? poly : base + (poly >> 16);
    vq = vq > 0 ? vq : 0;                             // 0 where u1 rounds to 1
    // ---- s = sqrt(v): vn = vq 2^sh in [2^61, 2^63), s^2 = vn 2^64, R = s 2^-32 - (sc + sh)/2
    const int sh = (clz64((uint64_t)vq | 1) - 1) & ~1;
    const uint64_t vn = (uint64_t)vq << sh;
    const float vf = (float)(uint32_t)(vn >> 32);
    const float y = rsqrt_seed(vf > 1.0f ? vf : 1.0f);
    const uint32_t s0 = (uint32_t)(vf * y * 65536.0f);
    const int64_t d1 = (int64_t)(vn - (uint64_t)s0 * s0);                // |d1| < 2^43
    const int32_t e1 = round_int((float)(int32_t)(d1 >> 12) * (y * 0x1p16f));   // d1 / (2 s0) 2^21
    const uint64_t s1 = ((uint64_t)s0 << 32) + (uint64_t)((int64_t)e1 << 11);
    const uint32_t s1h = (uint32_t)(s1 >> 32), s1l = (uint32_t)s1;
    // s1^2 / 2^64 (its lower word's square dropped: less than one unit)
    const uint64_t q1 = (uint64_t)s1h * s1h + ((((uint64_t)s1h * s1l) >> 31));
    const int32_t d2 = (int32_t)(uint32_t)(vn - q1);
    const uint64_t s = s1 + (uint64_t)(int64_t)round_int((float)d2 * (y * 32768.0f));
    // ---- the angle
    const uint32_t o = (uint32_t)(b >> 50);                              // octant
    uint64_t ph = b & ((1ULL << 50) - 1);
    if (o & 1) ph ^= (1ULL << 50) - 1;                                   // pi/4 - phi
    const TrigNode nt = t->tr[(int)(ph >> 41)];
    // d = pi kk 2^-75, kk = 2^22 (2 (ph mod 2^41) - 2^41 + 1); units 2^-72
    const int64_t kk = (int64_t)((ph << 23) + (1ULL << 63) + (1ULL << 22));
    const int64_t d = mul(kk, Limbs{0x6487ED51, 0x10B4611A});            // pi 2^61
    const Limbs dl = limbs(d);
    const int64_t dd = square(dl);                                       // d^2, units 2^-80
    const int32_t qs = (int32_t)(dd >> 29);                              // units 2^-51
    const int32_t d4 = mulhi(qs, qs);                                    // d^4, units 2^-70
    const int64_t cm = (dd >> 9) - ((int64_t)mulhi(d4, 178956971) << 2); // d^2/2 - d^4/24, units 2^-72
    // tan d = d (1 + d^2/3 + 2 d^4/15)
    const int32_t m3 = (int32_t)(((int64_t)qs * 1431655765) >> 31) + (mulhi(d4, 572662306) >> 18);   // units 2^-52
    const int64_t td = d + (((int64_t)dl.h * m3) >> 20);                 // units 2^-72
    // R cos d in units of 2^-59 (R < 8.66)
    const int rs = (sh >> 1) + (fine ? 8 : 0) + 1;
    const int64_t R = (int64_t)(s >> rs);
    const Limbs Rl = limbs(R - (mul(cm, limbs(R)) >> 8));
    // cos a - sin a tan d, sin a + cos a tan d, units 2^-62
    const Limbs cl = limbs(nt.c), sl = limbs(nt.s);
    const int64_t cf = nt.c - (mul(td, sl) >> 8);
    const int64_t sf = nt.s + (mul(td, cl) >> 8);
    const uint32_t q = o >> 1;
    const bool swap = ((o ^ q) & 1) != 0;
    const int64_t P = swap ? sf : cf, Q = swap ? cf : sf;
    // theta = q pi/2 + psi, (cos psi, sin psi) = (cf, sf) for even octants and
    // (sf, cf) for odd ones; then the quadrant's quarter turns
    z0 = mul((q == 1 || q == 2) ? -P : P, Rl);
    z1 = mul(q >= 2 ? -Q : Q, Rl);
}

}  // namespace fx
}  // namespace su
