// The amplitude estimator for systems of d = D x M coordinates (Sec. 2.2,
// Eq. EXP / Eq. MBrec): bisection paths of every coordinate (Sec. 4.1), the
// level-p effective potential W(x, xb; eps) of a polynomial potential per
// slice, per-sample log-weights of every level, per-item log-sum-exp tuples.
#include <cstdint>
#include <type_traits>

#include "sampler_impl.cuh"

namespace su {
namespace {

// Lanes of the evaluation: two slices in a packed pair of floats, or one double.
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
__device__ __forceinline__ void vzero(float2 &a) { a = make_float2(0.f, 0.f); }
__device__ __forceinline__ void vzero(double &a) { a = 0.0; }

// The variables of B lanes in program order: z_k, and the Horner variable of
// depth k (z_k or its square).
template <typename VT, int NV, int B>
struct Vars {
    VT z[NV][B], m[NV][B];
    unsigned one;   // 1, not known to the compiler (double)
    __device__ __forceinline__ void close(unsigned sq, unsigned once) {
        one = once;
#pragma unroll
        for (int k = 0; k < NV; ++k)
#pragma unroll
            for (int i = 0; i < B; ++i) m[k][i] = (sq >> k) & 1 ? vmul(z[k][i], z[k][i]) : z[k][i];
    }
};

// Steps that only some polynomials have -- the factor z_k, and a Horner chain's
// multiply-add after the first -- are loops of no or one pass in double, where an
// operation holds the pipe for 16 cycles: written as conditions the compiler
// computed both for all and selected (102 double operations a slice, two coordinates
// at p = 10; 54 now: 47.3 -> 29.7 ms for 100 003 paths of 1024 slices), and kept
// from that it left them to predicates, which hold the pipe too (37.4 ms).
// t = the polynomial in z_K.. at w (words) and c (coefficients), both moved past it
template <int K, typename VT, int NV, int B>
__device__ __forceinline__ void nd_poly(const uint32_t *__restrict__ &w, const VT *__restrict__ &c,
                                        const Vars<VT, NV, B> &v, VT (&t)[B]) {
    constexpr bool kSkip = std::is_same<VT, double>::value;
    const uint32_t hd = *w++;
    const int n = (int)(hd & 0xffffu);
    if constexpr (K == NV - 1) {
#pragma unroll
        for (int i = 0; i < B; ++i) vzero(t[i]);
        if (n) {
            const VT top = *c;
#pragma unroll
            for (int i = 0; i < B; ++i) t[i] = top;
#pragma unroll 1
            for (int e = 1; e < n; ++e) {
                const VT ce = c[e];
#pragma unroll
                for (int i = 0; i < B; ++i) t[i] = vfma(t[i], v.m[K][i], ce);
            }
            c += n;
        }
    } else {
#pragma unroll
        for (int i = 0; i < B; ++i) vzero(t[i]);
#pragma unroll 1
        for (int e = 0; e < n; ++e) {
            VT u[B];
            nd_poly<K + 1>(w, c, v, u);
            if constexpr (kSkip) {
#pragma unroll 1
                for (unsigned o = e ? v.one : 0u; o; --o)
#pragma unroll
                    for (int i = 0; i < B; ++i) u[i] = vfma(t[i], v.m[K][i], u[i]);
#pragma unroll
                for (int i = 0; i < B; ++i) t[i] = u[i];
            } else {
#pragma unroll
                for (int i = 0; i < B; ++i) t[i] = vfma(t[i], v.m[K][i], u[i]);
            }
        }
    }
    if constexpr (kSkip) {
#pragma unroll 1
        for (uint32_t o = hd >> 16; o; --o)   // kNdOdd
#pragma unroll
            for (int i = 0; i < B; ++i) t[i] = vmul(t[i], v.z[K][i]);
    } else if (hd & kNdOdd) {
#pragma unroll
        for (int i = 0; i < B; ++i) t[i] = vmul(t[i], v.z[K][i]);
    }
}

// The largest sum of the slices' single-precision parts over a path, of max(1, |w|):
// typically below 2^-30, where what single precision rounds is below 2^-55; at the
// limit some 2^-50 (the entries are two to four times their slices' sums).  Beyond
// it, about one path in a million, the second pass takes the path's own lane 7.5 ms
// (two coordinates, p = 10, one level of 512 slices), so that a limit of 2^-28
// doubled the time of a call of 50 001 such paths.
constexpr float kNdTail = 0x1p-27f;

// x (rounded to nearest) for |x| < 2^127 as a float, on the integer pipes
__device__ __forceinline__ float narrow(double x) {
    const uint64_t u = (uint64_t)__double_as_longlong(x);
    const uint64_t mag = (u & 0x7FFFFFFFFFFFFFFFULL) + (1ULL << 28);
    const uint32_t f = mag >= (897ULL << 52) ? (uint32_t)(mag >> 29) - (896u << 23) : 0u;
    return __uint_as_float(f | ((uint32_t)(u >> 32) & 0x80000000u));
}
__device__ __forceinline__ float narrow(float x) { return x; }

// the sum of 2 BP slices' -eps W in single precision (points pt(k0 stp).. of R), and
// the sum of its magnitudes
template <typename R, int D, int BP, typename PT>
__device__ __forceinline__ float2 nd_single(const NdParams &Q, const uint32_t *w, const float2 *c, PT &&pt, int k0, int stp) {
    Vars<float2, 2 * D, BP> v;
#pragma unroll
    for (int k = 0; k < 2 * D; ++k) {
        // l + r = 2x of a coordinate, or r - l = 2xb (the entries carry the powers of two)
        const int var = Q.order[k], cc = var >= D ? var - D : var;
        const R sg = var >= D ? (R)-1 : (R)1;
        R l = pt(k0 * stp, cc);
#pragma unroll
        for (int i = 0; i < BP; ++i) {
            const R a = pt((k0 + 2 * i + 1) * stp, cc), b = pt((k0 + 2 * i + 2) * stp, cc);
            v.z[k][i] = make_float2(narrow(fma(sg, l, a)), narrow(fma(sg, a, b)));
            l = b;
        }
    }
    v.close(Q.sq, Q.one);
    float2 t[BP];
    nd_poly<0>(w, c, v, t);
    float s = 0, m = 0;
#pragma unroll
    for (int i = 0; i < BP; ++i) {
        s += t[i].x + t[i].y;
        m += fabsf(t[i].x) + fabsf(t[i].y);
    }
    return make_float2(s, m);
}

// B slices' -eps W in double
template <int D, int B, typename PT>
__device__ __forceinline__ double nd_double(const NdParams &Q, unsigned sq, const uint32_t *w, const double *c, PT &&pt,
                                            int k0, int stp) {
    Vars<double, 2 * D, B> v;
#pragma unroll
    for (int k = 0; k < 2 * D; ++k) {
        const int var = Q.order[k], cc = var >= D ? var - D : var;
        const double sg = var >= D ? -1.0 : 1.0;
        double l = pt(k0 * stp, cc);
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const double e = pt((k0 + i + 1) * stp, cc);
            v.z[k][i] = fma(sg, l, e);
            l = e;
        }
    }
    v.close(sq, Q.one);
    double t[B];
    nd_poly<0>(w, c, v, t);
    double s = 0;
#pragma unroll
    for (int i = 0; i < B; i += 2) s += t[i] + t[i + 1];
    return s;
}

// R = double or float (the path and the per-level sums; the item's log-sum-exp
// tuples in double either way).
// Shared memory: sw[levels][kThreads] (R, reduced runs) | Box-Muller node tables
// (double) | where Q.staged: words | pairs [S][M] | double part's entries, words.
// Global scratch per slot: the 2^(S-F) + 1 segment endpoints (F = min(S, kNdSeg)).
//
// What bounds it.  Single precision: instruction issue, most of it the packed
// multiply-adds of the nest and the loops around them.  Double: the FP64 pipe
// (2 lanes a cycle; 56 % busy) in the double part, a tenth of the entries on fine
// levels, and the latency of its short chains: four slices a pass instead of two,
// where their variables fit the registers (D <= 2), took the case above from 29.7 to
// 24.4 ms.
template <typename R, int D>
__global__ void __launch_bounds__(kThreads, D == 3 ? 3 : 4) nd_kernel(const __grid_constant__ NdParams Q) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const SamplerParams &P = Q.base;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int L = P.levels, S = P.S;
    const bool per_sample = P.w_out != nullptr;
    R *sw = reinterpret_cast<R *>(smem_raw);
    size_t off = per_sample ? 0 : sizeof(R) * (size_t)L * kThreads;
    off = (off + 15) & ~(size_t)15;
    fx::Tables *bm_smem = reinterpret_cast<fx::Tables *>(smem_raw + off);
    if constexpr (sizeof(R) == 8) {
        fx::tables_load(bm_smem, tid, kThreads);
        off += sizeof(fx::Tables);
    }
    const uint32_t *words = Q.words, *hwords = Q.hwords;
    const float2 *pairs = sizeof(R) == 8 ? Q.tail : reinterpret_cast<const float2 *>(P.tables);
    const double *hcoef = Q.hcoef;
    if (Q.staged) {
        auto stage = [&](auto *&src, int n) {
            using T = typename std::remove_const<typename std::remove_pointer<typename std::remove_reference<decltype(src)>::type>::type>::type;
            T *dst = reinterpret_cast<T *>(smem_raw + off);
            for (int i = tid; i < n; i += kThreads) dst[i] = src[i];
            src = dst;
            off = (off + sizeof(T) * (size_t)n + 15) & ~(size_t)15;
        };
        stage(words, Q.n_words);
        stage(pairs, S * P.M);
        if constexpr (sizeof(R) == 8) {
            stage(hcoef, Q.n_hcoef);
            stage(hwords, Q.n_hwords);
        }
    }
    __syncthreads();

    Stream<R> st;
    st.key = make_uint2((uint32_t)P.seed, (uint32_t)(P.seed >> 32));
    st.inst = P.instance;
    st.bm = sizeof(R) == 8 ? bm_smem : nullptr;
    const int64_t ps = Q.pstride;
    // the path in segments of 2^F slices: the C + 1 segment endpoints (the
    // coarse levels' points) in this slot of the global scratch, one
    // segment's points at a time in local memory
    const int F = min(S, kNdSeg), Cn = S - F, C = 1 << Cn, NF = 1 << F;
    R *q = reinterpret_cast<R *>(Q.paths) + (int64_t)blockIdx.x * kThreads + tid;
    auto co = [&](int i, int c) -> R & { return q[((int64_t)i * D + c) * ps]; };
    R seg[((1 << kNdSeg) + 1) * D];
    constexpr int kBD = D <= 2 ? 4 : 2;          // slices per pass of the double part
    constexpr int kBP = D == 4 ? 2 : 4;          // pairs of slices per pass of the single-precision program

    for (int64_t item = P.item0 + blockIdx.x; item < P.n_items; item += gridDim.x) {
        const int64_t b = item / P.items_per_block;
        const int64_t r = item - b * P.items_per_block;
        const int64_t lo = b * P.n_mc / P.n_blocks;
        const int64_t hi = (b + 1) * P.n_mc / P.n_blocks;
        const int64_t start = lo + r * kThreads;
        const int cnt = (int)max((int64_t)0, min((int64_t)kThreads, hi - start));
        if (tid < cnt) {
            const uint64_t sample = (uint64_t)(P.sample0 + start + tid);
            st.slo = (uint32_t)sample;
            st.shi = (uint32_t)(sample >> 32);
            // normal g of the sample's stream: double, branch g & 1 of the
            // Box-Muller pair of call g >> 1; float, slot (g + 1) & 3 of the
            // four normals of call (g + 1) >> 2 (the one-dimensional layouts)
            uint32_t have = 0xffffffffu;   // the call last drawn
            R zc[4] = {0, 0, 0, 0};
            auto normal = [&](uint32_t g) -> R {
                if constexpr (sizeof(R) == 8) {
                    if ((g >> 1) != have) {
                        double z0, z1;
                        st.pair(g >> 1, z0, z1);
                        zc[0] = z0;
                        zc[1] = z1;
                        have = g >> 1;
                    }
                    return (g & 1u) ? zc[1] : zc[0];
                } else {
                    if (((g + 1) >> 2) != have) {
                        st.quad((g + 1) >> 2, zc);
                        have = (g + 1) >> 2;
                    }
                    return pick4(zc, g + 1);
                }
            };
            R wloc[SU_MAX_S];
            // pass 0 with the split levels; again in double for the levels whose
            // single-precision part is beyond kNdTail
            uint32_t todo = (1u << L) - 1u, far = 0;
            for (int pass = 0; pass < 2; ++pass) {
                float mag[sizeof(R) == 8 ? SU_MAX_S : 1];
                // coarse levels n = 1..S-F: midpoint i at segment endpoint (2i+1) 2^(S-F-n)
                have = 0xffffffffu;
                for (int c = 0; c < D; ++c) {
                    co(0, c) = Q.a[c];
                    co(C, c) = Q.b[c];
                }
                for (int n = 1; n <= Cn; ++n) {
                    const R sg = (R)P.sigma[n];
                    const int h = 1 << (Cn - n), j0 = (1 << (n - 1)) - 1;
                    for (int i = 0; i < (1 << (n - 1)); ++i) {
                        const int idx = (2 * i + 1) * h;
                        for (int c = 0; c < D; ++c)
                            co(idx, c) = fma(sg, normal((uint32_t)((j0 + i) * D + c)), (R)0.5 * (co(idx - h, c) + co(idx + h, c)));
                    }
                }
                // w_n = -eps_n sum_k W on the level-n subpath (level n = S - dl),
                // slices in ascending order, several at a time
                for (int dl = 0; dl < L; ++dl) {
                    if (todo >> dl & 1u) wloc[dl] = 0;
                    if constexpr (sizeof(R) == 8) mag[dl] = 0;
                }
                auto slices = [&](int dl, auto &&pt, int stp, int ns) {
                    if (sizeof(R) == 8 && !(todo >> dl & 1u)) return;
                    R w = 0;
                    if constexpr (sizeof(R) == 4) {
                        const float2 *c = pairs + (size_t)dl * P.M;
                        if (ns >= 2 * kBP) {
#pragma unroll 1
                            for (int k = 0; k < ns; k += 2 * kBP) w += nd_single<R, D, kBP>(Q, words, c, pt, k, stp).x;
                        } else {
#pragma unroll 1
                            for (int k = 0; k < ns; k += 2) w += nd_single<R, D, 1>(Q, words, c, pt, k, stp).x;
                        }
                    } else if (pass == 0 && Q.heads[dl] > 0) {
                        const float2 *c = pairs + (size_t)dl * P.M;
                        float2 tail = make_float2(0.f, 0.f);
                        if (ns >= 2 * kBP) {
#pragma unroll 1
                            for (int k = 0; k < ns; k += 2 * kBP) tail = __fadd2_rn(tail, nd_single<R, D, kBP>(Q, words, c, pt, k, stp));
                        } else {
#pragma unroll 1
                            for (int k = 0; k < ns; k += 2) tail = __fadd2_rn(tail, nd_single<R, D, 1>(Q, words, c, pt, k, stp));
                        }
                        mag[dl] += tail.y;
                        if (kBD > 2 && ns >= kBD) {
#pragma unroll 1
                            for (int k = 0; k < ns; k += kBD)
                                w += nd_double<D, kBD>(Q, Q.hsq[dl], hwords + Q.hw[dl], hcoef + Q.hc[dl], pt, k, stp);
                        } else {
#pragma unroll 1
                            for (int k = 0; k < ns; k += 2)
                                w += nd_double<D, 2>(Q, Q.hsq[dl], hwords + Q.hw[dl], hcoef + Q.hc[dl], pt, k, stp);
                        }
                        w += (double)tail.x;
                    } else {
#pragma unroll 1
                        for (int k = 0; k < ns; k += 2)
                            w += nd_double<D, 2>(Q, Q.sq, words, reinterpret_cast<const double *>(P.tables) + (size_t)dl * P.M, pt, k, stp);
                    }
                    wloc[dl] += w;
                };
#pragma unroll 1
                for (int dl = F; dl < L; ++dl)   // coarse levels: between segment endpoints
                    slices(dl, co, 1 << (dl - F), 1 << (S - dl));
                // fine levels n = S-F+1..S, one segment at a time
                auto fp = [&](int i, int c) -> R & { return seg[i * D + c]; };
#pragma unroll 1
                for (int sgi = 0; sgi < C; ++sgi) {
                    for (int c = 0; c < D; ++c) {
                        fp(0, c) = co(sgi, c);
                        fp(NF, c) = co(sgi + 1, c);
                    }
                    for (int n = Cn + 1; n <= S; ++n) {
                        const R sg = (R)P.sigma[n];
                        const int h = 1 << (S - n), m = 1 << (n - Cn - 1);
                        const int j0 = (1 << (n - 1)) - 1 + sgi * m;
                        for (int il = 0; il < m; ++il) {
                            const int idx = (2 * il + 1) * h;
                            for (int c = 0; c < D; ++c)
                                fp(idx, c) = fma(sg, normal((uint32_t)((j0 + il) * D + c)), (R)0.5 * (fp(idx - h, c) + fp(idx + h, c)));
                        }
                    }
#pragma unroll 1
                    for (int dl = 0; dl < min(F, L); ++dl) slices(dl, fp, 1 << dl, NF >> dl);
                }
                if constexpr (sizeof(R) == 8) {
                    if (pass == 0)
                        for (int dl = 0; dl < L; ++dl)
                            if (Q.heads[dl] > 0 && !(mag[dl] <= kNdTail * fmaxf(1.0f, fabsf(__double2float_rn(wloc[dl]))))) far |= 1u << dl;
                }
                todo = far;
                if (pass || !far) break;
            }
            bool bad = false;
            for (int dl = 0; dl < L; ++dl) bad |= isnan(wloc[dl]) || (isinf(wloc[dl]) && wloc[dl] > 0);
            if (bad) atomicOr(P.flags, 1);
            if (per_sample) {
                double *dst = P.w_out + (start + tid) * (int64_t)S;
                for (int dl = 0; dl < L; ++dl) dst[S - dl - 1] = (double)wloc[dl];
            } else {
                for (int dl = 0; dl < L; ++dl) sw[(size_t)dl * kThreads + tid] = wloc[dl];
            }
        }
        if (per_sample) continue;
        __syncthreads();
        item_lse<R>(sw, L, kThreads, cnt, P.partial, item, warp, lane);
        __syncthreads();
    }
}

template <typename R>
const void *nd_fn_r(int D) {
    switch (D) {
        case 1: return (const void *)nd_kernel<R, 1>;
        case 2: return (const void *)nd_kernel<R, 2>;
        case 3: return (const void *)nd_kernel<R, 3>;
        default: return (const void *)nd_kernel<R, 4>;
    }
}

const void *nd_fn(int D, int precision) {
    return precision == SU_FP32 ? nd_fn_r<float>(D) : nd_fn_r<double>(D);
}

}  // namespace

size_t nd_smem_bytes(const NdParams &Q, int precision) {
    const size_t rs = precision == SU_FP32 ? sizeof(float) : sizeof(double);
    auto up = [](size_t x) { return (x + 15) & ~(size_t)15; };
    size_t off = up(Q.base.w_out ? 0 : rs * (size_t)Q.base.levels * kThreads);
    if (precision != SU_FP32) off += sizeof(fx::Tables);
    if (Q.staged) {
        off = up(off + sizeof(uint32_t) * (size_t)Q.n_words);
        off = up(off + sizeof(float2) * (size_t)Q.base.S * Q.base.M);
        if (precision != SU_FP32) {
            off = up(off + sizeof(double) * (size_t)Q.n_hcoef);
            off = up(off + sizeof(uint32_t) * (size_t)Q.n_hwords);
        }
    }
    return off;
}

int nd_occupancy(const NdParams &Q, int precision, size_t smem) {
    const void *fn = nd_fn(Q.D, precision);
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, kThreads, smem) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb;
}

cudaError_t launch_nd(const NdParams &Q, int precision, int grid, size_t smem, cudaStream_t st) {
    const void *fn = nd_fn(Q.D, precision);
    cudaGetLastError();
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    void *args[] = {const_cast<NdParams *>(&Q)};
    return cudaLaunchKernel(fn, dim3(grid), dim3(kThreads), args, smem, st);
}

}  // namespace su
