#pragma once
// The double-precision sampler in fixed point (sm_103a): the same estimator,
// stream and outputs as sampler_kernel<double>, with path points, normals and
// the leading part of W_p in 64-bit integers and the rest of W_p, below 2^-29
// of it, in packed single precision (fx_plan.cpp: scales, ranges and error
// bounds; fixed_point.cuh: the arithmetic).
//
// What bounds it: sampler_kernel<double> keeps the FP64 pipe 93 % busy (2
// lanes a cycle on this part) with every other pipe idle.  Here nothing of the
// inner loops touches that pipe: about 300 integer and single-precision
// instructions per slice action, issue 58 %, ALU pipe 44 %, FMA pipe 39 %
// busy, the rest dependency waits and instruction fetch.  Anharmonic
// oscillator g = 10, p = 10, N = 1024 with every level, 400 003 samples:
// 45.7 ms in double, 14.1 ms with the tail's table shape read at run time,
// 11.4 ms with it compiled in (four CTAs an SM; five at 96 registers 11.8 ms,
// integer chains of eight slices instead of four 11.9 ms).  The weights' root
// mean square error against 128-bit arithmetic is 5e-17 to 1.5e-16 where the
// double sampler's is 1e-16 to 2e-16.
//
// One path per thread.  The path is walked depth first: the right endpoints
// of the current interval of every level above the register segment are a
// stack (at most 7 entries) in shared memory, instead of all segment
// endpoints, so that four CTAs fit an SM.  A normal of the coarse levels or a
// segment's 15 normals are drawn where they are needed (counter-based stream);
// the second normal of a Box-Muller pair waits in a row per level for the
// midpoint to its right.  A path whose points or steps leave the planned
// ranges (probability 1e-7) is taken again in double.
#include "sampler_impl.cuh"

namespace su {
namespace {

// 96-bit sum of 64-bit terms
struct Acc96 {
    uint32_t lo = 0, mid = 0, hi = 0;
    __device__ __forceinline__ void add(int64_t v) {
        const uint32_t vl = (uint32_t)v, vh = (uint32_t)((uint64_t)v >> 32), vs = (uint32_t)((int32_t)vh >> 31);
        asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
            : "+r"(lo), "+r"(mid), "+r"(hi)
            : "r"(vl), "r"(vh), "r"(vs));
    }
    // the sum in units of 2^-e
    __device__ __forceinline__ double value(int e) const {
        return fx::to_double((int64_t)(((uint64_t)hi << 32) | mid), 32 - e) + fx::to_double((int64_t)(uint64_t)lo, -e);
    }
};

// The kernel's shared memory as one thread sees it.  Rows (stride kThreads,
// this thread's column): right endpoints of levels 0..S-F, then the points of
// the segment at hand (first its normals, in their midpoints' places).
constexpr int kFxSeg = 4;                        // segments of 2^4 slices (fewer on shallow paths)
constexpr int kRowQ = SU_MAX_S - kFxSeg + 1;
constexpr int kFxRows = kRowQ + (1 << kFxSeg) + 1;
struct FxView {
    const fx::TanhNode *th;  // RING_TANH2: its nodes
    const float2 *tail;      // [S][M] single-precision entries as pairs {c, c}, zero where the entry is an integer one
    const int64_t *head;     // [S][hrow]
    int64_t *R;              // this thread's first row
    __device__ __forceinline__ int64_t &q(int i) const { return R[(kRowQ + i) * kThreads]; }
};

// ------------------------------------------------------------------ slices
// The sum of -eps W_p over B slices, integer part, in units of 2^-e: nested
// Horner over the leading entries (last column first), B chains side by side.
template <int B>
__device__ __forceinline__ int64_t fx_heads(const fx::Limbs (&Z)[B], const int64_t (&vs)[B], const FxLevel &L,
                                            const int64_t *__restrict__ h) {
    fx::Limbs Y[B];
    int64_t acc[B];
#pragma unroll
    for (int b = 0; b < B; ++b) Y[b] = fx::limbs(fx::square(fx::limbs(vs[b] << L.ky)) << 1);
    for (int j = L.nc - 1; j >= 0; --j) {
        int64_t g[B];
        const int64_t top = *h++;
#pragma unroll
        for (int b = 0; b < B; ++b) g[b] = top;
        for (int i = L.h[j] - 1; i > 0; --i) {
            const int64_t c = *h++;
#pragma unroll
            for (int b = 0; b < B; ++b) g[b] = fx::mul_add(g[b], Z[b], c);
        }
        if (j == L.nc - 1) {
#pragma unroll
            for (int b = 0; b < B; ++b) acc[b] = g[b];
        } else {
#pragma unroll
            for (int b = 0; b < B; ++b) acc[b] = fx::mul_add(acc[b], Y[b], g[b]);
        }
    }
    int64_t s = acc[0];
#pragma unroll
    for (int b = 1; b < B; ++b) s += acc[b];
    return s;
}

// z in units of 2^-63 from us
template <int RING>
__device__ __forceinline__ fx::Limbs fx_ring(int64_t us, const FxParams &X, const fx::TanhNode *th) {
    if constexpr (RING == RING_EVEN)
        return fx::limbs(fx::square(fx::limbs(us)) << 1);
    else
        return fx::limbs(fx::tanh2(fx::mul(fx::magnitude(us), fx::Limbs{X.ah, X.al}), th) << 1);
}

// a high word in units of 1
__device__ __forceinline__ float fx_unit(int32_t h) { return (float)h * 0x1p-31f; }

// BT slices between the points q[k stp], k = 0..BT: the single-precision
// entries (packed pairs of slices), then in batches of four the integer ones.
// (z = us^2 is cheaper made again for them than kept, tanh^2 is kept.)
template <int RING, int BT, typename SP>
__device__ __forceinline__ void fx_batch(const int64_t *__restrict__ q, int stp, const FxLevel &L, const FxParams &X,
                                         const fx::TanhNode *th, const float2 *__restrict__ tail,
                                         const int64_t *__restrict__ head, const SP &P, float2 &ts, Acc96 &acc,
                                         int &vm) {
    constexpr int BP = BT < 2 ? 1 : BT / 2;
    constexpr bool kKeep = RING != RING_EVEN;
    fx::Limbs Zk[kKeep ? BT : 1];
    float2 Zf[BP], Yf[BP], af[BP];
    {
        int64_t l = q[0];
#pragma unroll
        for (int m = 0; m < BP; ++m) {
            float u[2], v[2];
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                if (BT < 2 && s) {
                    u[1] = u[0];
                    v[1] = v[0];
                    break;
                }
                const int64_t r = q[(2 * m + s + 1) * stp];
                const int64_t us = l + r, vs = r - l;
                vm = max(vm, abs(fx::hi32(vs)));
                if constexpr (kKeep) {
                    Zk[2 * m + s] = fx_ring<RING>(us, X, th);
                    u[s] = fx_unit(Zk[2 * m + s].h);
                } else {
                    u[s] = fx_unit(fx::hi32(us));
                }
                v[s] = fx_unit((int32_t)__funnelshift_l(fx::lo32(vs), (uint32_t)fx::hi32(vs), L.ky));
                l = r;
            }
            Zf[m] = kKeep ? make_float2(u[0], u[1])
                          : __fmul2_rn(make_float2(u[0], u[1]), make_float2(u[0], u[1]));
            Yf[m] = __fmul2_rn(make_float2(v[0], v[1]), make_float2(v[0], v[1]));
        }
    }
    horner_packed<BP>(af, Yf, Zf, tail, P);
#pragma unroll
    for (int m = 0; m < BP; ++m) ts = __fadd2_rn(ts, BT < 2 ? make_float2(af[m].x, 0.f) : af[m]);
    constexpr int B = BT < 4 ? BT : 4;
    auto heads = [&](int k1) {
        fx::Limbs Z[B];
        int64_t vs[B], l = q[k1 * stp];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int64_t r = q[(k1 + b + 1) * stp];
            if constexpr (kKeep)
                Z[b] = Zk[k1 + b];
            else
                Z[b] = fx_ring<RING>(l + r, X, th);
            vs[b] = r - l;
            l = r;
        }
        acc.add(fx_heads<B>(Z, vs, L, head));
    };
    if constexpr (kKeep) {   // unrolled: Zk stays in registers
#pragma unroll
        for (int k1 = 0; k1 < BT; k1 += B) heads(k1);
    } else {
#pragma unroll 1
        for (int k1 = 0; k1 < BT; k1 += B) heads(k1);
    }
}

// One level of a segment: ns slices between points stp apart (2^F = ns stp / kThreads).
template <int RING, typename SP>
__device__ __forceinline__ void fx_level(const int64_t *__restrict__ q, int ns, int stp, const FxLevel &L,
                                         const FxParams &X, const fx::TanhNode *th, const float2 *__restrict__ tail, const int64_t *__restrict__ head, const SP &P,
                                         Acc96 &acc, bool &bad) {
    float2 ts = make_float2(0.f, 0.f);
    int vm = 0;
    if (ns >= 8) {
#pragma unroll 1
        for (int k = 0; k < ns; k += 8) fx_batch<RING, 8>(q + k * stp, stp, L, X, th, tail, head, P, ts, acc, vm);
    } else if (ns == 4) {
        fx_batch<RING, 4>(q, stp, L, X, th, tail, head, P, ts, acc, vm);
    } else {
#pragma unroll 1
        for (int k = 0; k < ns; ++k) fx_batch<RING, 1>(q + k * stp, stp, L, X, th, tail, head, P, ts, acc, vm);
    }
    acc.add(__float2ll_rn(ts.x + ts.y));
    bad |= vm >= L.vlim;
}

// one slice in double from the level's table in global memory (levels whose
// integer sums would not fit: few slices)
template <int RING>
__device__ __noinline__ double fx_slice_double(const SamplerParams &P, double ql, double qr, int d) {
    return slice<double, RING>(ql, qr, reinterpret_cast<const double *>(P.tables) + (size_t)d * P.M, P, P.alpha);
}

// ------------------------------------------------------------------ a path
// the same path in double, one slice at a time: paths out of the planned ranges
template <int RING>
__device__ __noinline__ void fx_slow_path(const SamplerParams &P, const Stream<double> &st, double *w) {
    const int S = P.S, N = 1 << S;
    double R[SU_MAX_S + 1], carry[SU_MAX_S + 1];
    double left = P.a;
    R[0] = P.b;
    for (int n = 1; n <= S; ++n) w[n] = 0;
    for (int c = 0; c < N; ++c) {
        const int n0 = c ? S - (__ffs(c) - 1) : 0;
        if (c) {
            left = R[S];
            R[n0] = R[n0 - 1];
        }
        for (int n = n0 + 1; n <= S; ++n) {
            const uint32_t i = (uint32_t)c >> (S - n + 1), j = (1u << (n - 1)) - 1u + i;
            double z = carry[n], z0, z1;
            if (!(j & 1u) || i == 0) {
                st.pair(j >> 1, z0, z1);
                z = (j & 1u) ? z1 : z0;
                if (!(j & 1u)) carry[n] = z1;
            }
            R[n] = fma(P.sigma[n], z, 0.5 * (left + R[n - 1]));
        }
        for (int n = max(n0, 1); n <= S; ++n)
            if (S - n < P.levels) w[n] += fx_slice_double<RING>(P, left, R[n], S - n);
    }
}

// Writes the log-weight of sampled level d (level n = S - d) to wout[d * wstride].
template <int RING, typename SP>
__device__ __forceinline__ void fx_path(const SamplerParams &P, const SP &V, const FxView &sm, const Stream<double> &st,
                                        double *wout, int wstride) {
    const FxParams &X = P.fx;
    const int S = P.S, F = P.F, NF = 1 << F, Cn = S - F, C = 1 << Cn;
    bool bad = false;
    uint32_t ov = 0;     // sign bit: a sum left 64 bits
    int qm = 0;          // largest |high word| of a point
    auto place = [&](int64_t l, int64_t r, int64_t z, int n) {
        const int64_t m = (l + r) >> 1;
        const int64_t d = fx::mul(z, fx::Limbs{X.sgh[n], X.sgl[n]}) << X.shl[n];
        const int64_t v = m + d;
        ov |= (uint32_t)((fx::hi32(v) ^ fx::hi32(m)) & (fx::hi32(v) ^ fx::hi32(d)));
        qm = max(qm, abs(fx::hi32(v)));
        return v;
    };
    // by level, in local memory: the second normal of its last pair, its sum
    int64_t carry[SU_MAX_S + 1];
    Acc96 acc[SU_MAX_S];
    double wsum[SU_MAX_S];
    for (int d = 0; d < P.levels; ++d) {
        acc[d] = Acc96{};
        wsum[d] = 0.0;
    }
    // the slices of level S - d between the points q[k stp]
    auto level = [&](const int64_t *q, int ns, int stp, int d) {
        const FxLevel &L = X.lv[d];
        if (L.ok) {
            Acc96 a = acc[d];
            fx_level<RING>(q, ns, stp, L, X, sm.th, sm.tail + d * P.M, sm.head + d * X.hrow, V, a, bad);
            acc[d] = a;
        } else {
            for (int k = 0; k < ns; ++k)
                wsum[d] += fx_slice_double<RING>(P, (double)q[k * stp] * X.q_unit, (double)q[(k + 1) * stp] * X.q_unit, d);
        }
    };
    int64_t left = X.qa;
    sm.R[0] = X.qb;
    for (int c = 0; c < C; ++c) {
        // ---- the intervals that begin here: levels n0..S-F, their right endpoints
        const int n0 = c ? Cn - (__ffs(c) - 1) : 0;
        if (c) {
            left = sm.R[Cn * kThreads];
            sm.R[n0 * kThreads] = sm.R[(n0 - 1) * kThreads];
        }
        int64_t right = sm.R[n0 * kThreads];
        sm.q(0) = left;
        // Normals: level n's midpoints i0..i0+m-1 (normals jb..) go to dst[k step];
        // the first one of an odd jb is the second of the pair to the left
        auto draw = [&](int n, uint32_t i0, int m, int64_t *dst, int step) {
            const uint32_t jb = (1u << (n - 1)) - 1u + i0;
            uint32_t k = (jb + 1) >> 1;
            if (jb & 1u) {
                if (i0 > 0)
                    dst[0] = carry[n];
                else if (C == 1 || n == 2)
                    dst[0] = carry[n - 1];   // the whole previous level has been drawn
                else
                    k = jb >> 1;             // drawn again: its other half comes later in the path
            }
#pragma unroll 1
            for (; k <= (jb + (uint32_t)m - 1u) >> 1; ++k) {
                int64_t z0, z1;
                st.fixed(k, z0, z1);
                const int a = (int)(2 * k - jb);
                if (a >= 0) dst[a * step] = z0;
                if (a + 1 < m)
                    dst[(a + 1) * step] = z1;
                else
                    carry[n] = z1;
            }
        };
        // levels n0+1..S-F: one midpoint each (taken through row q(1)), then the segment's
#pragma unroll 1
        for (int n = n0 + 1; n <= S; ++n) {
            const int l = n - Cn, h = NF >> max(l, 0);
            if (l <= 0) {
                draw(n, (uint32_t)c >> (1 - l), 1, &sm.q(1), 0);
                right = place(left, right, sm.q(1), n);
                sm.R[n * kThreads] = right;
            } else {
                draw(n, (uint32_t)c << (l - 1), 1 << (l - 1), &sm.q(h), 2 * h * kThreads);
            }
        }
        sm.q(NF) = right;
        for (int l = 1; l <= F; ++l) {
            const int h = NF >> l;
#pragma unroll 1
            for (int i = h; i < NF; i += 2 * h) sm.q(i) = place(sm.q(i - h), sm.q(i + h), sm.q(i), Cn + l);
        }
        // ---- the slices that begin here and, on the levels of the segment, inside it
        for (int d = 0; d < P.levels && d <= F; ++d) level(&sm.q(0), NF >> d, kThreads << d, d);
        if (P.levels > 1)
            for (int n = max(n0, 1); n < Cn; ++n) {
                sm.q(1) = sm.R[n * kThreads];
                level(&sm.q(0), 1, kThreads, S - n);
            }
    }
    bad |= (int32_t)ov < 0 || qm >= X.qlim;
    if (bad) {
        double w[SU_MAX_S + 1];
        fx_slow_path<RING>(P, st, w);
        for (int d = 0; d < P.levels; ++d) wout[d * wstride] = w[S - d];
        return;
    }
    for (int d = 0; d < P.levels; ++d)
        wout[d * wstride] = X.lv[d].ok ? fma((double)(1 << (S - d)), X.lv[d].res, acc[d].value(X.lv[d].e)) : wsum[d];
}

// ------------------------------------------------------------------ the kernel
// Shared memory: node tables | tail[S][M] pairs | head[S][hrow] | tanh nodes | rows[kFxRows][kThreads];
// the weights sw[levels][chunk] in the rows where one round needs no more,
// else after them.
__host__ __device__ inline bool fx_share_sw(const SamplerParams &P) {
    return P.rounds == 1 && P.levels <= kFxRows;
}

template <int RING, int KS>
__global__ void __launch_bounds__(kThreads, 4) sampler_fx_kernel(const __grid_constant__ SamplerParams P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int L = P.levels, chunk = kThreads * P.rounds;
    const bool per_sample = P.w_out != nullptr;
    fx::Tables *bm = reinterpret_cast<fx::Tables *>(smem_raw);
    size_t off = sizeof(fx::Tables);
    float2 *tail = reinterpret_cast<float2 *>(smem_raw + off);
    off += sizeof(float2) * (size_t)P.S * P.M;
    int64_t *head = reinterpret_cast<int64_t *>(smem_raw + off);
    off += sizeof(int64_t) * (size_t)P.S * P.fx.hrow;
    fx::TanhNode *th = reinterpret_cast<fx::TanhNode *>(smem_raw + off);
    if constexpr (RING == RING_TANH2) off += sizeof(fx::TanhNode) * (size_t)P.fx.nodes;
    int64_t *rows = reinterpret_cast<int64_t *>(smem_raw + off);
    double *sw = reinterpret_cast<double *>(rows + (fx_share_sw(P) ? 0 : kFxRows * kThreads));
    FxView sm;
    sm.th = th;
    sm.tail = tail;
    sm.head = head;
    sm.R = rows + tid;
    {
        const char *g = static_cast<const char *>(P.tables);
        const float *gt = reinterpret_cast<const float *>(g + P.fx.tail_off);
        const int64_t *gh = reinterpret_cast<const int64_t *>(g + P.fx.head_off);
        fx::tables_load(bm, tid, kThreads);
        if constexpr (RING == RING_TANH2) fx::tanh_load(th, P.fx.nodes, tid, kThreads);
        for (int i = tid; i < P.S * P.M; i += kThreads) tail[i] = make_float2(gt[i], gt[i]);
        for (int i = tid; i < P.S * P.fx.hrow; i += kThreads) head[i] = gh[i];
    }
    __syncthreads();

    const FixedView<(KS >= 0 ? KS : 0)> fv{};   // compiled shape: the tail's only

    Stream<double> st;
    st.key = make_uint2((uint32_t)P.seed, (uint32_t)(P.seed >> 32));
    st.inst = P.instance;
    st.bm = bm;
    st.zq = nullptr;
    for (int64_t item = P.item0 + blockIdx.x; item < P.n_items; item += gridDim.x) {
        const int64_t b = item / P.items_per_block;
        const int64_t r = item - b * P.items_per_block;
        const int64_t lo = b * P.n_mc / P.n_blocks;
        const int64_t hi = (b + 1) * P.n_mc / P.n_blocks;
        const int64_t start = lo + r * chunk;
        const int cnt = (int)max((int64_t)0, min((int64_t)chunk, hi - start));
        for (int rd = 0; rd < P.rounds; ++rd) {
            const int t = rd * kThreads + tid;
            if (t >= cnt) break;
            const uint64_t sample = (uint64_t)(P.sample0 + start + t);
            st.slo = (uint32_t)sample;
            st.shi = (uint32_t)(sample >> 32);
            double *wout = sw + t;
            if constexpr (KS >= 0)
                fx_path<RING>(P, fv, sm, st, wout, chunk);
            else
                fx_path<RING>(P, P, sm, st, wout, chunk);
            bool nonfinite = false;
            for (int d = 0; d < L; ++d) {
                const double w = wout[d * chunk];
                nonfinite |= isnan(w) || (isinf(w) && w > 0);
            }
            if (nonfinite) atomicOr(P.flags, 1);
            if (per_sample) {
                double *dst = P.w_out + (start + t) * (int64_t)P.S;
                for (int d = 0; d < L; ++d) dst[P.S - d - 1] = wout[d * chunk];
            }
        }
        if (per_sample) continue;
        __syncthreads();
        item_lse<double>(sw, L, chunk, cnt, P.partial, item, warp, lane);
        __syncthreads();
    }
}

}  // namespace
}  // namespace su
