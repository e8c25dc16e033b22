// The general potential's sampler with its monomial program split by the size of
// its entries (general_plan.cpp): per slice the potential's low derivatives and
// the few large entries in double, all derivatives and the whole program, with
// the large entries zero, in packed single precision.
//
// What bounds it: sampler_kernel<double, RING_GENERAL> spends about 1550 double
// operations a slice (p = 10: 585 entries, 155 monomials, 19 derivatives) on the
// FP64 pipe, 2 lanes a cycle on this part.  Here about 400 remain (FP64 pipe 69 %
// busy), most of them the derivatives that the large entries need; the packed program
// hides behind them.  Two features, p = 10, N = 64, 200 001 samples: 62.4 -> 24.7 ms.
//
// A level of a path whose single-precision entries are too large in sum, 2^-30 of
// max(1, |w|) (narrow features that the plan's moments missed, paths far out), is
// weighed again by the whole program in double: a few 2^-24 of the entries stay
// below what a double's rounding does to exp(w).
#include <cstdint>

#include "sampler_impl.cuh"

namespace su {
namespace {

constexpr int kGenSeg = 5;   // the path in segments of 2^5 slices
constexpr float kGenTail = 0x1p-30f;   // largest sum of the single-precision entries' magnitudes, of max(1, |w|)

// V^(j)(x) / j!, j = 0..J, of two slices.  (A feature's offset from x is taken in
// double: far from the origin a rounded x would be off by a part of the feature.)
__device__ __forceinline__ void taylor_pair(double xa, double xb, const GeneralDev *__restrict__ G, float2 (*U)[4], int m) {
    const int J = G->J;
    auto offset = [&](double c) { return make_float2(__double2float_rn(xa - c), __double2float_rn(xb - c)); };
    const float2 x = offset(0.0);
    for (int j = 0; j <= J; ++j) {
        float2 v = make_float2(0.f, 0.f);
        if (j <= G->deg)
            for (int i = G->deg; i >= j; --i) v = __ffma2_rn(v, x, make_float2(G->poly_tay[j][i], G->poly_tay[j][i]));
        U[j][m] = v;
    }
    for (int g = 0; g < G->ng; ++g) {
        const float beta = (float)G->gauss[g][1], A = (float)G->gauss[g][0];
        const float2 u = offset(G->gauss[g][2]);
        // g_n = (-sb)^n H_n(sb u) / n!: g_{n+1} = -2 beta (u g_n + g_{n-1}) / (n + 1)
        float2 p = make_float2(0.f, 0.f), q = make_float2(A * expf(-beta * u.x * u.x), A * expf(-beta * u.y * u.y));
        for (int n = 0; n <= J; ++n) {
            U[n][m] = __fadd2_rn(U[n][m], q);
            const float f = -2.0f * beta * G->invf[n + 1];
            const float2 r = __fmul2_rn(make_float2(f, f), __ffma2_rn(u, q, p));
            p = q;
            q = r;
        }
    }
    for (int s = 0; s < G->ns; ++s) {
        const float al = (float)G->sech[s][1];
        const float2 u = offset(G->sech[s][2]);
        float t[2], t1[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float w = al * (i ? u.y : u.x), em = expm1f(-2.0f * fabsf(w)), den = 2.0f + em;
            t[i] = copysignf(-em / den, w);               // tanh w
            t1[i] = 4.0f * (1.0f + em) / (den * den);     // sech^2 w
        }
        // Taylor coefficients a_n of tanh, as in general_derivatives
        float2 a[kGenMaxSym + 1];
        a[0] = make_float2(t[0], t[1]);
        a[1] = make_float2(t1[0], t1[1]);
        const float s0 = G->sech_tay[s][0];
        U[0][m] = __ffma2_rn(make_float2(s0, s0), a[1], U[0][m]);
        for (int n = 1; n <= J; ++n) {
            float2 acc = make_float2(0.f, 0.f);
            for (int k = 0; k < (n + 1) / 2; ++k) acc = __ffma2_rn(a[k], a[n - k], acc);
            acc = __fadd2_rn(acc, acc);
            if (!(n & 1)) acc = __ffma2_rn(a[n >> 1], a[n >> 1], acc);
            const float f = -G->invf[n + 1], sc = G->sech_tay[s][n];
            a[n + 1] = __fmul2_rn(acc, make_float2(f, f));
            U[n][m] = __ffma2_rn(make_float2(sc, sc), a[n + 1], U[n][m]);
        }
    }
    for (int q = 0; q < G->ne; ++q) {
        const float kap = (float)G->expo[q][1], E = (float)G->expo[q][0];
        const float2 u = offset(G->expo[q][2]);
        float2 e = make_float2(E * expf(-kap * u.x), E * expf(-kap * u.y));
        for (int n = 0; n <= J; ++n) {
            U[n][m] = __fadd2_rn(U[n][m], e);
            const float f = -kap * G->invf[n + 1];
            e = __fmul2_rn(e, make_float2(f, f));
        }
    }
}

// 2 BP slices between the points q[k0 stp ..]: the single-precision part of
// -eps W_p; adds to sum, and its nodes' magnitudes to mag (the roundings are of
// the entries: what cancels between them does not cancel there)
template <int BP>
__device__ __noinline__ void gen_single(const GeneralDev *__restrict__ G, const GeneralNode *__restrict__ nodes,
                                        const float *__restrict__ coef, const double *q, int k0, int stp, float &sum,
                                        float &mag) {
    float2 U[kGenMaxSym][4], stk[kGenMaxDepth + 1][BP], Y[BP], w[BP], m[BP];
#pragma unroll 1
    for (int i = 0; i < BP; ++i) {
        const double a = q[(k0 + 2 * i) * stp], b = q[(k0 + 2 * i + 1) * stp], c = q[(k0 + 2 * i + 2) * stp];
        taylor_pair(0.5 * (a + b), 0.5 * (b + c), G, U, i);
    }
#pragma unroll
    for (int i = 0; i < BP; ++i) {
        const double a = q[(k0 + 2 * i) * stp], b = q[(k0 + 2 * i + 1) * stp], c = q[(k0 + 2 * i + 2) * stp];
        const float2 vs = make_float2(__double2float_rn(b - a), __double2float_rn(c - b));
        Y[i] = __fmul2_rn(vs, vs);
        w[i] = m[i] = make_float2(0.f, 0.f);
    }
    const int nn = G->n_nodes;
#pragma unroll 1
    for (int t = 0; t < nn; ++t) {
        const GeneralNode nd = nodes[t];
        float2 mu[BP];
        if (t) {
#pragma unroll
            for (int i = 0; i < BP; ++i) {
                mu[i] = nd.depth > 1 ? __fmul2_rn(stk[nd.depth - 1][i], U[nd.sym][i]) : U[nd.sym][i];
                stk[nd.depth][i] = mu[i];
            }
        } else {
#pragma unroll
            for (int i = 0; i < BP; ++i) mu[i] = make_float2(1.f, 1.f);
        }
        const int cnt = nd.count;
        if (cnt) {
            const float *c = coef + nd.first;
            float2 h[BP];
            const float top = c[cnt - 1];
#pragma unroll
            for (int i = 0; i < BP; ++i) h[i] = make_float2(top, top);
#pragma unroll 2
            for (int e = cnt - 2; e >= 0; --e) {
                const float2 ce = make_float2(c[e], c[e]);
#pragma unroll
                for (int i = 0; i < BP; ++i) h[i] = __ffma2_rn(h[i], Y[i], ce);
            }
#pragma unroll
            for (int i = 0; i < BP; ++i) {
                const float2 x = __fmul2_rn(h[i], mu[i]);
                w[i] = __fadd2_rn(w[i], x);
                m[i].x += fabsf(x.x);
                m[i].y += fabsf(x.y);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < BP; ++i) {
        sum += w[i].x + w[i].y;
        mag += m[i].x + m[i].y;
    }
}

// Shared memory: sw[levels][chunk] | Box-Muller node tables | where staged:
// nodes, single-precision entries [S][M].
__global__ void __launch_bounds__(kThreads, 4) general_kernel(const __grid_constant__ SamplerParams P) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int L = P.levels, S = P.S, chunk = kThreads * P.rounds;
    const bool per_sample = P.w_out != nullptr;
    double *sw = reinterpret_cast<double *>(smem_raw);
    size_t off = per_sample ? 0 : sizeof(double) * (size_t)L * chunk;
    fx::Tables *bm = reinterpret_cast<fx::Tables *>(smem_raw + off);
    off += sizeof(fx::Tables);
    fx::tables_load(bm, tid, kThreads);
    const GeneralDev *G = P.general;
    const char *base = static_cast<const char *>(P.tables);
    const GeneralNode *nodes = G->nodes, *hnodes = reinterpret_cast<const GeneralNode *>(base + P.gs.hnodes);
    const float *tail = reinterpret_cast<const float *>(base + P.gs.tail);
    const double *hcoef = reinterpret_cast<const double *>(base + P.gs.hcoef);
    if (P.gs.staged) {
        GeneralNode *n = reinterpret_cast<GeneralNode *>(smem_raw + off);
        off += sizeof(GeneralNode) * (size_t)G->n_nodes;
        float *c = reinterpret_cast<float *>(smem_raw + off);
        for (int i = tid; i < G->n_nodes; i += kThreads) n[i] = nodes[i];
        for (int i = tid; i < S * P.M; i += kThreads) c[i] = tail[i];
        nodes = n;
        tail = c;
    }
    __syncthreads();
    Stream<double> st;
    st.key = make_uint2((uint32_t)P.seed, (uint32_t)(P.seed >> 32));
    st.inst = P.instance;
    st.bm = bm;
    st.zq = nullptr;
    const int F = min(S, kGenSeg), Cn = S - F, C = 1 << Cn, NF = 1 << F;
    double co[(1 << (SU_MAX_S - kGenSeg)) + 1], seg[(1 << kGenSeg) + 1];

    for (int64_t item = P.item0 + blockIdx.x; item < P.n_items; item += gridDim.x) {
        const int64_t b = item / P.items_per_block;
        const int64_t r = item - b * P.items_per_block;
        const int64_t lo = b * P.n_mc / P.n_blocks;
        const int64_t hi = (b + 1) * P.n_mc / P.n_blocks;
        const int64_t start = lo + r * chunk;
        const int cnt = (int)max((int64_t)0, min((int64_t)chunk, hi - start));
        for (int t0 = 0; t0 < cnt; t0 += kThreads) {
            // Pass 0: every lane its sample.  Then, one sample at a time by the whole warp, a
            // pair of slices a lane, the levels beyond the split's reach by the whole program,
            // summed in its order.  (By the sample's own lane that held a call of 30 001
            // samples up by a tenth: p = 12, N = 64, T = 1.)
            uint32_t todo = (1u << L) - 1u, far = 0;
            for (unsigned left = 1, pass = 0; left; ++pass) {
                const int t = t0 + (pass ? (tid & ~31) + __ffs(left) - 1 : tid);
                double w[SU_MAX_S];
                if (pass || t < cnt) {
                    const uint64_t sample = (uint64_t)(P.sample0 + start + t);
                    st.slo = (uint32_t)sample;
                    st.shi = (uint32_t)(sample >> 32);
                    uint32_t have = 0xffffffffu;
                    double z0 = 0, z1 = 0;
                    auto normal = [&](uint32_t g) {
                        if ((g >> 1) != have) {
                            st.pair(g >> 1, z0, z1);
                            have = g >> 1;
                        }
                        return (g & 1u) ? z1 : z0;
                    };
                    float tsum[SU_MAX_S], tmag[SU_MAX_S];
                    for (int d = 0; d < L; ++d) {
                        w[d] = 0;
                        tsum[d] = tmag[d] = 0;
                    }
                    auto slices = [&](int d, const double *q, int stp, int ns) {
                        if (!(todo >> d & 1u)) return;
                        const bool split = pass == 0 && P.gs.hn[d] > 0;
                        if (split) {
                            const float *c = tail + (size_t)d * P.M;
                            float s = 0, m = 0;
                            if (ns >= 8) {
#pragma unroll 1
                                for (int k = 0; k < ns; k += 8) gen_single<4>(G, nodes, c, q, k, stp, s, m);
                            } else {
#pragma unroll 1
                                for (int k = 0; k < ns; k += 2) gen_single<1>(G, nodes, c, q, k, stp, s, m);
                            }
                            tsum[d] += s;
                            tmag[d] += m;
                        }
                        const GeneralNode *nd = split ? hnodes + P.gs.h0[d] : nodes;
                        const int nn = split ? P.gs.hn[d] : G->n_nodes, J = split ? P.gs.hj[d] : G->J;
                        const double *c = split ? hcoef + P.gs.hc[d] : reinterpret_cast<const double *>(P.tables) + (size_t)d * P.M;
                        double sum = 0;   // of this segment (one running sum over the path rounds at its full size)
#pragma unroll 1
                        for (int k = pass ? 2 * lane : 0; k < ns; k += pass ? 64 : 2) {
                            const double2 v = slice_general<2>(q[k * stp], q[(k + 1) * stp], q[(k + 1) * stp], q[(k + 2) * stp],
                                                               c, G, nd, nn, J);
                            sum += v.x + v.y;
                        }
                        if (pass) {   // at most 32 pairs, in order
                            const double mine = sum;
                            sum = 0;
                            __syncwarp();
                            for (int k = 0; k < ns / 2; ++k) sum += __shfl_sync(0xffffffffu, mine, k);
                        }
                        w[d] += sum;
                    };
                    // coarse levels: the segment endpoints
                    co[0] = P.a;
                    co[C] = P.b;
                    for (int n = 1; n <= Cn; ++n) {
                        const int h = 1 << (Cn - n);
                        for (int i = 0; i < (1 << (n - 1)); ++i) {
                            const int x = (2 * i + 1) * h;
                            co[x] = fma(P.sigma[n], normal((1u << (n - 1)) - 1u + (uint32_t)i), 0.5 * (co[x - h] + co[x + h]));
                        }
                    }
#pragma unroll 1
                    for (int d = F; d < L; ++d) slices(d, co, 1 << (d - F), 1 << (S - d));
#pragma unroll 1
                    for (int sg = 0; sg < C; ++sg) {
                        seg[0] = co[sg];
                        seg[NF] = co[sg + 1];
                        for (int n = Cn + 1; n <= S; ++n) {
                            const int h = 1 << (S - n), m = 1 << (n - Cn - 1);
                            for (int i = 0; i < m; ++i) {
                                const int x = (2 * i + 1) * h;
                                seg[x] = fma(P.sigma[n], normal((1u << (n - 1)) - 1u + (uint32_t)(sg * m + i)), 0.5 * (seg[x - h] + seg[x + h]));
                            }
                        }
#pragma unroll 1
                        for (int d = 0; d < min(F, L); ++d) slices(d, seg, 1 << d, NF >> d);
                    }
                    if (pass == 0)
                        for (int d = 0; d < L; ++d)
                            if (P.gs.hn[d] > 0) {
                                w[d] += (double)tsum[d];
                                if (!(tmag[d] <= kGenTail * fmaxf(1.0f, fabsf(__double2float_rn(w[d]))))) far |= 1u << d;
                            }
                    if (pass == 0 || lane == 0) {
                        bool bad = false;
                        for (int d = 0; d < L; ++d)
                            if (pass ? todo >> d & 1u : !(far >> d & 1u)) {
                                bad |= isnan(w[d]) || (isinf(w[d]) && w[d] > 0);
                                if (per_sample)
                                    P.w_out[(start + t) * (int64_t)S + (S - d - 1)] = w[d];
                                else
                                    sw[(size_t)d * chunk + t] = w[d];
                            }
                        if (bad) atomicOr(P.flags, 1);
                    }
                }
                __syncwarp();
                left = pass ? left & (left - 1) : __ballot_sync(0xffffffffu, far != 0);
                if (left) todo = __shfl_sync(0xffffffffu, far, __ffs(left) - 1);
            }
        }
        if (per_sample) continue;
        __syncthreads();
        item_lse<double>(sw, L, chunk, cnt, P.partial, item, warp, lane);
        __syncthreads();
    }
}

}  // namespace

const void *general_entry() { return (const void *)general_kernel; }

size_t general_smem_bytes(const SamplerParams &P) {
    size_t off = (P.w_out ? 0 : sizeof(double) * (size_t)P.levels * kThreads * P.rounds) + sizeof(fx::Tables);
    if (P.gs.staged) off += sizeof(GeneralNode) * (size_t)P.gs.n_nodes + sizeof(float) * (size_t)P.S * P.M;
    return off;
}

}  // namespace su
