// Training of the proposal network on the tensor cores (sm_103a).
//
// The objective (weighted maximum likelihood of midpoints of plain-sampler
// paths): L = sum_r rw_r [ls_r + (u_r - shift_r)^2 e^{-2 ls_r} / 2] / sum_r rw_r,
// u_r = the midpoint's standardized offset (q - mu)/sigma_n.  One step on R
// rows (rows = the N-1 midpoints of each path of a minibatch):
//
//   forward   pre_l = H_{l-1} W_l^T + b_l, H_l = GELU(pre_l), Y = H_3 W_4^T + b_4
//   backward  dY = dL/dY; dH_3 = dY W_4; dPre_l = dH_l * GELU'(pre_l);
//             dW_l = dPre_l^T H_{l-1}; db_l = column sums of dPre_l;
//             dH_{l-1} = dPre_l W_l
//   update    Adam on the float master weights.
//
// step_kernel does all of forward and backward for tiles of 128 rows: weights,
// activations and gradients of a tile stay in shared memory as bfloat16 operands;
// products, and the sums of dW_l and db_l over the CTA's tiles, in tensor memory
// (float); GELU' of layers 2 and 3 in registers.  update_kernel adds the CTAs'
// weight gradients in a fixed order and does the update.  No transposed copies: an
// operand stored with its columns contiguous is read K-major or MN-major by the
// descriptor (dW_l = dPre_l^T H_{l-1} contracts over the rows).  The bias gradients
// ride on the constant seventh feature: dPre_l^T X0 has db_l in its column 6.
//
// What bounds it: the chain of ten dependent phases per tile (an MMA of under half
// a microsecond, a barrier, an elementwise epilogue whose polynomials and exps take
// most of the time): 12.6 us a tile, two tiles an SM at 512 paths x 63 rows, 9 us
// for the launch, the weights and the gradients; tensor cores 10 % busy.  That step
// takes 34 + 7 us; as one GEMM per product with transposed copies through global
// memory it was 22 launches and 263 us.  The CTAs' gradients by atomic adds, 128
// bytes apart in a warp, cost 12 us more than stores with the sum in update_kernel;
// keeping pre-activations of all three layers in registers spilled.  Minibatch draws
// (binary searches, 13 us a step) are made ahead for many steps at once.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "mlp.cuh"
#include "philox.cuh"
#include "train.h"

namespace su {
namespace train {
namespace {

using mlp::kHid;
using mlp::kIn;
using mlp::kK1;
using mlp::kOut;
using mlp::kRows;
using mlp::kX0Bytes;
using mlp::kHBytes;

constexpr int kThreads = 512, kColsPerWarp = kHid * 4 / (kThreads / 32);   // one tile: 16 warps, 32 columns each

// parameter offsets in the flat vector
constexpr int kPW1 = 0, kPb1 = kPW1 + kHid * kIn, kPW2 = kPb1 + kHid, kPb2 = kPW2 + kHid * kHid,
              kPW3 = kPb2 + kHid, kPb3 = kPW3 + kHid * kHid, kPW4 = kPb3 + kHid, kPb4 = kPW4 + kOut * kHid;
static_assert(kPb4 + kOut == mlp::kParams, "parameter layout");

// a CTA's gradients: W_2, W_3 as [column / 4][unit][column % 4], W_1 with its bias
// and a zero behind it the same way, b_2, b_3, W_4, b_4 with two zeros
constexpr int kQW2 = 0, kQW3 = kHid * kHid, kQW1 = 2 * kHid * kHid, kQB2 = kQW1 + 8 * kHid, kQB3 = kQB2 + kHid,
              kQW4 = kQB3 + kHid, kQb4 = kQW4 + kOut * kHid, kPart = kQb4 + 4;
static_assert(kPart % 4 == 0 && kQb4 % 4 == 0, "16-byte pieces");

// parameter index of gradient e, -1 for padding
__device__ __forceinline__ int param_of(int e) {
    if (e < kQB2) {
        const int s = e < kQW3 ? kPW2 : e < kQW1 ? kPW3 : kPW1;
        const int i = e < kQW3 ? e : e < kQW1 ? e - kQW3 : e - kQW1;
        const int c = i / (4 * kHid) * 4 + (i & 3), o = i / 4 % kHid;
        if (s != kPW1) return s + o * kHid + c;
        return c < kIn ? kPW1 + o * kIn + c : c == kIn ? kPb1 + o : -1;
    }
    if (e < kQB3) return kPb2 + e - kQB2;
    if (e < kQW4) return kPb3 + e - kQB3;
    if (e < kQb4) return kPW4 + e - kQW4;
    return e < kQb4 + kOut ? kPb4 + e - kQb4 : -1;
}

// tensor-memory columns
constexpr uint32_t kTD = 0, kTW2 = 128, kTW3 = 256, kTW1 = 384, kTB2 = 400, kTB3 = 416, kTW4 = 432, kTY = 448;

// shared memory: weight blob | X0 | dY | H1 | H2 | H3 | G
constexpr int kOffX0 = mlp::kBlobBytes, kOffDY = kOffX0 + kX0Bytes, kOffH = (kOffDY + kX0Bytes + 127) / 128 * 128;
constexpr int kStepSmem = kOffH + 4 * kHBytes;

// GELU(v) = v (1 + erf(v / sqrt 2)) / 2 of two values and its derivative, from one
// polynomial of erf (that of mlp::gelu2)
__device__ __forceinline__ float2 one_plus_erf(float2 v) {
    const float c = mlp::kErfClamp;
    const float2 x = make_float2(fminf(fmaxf(v.x, -c), c), fminf(fmaxf(v.y, -c), c));
    const float2 z = __fmul2_rn(x, x);
    float2 p = make_float2(mlp::erf_poly(mlp::kErfTerms - 1), mlp::erf_poly(mlp::kErfTerms - 1));
#pragma unroll
    for (int k = mlp::kErfTerms - 2; k >= 0; --k) p = __ffma2_rn(p, z, make_float2(mlp::erf_poly(k), mlp::erf_poly(k)));
    return __ffma2_rn(x, p, make_float2(1.0f, 1.0f));
}
__device__ __forceinline__ float2 gelu(float2 v) {
    return __fmul2_rn(__fmul2_rn(v, make_float2(0.5f, 0.5f)), one_plus_erf(v));
}
__device__ __forceinline__ float2 gelu_both(float2 v, float2 &grad) {
    const float2 half = make_float2(0.5f, 0.5f), o = one_plus_erf(v);
    const float2 e = make_float2(__expf(-0.5f * v.x * v.x), __expf(-0.5f * v.y * v.y));
    const float2 g = __fmul2_rn(__fmul2_rn(v, make_float2(0.39894228040143268f, 0.39894228040143268f)), e);
    grad = __ffma2_rn(half, o, g);
    return __fmul2_rn(__fmul2_rn(v, half), o);
}

__device__ __forceinline__ float2 unpack_bf16(uint32_t w) {
    return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

// MMA D[:, col..col+N) (+)= A B over K = 16 ks: descriptors with their byte
// offsets (lbo, sbo) and the advance per 16 of K; am, bm: the operand is MN-major
struct Operand {
    uint32_t addr, lbo, sbo, step;
    uint32_t mn;
};
__device__ __forceinline__ Operand k_major(uint32_t addr, int cols) { return {addr, 128u, (uint32_t)cols * 16u, 256u, 0u}; }
// the same bytes read with the columns as M or N and the rows as K: eight
// contiguous columns a core-matrix row, 8-column blocks 128 bytes apart, 8-row
// blocks cols * 16 bytes apart
__device__ __forceinline__ Operand mn_major(uint32_t addr, int cols) { return {addr, (uint32_t)cols * 16u, 128u, (uint32_t)cols * 32u, 1u}; }

__device__ __forceinline__ void mma(uint32_t tmem, Operand a, Operand b, int N, int ksteps, bool add) {
    const uint32_t id = mlp::instr_desc(kRows, N) | (a.mn << 15) | (b.mn << 16);
    for (int k = 0; k < ksteps; ++k) {
        const uint64_t ad = mlp::smem_desc(a.addr + k * a.step, a.lbo, a.sbo);
        const uint64_t bd = mlp::smem_desc(b.addr + k * b.step, b.lbo, b.sbo);
        asm volatile(
            "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
            "l"(ad), "l"(bd), "r"(id), "r"((uint32_t)(add || k > 0)));
    }
}
__device__ __forceinline__ void commit(const mlp::Tc &t) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(t.mbar));
}

// before the next MMA reads what this thread wrote or read
__device__ __forceinline__ void handover() {
    asm volatile("fence.proxy.async.shared::cta;");
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
}

struct StepArgs {
    const unsigned char *blob;      // weights as operands (mlp.cuh), biases
    // rows: midpoint j of path ids[r / (N-1)] of paths [n][N+1], or features F [n][6] with u and rw
    const float *paths;
    const int *ids;                 // of step *step: ids + *step * nb
    const int *step;
    int ids_steps;                  // steps that ids holds (a ring)
    int nb, np1, S;
    float a, b, T;
    const float *sig;
    const float *F, *u, *rw;
    int R;                          // rows
    double inv_norm;
    float *part;                    // [CTA][kPart]: the CTA's gradients, in the order of param_of
    double *loss;                   // [CTA]
    int *status;
};

__global__ void __launch_bounds__(kThreads, 1) step_kernel(const StepArgs P) {
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ uint32_t slot;
    __shared__ __align__(8) uint64_t bar;
    __shared__ double s_loss[4];
    __shared__ float s_db4[4][2];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char *X0 = sm + kOffX0, *DY = sm + kOffDY, *H = sm + kOffH, *Gb = H + 3 * kHBytes;
    {
        const uint4 *s = reinterpret_cast<const uint4 *>(P.blob);
        uint4 *d = reinterpret_cast<uint4 *>(sm);
        constexpr int kPieces = (mlp::kBlobBytes / 16 + kThreads - 1) / kThreads;
        uint4 w[kPieces];
#pragma unroll
        for (int i = 0; i < kPieces; ++i)
            if (tid + i * kThreads < mlp::kBlobBytes / 16) w[i] = s[tid + i * kThreads];
#pragma unroll
        for (int i = 0; i < kPieces; ++i)
            if (tid + i * kThreads < mlp::kBlobBytes / 16) d[tid + i * kThreads] = w[i];
        for (int i = tid; i < 2 * kX0Bytes / 16; i += kThreads) reinterpret_cast<uint4 *>(X0)[i] = make_uint4(0, 0, 0, 0);
    }
    const float *B = reinterpret_cast<const float *>(sm + mlp::kOffB);
    mlp::Tc tc = mlp::tc_begin(&slot, &bar, 512);
    const uint32_t ab = mlp::smem_u32(sm), aX = ab + kOffX0, aY = ab + kOffDY, aH = ab + kOffH, aG = aH + 3 * kHBytes;
    const Operand w1 = k_major(ab + mlp::kOffW1, kK1), w2 = k_major(ab + mlp::kOffW2, kHid), w3 = k_major(ab + mlp::kOffW3, kHid),
                  w4 = k_major(ab + mlp::kOffW4, kHid);
    const Operand w2t = mn_major(ab + mlp::kOffW2, kHid), w3t = mn_major(ab + mlp::kOffW3, kHid),
                  w4t = mn_major(ab + mlp::kOffW4, kHid);
    const int row = 32 * (warp & 3) + lane, c0 = kColsPerWarp * (warp >> 2);
    const uint32_t quad = (uint32_t)(32 * (warp & 3)) << 16;
    const int *ids = P.ids ? P.ids + (int64_t)(*P.step % P.ids_steps) * P.nb : nullptr;
    bool ok = true;
    double loss = 0;
    float db0 = 0, db1 = 0;
    bool first = true;

    // a hidden layer: bias + GELU; act(c, x) is the GELU of columns c0 + c, c0 + c + 1
    auto forward = [&](const float *bias, unsigned char *Ho, auto act) {
#pragma unroll
        for (int cc = 0; cc < kColsPerWarp; cc += 16) {
            float v[16];
            mlp::tmem_ld16(tc.tmem + kTD + quad + (uint32_t)(c0 + cc), v);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uint32_t w[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int c = cc + 8 * q + 2 * k;
                    const float2 bb = *reinterpret_cast<const float2 *>(bias + c0 + c);
                    const float2 x = __fadd2_rn(make_float2(v[8 * q + 2 * k], v[8 * q + 2 * k + 1]), bb);
                    const float2 g = act(c, x);
                    w[k] = mlp::pack_bf16(g.x, g.y);
                }
                *reinterpret_cast<uint4 *>(Ho + mlp::cm_off(row, c0 + cc + 8 * q, kHid)) = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
        handover();
    };
    // dPre = dH * GELU'(pre), grad(c) the GELU' of columns c0 + c, c0 + c + 1
    auto backward = [&](unsigned char *Go, auto grad) {
#pragma unroll
        for (int cc = 0; cc < kColsPerWarp; cc += 16) {
            float v[16];
            mlp::tmem_ld16(tc.tmem + kTD + quad + (uint32_t)(c0 + cc), v);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uint32_t w[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int c = cc + 8 * q + 2 * k;
                    const float2 g = __fmul2_rn(make_float2(v[8 * q + 2 * k], v[8 * q + 2 * k + 1]), grad(c));
                    w[k] = mlp::pack_bf16(g.x, g.y);
                }
                *reinterpret_cast<uint4 *>(Go + mlp::cm_off(row, c0 + cc + 8 * q, kHid)) = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
        handover();
    };
    auto arrived = [&] { return __syncthreads_and(mlp::tc_wait(tc) ? 1 : 0) != 0; };

    const int tiles = (P.R + kRows - 1) / kRows;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int r = tile * kRows + tid;
        float u = 0, rw = 0;
        if (tid < kRows) {
            float f[kIn] = {0, 0, 0, 0, 0, 0};
            if (r < P.R) {
                if (P.F) {
#pragma unroll
                    for (int c = 0; c < kIn; ++c) f[c] = P.F[(size_t)r * kIn + c];
                    u = P.u[r];
                    rw = P.rw[r];
                } else {
                    const int N = P.np1 - 1, pb = r / (N - 1), j = r - pb * (N - 1);
                    const int n = 32 - __clz(j + 1);        // level: 2^(n-1) <= j + 1 < 2^n
                    const int i = j - ((1 << (n - 1)) - 1), h = N >> n, k = (2 * i + 1) * h;
                    const float *q = P.paths + (size_t)ids[pb] * P.np1;
                    const float qL = q[k - h], qR = q[k + h];
                    f[0] = P.a;
                    f[1] = P.b;
                    f[2] = P.T;
                    f[3] = (float)n / (float)P.S;
                    f[4] = qL;
                    f[5] = qR;
                    u = (q[k] - 0.5f * (qL + qR)) / P.sig[n];
                    rw = 1.0f;
                }
            }
            uint4 w;
            w.x = mlp::pack_bf16(f[0], f[1]);
            w.y = mlp::pack_bf16(f[2], f[3]);
            w.z = mlp::pack_bf16(f[4], f[5]);
            w.w = mlp::pack_bf16(1.0f, 0.0f);               // the constant behind the bias gradients (W1 has a zero there)
            *reinterpret_cast<uint4 *>(X0 + mlp::cm_off(tid, 0, kK1)) = w;
        }
        handover();
        float2 g2[16], g3[16];   // GELU' of layers 2 and 3; layer 1's come from its six products a unit, made again
        // ---- forward
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            mma(tc.tmem + kTD, k_major(aX, kK1), w1, kHid, 1, false);
            commit(tc);
        }
        if (!(ok = arrived())) break;
        forward(B, H, [](int, float2 x) { return gelu(x); });
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            mma(tc.tmem + kTD, k_major(aH, kHid), w2, kHid, 8, false);
            commit(tc);
        }
        if (!(ok = arrived())) break;
        forward(B + kHid, H + kHBytes, [&](int c, float2 x) { return gelu_both(x, g2[c / 2]); });
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            mma(tc.tmem + kTD, k_major(aH + kHBytes, kHid), w3, kHid, 8, false);
            commit(tc);
        }
        if (!(ok = arrived())) break;
        forward(B + 2 * kHid, H + 2 * kHBytes, [&](int c, float2 x) { return gelu_both(x, g3[c / 2]); });
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            mma(tc.tmem + kTY, k_major(aH + 2 * kHBytes, kHid), w4, mlp::kNOut, 8, false);
            commit(tc);
        }
        if (!(ok = arrived())) break;
        // ---- loss and dL/dY (row r of the tile: thread r)
        if (warp < 4) {
            uint32_t y0, y1;
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];"
                         : "=r"(y0), "=r"(y1)
                         : "r"(tc.tmem + kTY + quad));
            asm volatile("tcgen05.wait::ld.sync.aligned;");
            const float sh = __uint_as_float(y0) + B[3 * kHid], ls = __uint_as_float(y1) + B[3 * kHid + 1];
            const float d = u - sh, e2 = __expf(-2.f * ls);
            __nv_bfloat16 h0 = __float2bfloat16_rn(0.f), h1 = h0;
            if (r < P.R) {
                loss += (double)rw * ((double)ls + 0.5 * (double)d * d * e2) * P.inv_norm;
                h0 = __float2bfloat16_rn((float)(-(double)d * e2 * rw * P.inv_norm));
                h1 = __float2bfloat16_rn((float)((1.0 - (double)d * d * e2) * rw * P.inv_norm));
            }
            db0 += __bfloat162float(h0);
            db1 += __bfloat162float(h1);
            const __nv_bfloat162 hh = __halves2bfloat162(h0, h1);
            *reinterpret_cast<uint32_t *>(DY + mlp::cm_off(tid, 0, kK1)) = *reinterpret_cast<const uint32_t *>(&hh);
        }
        handover();
        // ---- backward: dPre_3 into G, dPre_2 into H3's place, dPre_1 into G; each
        // layer's weight gradient behind the product that the next epilogue waits for
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            mma(tc.tmem + kTD, k_major(aY, kK1), w4t, kHid, 1, false);
            mma(tc.tmem + kTW4, mn_major(aH + 2 * kHBytes, kHid), mn_major(aY, kK1), mlp::kNOut, 8, !first);
            commit(tc);
        }
        if (!(ok = arrived())) break;
        backward(Gb, [&](int c) { return g3[c / 2]; });
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            mma(tc.tmem + kTD, k_major(aG, kHid), w3t, kHid, 8, false);
            commit(tc);
            mma(tc.tmem + kTW3, mn_major(aG, kHid), mn_major(aH + kHBytes, kHid), kHid, 8, !first);
            mma(tc.tmem + kTB3, mn_major(aG, kHid), mn_major(aX, kK1), kK1, 8, !first);
        }
        if (!(ok = arrived())) break;
        backward(H + 2 * kHBytes, [&](int c) { return g2[c / 2]; });
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            mma(tc.tmem + kTD, k_major(aH + 2 * kHBytes, kHid), w2t, kHid, 8, false);
            commit(tc);
            mma(tc.tmem + kTW2, mn_major(aH + 2 * kHBytes, kHid), mn_major(aH, kHid), kHid, 8, !first);
            mma(tc.tmem + kTB2, mn_major(aH + 2 * kHBytes, kHid), mn_major(aX, kK1), kK1, 8, !first);
        }
        if (!(ok = arrived())) break;
        {
            const uint4 xr = *reinterpret_cast<const uint4 *>(X0 + mlp::cm_off(row, 0, kK1));
            const float2 x01 = unpack_bf16(xr.x), x23 = unpack_bf16(xr.y), x45 = unpack_bf16(xr.z);
            backward(Gb, [&](int c) {
                float2 p = *reinterpret_cast<const float2 *>(B + c0 + c);
                const uint4 wa = *reinterpret_cast<const uint4 *>(sm + mlp::kOffW1 + mlp::cm_off(c0 + c, 0, kK1));
                const uint4 wb = *reinterpret_cast<const uint4 *>(sm + mlp::kOffW1 + mlp::cm_off(c0 + c + 1, 0, kK1));
                auto dot = [&](uint32_t ua, uint32_t ub, float2 x) {
                    const float2 a = unpack_bf16(ua), b = unpack_bf16(ub);
                    p = __ffma2_rn(make_float2(a.x, b.x), make_float2(x.x, x.x), p);
                    p = __ffma2_rn(make_float2(a.y, b.y), make_float2(x.y, x.y), p);
                };
                dot(wa.x, wb.x, x01);
                dot(wa.y, wb.y, x23);
                dot(wa.z, wb.z, x45);
                float2 g;
                gelu_both(p, g);
                return g;
            });
        }
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            mma(tc.tmem + kTW1, mn_major(aG, kHid), mn_major(aX, kK1), kK1, 8, !first);
            commit(tc);
        }
        if (!(ok = arrived())) break;   // all of the tile's operands are free
        first = false;
    }
    // ---- the CTA's gradients and loss: lane = output unit of dW_l (input unit of
    // dW_4^T), four columns a store, neighbouring units next to each other
    if (ok) {
        float *g = P.part + (size_t)blockIdx.x * kPart;
#pragma unroll 1
        for (int l = 0; l < 2; ++l) {
            float4 *d = reinterpret_cast<float4 *>(g + (l ? kQW3 : kQW2)) + row;
#pragma unroll
            for (int cc = 0; cc < kColsPerWarp; cc += 16) {
                float v[16];
                mlp::tmem_ld16(tc.tmem + (l ? kTW3 : kTW2) + quad + (uint32_t)(c0 + cc), v);
#pragma unroll
                for (int k = 0; k < 16; k += 4)
                    d[(c0 + cc + k) / 4 * kHid] = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
            }
        }
        float v[16];
        if (warp < 4) {
            mlp::tmem_ld16(tc.tmem + kTW1 + quad, v);
            float4 *d = reinterpret_cast<float4 *>(g + kQW1) + row;
            d[0] = make_float4(v[0], v[1], v[2], v[3]);
            d[kHid] = make_float4(v[4], v[5], v[6], 0.f);
        } else if (warp < 8) {
            mlp::tmem_ld16(tc.tmem + kTB2 + quad, v);
            g[kQB2 + row] = v[kIn];
        } else if (warp < 12) {
            mlp::tmem_ld16(tc.tmem + kTB3 + quad, v);
            g[kQB3 + row] = v[kIn];
        } else {
            mlp::tmem_ld16(tc.tmem + kTW4 + quad, v);
            g[kQW4 + row] = v[0];
            g[kQW4 + kHid + row] = v[1];
        }
        if (warp < 4) {
            for (int o = 16; o; o >>= 1) {
                loss += __shfl_xor_sync(0xffffffffu, loss, o);
                db0 += __shfl_xor_sync(0xffffffffu, db0, o);
                db1 += __shfl_xor_sync(0xffffffffu, db1, o);
            }
            if (lane == 0) {
                s_loss[warp] = loss;
                s_db4[warp][0] = db0;
                s_db4[warp][1] = db1;
            }
        }
        __syncthreads();
        if (tid == 0) {
            P.loss[blockIdx.x] = (s_loss[0] + s_loss[1]) + (s_loss[2] + s_loss[3]);
            float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
            d.x = (s_db4[0][0] + s_db4[1][0]) + (s_db4[2][0] + s_db4[3][0]);
            d.y = (s_db4[0][1] + s_db4[1][1]) + (s_db4[2][1] + s_db4[3][1]);
            *reinterpret_cast<float4 *>(g + kQb4) = d;
        }
    }
    if (!ok && tid == 0) atomicOr(P.status, 1);
    mlp::tc_end(tc);
}

// where parameter k lies in the operand blob: byte offset, or -1 for a bias (kept
// as a float at `bias`)
__device__ __forceinline__ int blob_at(int k, int &bias) {
    bias = -1;
    if (k < kPb1) return mlp::kOffW1 + mlp::cm_off(k / kIn, k % kIn, kK1);
    if (k < kPW2) { bias = k - kPb1; return -1; }
    if (k < kPb2) return mlp::kOffW2 + mlp::cm_off((k - kPW2) / kHid, (k - kPW2) % kHid, kHid);
    if (k < kPW3) { bias = kHid + k - kPb2; return -1; }
    if (k < kPb3) return mlp::kOffW3 + mlp::cm_off((k - kPW3) / kHid, (k - kPW3) % kHid, kHid);
    if (k < kPW4) { bias = 2 * kHid + k - kPb3; return -1; }
    if (k < kPb4) return mlp::kOffW4 + mlp::cm_off((k - kPW4) / kHid, (k - kPW4) % kHid, kHid);
    bias = 3 * kHid + k - kPb4;
    return -1;
}
__device__ __forceinline__ void put_blob(unsigned char *blob, int k, float v) {
    int bias;
    const int at = blob_at(k, bias);
    if (at >= 0)
        *reinterpret_cast<__nv_bfloat16 *>(blob + at) = __float2bfloat16_rn(v);
    else
        reinterpret_cast<float *>(blob + mlp::kOffB)[bias] = v;
}

__global__ void pack_kernel(const float *__restrict__ th, unsigned char *blob) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < mlp::kParams) put_blob(blob, k, th[k]);
}

// The gradient, summed over the step kernel's CTAs in a fixed order; then (adam)
// one Adam step with t = *step + 1, the new weights as operands, the loss recorded
// and the counter advanced by the last thread block, or (else) gradient and loss
// written.  A block has 64 gradients, 16 threads for each four of them; one read of
// the CTAs' 17 MB (126 of them) from L2 bounds it.
constexpr int kUpThreads = 256, kUpSlices = 16;
struct UpArgs {
    const float *part;
    const double *loss;
    int parts;
    float *th, *m, *v, *grad;
    unsigned char *blob;
    float lr, b1, b2, eps;
    int *step, *done;
    double *losses;
};
template <bool adam>
__global__ void __launch_bounds__(kUpThreads) update_kernel(const UpArgs P) {
    __shared__ float4 sg[kUpSlices][kUpThreads / kUpSlices];
    constexpr int kGroups = kUpThreads / kUpSlices;
    const int tid = threadIdx.x, gi = tid % kGroups, sl = tid / kGroups, grp = blockIdx.x * kGroups + gi;
    const int s = adam ? *P.step : 0;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    if (grp < kPart / 4) {
        const float4 *p = reinterpret_cast<const float4 *>(P.part) + grp;
#pragma unroll 4
        for (int c = sl; c < P.parts; c += kUpSlices) {
            const float4 x = p[(size_t)c * (kPart / 4)];
            a.x += x.x;
            a.y += x.y;
            a.z += x.z;
            a.w += x.w;
        }
    }
    sg[sl][gi] = a;
    __syncthreads();
    const int e = blockIdx.x * 4 * kGroups + tid;
    if (tid < 4 * kGroups && e < kPart) {
        float gk = 0.f;
#pragma unroll
        for (int q = 0; q < kUpSlices; ++q) gk += reinterpret_cast<const float *>(sg[q])[tid];
        const int k = param_of(e);
        if (k >= 0) {
            if (adam) {
                const float t = (float)(s + 1);
                const float c1 = 1.f - powf(P.b1, t), c2 = 1.f - powf(P.b2, t);
                const float mk = P.b1 * P.m[k] + (1.f - P.b1) * gk;
                const float vk = P.b2 * P.v[k] + (1.f - P.b2) * gk * gk;
                P.m[k] = mk;
                P.v[k] = vk;
                const float x = P.th[k] - P.lr * (mk / c1) / (sqrtf(vk / c2) + P.eps);
                P.th[k] = x;
                put_blob(P.blob, k, x);
            } else {
                P.grad[k] = gk;
            }
        }
    }
    if (blockIdx.x == 0 && tid >= kUpThreads - 32) {
        double l = 0;
        for (int c = tid & 31; c < P.parts; c += 32) l += P.loss[c];
        for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if ((tid & 31) == 0) P.losses[s] = l;
    }
    if (adam) {
        __syncthreads();
        if (tid == 0) {
            __threadfence();
            if (atomicAdd(P.done, 1) == (int)gridDim.x - 1) {   // every block has read the counter
                *P.done = 0;
                *P.step = s + 1;
            }
        }
    }
}

// Minibatch path ids of the steps step0.. step0 + n_steps - 1: draw k of a step is
// the 53-bit uniform u of Philox call (step, k, 0x7261696E, 0) under the key (seed
// lo, seed hi), and the id is the first index whose cumulative weight exceeds u *
// total (a draw in proportion to the weights).
__global__ void sample_ids_kernel(const double *__restrict__ cdf, int64_t n, double total, uint2 key, int step0,
                                  int n_steps, int nb, int *ids) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)n_steps * nb) return;
    const int s = (int)(t / nb), k = (int)(t - (int64_t)s * nb);
    const uint4 w = philox4x32_10(make_uint4((uint32_t)(step0 + s), (uint32_t)k, 0x7261696Eu, 0u), key);
    const double u = ((double)(((uint64_t)w.x << 21) | (w.y >> 11)) + 0.5) * 0x1p-53;
    const double x = u * total;
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (cdf[mid] > x)
            hi = mid;
        else
            lo = mid + 1;
    }
    ids[t] = (int)(lo < n ? lo : n - 1);
}

// level S of every path's weights
__global__ void top_weights_kernel(const double *__restrict__ w, int64_t n, int S, double *out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = w[i * S + S - 1];
}

}  // namespace

// ------------------------------------------------------------------ host

Workspace::~Workspace() {
    if (base) cudaFree(base);
}

cudaError_t Workspace::make(int rows) {
    cudaError_t e = cudaFuncSetAttribute(step_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kStepSmem);
    int dev = 0, sms = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // as few CTAs as keep the longest run of tiles: each leaves 137 KB of gradients
    const int tiles = std::max(1, (rows + kRows - 1) / kRows), per = (tiles + sms - 1) / sms;
    ctas = (tiles + per - 1) / per;
    const size_t flat = ((size_t)mlp::kParams * 4 + 255) / 256 * 256, blob_bytes = ((size_t)mlp::kBlobBytes + 255) / 256 * 256;
    const size_t zeroed = 4 * flat + blob_bytes + 256, sums = ((size_t)ctas * 8 + 255) / 256 * 256;
    e = cudaMalloc(&base, zeroed + sums + (size_t)ctas * kPart * 4);
    if (e != cudaSuccess) {
        base = nullptr;
        return e;
    }
    unsigned char *p = static_cast<unsigned char *>(base);
    theta = (float *)p;
    grad = (float *)(p + flat);
    m = (float *)(p + 2 * flat);
    v = (float *)(p + 3 * flat);
    blob = p + 4 * flat;
    loss = (double *)(p + 4 * flat + blob_bytes);
    step = (int *)(loss + 1);
    done = step + 1;
    status = step + 2;
    loss_part = (double *)(p + zeroed);
    part = (float *)(p + zeroed + sums);
    return cudaMemset(base, 0, zeroed);
}

cudaError_t pack(Workspace &ws, cudaStream_t st) {
    cudaGetLastError();
    pack_kernel<<<(mlp::kParams + 255) / 256, 256, 0, st>>>(ws.theta, ws.blob);
    return cudaGetLastError();
}

static cudaError_t launch_step(StepArgs a, const Workspace &ws, cudaStream_t st) {
    a.blob = ws.blob;
    a.step = ws.step;
    a.part = ws.part;
    a.loss = ws.loss_part;
    a.status = ws.status;
    cudaGetLastError();
    step_kernel<<<ws.ctas, kThreads, kStepSmem, st>>>(a);
    return cudaGetLastError();
}

static UpArgs update_args(const Workspace &ws) {
    UpArgs u{};
    u.part = ws.part;
    u.loss = ws.loss_part;
    u.parts = ws.ctas;
    u.th = ws.theta;
    u.m = ws.m;
    u.v = ws.v;
    u.grad = ws.grad;
    u.blob = ws.blob;
    u.step = ws.step;
    u.done = ws.done;
    u.losses = ws.loss;
    return u;
}
constexpr int kUpBlocks = (kPart + 4 * (kUpThreads / kUpSlices) - 1) / (4 * (kUpThreads / kUpSlices));

cudaError_t loss_grad(Workspace &ws, const float *F, const float *u, const float *rw, int n, double inv_norm,
                      cudaStream_t st) {
    StepArgs a{};
    a.F = F;
    a.u = u;
    a.rw = rw;
    a.R = n;
    a.inv_norm = inv_norm;
    const cudaError_t e = launch_step(a, ws, st);
    if (e != cudaSuccess) return e;
    update_kernel<false><<<kUpBlocks, kUpThreads, 0, st>>>(update_args(ws));
    return cudaGetLastError();
}

cudaError_t path_step(Workspace &ws, const float *paths, int np1, const int *ids, int ids_steps, int nb, float a, float b,
                      float T, int S, const float *sig, cudaStream_t st) {
    StepArgs s{};
    s.paths = paths;
    s.ids = ids;
    s.ids_steps = ids_steps;
    s.nb = nb;
    s.np1 = np1;
    s.S = S;
    s.a = a;
    s.b = b;
    s.T = T;
    s.sig = sig;
    s.R = nb * (np1 - 2);
    s.inv_norm = 1.0 / s.R;
    return launch_step(s, ws, st);
}

cudaError_t sample_ids(const double *cdf, int64_t n, double total, uint64_t seed, int step0, int n_steps, int nb,
                       int *ids, cudaStream_t st) {
    cudaGetLastError();
    const int64_t k = (int64_t)n_steps * nb;
    sample_ids_kernel<<<(unsigned)((k + 127) / 128), 128, 0, st>>>(cdf, n, total, make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)),
                                                                 step0, n_steps, nb, ids);
    return cudaGetLastError();
}

cudaError_t top_weights(const double *w, int64_t n, int S, double *out, cudaStream_t st) {
    cudaGetLastError();
    top_weights_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(w, n, S, out);
    return cudaGetLastError();
}

cudaError_t adam_step(Workspace &ws, float lr, double *losses, cudaStream_t st) {
    cudaGetLastError();
    UpArgs u = update_args(ws);
    u.lr = lr;
    u.b1 = 0.9f;
    u.b2 = 0.999f;
    u.eps = 1e-8f;
    u.losses = losses;
    update_kernel<true><<<kUpBlocks, kUpThreads, 0, st>>>(u);
    return cudaGetLastError();
}

}  // namespace train
}  // namespace su
