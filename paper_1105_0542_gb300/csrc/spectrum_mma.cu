// The band matrix-block product of the eigensolver on the tensor cores
// (sm_103a), exact in integers: U and X are split into signed 8-bit digits, the
// digits' products are summed by tcgen05.mma (bfloat16 holds the digits, the
// float accumulator every sum, exactly), and the sums are put together in
// 64-bit integers (the scheme of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines", 2012).
//
// With U = 2^(ea - 55) sum_i d_i 2^(8 (6 - i)), i = 0..6, |d_i| <= 128 (ea: the
// exponent of max |U|), and column c of X likewise (its own exponent), the sums
//   D_g = sum_k sum_{i + j = g} d_i[k] x_j[k],  g = 0..6
// over K = 128 columns of U stay below 7 * 128 * 2^14 < 2^24: exact.  Dropped: the
// digits' rounding, 2^-57 of the largest element, and the pairs i + j >= 7, 2^-55.
// Against the product in double, whose rounding is that of its running sums, the
// root mean square error on bands of 36 diagonals and more is between 0.01 (smooth
// columns) and 0.9 (random ones) times as large; narrower bands stay in double
// (band_spectrum).  With six digits it was 1.4 to 240 times as large.
//
// Layout: U as row tiles of 128 rows, each over its band in chunks of 32 columns;
// a chunk is seven digit planes of 128 x 32 bfloat16 in the operand layout of
// mlp.cuh (core matrices of 8 rows x 16 bytes, no swizzle), 56 KB contiguous, so
// that one bulk copy brings it to shared memory.  X's digits lie in chunks of
// 32 rows of U's columns: rows j * 16 + c (digit j of column c), 7 KB.
// Per 16 columns of U and digit i one MMA of M = 128, N = 16 (7 - i): A = plane
// i, B = digits 0..6-i of the 16 columns, D at tensor-memory column 16 i, so that
// pairs of equal i + j share an accumulator.
//
// What bounds it: reading the digit planes, 14 bytes an element once per
// product (617 MB at n = 16 385, w = 1297, in 98 us: 6.3 TB/s of a copy's 6.8; tensor
// cores 21 % busy; 0.106 ms with the digits of X, 0.090 with six digits); the
// product in double took 1161 us at 96 % of the FP64 pipe.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include <cooperative_groups.h>

#include "mlp.cuh"
#include "sampler.h"

namespace su {
namespace {

constexpr int kDig = 7;                        // digits of 8 bits
constexpr int kBits = 8 * kDig - 1;            // of an element, of its largest one's power of two
constexpr int kCols = 16;                      // columns of X per pass
constexpr int kChunk = 32;                     // columns of U per stage
constexpr int kWindow = 128 / kChunk;          // stages whose sums share an accumulator buffer
constexpr int kPlane = 128 * kChunk * 2;       // bytes of one digit plane of a chunk
constexpr int kABytes = kDig * kPlane;         // 56 KB
constexpr int kBBytes = kDig * kCols * kChunk * 2;   // 7 KB
constexpr int kStages = 3;
constexpr int kMmaThreads = 320;               // eight epilogue warps, one that issues, one that copies
constexpr int kMmaSmem = kStages * (kABytes + kBBytes) + 128;

__device__ __forceinline__ int exponent_of(unsigned long long bits) {   // v = m 2^e, m in [1/2, 1)
    return (int)((bits >> 52) & 0x7FF) - 1022;
}
__device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }

// the digits of q (|q| <= 2^kBits), most significant first
__device__ __forceinline__ void digits(long long q, int (&d)[kDig]) {
#pragma unroll
    for (int i = kDig - 1; i > 0; --i) {
        d[i] = (int)(signed char)(q & 255);
        q = (q - d[i]) >> 8;
    }
    d[0] = (int)q;
}

__device__ __forceinline__ uint32_t pair_bf16(int lo, int hi) { return mlp::pack_bf16((float)lo, (float)hi); }

// dmax[k] = the largest |D[k pitch + i]| (as bits), one thread block per diagonal
__global__ void __launch_bounds__(256) diag_max_kernel(const double *__restrict__ D, int64_t pitch, int n,
                                                       unsigned long long *dmax) {
    const double *d = D + (int64_t)blockIdx.x * pitch;
    unsigned long long m = 0;
    for (int i = threadIdx.x; i < n; i += 256) m = max(m, (unsigned long long)__double_as_longlong(d[i]) & 0x7FFFFFFFFFFFFFFFULL);
    for (int o = 16; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    __shared__ unsigned long long red[8];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < 8; ++k) m = max(m, red[k]);
        dmax[blockIdx.x] = m;
    }
}

// first column (a multiple of kChunk) of row tile rt
__device__ __forceinline__ int tile_col0(int rt, int w) { return max(0, rt * 128 - w) / kChunk * kChunk; }

// the digit planes of U from its upper band; one thread block per (chunk, row tile)
__global__ void __launch_bounds__(256) digits_a_kernel(const double *__restrict__ D, int64_t pitch, int n, int w,
                                                       int nk, int ea, unsigned char *__restrict__ A) {
    const int rt = blockIdx.y, kc = blockIdx.x;
    const double scale = pow2(kBits - ea);
    unsigned char *out = A + ((int64_t)rt * nk + kc) * kABytes;
    for (int g = threadIdx.x; g < 128 * (kChunk / 8); g += 256) {
        const int lr = g & 127, kg = g >> 7, r = rt * 128 + lr;
        const int c0 = tile_col0(rt, w) + kc * kChunk + kg * 8;
        int d[8][kDig];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int c = c0 + j, k = abs(r - c);
            const double v = (r < n && c < n && k <= w) ? D[(int64_t)k * pitch + min(r, c)] : 0.0;
            digits(__double2ll_rn(v * scale), d[j]);
        }
#pragma unroll
        for (int i = 0; i < kDig; ++i) {
            uint4 q;
            q.x = pair_bf16(d[0][i], d[1][i]);
            q.y = pair_bf16(d[2][i], d[3][i]);
            q.z = pair_bf16(d[4][i], d[5][i]);
            q.w = pair_bf16(d[6][i], d[7][i]);
            *reinterpret_cast<uint4 *>(out + i * kPlane + mlp::cm_off(lr, kg * 8, kChunk)) = q;
        }
    }
}

// max |X[:, c]| of the columns col0..col0+15
__global__ void __launch_bounds__(256) col_max_kernel(const double *__restrict__ X, int n, int B, int col0,
                                                      unsigned long long *xmax) {
    const int c = threadIdx.x & 15;
    unsigned long long m = 0;
    if (col0 + c < B)
        for (int64_t i = (int64_t)blockIdx.x * 16 + (threadIdx.x >> 4); i < n; i += (int64_t)gridDim.x * 16)
            m = max(m, (unsigned long long)__double_as_longlong(X[i * B + col0 + c]) & 0x7FFFFFFFFFFFFFFFULL);
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 16));
    if ((threadIdx.x & 31) < 16 && m) atomicMax(xmax + c, m);
}

// the digits of X's columns; one thread per (8 rows, column); also clears the
// maxima of the product to come
__global__ void __launch_bounds__(256) digits_x_kernel(const double *__restrict__ X, int n, int B, int col0,
                                                       const unsigned long long *__restrict__ xmax,
                                                       unsigned char *__restrict__ Xd, int rows8,
                                                       unsigned long long *__restrict__ clear) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < kCols) clear[t] = 0;
    const int c = t & 15, g = t >> 4;
    if (g >= rows8) return;
    const unsigned long long m = xmax[c];
    const double scale = m ? pow2(kBits - exponent_of(m)) : 0.0;
    int d[8][kDig];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int r = g * 8 + j;
        const double v = (r < n && col0 + c < B) ? X[(int64_t)r * B + col0 + c] : 0.0;
        digits(__double2ll_rn(v * scale), d[j]);
    }
    unsigned char *out = Xd + (int64_t)(g / (kChunk / 8)) * kBBytes;
#pragma unroll
    for (int i = 0; i < kDig; ++i) {
        uint4 q;
        q.x = pair_bf16(d[0][i], d[1][i]);
        q.y = pair_bf16(d[2][i], d[3][i]);
        q.z = pair_bf16(d[4][i], d[5][i]);
        q.w = pair_bf16(d[6][i], d[7][i]);
        *reinterpret_cast<uint4 *>(out + mlp::cm_off(i * kCols + c, g % (kChunk / 8) * 8, kChunk)) = q;
    }
}

// ---- barriers (bounded waits: one second, then false)
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {
    const unsigned long long t0 = mlp::global_ns();
    for (int it = 0; it < mlp::kWaitPolls; ++it) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if ((it & 255) == 255 && mlp::global_ns() - t0 > mlp::kWaitNs) return false;
    }
    return false;
}
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void bar_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar));
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t addr, int (&v)[8]) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = __float2int_rn(__uint_as_float(r[j]));
}

// Ynew = alpha U X + beta Ycur + gamma Yprev for 16 columns of X, one row tile per
// CTA.  Warp 9 copies chunks (three stages), warp 8 issues their MMAs into one of two
// accumulator buffers per 128 columns of U, warps 0..7 read a finished buffer (two
// warps per lane quadrant, eight columns each) into 64-bit sums while the other
// fills.
struct MmaArgs {
    const unsigned char *A, *Xd;
    int ea;                            // exponent of max |U|
    const unsigned long long *xmax;
    unsigned long long *ymax;          // max |Ynew[:, c]| (null: not wanted)
    const double *Ycur, *Yprev;
    double *Ynew;
    double alpha, beta, gamma;
    int n, w, nk, B, col0;
    int *status;
};

__global__ void __launch_bounds__(kMmaThreads, 1) band_mma_kernel(const MmaArgs P) {
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ __align__(8) uint64_t bars[2 * kStages + 4];
    __shared__ uint32_t slot;
    __shared__ int dead;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rt = blockIdx.x;
    const uint32_t full = mlp::smem_u32(bars), empty = full + 8 * kStages, wfull = empty + 8 * kStages, wfree = wfull + 16;
    const uint32_t base = (mlp::smem_u32(sm) + 127u) & ~127u;
    const int c0 = tile_col0(rt, P.w);
    const int cend = min(P.n, rt * 128 + 128 + P.w);
    const int nk = (cend - c0 + kChunk - 1) / kChunk, nw = (nk + kWindow - 1) / kWindow;
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            bar_init(full + 8 * s, 1);
            bar_init(empty + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            bar_init(wfull + 8 * b, 1);
            bar_init(wfree + 8 * b, 8);
        }
        asm volatile("fence.mbarrier_init.release.cluster;");
        dead = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(mlp::smem_u32(&slot)));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = slot;
    bool ok = true;
    long long hi[8], lo[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) hi[c] = lo[c] = 0;

    if (warp == 9) {
        if (lane == 0) {
            int k = 0;
            for (; k < nk; ++k) {
                const int s = k % kStages;
                if (k >= kStages && !bar_wait(empty + 8 * s, (uint32_t)(k / kStages - 1) & 1u)) {
                    ok = false;
                    break;
                }
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full + 8 * s),
                             "r"((uint32_t)(kABytes + kBBytes))
                             : "memory");
                const uint32_t dst = base + s * (kABytes + kBBytes);
                bulk_copy(dst, P.A + ((int64_t)rt * P.nk + k) * kABytes, kABytes, full + 8 * s);
                bulk_copy(dst + kABytes, P.Xd + (int64_t)(c0 / kChunk + k) * kBBytes, kBBytes, full + 8 * s);
            }
            // nothing of this CTA's is in flight when it ends
            for (int q = max(0, k - kStages); q < k; ++q) {
                bar_wait(full + 8 * (q % kStages), (uint32_t)(q / kStages) & 1u);
                bar_wait(empty + 8 * (q % kStages), (uint32_t)(q / kStages) & 1u);
            }
        }
        __syncwarp();
    } else if (warp == 8) {
        if (lane == 0) {
            for (int k = 0; k < nk && ok; ++k) {
                const int s = k % kStages, win = k / kWindow, buf = win & 1;
                if (k % kWindow == 0 && win >= 2 && !bar_wait(wfree + 8 * buf, (uint32_t)(win / 2 - 1) & 1u)) {
                    ok = false;
                    break;
                }
                if (!bar_wait(full + 8 * s, (uint32_t)(k / kStages) & 1u)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;");
                const uint32_t a = base + s * (kABytes + kBBytes), b = a + kABytes;
                for (int ks = 0; ks < kChunk / 16; ++ks)
                    for (int i = 0; i < kDig; ++i) {
                        const uint64_t ad = mlp::smem_desc(a + i * kPlane + ks * 256, 128, kChunk / 8 * 128);
                        const uint64_t bd = mlp::smem_desc(b + ks * 256, 128, kChunk / 8 * 128);
                        const uint32_t id = mlp::instr_desc(128, kCols * (kDig - i));
                        asm volatile(
                            "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem + buf * 128 + i * kCols),
                            "l"(ad), "l"(bd), "r"(id), "r"((uint32_t)(k % kWindow || ks || i)));
                    }
                bar_commit(empty + 8 * s);
                if (k % kWindow == kWindow - 1 || k == nk - 1) bar_commit(wfull + 8 * buf);
            }
        }
        __syncwarp();
    } else {
        const uint32_t at = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(8 * (warp >> 2));
        for (int win = 0; win < nw; ++win) {
            const int buf = win & 1;
            if (!__all_sync(0xffffffffu, bar_wait(wfull + 8 * buf, (uint32_t)(win / 2) & 1u))) {
                ok = false;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
            for (int g = 0; g < kDig; ++g) {
                int v[8];
                tmem_ld8(at + buf * 128 + g * kCols, v);
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    if (g < 4)
                        hi[c] += (long long)v[c] << (8 * (3 - g));
                    else
                        lo[c] += (long long)v[c] << (8 * (6 - g));
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(wfree + 8 * buf) : "memory");
        }
    }
    if (!ok) dead = 1;
    __syncthreads();
    if (warp < 8 && !dead) {
        const int r = rt * 128 + 32 * (warp & 3) + lane;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int cc = 8 * (warp >> 2) + c, col = P.col0 + cc;
            double y = 0.0;
            const unsigned long long xm = P.xmax[cc];
            if (r < P.n && col < P.B) {
                // 2^48 (hi 2^24 + lo) in units of both scales
                y = xm ? fma((double)hi[c], 0x1p24, (double)lo[c]) * pow2(P.ea - 31) * pow2(exponent_of(xm) - 31) : 0.0;
                const int64_t at = (int64_t)r * P.B + col;
                y *= P.alpha;
                if (P.beta != 0.0) y = fma(P.beta, P.Ycur[at], y);
                if (P.gamma != 0.0) y = fma(P.gamma, P.Yprev[at], y);
                P.Ynew[at] = y;
            }
            if (P.ymax) {
                unsigned long long m = (unsigned long long)__double_as_longlong(y) & 0x7FFFFFFFFFFFFFFFULL;
                for (int o = 16; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
                if (lane == 0 && m) atomicMax(P.ymax + cc, m);
            }
        }
    }
    if (dead && tid == 0) atomicOr(P.status, 1);
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem));
}

// One Lanczos step on one vector after wv = U v: alpha = v.w, w -= alpha v +
// beta vp, beta' = |w|; then vp <- v, v <- w / beta'.  One cluster of eight CTAs,
// each an eighth of the vector, sums exchanged through distributed shared memory
// in a fixed order (one CTA took 66 us at n = 16 385: about sixteen double
// operations per element on one SM's FP64 pipe, a division among them).
constexpr int kLanCtas = 8, kLanThreads = 512;
__global__ void __cluster_dims__(kLanCtas, 1, 1) __launch_bounds__(kLanThreads)
    lanczos_kernel(int n, int j, double *__restrict__ v, double *__restrict__ vp, double *__restrict__ wv, double *al,
                   double *be) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ double red[kLanThreads / 32], total[2];
    auto sum = [&](double x, int slot) {
        for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
        __syncthreads();
        if (threadIdx.x == 0) {
            double y = 0;
            for (int k = 0; k < kLanThreads / 32; ++k) y += red[k];
            total[slot] = y;
        }
        cluster.sync();
        double r = 0;
        for (int c = 0; c < kLanCtas; ++c) r += *cluster.map_shared_rank(&total[slot], c);
        return r;
    };
    const int step = kLanCtas * kLanThreads, i0 = blockIdx.x * kLanThreads + threadIdx.x;
    const double beta = j ? be[j - 1] : 0.0;
    double a = 0;
#pragma unroll 4
    for (int i = i0; i < n; i += step) a = fma(v[i], wv[i], a);
    a = sum(a, 0);
    double b2 = 0;
#pragma unroll 4
    for (int i = i0; i < n; i += step) {
        const double x = wv[i] - (a * v[i] + beta * (j ? vp[i] : 0.0));
        wv[i] = x;
        b2 = fma(x, x, b2);
    }
    const double b = sqrt(sum(b2, 1)), inv = b > 0 ? 1.0 / b : 0.0;
#pragma unroll 4
    for (int i = i0; i < n; i += step) {
        vp[i] = v[i];
        v[i] = wv[i] * inv;
    }
    if (i0 == 0) {
        al[j] = a;
        be[j] = b;
    }
    cluster.sync();   // no CTA's shared memory goes before the others have read it
}

}  // namespace

static int64_t band_mma_tiles(int n) { return ((int64_t)n + 127) / 128; }
static int band_mma_chunks(int n, int w) { return (std::min(n, 2 * w + 128 + kChunk) + kChunk - 1) / kChunk; }
int64_t band_mma_bytes_a(int n, int w) { return band_mma_tiles(n) * band_mma_chunks(n, w) * (int64_t)kABytes; }
// (the last tile's last chunk may start up to a chunk past n)
int64_t band_mma_bytes_x(int n) { return ((int64_t)n / kChunk + 2) * kBBytes; }

int band_mma_bits() { return kBits; }
int band_exponent(unsigned long long bits) { return (int)((bits >> 52) & 0x7FF) - 1022; }

cudaError_t launch_diag_max(const double *D, int64_t pitch, int n, int w, unsigned long long *dmax, cudaStream_t st) {
    cudaGetLastError();
    diag_max_kernel<<<(unsigned)(w + 1), 256, 0, st>>>(D, pitch, n, dmax);
    return cudaGetLastError();
}

cudaError_t launch_band_digits(const BandMma &M, const double *D, int64_t pitch, cudaStream_t st) {
    cudaGetLastError();
    const int nk = band_mma_chunks(M.n, M.w);
    digits_a_kernel<<<dim3((unsigned)nk, (unsigned)band_mma_tiles(M.n)), 256, 0, st>>>(D, pitch, M.n, M.w, nk, M.ea, M.A);
    return cudaGetLastError();
}

cudaError_t launch_col_max(const double *X, int n, int B, int col0, unsigned long long *xmax, cudaStream_t st) {
    cudaGetLastError();
    cudaError_t e = cudaMemsetAsync(xmax, 0, kCols * sizeof *xmax, st);
    if (e != cudaSuccess) return e;
    col_max_kernel<<<(unsigned)std::min(128, (n + 15) / 16), 256, 0, st>>>(X, n, B, col0, xmax);
    return cudaGetLastError();
}

cudaError_t launch_band_mma(const BandMma &M, const double *X, const unsigned long long *xmax, unsigned long long *ymax,
                            int B, int col0, const double *Ycur, const double *Yprev, double *Ynew, double alpha,
                            double beta, double gamma, cudaStream_t st) {
    cudaGetLastError();
    cudaError_t e = cudaFuncSetAttribute(band_mma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMmaSmem);
    if (e != cudaSuccess) return e;
    const int rows8 = (int)(band_mma_bytes_x(M.n) / kBBytes * (kChunk / 8));
    digits_x_kernel<<<(unsigned)((rows8 * 16 + 255) / 256), 256, 0, st>>>(X, M.n, B, col0, xmax, M.Xd, rows8,
                                                                        ymax ? ymax : M.scratch_max);
    MmaArgs a{M.A, M.Xd, M.ea, xmax, ymax, Ycur, Yprev, Ynew, alpha, beta, gamma, M.n, M.w, band_mma_chunks(M.n, M.w),
              B, col0, M.status};
    band_mma_kernel<<<(unsigned)band_mma_tiles(M.n), kMmaThreads, kMmaSmem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_lanczos(int n, int j, double *v, double *vp, double *wv, double *al, double *be, cudaStream_t st) {
    cudaGetLastError();
    lanczos_kernel<<<kLanCtas, kLanThreads, 0, st>>>(n, j, v, vp, wv, al, be);
    return cudaGetLastError();
}

}  // namespace su
