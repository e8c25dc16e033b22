#pragma once
// The proposal network on the 5th-generation tensor cores (sm_103a):
// tcgen05.mma with bfloat16 operands in shared memory and float accumulators
// in tensor memory, 128 rows (paths) at a time.
//
// x = (a, b, T, n/s, q_L, q_R) -> Linear(6,128) -> GELU -> Linear(128,128)
// -> GELU -> Linear(128,128) -> GELU -> Linear(128,2) = (shift, log-scale),
// GELU(v) = v (1 + erf(v/sqrt 2))/2.  Host weights: one float vector
// (W1[128][6], b1, W2[128][128], b2, W3[128][128], b3, W4[2][128], b4),
// matrices stored [out][in].
//
// Operand layout (A = activations [128 rows][K], B = weights [N rows][K],
// both K-major): core matrices of 8 rows x 16 bytes (8 bf16), stored
// contiguously; K-adjacent core matrices 128 bytes apart (the descriptor's
// leading byte offset), 8-row groups K/8 * 128 bytes apart (stride byte
// offset); no swizzle.  A CTA copies the weight blob (this layout, plus the
// float biases) once and keeps it resident.
//
// One layer = K/16 MMAs of M = 128, N = 128 (N = 16 for the output layer,
// rows 2..15 of W4 zero) issued by one thread into tensor-memory columns
// [0, 128) (outputs: [128, 144)), a commit to an mbarrier, and an epilogue
// in which warp w reads tensor-memory lanes 32 (w % 4) .. +31 (its rows) and
// a quarter of the columns of its quadrant's rows, adds the bias, applies GELU (erf
// by a polynomial, two values per packed multiply-add) and writes the bfloat16
// activations back into the A tile for the next layer.
//
// A tile belongs to a group of sixteen warps with its own accumulators, A tiles,
// named barrier and mbarrier; a CTA runs two groups on one copy of the weights, so
// that one group's epilogue fills the other's wait for its MMAs (1 000 003 paths of
// 64 slices through the network: 17.8 ms with one group, 13.8 with two of eight
// warps, 13.4 with two of sixteen).  Bound by the epilogue's multiply-adds (FMA
// pipes 54 % busy) and the four dependent layers of a tile; tensor cores 16 %.
#include <cuda_bf16.h>
#include <cstdint>

#include "erf_poly.h"

namespace su {
namespace mlp {

constexpr int kIn = 6, kHid = 128, kOut = 2;
constexpr int kParams = kHid * kIn + kHid + 2 * (kHid * kHid + kHid) + kOut * kHid + kOut;   // 34178
constexpr int kK1 = 16;        // layer-1 K: the 6 features, zero-padded
constexpr int kNOut = 16;      // output-layer N: 2 outputs, zero-padded
constexpr int kRows = 128;     // rows per tile = the MMA's M
constexpr int kGroups = 2;     // groups of a CTA
constexpr int kGroup = 512;    // threads of a group: four warps per tensor-memory lane quadrant
constexpr int kThreads = kGroups * kGroup;
constexpr int kColsPerWarp = kHid * 4 / (kGroup / 32);     // epilogue columns of a warp
constexpr int kTmemCols = 256; // a group's: [0, 128) hidden accumulator, [128, 144) outputs

// byte offset of element (r, k) of an operand with K columns
__host__ __device__ constexpr int cm_off(int r, int k, int K) {
    return (r >> 3) * (K / 8) * 128 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2;
}

// blob layout (the shared-memory image), byte offsets
constexpr int kOffW1 = 0;                                 // [128][16]
constexpr int kOffW2 = kOffW1 + kHid * kK1 * 2;           // [128][128]
constexpr int kOffW3 = kOffW2 + kHid * kHid * 2;          // [128][128]
constexpr int kOffW4 = kOffW3 + kHid * kHid * 2;          // [16][128]
constexpr int kOffB = kOffW4 + kNOut * kHid * 2;          // b1, b2, b3 [128], b4 [2] (+ pad), float
constexpr int kBlobBytes = kOffB + (3 * kHid + 8) * 4;    // 75296
static_assert(kBlobBytes % 16 == 0, "blob copies in 16-byte pieces");

// tile buffers (shared memory, byte sizes)
constexpr int kX0Bytes = kRows * kK1 * 2;
constexpr int kHBytes = kRows * kHid * 2;

#ifdef __CUDACC__
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// GELU of two values, v (1/2 + erf(v/sqrt 2)/2), with erf(v/sqrt 2) from the
// odd polynomial v Q(v^2) of erf_poly.h (v clamped to [-3 sqrt 2, 3 sqrt 2],
// error <= 1e-4, below the bfloat16 rounding the epilogue applies; the halves
// of its coefficients are exact) evaluated on the pair by packed multiply-adds
// (fma.rn.f32x2): one instruction for both values.
__device__ __forceinline__ float2 gelu2(float2 v) {
    const float2 x = make_float2(fminf(fmaxf(v.x, -kErfClamp), kErfClamp), fminf(fmaxf(v.y, -kErfClamp), kErfClamp));
    const float2 z = __fmul2_rn(x, x);
    float2 p = make_float2(0.5f * erf_poly(kErfTerms - 1), 0.5f * erf_poly(kErfTerms - 1));
#pragma unroll
    for (int k = kErfTerms - 2; k >= 0; --k) p = __ffma2_rn(p, z, make_float2(0.5f * erf_poly(k), 0.5f * erf_poly(k)));
    return __fmul2_rn(v, __ffma2_rn(x, p, make_float2(0.5f, 0.5f)));
}

// ---- tcgen05 plumbing
// shared-memory matrix descriptor: start address, leading (K) and stride
// (8-row) byte offsets, descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}

// instruction descriptor, kind::f16: float accumulator, bf16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24
__host__ __device__ constexpr uint32_t instr_desc(int m, int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

constexpr unsigned long long kWaitNs = 1000000000ull;   // a wait gives up after one second
constexpr int kWaitPolls = 1 << 28;                      // and after this many polls in any case

struct Tc {
    uint32_t tmem;     // tensor-memory base address (lane 0, first column)
    uint32_t mbar;     // shared address of the MMA-completion mbarrier
    uint32_t phase;    // parity of the next completion to wait for
    uint32_t ncols;    // allocated columns
};

// A group of a CTA: its threads, named barrier and tensor-core state (tmem and
// mbar its own)
struct Group {
    int tid;           // thread within the group
    uint32_t bar;      // named barrier
    Tc tc;
    // every thread of the group; false on all where any came with !ok
    __device__ __forceinline__ bool sync(bool ok) const {
        uint32_t all;
        asm volatile(
            "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.and.pred q, %2, %3, p;\nselp.u32 %0, 1, 0, q;\n}\n"
            : "=r"(all)
            : "r"((uint32_t)ok), "r"(bar), "n"(kGroup)
            : "memory");
        return all != 0;
    }
};

// All threads: initialisation of n mbarriers (thread 0), allocation of ncols
// tensor-memory columns (warp 0; a power of two >= 32).  slot and bar are
// shared-memory words of the CTA.
__device__ __forceinline__ Tc tc_begin(uint32_t *slot, uint64_t *bar, uint32_t ncols, int n = 1) {
    const int tid = threadIdx.x;
    if (tid == 0) {
        for (int k = 0; k < n; ++k) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar + k)));
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if ((tid >> 5) == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)),
                     "r"(ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    Tc t;
    t.tmem = *slot;
    t.mbar = smem_u32(bar);
    t.phase = 0;
    t.ncols = ncols;
    return t;
}

// The group of this thread, of a CTA of blockDim.x / kGroup groups (bar: one
// mbarrier each; the CTA's allocation is kTmemCols columns each)
__device__ __forceinline__ Group group_begin(uint32_t *slot, uint64_t *bar) {
    const int n = (int)blockDim.x / kGroup, g = (int)threadIdx.x / kGroup;
    Group r;
    r.tid = (int)threadIdx.x % kGroup;
    r.bar = 1u + (uint32_t)g;
    r.tc = tc_begin(slot, bar, (uint32_t)(n * kTmemCols), n);
    r.tc.tmem += (uint32_t)(g * kTmemCols);
    r.tc.mbar += (uint32_t)(g * 8);
    return r;
}

// All threads, after the last use: warp 0 frees the tensor memory.
__device__ __forceinline__ void tc_end(const Tc &t) {
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    if ((threadIdx.x >> 5) == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(t.tmem), "r"(t.ncols));
}

// All threads of the CTA, after its groups' last use
__device__ __forceinline__ void group_end(const Group &g) {
    Tc t = g.tc;
    t.tmem -= (threadIdx.x / kGroup) * kTmemCols;
    tc_end(t);
}

// One layer's MMAs, D[:, col..col+N) = A[128][K] B[N][K]^T, issued by the
// group's thread 0 after the other threads' shared-memory writes (fenced for the async
// proxy and synchronised by the caller), then committed to the mbarrier.
// withhold (fault injection): issue nothing, so the wait runs out.
__device__ __forceinline__ void tc_layer(const Group &g, uint32_t a, uint32_t b, int K, int N, uint32_t col,
                                         bool withhold = false) {
    const Tc &t = g.tc;
    if (g.tid == 0 && !withhold) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t sbo = (uint32_t)(K / 8) * 128;
        const uint32_t id = instr_desc(kRows, N);
        for (int ks = 0; ks < K / 16; ++ks) {
            const uint64_t ad = smem_desc(a + ks * 256, 128, sbo);
            const uint64_t bd = smem_desc(b + ks * 256, 128, sbo);
            asm volatile(
                "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(t.tmem + col),
                "l"(ad), "l"(bd), "r"(id), "r"((uint32_t)(ks > 0)));
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(t.mbar));
    }
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long v;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(v));
    return v;
}

// All threads: wait (bounded: one second of the global timer) for the last
// commit; false if it never came.
__device__ __forceinline__ bool tc_wait(Tc &t) {
    uint32_t done = 0;
    const unsigned long long t0 = global_ns();
    for (int it = 0; it < kWaitPolls && !done; ++it) {
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(t.mbar), "r"(t.phase));
        if (!done && (it & 255) == 255 && global_ns() - t0 > kWaitNs) break;
    }
    t.phase ^= 1u;
    asm volatile("tcgen05.fence::after_thread_sync;");
    return done != 0;
}

__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

__device__ __forceinline__ void tmem_ld32(uint32_t addr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
        "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;");
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&h);
}

// Epilogue of a hidden layer: bias + GELU of the accumulator, bfloat16, into
// the A tile H ([128][128], operand layout); fenced for the next MMA.
__device__ __forceinline__ void tc_store_gelu(const Group &g, const float *bias, unsigned char *H) {
    const int warp = g.tid >> 5, lane = g.tid & 31;
    const int row = 32 * (warp & 3) + lane;
    const int c0 = kColsPerWarp * (warp >> 2);
    const uint32_t base = g.tc.tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0;
    unsigned char *h = H + cm_off(row, c0, kHid);
#pragma unroll 1
    for (int cc = 0; cc < kColsPerWarp; cc += 32) {
        uint32_t v[32];
        tmem_ld32(base + (uint32_t)cc, v);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            // eight columns' biases (16-byte aligned: the blob's bias block is)
            const float4 b0 = *reinterpret_cast<const float4 *>(bias + c0 + cc + 8 * q);
            const float4 b1 = *reinterpret_cast<const float4 *>(bias + c0 + cc + 8 * q + 4);
            auto act = [&](int k, float x, float y) {
                const float2 u = make_float2(__uint_as_float(v[8 * q + k]), __uint_as_float(v[8 * q + k + 1]));
                const float2 a = gelu2(__fadd2_rn(u, make_float2(x, y)));
                return pack_bf16(a.x, a.y);
            };
            uint4 w;
            w.x = act(0, b0.x, b0.y);
            w.y = act(2, b0.z, b0.w);
            w.z = act(4, b1.x, b1.y);
            w.w = act(6, b1.z, b1.w);
            *reinterpret_cast<uint4 *>(h + cm_off(0, cc + 8 * q, kHid)) = w;
        }
    }
    asm volatile("fence.proxy.async.shared::cta;");
    asm volatile("tcgen05.fence::before_thread_sync;");
}

// The whole network on the group's 128-row tile.  X0: the features in operand
// layout ([128][16], columns 6..15 zero), written by the caller's threads; H: the
// hidden tile.  (sh, ls) = outputs of row tid on the group's first 128 threads.
// All threads of the group.  A thread whose MMA never completed clears its ok and
// goes on to the group's next barrier (a layer on the sums of an unfinished MMA
// computes what is thrown away); from there all return false, and the caller stops
// (after the last tile: sync(ok)).  withhold: fault injection (see tc_layer).
__device__ __forceinline__ bool tile_forward(Group &g, const unsigned char *blob, const unsigned char *X0,
                                             unsigned char *H, float &sh, float &ls, bool &ok, bool withhold = false) {
    const float *B = reinterpret_cast<const float *>(blob + kOffB);
    const uint32_t sb = smem_u32(blob), sx = smem_u32(X0), ah = smem_u32(H);
    asm volatile("fence.proxy.async.shared::cta;");
    if (!g.sync(ok)) return false;
    tc_layer(g, sx, sb + kOffW1, kK1, kHid, 0, withhold);
    ok = tc_wait(g.tc);
    tc_store_gelu(g, B, H);
    if (!g.sync(ok)) return false;
    tc_layer(g, ah, sb + kOffW2, kHid, kHid, 0);
    ok = tc_wait(g.tc);
    tc_store_gelu(g, B + kHid, H);
    if (!g.sync(ok)) return false;
    tc_layer(g, ah, sb + kOffW3, kHid, kHid, 0);
    ok = tc_wait(g.tc);
    tc_store_gelu(g, B + 2 * kHid, H);
    if (!g.sync(ok)) return false;
    tc_layer(g, ah, sb + kOffW4, kHid, kNOut, kHid);
    if (g.tid < kRows) {   // the other threads' next wait comes after a barrier that these reach later
        ok = tc_wait(g.tc);
        uint32_t r0, r1;
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];"
                     : "=r"(r0), "=r"(r1)
                     : "r"(g.tc.tmem + ((uint32_t)(g.tid & ~31) << 16) + (uint32_t)kHid));
        asm volatile("tcgen05.wait::ld.sync.aligned;");
        asm volatile("tcgen05.fence::before_thread_sync;");
        sh = __uint_as_float(r0) + B[3 * kHid];
        ls = __uint_as_float(r1) + B[3 * kHid + 1];
    } else {
        g.tc.phase ^= 1u;
    }
    return true;
}

// features of one row into the X0 tile (operand layout): columns 0..5, the
// zero padding of columns 6..7 in the same 16-byte chunk
__device__ __forceinline__ void store_features(unsigned char *X0, int row, __nv_bfloat16 f0, __nv_bfloat16 f1,
                                               __nv_bfloat16 f2, __nv_bfloat16 f3, __nv_bfloat16 f4,
                                               __nv_bfloat16 f5) {
    __nv_bfloat162 p0 = __halves2bfloat162(f0, f1), p1 = __halves2bfloat162(f2, f3), p2 = __halves2bfloat162(f4, f5);
    uint4 w;
    w.x = *reinterpret_cast<uint32_t *>(&p0);
    w.y = *reinterpret_cast<uint32_t *>(&p1);
    w.z = *reinterpret_cast<uint32_t *>(&p2);
    w.w = 0u;
    *reinterpret_cast<uint4 *>(X0 + cm_off(row, 0, kK1)) = w;
}
#endif

// host: float parameter vector -> device blob image (kBlobBytes)
void pack_blob(const float *theta, unsigned char *blob);

}  // namespace mlp
}  // namespace su
