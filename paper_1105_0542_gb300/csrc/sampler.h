// Internal interface between the host API and the device kernels.
#pragma once

#include <cstdint>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/speedup.h"
#include "generator.h"

namespace su {

constexpr int kThreads = 128;   // threads per CTA of the sampler: one path per thread
constexpr int kMaxFine = 5;     // depth of the register-resident bisection subtree

// Everything the sampler needs, passed by value (it lives in the constant bank).
// General potential (RING_GENERAL): the device image of the monomial program
// and of the potential's families (built by the host from GeneralEffective
// and GeneralPotential, in device memory).
constexpr int kGenMaxSym = 2 * kGenMaxP - 1;   // V_0..V_{2p-2}
constexpr int kGenMaxDepth = 16;               // deepest monomial (6 at p = 12, 9 at p = 18; checked by the host)

struct GeneralNode {
    unsigned char depth, sym;                  // depth in the trie, symbol j of V_j
    unsigned short count;                      // entries of this monomial
    int first;                                 // its first entry
};

struct GeneralDev {
    int J, K, n_nodes, n_entries, ng, ns, ne;
    const GeneralNode *nodes;                  // depth-first; node 0 = the constant monomial;
                                               // a node's entries are vs^0, vs^2, .. in order
    double poly_der[kGenMaxSym][9];            // V^(j) polynomial part: sum_i poly_der[j][i] x^(i-j)
    double gauss[4][4];                        // A, beta, c, sqrt(beta)
    double sech[4][3];                         // B, alpha, d
    double sech_scale[4][kGenMaxSym];          // B alpha^n (n+1)!
    double expo[4][3];                         // E, kappa, x0
    double inv[kGenMaxSym + 1];                // 1 / n
    // single precision, derivatives over j!
    int deg;                                   // degree of the polynomial part
    float poly_tay[9][9];                      // a_i C(i, j)
    float sech_tay[4][kGenMaxSym];             // B alpha^n (n+1)
    float invf[kGenMaxSym + 2];
};

// The fixed-point sampler's plan (sampler_fx.cuh; built by fx_plan).  Path
// points are integers in units of q_unit; row d of the arrays is level n = S - d.
constexpr int kFxCols = 8;
struct FxLevel {
    int ok;                   // evaluated in fixed point, else in double
    int nc, h[kFxCols];       // columns with integer entries, and how many each (the others in single precision)
    int ky;                   // vs is shifted left by ky before it is squared
    int vlim;                 // |high word of vs| stays below this
    int e;                    // weights in units of 2^-e
    double res;               // what rounding to a unit takes from the constant entry, per slice
};
struct FxParams {
    int on;
    int qlim;                 // |high word of q| stays below this
    int hrow;                 // room for integer entries per level
    int ah, al, nodes;        // RING_TANH2: limbs of us -> alpha us / 2 in node steps, nodes in reach
    int sgh[SU_MAX_S + 1], sgl[SU_MAX_S + 1], shl[SU_MAX_S + 1];   // sigma_n: limbs and left shift of the product
    int64_t qa, qb;           // endpoints
    double q_unit;
    FxLevel lv[SU_MAX_S];
    int64_t head_off, tail_off;   // from the tables: [S][hrow] int64, [S][M] float
};

// The split general program (general.cu; built by general_split): byte offsets
// from the tables, and per level (row d) the double part's nodes, entries and
// highest derivative (hn = 0: the whole program in double).
struct GeneralSplit {
    int on, staged, n_nodes;
    int64_t tail, hnodes, hcoef;
    int hn[SU_MAX_S], h0[SU_MAX_S], hc[SU_MAX_S], hj[SU_MAX_S];
};

struct SamplerParams {
    // path: q_0 = a, q_N = b, N = 2^S, bisection widths sigma[n] (n = 1..S)
    double a, b;
    double sigma[SU_MAX_S + 1];
    int S;
    int F;                    // fine subtree depth, min(S, kMaxFine)
    int levels;               // sampled levels: S with the hierarchy, else 1
    // width-factor reweighting (Sec. 4.1 literal width): w_n += n_mid(n) lwf + hcoef * sum z^2
    int wf_on;
    double lwf, hcoef;
    // effective potential tables: row d (level n = S - d), M entries each
    int ring, ncol, M;
    int len[SU_MAX_P];
    int tab_global;           // 1: the level tables are read from global memory (too large to stage)
    int generic;              // 1: never the compiled-shape sampler (su_options.kernel = 1)
    double alpha;
    const void *tables;       // device, levels * M elements of the kernel's precision
    // Philox stream
    uint64_t seed;
    uint32_t instance;
    // work decomposition: items = (block b, chunk r), chunk = kThreads * rounds samples
    int64_t n_mc, sample0;
    int64_t n_blocks;
    int64_t items_per_block;
    int64_t n_items;          // items [item0, n_items) are this launch's (block ranges)
    int64_t item0;
    int rounds;
    // outputs
    double *partial;          // device: per item and level, (M, S, Q, n)
    double *w_out;            // device: per-sample mode when non-null, [sample][S]
    float *q_out;             // device: per-sample mode, single precision only: path points [sample][N+1] (or null)
    int *flags;               // device: bit 0 = non-finite weight seen
    const GeneralDev *general;  // device: RING_GENERAL only
    GeneralSplit gs;            // RING_GENERAL: the split program where gs.on
    FxParams fx;                // double precision: the fixed-point sampler where fx.on
};

// The split of the general program (rows of entries for levels n = S..1, the
// first `levels` of them): fills gs but its offsets, and the images that belong
// there -- the single-precision entries [S][M] (times the factorials that the
// kernel's derivatives are short of), the double parts' nodes and entries.
// False (gs.on = 0) where no level has a short enough double part.  Host work.
struct GeneralImages {
    std::vector<float> tail;
    std::vector<GeneralNode> hnodes;
    std::vector<double> hcoef;
};
bool general_split(const GeneralEffective &G, const GeneralPotential &V, double a, double b, double T, int S, int levels,
                   const double *tables, GeneralSplit &gs, GeneralImages &im);

// The fixed-point plan of a double-precision plan's tables (rows of M entries,
// kernel_table's, for levels n = S..1): fills P.fx (on = 0 where the ranges do
// not allow it) and the images head [S][hrow] and tail [S][M].  Host work.
void fx_plan(SamplerParams &P, double T, const double *tables, std::vector<int64_t> &head, std::vector<float> &tail);

// One instance of a batch: its path (a, b, N = 2^S, widths), its table
// shape (one per distinct level p), its tables (L rows of M entries from
// element tab: row d for level n = S - d), its samples and error blocks,
// the chunks each block is split into (work items), and where its tuples go.
struct BatchInstance {
    double a, b;
    int S, F;
    int L;                    // sampled levels: 1 (top level only) or S (hierarchy)
    int shape;                // index into BatchParams::shapes
    int64_t tab;              // first table element of this instance
    int64_t n_mc;             // samples
    int n_blocks, chunks;     // error blocks; work items per block
    int64_t tup;              // first tuple: [block][chunk][level], 4 doubles each
    double sigma[SU_MAX_S + 1];
};

// The Horner shape of one level p's tables (columns in x-bar^2, entries per
// column), or for the general potential its program (M = the program's entries).
struct BatchShape {
    int ncol, M;
    int len[SU_MAX_P];
    const GeneralDev *general;   // the general potential: this level's program (device), else null
};

// The batched kernel's parameters: the model fields of base (ring, alpha,
// seed, stream id, tables, flags) are shared by all instances; the
// per-instance fields of base are unused.
struct BatchParams {
    SamplerParams base;
    const BatchInstance *inst;
    const BatchShape *shapes;
    const int2 *items;        // (instance, block * chunks + chunk), costliest first
    int n_items;
    int S_max;
    int C_max;                // largest 2^(S - F): segment endpoints per path
    int L_max;                // most sampled levels of an instance
    int64_t tab_max;          // largest L * M: table elements staged per item
    double *tuples;           // per instance from its tup offset
    int *counter;             // work-queue head, zeroed before every launch
    int fixed_shape;          // >= 0: every item's instance has this compiled table shape (fixed_shapes.h)
    int fixed_src;            // ... which is shapes[fixed_src]
};

// dynamic shared memory the sampler needs
size_t sampler_smem_bytes(const SamplerParams &P, int precision);
// the compiled table shape the sampler launch of P runs with, or -1 (generic)
int sampler_fixed_shape(const SamplerParams &P, int precision);
// max resident CTAs per SM for the sampler (after opting in to its smem)
int sampler_occupancy(const SamplerParams &P, int precision, size_t smem);

// U[i * n + j] = exp(lognorm - (x_j - x_i)^2 / (2t) - t W_p) on the grid
// x_i = -L + i delta (evolution.cu); tab: the device table for eps = t
cudaError_t launch_evolution(const SamplerParams &P, int precision, const void *tab, double L, double delta, int n,
                             double t, double lognorm, double *U, cudaStream_t st);

// The upper band of the evolution operator, diagonal-major:
// D[k * pitch + i] = U_{i,i+k}, k = 0..w (evolution.cu)
cudaError_t launch_band(const SamplerParams &P, int precision, const void *tab, double L, double delta, int n,
                        double t, double lognorm, int w, int64_t pitch, double *D, cudaStream_t st);
// part[split][i][c] = partial sums of (U X)[i][c] over the split's diagonals, B in {1, 8, 16, 32}
cudaError_t launch_band_matvec(int B, const double *D, int64_t pitch, int n, int w, int splits, const double *X,
                               double *part, cudaStream_t st);
// Ynew = alpha * sum_split part + beta * Ycur + gamma * Yprev (nb = n * B elements)
cudaError_t launch_cheb(const double *part, int splits, int64_t nb, const double *Ycur, const double *Yprev,
                        double *Ynew, double alpha, double beta, double gamma, cudaStream_t st);
// op 0: out[chunk][B][B] = A^T C over the chunk's rows; op 1: out = A Q (Q: B x B);
// op 2: out[chunk][B] = sum (A - Q[c] C)^2 over the chunk's rows (Q: B Ritz values)
cudaError_t launch_block_op(int op, int B, const double *A, const double *C, const double *Q, int n, int chunks,
                            double *out, cudaStream_t st);
// The same product on the tensor cores from digit planes (spectrum_mma.cu):
// Ynew = alpha U X + beta Ycur + gamma Yprev for the columns col0..col0+15 of X
// (n x B), xmax their largest magnitudes as bits; ymax (or null) receives Ynew's.
struct BandMma {
    int n, w;                          // elements beyond w diagonals have no digits
    int ea;                            // exponent of the largest element
    unsigned char *A, *Xd;
    unsigned long long *scratch_max;
    int *status;                       // bit 0: a wait ran out
};
int band_mma_bits();                          // of an element's digits, below the largest one's power of two
int band_exponent(unsigned long long bits);   // e of |v| = m 2^e, m in [1/2, 1), from v's bits
cudaError_t launch_diag_max(const double *D, int64_t pitch, int n, int w, unsigned long long *dmax, cudaStream_t st);
int64_t band_mma_bytes_a(int n, int w);
int64_t band_mma_bytes_x(int n);
cudaError_t launch_band_digits(const BandMma &M, const double *D, int64_t pitch, cudaStream_t st);
cudaError_t launch_col_max(const double *X, int n, int B, int col0, unsigned long long *xmax, cudaStream_t st);
cudaError_t launch_band_mma(const BandMma &M, const double *X, const unsigned long long *xmax, unsigned long long *ymax,
                            int B, int col0, const double *Ycur, const double *Yprev, double *Ynew, double alpha,
                            double beta, double gamma, cudaStream_t st);
// one Lanczos step after wv = U v (alpha and beta into al[j] and be[j])
cudaError_t launch_lanczos(int n, int j, double *v, double *vp, double *wv, double *al, double *be, cudaStream_t st);
// vec[k n + i] = scale X[i][k], k < nev
cudaError_t launch_vectors(int B, const double *X, int n, int nev, double scale, double *vec, cudaStream_t st);

// Systems of d = D x M coordinates (Sec. 2.2): one bisection path per
// thread, every coordinate an exact Brownian bridge (coordinate c of heap
// midpoint j takes normal j D + c of the sample's stream), built and weighed
// in segments of 2^kNdSeg slices (segment endpoints in a global scratch, one
// segment's points in local memory); W(x, xb; eps) per slice by nested Horner
// (nd_plan.cpp), several slices at a time; weights and per-item tuples as the
// one-dimensional sampler's.
constexpr int kNdSeg = 5;     // the several-coordinates path in segments of 2^5 slices
constexpr uint32_t kNdOdd = 1u << 16;   // program word: the polynomial has a factor z_k
// The nested-Horner program of a set of monomials (nd_plan.cpp).
struct NdProgram {
    std::vector<uint32_t> words;
    std::vector<int> slot;    // table entry of each coefficient in program order, -1: zero
    unsigned sq = 0;          // depths whose Horner variable is z_k^2
};
// the order of the variables for these monomials (nv exponents each)
void nd_order(const std::vector<std::vector<unsigned char>> &mono, int nv, int *order);
void nd_program(const std::vector<std::vector<unsigned char>> &mono, const std::vector<int> &pick, int nv,
                const int *order, NdProgram &G);
// where the entries of level n's table go (part: one of these each)
enum : char { kNdFloat = 0, kNdDouble = 1, kNdNone = 2 };   // single precision, double, too small to count
void nd_split(const std::vector<std::vector<unsigned char>> &mono, int D, const double *a, const double *b, double T,
              int n, const double *table, std::vector<char> &part);

struct NdParams {
    SamplerParams base;       // S, levels, M = coefficients of the program per level, sigma, stream, items, outputs
    int D;
    int order[2 * kNdMaxDim]; // variable of each depth: x_c = c, xb_c = D + c
    unsigned sq;              // depths whose Horner variable is z_k^2
    int n_words;
    const uint32_t *words;    // device: the program
    // base.tables: [S][M], pairs {c, c} in single precision
    // double precision: the single-precision part's pairs [S][M], and per level the program and entries of
    // the double part (heads = 0: the whole program in double)
    const float2 *tail;
    const uint32_t *hwords;   // all levels' words
    const double *hcoef;
    int n_hwords, n_hcoef;
    int heads[SU_MAX_S], hw[SU_MAX_S], hc[SU_MAX_S];   // row d: its double entries, first word, first coefficient
    unsigned hsq[SU_MAX_S];
    int staged;               // program and tables in shared memory
    unsigned one;             // 1
    double a[kNdMaxDim], b[kNdMaxDim];
    void *paths;              // device (double or float): segment endpoint i, coordinate c of slot t
                              // at [(i D + c) pstride + t]
    int64_t pstride;          // slots = grid x kThreads
};
size_t nd_smem_bytes(const NdParams &Q, int precision);
int nd_occupancy(const NdParams &Q, int precision, size_t smem);
cudaError_t launch_nd(const NdParams &Q, int precision, int grid, size_t smem, cudaStream_t st);

cudaError_t launch_sampler(const SamplerParams &P, int precision, int grid, size_t smem,
                           cudaStream_t st);
size_t batch_smem_bytes(const BatchParams &B, int precision);
int batch_occupancy(const BatchParams &B, int precision, size_t smem);
const void *batch_fn(const BatchParams &B, int precision);
// tuples of blocks [b0, b0 + n_blocks) from their items' partial tuples
cudaError_t launch_combine(const double *partial, double *tuples, int64_t b0, int64_t n_blocks, int levels,
                           int64_t items_per_block, cudaStream_t st);
cudaError_t launch_normals(uint64_t seed, uint32_t instance, int64_t sample0, int64_t n_samples,
                           int n_normals, int precision, double *out, cudaStream_t st);
cudaError_t launch_philox_words(uint64_t seed, uint32_t instance, int64_t sample0,
                                int64_t n_samples, int n_calls, uint32_t *out, cudaStream_t st);

}  // namespace su
