// The lowest energies of the space-discretized evolution operator (Sec. 5,
// Fig. 3): the largest eigenvalues lambda_k = exp(-t E_k) of the symmetric
// band matrix U, from its upper band in diagonal-major storage
// (D[k * pitch + i] = U_{i,i+k}, k = 0..w), by Chebyshev-filtered block
// subspace iteration with Rayleigh-Ritz (Zhou and Saad, "A Chebyshev-Davidson
// algorithm"/"Self-consistent-field calculations using Chebyshev-filtered
// subspace iteration", 2006-2007), all in double precision:
//
//   bounds   a few Lanczos steps (Lanczos 1950) give the lower end lo of the
//            spectrum (smallest Ritz value minus the last off-diagonal);
//   filter   Y = T_m((U - c)/e) X with the interval [lo, cut] mapped onto
//            [-1, 1] (c = (cut + lo)/2, e = (cut - lo)/2), cut = the
//            smallest Ritz value of the block: components above cut grow
//            like T_m of their mapped value, the rest stay bounded;
//   basis    shifted Cholesky QR followed by two plain passes (Fukaya,
//            Kannan, Nakatsukasa, Yamamoto, Yanagisawa 2020) on the
//            column-scaled Gram matrix;
//   Ritz     H = Y^T U Y, its eigenpairs by cyclic Jacobi rotations (Golub
//            and Van Loan, Sec. 8.5), X = Y Q, residuals |U x_k - theta_k x_k|.
//
// The block width (8, 16 or 32 columns) holds nev wanted pairs plus at least
// six guard vectors, so nearly degenerate pairs (a tunnelling doublet) sit
// inside the block and are separated by the Rayleigh-Ritz step, not by the
// filter.  Device work: the band matrix-block product with the Chebyshev update
// (on the tensor cores in exact digits, spectrum_mma.cu; in double, FP64 bound,
// where the digit planes have no room), Gram products and rotations; host work:
// B x B Cholesky and Jacobi.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include <cuda_runtime.h>

#include "sampler.h"
#include "spectrum.h"

namespace su {
namespace {

// least n w B for the tensor-core product: at n = 1201, w = 158, B = 8 a product
// takes 0.023 ms there and 0.013 in double, at n = 2001, w = 212, B = 16 0.032
// and 0.050, at n = 16 385, w = 1297, B = 16 0.106 and 1.16
constexpr int64_t kMmaLeast = 3000000;
// and its least band: below some 36 diagonals the digits' rounding, of the largest
// element, would pass that of the double product's running sums (spectrum_mma.cu)
constexpr int kMmaBand = 48;

// symmetric eigenpairs of the k x k matrix A (row-major) by cyclic Jacobi
// rotations; eigenvalues descending in ev, eigenvectors in the columns of V
void jacobi_eig(std::vector<double> A, int k, std::vector<double> &ev, std::vector<double> &V) {
    V.assign((size_t)k * k, 0.0);
    for (int i = 0; i < k; ++i) V[(size_t)i * k + i] = 1.0;
    auto a = [&](int i, int j) -> double & { return A[(size_t)i * k + j]; };
    for (int sweep = 0; sweep < 100; ++sweep) {
        double off = 0.0, tot = 0.0;
        for (int i = 0; i < k; ++i)
            for (int j = 0; j < k; ++j) {
                tot += a(i, j) * a(i, j);
                if (i != j) off += a(i, j) * a(i, j);
            }
        if (off <= 1e-34 * tot || off == 0.0) break;
        for (int p = 0; p < k - 1; ++p)
            for (int q = p + 1; q < k; ++q) {
                const double apq = a(p, q);
                if (apq == 0.0) continue;
                // rotation that annihilates a(p, q): tan(phi) = t, t the smaller root
                const double theta = (a(q, q) - a(p, p)) / (2.0 * apq);
                const double t = (theta >= 0 ? 1.0 : -1.0) / (std::fabs(theta) + std::sqrt(theta * theta + 1.0));
                const double c = 1.0 / std::sqrt(t * t + 1.0), s = t * c;
                for (int r = 0; r < k; ++r) {   // A <- A J (columns p, q)
                    const double arp = a(r, p), arq = a(r, q);
                    a(r, p) = c * arp - s * arq;
                    a(r, q) = s * arp + c * arq;
                }
                for (int r = 0; r < k; ++r) {   // A <- J^T A (rows p, q)
                    const double apr = a(p, r), aqr = a(q, r);
                    a(p, r) = c * apr - s * aqr;
                    a(q, r) = s * apr + c * aqr;
                }
                for (int r = 0; r < k; ++r) {   // V <- V J
                    const double vrp = V[(size_t)r * k + p], vrq = V[(size_t)r * k + q];
                    V[(size_t)r * k + p] = c * vrp - s * vrq;
                    V[(size_t)r * k + q] = s * vrp + c * vrq;
                }
            }
    }
    std::vector<int> ord((size_t)k);
    for (int i = 0; i < k; ++i) ord[(size_t)i] = i;
    std::sort(ord.begin(), ord.end(), [&](int x, int y) { return a(x, x) > a(y, y); });
    ev.resize((size_t)k);
    std::vector<double> W((size_t)k * k);
    for (int c = 0; c < k; ++c) {
        ev[(size_t)c] = a(ord[(size_t)c], ord[(size_t)c]);
        for (int r = 0; r < k; ++r) W[(size_t)r * k + c] = V[(size_t)r * k + ord[(size_t)c]];
    }
    V.swap(W);
}

// The smallest and largest eigenvalue of the symmetric tridiagonal matrix with
// diagonal al and off-diagonal be, by bisection on the Sturm sequence's count of
// negative pivots (Golub and Van Loan, Sec. 8.4).
void tridiagonal_ends(const std::vector<double> &al, const std::vector<double> &be, double &least, double &most) {
    const size_t k = al.size();
    double lo = al[0], hi = al[0];
    for (size_t i = 0; i < k; ++i) {   // Gershgorin
        const double r = (i ? std::fabs(be[i - 1]) : 0.0) + (i + 1 < k ? std::fabs(be[i]) : 0.0);
        lo = std::min(lo, al[i] - r);
        hi = std::max(hi, al[i] + r);
    }
    auto below = [&](double x) {   // eigenvalues smaller than x
        size_t n = 0;
        double d = 1.0;
        for (size_t i = 0; i < k; ++i) {
            d = al[i] - x - (i ? be[i - 1] * be[i - 1] / d : 0.0);
            if (d == 0.0) d = -1e-300;
            n += d < 0.0;
        }
        return n;
    };
    auto find = [&](size_t want) {   // the eigenvalue that has `want` below it
        double a = lo, b = hi;
        for (int it = 0; it < 200 && a < b; ++it) {
            const double m = 0.5 * (a + b);
            if (m <= a || m >= b) break;
            if (below(m) > want)
                b = m;
            else
                a = m;
        }
        return 0.5 * (a + b);
    };
    least = find(0);
    most = find(k - 1);
}

// lower Cholesky factor of the k x k matrix G (row-major); false if not
// positive definite
bool cholesky(const std::vector<double> &G, int k, std::vector<double> &Lf) {
    Lf.assign((size_t)k * k, 0.0);
    for (int j = 0; j < k; ++j) {
        double d = G[(size_t)j * k + j];
        for (int r = 0; r < j; ++r) d -= Lf[(size_t)j * k + r] * Lf[(size_t)j * k + r];
        if (!(d > 0.0)) return false;
        const double l = std::sqrt(d);
        Lf[(size_t)j * k + j] = l;
        for (int i = j + 1; i < k; ++i) {
            double s = G[(size_t)i * k + j];
            for (int r = 0; r < j; ++r) s -= Lf[(size_t)i * k + r] * Lf[(size_t)j * k + r];
            Lf[(size_t)i * k + j] = s / l;
        }
    }
    return true;
}

// (L^T)^{-1}: the inverse of the upper factor R = L^T, row-major
std::vector<double> inverse_upper(const std::vector<double> &Lf, int k) {
    std::vector<double> X((size_t)k * k, 0.0);   // X = R^{-1}, R[i][j] = L[j][i]
    for (int c = 0; c < k; ++c) {
        // solve R x = e_c by back substitution
        for (int i = k - 1; i >= 0; --i) {
            double s = i == c ? 1.0 : 0.0;
            for (int j = i + 1; j < k; ++j) s -= Lf[(size_t)j * k + i] * X[(size_t)j * k + c];
            X[(size_t)i * k + c] = s / Lf[(size_t)i * k + i];
        }
    }
    return X;
}

// device buffers, freed together
struct Bufs {
    std::vector<void *> v;
    ~Bufs() {
        for (void *p : v) cudaFree(p);
    }
    template <typename T>
    cudaError_t get(T **p, size_t count) {
        void *q = nullptr;
        cudaError_t e = cudaMalloc(&q, count * sizeof(T));
        if (e == cudaSuccess) v.push_back(q);
        *p = static_cast<T *>(q);
        return e;
    }
};

struct Work {
    double *D = nullptr;
    int64_t pitch = 0;
    int n = 0, w = 0, B = 0, splits = 1, chunks = 1;
    cudaStream_t st = nullptr;
    double *part = nullptr;      // splits x n x B
    double *gpart = nullptr;     // chunks x B x B
    double *dQ = nullptr;        // B x B (or B values)
    bool mma = false;            // block products on the tensor cores
    BandMma M{};
    unsigned long long *mx[2] = {nullptr, nullptr};   // column maxima (32 each) of a product's input and output
    std::vector<double> hpart;
    int64_t matvecs = 0;         // vector products with U
    std::vector<cudaEvent_t> ev; // pairs around the block products (their device time)
    ~Work() {
        for (cudaEvent_t e : ev) cudaEventDestroy(e);
    }
};

#define SPC(call)                               \
    do {                                        \
        cudaError_t e_ = (call);                \
        if (e_ != cudaSuccess) return e_;       \
    } while (0)

// Ynew = alpha U X + beta Ycur + gamma Yprev for the block: on the tensor cores
// (in: which of W.mx holds X's column maxima; the other receives Ynew's), or in
// double from split partial sums.  Bracketed by a pair of events for its device time.
cudaError_t product(Work &W, const double *X, const double *Ycur, const double *Yprev, double *Ynew, double alpha,
                    double beta, double gamma, int in) {
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    SPC(cudaEventCreate(&e0));
    W.ev.push_back(e0);
    SPC(cudaEventCreate(&e1));
    W.ev.push_back(e1);
    SPC(cudaEventRecord(e0, W.st));
    if (W.mma) {
        for (int c = 0; c < W.B; c += 16)
            SPC(launch_band_mma(W.M, X, W.mx[in] + c, W.mx[in ^ 1] + c, W.B, c, Ycur, Yprev, Ynew, alpha, beta, gamma, W.st));
    } else {
        SPC(launch_band_matvec(W.B, W.D, W.pitch, W.n, W.w, W.splits, X, W.part, W.st));
        SPC(launch_cheb(W.part, W.splits, (int64_t)W.n * W.B, Ycur, Yprev, Ynew, alpha, beta, gamma, W.st));
    }
    SPC(cudaEventRecord(e1, W.st));
    W.matvecs += W.B;
    return cudaSuccess;
}

// W.mx[0] = the column maxima of X
cudaError_t maxima(Work &W, const double *X) {
    if (W.mma)
        for (int c = 0; c < W.B; c += 16) SPC(launch_col_max(X, W.n, W.B, c, W.mx[0] + c, W.st));
    return cudaSuccess;
}

// G = A^T C (B x B, row-major), the chunks summed in order on the host
cudaError_t gram(Work &W, const double *A, const double *C, std::vector<double> &G) {
    const int B = W.B;
    SPC(launch_block_op(0, B, A, C, nullptr, W.n, W.chunks, W.gpart, W.st));
    W.hpart.resize((size_t)W.chunks * B * B);
    SPC(cudaMemcpyAsync(W.hpart.data(), W.gpart, W.hpart.size() * sizeof(double), cudaMemcpyDeviceToHost, W.st));
    SPC(cudaStreamSynchronize(W.st));
    G.assign((size_t)B * B, 0.0);
    for (int q = 0; q < W.chunks; ++q)
        for (int e = 0; e < B * B; ++e) G[(size_t)e] += W.hpart[(size_t)q * B * B + e];
    return cudaSuccess;
}

// out = A Q for a host B x B matrix Q
cudaError_t rotate(Work &W, const double *A, const std::vector<double> &Q, double *out) {
    SPC(cudaMemcpyAsync(W.dQ, Q.data(), Q.size() * sizeof(double), cudaMemcpyHostToDevice, W.st));
    SPC(launch_block_op(1, W.B, A, nullptr, W.dQ, W.n, W.chunks, out, W.st));
    // the host copy of Q must outlive the copy
    return cudaStreamSynchronize(W.st);
}

// orthonormal basis of the columns of Y into out: column scaling, one
// shifted Cholesky QR pass and two plain ones.  Returns false (in ok) when
// the block has lost rank.
cudaError_t orthonormalize(Work &W, const double *Y, double *tmp, double *out, bool &ok) {
    const int B = W.B;
    std::vector<double> G, Lf;
    SPC(gram(W, Y, Y, G));
    std::vector<double> dsc((size_t)B);
    for (int c = 0; c < B; ++c) dsc[(size_t)c] = G[(size_t)c * B + c] > 0 ? 1.0 / std::sqrt(G[(size_t)c * B + c]) : 0.0;
    for (int i = 0; i < B; ++i)
        for (int j = 0; j < B; ++j) G[(size_t)i * B + j] *= dsc[(size_t)i] * dsc[(size_t)j];
    double tr = 0.0;
    for (int c = 0; c < B; ++c) tr += G[(size_t)c * B + c];
    const double shift = 11.0 * ((double)W.n * B + (double)B * (B + 1)) * 0x1p-53 * tr;
    for (int c = 0; c < B; ++c) G[(size_t)c * B + c] += shift;
    ok = cholesky(G, B, Lf);
    if (!ok) return cudaSuccess;
    std::vector<double> Q = inverse_upper(Lf, B);
    for (int i = 0; i < B; ++i)
        for (int j = 0; j < B; ++j) Q[(size_t)i * B + j] *= dsc[(size_t)i];
    SPC(rotate(W, Y, Q, out));
    for (int pass = 0; pass < 2; ++pass) {
        SPC(gram(W, out, out, G));
        ok = cholesky(G, B, Lf);
        if (!ok) return cudaSuccess;
        Q = inverse_upper(Lf, B);
        SPC(rotate(W, out, Q, tmp));
        SPC(cudaMemcpyAsync(out, tmp, (size_t)W.n * B * sizeof(double), cudaMemcpyDeviceToDevice, W.st));
    }
    return cudaSuccess;
}

}  // namespace

int band_spectrum(const double *D, int64_t pitch, int n, int w, int nev, int degree, double tol, int max_iter,
                  uint64_t seed, double *d_vectors, double vec_scale, cudaStream_t st, SpectrumResult &res,
                  std::string &err) {
    res = SpectrumResult{};
    const int B = nev + 6 <= 8 ? 8 : nev + 6 <= 16 ? 16 : 32;
    if (nev < 1 || nev + 6 > 32 || nev > n / 2) {
        err = "nev must be in 1..26 and at most n/2";
        return SU_EINVAL;
    }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    Work W;
    W.D = const_cast<double *>(D);
    W.pitch = pitch;
    W.n = n;
    W.w = w;
    W.B = B;
    W.st = st;
    const int rblocks = (n + 63) / 64;
    // split the diagonals so that about 32 CTAs of two warps per SM are
    // resident: the FP64 multiply-adds need the warps to hide load latency
    W.splits = std::max(1, std::min(w + 1, (32 * std::max(sms, 1) + rblocks - 1) / rblocks));
    W.chunks = std::max(1, std::min(std::max(sms, 1), (n + 31) / 32));
    Bufs bufs;
    const size_t nb = (size_t)n * B;
    const int steps = std::min(40, n);
    double *X, *Y0, *Y1, *Y2, *Z, *UX, *T, *ab;
    unsigned long long *dmax = nullptr;
    cudaError_t e = cudaSuccess;
    for (double **p : {&X, &Y0, &Y1, &Y2, &Z, &UX, &T})
        if (e == cudaSuccess) e = bufs.get(p, nb);
    if (e == cudaSuccess) e = bufs.get(&W.gpart, (size_t)W.chunks * B * B);
    if (e == cudaSuccess) e = bufs.get(&W.dQ, (size_t)B * B);
    if (e == cudaSuccess) e = bufs.get(&ab, (size_t)2 * steps);
    if (e == cudaSuccess) e = bufs.get(&dmax, (size_t)w + 1 + 4 * 32);
    if (e == cudaSuccess) e = bufs.get(&W.part, (size_t)W.splits * n);
    auto no_buffers = [&] {
        cudaGetLastError();
        err = std::string("eigensolver buffers: ") + cudaGetErrorString(e);
        return e == cudaErrorMemoryAllocation ? SU_ENOMEM : SU_ECUDA;
    };
    if (e != cudaSuccess) return no_buffers();
    auto cuda_err = [&](cudaError_t c, const char *what) {
        err = std::string(what) + ": " + cudaGetErrorString(c);
        cudaGetLastError();
        return SU_ECUDA;
    };

    // ---- the lower end of the spectrum: Lanczos steps on one vector, all on
    // the device; the host draws the start block meanwhile
    std::mt19937_64 rng(seed);
    std::normal_distribution<double> nd(0.0, 1.0);
    std::vector<double> v((size_t)n), h(nb), hab((size_t)2 * steps);
    std::vector<unsigned long long> dm((size_t)w + 1);
    {
        double nrm = 0;
        for (double &x : v) {
            x = nd(rng);
            nrm += x * x;
        }
        nrm = std::sqrt(nrm);
        for (double &x : v) x /= nrm;
    }
    if ((e = cudaMemcpyAsync(X, v.data(), (size_t)n * sizeof(double), cudaMemcpyHostToDevice, st)) ||
        (e = launch_diag_max(D, pitch, n, w, dmax, st)))
        return cuda_err(e, "Lanczos bounds");
    for (int j = 0; j < steps; ++j) {
        if ((e = launch_band_matvec(1, W.D, W.pitch, n, w, W.splits, X, W.part, st)) ||
            (e = launch_cheb(W.part, W.splits, n, nullptr, nullptr, Y2, 1.0, 0.0, 0.0, st)) ||
            (e = launch_lanczos(n, j, X, Y1, Y2, ab, ab + steps, st)))
            return cuda_err(e, "Lanczos bounds");
        W.matvecs += 1;
    }
    for (double &x : h) x = nd(rng);
    if ((e = cudaMemcpyAsync(dm.data(), dmax, dm.size() * sizeof(dm[0]), cudaMemcpyDeviceToHost, st)) ||
        (e = cudaMemcpyAsync(hab.data(), ab, hab.size() * sizeof(double), cudaMemcpyDeviceToHost, st)) ||
        (e = cudaStreamSynchronize(st)))
        return cuda_err(e, "Lanczos bounds");
    {
        std::vector<double> al, be;
        for (int j = 0; j < steps; ++j) {
            al.push_back(hab[(size_t)j]);
            be.push_back(hab[(size_t)(steps + j)]);
            if (!(be.back() > 0)) break;
        }
        double least = 0, most = 0;
        tridiagonal_ends(al, be, least, most);
        res.upper = most + be.back();
        res.lower = least - be.back();
    }
    // ---- digit planes for the tensor-core product, where the band's values
    // are finite and the planes fit the device
    {
        const unsigned long long top = *std::max_element(dm.begin(), dm.end());
        W.M.n = n;
        W.M.ea = band_exponent(top);
        // diagonals whose elements all round to zero digits
        W.M.w = w;
        while (W.M.w > 0 && band_exponent(dm[(size_t)W.M.w]) < W.M.ea - band_mma_bits() - 1) --W.M.w;
        if (W.M.ea > -400 && W.M.ea < 400 && W.M.w >= kMmaBand && (int64_t)n * w * B >= kMmaLeast) {
            W.mx[0] = dmax + w + 1;
            W.mx[1] = W.mx[0] + 32;
            W.M.scratch_max = W.mx[1] + 32;
            W.M.status = reinterpret_cast<int *>(W.M.scratch_max + 32);
            W.mma = bufs.get(&W.M.A, (size_t)band_mma_bytes_a(n, W.M.w)) == cudaSuccess &&
                    bufs.get(&W.M.Xd, (size_t)band_mma_bytes_x(n)) == cudaSuccess;
            if (!W.mma) cudaGetLastError();
        }
        // (in double the split partial sums of the whole block)
        if (!W.mma && (e = bufs.get(&W.part, (size_t)W.splits * nb)) != cudaSuccess) return no_buffers();
        if (W.mma && ((e = cudaMemsetAsync(W.M.status, 0, sizeof(int), st)) || (e = launch_band_digits(W.M, D, pitch, st))))
            return cuda_err(e, "digit planes");
    }
    const double lo = res.lower;

    // ---- a random block, orthonormalized, and its Rayleigh-Ritz pairs
    if ((e = cudaMemcpyAsync(Y0, h.data(), nb * sizeof(double), cudaMemcpyHostToDevice, st)) ||
        (e = cudaStreamSynchronize(st)))
        return cuda_err(e, "initial block");
    std::vector<double> theta((size_t)B, 0.0), H, Q, r((size_t)B);
    const double *src = Y0;
    for (int it = 0; it <= max_iter; ++it) {
        bool ok = true;
        if ((e = orthonormalize(W, src, T, X, ok))) return cuda_err(e, "orthonormalization");
        if (!ok) {
            err = "the block lost rank (Cholesky QR failed)";
            return SU_ECUDA;
        }
        if ((e = maxima(W, X)) || (e = product(W, X, nullptr, nullptr, Z, 1.0, 0.0, 0.0, 0)) || (e = gram(W, X, Z, H)))
            return cuda_err(e, "Rayleigh-Ritz");
        for (int i = 0; i < B; ++i)   // symmetrize the projection's rounding
            for (int j = i + 1; j < B; ++j)
                H[(size_t)i * B + j] = H[(size_t)j * B + i] = 0.5 * (H[(size_t)i * B + j] + H[(size_t)j * B + i]);
        jacobi_eig(H, B, theta, Q);
        if ((e = rotate(W, X, Q, Y1)) || (e = rotate(W, Z, Q, UX))) return cuda_err(e, "Ritz vectors");
        std::swap(X, Y1);
        // residual norms of the Ritz pairs
        if ((e = cudaMemcpyAsync(W.dQ, theta.data(), (size_t)B * sizeof(double), cudaMemcpyHostToDevice, st)) ||
            (e = launch_block_op(2, B, UX, X, W.dQ, n, W.chunks, W.gpart, st)))
            return cuda_err(e, "residuals");
        std::vector<double> rp((size_t)W.chunks * B);
        int waits = 0;
        if ((e = cudaMemcpyAsync(rp.data(), W.gpart, rp.size() * sizeof(double), cudaMemcpyDeviceToHost, st)) ||
            (W.mma && (e = cudaMemcpyAsync(&waits, W.M.status, sizeof(int), cudaMemcpyDeviceToHost, st))) ||
            (e = cudaStreamSynchronize(st)))
            return cuda_err(e, "residuals");
        if (waits) {
            err = "a block product's wait ran out";
            return SU_ETIMEOUT;
        }
        double worst = 0.0;
        for (int c = 0; c < B; ++c) {
            double s = 0;
            for (int q = 0; q < W.chunks; ++q) s += rp[(size_t)q * B + c];
            r[(size_t)c] = std::sqrt(s);
            if (c < nev) worst = std::max(worst, r[(size_t)c]);
        }
        res.iterations = it;
        res.converged = worst <= tol * std::fabs(theta[0]) ? 1 : 0;
        if (res.converged || it == max_iter) break;
        // ---- filter: Y = T_m((U - c)/e) X on the interval [lo, cut]
        double cut = theta[(size_t)B - 1];
        cut = std::max(cut, lo + 1e-3 * (theta[0] - lo));
        const double c0 = 0.5 * (cut + lo), e0 = 0.5 * (cut - lo);
        // A degree at which the largest pair is amplified by no more than 2^64 against
        // the smallest of the block: the rounding left of it in the others' vectors,
        // 2^-53, then outgrows them by no more than 2^11, which the orthonormalization
        // takes; much further on the block loses rank.  (T_m(x) < e^(m acosh x); it
        // matters where the block reaches down to the spectrum's flat end, short
        // intervals or long times.)
        const double x = (theta[0] - c0) / e0;
        const int reach = x > 1.0 ? (int)(64 * 0.69314718055994531 / std::acosh(x)) : degree;
        const int m = std::max(2, std::min(it == 0 ? std::min(4, degree) : degree, reach));
        double *ym1 = X, *y = Y0, *yp = Y1;
        if ((e = maxima(W, X)) || (e = product(W, X, X, nullptr, Y0, 1.0 / e0, -c0 / e0, 0.0, 0))) return cuda_err(e, "filter");
        for (int j = 1; j < m; ++j) {
            if ((e = product(W, y, y, ym1, yp, 2.0 / e0, -2.0 * c0 / e0, -1.0, j & 1))) return cuda_err(e, "filter");
            // rotate the three buffers: the oldest becomes the next output
            double *old = ym1;
            ym1 = y;
            y = yp;
            yp = old == X ? Y2 : old;
        }
        src = y;
        if (src == X) {   // cannot happen for m >= 1; keep the orthonormalizer's output separate
            err = "internal: filter output aliases the basis";
            return SU_ECUDA;
        }
    }
    res.theta.assign(theta.begin(), theta.begin() + nev);
    res.resid.assign(r.begin(), r.begin() + nev);
    res.block = B;
    res.matvecs = W.matvecs;
    if ((e = cudaStreamSynchronize(st))) return cuda_err(e, "eigensolver");
    for (size_t q = 0; q + 1 < W.ev.size(); q += 2) {
        float ms = 0;
        if ((e = cudaEventElapsedTime(&ms, W.ev[q], W.ev[q + 1]))) return cuda_err(e, "event time");
        res.block_matvec_ms += ms;
        ++res.block_matvecs;
    }
    if (d_vectors) {
        if ((e = launch_vectors(B, X, n, nev, vec_scale, d_vectors, st)) || (e = cudaStreamSynchronize(st)))
            return cuda_err(e, "eigenvectors");
    }
    return SU_OK;
}

}  // namespace su
