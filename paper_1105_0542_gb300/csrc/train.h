// Internal interface of the proposal-network training kernels.
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

namespace su {
namespace train {

// Device state of a training run: flat parameter vectors (mlp::kParams each), the
// weights as operands, the loss sum, the step counter.
struct Workspace {
    void *base = nullptr;
    float *theta = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    unsigned char *blob = nullptr;
    double *loss = nullptr;
    int *step = nullptr, *done = nullptr;
    int *status = nullptr;                               // set when a tensor-core wait gave up
    int ctas = 0;                                        // of the step kernel
    float *part = nullptr;                               // their gradients
    double *loss_part = nullptr;                         // and losses

    ~Workspace();
    cudaError_t make(int rows);                          // for steps of that many rows; everything zero
};

// the operands of ws.theta
cudaError_t pack(Workspace &ws, cudaStream_t st);
// ws.loss and ws.grad = those of n rows of features (n x 6), targets and weights
cudaError_t loss_grad(Workspace &ws, const float *F, const float *u, const float *rw, int n, double inv_norm,
                      cudaStream_t st);
// the CTAs' parts of the same for the midpoints of the paths ([n][np1] floats) that ids lists for
// step *ws.step (nb a step, a ring of ids_steps steps), weights one
cudaError_t path_step(Workspace &ws, const float *paths, int np1, const int *ids, int ids_steps, int nb, float a, float b,
                      float T, int S, const float *sig, cudaStream_t st);
// minibatch path ids of the steps step0.. step0 + n_steps - 1: nb draws each in
// proportion to the weights whose running sums are cdf[0..n) (total = cdf[n-1]),
// Philox under the key seed
cudaError_t sample_ids(const double *cdf, int64_t n, double total, uint64_t seed, int step0, int n_steps, int nb,
                       int *ids, cudaStream_t st);
// out[i] = w[i][S - 1] of w [n][S]
cudaError_t top_weights(const double *w, int64_t n, int S, double *out, cudaStream_t st);
// one Adam step from those parts with t = *ws.step + 1; losses[*ws.step] = the loss,
// ++*ws.step
cudaError_t adam_step(Workspace &ws, float lr, double *losses, cudaStream_t st);

}  // namespace train
}  // namespace su
