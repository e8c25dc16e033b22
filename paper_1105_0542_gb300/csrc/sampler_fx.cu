// The fixed-point double sampler for table shapes that are not compiled in and
// for the tanh^2 ring, and its shared memory.  (The compiled shapes' instances:
// sampler_inst.cu.)
#include "sampler_fx.cuh"

namespace su {

const void *sampler_fx_entry(int ring) {
    return ring == RING_TANH2 ? (const void *)sampler_fx_kernel<RING_TANH2, -1>
                              : (const void *)sampler_fx_kernel<RING_EVEN, -1>;
}

size_t sampler_fx_smem_bytes(const SamplerParams &P) {
    size_t off = sizeof(fx::Tables) + (sizeof(float2) * (size_t)P.M + sizeof(int64_t) * (size_t)P.fx.hrow) * P.S;
    if (P.ring == RING_TANH2) off += sizeof(fx::TanhNode) * (size_t)P.fx.nodes;
    off += sizeof(int64_t) * (size_t)kFxRows * kThreads;
    if (!fx_share_sw(P)) off += sizeof(double) * (size_t)P.levels * kThreads * P.rounds;
    return off;
}

}  // namespace su
