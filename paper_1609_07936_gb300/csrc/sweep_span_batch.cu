// Batched span sweep (sweep_span.cuh): the plain loop with 8 and 4 lanes per walker.
#include "sweep_span.cuh"

namespace sail {

cudaError_t launch_span_batch_modes(const BatchProblem *d_probs, const BatchItem *d_items, int n_items, int *d_counter,
                                    size_t smem, int warps, int mode, cudaStream_t st);

size_t span_batch_smem(const DevProblem &P, int smem_max) {
    const size_t base = span_ring_bytes(kSpanWarps) + (size_t)span_vec_floats(P.n_omega) * 4;
    const size_t all = base + (size_t)P.n_omega * P.span * 4;
    return all <= (size_t)smem_max ? all : base;
}

// 4 lanes once 8 would fill every SM's 16 warps (see launch_span).
int span_batch_lanes(long long walkers) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return walkers > 4ll * kSpanWarps * sms ? 4 : 8;
}

cudaError_t launch_span_batch(const BatchProblem *d_probs, const BatchItem *d_items, int n_items, int *d_counter, size_t smem,
                              int warps, int lanes, int mode, cudaStream_t st) {
    if (mode != kPlain) return launch_span_batch_modes(d_probs, d_items, n_items, d_counter, smem, warps, mode, st);
    if (lanes == 4) return launch_span_batch_g<4, kPlain>(d_probs, d_items, n_items, d_counter, smem, warps, st);
    return launch_span_batch_g<8, kPlain>(d_probs, d_items, n_items, d_counter, smem, warps, st);
}

}  // namespace sail
