// Batched span sweep (sweep_span.cuh): the index walk and the Hastings acceptance, 8 lanes per walker.
#include "sweep_span.cuh"

namespace sail {

cudaError_t span_batch_static_modes(int mode, size_t *bytes) {
    return mode == kWalk ? static_smem(sweep_span_batch_kernel<8, kWalk>, bytes) : static_smem(sweep_span_batch_kernel<8, kHastings>, bytes);
}

cudaError_t launch_span_batch_modes(const BatchProblem *d_probs, const BatchItem *d_items, int n_items, int *d_counter,
                                    size_t smem, int warps, int mode, cudaStream_t st) {
    if (mode == kWalk) return launch_span_batch_g<8, kWalk>(d_probs, d_items, n_items, d_counter, smem, warps, st);
    return launch_span_batch_g<8, kHastings>(d_probs, d_items, n_items, d_counter, smem, warps, st);
}

}  // namespace sail
