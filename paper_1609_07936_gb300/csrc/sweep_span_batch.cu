// Batched span sweep (sweep_span.cuh): the plain loop with 4 lanes per walker (its spectra stay in
// global memory, where 4 lanes are the faster layout at every population: see launch_span).
#include "sweep_span.cuh"

namespace sail {

cudaError_t launch_span_batch_modes(const BatchProblem *d_probs, const BatchItem *d_items, int n_items, int *d_counter,
                                    size_t smem, int warps, int mode, cudaStream_t st);

cudaError_t span_batch_static_modes(int mode, size_t *bytes);

cudaError_t span_batch_smem(const DevProblem &P, int mode, size_t *bytes) {
    int dev = 0, smem_max = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    size_t fixed = 0;
    const cudaError_t e = mode == kPlain ? static_smem(sweep_span_batch_kernel<4, kPlain>, &fixed) : span_batch_static_modes(mode, &fixed);
    if (e != cudaSuccess) return e;
    const size_t base = span_ring_bytes(kSpanWarps) + (size_t)span_vec_floats(P.n_omega) * 4;
    const size_t all = base + (size_t)P.n_omega * P.span * 4;
    *bytes = all + fixed <= (size_t)smem_max ? all : base;
    return cudaSuccess;
}

cudaError_t launch_span_batch(const BatchProblem *d_probs, const BatchItem *d_items, int n_items, int *d_counter, size_t smem,
                              int warps, int mode, cudaStream_t st) {
    if (mode != kPlain) return launch_span_batch_modes(d_probs, d_items, n_items, d_counter, smem, warps, mode, st);
    return launch_span_batch_g<4, kPlain>(d_probs, d_items, n_items, d_counter, smem, warps, st);
}

}  // namespace sail
