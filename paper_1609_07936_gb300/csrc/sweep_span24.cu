// The span sweep with 24 basis directions (sweep_span.cuh; one translation unit per width, compiled
// in parallel).
#include "sweep_span.cuh"

namespace sail {

cudaError_t launch_sweep_span24(const DevProblem &P, const DevState &S, int n0, int n1, cudaStream_t st) {
    return launch_span_mode<24>(P, S, n0, n1, st);
}

}  // namespace sail
