// The basis of the kernel's columns (see sweep_span.cuh): built on the host from sampled columns,
// applied to all columns and checked on the device, in FP64.  Compiled without contraction.
#include <algorithm>
#include <cmath>
#include <vector>

#include "sail_internal.cuh"

namespace sail {

namespace {

// Largest part of a column outside the basis, relative to its norm: a quarter of FP32's rounding
// unit, below the rounding of the stored columns themselves.
constexpr double kSpanTol = 1.4901161193847656e-08;   // 2^-26

// One warp per column j: K'_jk = sum_i U_ki Khat_ij, and the norm of what the basis leaves of
// the column against the column's (the largest ratio over all columns goes to *worst).
__global__ void __launch_bounds__(128) span_table_kernel(DevProblem P, const double *U, float *Kspan, double *worst) {
    const int j = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (j >= P.n_omega) return;
    const int PAD = P.n_tau_pad, RR = P.span;
    const double *K = P.Khat64 + (size_t)j * PAD;
    double top = 0.0;
    for (int i = lane; i < PAD; i += 32) top = fmax(top, fabs(K[i]));
    for (int o = 16; o > 0; o >>= 1) top = fmax(top, __shfl_xor_sync(0xFFFFFFFFu, top, o));
    double coef = 0.0;                 // lane k: K'_jk
    for (int k = 0; k < RR; ++k) {
        const double *u = U + (size_t)k * PAD;
        double c = 0.0;
        for (int i = lane; i < PAD; i += 32) c += u[i] * K[i];
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
        if (lane == k) coef = c;
    }
    if (lane < RR) Kspan[(size_t)j * RR + lane] = (float)coef;
    double left = 0.0, all = 0.0;
    if (!(top > 0.0)) return;          // an underflown column is zero in either form
    for (int i0 = 0; i0 < PAD; i0 += 32) {
        const int i = i0 + lane;
        double e = K[i];
        const double x = e / top;
        for (int k = 0; k < RR; ++k) e -= __shfl_sync(0xFFFFFFFFu, coef, k) * U[(size_t)k * PAD + i];
        left += (e / top) * (e / top);
        all += x * x;
    }
    for (int o = 16; o > 0; o >>= 1) {
        left += __shfl_xor_sync(0xFFFFFFFFu, left, o);
        all += __shfl_xor_sync(0xFFFFFFFFu, all, o);
    }
    // non-negative doubles compare as their bit patterns
    if (lane == 0) atomicMax((unsigned long long *)worst, (unsigned long long)__double_as_longlong(sqrt(left / all)));
}

}  // namespace

bool span_fits(double worst) { return worst <= kSpanTol; }

int span_basis(const double *K64, int n_tau, int pad, int n_omega, int n_samples, std::vector<double> &U) {
    // columns at Chebyshev nodes over the bins (the kernel is smooth in omega), scaled to norm 1
    std::vector<double> A;
    int m = 0, last = -1;
    const int want = std::min(n_samples, n_omega);
    for (int q = 0; q < want; ++q) {
        const double t = 0.5 * (1.0 - std::cos(3.14159265358979323846 * q / std::max(1, want - 1)));
        const int j = want == n_omega ? q : (int)std::lround(t * (n_omega - 1));
        if (j == last) continue;
        last = j;
        const double *k = K64 + (size_t)j * pad;
        double top = 0.0, s = 0.0;
        for (int i = 0; i < n_tau; ++i) top = std::max(top, std::fabs(k[i]));
        if (!(top > 0.0)) continue;
        for (int i = 0; i < n_tau; ++i) s += (k[i] / top) * (k[i] / top);
        const double scale = 1.0 / std::sqrt(s);
        A.resize((size_t)(m + 1) * n_tau);
        for (int i = 0; i < n_tau; ++i) A[(size_t)m * n_tau + i] = k[i] / top * scale;
        ++m;
    }
    // dot product in eight interleaved sums (independent chains)
    auto dot = [n_tau](const double *x, const double *y) {
        double s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        int i = 0;
        for (; i + 8 <= n_tau; i += 8)
            for (int e = 0; e < 8; ++e) s[e] += x[i + e] * y[i + e];
        for (; i < n_tau; ++i) s[0] += x[i] * y[i];
        return ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
    };
    auto axpy = [n_tau](double c, const double *x, double *y) {
        for (int i = 0; i < n_tau; ++i) y[i] -= c * x[i];
    };
    // Gram-Schmidt with column pivoting; each direction is orthogonalised against the earlier ones
    // once more before use.  need: directions until every sample is within half the tolerance.
    std::vector<double> norm2(m, 1.0);
    U.assign((size_t)kSpanMax * pad, 0.0);
    int need = -1, k = 0;
    for (; k < kSpanMax; ++k) {
        int j = -1;
        double big = 0.0;
        for (int c = 0; c < m; ++c)
            if (norm2[c] > big) { big = norm2[c]; j = c; }
        if (need < 0 && !(std::sqrt(big) > 0.5 * kSpanTol)) need = k;
        if (need >= 0 && k >= span_width(need)) break;
        if (j < 0 || !(std::sqrt(big) > 1e-13)) break;     // the samples' span is exhausted
        double *u = U.data() + (size_t)k * pad;
        std::copy(A.begin() + (size_t)j * n_tau, A.begin() + (size_t)(j + 1) * n_tau, u);
        const double s0 = 1.0 / std::sqrt(dot(u, u));
        for (int i = 0; i < n_tau; ++i) u[i] *= s0;
        for (int q = 0; q < k; ++q) axpy(dot(U.data() + (size_t)q * pad, u), U.data() + (size_t)q * pad, u);
        const double s1 = 1.0 / std::sqrt(dot(u, u));
        for (int i = 0; i < n_tau; ++i) u[i] *= s1;
        for (int c = 0; c < m; ++c) {
            double *a = A.data() + (size_t)c * n_tau;
            axpy(dot(u, a), u, a);
            norm2[c] = dot(a, a);
        }
    }
    if (need < 0) {
        double big = 0.0;
        for (int c = 0; c < m; ++c) big = std::max(big, norm2[c]);
        if (std::sqrt(big) > kSpanTol) return 0;
        need = k;
    }
    // mix the directions evenly (orthonormal cosine transform over them; unused ones are zero)
    const int rr = span_width(need);
    std::vector<double> V((size_t)kSpanMax * pad, 0.0);
    for (int q = 0; q < rr; ++q)
        for (int d = 0; d < std::min(k, rr); ++d) {
            const double c = std::sqrt((d ? 2.0 : 1.0) / rr) * std::cos(3.14159265358979323846 * (q + 0.5) * d / rr);
            axpy(-c, U.data() + (size_t)d * pad, V.data() + (size_t)q * pad);
        }
    U.swap(V);
    return rr;
}

cudaError_t launch_span_table(const DevProblem &P, const double *U, float *Kspan, double *worst, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(worst, 0, sizeof(double), st);
    if (e != cudaSuccess) return e;
    span_table_kernel<<<(P.n_omega + 3) / 4, 128, 0, st>>>(P, U, Kspan, worst);
    return cudaGetLastError();
}

cudaError_t launch_sweep_span16(const DevProblem &P, const DevState &S, int n0, int n1, cudaStream_t st);
cudaError_t launch_sweep_span24(const DevProblem &P, const DevState &S, int n0, int n1, cudaStream_t st);
cudaError_t launch_sweep_span32(const DevProblem &P, const DevState &S, int n0, int n1, cudaStream_t st);

cudaError_t launch_sweep_span(const DevProblem &P, const DevState &S, int n0, int n1, cudaStream_t st) {
    switch (P.span) {
        case 16: return launch_sweep_span16(P, S, n0, n1, st);
        case 24: return launch_sweep_span24(P, S, n0, n1, st);
        case 32: return launch_sweep_span32(P, S, n0, n1, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace sail
