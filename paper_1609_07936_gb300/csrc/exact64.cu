// FP64 kernels whose every operation is rounded on its own (this file is compiled with
// -fmad=false): the validation sweep, the residual recomputation, the branching solve and
// imprint, the stochastic average and the state initialisation.  On an FP64 state sums run in the
// order the method's definition states them (j ascending for a model value, i ascending for chi2,
// walkers ascending for an average), so these kernels reproduce a plain sequential FP64
// evaluation of the same formulas bit for bit, up to the library exp of the Metropolis test; so does
// the branching solve for either state.  Averages, smoothing and block statistics of an FP32 state
// sum in FP64 over lanes, threads or parts of the walkers.
#include <cfloat>
#include <cmath>
#include <cstdint>

#include "moves.cuh"
#include "philox.cuh"
#include <cuda_bf16.h>

#include "sail_internal.cuh"

namespace sail {

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

// ------------------------------------------------------------------ state set-up
__global__ void init_state_kernel(DevProblem P, DevState S, int precision, const double *a0,
                                  const double *R0, double chi2_0) {
    const int w = blockIdx.x;
    if (w >= P.n_walkers) return;
    for (int j = threadIdx.x; j < P.n_omega; j += blockDim.x) {
        if (precision == 0) S.a64[(size_t)w * P.n_omega + j] = a0[j];
        else S.b32[(size_t)w * P.n_omega + j] = (float)a0[j];
    }
    for (int i = threadIdx.x; i < P.n_tau_pad; i += blockDim.x) {
        const double r = i < P.n_tau ? R0[i] : 0.0;
        if (precision == 0) S.R64[(size_t)w * P.n_tau_pad + i] = r;
        else S.R32[(size_t)w * P.n_tau_pad + i] = (float)r;
    }
    if (threadIdx.x == 0) {
        S.chi2[w] = chi2_0;
        S.acc_prev[w] = P.n_omega;
        S.hash[w] = kFnvOffset;
        S.n_acc[w] = 0;
        S.n_pos[w] = 0;
        if (precision != 0) {
            S.g2[2 * w] = 1.0f;
            S.g2[2 * w + 1] = 0.0f;
        }
    }
}

// ------------------------------------------------------------------ validation sweep
// One warp per walker.  Lane l holds R_i for i = l + 32 c.  Every move is Sec. 2.2:
//   eps = 1 - r, delta_p = eps (B - A x_s) / (x_p - x_s), delta_s = eps (B - A x_p) / (x_s - x_p),
//   a_p' = r a_p + delta_p, a_s' = r a_s + delta_s (rejected if either is negative),
//   d_i = eps (Fhat_i - R_i) - delta_p Khat_ip - delta_s Khat_is,
//   Delta chi2 = sum_i d_i (2 R_i + d_i), summed over i ascending,
// accepted with probability min(1, exp(-Delta chi2 / T)) (Eq. probability-density); an
// accepted move rescales every bin by r, writes a_p', a_s' and adds d to R.
// Bins of a move (Sec. 2.3) in the oracle's order: p from word w0, then its index walk of
// L = P.walk_len steps (step t: Philox counter (mv, n, w, 1 + t), proposal word x, acceptance
// word y; move when u a_p <= a_j); s from word w1 on the bins other than the final p, then its
// walk (words z, w; proposals on the bins other than p).  Each walk is skipped with
// probability walk_rho (words x, y of counter (mv, n, w, 2 + L)).
__device__ void walk_bins64(const DevProblem &P, const double *a, uint32_t w0, uint32_t w1, int mv, int n, int w,
                            uint2 key, int &p_out, int &s_out) {
    const int NO = P.n_omega, L = P.walk_len;
    int p = (int)(((uint64_t)w0 * (uint64_t)NO) >> 32);
    bool walk_p = false, walk_s = false;
    if (L > 0) {
        const uint4 mix = philox4x32_10(make_uint4((uint32_t)mv, (uint32_t)n, (uint32_t)w, (uint32_t)(2 + L)), key);
        walk_p = !(unit64(mix.x) < P.walk_rho);
        walk_s = !(unit64(mix.y) < P.walk_rho);
    }
    for (int t = 1; t <= L && walk_p; ++t) {
        const uint4 r = philox4x32_10(make_uint4((uint32_t)mv, (uint32_t)n, (uint32_t)w, (uint32_t)(1 + t)), key);
        const int j = (int)(((uint64_t)r.x * (uint64_t)NO) >> 32);
        if (unit64(r.y) * a[p] <= a[j]) p = j;
    }
    int s = (int)(((uint64_t)w1 * (uint64_t)(NO - 1)) >> 32);
    s += (s >= p);
    for (int t = 1; t <= L && walk_s; ++t) {
        const uint4 r = philox4x32_10(make_uint4((uint32_t)mv, (uint32_t)n, (uint32_t)w, (uint32_t)(1 + t)), key);
        int j = (int)(((uint64_t)r.z * (uint64_t)(NO - 1)) >> 32);
        j += (j >= p);
        if (unit64(r.w) * a[s] <= a[j]) s = j;
    }
    p_out = p;
    s_out = s;
}

// What a move needs besides the state, drawn by one lane for one of the next 32 moves (the
// divisions of the two deltas cost the FP64 pipe one instruction for 32 moves instead of one each).
struct Ring64 {
    double eps[32], dp[32], ds[32], u[32];
    double hl[32];        // Hastings: (N - 4) ln r, or NaN where the reverse move cannot be proposed
    float lnu[32];        // -ln u
    int p[32], s[32];     // the bins (without an index walk)
};

// A warp's shared memory: its draws, the terms of delta chi2 on their way to the ordered sum, and the
// spectrum if it is staged.
__host__ __device__ __forceinline__ size_t sweep64_warp_bytes(bool staged, int n_omega, int C) {
    return sizeof(Ring64) + (size_t)(32 * C) * 8 + (staged ? (size_t)n_omega * 8 : 0);
}

// One warp per walker; every state value and every decision is the oracle's bit for bit.  The FP64
// pipe answers after some 60 cycles, so the chain of a move was its ordered sum of n_tau additions
// (needed only where the decision is close: see below), two divisions and an exponential in FP64, and
// the L2 latency of a[p] and a[s].  Now the draws are made 32 moves at a time, the spectrum is staged
// in shared memory where it fits, the next move's columns are loaded during the reduction, and a
// butterfly sum and FP32 take the clear decisions.  chi2 is not tracked: every sweep launch is
// followed by its recomputation.  32 tau x 64 bins x 64 walkers, per move: 3.87 us -> 1.1 us.
template <int C, bool STAGED>
__global__ void __launch_bounds__(128) sweep_fp64_kernel(DevProblem P, DevState S, int n0, int n1) {
    extern __shared__ double s_mem64[];
    const int lane = threadIdx.x & 31;
    const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (w >= P.n_walkers) return;
    const int NT = P.n_tau, NO = P.n_omega, PAD = P.n_tau_pad;
    char *mem = reinterpret_cast<char *>(s_mem64) + (threadIdx.x >> 5) * sweep64_warp_bytes(STAGED, NO, C);
    Ring64 &ring = *reinterpret_cast<Ring64 *>(mem);
    double *s_t = reinterpret_cast<double *>(mem + sizeof(Ring64));
    double *ag = S.a64 + (size_t)w * NO;
    double *a = STAGED ? s_t + 32 * C : ag;
    if constexpr (STAGED)
        for (int j = lane; j < NO; j += 32) a[j] = ag[j];
    double R[C], Fh[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
        R[c] = S.R64[(size_t)w * PAD + lane + 32 * c];
        Fh[c] = P.Fhat64[lane + 32 * c];
    }
    int accp = S.acc_prev[w];
    unsigned long long h = S.hash[w], nacc = 0, npos = 0;
    const uint2 key = philox_key(P.seed);
    const double dmove = P.move_scale > 0.0 ? P.move_scale : 1.0 / NO;
    const int wg = w + P.walker_base;   // the walker's index in the whole population
    const bool walk = P.walk_len > 0;
    constexpr bool AHEAD = C <= 4;      // the next move's columns in registers

    // delta_p, delta_s of Eqs. (update-delta-p/s)
    auto deltas64 = [&](double eps, int p, int s, double &dp, double &ds) {
        const double xp = P.x64[p], xs = P.x64[s];
        dp = eps * (P.B - P.A * xs) / (xp - xs);
        ds = eps * (P.B - P.A * xp) / (xs - xp);
    };
    for (int n = n0; n < n1; ++n) {
        const double T = P.Tsweep[n];
        const float inv_T = (float)(1.0 / T);
        const double y = amplitude(accp, NO, P.y_p, P.y_m, P.y_min);
        int acc = 0;
        for (int base = 0; base < NO; base += 32) {
            const int count = min(32, NO - base);
            __syncwarp();
            if (lane < count) {
                const int mv = base + lane;
                const uint4 rnd = philox4x32_10(make_uint4((uint32_t)mv, (uint32_t)n, (uint32_t)wg, 0u), key);
                const double eps = (y * dmove) * (2.0 * unit64(rnd.z) - 1.0);
                const double u = unit64(rnd.w);
                ring.eps[lane] = eps;
                ring.u[lane] = u;
                ring.lnu[lane] = -logf((float)u);
                if (!walk) {
                    // shared bins: the group's first walker's words 0 and 1 (its own counter)
                    uint2 bw = make_uint2(rnd.x, rnd.y);
                    if (P.shared_bins > 1 && wg % P.shared_bins != 0) {
                        const uint4 g = philox4x32_10(
                            make_uint4((uint32_t)mv, (uint32_t)n, (uint32_t)(wg - wg % P.shared_bins), 0u), key);
                        bw = make_uint2(g.x, g.y);
                    }
                    int p, s;
                    move_bins(bw.x, bw.y, NO, p, s);
                    double dp, ds;
                    deltas64(eps, p, s, dp, ds);
                    ring.dp[lane] = dp;
                    ring.ds[lane] = ds;
                    ring.p[lane] = p;
                    ring.s[lane] = s;
                }
                if (P.hastings) {
                    // the move's Jacobian r^(N-4), the reverse amplitude -eps/r proposable only when
                    // |eps/r| < y d (the oracle's or_accept)
                    const double r = 1.0 - eps;
                    ring.hl[lane] = fabs(eps / r) < y * dmove ? (double)(NO - 4) * log(r) : NAN;
                }
            }
            __syncwarp();
            double Kp[C], Ks[C];
            auto load_columns = [&](int p, int s) {
                const double *kp = P.Khat64 + (size_t)p * PAD, *ks = P.Khat64 + (size_t)s * PAD;
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    Kp[c] = kp[lane + 32 * c];
                    Ks[c] = ks[lane + 32 * c];
                }
            };
            if (AHEAD && !walk) load_columns(ring.p[0], ring.s[0]);
            for (int i = 0; i < count; ++i) {
                const double eps = ring.eps[i], r = 1.0 - eps;
                double dp, ds;
                int p, s;
                if (walk) {
                    const int mv = base + i;
                    const uint4 rnd = philox4x32_10(make_uint4((uint32_t)mv, (uint32_t)n, (uint32_t)wg, 0u), key);
                    walk_bins64(P, a, rnd.x, rnd.y, mv, n, wg, key, p, s);
                    deltas64(eps, p, s, dp, ds);
                } else {
                    dp = ring.dp[i];
                    ds = ring.ds[i];
                    p = ring.p[i];
                    s = ring.s[i];
                }
                if (!AHEAD || walk) load_columns(p, s);
                const double ap = r * a[p] + dp;
                const double as = r * a[s] + ds;
                unsigned code;
                if (ap < 0.0 || as < 0.0) {
                    if (AHEAD && !walk && i + 1 < count) load_columns(ring.p[i + 1], ring.s[i + 1]);
                    code = 2;
                    ++npos;
                } else {
                    double d[C], t[C];
                    double D = 0.0;              // sum in butterfly order; the decision's own unless it is close
                    float mag = 0.0f;            // sum of the terms' magnitudes
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        const double M = Fh[c] - R[c];
                        d[c] = eps * M - dp * Kp[c] - ds * Ks[c];
                        t[c] = d[c] * (2.0 * R[c] + d[c]);
                        D = D + t[c];
                        mag += fabsf((float)t[c]);
                    }
                    if (AHEAD && !walk && i + 1 < count) load_columns(ring.p[i + 1], ring.s[i + 1]);
                    for (int o = 16; o > 0; o >>= 1) {
                        D = D + __shfl_xor_sync(kFull, D, o);
                        mag += __shfl_xor_sync(kFull, mag, o);
                    }
                    // accept with probability min(1, exp(-D / T)) (Hastings: times r^(N-4)).  The sums in
                    // two orders differ by at most n_tau 2^-53 of the terms' magnitudes (512 points:
                    // 6e-14) and FP32 rounds x = D / T and -ln u (+ (N-4) ln r) to about 1e-7 of
                    // themselves; where the decision lies outside both it is taken, else the terms
                    // are added in the oracle's order and the test is evaluated in FP64.
                    const double hl = P.hastings ? ring.hl[i] : 0.0;
                    const float Df = (float)D, close = 1e-12f * mag;
                    const float x = Df * inv_T, lnu = ring.lnu[i], hf = (float)hl, gap = x - (lnu + hf);
                    const float tol = 1e-5f * (fabsf(x) + lnu + fabsf(hf)) + 1e-6f + close * inv_T;
                    bool accept;
                    if (hl != hl) {
                        accept = false;
                    } else if (!P.hastings && Df < -close) {
                        accept = true;
                    } else if (fabsf(gap) > tol && (P.hastings || Df > close)) {
                        accept = gap < 0.0f;
                    } else {
#pragma unroll
                        for (int c = 0; c < C; ++c) s_t[lane + 32 * c] = t[c];
                        __syncwarp();
                        D = 0.0;
                        for (int q = 0; q < NT; ++q) D = D + s_t[q];
                        if (!P.hastings) accept = D <= 0.0 || ring.u[i] < exp(-D / T);
                        else accept = ring.u[i] < exp(-D / T + hl);
                    }
                    if (accept) {
                        for (int j = lane; j < NO; j += 32) a[j] = r * a[j];
                        __syncwarp();
                        if (lane == 0) {
                            a[p] = ap;
                            a[s] = as;
                        }
#pragma unroll
                        for (int c = 0; c < C; ++c) R[c] = R[c] + d[c];
                        ++acc;
                        code = 1;
                    } else {
                        code = 0;
                    }
                    __syncwarp();
                }
                h = (h ^ code) * kFnvPrime;
            }
        }
        accp = acc;
        nacc += acc;
        if (S.acc_trace && lane == 0) S.acc_trace[(size_t)n * P.n_walkers + w] = acc;
    }
    if constexpr (STAGED) {
        __syncwarp();
        for (int j = lane; j < NO; j += 32) ag[j] = a[j];
    }
#pragma unroll
    for (int c = 0; c < C; ++c) S.R64[(size_t)w * PAD + lane + 32 * c] = R[c];
    if (lane == 0) {
        S.acc_prev[w] = accp;
        S.hash[w] = h;
        S.n_acc[w] += nacc;
        S.n_pos[w] += npos;
    }
}

// ------------------------------------------------------------------ residual recomputation
// R_i = Fhat_i - sum_j Khat_ij a_j with j ascending, chi2 = sum_i R_i^2 with i ascending.
// One block per walker.  FP32 state enters as (double) b_j; the sweep kernel folds its
// common scale into b before this runs.
//
// FP32 state only: rounding in the moves lets sum a and sum a x wander by ~1e-6 of A and B
// over a resync interval (exact arithmetic keeps them fixed, Sec. 2.2), so before the residual
// is formed each walker is put back on both sum rules with the
// affine reweighting b_j <- b_j kappa (1 + lambda (x_j - c)): c = B'/A', kappa = A / A',
// lambda = (B/A - c) / var', where A' = sum b, B' = sum b x and var' = sum b x^2 / A' - c^2 are
// the walker's current moments (lambda = 0 if the tilt could make a factor negative).  One
// warp per walker, one pass for the moments: FP32 per bin, in the offset t_j = x_j - x_mid =
// (j - (N-1)/2) dw from the grid's midpoint (uniform bins), with compensated per-lane sums and
// FP64 across lanes; the factor is applied in FP32, the state's own precision (FP64 runs at a
// small fraction of the FP32 rate on this GPU).
__device__ __forceinline__ void kahan_add(float &s, float &comp, float v) {
    const float y = v - comp;
    const float t = s + y;
    comp = (t - s) - y;
    s = t;
}

// The three BF16 pieces (each the round-to-nearest BF16 of what is left) of 8 consecutive
// spectrum values for the tensor-copy recomputation, stored as three 16-byte rows at
// [piece][walker][bin] of At (v past the last bin is 0).
__device__ __forceinline__ void put_pieces8(unsigned short *At, size_t plane, size_t at, const float (&v)[8]) {
    uint32_t w1[4], w2[4], w3[4];
#pragma unroll
    for (int e = 0; e < 8; e += 2) {
        uint32_t p1[2], p2[2], p3[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const __nv_bfloat16 b1 = __float2bfloat16_rn(v[e + h]);
            const float r = v[e + h] - __bfloat162float(b1);
            const __nv_bfloat16 b2 = __float2bfloat16_rn(r);
            const __nv_bfloat16 b3 = __float2bfloat16_rn(r - __bfloat162float(b2));
            p1[h] = __bfloat16_as_ushort(b1);
            p2[h] = __bfloat16_as_ushort(b2);
            p3[h] = __bfloat16_as_ushort(b3);
        }
        w1[e / 2] = p1[0] | (p1[1] << 16);
        w2[e / 2] = p2[0] | (p2[1] << 16);
        w3[e / 2] = p3[0] | (p3[1] << 16);
    }
    *reinterpret_cast<uint4 *>(At + at) = make_uint4(w1[0], w1[1], w1[2], w1[3]);
    *reinterpret_cast<uint4 *>(At + plane + at) = make_uint4(w2[0], w2[1], w2[2], w2[3]);
    *reinterpret_cast<uint4 *>(At + 2 * plane + at) = make_uint4(w3[0], w3[1], w3[2], w3[3]);
}

// At (optional): also write the restored spectra's BF16 pieces for the tensor-copy
// recomputation, rows of nop bins, planes of `plane` elements (the padding stays zero).
__global__ void __launch_bounds__(256) restore_kernel(DevProblem P, DevState S, unsigned short *At, int nop,
                                                      size_t plane) {
    const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (w >= P.n_walkers) return;
    float *b = S.b32 + (size_t)w * P.n_omega;
    const float dw = (float)P.dw, half = 0.5f * (float)(P.n_omega - 1);
    float a0 = 0.f, c0 = 0.f, a1 = 0.f, c1 = 0.f, a2 = 0.f, c2 = 0.f;
    for (int j = lane; j < P.n_omega; j += 32) {
        const float v = b[j], xj = ((float)j - half) * dw;
        kahan_add(a0, c0, v);
        kahan_add(a1, c1, v * xj);
        kahan_add(a2, c2, v * xj * xj);
    }
    double s0 = (double)a0 - (double)c0, s1 = (double)a1 - (double)c1, s2 = (double)a2 - (double)c2;
    for (int o = 16; o > 0; o >>= 1) {
        s0 += __shfl_xor_sync(0xFFFFFFFFu, s0, o);
        s1 += __shfl_xor_sync(0xFFFFFFFFu, s1, o);
        s2 += __shfl_xor_sync(0xFFFFFFFFu, s2, o);
    }
    if (s0 > 0.0) {
        const double xmid = 0.5 * (P.x64[0] + P.x64[P.n_omega - 1]);
        const double c = s1 / s0;                               // centre, as an offset from xmid
        const double var = s2 / s0 - c * c;
        const double kappa = P.A / s0;
        double lambda = var > 0.0 ? (P.B / P.A - xmid - c) / var : 0.0;
        if (!(fabs(lambda * (P.n_omega - 1) * P.dw) < 0.5)) lambda = 0.0;
        const float kf = (float)kappa, lk = (float)(kappa * lambda), cf = (float)c;
        for (int j = lane; j < P.n_omega; j += 32) {
            const float xj = ((float)j - half) * dw;
            b[j] = b[j] * fmaf(lk, xj - cf, kf);
        }
    }
    if (!At) return;
    // the pieces of the restored spectrum, 8 bins a lane (16-byte stores)
    __syncwarp();
    const size_t row = (size_t)w * nop;
    for (int j0 = 8 * lane; j0 < P.n_omega; j0 += 256) {
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = j0 + e < P.n_omega ? b[j0 + e] : 0.0f;
        put_pieces8(At, plane, row + j0, v);
    }
}

__global__ void __launch_bounds__(128) resync_kernel(DevProblem P, DevState S, int precision) {
    __shared__ double Rs[kMaxTau];
    const int w = blockIdx.x;
    const int NO = P.n_omega, PAD = P.n_tau_pad;
    for (int i = threadIdx.x; i < PAD; i += blockDim.x) {
        double r = 0.0;
        if (i < P.n_tau) {
            double model = 0.0;
            if (precision == 0) {
                const double *a = S.a64 + (size_t)w * NO;
                for (int j = 0; j < NO; ++j) model = model + P.Khat64[(size_t)j * PAD + i] * a[j];
            } else {
                const float *b = S.b32 + (size_t)w * NO;
                for (int j = 0; j < NO; ++j) model = model + P.Khat64[(size_t)j * PAD + i] * (double)b[j];
            }
            r = P.Fhat64[i] - model;
        }
        Rs[i] = r;
        if (precision == 0) S.R64[(size_t)w * PAD + i] = r;
        else S.R32[(size_t)w * PAD + i] = (float)r;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double c2 = 0.0;
        for (int i = 0; i < P.n_tau; ++i) c2 = c2 + Rs[i] * Rs[i];
        S.chi2[w] = c2;
    }
}

// ------------------------------------------------------------------ branching (Sec. 2.5)
// Walker l has weight w_l = exp[-Delta (z_l - P_r)], z_l = (chi2_l - min) / (mean - min), and
// multiplier m_l = floor(w_l + xi_l).  Writing Theta = exp(Delta P_r) and E_l = exp(-Delta z_l),
// m_l = floor(Theta E_l + xi_l), which steps up by one at each "break point"
// Delta z_l + ln(k - xi_l) = ln Theta, k = 1, 2, ...  P_r is fixed by sum m = N: ln Theta lies
// between the N-th and (N+1)-th smallest break points of all walkers, found by bisection on
// ln Theta until the count is exactly N.  Z(Delta) = #{m_l = 0}; Delta doubles from 1 until
// Z >= round(f N), then bisects, stopping at the first Delta with Z = round(f N).
struct SolveShared {
    double red_d[32];
    int red_i[32];
    double bcast_d;
    int bcast_i;
    double theta;
    double cmin, spread;
    int scan[kSolveThreads / 32];
};

__device__ double block_sum_d(double v, SolveShared &sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) sh.red_d[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = lane < (int)(blockDim.x >> 5) ? sh.red_d[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
        if (lane == 0) sh.bcast_d = v;
    }
    __syncthreads();
    return sh.bcast_d;
}

__device__ int block_sum_i(int v, SolveShared &sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) sh.red_i[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = lane < (int)(blockDim.x >> 5) ? sh.red_i[lane] : 0;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
        if (lane == 0) sh.bcast_i = v;
    }
    __syncthreads();
    return sh.bcast_i;
}

// Exclusive prefix sum over the block in thread order; returns this thread's offset and
// writes the total to *total.
__device__ int block_scan_excl(int v, int *total, SolveShared &sh) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int incl = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
    }
    __syncthreads();
    if (lane == 31) sh.scan[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int nw = (int)(blockDim.x >> 5);
        int x = lane < nw ? sh.scan[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(kFull, x, o);
            if (lane >= o) x += t;
        }
        if (lane < nw) sh.scan[lane] = x;  // inclusive over warps
    }
    __syncthreads();
    const int warp_off = warp > 0 ? sh.scan[warp - 1] : 0;
    *total = sh.scan[(blockDim.x >> 5) - 1];
    return warp_off + incl - v;
}

// Multipliers at one Delta; returns Z.  Walker l = threadIdx.x + kSolveThreads * q, q < PT.
template <int PT>
__device__ int multipliers_at(int N, const double *z, const double *xi, double Delta, int *m,
                              SolveShared &sh) {
    const int tid = threadIdx.x;
    double E[PT];
    double sE = 0.0;
#pragma unroll
    for (int q = 0; q < PT; ++q) {
        const int l = tid + kSolveThreads * q;
        E[q] = l < N ? exp(-Delta * z[q]) : 0.0;
        sE += E[q];
    }
    sE = block_sum_d(sE, sh);
    auto count_at = [&](double lnTheta, bool store) -> int {
        if (tid < 32) {
            const double Th = exp(lnTheta);
            if (tid == 0) sh.theta = Th;
        }
        __syncthreads();
        const double Th = sh.theta;
        int c = 0;
#pragma unroll
        for (int q = 0; q < PT; ++q) {
            const int l = tid + kSolveThreads * q;
            int mq = 0;
            if (l < N) {
                const double v = floor(Th * E[q] + xi[q]);
                mq = v >= (double)N ? N : (int)v;
            }
            if (store) m[q] = mq;
            c += mq;
        }
        return block_sum_i(c, sh);
    };
    // Sum m is close to Theta * sum E; bracket ln Theta around ln(N / sum E).
    const double guess = log((double)N / sE);
    double lo = guess - 0.25, hi = guess + 0.25;
    int clo = count_at(lo, false), chi = count_at(hi, false);
    for (int it = 0; it < 200 && clo >= N; ++it) { lo -= (hi - lo); clo = count_at(lo, false); }
    for (int it = 0; it < 200 && chi < N; ++it) { hi += (hi - lo); chi = count_at(hi, false); }
    bool hit = false;
    for (int it = 0; it < 200; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (!(mid > lo && mid < hi)) break;
        const int c = count_at(mid, true);
        if (c == N) { hit = true; break; }
        if (c < N) lo = mid; else hi = mid;
    }
    if (!hit) {
        // Break points tied at ln Theta: take the upper end and drop the surplus copies
        // from the highest walker indices whose count rises across the final bracket.
        int c = count_at(hi, true);
        int mlo[PT];
        {
            if (tid < 32) { const double Th = exp(lo); if (tid == 0) sh.theta = Th; }
            __syncthreads();
            const double Th = sh.theta;
#pragma unroll
            for (int q = 0; q < PT; ++q) {
                const int l = tid + kSolveThreads * q;
                const double v = l < N ? floor(Th * E[q] + xi[q]) : 0.0;
                mlo[q] = v >= (double)N ? N : (int)v;
            }
            __syncthreads();
        }
        for (int q = PT - 1; q >= 0 && c > N; --q) {
            for (int t = kSolveThreads - 1; t >= 0 && c > N; --t) {
                // serial over walkers in descending index order; thread t owns walker l
                if (tid == t) {
                    const int l = t + kSolveThreads * q;
                    int take = 0;
                    if (l < N) {
                        const int extra = m[q] - mlo[q];
                        take = extra < (c - N) ? extra : (c - N);
                        m[q] -= take;
                    }
                    sh.bcast_i = take;
                }
                __syncthreads();
                c -= sh.bcast_i;
                __syncthreads();
            }
        }
    }
    int zc = 0;
#pragma unroll
    for (int q = 0; q < PT; ++q) {
        const int l = tid + kSolveThreads * q;
        zc += (l < N && m[q] == 0);
    }
    return block_sum_i(zc, sh);
}

// The sum of the walkers' residues in walker order, every partial sum rounded as one FP64 addition
// rounds it, by a whole block.  While the running sum stays in one binade it is an integer S in units
// of its last place, and adding c adds an integer to S: c in that unit, rounded to nearest, a tie to
// the even sum.  A step is then what S grows by if it is even and if it is odd; steps compose, so a
// scan over the walkers gives S at every walker up to the one whose addition leaves the binade, and
// that addition is done as such.  One thread's chain of additions (some 60 cycles each) took 0.53 ms
// at 16384 walkers (block of 512 x 2048, 10 sweeps: 14.80 -> 15.32 ms); this takes a scan for every
// doubling of the sum past its first 32 terms, over a little more than the walkers that double it
// (14.90 ms; one solve of 1023 walkers 11 us).
struct SumStep { unsigned long long even, odd; };
constexpr unsigned long long kSumTop = 1ull << 53;      // S leaves the binade
__host__ __device__ __forceinline__ SumStep sum_then(SumStep a, SumStep b) {
    // saturated well past the binade, where the parity no longer matters
    const unsigned long long e = a.even + (a.even & 1 ? b.odd : b.even), o = a.odd + (a.odd & 1 ? b.even : b.odd);
    return {e < 2 * kSumTop ? e : 2 * kSumTop, o < 2 * kSumTop ? o : 2 * kSumTop};
}
// The step of adding c >= 0 (its bits) to a sum whose biased exponent is e.
__host__ __device__ __forceinline__ SumStep sum_step(unsigned long long c, int e) {
    const int k = (int)(c >> 52) & 0x7FF;
    const unsigned long long m = (c & (kSumTop / 2 - 1)) | (k ? kSumTop / 2 : 0);
    const int low = e - (k ? k : 1);                    // places of c below the sum's last
    if (low <= 0) {
        const unsigned long long q = low < -1 ? 2 * kSumTop : m << -low;
        return {q, q};
    }
    if (low > 53) return {0, 0};
    const unsigned long long q = m >> low, rest = m & ((1ull << low) - 1), half = 1ull << (low - 1);
    if (rest == half) return {q + (q & 1), q + ((q + 1) & 1)};
    return {q + (rest > half), q + (rest > half)};
}
// Where walker l's residue stands in shared memory: threads that read 2^k consecutive ones meet different
// banks.
__host__ __device__ __forceinline__ int sum_at(int l) { return l + (l >> 4); }

constexpr int kSumWarps = 8;                           // a scan is short: more warps wait longer for one another
struct SumShared {
    double s;            // the sum of the first `at` residues
    int at;
    SumStep warp[kSumWarps];
};
// c: N residues at sum_at(l), stored by all threads before a barrier.  Values that are not residues (NaN,
// negative, huge) and sums below the normal range are added one by one.
__device__ double ordered_sum(const double *c, int N, SumShared &sh) {
    constexpr int kThreads = 32 * kSumWarps;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    bool plain = true;
    for (int l = tid; l < N; l += kSolveThreads) plain = plain && c[sum_at(l)] >= 0.0 && c[sum_at(l)] <= 1e300;
    const bool scan = __syncthreads_and(plain);
    if (tid == 0) {
        double s = 0.0;
        const int n = scan ? min(N, 32) : N;
        for (int l = 0; l < n; ++l) s += c[sum_at(l)];
        if (!(s >= 1e-290))
            for (int l = n; l < N; ++l) s += c[sum_at(l)];
        sh.s = s;
        sh.at = s >= 1e-290 ? n : N;
    }
    auto barrier = [] { asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory"); };
    while (warp < kSumWarps) {
        barrier();
        const double s = sh.s;
        const int at = sh.at;
        if (at >= N) break;
        const unsigned long long bits = __double_as_longlong(s);
        const int e = (int)(bits >> 52);
        const unsigned long long S = (bits & (kSumTop / 2 - 1)) | kSumTop / 2;
        // this scan: the walkers up to `end`, each thread some of them
        const int end = min(N, at + max(kThreads, at + at / 4)), per = (end - at + kThreads - 1) / kThreads;
        const int first = min(end, at + tid * per), last = min(end, first + per);
        SumStep own = {0, 0};
        for (int l = first; l < last; ++l) own = sum_then(own, sum_step(__double_as_longlong(c[sum_at(l)]), e));
        SumStep incl = own;
        auto up = [&](SumStep v, int o) -> SumStep { return {__shfl_up_sync(kFull, v.even, o), __shfl_up_sync(kFull, v.odd, o)}; };
        for (int o = 1; o < 32; o <<= 1) {
            const SumStep t = up(incl, o);
            if (lane >= o) incl = sum_then(t, incl);
        }
        if (lane == 31) sh.warp[warp] = incl;
        SumStep before = up(incl, 1);
        if (lane == 0) before = {0, 0};
        barrier();
        SumStep all = {0, 0}, off = {0, 0};
        for (int k = 0; k < kSumWarps; ++k) {
            if (k == warp) off = all;
            all = sum_then(all, sh.warp[k]);
        }
        before = sum_then(off, before);
        const SumStep after = sum_then(before, own);
        auto at_S = [S](SumStep v) { return S + (S & 1 ? v.odd : v.even); };
        auto value = [e](unsigned long long v) { return __longlong_as_double(((unsigned long long)e << 52) | (v & (kSumTop / 2 - 1))); };
        if (at_S(before) < kSumTop && at_S(after) >= kSumTop) {
            unsigned long long v = at_S(before);
            for (int l = first; l < last; ++l) {
                const SumStep step = sum_step(__double_as_longlong(c[sum_at(l)]), e);
                const unsigned long long next = v + (v & 1 ? step.odd : step.even);
                if (next >= kSumTop) {
                    sh.s = value(v) + c[sum_at(l)];
                    sh.at = l + 1;
                    break;
                }
                v = next;
            }
        } else if (tid == 0 && at_S(all) < kSumTop) {
            sh.s = value(at_S(all));
            sh.at = end;
        }
    }
    __syncthreads();
    return sh.s;
}

// The whole solve in one block: the search over Delta is sequential, and a trial is cheap because
// FP32 decides nearly every multiplier.  At a trial Delta each thread holds e^(-Delta z_l) in FP32
// with a bound on its error; a count of sum m at some Theta forms Theta E + xi in FP32 and goes to
// FP64 (the arithmetic of multipliers_at) only for a walker whose value lies within that bound of
// an integer, about one in 1e5.  So every count is the FP64 count, and since each m_l rises with
// Theta, the multipliers with sum N are the same whichever Theta with that sum is found; the
// Theta search may therefore interpolate in FP32, and needs 5 to 8 counts.  Where no FP32 Theta has
// sum N (ties, or two break points within 6e-8) multipliers_at decides.  The FP64 pipe (2 lanes a
// clock and SM: one FP64 instruction of all 32 warps is 512 cycles) is what a solve in FP64 waits
// for, so FP64 is kept to the walkers' differences from the smallest chi2 and to one warp's
// scalars.  Against one block per speculative trial in FP64 (23 launches; the same multipliers):
// 1013 -> 105 us at 4096 walkers, 4050 -> 522 us at 16384, 350 -> 62 us at 1500, 220 -> 28 us at 64
// (first block of an anneal, the mean summed over threads; its ordered sum, above, comes on top).
constexpr float kSolveErr = 3e-7f;     // rounding of Theta E + xi and of xi, absolute part

template <int PT>
__device__ __noinline__ int multipliers_tied(int N, const double *chi2, double cmin, double spread, const uint32_t *word,
                                             double Delta, int *m, SolveShared &sh) {
    double z[PT], xi[PT];
#pragma unroll
    for (int q = 0; q < PT; ++q) {
        const int l = threadIdx.x + kSolveThreads * q;
        z[q] = l < N && spread > 0.0 ? (chi2[l] - cmin) / spread : 0.0;
        xi[q] = l < N ? unit64(word[l]) : 0.5;
    }
    return multipliers_at<PT>(N, z, xi, Delta, m, sh);
}

// One walker's multiplier in FP64, as multipliers_at forms it.
__device__ __noinline__ int multiplier64(float Theta, double Delta, double chi2, double cmin, double spread, uint32_t word, int N) {
    const double z = spread > 0.0 ? (chi2 - cmin) / spread : 0.0;
    const double v = floor((double)Theta * exp(-Delta * z) + unit64(word));
    return v >= (double)N ? N : (int)v;
}

// Sums of a and b over the block, the same in every thread (one barrier; red alternates).
template <typename T>
__device__ __forceinline__ T block_sum1(T v, T (*red)[32], int buf) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    if ((threadIdx.x & 31) == 0) red[buf][threadIdx.x >> 5] = v;
    __syncthreads();
    v = red[buf][threadIdx.x & 31];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}
__device__ __forceinline__ int2 block_sum2(int a, int b, int2 (*red)[32], int &buf) {
    a = __reduce_add_sync(kFull, a);
    b = __reduce_add_sync(kFull, b);
    if ((threadIdx.x & 31) == 0) red[buf][threadIdx.x >> 5] = make_int2(a, b);
    __syncthreads();
    const int2 v = red[buf][threadIdx.x & 31];
    buf ^= 1;
    return make_int2(__reduce_add_sync(kFull, v.x), __reduce_add_sync(kFull, v.y));
}

// The search over Delta, advanced by one warp: Delta doubles from 1 until Z >= the target, at
// most 64 times, then bisects, at most 64 times, and stops at the first Z equal to the target.
struct SolveSearch {
    double lo, hi, D;
    int doublings, halvings, state;    // 0 doubling, 1 bisecting, 2 done (D is the result)
    __device__ void begin() { lo = 0.0; hi = D = 1.0; doublings = halvings = state = 0; }
    __device__ void next(int Z, int Zt) {
        if (state == 0) {
            if (Z < Zt && doublings < 64) {
                lo = hi;
                hi = D = 2.0 * hi;
                ++doublings;
                return;
            }
            state = 1;
            if (Z == Zt) { state = 2; return; }
        } else {
            if (Z == Zt) { state = 2; return; }
            if (Z < Zt) lo = D; else hi = D;
        }
        const double mid = 0.5 * (lo + hi);
        if (halvings >= 64 || mid <= lo || mid >= hi) {
            D = hi;
            state = 2;
            return;
        }
        D = mid;
        ++halvings;
    }
};

template <int PT>
__global__ void __launch_bounds__(kSolveThreads, 1) branch_solve_kernel(DevProblem P, DevState S, BranchScratch B, int block_index,
                                                                        double fraction, int event) {
    extern __shared__ double s_chi2[];           // chi2 for the ordered sum; then z [N] and the draws [N]
    __shared__ SolveShared sh;
    __shared__ SolveSearch s_search;
    __shared__ SumShared s_sum;
    __shared__ int2 red[2][32];
    __shared__ float red_f[2][32];
    const int N = P.n_walkers, tid = threadIdx.x;
    float *s_z = reinterpret_cast<float *>(s_chi2);
    uint32_t *s_word = reinterpret_cast<uint32_t *>(s_z + N);
    int Zt = (int)floor(fraction * N + 0.5);
    if (Zt > N - 1) Zt = N - 1;
    double cmin = S.chi2[0];
    for (int l = tid; l < N; l += kSolveThreads) {
        const double c = S.chi2[l];
        s_chi2[sum_at(l)] = c;
        cmin = c < cmin ? c : cmin;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const double c = __shfl_xor_sync(kFull, cmin, o);
        cmin = c < cmin ? c : cmin;
    }
    if ((tid & 31) == 0) sh.red_d[tid >> 5] = cmin;
    __syncthreads();
    cmin = sh.red_d[tid & 31];
    for (int o = 16; o > 0; o >>= 1) {
        const double c = __shfl_xor_sync(kFull, cmin, o);
        cmin = c < cmin ? c : cmin;
    }
    // the mean, summed in the oracle's order: where the residues lie close together, z hangs on its last bits
    const double csum = ordered_sum(s_chi2, N, s_sum);
    const double spread = csum / N - cmin;
    const double scale = spread > 0.0 ? 1.0 / spread : 0.0;    // FP64: residues and mean may leave FP32's range, z does not
    const uint2 key = philox_key(P.seed);
    __syncthreads();
    float xif[PT], E[PT];                        // this thread's walkers: draws, and E at the trial Delta
    int m[PT];
#pragma unroll
    for (int q = 0; q < PT; ++q) {
        const int l = tid + kSolveThreads * q;
        E[q] = 0.0f;
        xif[q] = 0.5f;
        m[q] = 1;
        if (l < N) {
            const uint32_t w = philox4x32_10(make_uint4((uint32_t)(l + P.walker_base), (uint32_t)block_index, 0u, 1u), key).x;
            s_z[l] = (float)(scale * (S.chi2[l] - cmin));
            s_word[l] = w;
            xif[q] = fmaf((float)w, 2.3283064e-10f, 1.1641532e-10f);
        }
    }
    int buf = 0, fbuf = 0;
    float Theta = 0.0f;                          // of the last trial: sum m = N
    bool tied = false;
    double Delta = 0.0;
    float Df = 0.0f;
    // multiplier of walker q of this thread at Theta
    auto mult = [&](int q, float Th) -> int {
        const int l = tid + kSolveThreads * q;
        if (l >= N) return 0;
        const float v = fmaf(Th, E[q], xif[q]);
        // E's relative error: the exponent's rounding (4e-7 of it) and expf's
        const float tol = fmaf(v, fmaf(4e-7f, Df * s_z[l], 2e-6f), kSolveErr);
        const float lo = floorf(v - tol), hi = floorf(v + tol);
        if (lo == hi && hi < 1e6f) return min((int)lo, N);
        return multiplier64(Th, Delta, S.chi2[l], cmin, spread, s_word[l], N);
    };
    auto count = [&](float Th) -> int2 {         // (sum m, zero multipliers)
        int c = 0, zc = 0;
#pragma unroll
        for (int q = 0; q < PT; ++q) {
            const int k = mult(q, Th);
            c += k;
            zc += (k == 0 && tid + kSolveThreads * q < N);
        }
        return block_sum2(c, zc, red, buf);
    };
    // Z at the trial Delta; leaves Theta (or, tied, the multipliers in m)
    auto trial = [&]() -> int {
        tied = false;
        float sE = 0.0f;
#pragma unroll
        for (int q = 0; q < PT; ++q) {
            const int l = tid + kSolveThreads * q;
            E[q] = l < N ? expf(-Df * s_z[l]) : 0.0f;
            sE += E[q];
        }
        const float guess = (float)N / block_sum1(sE, red_f, fbuf);
        fbuf ^= 1;
        float lo = 0.9f * guess, hi = 1.1f * guess;
        int2 clo = count(lo), chi = count(hi);
        for (int it = 0; it < 100 && clo.x >= N; ++it) { lo *= 0.5f; clo = count(lo); }
        for (int it = 0; it < 100 && chi.x < N; ++it) { hi *= 2.0f; chi = count(hi); }
        if (clo.x < N && chi.x == N) { Theta = hi; return chi.y; }
        for (int it = 0; it < 200; ++it) {
            float mid = 0.5f * (lo + hi);
            if (it % 3 != 2 && chi.x > clo.x) {
                const float at = fmaf(hi - lo, ((float)(N - clo.x) + 0.5f) / (float)(chi.x - clo.x), lo);
                if (at > lo && at < hi) mid = at;
            }
            if (!(mid > lo && mid < hi)) break;
            const int2 c = count(mid);
            if (c.x == N) { Theta = mid; return c.y; }
            if (c.x < N) { lo = mid; clo = c; } else { hi = mid; chi = c; }
        }
        tied = true;
        return multipliers_tied<PT>(N, S.chi2, cmin, spread, s_word, Delta, m, sh);
    };

    double result = 0.0;
    if (Zt > 0) {
        if (tid == 0) s_search.begin();
        __syncthreads();
        int Z = 0;
        for (;;) {
            const double D = s_search.D;
            const int state = s_search.state;
            if (state == 2) {
                result = D;
                if (D == Delta) break;           // the last trial was at the result
            }
            Delta = D;
            Df = __double2float_rn(D);
            Z = trial();
            if (state == 2) break;
            __syncthreads();
            if (tid == 0) s_search.next(Z, Zt);
            __syncthreads();
        }
        if (!tied) {
#pragma unroll
            for (int q = 0; q < PT; ++q) m[q] = mult(q, Theta);
        }
    }
    // the imprint pairing: zero-multiplier walkers ascending, matched with surplus copies (walker l
    // listed m_l - 1 times) ascending; one scan carries both counts (each at most 2^14)
    int zero_base = 0, copy_base = 0;
#pragma unroll
    for (int q = 0; q < PT; ++q) {
        const int l = tid + kSolveThreads * q;
        const bool valid = l < N;
        const int isz = valid && m[q] == 0;
        const int surplus = valid && m[q] > 1 ? m[q] - 1 : 0;
        int total;
        const int at = block_scan_excl(isz | (surplus << 16), &total, sh);
        if (valid) {
            B.m[l] = m[q];
            if (isz) B.zero_l[zero_base + (at & 0xFFFF)] = l;
            for (int k = 0; k < surplus; ++k) B.donor_l[copy_base + (at >> 16) + k] = l;
            if (B.m_trace) B.m_trace[(size_t)event * N + l] = m[q];
        }
        zero_base += total & 0xFFFF;
        copy_base += total >> 16;
    }
    if (tid == 0) {
        B.n_pairs[0] = zero_base < copy_base ? zero_base : copy_base;
        B.delta[0] = result;
        if (B.delta_trace) B.delta_trace[event] = result;
    }
}

// room for the kernel's static shared memory (its reductions, under 2 KiB) beside the 136 KiB
constexpr size_t kSolveStatic = 4096;
template <int PT>
cudaError_t launch_solve(const DevProblem &P, const DevState &S, const BranchScratch &B, int block_index, double fraction,
                         int event, cudaStream_t st, int *launches) {
    const size_t staged = (size_t)(sum_at(P.n_walkers - 1) + 1) * sizeof(double);   // <= 136 KiB (16384 walkers)
    const cudaError_t e = allow_smem(branch_solve_kernel<PT>, kSolveStatic);
    if (e != cudaSuccess) return e;
    branch_solve_kernel<PT><<<1, kSolveThreads, staged, st>>>(P, S, B, block_index, fraction, event);
    *launches += 1;
    return cudaGetLastError();
}

template <typename... Args>
cudaError_t launch_solve_n(const DevProblem &P, Args... args) {
    if (P.n_walkers <= kSolveThreads) return launch_solve<1>(P, args...);
    if (P.n_walkers <= kSolveThreads * 4) return launch_solve<4>(P, args...);
    if (P.n_walkers <= kSolveThreads * 8) return launch_solve<8>(P, args...);
    return launch_solve<16>(P, args...);
}

// Imprinting (Sec. 2.5): a^(l1) <- t a^(l2) + (1 - t) a^(l1); the residual mixes the same way
// by linearity and chi2 of l1 is summed again.  One block per pair; no donor is imprinted.
__global__ void __launch_bounds__(128) imprint_kernel(DevProblem P, DevState S, BranchScratch B,
                                                      int precision, double t) {
    __shared__ double Rs[kMaxTau];
    const int q = blockIdx.x;
    if (q >= B.n_pairs[0]) return;
    const int l1 = B.zero_l[q], l2 = B.donor_l[q];
    const double omt = 1.0 - t;
    const int NO = P.n_omega, PAD = P.n_tau_pad;
    if (precision == 0) {
        double *a1 = S.a64 + (size_t)l1 * NO;
        const double *a2 = S.a64 + (size_t)l2 * NO;
        for (int j = threadIdx.x; j < NO; j += blockDim.x) a1[j] = t * a2[j] + omt * a1[j];
        for (int i = threadIdx.x; i < PAD; i += blockDim.x) {
            const double r = t * S.R64[(size_t)l2 * PAD + i] + omt * S.R64[(size_t)l1 * PAD + i];
            S.R64[(size_t)l1 * PAD + i] = r;
            Rs[i] = r;
        }
    } else {
        float *b1 = S.b32 + (size_t)l1 * NO;
        const float *b2 = S.b32 + (size_t)l2 * NO;
        const float tf = (float)t, omtf = (float)omt;
        for (int j = threadIdx.x; j < NO; j += blockDim.x) b1[j] = tf * b2[j] + omtf * b1[j];
        for (int i = threadIdx.x; i < PAD; i += blockDim.x) {
            const double r = t * (double)S.R32[(size_t)l2 * PAD + i] + omt * (double)S.R32[(size_t)l1 * PAD + i];
            S.R32[(size_t)l1 * PAD + i] = (float)r;
            Rs[i] = (double)(float)r;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double c2 = 0.0;
        for (int i = 0; i < P.n_tau; ++i) c2 = c2 + Rs[i] * Rs[i];
        S.chi2[l1] = c2;
    }
}

// Walker rows for another handle of the population: spectrum and residual of idx[q] in FP64.
__global__ void walker_rows_kernel(DevProblem P, DevState S, int precision, const int *idx, double *a_rows,
                                   double *R_rows) {
    const int q = blockIdx.x, l = idx[q];
    const int NO = P.n_omega, NT = P.n_tau, PAD = P.n_tau_pad;
    for (int j = threadIdx.x; j < NO; j += blockDim.x)
        a_rows[(size_t)q * NO + j] = precision == 0 ? S.a64[(size_t)l * NO + j] : (double)S.b32[(size_t)l * NO + j];
    for (int i = threadIdx.x; i < NT; i += blockDim.x)
        R_rows[(size_t)q * NT + i] = precision == 0 ? S.R64[(size_t)l * PAD + i] : (double)S.R32[(size_t)l * PAD + i];
}

// Elements [q0, q0 + n) of an FP32 array of rows of `cols` (`pitch` apart) as FP64, and the way back (rows
// without gaps): states cross to the host in FP64, and the conversion is bound by memory here, 3 us for
// 512000 elements, where a host thread took 130 (in) to 230 us (out), page faults of its buffer included.
// set_state and state of 1024 walkers x 500 bins x 200 tau: 0.66 -> 0.39 ms.
__global__ void __launch_bounds__(256) widen_kernel(const float *src, int cols, int pitch, size_t q0, size_t n, double *out) {
    const size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const size_t at = q0 + q;
    out[q] = (double)src[cols == pitch ? at : at / cols * pitch + at % cols];
}
__global__ void __launch_bounds__(256) narrow_kernel(const double *in, size_t n, float *dst) {
    const size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q < n) dst[q] = (float)in[q];
}
// every walker's common scale = 1
__global__ void __launch_bounds__(256) unit_scale_kernel(int n_walkers, float *g2) {
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= n_walkers) return;
    g2[2 * w] = 1.0f;
    g2[2 * w + 1] = 0.0f;
}

// Imprinting from donor rows (Sec. 2.5), the arithmetic of imprint_kernel with the donor's
// values read from rows in this device's memory: walker idx[q] <- t row q + (1 - t) itself.
__global__ void __launch_bounds__(128) imprint_rows_kernel(DevProblem P, DevState S, int precision, const int *idx,
                                                           const double *a_rows, const double *R_rows, double t) {
    __shared__ double Rs[kMaxTau];
    const int q = blockIdx.x, l1 = idx[q];
    const double omt = 1.0 - t;
    const int NO = P.n_omega, NT = P.n_tau, PAD = P.n_tau_pad;
    const double *a2 = a_rows + (size_t)q * NO, *R2 = R_rows + (size_t)q * NT;
    if (precision == 0) {
        double *a1 = S.a64 + (size_t)l1 * NO;
        for (int j = threadIdx.x; j < NO; j += blockDim.x) a1[j] = t * a2[j] + omt * a1[j];
        for (int i = threadIdx.x; i < PAD; i += blockDim.x) {
            const double r = t * (i < NT ? R2[i] : 0.0) + omt * S.R64[(size_t)l1 * PAD + i];
            S.R64[(size_t)l1 * PAD + i] = r;
            Rs[i] = r;
        }
    } else {
        float *b1 = S.b32 + (size_t)l1 * NO;
        const float tf = (float)t, omtf = (float)omt;
        for (int j = threadIdx.x; j < NO; j += blockDim.x) b1[j] = tf * (float)a2[j] + omtf * b1[j];
        for (int i = threadIdx.x; i < PAD; i += blockDim.x) {
            const double r = t * (i < NT ? R2[i] : 0.0) + omt * (double)S.R32[(size_t)l1 * PAD + i];
            S.R32[(size_t)l1 * PAD + i] = (float)r;
            Rs[i] = (double)(float)r;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double c2 = 0.0;
        for (int i = 0; i < NT; ++i) c2 = c2 + Rs[i] * Rs[i];
        S.chi2[l1] = c2;
    }
}

// ------------------------------------------------------------------ statistics
__global__ void block_stats_kernel(DevProblem P, DevState S, BlockCounters *out) {
    double cmin = DBL_MAX, csum = 0.0;
    unsigned long long acc = 0, pos = 0;
    for (int w = threadIdx.x; w < P.n_walkers; w += blockDim.x) {
        const double c = S.chi2[w];
        cmin = c < cmin ? c : cmin;
        csum += c;
        acc += S.n_acc[w];
        pos += S.n_pos[w];
    }
    for (int o = 16; o > 0; o >>= 1) {
        const double c = __shfl_xor_sync(kFull, cmin, o);
        cmin = c < cmin ? c : cmin;
        csum += __shfl_xor_sync(kFull, csum, o);
        acc += __shfl_xor_sync(kFull, acc, o);
        pos += __shfl_xor_sync(kFull, pos, o);
    }
    __shared__ double smin[32], ssum[32];
    __shared__ unsigned long long sacc[32], spos[32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) { smin[warp] = cmin; ssum[warp] = csum; sacc[warp] = acc; spos[warp] = pos; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) {
            cmin = smin[k] < cmin ? smin[k] : cmin;
            csum += ssum[k];
            acc += sacc[k];
            pos += spos[k];
        }
        out->chi2_min = cmin;
        out->chi2_sum = csum;
        out->acc = acc;
        out->pos = pos;
    }
}

// ------------------------------------------------------------------ stochastic average
// Walkers with chi2 <= factor * min chi2; mean over them and the standard error
// sqrt(sum (a - mean)^2 / (n - 1)) / sqrt(n) per bin (Sec. 1).
//
// One block selects: the smallest chi2 (a NaN in walker 0's place stands, elsewhere it is passed
// over), the cut, and the list of the walkers below it, ascending.  (One thread over all walkers
// took 0.46 ms at 4096 and 1.8 ms at 16384; the block takes about 10 us.)
constexpr int kSelectThreads = 1024;
__global__ void __launch_bounds__(kSelectThreads) average_select_kernel(DevProblem P, DevState S, double factor, int *n_used,
                                                                        double *cut_out, int *idx) {
    __shared__ SolveShared sh;
    const int W = P.n_walkers, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double c0 = S.chi2[0];
    double cmin = c0;
    for (int w = tid; w < W; w += kSelectThreads) {
        const double c = S.chi2[w];
        cmin = c < cmin ? c : cmin;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const double c = __shfl_xor_sync(kFull, cmin, o);
        cmin = c < cmin ? c : cmin;
    }
    if (lane == 0) sh.red_d[warp] = cmin;
    __syncthreads();
    cmin = c0;
    for (int k = 0; k < kSelectThreads / 32; ++k) cmin = sh.red_d[k] < cmin ? sh.red_d[k] : cmin;
    const double cut = factor * cmin;
    int used = 0;
    for (int w0 = 0; w0 < W; w0 += kSelectThreads) {
        const int w = w0 + tid;
        const int in = w < W && S.chi2[w] <= cut;
        int total;
        const int at = block_scan_excl(in, &total, sh);
        if (in) idx[used + at] = w;
        used += total;
    }
    if (tid == 0) {
        *n_used = used;
        *cut_out = cut;
    }
}

// FP64 state: one thread per bin, sums over the selected walkers in ascending order (the
// validation path's order), eight loads in flight before their eight ordered additions.
__global__ void __launch_bounds__(32) average_bins64_kernel(DevProblem P, DevState S, const int *n_used, const int *idx,
                                                            double *mean, double *err) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= P.n_omega) return;
    const int used = *n_used;
    const double *a = S.a64 + j;
    const size_t NO = P.n_omega;
    auto walk = [&](auto &&term) {
        int k = 0;
        for (; k + 8 <= used; k += 8) {
            double v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = a[(size_t)idx[k + q] * NO];
#pragma unroll
            for (int q = 0; q < 8; ++q) term(v[q]);
        }
        for (; k < used; ++k) term(a[(size_t)idx[k] * NO]);
    };
    double m = 0.0, e = 0.0;
    walk([&](double v) { m += v; });
    m /= used;
    if (used > 1) {
        walk([&](double v) {
            const double d = v - m;
            e += d * d;
        });
        e = sqrt(e / (used - 1)) / sqrt((double)used);
    }
    mean[j] = m;
    err[j] = e;
}

// FP32 state: FP64 sums over kAvgChunks equal parts of the selected walkers, one block per part
// and 128 bins, then over the parts in order.  The bound is the FP64 pipe (two conversions, two
// additions and a fused multiply-add per element at 2 lanes a clock and SM) once enough blocks
// are in flight; one thread per bin over all walkers was bound by one load's latency at a time
// (1.48 ms at 4096 x 1000, 4.7 ms at 16384 x 2048).  A whole sail_average call: 2.41 -> 0.24 ms at
// 200 tau x 1000 bins x 4096 walkers, 9.65 -> 0.37 ms at 512 x 2048 x 16384.
constexpr int kAvgBins = 128;
template <bool VAR>
__global__ void __launch_bounds__(kAvgBins) average_part_kernel(DevProblem P, DevState S, const int *n_used, const int *idx,
                                                                const double *sums, double *out, double *mean) {
    const int j = blockIdx.x * kAvgBins + threadIdx.x, part = blockIdx.y;
    if (j >= P.n_omega) return;
    const size_t NO = P.n_omega;
    const int used = *n_used, per = (used + kAvgChunks - 1) / kAvgChunks;
    const int k0 = min(part * per, used), k1 = min(k0 + per, used);
    double m = 0.0;
    if constexpr (VAR) {
        for (int c = 0; c < kAvgChunks; ++c) m += sums[c * NO + j];
        m /= used;
        if (part == 0) mean[j] = m;
    }
    const float *b = S.b32 + j;
    double s0 = 0.0, s1 = 0.0;
    auto term = [&](double &s, float v) {
        if constexpr (VAR) {
            const double d = (double)v - m;
            s = fma(d, d, s);
        } else {
            s += (double)v;
        }
    };
    int k = k0;
    for (; k + 8 <= k1; k += 8) {
        float v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = b[(size_t)idx[k + q] * NO];
#pragma unroll
        for (int q = 0; q < 8; q += 2) {
            term(s0, v[q]);
            term(s1, v[q + 1]);
        }
    }
    for (; k < k1; ++k) term(s0, b[(size_t)idx[k] * NO]);
    out[part * NO + j] = s0 + s1;
}

__global__ void __launch_bounds__(kAvgBins) average_err_kernel(DevProblem P, const int *n_used, const double *squares, double *err) {
    const int j = blockIdx.x * kAvgBins + threadIdx.x;
    if (j >= P.n_omega) return;
    const int used = *n_used;
    double e = 0.0;
    if (used > 1) {
        for (int c = 0; c < kAvgChunks; ++c) e += squares[(size_t)c * P.n_omega + j];
        e = sqrt(e / (used - 1)) / sqrt((double)used);
    }
    err[j] = e;
}

// Residual of one spectrum: thread i sums the model over the bins in order (eight products in
// flight ahead of their ordered additions), one warp a block so that every SM's FP64 pipe serves
// one of them; then one thread sums chi2 in order.  (One block of 128 threads, a load at a time:
// 0.47 ms at 200 x 1000, 2.0 ms at 512 x 2048.)
__global__ void __launch_bounds__(32) residual_of_kernel(DevProblem P, const double *a, double *R) {
    const int i = blockIdx.x * 32 + threadIdx.x;
    const size_t PAD = P.n_tau_pad;
    double r = 0.0;
    if (i < P.n_tau) {
        const double *K = P.Khat64 + i;
        double model = 0.0;
        int j = 0;
        for (; j + 8 <= P.n_omega; j += 8) {
            double p[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) p[q] = K[(j + q) * PAD] * a[j + q];
#pragma unroll
            for (int q = 0; q < 8; ++q) model = model + p[q];
        }
        for (; j < P.n_omega; ++j) model = model + K[j * PAD] * a[j];
        r = P.Fhat64[i] - model;
    }
    R[i] = r;
}
__global__ void __launch_bounds__(128) chi2_of_kernel(DevProblem P, const double *R, double *chi2) {
    __shared__ double Rs[kMaxTau];
    for (int i = threadIdx.x; i < P.n_tau; i += blockDim.x) Rs[i] = R[i] * R[i];
    __syncthreads();
    if (threadIdx.x == 0) {
        double c2 = 0.0;
#pragma unroll 8
        for (int i = 0; i < P.n_tau; ++i) c2 = c2 + Rs[i];
        *chi2 = c2;
    }
}

__global__ void philox_kernel(int n, const uint32_t *ctr, uint64_t seed, uint32_t *out) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const uint4 c = make_uint4(ctr[4 * q], ctr[4 * q + 1], ctr[4 * q + 2], ctr[4 * q + 3]);
    const uint4 r = philox4x32_10(c, philox_key(seed));
    out[4 * q] = r.x;
    out[4 * q + 1] = r.y;
    out[4 * q + 2] = r.z;
    out[4 * q + 3] = r.w;
}

template <int C>
cudaError_t launch_sweep64_c(const DevProblem &P, const DevState &S, int n0, int n1, cudaStream_t st) {
    // one warp a block while the walkers do not fill the SMs (a warp's FP64 chain wants an SM's FP64
    // pipe for itself), up to four otherwise
    int dev = 0, sms = 1, smem_max = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    int warps = (P.n_walkers + sms - 1) / sms;
    warps = warps > 4 ? 4 : warps;
    const int blocks = (P.n_walkers + warps - 1) / warps;
    const size_t staged = warps * sweep64_warp_bytes(true, P.n_omega, C);
    if (staged <= (size_t)smem_max) {
        const cudaError_t e = allow_smem(sweep_fp64_kernel<C, true>);
        if (e != cudaSuccess) return e;
        sweep_fp64_kernel<C, true><<<blocks, 32 * warps, staged, st>>>(P, S, n0, n1);
    } else {
        sweep_fp64_kernel<C, false><<<blocks, 32 * warps, warps * sweep64_warp_bytes(false, P.n_omega, C), st>>>(P, S, n0, n1);
    }
    return cudaGetLastError();
}

// Smoothing of one spectrum (Sec. smoothing), in the oracle's order of operations: the
// three-point stencil of strength s from the old values, ends (1 - s) a_0 + s a_1 and
// (1 - s) a_{N-1} + s a_{N-2}; then sums in bin order and the tilt a_j (1 + beta (x_j - m)),
// m = B'/A', beta = (B - B') / sum_j a_j (x_j - m)^2, which restores sum_j a_j x_j = B and
// keeps sum_j a_j (skipped when |beta| max_j |x_j - m| >= 1/2).  FP64 arithmetic; E is the
// element type of the state.
template <typename E>
__device__ void smooth_one(E *a, int N, const double *x, double B, double s) {
    const double c = 1.0 - 2.0 * s, e = 1.0 - s;
    double prev = (double)a[0];
    a[0] = (E)(e * (double)a[0] + s * (double)a[1]);
    for (int j = 1; j < N - 1; ++j) {
        const double cur = (double)a[j];
        a[j] = (E)(s * prev + c * cur + s * (double)a[j + 1]);
        prev = cur;
    }
    a[N - 1] = (E)(e * (double)a[N - 1] + s * prev);
    double A1 = 0.0, B1 = 0.0;
    for (int j = 0; j < N; ++j) {
        const double v = (double)a[j];
        A1 += v;
        B1 += v * x[j];
    }
    if (!(A1 > 0.0)) return;
    const double m = B1 / A1;
    double V = 0.0;
    for (int j = 0; j < N; ++j) {
        const double d = x[j] - m;
        V += (double)a[j] * d * d;
    }
    double beta = V > 0.0 ? (B - B1) / V : 0.0;
    const double span = fabs(x[0] - m) > fabs(x[N - 1] - m) ? fabs(x[0] - m) : fabs(x[N - 1] - m);
    if (!(fabs(beta) * span < 0.5)) beta = 0.0;
    for (int j = 0; j < N; ++j) a[j] = (E)((double)a[j] * (1.0 + beta * (x[j] - m)));
}

// Puts each FP64 spectrum back on both sum rules in the oracle's order (or_restore): sums in
// bin order, then a_j kappa (1 + lambda (x_j - c)).  One thread per walker.
__global__ void __launch_bounds__(128) restore_seq_kernel(DevProblem P, DevState S) {
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= P.n_walkers) return;
    const int N = P.n_omega;
    double *a = S.a64 + (size_t)w * N;
    const double *x = P.x64;
    double A1 = 0.0, B1 = 0.0;
    for (int j = 0; j < N; ++j) {
        A1 += a[j];
        B1 += a[j] * x[j];
    }
    if (!(A1 > 0.0)) return;
    const double c = B1 / A1;
    double V = 0.0;
    for (int j = 0; j < N; ++j) {
        const double d = x[j] - c;
        V += a[j] * d * d;
    }
    const double kappa = P.A / A1;
    double lambda = V > 0.0 ? (P.B / P.A - c) * A1 / V : 0.0;
    if (!(fabs(lambda * (x[N - 1] - x[0])) < 0.5)) lambda = 0.0;
    for (int j = 0; j < N; ++j) a[j] = a[j] * (kappa * (1.0 + lambda * (x[j] - c)));
}

__global__ void __launch_bounds__(128) smooth_kernel(DevProblem P, DevState S, double s) {
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= P.n_walkers) return;
    smooth_one(S.a64 + (size_t)w * P.n_omega, P.n_omega, P.x64, P.B, s);
}

// The same for an FP32 population, one warp per walker: the stencil and the sums in one pass over
// chunks of 32 bins (neighbours by shuffle; the chunk's right neighbour is read before it is
// written), then the tilt's second moment and the tilt, all in FP64, sums over lanes.  One thread
// per walker took 0.97 ms at 1500 x 1000, strided over the spectra.
__global__ void __launch_bounds__(256) smooth32_kernel(DevProblem P, DevState S, double s) {
    const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (w >= P.n_walkers) return;
    const int N = P.n_omega;
    float *a = S.b32 + (size_t)w * N;
    const double *x = P.x64;
    const double c = 1.0 - 2.0 * s, e = 1.0 - s;
    auto sum = [](double v) {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
        return v;
    };
    double A1 = 0.0, B1 = 0.0;
    float before = 0.0f;                         // the last old value of the chunk before
    for (int j0 = 0; j0 < N; j0 += 32) {
        const int j = j0 + lane;
        const float cur = j < N ? a[j] : 0.0f, after = j0 + 32 < N ? a[j0 + 32] : 0.0f;
        float left = __shfl_up_sync(kFull, cur, 1), right = __shfl_down_sync(kFull, cur, 1);
        if (lane == 0) left = before;
        if (lane == 31) right = after;
        before = __shfl_sync(kFull, cur, 31);
        __syncwarp();                            // the chunk is read before any of it is written
        if (j < N) {
            const double v = j == 0 ? e * (double)cur + s * (double)right
                             : j == N - 1 ? e * (double)cur + s * (double)left
                                          : s * (double)left + c * (double)cur + s * (double)right;
            const float f = (float)v;
            a[j] = f;
            A1 += (double)f;
            B1 += (double)f * x[j];
        }
    }
    A1 = sum(A1);
    B1 = sum(B1);
    if (!(A1 > 0.0)) return;
    const double m = B1 / A1;
    double V = 0.0;
    for (int j = lane; j < N; j += 32) {
        const double d = x[j] - m;
        V += (double)a[j] * d * d;
    }
    V = sum(V);
    double beta = V > 0.0 ? (P.B - B1) / V : 0.0;
    const double span = fabs(x[0] - m) > fabs(x[N - 1] - m) ? fabs(x[0] - m) : fabs(x[N - 1] - m);
    if (!(fabs(beta) * span < 0.5)) beta = 0.0;
    for (int j = lane; j < N; j += 32) a[j] = (float)((double)a[j] * (1.0 + beta * (x[j] - m)));
}

}  // namespace

// ------------------------------------------------------------------ launchers
cudaError_t launch_init_state(const DevProblem &P, const DevState &S, int precision, const double *a0,
                              const double *R0, double chi2_0, cudaStream_t st) {
    init_state_kernel<<<P.n_walkers, 128, 0, st>>>(P, S, precision, a0, R0, chi2_0);
    return cudaGetLastError();
}

cudaError_t launch_sweep_fp64(const DevProblem &P, const DevState &S, int n0, int n1, cudaStream_t st) {
    switch (P.n_tau_pad / 32) {
        case 1: return launch_sweep64_c<1>(P, S, n0, n1, st);
        case 2: return launch_sweep64_c<2>(P, S, n0, n1, st);
        case 3: return launch_sweep64_c<3>(P, S, n0, n1, st);
        case 4: return launch_sweep64_c<4>(P, S, n0, n1, st);
        case 5: return launch_sweep64_c<5>(P, S, n0, n1, st);
        case 6: return launch_sweep64_c<6>(P, S, n0, n1, st);
        case 7: return launch_sweep64_c<7>(P, S, n0, n1, st);
        case 8: return launch_sweep64_c<8>(P, S, n0, n1, st);
        case 9: return launch_sweep64_c<9>(P, S, n0, n1, st);
        case 10: return launch_sweep64_c<10>(P, S, n0, n1, st);
        case 11: return launch_sweep64_c<11>(P, S, n0, n1, st);
        case 12: return launch_sweep64_c<12>(P, S, n0, n1, st);
        case 13: return launch_sweep64_c<13>(P, S, n0, n1, st);
        case 14: return launch_sweep64_c<14>(P, S, n0, n1, st);
        case 15: return launch_sweep64_c<15>(P, S, n0, n1, st);
        case 16: return launch_sweep64_c<16>(P, S, n0, n1, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_resync(const DevProblem &P, const DevState &S, int precision, int restore, int kind,
                          int *status, cudaStream_t st, int *launches) {
    if (precision == 0) {
        if (P.hastings && restore) {
            // the Hastings chain drifts off the sum rules by rounding: put it back first
            restore_seq_kernel<<<(P.n_walkers + 127) / 128, 128, 0, st>>>(P, S);
            *launches += 1;
        }
        resync_kernel<<<P.n_walkers, 128, 0, st>>>(P, S, precision);
        *launches += 1;
        return cudaGetLastError();
    }
    if (kind == 2 && !P.tma) return cudaErrorInvalidValue;
    if (restore) {
        // with the tensor-copy recomputation the restoration also writes the BF16 pieces
        unsigned short *At = kind == 2 ? (unsigned short *)P.tma->At : nullptr;
        const int nop = kind == 2 ? P.tma->nop : 0;
        const size_t plane = kind == 2 ? (size_t)P.tma->n_blocks_walkers * 128 * nop : 0;
        restore_kernel<<<(P.n_walkers * 32 + 255) / 256, 256, 0, st>>>(P, S, At, nop, plane);
        *launches += 1;
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (kind == 3) {                  // FP64 GEMM
        *launches += 1;
        return launch_resync_fp64(P, S, st);
    }
    if (kind == 2) {                  // (pieces of the spectra), tensor-copy GEMM, chi2 pass
        *launches += restore ? 2 : 3;
        return launch_resync_tma(P, S, *P.tma, status, !restore, st);
    }
    *launches += kind == 1 ? 2 : 1;   // tensor-core GEMM + chi2 pass, or the FP32 GEMM
    return kind == 1 ? launch_resync_tc(P, S, status, false, st) : launch_resync_fp32(P, S, st);
}

cudaError_t launch_branch(const DevProblem &P, const DevState &S, const BranchScratch &B, int precision,
                          int block_index, double fraction, double imprint_t, int event, cudaStream_t st,
                          int *launches) {
    const cudaError_t e = launch_solve_n(P, S, B, block_index, fraction, event, st, launches);
    if (e != cudaSuccess) return e;
    imprint_kernel<<<P.n_walkers, 128, 0, st>>>(P, S, B, precision, imprint_t);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_branch_solve(const DevProblem &P, const DevState &S, const BranchScratch &B, int block_index,
                                double fraction, cudaStream_t st, int *launches) {
    return launch_solve_n(P, S, B, block_index, fraction, 0, st, launches);
}

cudaError_t launch_walker_rows(const DevProblem &P, const DevState &S, int precision, int n, const int *idx,
                               double *a_rows, double *R_rows, cudaStream_t st) {
    walker_rows_kernel<<<n, 128, 0, st>>>(P, S, precision, idx, a_rows, R_rows);
    return cudaGetLastError();
}

cudaError_t launch_widen(const float *src, int cols, int pitch, size_t q0, size_t n, double *out, cudaStream_t st) {
    widen_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(src, cols, pitch, q0, n, out);
    return cudaGetLastError();
}

cudaError_t launch_narrow(const double *in, size_t n, float *dst, cudaStream_t st) {
    narrow_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(in, n, dst);
    return cudaGetLastError();
}

cudaError_t launch_unit_scale(int n_walkers, float *g2, cudaStream_t st) {
    unit_scale_kernel<<<(n_walkers + 255) / 256, 256, 0, st>>>(n_walkers, g2);
    return cudaGetLastError();
}

cudaError_t launch_imprint_rows(const DevProblem &P, const DevState &S, int precision, int n, const int *idx,
                                const double *a_rows, const double *R_rows, double t, cudaStream_t st) {
    imprint_rows_kernel<<<n, 128, 0, st>>>(P, S, precision, idx, a_rows, R_rows, t);
    return cudaGetLastError();
}

cudaError_t launch_smooth(const DevProblem &P, const DevState &S, int precision, double s, cudaStream_t st) {
    if (precision == 0) smooth_kernel<<<(P.n_walkers + 127) / 128, 128, 0, st>>>(P, S, s);
    else smooth32_kernel<<<(P.n_walkers + 7) / 8, 256, 0, st>>>(P, S, s);
    return cudaGetLastError();
}

cudaError_t launch_block_stats(const DevProblem &P, const DevState &S, BlockCounters *out, cudaStream_t st) {
    block_stats_kernel<<<1, 1024, 0, st>>>(P, S, out);
    return cudaGetLastError();
}

cudaError_t launch_average(const DevProblem &P, const DevState &S, int precision, double factor, double *mean,
                           double *err, int *n_used, double *cut, int *idx, double *parts, double *R_mean,
                           double *chi2_mean, cudaStream_t st, int *launches) {
    average_select_kernel<<<1, kSelectThreads, 0, st>>>(P, S, factor, n_used, cut, idx);
    if (precision == 0) {
        average_bins64_kernel<<<(P.n_omega + 31) / 32, 32, 0, st>>>(P, S, n_used, idx, mean, err);
        *launches += 4;
    } else {
        double *squares = parts + (size_t)kAvgChunks * P.n_omega;
        const dim3 grid((P.n_omega + kAvgBins - 1) / kAvgBins, kAvgChunks);
        average_part_kernel<false><<<grid, kAvgBins, 0, st>>>(P, S, n_used, idx, nullptr, parts, nullptr);
        average_part_kernel<true><<<grid, kAvgBins, 0, st>>>(P, S, n_used, idx, parts, squares, mean);
        average_err_kernel<<<grid.x, kAvgBins, 0, st>>>(P, n_used, squares, err);
        *launches += 6;
    }
    residual_of_kernel<<<P.n_tau_pad / 32, 32, 0, st>>>(P, mean, R_mean);
    chi2_of_kernel<<<1, 128, 0, st>>>(P, R_mean, chi2_mean);
    return cudaGetLastError();
}

cudaError_t launch_philox(int n, const uint32_t *ctr, uint64_t seed, uint32_t *out, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    philox_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, ctr, seed, out);
    return cudaGetLastError();
}

}  // namespace sail
