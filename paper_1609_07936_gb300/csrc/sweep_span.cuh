// The FP32 sweep in the span of the kernel's columns.
//
// A move changes a walker's residual by d = eps M - delta_p Khat_p - delta_s Khat_s (Sec. 2.2),
// and M = Fhat - R = Khat a: every vector of it lies in the span of the columns of Khat.  The
// bin kernel is a smooth function of omega, so that span is small: within 2^-26 of each
// column's norm (a quarter of FP32's rounding unit) it has 12 to 24 dimensions on every
// recipe of this repository, whatever n_tau is.  With an orthonormal basis U of it (span.cu),
// R' = U^T R, F' = U^T Fhat and K' = U^T Khat (rows of RR floats, RR = 16, 24 or 32),
//     delta chi2 = sum_i d_i (2 R_i + d_i) = sum_k d'_k (2 R'_k + d'_k),
// the same number up to rounding: the part of R outside the span is constant and drops out.
// A move costs RR elements instead of n_tau, and its two columns are two rows of a table that
// fits in shared memory whole (96 KB at 1000 bins), not products of factor rows.  The residual
// and chi2 are not written back: every sweep launch is followed by their recomputation.
//
// Rounding.  Fewer elements average out less rounding error, so three things keep the error of
// delta chi2 below that of the loops over tau (measured in FP32 emulation against FP64 on the
// moves within 5 T of the threshold, mean error over T, both sides: 200 tau 9.2e-8 -> 3.0e-8,
// 32 tau at the noise floor 2.6e-5 -> 3.5e-6, 100 tau 7.7e-7 -> 4.4e-7, 512 tau 3.8e-7 ->
// 3.9e-7 in its first 20 sweeps and 2.3e-6 -> 7.7e-7 colder): the basis mixes its directions
// evenly (a cosine transform over them: without it the first direction carries nearly all of
// Fhat and of every column, and its rounding alone sets the error, 6 times larger); M is not
// kept but formed as F' - R', so it does not drift; and R' is summed with its rounding error
// carried along (Kahan), so it does not drift either.
//
// Measured against the loops over tau (sweep_group.cuh), sweep time, same box: 200 tau x 1000 bins
// x 4096 walkers, 100 sweeps 47.1 -> 14.0 ms (2.9e10 walker-moves/s; 100 warp instructions an
// iteration of four walkers, 290 cycles at two warps on a scheduler, 64% of its issue slots and 67%
// of the shared-memory data pipe), 16384 walkers 198 -> 45 ms; 512 x 2048 x 16384, 10 sweeps 90 ->
// 14 ms (spectra in L2); 160 x 1000 x 1500, 100 sweeps 35.5 -> 9.6 ms (203 cycles an iteration,
// one warp); Hastings 72 -> 15.7 ms; index walk (L = 2, 1500 walkers, 50 sweeps) 47 -> 15 ms.  The
// warp barrier a move (below) is in the noise of these.
//
// Layout.  G lanes per walker (8 or 4: four or eight walkers a warp).  The RR elements belong to
// eight virtual lanes, RR / 8 each; delta chi2 is the xor-butterfly sum (4, 2, 1) of the virtual
// lanes' parts.  With G = 4 a lane holds virtual lanes l and l + 4 and does the first step of
// the butterfly by itself, so both layouts form the same sums bit for bit, and a walker's
// trajectory does not depend on the layout, the launch or the other walkers.
//
// Chain.  One move at a time; the loop is bound by one warp's dependent chain (update -> d ->
// delta chi2 -> butterfly -> test -> update), so everything else is kept off it: move k+1's
// words and columns are read while move k is reduced, the amplitudes that move k would set are
// formed before its test, and its update is branch-free.  The words of G consecutive moves are
// drawn at once, one move per lane, and handed over through a ring in shared memory.
//
// One basic block.  The G moves of a batch are unrolled without a branch (stores under a predicate,
// masked updates, a reciprocal without its slow path, null moves past the sweep's end), so that the
// compiler fills a move's butterfly with the work around it: the same loop with branches for the
// accepted move and the division ran 310 cycles an iteration instead of 203 (one warp), 387 instead
// of 290 (4096 walkers).  Evaluating two moves at once (the second for both outcomes of the first)
// halves the butterflies but costs 128 instructions a move: 2.28 against 1.98 ms.
#pragma once
#include "sweep_group.cuh"

namespace sail {

namespace {

constexpr int kSpanWarps = 16;         // at most 16 warps a block (128 registers a thread)

struct SpanGeom {
    int groups_total;     // walker groups (one warp each)
    int groups_per_cta;
    int warps;            // warps per block
    int rounds;           // groups handled one after another by each warp
    int stage_t;          // column table in shared memory
    int stage_b;          // spectra in shared memory
};

// One move's words in the ring, as its users take them: -delta_p, -delta_s and -eps twice each
// (operand pairs of the f32x2 arithmetic), the acceptance threshold and the bins p | s << 16.
struct SpanRing {
    float4 a[2][32];      // -delta_p, -delta_p, -delta_s, -delta_s; [batch][lane that drew it]
    float4 b[2][32];      // -eps, -eps, threshold, bins
};
struct SpanMove {
    f2 mdp2, mds2, me2;
    float mdp, mds, me, thr;
    int ps;
};

// The elements of one virtual lane: RR / 8 floats, as pairs and (RR = 24) a single.
template <int RR>
struct SpanVec {
    static constexpr int NP = RR / 16;
    static constexpr bool ODD = (RR / 8) % 2 != 0;
    f2 p[NP];
    float s;
};
// the basis direction of element e of virtual lane v
template <int RR>
__device__ __forceinline__ int span_dim(int v, int e) {
    if (RR == 24) return e < 2 ? 2 * v + e : 16 + v;
    return (RR / 8) * v + e;
}

// A virtual lane's elements of one table row (row: its first float).
template <int RR, bool SMEM>
__device__ __forceinline__ SpanVec<RR> span_row(const float *row, int v) {
    SpanVec<RR> r;
    if constexpr (RR == 32) {
        const float4 x = SMEM ? *reinterpret_cast<const float4 *>(row + 4 * v)
                              : __ldg(reinterpret_cast<const float4 *>(row + 4 * v));
        r.p[0] = pk(x.x, x.y);
        r.p[1] = pk(x.z, x.w);
    } else {
        const float2 x = SMEM ? *reinterpret_cast<const float2 *>(row + 2 * v)
                              : __ldg(reinterpret_cast<const float2 *>(row + 2 * v));
        r.p[0] = pk(x.x, x.y);
    }
    r.s = 0.0f;
    if constexpr (SpanVec<RR>::ODD) r.s = SMEM ? row[16 + v] : __ldg(row + 16 + v);
    return r;
}

// a virtual lane's part of delta chi2: sum of d (2 R + d) over its elements, R = (R, c)
template <int RR>
__device__ __forceinline__ float span_part(const SpanVec<RR> &d, const SpanVec<RR> &R, const SpanVec<RR> &c, f2 two) {
    f2 acc = mul2(d.p[0], fma2(two, c.p[0], fma2(two, R.p[0], d.p[0])));
    if constexpr (SpanVec<RR>::NP > 1) acc = fma2(d.p[1], fma2(two, c.p[1], fma2(two, R.p[1], d.p[1])), acc);
    const float2 a = up(acc);
    if constexpr (SpanVec<RR>::ODD) return fmaf(d.s, fmaf(2.0f, c.s, fmaf(2.0f, R.s, d.s)), a.x) + a.y;
    return a.x + a.y;
}

// R <- R + m d (m = 1 or 0) with the rounding error carried in c; m = 0 leaves R + c as it is.
template <int RR>
__device__ __forceinline__ void span_add(SpanVec<RR> &R, SpanVec<RR> &c, const SpanVec<RR> &d, float m, f2 m2, f2 minus_one) {
#pragma unroll
    for (int q = 0; q < SpanVec<RR>::NP; ++q) {
        const f2 y = fma2(m2, d.p[q], c.p[q]);
        const f2 t = add2(R.p[q], y);
        c.p[q] = fma2(minus_one, fma2(minus_one, R.p[q], t), y);
        R.p[q] = t;
    }
    if constexpr (SpanVec<RR>::ODD) {
        const float y = fmaf(m, d.s, c.s);
        const float t = __fadd_rn(R.s, y);
        c.s = __fadd_rn(y, -__fadd_rn(t, -R.s));
        R.s = t;
    }
}

// R'_k = sum_i U_ik R_i of the lane's elements: compensated dot products (Ogita, Rump and Oishi's
// Dot2), U as a pair of floats, the result as (R, c);
// F = -F' of those elements.
template <int RR, int NV>
__device__ __forceinline__ void span_project(const DevProblem &P, const float *Rrow, const int (&vl)[NV],
                                             SpanVec<RR> (&R)[NV], SpanVec<RR> (&C)[NV], SpanVec<RR> (&F)[NV]) {
    constexpr int E = RR / 8;
#pragma unroll
    for (int u = 0; u < NV; ++u) {
        float s[E], c[E], f[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            s[e] = c[e] = 0.0f;
            f[e] = -P.Fspan[span_dim<RR>(vl[u], e)];
        }
#pragma unroll 8
        for (int i = 0; i < P.n_tau; ++i) {
            const float r = __ldg(Rrow + i);
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const float2 U = __ldg(reinterpret_cast<const float2 *>(P.Uspan) + (size_t)i * RR + span_dim<RR>(vl[u], e));
                const float p = __fmul_rn(r, U.x);
                const float pe = fmaf(r, U.x, -p);
                const float t = __fadd_rn(s[e], p);
                const float b = __fadd_rn(t, -s[e]);
                const float se = __fadd_rn(__fadd_rn(s[e], -__fadd_rn(t, -b)), __fadd_rn(p, -b));
                c[e] = fmaf(r, U.y, __fadd_rn(c[e], __fadd_rn(pe, se)));
                s[e] = t;
            }
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const float t = __fadd_rn(s[e], c[e]);
            c[e] = __fadd_rn(c[e], -__fadd_rn(t, -s[e]));
            s[e] = t;
        }
#pragma unroll
        for (int q = 0; q < SpanVec<RR>::NP; ++q) {
            R[u].p[q] = pk(s[2 * q], s[2 * q + 1]);
            C[u].p[q] = pk(c[2 * q], c[2 * q + 1]);
            F[u].p[q] = pk(f[2 * q], f[2 * q + 1]);
        }
        R[u].s = SpanVec<RR>::ODD ? s[E - 1] : 0.0f;
        C[u].s = SpanVec<RR>::ODD ? c[E - 1] : 0.0f;
        F[u].s = SpanVec<RR>::ODD ? f[E - 1] : 0.0f;
    }
}

// g = eps F' - delta_p K'_p - delta_s K'_s: a move's change but for -eps R' (F = -F'; tab: the column
// table)
template <int RR, int NV, bool TS>
__device__ __forceinline__ void span_g(const float *tab, const int (&vl)[NV], const SpanVec<RR> (&F)[NV], const SpanMove &m,
                                       SpanVec<RR> (&g)[NV]) {
    using V = SpanVec<RR>;
    const float *rp = tab + (size_t)(uint32_t)((m.ps & 0xFFFF) * RR), *rs = tab + (size_t)(uint32_t)((m.ps >> 16) * RR);
#pragma unroll
    for (int u = 0; u < NV; ++u) {
        const V kp = span_row<RR, TS>(rp, vl[u]), ks = span_row<RR, TS>(rs, vl[u]);
#pragma unroll
        for (int q = 0; q < V::NP; ++q) g[u].p[q] = fma2(m.me2, F[u].p[q], fma2(m.mds2, ks.p[q], mul2(m.mdp2, kp.p[q])));
        g[u].s = V::ODD ? fmaf(m.me, F[u].s, fmaf(m.mds, ks.s, m.mdp * kp.s)) : 0.0f;
    }
}

// d = g - eps R'
template <int RR, int NV>
__device__ __forceinline__ void span_d(const SpanVec<RR> (&g)[NV], const SpanVec<RR> (&R)[NV], const SpanMove &m,
                                       SpanVec<RR> (&d)[NV]) {
#pragma unroll
    for (int u = 0; u < NV; ++u) {
#pragma unroll
        for (int q = 0; q < SpanVec<RR>::NP; ++q) d[u].p[q] = fma2(m.me2, R[u].p[q], g[u].p[q]);
        d[u].s = SpanVec<RR>::ODD ? fmaf(m.me, R[u].s, g[u].s) : 0.0f;
    }
}

// Lane's draw of move mv of walker wr.  The Metropolis test is D < threshold: D <= 0 passes, so a
// plain threshold is at least the smallest positive float (the Hastings threshold may be negative).
// Past the sweep's end, and for walkers that do not exist, a null move: eps = 1 makes its
// amplitudes 0, which passes the positivity test (it is not counted), and the threshold is never met.
template <int MODE>
__device__ __forceinline__ MoveDraw span_draw(const DevProblem &P, int mv, int n, int wr, bool active, uint2 key, float yd,
                                              float T, const float *sBeta, const float *sRgap) {
    MoveDraw m = draw_move<MODE>(mv, n, wr + P.walker_base, key, P.n_omega, yd, T, sBeta, sRgap);
    if constexpr (MODE != kHastings) m.thr = fmaxf(m.thr, 1.401298464e-45f);
    if (mv >= P.n_omega || !active) {
        m.eps = 1.0f;
        m.dp = m.ds = 0.0f;
        m.thr = -INFINITY;
    }
    return m;
}
__device__ __forceinline__ void span_put(SpanRing &ring, int batch, const MoveDraw &m) {
    const int lane = threadIdx.x & 31;
    ring.a[batch][lane] = make_float4(-m.dp, -m.dp, -m.ds, -m.ds);
    ring.b[batch][lane] = make_float4(-m.eps, -m.eps, m.thr, __int_as_float(m.ps));
}
// Move i of the batch of this lane's walker.
template <int G>
__device__ __forceinline__ SpanMove span_get(const SpanRing &ring, int batch, int i) {
    const int at = (threadIdx.x & 31) / G * G + i;
    const float4 x = ring.a[batch][at], y = ring.b[batch][at];
    SpanMove m;
    m.mdp2 = pk(x.x, x.y);
    m.mds2 = pk(x.z, x.w);
    m.me2 = pk(y.x, y.y);
    m.mdp = x.x;
    m.mds = x.z;
    m.me = y.x;
    m.thr = y.z;
    m.ps = __float_as_int(y.w);
    return m;
}

// The steps of one move's index walk (Sec. 2.3): proposed bins for p and (before skipping p) for s, and
// the uniforms of their acceptance; a step that is not taken (past P.walk_len, or the whole walk
// skipped by the uniform admixture) has a NaN, which no proposal passes.
template <int LM>
struct SpanSteps {
    int jp[LM], js[LM];
    float up[LM], us[LM];
};
template <int G, int LM>
__device__ __forceinline__ SpanSteps<LM> span_steps(const DevProblem &P, int mv, int n, int wr, uint2 key, float rho, int gl) {
    // lane t of the group draws step t + 1's words (counter (mv, n, w, 2 + t)), lane L the admixture's
    const int L = P.walk_len, NO = P.n_omega;
    const uint4 w4 = philox4x32_10(make_uint4((uint32_t)mv, (uint32_t)n, (uint32_t)(wr + P.walker_base), 2u + gl), key);
    const bool walk_p = !(unit32(__shfl_sync(kFull, w4.x, L, G)) < rho);
    const bool walk_s = !(unit32(__shfl_sync(kFull, w4.y, L, G)) < rho);
    const int jp = (int)(((uint64_t)w4.x * (uint64_t)NO) >> 32), js = (int)(((uint64_t)w4.z * (uint64_t)(NO - 1)) >> 32);
    const float up = walk_p && gl < L ? unit32(w4.y) : NAN, us = walk_s && gl < L ? unit32(w4.w) : NAN;
    SpanSteps<LM> s;
#pragma unroll
    for (int t = 0; t < LM; ++t) {
        s.jp[t] = __shfl_sync(kFull, jp, t, G);
        s.js[t] = __shfl_sync(kFull, js, t, G);
        s.up[t] = __shfl_sync(kFull, up, t, G);
        s.us[t] = __shfl_sync(kFull, us, t, G);
    }
    return s;
}
// Move m proposes bins p and s.
__device__ __forceinline__ void span_walk_to(SpanMove &m, int p, int s, const float *sBeta, const float *sRgap) {
    float dp, ds;
    m.ps = p | (s << 16);
    deltas(-m.me, p, s, sBeta, sRgap, dp, ds);
    m.mdp = -dp;
    m.mds = -ds;
    m.mdp2 = pk(-dp, -dp);
    m.mds2 = pk(-ds, -ds);
}

// Folds the common scale into walker w's spectrum b and writes the walker back (lane gl of its G).
template <int G>
__device__ __forceinline__ void span_write_back(const DevProblem &P, const DevState &S, int w, int gl, const float *b, float ghi,
                                                float glo, int accp, unsigned long long nacc,
                                                unsigned long long npos) {
    float *bg = S.b32 + (size_t)w * P.n_omega;
    for (int j = gl; j < P.n_omega; j += G) {
        const float v = b[j];
        bg[j] = fmaf(glo, v, ghi * v);
    }
    if (gl == 0) {
        S.g2[2 * w] = 1.0f;
        S.g2[2 * w + 1] = 0.0f;
        S.acc_prev[w] = accp;
        S.n_acc[w] += nacc;
        S.n_pos[w] += npos;
    }
}

// Sweeps [n0, n1) for the 32 / G walkers of group grp of one problem on one warp.
//   tab    the column table (shared memory if TS, else global memory), rows of RR floats
//   sBeta, sRgap  beta and the reciprocal gaps (shared memory)
//   b      STAGED: the spectra of walkers walker_lo.. in shared memory.  Else in global memory,
//          where a read takes longer than several moves; each lane reads b_p, b_s of the move it
//          drew a batch ahead and keeps them, replaces them when a move before it writes one of
//          those bins (until the batch turns over the replacement waits apart, so that nothing
//          waits for the read), and hands them over by shuffle
// Every lane of a walker writes an accepted move's two amplitudes (the same values), so each
// lane later reads its own write.  The warp barrier before the write orders it against the other
// lanes' reads of the same move and their writes of the move before, whose shuffles order no memory.
//
// LM > 0 (index walk): the walk's steps unrolled to LM >= P.walk_len.  The proposals of a walk do not
// depend on the state, so the steps' words are drawn and handed out one move ahead, and b at all of
// them (for s, at the bin and the one after: the proposals skip p) is read at once; what is left on the
// chain is a comparison a step.  LM = 0: steps in a loop, each with its own reads (the batched sweep).
// 200 x 1000, 10 sweeps: L = 2, 1500 walkers 6.0 -> 3.2 ms (9.4 over tau), 4096 4.0, L = 7 5.5 (12.1).
template <int RR, int G, bool TS, bool STAGED, int MODE, int LM = 0>
__device__ __forceinline__ void run_span(const DevProblem &P, const DevState &S, int n0, int n1, int grp,
                                         const float *tab, const float *sBeta, const float *sRgap, SpanRing &ring,
                                         float *b_stage, int walker_lo) {
    static_assert(G == 8 || G == 4, "eight virtual lanes on 8 or 4 lanes");
    static_assert(MODE != kWalk || G == 8, "the walk's words are drawn by 8 lanes");
    constexpr int WPW = 32 / G, NV = 8 / G;
    constexpr bool WALK = MODE == kWalk;
    constexpr bool OWN = !STAGED && !WALK;      // b_p, b_s held by the lane that drew the move (above)
    using V = SpanVec<RR>;
    const int NO = P.n_omega;
    const int lane = threadIdx.x & 31, gl = lane & (G - 1), sub = lane / G;
    const uint2 key = philox_key(P.seed);
    const double dmove = P.move_scale > 0.0 ? P.move_scale : 1.0 / NO;
    const float rho = (float)P.walk_rho;
    // virtual lanes of this lane; with G = 4 odd walkers take their halves in the other order, so
    // that two walkers' 16-byte accesses fall on different banks
    int vl[NV];
#pragma unroll
    for (int u = 0; u < NV; ++u) vl[u] = G == 8 ? gl : gl + 4 * (u ^ (sub & 1));

    const int w = WPW * grp + sub;
    const bool active = w < P.n_walkers;
    const int wr = active ? w : WPW * grp;            // a valid walker to read from
    float *b = STAGED ? b_stage + (size_t)(wr - walker_lo) * NO : S.b32 + (size_t)wr * NO;

    V R[NV], C[NV], F[NV];
    span_project<RR, NV>(P, S.R32 + (size_t)wr * P.n_tau_pad, vl, R, C, F);
    float ghi = S.g2[2 * wr], glo = S.g2[2 * wr + 1];
    int accp = S.acc_prev[wr];
    unsigned long long nacc = 0, npos = 0;
    const f2 two = pk(2.0f, 2.0f), minus_one = pk(-1.0f, -1.0f);

    for (int n = n0; n < n1; ++n) {
        const float T = (float)P.Tsweep[n];
        const float yd = (float)(amplitude(accp, NO, P.y_p, P.y_m, P.y_min) * dmove);
        int acc = 0, pos = 0;
        __syncwarp();
        const MoveDraw first = span_draw<MODE>(P, gl, n, wr, active, key, yd, T, sBeta, sRgap);
        span_put(ring, 0, first);
        __syncwarp();
        SpanMove cur = span_get<G>(ring, 0, 0), nxt = span_get<G>(ring, 0, 1);
        V g[NV];
        if constexpr (!WALK) span_g<RR, NV, TS>(tab, vl, F, cur, g);
        // OWN: this lane's move of the batch: its bins and b there
        int own_p = first.ps & 0xFFFF, own_s = first.ps >> 16;
        float own_bp = 0.0f, own_bs = 0.0f;
        if constexpr (OWN) {
            own_bp = b[own_p];
            own_bs = b[own_s];
        }
        SpanSteps<LM == 0 ? 1 : LM> steps;
        if constexpr (LM > 0) steps = span_steps<G, LM == 0 ? 1 : LM>(P, 0, n, wr, key, rho, gl);
        int batch = 0;
        for (int base = 0; base < NO; base += G, batch ^= 1) {
            const MoveDraw mine = span_draw<MODE>(P, base + G + gl, n, wr, active, key, yd, T, sBeta, sRgap);
            // OWN: b at the next batch's move, read now, and what this batch's moves write there meanwhile
            const int next_p = mine.ps & 0xFFFF, next_s = mine.ps >> 16;
            float next_bp = 0.0f, next_bs = 0.0f, new_bp = __int_as_float(-1), new_bs = __int_as_float(-1);
            if constexpr (OWN) {
                next_bp = b[next_p];
                next_bs = b[next_s];
            }
#pragma unroll
            for (int i = 0; i < G; ++i) {
                if (i == (G > 4 ? G - 3 : 1)) {
                    span_put(ring, batch ^ 1, mine);
                    __syncwarp();
                }
                float walk_bp = 0.0f, walk_bs = 0.0f;
                if constexpr (WALK && LM > 0) {
                    const int p0 = cur.ps & 0xFFFF, s0 = cur.ps >> 16;
                    float bpt[LM], bst[LM], bsu[LM];
                    float bp = b[p0];
                    const float b0 = b[s0], b1 = b[s0 + 1];
#pragma unroll
                    for (int t = 0; t < LM; ++t) {
                        bpt[t] = b[steps.jp[t]];
                        bst[t] = b[steps.js[t]];
                        bsu[t] = b[steps.js[t] + 1];
                    }
                    int wp = p0;
#pragma unroll
                    for (int t = 0; t < LM; ++t) {
                        const bool go = steps.up[t] * bp <= bpt[t];
                        wp = go ? steps.jp[t] : wp;
                        bp = go ? bpt[t] : bp;
                    }
                    int ws = s0 + (s0 >= wp);
                    float bs = s0 >= wp ? b1 : b0;
#pragma unroll
                    for (int t = 0; t < LM; ++t) {
                        const bool past = steps.js[t] >= wp;
                        const float bj = past ? bsu[t] : bst[t];
                        const bool go = steps.us[t] * bs <= bj;
                        ws = go ? steps.js[t] + past : ws;
                        bs = go ? bj : bs;
                    }
                    walk_bp = bp;
                    walk_bs = bs;
                    span_walk_to(cur, wp, ws, sBeta, sRgap);
                    span_g<RR, NV, TS>(tab, vl, F, cur, g);
                    steps = span_steps<G, LM == 0 ? 1 : LM>(P, base + i + 1, n, wr, key, rho, gl);
                } else if constexpr (WALK) {
                    // the index walk (Sec. 2.3) on the spectrum as it is now: lane t of the group
                    // draws step t + 1's words (counter (mv, n, w, 2 + t)), lane L the admixture's
                    const int mv = base + i;
                    const int L = P.walk_len;
                    const uint4 wr4 = philox4x32_10(make_uint4((uint32_t)mv, (uint32_t)n, (uint32_t)(wr + P.walker_base), 2u + gl), key);
                    const bool walk_p = !(unit32(__shfl_sync(kFull, wr4.x, L, G)) < rho);
                    const bool walk_s = !(unit32(__shfl_sync(kFull, wr4.y, L, G)) < rho);
                    int wp = cur.ps & 0xFFFF;
                    float bp = b[wp];
                    for (int t = 0; t < L; ++t) {
                        const uint32_t xj = __shfl_sync(kFull, wr4.x, t, G), xu = __shfl_sync(kFull, wr4.y, t, G);
                        const int j = (int)(((uint64_t)xj * (uint64_t)NO) >> 32);
                        const float bj = b[j];
                        if (walk_p && unit32(xu) * bp <= bj) {
                            wp = j;
                            bp = bj;
                        }
                    }
                    int ws = cur.ps >> 16;
                    ws += (ws >= wp);
                    float bs = b[ws];
                    for (int t = 0; t < L; ++t) {
                        const uint32_t xj = __shfl_sync(kFull, wr4.z, t, G), xu = __shfl_sync(kFull, wr4.w, t, G);
                        int j = (int)(((uint64_t)xj * (uint64_t)(NO - 1)) >> 32);
                        j += (j >= wp);
                        const float bj = b[j];
                        if (walk_s && unit32(xu) * bs <= bj) {
                            ws = j;
                            bs = bj;
                        }
                    }
                    span_walk_to(cur, wp, ws, sBeta, sRgap);
                    span_g<RR, NV, TS>(tab, vl, F, cur, g);
                }
                // move k: d and its part of delta chi2; then the columns of move k+1 take the place of
                // its own, and move k+2's words are fetched
                V d[NV];
                span_d<RR, NV>(g, R, cur, d);
                float D = span_part<RR>(d[0], R[0], C[0], two);
                if constexpr (NV == 2) D += span_part<RR>(d[1], R[1], C[1], two);
                const int p = cur.ps & 0xFFFF, s = cur.ps >> 16;
                float bp, bs;
                if constexpr (OWN) {
                    bp = __shfl_sync(kFull, own_bp, i, G);
                    bs = __shfl_sync(kFull, own_bs, i, G);
                } else if constexpr (LM > 0) {
                    bp = walk_bp;
                    bs = walk_bs;
                } else {
                    bp = b[p];
                    bs = b[s];
                }
                if constexpr (!WALK) span_g<RR, NV, TS>(tab, vl, F, nxt, g);
                const SpanMove far = i < G - 2 ? span_get<G>(ring, batch, i + 2) : span_get<G>(ring, batch ^ 1, i + 2 - G);
                // positivity (Eq. probability-density) on the spectrum as it is now, and the spectrum
                // if the move is accepted
                const float r = 1.0f + cur.me;
                const float ap = fmaf(r, ghi * bp, -cur.mdp);
                const float as = fmaf(r, ghi * bs, -cur.mds);
                const bool ok = ap >= 0.0f && as >= 0.0f;
                // an index walk forms its amplitudes anew, also a null move's, whose threshold alone is negative
                pos += WALK ? !ok && cur.thr > 0.0f : !ok;
                float gah = ghi, gal = glo;
                pair_scale(gah, gal, r);
                const float inv_g = rcp_rn(gah);
                const float ap_b = ap * inv_g, as_b = as * inv_g;
                // delta chi2 and the test
                D = group_sum<G>(D);
                const bool acc_k = ok && D < cur.thr;
                const float am = acc_k ? 1.0f : 0.0f;
                const f2 am2 = pk(am, am);
#pragma unroll
                for (int u = 0; u < NV; ++u) span_add<RR>(R[u], C[u], d[u], am, am2, minus_one);
                __syncwarp();          // orders the lanes' stores of b (see above)
                put_if<STAGED>(am, b, p, s, ap_b, as_b);
                ghi = acc_k ? gah : ghi;
                glo = acc_k ? gal : glo;
                acc += acc_k;
                if constexpr (OWN) {
                    const int wp = acc_k ? p : -1, ws = acc_k ? s : -1;
                    own_bp = own_p == wp ? ap_b : (own_p == ws ? as_b : own_bp);
                    own_bs = own_s == wp ? ap_b : (own_s == ws ? as_b : own_bs);
                    new_bp = next_p == wp ? ap_b : (next_p == ws ? as_b : new_bp);
                    new_bs = next_s == wp ? ap_b : (next_s == ws ? as_b : new_bs);
                }
                cur = nxt;
                nxt = far;
            }
            if constexpr (OWN) {
                own_p = next_p;
                own_s = next_s;
                own_bp = __float_as_int(new_bp) == -1 ? next_bp : new_bp;
                own_bs = __float_as_int(new_bs) == -1 ? next_bs : new_bs;
            }
        }
        accp = acc;
        nacc += acc;
        npos += pos;
        if (active && S.acc_trace && gl == 0) S.acc_trace[(size_t)n * P.n_walkers + w] = acc;
    }
    __syncwarp();                      // the lanes' writes of b, before other lanes fold them
    if (!active) return;
    span_write_back<G>(P, S, w, gl, b, ghi, glo, accp, nacc, npos);
}

// Shared memory of a span launch: rings, beta, gaps, then the table and the spectra if staged.
__host__ __device__ __forceinline__ size_t span_ring_bytes(int warps) { return (size_t)warps * sizeof(SpanRing); }

template <int RR>
__device__ __forceinline__ void span_load(const DevProblem &P, float *sBeta, float *sRgap, float *sTab, bool stage_t) {
    const int NO = P.n_omega;
    for (int q = threadIdx.x; q < NO; q += blockDim.x) {
        sBeta[q] = P.beta32[q];
        sRgap[q] = P.rgap32[q];
    }
    if (stage_t) {
        const float4 *g4 = reinterpret_cast<const float4 *>(P.Kspan);
        float4 *s4 = reinterpret_cast<float4 *>(sTab);
        for (int q = threadIdx.x; q < NO * RR / 4; q += blockDim.x) s4[q] = g4[q];
    }
}

// floats of the beta and gap vectors, rounded up so that what follows is 16-byte aligned
__host__ __device__ __forceinline__ int span_vec_floats(int NO) { return (2 * NO + 3) / 4 * 4; }

template <int RR, int G, int MODE, int LM>
__global__ void __launch_bounds__(32 * kSpanWarps, 1) sweep_span_kernel(DevProblem P, DevState S, int n0, int n1, SpanGeom Gm) {
    extern __shared__ float4 smem4[];
    constexpr int WPW = 32 / G;
    const int NO = P.n_omega;
    SpanRing *rings = reinterpret_cast<SpanRing *>(smem4);
    float *sBeta = reinterpret_cast<float *>(rings + Gm.warps), *sRgap = sBeta + NO;
    float *sTab = sBeta + span_vec_floats(NO);
    float *sB = sTab + (Gm.stage_t ? (size_t)NO * RR : 0);
    span_load<RR>(P, sBeta, sRgap, sTab, Gm.stage_t);
    const int grp_lo = blockIdx.x * Gm.groups_per_cta;
    const int grp_hi = min(grp_lo + Gm.groups_per_cta, Gm.groups_total);
    const int walker_lo = WPW * grp_lo;
    const int walker_hi = min(WPW * grp_hi, P.n_walkers);
    if (Gm.stage_b) {
        const size_t n = (size_t)(walker_hi - walker_lo) * NO;
        const float *src = S.b32 + (size_t)walker_lo * NO;
        for (size_t q = threadIdx.x; q < n; q += blockDim.x) sB[q] = src[q];
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5;
    for (int round = 0; round < Gm.rounds; ++round) {
        const int grp = grp_lo + round * Gm.warps + warp;
        if (grp >= grp_hi) break;                         // uniform across the warp
        if (Gm.stage_t && Gm.stage_b)
            run_span<RR, G, true, true, MODE, LM>(P, S, n0, n1, grp, sTab, sBeta, sRgap, rings[warp], sB, walker_lo);
        else if (Gm.stage_t)
            run_span<RR, G, true, false, MODE, LM>(P, S, n0, n1, grp, sTab, sBeta, sRgap, rings[warp], nullptr, 0);
        else
            run_span<RR, G, false, false, MODE, LM>(P, S, n0, n1, grp, P.Kspan, sBeta, sRgap, rings[warp], nullptr, 0);
    }
}

// How a problem's sweep is laid out over the device with G lanes per walker.
template <int RR, int G>
SpanGeom span_geom(const DevProblem &P, int sms, int smem_max, size_t *smem) {
    constexpr int WPW = 32 / G;
    SpanGeom Gm;
    Gm.groups_total = (P.n_walkers + WPW - 1) / WPW;
    const int ctas = Gm.groups_total < sms ? Gm.groups_total : sms;
    Gm.groups_per_cta = (Gm.groups_total + ctas - 1) / ctas;
    Gm.rounds = (Gm.groups_per_cta + kSpanWarps - 1) / kSpanWarps;
    const size_t tab = (size_t)P.n_omega * RR * 4, spec = (size_t)WPW * Gm.groups_per_cta * P.n_omega * 4;
    Gm.warps = (Gm.groups_per_cta + Gm.rounds - 1) / Gm.rounds;
    *smem = span_ring_bytes(Gm.warps) + (size_t)span_vec_floats(P.n_omega) * 4;
    Gm.stage_t = *smem + tab <= (size_t)smem_max;
    *smem += Gm.stage_t ? tab : 0;
    Gm.stage_b = Gm.stage_t && *smem + spec <= (size_t)smem_max;
    *smem += Gm.stage_b ? spec : 0;
    return Gm;
}

template <int RR, int G, int MODE, int LM = 0>
cudaError_t launch_span_g(const DevProblem &P, const DevState &S, int n0, int n1, const SpanGeom &Gm, size_t smem,
                          cudaStream_t st) {
    cudaError_t e = allow_smem(sweep_span_kernel<RR, G, MODE, LM>);
    if (e != cudaSuccess) return e;
    const int n_ctas = (Gm.groups_total + Gm.groups_per_cta - 1) / Gm.groups_per_cta;
    sweep_span_kernel<RR, G, MODE, LM><<<n_ctas, Gm.warps * 32, smem, st>>>(P, S, n0, n1, Gm);
    return cudaGetLastError();
}

// Lanes per walker of a launch (either gives the same trajectories).  8 lanes keep one warp's chain
// shortest: they run while the spectra are staged and the SM's schedulers have room (20 sweeps, 200
// x 1000: 1500 walkers 2.01 ms against 2.79 with 4 lanes, 4096: 2.85 against 5.7, which does not
// stage).  4 lanes need 0.8 of the instructions per walker: they run where the spectra stay in
// global memory anyway (8192 walkers 6.1 against 7.9 ms, 16384: 9.0 against 15.6; 512 x 2048: 608
// walkers 7.9 against 14.9), and where the population fills the schedulers and is staged (32 x 64,
// 200 sweeps: 4096 walkers 1.70 against 1.86 ms; 608: 1.63 against 1.36).
template <int RR, int MODE>
cudaError_t launch_span(const DevProblem &P, const DevState &S, int n0, int n1, cudaStream_t st) {
    int dev = 0, sms = 0, smem_max = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    size_t m8 = 0;
    const SpanGeom g8 = span_geom<RR, 8>(P, sms, smem_max, &m8);
    if (m8 > (size_t)smem_max) return cudaErrorInvalidValue;
    if constexpr (MODE != kWalk) {
        size_t m4 = 0;
        const SpanGeom g4 = span_geom<RR, 4>(P, sms, smem_max, &m4);
        if (m4 <= (size_t)smem_max && (!g8.stage_b || (g4.stage_b && g8.groups_per_cta >= 6)))
            return launch_span_g<RR, 4, MODE>(P, S, n0, n1, g4, m4, st);
    }
    if constexpr (MODE == kWalk) {
        if (P.walk_len <= 2) return launch_span_g<RR, 8, MODE, 2>(P, S, n0, n1, g8, m8, st);
        if (P.walk_len <= 4) return launch_span_g<RR, 8, MODE, 4>(P, S, n0, n1, g8, m8, st);
        return launch_span_g<RR, 8, MODE, 7>(P, S, n0, n1, g8, m8, st);
    } else {
        return launch_span_g<RR, 8, MODE>(P, S, n0, n1, g8, m8, st);
    }
}

template <int RR>
cudaError_t launch_span_mode(const DevProblem &P, const DevState &S, int n0, int n1, cudaStream_t st) {
    if (P.walk_len > 0) return launch_span<RR, kWalk>(P, S, n0, n1, st);
    if (P.hastings) return launch_span<RR, kHastings>(P, S, n0, n1, st);
    return launch_span<RR, kPlain>(P, S, n0, n1, st);
}

// Many inversions in one persistent launch: blocks take (problem, group range) items from a
// queue, load the item's tables when the problem changes, and run one walker group per warp.  The
// spectra stay in global memory; the column table is staged where it fits in what the launch has
// (smem bytes).
template <int RR, int G, int MODE>
__device__ __forceinline__ void span_item(const BatchProblem &BP, int grp, bool valid, bool reload, char *sm, size_t smem) {
    const int NO = BP.P.n_omega, warps = blockDim.x >> 5;
    SpanRing *rings = reinterpret_cast<SpanRing *>(sm);
    float *sBeta = reinterpret_cast<float *>(rings + warps), *sRgap = sBeta + NO;
    float *sTab = sBeta + span_vec_floats(NO);
    const bool stage_t = span_ring_bytes(warps) + ((size_t)span_vec_floats(NO) + (size_t)NO * RR) * 4 <= smem;
    if (reload) span_load<RR>(BP.P, sBeta, sRgap, sTab, stage_t);
    __syncthreads();
    if (!valid) return;
    if (stage_t)
        run_span<RR, G, true, false, MODE>(BP.P, BP.S, BP.n0, BP.n1, grp, sTab, sBeta, sRgap, rings[threadIdx.x >> 5], nullptr, 0);
    else
        run_span<RR, G, false, false, MODE>(BP.P, BP.S, BP.n0, BP.n1, grp, BP.P.Kspan, sBeta, sRgap, rings[threadIdx.x >> 5], nullptr, 0);
}

template <int G, int MODE>
__global__ void __launch_bounds__(32 * kSpanWarps, 1) sweep_span_batch_kernel(const BatchProblem *probs, const BatchItem *items,
                                                                             int n_items, int *counter, size_t smem) {
    extern __shared__ float4 smem4[];
    char *sm = reinterpret_cast<char *>(smem4);
    __shared__ int s_item;
    int loaded = -1;
    for (;;) {
        __syncthreads();                       // the previous item is finished with the tables
        if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= n_items) break;
        const BatchItem I = items[it];
        const BatchProblem &BP = probs[I.prob];
        const int grp = I.grp_lo + (threadIdx.x >> 5);
        const bool valid = grp < I.grp_hi && BP.n0 < BP.n1, reload = I.prob != loaded;
        loaded = I.prob;
        switch (BP.P.span) {
            case 16: span_item<16, G, MODE>(BP, grp, valid, reload, sm, smem); break;
            case 24: span_item<24, G, MODE>(BP, grp, valid, reload, sm, smem); break;
            default: span_item<32, G, MODE>(BP, grp, valid, reload, sm, smem); break;
        }
    }
}

template <int G, int MODE>
cudaError_t launch_span_batch_g(const BatchProblem *d_probs, const BatchItem *d_items, int n_items, int *d_counter,
                                size_t smem, int warps, cudaStream_t st) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (warps > kSpanWarps) warps = kSpanWarps;
    size_t fixed = 0;
    cudaError_t e = static_smem(sweep_span_batch_kernel<G, MODE>, &fixed);
    if (e == cudaSuccess) e = allow_smem(sweep_span_batch_kernel<G, MODE>, fixed);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(d_counter, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    // persistent: as many blocks as fit on the SMs at once
    int per_sm = 1;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sweep_span_batch_kernel<G, MODE>, warps * 32, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int blocks = n_items < sms * per_sm ? n_items : sms * per_sm;
    sweep_span_batch_kernel<G, MODE><<<blocks, warps * 32, smem, st>>>(d_probs, d_items, n_items, d_counter, smem);
    return cudaGetLastError();
}

}  // namespace

}  // namespace sail
