// FP64 per-hypothesis part of an LM iteration (device functions shared by the evaluation's
// epilogue, the build pass' fused last-CTA epilogue and the kernels that run whole levels).
//
//   gravity term  Eq. 3: r = R gamma^W - gamma^imu, J = [0 | -[a]x], a = R gamma^W
//   range term    Eq. 4-6: P = R^T (q - t), r = P_z - D(P_x, P_y), J = [-n | n x q]
//                 with n = R (-D_x, -D_y, 1) and q = d v
//   assembly      Supp. "Sensor-Prior Fusion in LM": H, g are sums over the terms
//   LM step       Eq. 8: (H + lambda I) dxi = -g by 6x6 Cholesky, Eq. 9: T' = exp(dxi) T
//   acceptance    keep T' iff its objective is lower and enough anchors stay visible
#pragma once

#include <math.h>

#include "pilot_bits.cuh"
#include "pilot_internal.cuh"

namespace pilot {

constexpr double kLambdaMin = 1e-12;
constexpr double kLambdaMax = 1e12;

__device__ __forceinline__ int tri_index(int a, int b) {
    // row-major upper triangle of a 6x6 matrix, a <= b
    return a * 6 - (a * (a - 1)) / 2 + (b - a);
}

// rho and rho' of the Huber function at s >= 0 (delta2 = delta^2).
__device__ __forceinline__ void huber64(double s, double delta, double delta2, double* rho, double* drho) {
    if (within(s, delta2)) {
        *rho = s;
        *drho = 1.0;
    } else {
        const double q = sqrt(s);
        *rho = fma(2.0 * delta, q, -delta2);
        *drho = delta / q;
    }
}

// The step is warp-cooperative: all 32 lanes of one warp run it together.  What bounds it is the
// number of FP64 warp instructions (64 cycles each, however few lanes are active; see
// pilot_bits.cuh), so independent operations of one kind run in one instruction on different
// lanes -- the three rows of a matrix-vector product, the 28 entries a prior adds, the matrix
// entries a Cholesky step updates, the three series, the entries of Exp, V and T' -- values move
// between lanes by shuffles, and comparisons, conversions and truncations are integer
// operations.  About 150 FP64 instructions per step instead of 415: 27 000 -> 17 000 cycles with
// both priors at the paper's schedule.  Each value's arithmetic (operations, order, rounding) is
// the one a single thread would do.

// tri_pair's table: the smaller (or larger) index of upper-triangle entry k (row-major)
__host__ __device__ constexpr unsigned long long pack_tri(bool second) {
    unsigned long long v = 0;
    int k = 0;
    for (int a = 0; a < 6; ++a)
        for (int b = a; b < 6; ++b, ++k) v |= (unsigned long long)(second ? b : a) << (3 * k);
    return v;
}

// Chain c of the FP64 sum of n tile records in 8 chains: records c, c + 8, ..., in order (0 if
// there is none).  A sum starts at its first term and leaves out empty chains: adding them to or
// from zero changes nothing.
template <typename Load>
__device__ __forceinline__ double chain_sum(Load load, int c, int n) {
    if (c >= n) return 0.0;
    double a = widen(load(c));
    for (int t = c + 8; t < n; t += 8) a += widen(load(t));
    return a;
}

__device__ __forceinline__ double shfl_d(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// x0 y0 + x1 y1 + x2 y2 and x0 y0 - x1 y1 with the contractions written out.
__device__ __forceinline__ double dot3(double x0, double y0, double x1, double y1, double x2, double y2) {
    return fma(x2, y2, fma(x0, y0, __dmul_rn(x1, y1)));
}
__device__ __forceinline__ double minus_products(double x0, double y0, double x1, double y1) {
    return fma(x0, y0, -__dmul_rn(x1, y1));
}

// (column, row) of the upper triangle for lane l < 21, three bits per lane
__device__ __forceinline__ void tri_pair(int l, int* a, int* b) {
    // lanes 0-5: a = 0; 6-10: 1; 11-14: 2; 15-17: 3; 18-19: 4; 20: 5
    constexpr unsigned long long ka = pack_tri(false), kb = pack_tri(true);
    *a = (int)(ka >> (3 * l)) & 7;
    *b = (int)(kb >> (3 * l)) & 7;
}

// What the priors add to this lane's entry of H21 | g6 | cost: entry + gw gx (gravity), then + rw rx
// (range), each fused.  They depend on the pose only, so they can be had before the photo sums.
struct PriorTerms {
    double gw, gx, rw, rx;
};

__device__ __forceinline__ double with_priors(double e, const PriorTerms& t) { return fma(t.rw, t.rx, fma(t.gw, t.gx, e)); }

// Gravity direction prior (Eq. 3) and laser range prior (Eq. 4-6; dropped when the range point
// leaves the DSM) at the pose of which lane l < 12 holds entry l.  Gravity: lane i computes a_i and
// r_i; rotation block w [a]x^T [a]x = w (|a|^2 I - a a^T), gradient w [a]x r = w (a x r).
__device__ __forceinline__ PriorTerms prior_terms(const PriorParams& pp, double T, int lane, int ta, int tb) {
    PriorTerms out{0.0, 0.0, 0.0, 0.0};
    const int li = lane % 3, lu = li == 2 ? 0 : li + 1, lv = lu == 2 ? 0 : lu + 1;
    const double R0 = shfl_d(T, 4 * li), R1 = shfl_d(T, 4 * li + 1), R2 = shfl_d(T, 4 * li + 2);
    if (pp.use_gravity) {
        const double ai = dot3(R0, pp.g_world[0], R1, pp.g_world[1], R2, pp.g_world[2]);
        const double ri = ai - pp.g_cam[li];
        // even lanes |a|^2, odd lanes |r|^2: a on lanes 0..2, r on lanes 3..5
        const double y = lane < 3 ? ai : ri;
        const int o = (lane & 1) ? 3 : 0;
        const double v0 = shfl_d(y, o), v1 = shfl_d(y, o + 1), v2 = shfl_d(y, o + 2);
        const double vv = dot3(v0, v0, v1, v1, v2, v2);
        const double aa = shfl_d(vv, 0), s = shfl_d(vv, 1);
        // H entries (3 + i, 3 + k) on lanes 15..20, g entries 3 + i on lanes 24..26, the cost on lane 27
        const bool h = lane < 21;
        const int i = h ? max(ta - 3, 0) : (lane >= 24 && lane < 27 ? lane - 24 : 0), k = h ? max(tb - 3, 0) : 0;
        const int u = i == 2 ? 0 : i + 1, v = u == 2 ? 0 : u + 1;
        // p q - m with p q = -a_i a_k (H) or a_u r_v (g)
        const double p = shfl_d(y, h ? i : u), q = shfl_d(y, h ? k : 3 + v);
        const double m = __dmul_rn(shfl_d(y, v), shfl_d(y, 3 + u));
        const double val = fma(h ? -p : p, q, h ? (i == k ? aa : 0.0) : -m);
        double rho, drho;
        const bool gated = bits(pp.gate_grav) != 0ull && bits(s) > bits(pp.gate_grav2) && bits(s) <= kInfBits;
        huber64(gated ? pp.gate_grav2 : s, pp.huber_grav, pp.huber_grav2, &rho, &drho);
        const double w = bits(drho) == kOneBits ? pp.w_grav : pp.w_grav * drho;
        if (lane == 27) out.gw = pp.w_grav, out.gx = rho;
        else if (!gated && ((lane >= 15 && lane < 21) || (lane >= 24 && lane < 27))) out.gw = w, out.gx = val;
    }
    if (pp.use_range) {
        const double C0 = shfl_d(T, li), C1 = shfl_d(T, 4 + li), C2 = shfl_d(T, 8 + li);
        const double di = pp.q[li] - shfl_d(T, 4 * li + 3);
        const double d0 = shfl_d(di, 0), d1 = shfl_d(di, 1), d2 = shfl_d(di, 2);
        const double Pi = dot3(C0, d0, C1, d1, C2, d2);                           // R^T d
        // x on lanes 0 mod 3, y on lanes 1 mod 3
        const double inv_gsd = pp.dsm_inv_gsd;
        const double gi = fma(Pi - (li == 0 ? pp.dsm_x0 : pp.dsm_y0), inv_gsd, -0.5);
        const bool in = within(gi, li == 0 ? pp.dsm_wmax : pp.dsm_hmax);
        if ((__ballot_sync(0xffffffffu, in) & 3u) != 3u) return out;
        const int ci = min(whole_part(gi), (li == 0 ? pp.dsm_W : pp.dsm_H) - 2);
        const double fi = gi - as_double(ci);
        const int c0 = __shfl_sync(0xffffffffu, ci, 0), r0 = __shfl_sync(0xffffffffu, ci, 1);
        const float* row0 = pp.dsm + (size_t)r0 * pp.dsm_W + c0;
        const float* row1 = row0 + pp.dsm_W;
        const float f00 = row0[0], f01 = row0[1], f10 = row1[0], f11 = row1[1];
        const double ax = shfl_d(fi, 0), ay = shfl_d(fi, 1);
        const double h00 = widen(f00), h10 = widen(f10);
        // bx on lanes 0 mod 3, cy on lanes 1 mod 3, the lower difference on lanes 2 mod 3
        const double diff = (li == 0 ? widen(f01) : (li == 1 ? h10 : widen(f11))) - (li == 2 ? h10 : h00);
        const double bx = shfl_d(diff, 0), cy = shfl_d(diff, 1);
        const double dxy = shfl_d(diff, 2) - bx;
        const double ui = fma(dxy, li == 0 ? ay : ax, li == 0 ? bx : cy);
        const double gradi = ui * inv_gsd;
        const double D = fma(ay, cy, fma(ax, shfl_d(ui, 0), h00));
        const double Dx = shfl_d(gradi, 0), Dy = shfl_d(gradi, 1);
        const double r = shfl_d(Pi, 2) - D;
        const unsigned long long ra = bits(r) & 0x7fffffffffffffffull;
        const bool gated = bits(pp.gate_range) != 0ull && ra > bits(pp.gate_range) && ra <= kInfBits;
        // dr/dP = (-Dx, -Dy, 1); dP/ddelta = R^T [-I | [q]x]  =>  J = [-n | n x q], n = R (-Dx, -Dy, 1)
        const double ni = fma(R0, -Dx, __dmul_rn(R1, -Dy)) + R2;
        const double xi = minus_products(shfl_d(ni, lu), pp.q[lv], shfl_d(ni, lv), pp.q[lu]);
        double rho, drho;
        huber64(gated ? pp.gate_range2 : r * r, pp.huber_range, pp.huber_range2, &rho, &drho);
        const double w = bits(drho) == kOneBits ? pp.w_range : pp.w_range * drho;
        // this lane's J[a] and its factor: J[b] (H), r (g), rho (cost)
        const int a = lane < 21 ? ta : (lane < 27 ? lane - 21 : 0), b = lane < 21 ? tb : 0;
        const double y = lane < 3 ? -ni : xi;                                     // J on lanes 0..5
        const double Ja = shfl_d(y, a), Jb = shfl_d(y, b);
        const double m = w * Ja;
        if (lane == 27) out.rw = pp.w_range, out.rx = rho;
        else if (!gated && lane < 27) out.rw = m, out.rx = lane < 21 ? Jb : r;
    }
    return out;
}

// s = sqrt(d) and inv = 1 / s, each rounded to nearest, for d > 0.  An FP32 estimate of 1 / sqrt(d)
// is refined by Newton's iteration of third order; the square root and the reciprocal are then
// corrected by their remainders, which FMA gives exactly (Markstein, IBM J. Res. Dev. 34(1),
// 1990).  Ten FP64 instructions; the operations themselves outside 2^+-900.
__device__ __forceinline__ void sqrt_inverse(double d, double* s, double* inv) {
    const int e = (int)(((unsigned)__double2hiint(d) >> 20) & 0x7ffu) - 1023;
    if (e < -900 || e > 900) {
        *s = sqrt(d);
        *inv = 1.0 / *s;
        return;
    }
    const int k = e >> 1;
    const double m = scale2(d, -2 * k);                      // in [1, 4)
    float f = __uint_as_float(((unsigned)__double2hiint(m) - 0x38000000u) << 3 | (unsigned)__double2loint(m) >> 29);
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(f));
    const double y0 = widen(f);
    const double t = m * y0;
    const double r = fma(-t, y0, 1.0);
    const double y = fma(fma(0.375, r, 0.5), y0 * r, y0);
    const double s0 = m * y;
    const double sm = fma(fma(-s0, s0, m), scale2(y, -1), s0);
    *s = scale2(sm, k);
    // (a root just below 2 has its reciprocal next to a rounding boundary)
    *inv = (__double2hiint(sm) & 0xfffff) == 0xfffff ? 1.0 / *s : scale2(fma(fma(-sm, y, 1.0), y, y), -k);
}

// lambda / 10, rounded to nearest (a product and a correction by its remainder).
__device__ __forceinline__ double tenth(double v) { return quotient(v, 10.0, 0.1); }

// (H + damping) x = -g by Cholesky.  Lane l < 21 holds entry l of H's upper triangle, (a, b) of
// tri_pair, i.e. entry (b, a) of the factor; lanes 21..26 hold g, treated as a seventh row of the
// matrix (its row of the factor is y, L y = -g), so that one instruction updates every entry
// behind a column.  x on every lane; false (on every lane) if the damped matrix is not positive
// definite.
__device__ __forceinline__ bool damped_solve(double hg, int ta, int tb, double lambda, int mode, double* x, int lane) {
    const int col = lane < 21 ? ta : lane - 21, row = lane < 21 ? tb : 6;
    double v = lane < 21 ? hg : -hg;
    if (row == col) v += mode == 1 ? __dmul_rn(lambda, v) : lambda;
    auto at = [](int r, int c) { return r == 6 ? 21 + c : tri_index(c, r); };    // lane of entry (r, c)
    double inv[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
        const double d = shfl_d(v, tri_index(j, j));
        // d > 0 (a zero, negative or NaN pivot ends the solve)
        if (bits(d) - 1ull >= kInfBits) return false;
        double s;
        sqrt_inverse(d, &s, &inv[j]);
        const double l = v * inv[j];
        if (col == j) v = row == j ? s : l;
        if (j < 5) {
            const double lr = shfl_d(v, at(row, j) & 31), lc = shfl_d(v, at(max(col, j), j) & 31);
            if (col > j) v = fma(-lr, lc, v);
        }
    }
    // L^T x = y: lane 21 + i runs row i
#pragma unroll
    for (int k = 5; k >= 0; --k) {
        x[k] = shfl_d(v, 21 + k) * inv[k];
        if (k > 0) {
            const int i = lane >= 21 ? lane - 21 : 0;
            const double l = shfl_d(v, tri_index(min(i, k), k));
            if (lane >= 21 && i < k) v = fma(-l, x[k], v);
        }
    }
    return true;
}

// Coefficients of Exp and V: A = sin(th)/th, B = (1 - cos th)/th^2, C = (th - sin th)/th^3.
// For th <= 0.25 rad (every LM step in practice) their Maclaurin series in x = th^2,
//   A = sum_k (-x)^k / (2k+1)!,  B = sum_k (-x)^k / (2k+2)!,  C = sum_k (-x)^k / (2k+3)!,
// are summed for k = 0..8 by Horner (the first omitted term is below 1e-27), lane 0 summing
// A, lane 1 B and lane 2 C; larger angles use sin and cos.
__device__ __forceinline__ void exp_coefficients(double x, double* A, double* B, double* C, int lane) {
    if (within(x, 0.0625)) {
        // reciprocal factorials 1/n!, n = 1..19
        constexpr double f[20] = {1.0, 1.0, 1.0 / 2, 1.0 / 6, 1.0 / 24, 1.0 / 120, 1.0 / 720, 1.0 / 5040,
                                  1.0 / 40320, 1.0 / 362880, 1.0 / 3628800, 1.0 / 39916800,
                                  1.0 / 479001600, 1.0 / 6227020800.0, 1.0 / 87178291200.0,
                                  1.0 / 1307674368000.0, 1.0 / 20922789888000.0,
                                  1.0 / 355687428096000.0, 1.0 / 6402373705728000.0,
                                  1.0 / 121645100408832000.0};
        const int o = lane < 3 ? lane : 0;     // series o: coefficients f[2k + 1 + o]
        double v = o == 0 ? f[17] : (o == 1 ? f[18] : f[19]);
#pragma unroll
        for (int k = 7; k >= 0; --k) {
            const double c = o == 0 ? f[2 * k + 1] : (o == 1 ? f[2 * k + 2] : f[2 * k + 3]);
            v = fma(-x, v, c);
        }
        *A = shfl_d(v, 0);
        *B = shfl_d(v, 1);
        *C = shfl_d(v, 2);
    } else {
        const double th = sqrt(x);
        double sn, cs;
        sincos(th, &sn, &cs);
        *A = sn / th;
        *B = (1.0 - cs) / x;
        *C = (th - sn) / (x * th);
    }
}

// T' = exp(xi) T with xi = (nu, omega):  Exp(w) = I + A K + B K^2, V = I + B K + C K^2, K = [w]x,
// K^2 = w w^T - th^2 I.  Lanes 0..8 form Exp, 9..17 V, then lanes 0..11 an entry of Exp T each and
// lanes 12..14 an entry of V nu.  T: lane l < 12 holds entry l; returns entry l of T'.
__device__ __forceinline__ double pose_update(const double* xi, double T, int lane) {
    const double w0 = xi[3], w1 = xi[4], w2 = xi[5];
    const double th2 = dot3(w0, w0, w1, w1, w2, w2);
    double A, B, Cc;
    exp_coefficients(th2, &A, &B, &Cc, lane);
    double W;
    {
        const bool ex = lane < 9;
        const int e = ex ? lane : (lane < 18 ? lane - 9 : 0);
        const int i = e / 3, k = e % 3;
        const double wi = i == 0 ? w0 : (i == 1 ? w1 : w2);
        const double wk = k == 0 ? w0 : (k == 1 ? w1 : w2);
        // K[i][k] = -eps_ikl w_l
        double Kik = 0.0;
        if (i == 0 && k == 1) Kik = -w2;
        if (i == 0 && k == 2) Kik = w1;
        if (i == 1 && k == 0) Kik = w2;
        if (i == 1 && k == 2) Kik = -w0;
        if (i == 2 && k == 0) Kik = -w1;
        if (i == 2 && k == 1) Kik = w0;
        const double K2 = fma(wi, wk, -(i == k ? th2 : 0.0));
        const double I = (i == k) ? 1.0 : 0.0;
        W = fma(ex ? B : Cc, K2, fma(ex ? A : B, Kik, I));
    }
    const bool rot = lane < 12;
    const int i = rot ? lane >> 2 : (lane < 15 ? lane - 12 : 0), k = lane & 3;
    const int w = rot ? 3 * i : 9 + 3 * i;
    const double m0 = shfl_d(W, w), m1 = shfl_d(W, w + 1), m2 = shfl_d(W, w + 2);
    const double t0 = shfl_d(T, k), t1 = shfl_d(T, 4 + k), t2 = shfl_d(T, 8 + k);
    const double b0 = rot ? t0 : xi[0], b1 = rot ? t1 : xi[1], b2 = rot ? t2 : xi[2];
    const double v = dot3(m0, b0, m1, b1, m2, b2);
    const double shift = shfl_d(v, 12 + i);
    return k == 3 ? v + shift : v;
}

__device__ __forceinline__ void store_pose32(float* dst, const double* T) {
    for (int i = 0; i < 12; ++i) dst[i] = (float)T[i];
}

// LM state of one hypothesis on a warp: entry l of T and of the candidate Tc on lane l < 12, of H
// and g on lanes l < 27; the rest on every lane.
struct LmLanes {
    double T, Tc, hg, cost, lambda;
    int n_valid, has_cand, last_fail;
};

// The LM step (kEpiInit or kEpiStep) after a build pass at the candidate: e is this lane's entry of
// the sums, priors included (lane 27: cost, lane 28: visible anchors), read only when evaluated.
// Accepts or rejects, then solves for the next candidate (solve_next).  All 32 lanes.
__device__ __forceinline__ void lm_lanes_step(LmLanes& s, int mode, bool evaluated, int solve_next, int damping_mode,
                                              double e, double min_valid, int lane, int ta, int tb, bool* take) {
    *take = false;
    if (mode == kEpiInit) {
        *take = true;
    } else if (evaluated) {
        *take = shfl_d(e, 27) < s.cost && bits(min_valid) <= bits(shfl_d(e, 28));  // a count and a threshold >= 0
        s.lambda = *take ? fmax(tenth(s.lambda), kLambdaMin) : fmin(s.lambda * 10.0, kLambdaMax);
    }
    if (*take) {
        s.hg = e;
        s.cost = shfl_d(e, 27);
        s.n_valid = whole_part(shfl_d(e, 28));
        if (mode == kEpiStep) s.T = s.Tc;
    }
    s.has_cand = 0;
    if (solve_next) {
        double dxi[6];
        if (!damped_solve(s.hg, ta, tb, s.lambda, damping_mode, dxi, lane)) {
            s.lambda = fmin(s.lambda * 10.0, kLambdaMax);
            s.last_fail = 1;
        } else {
            s.last_fail = 0;
            s.Tc = pose_update(dxi, s.T, lane);
            s.has_cand = 1;
        }
    }
}

// One hypothesis' FP64 step after a build pass at its candidate, its state in memory.  E (29 sums,
// photo term only, in the warp's shared memory) gets the priors at the evaluated pose; then
// (init) it becomes the current state, or (step) the candidate is accepted or rejected; then
// the next candidate is solved for and, if cand32 is given, written there in FP32; or (eval) the
// sums go to eval_out.  All 32 lanes of one warp call it with the same arguments.  Returns whether
// there is a candidate.  The contractions of its products are written out, so that every kernel
// computes the same bits; not inlined, to keep the callers' registers.
static __device__ __noinline__ int lm_update(HypState& st, int mode, int solve_next, int damping_mode,
                                             const PriorParams& prior, const double* E,
                                             double min_valid, float* cand32, double* eval_out, int lane) {
    // every read of the state is issued here, before any write, as one round trip, from L2:
    // the persistent level kernel may step a hypothesis on another SM than the last time
    LmLanes s;
    const int has_cand = __ldcg(&st.has_cand);
    s.cost = __ldcg(&st.cost);
    s.lambda = __ldcg(&st.lambda);
    s.hg = lane < 21 ? __ldcg(st.H + lane) : (lane < 27 ? __ldcg(st.g + lane - 21) : 0.0);
    s.T = lane < 12 ? __ldcg(st.T + lane) : 0.0;
    s.Tc = lane < 12 ? __ldcg(st.Tc + lane) : 0.0;
    s.last_fail = -1;
    const bool evaluated = (mode == kEpiStep) ? (has_cand != 0) : true;
    int ta = 0, tb = 0;
    if (lane < 21) tri_pair(lane, &ta, &tb);
    double e = evaluated && lane < kNumSums ? E[lane] : 0.0;
    if (evaluated) e = with_priors(e, prior_terms(prior, mode == kEpiStep ? s.Tc : s.T, lane, ta, tb));
    if (mode == kEpiEval) {
        if (lane < kNumSums) eval_out[lane] = e;
        if (lane == 0) st.has_cand = 0;
        return 0;
    }
    bool take;
    lm_lanes_step(s, mode, evaluated, solve_next, damping_mode, e, min_valid, lane, ta, tb, &take);
    if (take) {
        if (lane < 21) st.H[lane] = s.hg;
        else if (lane < 27) st.g[lane - 21] = s.hg;
        if (mode == kEpiStep && lane < 12) st.T[lane] = s.T;
    }
    if (s.has_cand && lane < 12) {
        st.Tc[lane] = s.Tc;
        if (cand32) cand32[lane] = narrow(s.Tc);
    }
    if (lane == 0) {
        if (take) {
            st.cost = s.cost;
            st.n_valid = s.n_valid;
        }
        st.lambda = s.lambda;
        if (s.last_fail >= 0) st.last_fail = s.last_fail;
        st.has_cand = s.has_cand;
    }
    __syncwarp();
    return s.has_cand;
}

// A hypothesis whose LM state stays in shared memory through a level, and what its priors add to
// the sums at the pose being evaluated (lane l's factors in terms[l]).
struct ResidentHyp {
    double T[12], Tc[12], hg[27], cost, lambda;
    PriorTerms terms[32];
    int n_valid, has_cand, last_fail, pad;
};

// Level start, by one warp: T is lane l's entry of the pose (l < 12).
__device__ __forceinline__ void resident_begin(ResidentHyp& h, double T, double lambda0, int lane) {
    if (lane < 12) h.T[lane] = T;
    if (lane == 0) {
        h.lambda = lambda0;
        h.cost = 0.0;
        h.n_valid = 0;
        h.has_cand = 1;
        h.last_fail = 0;
    }
}

// The priors at the pose to be evaluated (first: T, else the candidate), by the hypothesis' warp
// before the gathers: they depend on the pose only, and the other warps gather meanwhile.
static __device__ __noinline__ void resident_priors(ResidentHyp& h, const PriorParams& prior, int first, int lane) {
    int ta = 0, tb = 0;
    if (lane < 21) tri_pair(lane, &ta, &tb);
    const double T = lane < 12 ? (first ? h.T[lane] : h.Tc[lane]) : 0.0;
    h.terms[lane] = prior_terms(prior, T, lane, ta, tb);
}

// The LM step on the photo sums E (29, shared memory), by the hypothesis' warp; the next candidate's
// FP32 pose goes to pose.  Returns whether there is one.
static __device__ __noinline__ int resident_step(ResidentHyp& h, const double* E, int mode, int solve_next,
                                                 int damping_mode, double min_valid, float* pose, int lane) {
    int ta = 0, tb = 0;
    if (lane < 21) tri_pair(lane, &ta, &tb);
    LmLanes s;
    s.T = lane < 12 ? h.T[lane] : 0.0;
    s.Tc = lane < 12 && mode == kEpiStep ? h.Tc[lane] : 0.0;
    s.hg = lane < 27 && mode == kEpiStep ? h.hg[lane] : 0.0;
    s.cost = h.cost;
    s.lambda = h.lambda;
    s.n_valid = h.n_valid;
    s.last_fail = h.last_fail;
    const bool evaluated = h.has_cand != 0;
    double e = 0.0;
    if (evaluated) e = with_priors(lane < kNumSums ? E[lane] : 0.0, h.terms[lane]);
    bool take;
    lm_lanes_step(s, mode, evaluated, solve_next, damping_mode, e, min_valid, lane, ta, tb, &take);
    __syncwarp();
    if (lane < 12) {
        h.T[lane] = s.T;
        if (s.has_cand) {
            h.Tc[lane] = s.Tc;
            pose[lane] = narrow(s.Tc);
        }
    }
    if (lane < 27) h.hg[lane] = s.hg;
    if (lane == 0) {
        h.cost = s.cost;
        h.lambda = s.lambda;
        h.n_valid = s.n_valid;
        h.has_cand = s.has_cand;
        h.last_fail = s.last_fail;
    }
    __syncwarp();
    return s.has_cand;
}

// Level end: what the next level, the top-K and the selection read.
__device__ __forceinline__ void resident_end(const ResidentHyp& h, HypState& st, int lane) {
    if (lane < 12) st.T[lane] = h.T[lane];
    if (lane == 0) {
        st.cost = h.cost;
        st.lambda = h.lambda;
        st.n_valid = h.n_valid;
        st.has_cand = h.has_cand;
        st.last_fail = h.last_fail;
    }
}

// lm_update for slot `slot` of a launch described by p (candidate written to p.pose32); all
// 32 lanes of one warp call it.
__device__ inline void lm_step(const EpilogueParams& p, int slot, const double* E, double min_valid, int lane) {
    const int hyp = p.active_idx[slot];
    lm_update(p.state[hyp], p.mode, p.solve_next, p.damping_mode, p.prior, E, min_valid,
              p.pose32 + 12 * hyp, p.eval_out ? p.eval_out + (size_t)slot * kNumSums : nullptr, lane);
}

}  // namespace pilot
