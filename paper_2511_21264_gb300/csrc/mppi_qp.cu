// QP smoothing projection (Eq. 5): each sampled joint-velocity sequence is
// moved to the nearest sequence (in the 2-norm) whose position, velocity,
// acceleration and jerk (r = 0..3, Sec. III) stay within their bounds.
//
// Solver: a fixed number of ADMM iterations (the paper names none).  An
// iteration clips every row, updates its dual and solves
//   (I + rho D^T D) v = vt + rho D^T (w - y).
//
// H <= 80: in the velocities themselves.  With P_t = sum_{i<=t} v_i the rows
// at step t are P_t, v_t, v_t - v_{t-1} and v_t - 2 v_{t-1} + v_{t-2}
// (v_{-1} = the present velocity), their bounds divided by dt, 1, 1/dt,
// 1/dt^2.  The solve is a linear-quadratic control problem in the state
// (P_{t-1}, v_{t-1}, v_{t-2}): one backward pass carries the three costates
// g and leaves a feed-forward term per step, one forward pass plays it out
// against the state feedback (three gains per step).  The gains depend on H,
// rho and the row scales only and come from a Riccati recursion on the host
// in FP64.  Both passes are affine in the three numbers that enter a piece of
// the horizon, so L lanes share one sequence, each with C = ceil(H / L)
// consecutive steps whose velocities and duals stay in registers for all
// iterations: a local pass from zero, log2(L) shuffle rounds with
// precomputed 3 x 3 maps, and a correction (backward: three products per
// step; forward: the pass again from the true state).  When L does not divide
// H, slot 0 of the last lanes is empty; lane 0 is always full.
// Bound: at C = 16 the latency of two warps per scheduler (63-65 warp
// instructions per 32 steps and iteration, 51-53% of the issue slots); with
// more warps and the gains in shared memory the issue slots (72-79
// instructions, 65-70%) and the 128-bit loads (four wavefronts each even when
// the lanes share addresses), which is no faster: a shape's register bound is
// set so that most gains stay in registers.  One GB300, 30 iterations:
// 57344 x 64 takes 312-319 us against 676 with the long form below (one warp per
// scheduler, 30% of the issue slots); 5000 x 27 takes 31 us against 38 with one
// lane per step and a dense inverse; 1024 samples x 14 joints x 32 drawn and
// projected 48 us against 92.
//
// Longer horizons: one thread per sequence, in the coordinates
//   x_i = sum_{t<i} v_t   (i = 1..H, the position offset over dt),
// where every constraint row touches at most four consecutive x_i and the
// system  N x = B^T vt + rho D^T (w - y),  N = B^T B + rho D^T D  (B: first
// differences, D: the scaled rows) is banded with bandwidth 3; its FP32 band
// Cholesky factor is shared by every sequence of a class (one class per
// joint).  The differences of positions cost a digit: at H = 96 any other
// order of the same FP32 operations moves the result by 1.5e-5 of its norm,
// at H = 128 by 2e-5, so this form keeps its horizons.  For 32 < H <= 80 the
// lane form solves the system of the same FP32 band factor (its rounding
// alone moves the solution by 2e-5 at H = 64) and agrees with this form to
// 1e-5 at H = 64, 1.3e-5 at H = 80.
//
// Per iteration a thread of the long form makes one forward sweep over t that
// evaluates the four rows at t, updates their scaled duals y (w = clip(D x +
// y), y = D x + y - w), accumulates the right-hand side D^T (w - y) and runs
// the forward substitution three indices behind, then one backward
// substitution sweep.  The per-thread vectors live in shared memory, laid
// out [t][thread] so that a warp's accesses are conflict-free.
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <cstring>
#include <vector>

#include "../../include/mppi.h"
#include "mppi_device.cuh"
#include "mppi_internal.h"

namespace mppi {

namespace {

constexpr int QP_MAX_C = 16;      // steps per lane
constexpr int QP_MAX_L = 16;      // lanes per sequence
constexpr int QP_DENSE_MAX_H = 32;  // up to here no band factor is rounded to FP32
constexpr int QP_LANES_MAX_H = 80;  // longest horizon of the lane form
constexpr int QP_THREADS = 128;   // standalone lane form
// float4s of the largest table: the long form's, or the lane form's with L = 16
constexpr int QP_MAX_TABLE = 2 * (QP_LANES_MAX_H + QP_MAX_L) + 6 * 4 * QP_MAX_L;
static_assert(QP_MAX_TABLE >= 2 * MPPI_QP_MAX_H, "the long form's rows fit");

int log2i(int v) {
    int r = 0;
    while ((1 << r) < v) ++r;
    return r;
}

struct Mat3 {
    double m[3][3];
};
Mat3 identity3() { return {{{1, 0, 0}, {0, 1, 0}, {0, 0, 1}}}; }
Mat3 mul3(const Mat3& a, const Mat3& b) {
    Mat3 c{};
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j)
            for (int k = 0; k < 3; ++k) c.m[i][j] += a.m[i][k] * b.m[k][j];
    return c;
}

// N of one factor in band form, N[i][d] = N(i, i - d), and its Cholesky factor
// in the same form.  Entries with d > i couple to the fixed x before the first
// step (x_0 = 0, x_{-1} = -qd); the factor ignores them.
using Band = std::vector<std::array<double, 4>>;

// x-coordinate form of one scaled row group: value at t is
// s * (x_{t+1} + c1 x_t + c2 x_{t-1} + c3 x_{t-2})
void add_group(Band& N, int H, double w, const double* c, int t0) {
    for (int t = t0; t < H; ++t)
        for (int a = 0; a < 4 && a <= t; ++a)  // x index t + 1 - a (1-based)
            for (int b = a; b < 4; ++b) N[t - a][b - a] += w * c[a] * c[b];
}

Band system_band(int H, double rho, const double sc[4]) {
    Band N(H, {0.0, 0.0, 0.0, 0.0});
    static const double cB[4] = {1, -1, 0, 0}, cP[4] = {1, 0, 0, 0}, cA[4] = {1, -2, 1, 0}, cJ[4] = {1, -3, 3, -1};
    add_group(N, H, 1.0, cB, 0);                  // objective 1/2 |B x - vt|^2
    add_group(N, H, rho * sc[0] * sc[0], cP, 0);  // position rows
    add_group(N, H, rho * sc[1] * sc[1], cB, 0);  // velocity rows
    add_group(N, H, rho * sc[2] * sc[2], cA, 0);  // acceleration rows
    add_group(N, H, rho * sc[3] * sc[3], cJ, 1);  // jerk rows, t >= 1
    return N;
}

bool band_cholesky(Band& N) {
    const int H = (int)N.size();
    for (int i = 0; i < H; ++i)
        for (int d = std::min(i, 3); d >= 0; --d) {
            double t = N[i][d];
            for (int e = d + 1; e <= 3 && i - e >= 0; ++e) t -= N[i][e] * N[i - d][e - d];
            if (d == 0) {
                if (!(t > 0.0) || !std::isfinite(t)) return false;
                N[i][0] = std::sqrt(t);
            } else {
                N[i][d] = t / N[i - d][0];
            }
        }
    return true;
}

// Standalone table, handed over as a kernel parameter.
struct QPTable {
    float4 v[QP_MAX_TABLE];
};

}  // namespace

// Lanes per sequence for n sequences of H steps (0: the long form): the
// fewest that keep C <= 16 steps per lane (fewer shuffle rounds and tails),
// then twice as many while the launch has less than 16 warps per SM (4 in the
// controller form, whose CTAs are whole samples) and a lane keeps seven steps, or
// less than two warps per SM and three steps.  So lanes of a shared sequence
// hold at least two steps.  The 152 SMs of a GB300 are a constant here, not the
// device's count: the split orders the sums, so a result follows from n and H
// alone (one split for every n would cost 38% at n = 1000, H = 32, 33% at n = 300,
// H = 64).  One GB300, 30 iterations, us with
// 1 / 2 / 4 / 8 / 16 lanes:
//   n = 57344, H = 64:  - / - / 312 / 318 / 474     H = 32: - / 140 / 148 / 195 / 404
//   n = 57344, H = 16:  101 / 75 / 91 / 162 / 386   n = 14336, H = 64: - / - / 107 / 92 / 134
//   n = 14336, H = 32:  - / 50 / 44 / 56 / 113      n = 5000, H = 27:  - / 36 / 32 / 33 / 54
//   n = 1000, H = 32:   - / 37 / 29 / 21 / 21       n = 300, H = 64:   - / - / 41 / 32 / 24
// and drawn and projected, K samples x 14 joints:
//   K = 1024, H = 32:   - / 48 / 55 / 77 / 110      K = 1024, H = 20: - / 33 / 39 / 68 / 110
//   K = 4096, H = 64:   - / - / 336 / 358 / 499     K = 256, H = 16: 45 / 31 / 28 / 22 / 36
int qp_lanes(int n, int H, bool drawn) {
    if (H > QP_LANES_MAX_H) return 0;
    int L = 1;
    while ((H + L - 1) / L > QP_MAX_C) L *= 2;
    const auto grow = [&](int warps_per_sm, int min_c) {
        while (L < QP_MAX_L && (long long)n * L < 152LL * 32 * warps_per_sm && (H + 2 * L - 1) / (2 * L) >= min_c) L *= 2;
    };
    grow(drawn ? 4 : 16, 7);
    grow(2, 3);
    return L;
}

// float4s of a table: the band factor's rows (L = 0), or per slot and lane the
// gains (1/Q, K_P, K_1, K_2) and the costate correction, then per shuffle round
// the backward and forward maps.
int qp_table_size(int H, int L) { return L == 0 ? 2 * H : 2 * ((H + L - 1) / L) * L + 6 * log2i(L) * L; }

// Table of one factor (horizon H, penalty rho, row scales sc; 0 = free group).
// L = 0: the long form, 2 H rows of the band factor, forward then backward.
// Else the lane form for L lanes per sequence.
int qp_table(int H, int L, double rho, const double sc[4], float4* out) {
    Band N = system_band(H, rho, sc);
    if (H > QP_DENSE_MAX_H) {
        Band F = N;
        if (!band_cholesky(F)) return MPPI_ERR_CHOLESKY;
        auto l = [&](int i, int d) { return i < H && d <= i ? (float)F[i][d] : 0.0f; };
        if (L == 0) {
            for (int i = 0; i < H; ++i) {
                const float dinv = (float)(1.0 / F[i][0]);
                out[i] = make_float4(dinv, l(i, 1), l(i, 2), l(i, 3));
                out[H + i] = make_float4(dinv, l(i + 1, 1), l(i + 2, 2), l(i + 3, 3));
            }
            return MPPI_OK;
        }
        // the system of the FP32 factor, as the long form solves it
        for (int i = 0; i < H; ++i) {
            F[i][0] = 1.0 / (double)(float)(1.0 / F[i][0]);
            for (int d = 1; d <= 3; ++d) F[i][d] = (double)(float)F[i][d];
        }
        for (int i = 0; i < H; ++i)
            for (int d = 0; d <= 3 && d <= i; ++d) {
                N[i][d] = 0.0;
                for (int e = d; e <= 3 && e <= i; ++e) N[i][d] += F[i][e] * F[i - d][e - d];
            }
    }
    // Riccati recursion over x_H .. x_1 with the value function S of (x_{t-1},
    // x_{t-2}, x_{t-3}); the gains in terms of (P, v1, v2) = (x_{t-1}, x_{t-1} -
    // x_{t-2}, x_{t-2} - x_{t-3}) and of v = x_t - x_{t-1}
    std::vector<double> iq(H);
    std::vector<Mat3> F(H);  // closed-loop map of step t on (P, v1, v2)
    std::vector<double> K(3 * (size_t)H);
    double S[3][3] = {};
    for (int t = H - 1; t >= 0; --t) {
        const double qxx = N[t][0] + S[0][0];
        const double qx[3] = {N[t][1] + S[0][1], N[t][2] + S[0][2], N[t][3]};
        if (!(qxx > 0.0) || !std::isfinite(qxx)) return MPPI_ERR_CHOLESKY;
        double Sn[3][3] = {{S[1][1], S[1][2], 0.0}, {S[1][2], S[2][2], 0.0}, {0.0, 0.0, 0.0}};
        for (int i = 0; i < 3; ++i)
            for (int k = 0; k < 3; ++k) Sn[i][k] -= qx[i] * qx[k] / qxx;
        std::memcpy(S, Sn, sizeof S);
        iq[t] = 1.0 / qxx;
        double* k3 = &K[3 * t];
        k3[0] = 1.0 + (qx[0] + qx[1] + qx[2]) / qxx;
        k3[1] = -(qx[1] + qx[2]) / qxx;
        k3[2] = -qx[2] / qxx;
        F[t] = {{{1.0 - k3[0], -k3[1], -k3[2]}, {-k3[0], -k3[1], -k3[2]}, {0.0, 1.0, 0.0}}};
    }
    const int C = (H + L - 1) / L, full = H - L * (C - 1), R = log2i(L);
    std::memset(out, 0, (size_t)qp_table_size(H, L) * sizeof(float4));
    std::vector<Mat3> Bm(L), Fm(L);  // costate and state maps of a lane's steps
    int t0 = 0;
    for (int p = 0; p < L; ++p) {
        const int n = p < full ? C : C - 1, e = C - n;  // slot of the lane's first step
        Mat3 G = identity3(), X = identity3();
        for (int s = n - 1; s >= 0; --s) {
            const int t = t0 + s;
            float4& kc = out[(e + s) * L + p];
            kc = make_float4((float)iq[t], (float)K[3 * t], (float)K[3 * t + 1], (float)K[3 * t + 2]);
            float4& ps = out[(C + e + s) * L + p];  // iq B^T G: v takes g_P + g_1 of the costate entering the lane
            ps = make_float4((float)(iq[t] * (G.m[0][0] + G.m[1][0])), (float)(iq[t] * (G.m[0][1] + G.m[1][1])),
                             (float)(iq[t] * (G.m[0][2] + G.m[1][2])), 0.0f);
            Mat3 Ft{};
            for (int i = 0; i < 3; ++i)
                for (int k = 0; k < 3; ++k) Ft.m[i][k] = F[t].m[k][i];
            G = mul3(Ft, G);
            X = mul3(X, F[t]);
        }
        Bm[p] = G;
        Fm[p] = X;
        t0 += n;
    }
    for (int r = 0; r < R; ++r) {
        const int off = 1 << r;
        float4* b = out + 2 * C * L + 6 * r * L;
        for (int p = 0; p < L; ++p)
            for (int i = 0; i < 3; ++i) {
                if (p + off < L)
                    b[i * L + p] = make_float4((float)Bm[p].m[i][0], (float)Bm[p].m[i][1], (float)Bm[p].m[i][2], 0.0f);
                if (p - off >= 0)
                    b[(3 + i) * L + p] = make_float4((float)Fm[p].m[i][0], (float)Fm[p].m[i][1], (float)Fm[p].m[i][2], 0.0f);
            }
        std::vector<Mat3> Bn = Bm, Fn = Fm;
        for (int p = 0; p < L; ++p) {
            if (p + off < L) Bn[p] = mul3(Bm[p], Bm[p + off]);
            if (p - off >= 0) Fn[p] = mul3(Fm[p], Fm[p - off]);
        }
        Bm = Bn;
        Fm = Fn;
    }
    return MPPI_OK;
}

// Class record from 8 physical bounds: free groups get scale 0.
void qp_make_class(const float b[8], const float sc[4], float rho, QPClass* c) {
    std::memset(c, 0, sizeof *c);
    for (int g = 0; g < 4; ++g) {
        c->lo[g] = b[2 * g];
        c->hi[g] = b[2 * g + 1];
        const bool free_g = std::isinf(b[2 * g]) && b[2 * g] < 0 && std::isinf(b[2 * g + 1]) && b[2 * g + 1] > 0;
        c->s[g] = free_g ? 0.0f : sc[g];
    }
    c->rho = rho;
}

int qp_validate(const float b[8], const float sc[4], float rho) {
    if (!(rho > 0.0f) || !std::isfinite(rho)) return MPPI_ERR_INVALID_ARG;
    for (int g = 0; g < 4; ++g) {
        if (std::isnan(b[2 * g]) || std::isnan(b[2 * g + 1]) || !(b[2 * g] <= b[2 * g + 1])) return MPPI_ERR_INVALID_ARG;
        if (!(sc[g] > 0.0f) || !std::isfinite(sc[g])) return MPPI_ERR_INVALID_ARG;
    }
    return MPPI_OK;
}

// ---------------------------------------------------------------------------
// device
// ---------------------------------------------------------------------------

// One row: s = val + y, w = clip(s), y = s - w; returns w - y = 2 w - s.
__device__ __forceinline__ float qp_row(float val, float& y, float lo, float hi) {
    const float s = val + y;
    const float w = fminf(fmaxf(s, lo), hi);
    y = s - w;
    return __fmaf_rn(2.0f, w, -s);
}

// acc += m x, m the rows at t[0], t[L], t[2 L]
__device__ __forceinline__ void qp_map(Run<const float4> t, int L, const float (&x)[3], float (&acc)[3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float4 m = t[i * L];
        acc[i] = __fmaf_rn(m.z, x[2], __fmaf_rn(m.y, x[1], __fmaf_rn(m.x, x[0], acc[i])));
    }
}

// ADMM iterations of one sequence held by L consecutive lanes of a warp, this
// one (p) with the C slots v (the input on entry, the last iterate on exit;
// slot 0 unused when `empty`).  T: the table, lane p's entries from p on.
template <int C>
__device__ __forceinline__ void qp_admm(const QPClass& c, Run<const float4> T, int L, int p, bool empty, int iters, float dt,
                                        float q, float qd, float (&v)[C]) {
    const float idt = 1.0f / dt, dt2 = dt * dt;
    const float Plo = (c.lo[0] - q) * idt, Phi = (c.hi[0] - q) * idt, Vlo = c.lo[1], Vhi = c.hi[1];
    const float Alo = c.lo[2] * dt, Ahi = c.hi[2] * dt, Jlo = c.lo[3] * dt2, Jhi = c.hi[3] * dt2;
    const float rP = c.rho * c.s[0] * c.s[0], rV = c.rho * c.s[1] * c.s[1], rA = c.rho * c.s[2] * c.s[2];
    const float rJ = c.rho * c.s[3] * c.s[3], rJ2 = -2.0f * rJ;
    const float on0 = empty ? 0.0f : 1.0f, onJ = empty || p == 0 ? 0.0f : 1.0f;  // slot 0's rows; step 0 has no jerk row
    const float qd0 = p == 0 ? qd : 0.0f;
    const Run<const float4> kc = sub_run(T, p), psi = sub_run(T, C * L + p), maps = sub_run(T, 2 * C * L + p);

    float vt[C], P[C], y[4][C];
    // positions of the start point, and the two velocities before slot 0
    float acc = 0.0f;
#pragma unroll
    for (int i = 0; i < C; ++i) {
        vt[i] = v[i];
        y[0][i] = y[1][i] = y[2][i] = y[3][i] = 0.0f;
        acc += i == 0 && empty ? 0.0f : v[i];
        P[i] = acc;
    }
    float pre = acc;
    for (int off = 1; off < L; off <<= 1) {
        const float o = __shfl_up_sync(FULL, pre, off, L);
        if (p >= off) pre += o;
    }
    pre = __shfl_up_sync(FULL, pre, 1, L);
    if (p == 0) pre = 0.0f;
#pragma unroll
    for (int i = 0; i < C; ++i) P[i] += pre;
    float x1, x2;
    {
        // last two velocities of the lanes before; the case of a lane with one
        // step is for any split (qp_lanes makes none: without it, the compiler
        // spills 96 bytes of 16 steps per lane instead of 12, and 4096 samples x 64
        // take 652 us an iteration instead of 603)
        float l1 = v[C - 1], l2 = C > 1 ? v[C > 1 ? C - 2 : 0] : 0.0f;
        const bool one = C == 1 || (C == 2 && empty);
        float a1 = __shfl_up_sync(FULL, l1, 1, L), a2 = __shfl_up_sync(FULL, l2, 1, L);
        const float b1 = __shfl_up_sync(FULL, l1, 2, L);
        const bool onep = __shfl_up_sync(FULL, (int)one, 1, L) != 0;
        if (onep) a2 = p >= 2 ? b1 : qd;
        x1 = p == 0 ? qd : a1;
        x2 = p == 0 ? 0.0f : a2;
    }
    // the velocities before slot 0; an empty slot 0 holds the last one itself
    float a1 = empty ? x2 : x1, a2 = x2;
    if (empty) v[0] = x1;

    for (int it = 0; it < iters; ++it) {
        // rows and costate, last slot first; ff replaces P
        float gP = 0.0f, g1 = 0.0f, g2 = 0.0f;
        float d1 = v[C - 1] - (C > 1 ? v[C > 1 ? C - 2 : 0] : a1);
#pragma unroll
        for (int i = C - 1; i >= 0; --i) {
            const float vm1 = i >= 1 ? v[i - 1] : a1, vm2 = i >= 2 ? v[i - 2] : (i == 1 ? a1 : a2);
            const float dp = vm1 - vm2;
            float tP = qp_row(P[i], y[0][i], Plo, Phi);
            float tV = qp_row(v[i], y[1][i], Vlo, Vhi);
            float tA = qp_row(d1, y[2][i], Alo, Ahi);
            float tJ = qp_row(d1 - dp, y[3][i], Jlo, Jhi);
            if (i == 0) {
                tP *= on0;
                tV *= on0;
                tA *= on0;
                tJ *= onJ;
            }
            const float4 k = kc[i * L];
            float cc = __fmaf_rn(rP, tP, vt[i]);
            cc = __fmaf_rn(rV, tV, cc);
            cc = __fmaf_rn(rA, tA, cc);
            cc = __fmaf_rn(rJ, tJ, cc) + (gP + g1);
            P[i] = k.x * cc;
            const float nP = __fmaf_rn(-k.y, cc, __fmaf_rn(rP, tP, gP));
            const float n1 = __fmaf_rn(-k.z, cc, __fmaf_rn(-rA, tA, __fmaf_rn(rJ2, tJ, g2)));
            const float n2 = __fmaf_rn(-k.w, cc, rJ * tJ);
            gP = nP;
            g1 = i == 0 && empty ? g1 : n1;
            g2 = i == 0 && empty ? g2 : n2;
            d1 = dp;
        }
        float g[3] = {gP, g1, g2}, s[3];
        Run<const float4> mp = maps;
        for (int off = 1; off < L; off <<= 1, mp = sub_run(mp, 6 * L)) {
#pragma unroll
            for (int k = 0; k < 3; ++k) s[k] = __shfl_down_sync(FULL, g[k], off, L);
            qp_map(mp, L, s, g);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            s[k] = __shfl_down_sync(FULL, g[k], 1, L);
            if (p == L - 1) s[k] = 0.0f;
        }
        // feed-forward with the true costate; the forward pass from zero
        float st[3] = {0.0f, qd0, 0.0f};
#pragma unroll
        for (int i = 0; i < C; ++i) {
            const float4 w = psi[i * L];
            P[i] = __fmaf_rn(w.z, s[2], __fmaf_rn(w.y, s[1], __fmaf_rn(w.x, s[0], P[i])));
            const float4 k = kc[i * L];
            const float x = __fmaf_rn(-k.z, st[1], __fmaf_rn(-k.w, st[2], __fmaf_rn(-k.y, st[0], P[i])));
            const bool skip = i == 0 && empty;
            st[0] += skip ? 0.0f : x;
            st[2] = skip ? st[2] : st[1];
            st[1] = skip ? st[1] : x;
        }
        mp = sub_run(maps, 3 * L);
        for (int off = 1; off < L; off <<= 1, mp = sub_run(mp, 6 * L)) {
#pragma unroll
            for (int k = 0; k < 3; ++k) s[k] = __shfl_up_sync(FULL, st[k], off, L);
            qp_map(mp, L, s, st);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            s[k] = __shfl_up_sync(FULL, st[k], 1, L);
            st[k] = p == 0 ? (k == 1 ? qd : 0.0f) : s[k];
        }
        a1 = empty ? st[2] : st[1];
        a2 = st[2];
#pragma unroll
        for (int i = 0; i < C; ++i) {
            const float4 k = kc[i * L];
            const float x = __fmaf_rn(-k.z, st[1], __fmaf_rn(-k.w, st[2], __fmaf_rn(-k.y, st[0], P[i])));
            const bool skip = i == 0 && empty;
            v[i] = skip ? st[1] : x;
            st[0] += skip ? 0.0f : x;
            P[i] = st[0];
            st[2] = skip ? st[2] : st[1];
            st[1] = skip ? st[1] : x;
        }
    }
}

// Shared memory of a CTA: the stage (one padded row of H values per
// sequence), then the tables (and, while sampling, the normals).
__device__ __forceinline__ int qp_row_stride(int H) { return H | 1; }

// The CTA's sequences from the stage through the iterations and back.
template <int C>
__device__ __forceinline__ void qp_solve(const QPArgs& a, const QPClass& c, Run<const float4> T, Run<float> row, int p,
                                         float q, float qd) {
    const int full = a.H - a.L * (C - 1);  // lanes with C steps; the others leave slot 0 empty
    const bool empty = p >= full;
    const int t0 = p * C - (empty ? p - full + 1 : 0);  // step of slot 0
    float v[C];
#pragma unroll
    for (int i = 0; i < C; ++i) v[i] = i == 0 && empty ? 0.0f : row[t0 + i];
    qp_admm<C>(c, T, a.L, p, empty, a.iters, a.dt, q, qd, v);
#pragma unroll
    for (int i = 0; i < C; ++i)
        if (!(i == 0 && empty)) row[t0 + i] = v[i];
}

// Standalone form: one class, the table as a kernel parameter.
template <int C>
__global__ void __launch_bounds__(QP_THREADS, C <= 4 ? 6 : C <= 8 ? 4 : C <= 12 ? 3 : 2) qp_project_kernel(QPArgs a, const __grid_constant__ QPClass c,
                                                               const __grid_constant__ QPTable table) {
    extern __shared__ __align__(16) float4 qsm[];
    const int tid = threadIdx.x, L = a.L, p = tid & (L - 1), seqs = QP_THREADS / L, rs = qp_row_stride(a.H);
    const int nt = a.tab_size;
    const Run<float4> tab = make_run(qsm, nt);
    const Run<float> stage = make_run(reinterpret_cast<float*>(qsm + nt), seqs * rs);
    for (int t = tid; t < nt; t += QP_THREADS) tab[t] = table.v[MPPI_IN_RANGE(t, QP_MAX_TABLE) ? t : 0];
    const long long i0 = (long long)blockIdx.x * seqs;
    const int ns = (int)(a.n - i0 < seqs ? a.n - i0 : seqs);  // sequences of this CTA
    const int lane = tid & 31, warp = tid >> 5;
    for (int r = warp; r < seqs; r += QP_THREADS / 32)
        for (int t = lane; t < a.H; t += 32)  // rows past the last sequence run on zeros
            stage[r * rs + t] = r < ns ? ld_checked(a.vin, (i0 + r) * a.H + t, a.in_n) : 0.0f;
    __syncthreads();
    const int sq = tid / L;
    const long long i = i0 + (sq < ns ? sq : ns - 1);
    qp_solve<C>(a, c, tab, sub_run(stage, sq * rs, a.H), p, ld_checked(a.q0, i, a.n), ld_checked(a.qd0, i, a.n));
    __syncthreads();
    for (int r = warp; r < ns; r += QP_THREADS / 32)
        for (int t = lane; t < a.H; t += 32)
            if (MPPI_IN_RANGE((i0 + r) * a.H + t, a.out_n)) a.out[(i0 + r) * a.H + t] = stage[r * rs + t];
}

// Controller form: S = 16 / L samples per CTA, every joint of each (sequence
// s * nu + j), drawn here (one thread per Philox block, then the row
// products), projected and written to the h-major sample buffer as
// contiguous rows of S nu values.
template <int C>
__global__ void __launch_bounds__(224, C <= 4 ? 3 : C <= 8 ? 2 : 1) qp_sample_kernel(QPArgs a) {
    extern __shared__ __align__(16) float4 qsm[];
    const int tid = threadIdx.x, T = blockDim.x, L = a.L, p = tid & (L - 1), S = QP_MAX_L / L, nu = a.nu, H = a.H;
    const int rs = qp_row_stride(H), k0 = blockIdx.x * S, nb = (nu + 3) / 4;
    const int ns = a.per_cls - k0 < S ? a.per_cls - k0 : S;  // samples of this CTA
    const Run<float> stage = make_run(reinterpret_cast<float*>(qsm), S * nu * rs);
    float4* const after = qsm + ((S * nu * rs + 3) >> 2);
    const Run<float4> draws = make_run(after, S * H * nb), tab = make_run(after, a.n_tab * a.tab_size);
    const Run<float> z = make_run(reinterpret_cast<float*>(after), 4 * S * H * nb);
    const uint2 key = make_uint2((uint32_t)a.seed, (uint32_t)(a.seed >> 32));
    const uint32_t iter = (uint32_t)(a.iter_ptr ? *a.iter_ptr : a.iter_val);
    for (int b = tid; b < S * H * nb; b += T) {
        const int s = b / (H * nb), h = b / nb - s * H, jb = b % nb;
        float z4[4];
        block_normals4(philox4x32_10(make_uint4((uint32_t)jb, (uint32_t)h, (uint32_t)(k0 + s), iter), key), z4);
        draws[b] = make_float4(z4[0], z4[1], z4[2], z4[3]);
    }
    __syncthreads();
    const int jt = tid % nu;  // 16 nu threads: a thread stays with its joint
    for (int e = tid / nu; e < S * H; e += QP_MAX_L) {
        // the value the rollout's sampler draws, unclamped
        const int j = jt, s = e / H, h = e - s * H;
        const Run<float> zr = sub_run(z, e * 4 * nb, 4 * nb);
        float v = ld_checked(a.u_nom, (long long)h * nu + j, (long long)H * nu);
        if (a.Lfac) {
            const long long r0 = ((long long)h * nu + j) * nu, n_l = (long long)H * nu * nu;
            for (int i = 0; i <= j; ++i) v = __fmaf_rn(ld_checked(a.Lfac, r0 + i, n_l), zr[i], v);
        } else {
            v = __fmaf_rn(ld_checked(a.sigma, j, nu), zr[j], v);
        }
        stage[(s * nu + j) * rs + h] = v;
    }
    __syncthreads();
    for (int t = tid; t < a.n_tab * a.tab_size; t += T) tab[t] = __ldg(&a.tab[t]);
    __syncthreads();
    const int sq = tid / L, j = sq % nu;
    const QPClass c = a.cls[MPPI_IN_RANGE(j, a.n_cls) ? j : 0];
    qp_solve<C>(a, c, sub_run(tab, a.n_tab > 1 ? j * a.tab_size : 0, a.tab_size), sub_run(stage, sq * rs, H), p, ld_checked(a.q0, j, a.n_cls),
                ld_checked(a.qd0, j, a.n_cls));
    __syncthreads();
    const int i = tid % (S * nu);  // L rows of S nu values at a time
    if (i < ns * nu)
        for (int h = tid / (S * nu); h < H; h += L) {
            const long long o = ((long long)h * a.per_cls + k0) * nu + i;
            if (MPPI_IN_RANGE(o, a.out_n)) a.out[o] = stage[i * rs + h];
        }
}

// ---------------------------------------------------------------------------
// long form
// ---------------------------------------------------------------------------
// scaled bounds of one row group: [s lo, s hi], or unbounded for a free group
__device__ __forceinline__ void qp_bound(float s, float lo, float hi, float& blo, float& bhi) {
    if (s == 0.0f) {
        blo = -INFINITY;
        bhi = INFINITY;
    } else {
        blo = s * lo;
        bhi = s * hi;
    }
}

// One row: s = val + y; w = clip(s); y = s - w; returns e = rho s_g (w - y).
__device__ __forceinline__ float qp_scaled_row(float val, float& y, float lo, float hi, float rs) {
    const float s = val + y;
    const float w = fminf(fmaxf(s, lo), hi);
    y = s - w;
    return rs * (w - y);
}

// ADMM iterations of one thread's sequence.  xs[t*T] = x_{t+1} on entry holds
// the start point, the prefix sums of vt; y[t*T] = 0; rhs(t) = (B^T vt)_{t+1},
// row(r) = row r of the band factor.  On exit xs holds the last iterate.
template <class Row, class Rhs>
__device__ __forceinline__ void qp_long_admm(const QPClass& c, const Row& row, const Rhs& rhs, int H, int iters, float dt,
                                             float q, float qd, float* xs, float4* yv, int T) {
    const float s0 = c.s[0], s1 = c.s[1], s2 = c.s[2], s3 = c.s[3];
    const float rs0 = c.rho * s0, rs1 = c.rho * s1, rs2 = c.rho * s2, rs3 = c.rho * s3;
    float Plo, Phi, Vlo, Vhi, Alo, Ahi, A0lo, A0hi, Jlo, Jhi, J1lo, J1hi;
    const float idt = 1.0f / dt, dt2 = dt * dt;
    qp_bound(s0, (c.lo[0] - q) * idt, (c.hi[0] - q) * idt, Plo, Phi);
    qp_bound(s1, c.lo[1], c.hi[1], Vlo, Vhi);
    qp_bound(s2, c.lo[2] * dt, c.hi[2] * dt, Alo, Ahi);
    qp_bound(s2, c.lo[2] * dt + qd, c.hi[2] * dt + qd, A0lo, A0hi);  // v_{-1} = qd moved into the bounds
    qp_bound(s3, c.lo[3] * dt2, c.hi[3] * dt2, Jlo, Jhi);
    qp_bound(s3, c.lo[3] * dt2 - qd, c.hi[3] * dt2 - qd, J1lo, J1hi);
    // slot index i (0 <= i < H) of this thread's vectors and band rows;
    // checked in the bounds-check build, the identity otherwise
    auto sl = [H](int i) { return MPPI_IN_RANGE(i, H) ? i : 0; };

    for (int it = 0; it < iters; ++it) {
        // forward sweep: rows at t, right-hand side, forward substitution
        float x0 = 0.0f;                         // x_t (x_0 and earlier are zero)
        float d1p = 0.0f, d2p = 0.0f;            // first and second differences at t-1
        float r0 = 0.0f, r1 = 0.0f, r2 = 0.0f;   // rhs of x_{t-2}, x_{t-1}, x_t
        float z1 = 0.0f, z2 = 0.0f, z3 = 0.0f;   // z_{i-1}, z_{i-2}, z_{i-3} of the substitution
        // unrolled so that the next steps' loads are in flight during the
        // substitution chain (the operations and their order are unchanged)
#pragma unroll 4
        for (int t = 0; t < H; ++t) {
            const float xp1 = xs[(size_t)sl(t) * T], bt = rhs(t);
            float4 y = yv[(size_t)sl(t) * T];
            const float d1 = xp1 - x0, d2 = d1 - d1p, d3 = d2 - d2p;
            const float eP = qp_scaled_row(s0 * xp1, y.x, Plo, Phi, rs0);
            const float eV = qp_scaled_row(s1 * d1, y.y, Vlo, Vhi, rs1);
            const float eA = qp_scaled_row(s2 * d2, y.z, t == 0 ? A0lo : Alo, t == 0 ? A0hi : Ahi, rs2);
            float eJ = 0.0f;
            if (t >= 1) eJ = qp_scaled_row(s3 * d3, y.w, t == 1 ? J1lo : Jlo, t == 1 ? J1hi : Jhi, rs3);
            yv[(size_t)sl(t) * T] = y;
            // row t touches x_{t+1} (+1), x_t (-1, -2, -3), x_{t-1} (+1, +3), x_{t-2} (-1)
            const float r3 = bt + eP + eV + eA + eJ;
            r2 = r2 - eV - 2.0f * eA - 3.0f * eJ;
            r1 = r1 + eA + 3.0f * eJ;
            r0 = r0 - eJ;
            if (t >= 3) {  // x_{t-2} is complete: substitute (index i = t-2, slot t-3)
                const float4 L = row(sl(t - 3));
                const float z = (r0 - L.y * z1 - L.z * z2 - L.w * z3) * L.x;
                xs[(size_t)sl(t - 3) * T] = z;
                z3 = z2;
                z2 = z1;
                z1 = z;
            }
            r0 = r1;
            r1 = r2;
            r2 = r3;
            x0 = xp1;
            d2p = d2;
            d1p = d1;
        }
        // the last (up to) three indices: r0, r1, r2 belong to x_{H-2}, x_{H-1}, x_H
        for (int i = H - 2; i <= H; ++i) {
            const float r = i == H - 2 ? r0 : (i == H - 1 ? r1 : r2);
            if (i < 1) continue;
            const float4 L = row(sl(i - 1));
            const float z = (r - L.y * z1 - L.z * z2 - L.w * z3) * L.x;
            xs[(size_t)sl(i - 1) * T] = z;
            z3 = z2;
            z2 = z1;
            z1 = z;
        }
        // backward substitution L^T x = z
        float p1 = 0.0f, p2 = 0.0f, p3 = 0.0f;  // x_{i+1}, x_{i+2}, x_{i+3}
#pragma unroll 4
        for (int i = H; i >= 1; --i) {
            const float4 L = row(H + sl(i - 1));
            float* slot = &xs[(size_t)sl(i - 1) * T];
            const float xi = (*slot - L.y * p1 - L.z * p2 - L.w * p3) * L.x;
            *slot = xi;
            p3 = p2;
            p2 = p1;
            p1 = xi;
        }
    }
}

// Raw sample h of member k (sample) in class j (joint): the value the
// rollout's sampler draws, unclamped.
__device__ __forceinline__ float qp_sample(const QPArgs& a, uint2 key, uint32_t iter, int k, int j, int h) {
    float v = ld_checked(a.u_nom, (long long)h * a.nu + j, (long long)a.H * a.nu);
    if (a.Lfac) {
        const long long r0 = ((long long)h * a.nu + j) * a.nu, n_l = (long long)a.H * a.nu * a.nu;
        for (int jb = 0; 4 * jb <= j; ++jb) {
            const uint4 w = philox4x32_10(make_uint4((uint32_t)jb, (uint32_t)h, (uint32_t)k, iter), key);
            for (int t = 0; t < 4 && 4 * jb + t <= j; ++t)
                v = __fmaf_rn(ld_checked(a.Lfac, r0 + 4 * jb + t, n_l), block_normal(w, t), v);
        }
    } else {
        const uint4 w = philox4x32_10(make_uint4((uint32_t)(j >> 2), (uint32_t)h, (uint32_t)k, iter), key);
        v = __fmaf_rn(ld_checked(a.sigma, j, a.nu), block_normal(w, j & 3), v);
    }
    return v;
}

// ALONE: the standalone form, sequence i of class `own` with the table as a
// parameter: its rows are uniform reads of constant memory, which a chain of
// dependent steps waits for less than for cached global ones (43,973 x 110,
// 20 iterations: 1,259 -> 1,094 us; 1,335 x 106, 30 iterations: 370 -> 313).
// Else sequence i = j K + k is sample k of joint (class) j, drawn here.
template <bool ALONE>
__global__ void __launch_bounds__(64) qp_long_kernel(QPArgs a, const __grid_constant__ QPClass own,
                                                     const __grid_constant__ QPTable table) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int T = blockDim.x, tid = threadIdx.x, H = a.H;
    float4* yv = reinterpret_cast<float4*>(smem) + tid;
    float* xs = reinterpret_cast<float*>(smem + (size_t)H * T * sizeof(float4)) + tid;
    float* bs = xs + (size_t)H * T;  // B^T vt
    const int i = blockIdx.x * T + tid;
    if (i >= a.n) return;
    const int cls = ALONE ? 0 : i / a.per_cls, mem = ALONE ? i : i % a.per_cls;
    const QPClass c = ALONE ? own : a.cls[MPPI_IN_RANGE(cls, a.n_cls) ? cls : 0];
    const long long nq = ALONE ? a.n : a.n_cls;
    const float q = ld_checked(a.q0, ALONE ? i : cls, nq), qd = ld_checked(a.qd0, ALONE ? i : cls, nq);
    auto sl = [H](int h) { return MPPI_IN_RANGE(h, H) ? h : 0; };  // this thread's slots
    auto rhs = [&](int t) { return bs[(size_t)sl(t) * T]; };
    uint2 key{};
    uint32_t iter = 0;
    if (!ALONE) {
        key = make_uint2((uint32_t)a.seed, (uint32_t)(a.seed >> 32));
        iter = (uint32_t)(a.iter_ptr ? *a.iter_ptr : a.iter_val);
    }
    // start point x = prefix sums of vt, and (B^T vt)_i = vt_{i-1} - vt_i (vt_H for i = H)
    float prev = 0.0f, acc = 0.0f;
    for (int h = 0; h < H; ++h) {
        const float vt =
            ALONE ? ld_checked(a.vin, (long long)i * H + h, a.in_n) : qp_sample(a, key, iter, mem, cls, h);
        acc += vt;
        if (h > 0) bs[(size_t)sl(h - 1) * T] = prev - vt;
        xs[(size_t)sl(h) * T] = acc;
        yv[(size_t)sl(h) * T] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        prev = vt;
    }
    bs[(size_t)sl(H - 1) * T] = prev;
    if (ALONE) {
        qp_long_admm(c, [&](int r) { return table.v[r]; }, rhs, H, a.iters, a.dt, q, qd, xs, yv, T);
    } else {
        const float4* band = a.tab + (size_t)(a.n_tab > 1 ? cls : 0) * a.tab_size;
        qp_long_admm(c, [&](int r) { return __ldg(&band[r]); }, rhs, H, a.iters, a.dt, q, qd, xs, yv, T);
    }
    float xp = 0.0f;
    for (int h = 0; h < H; ++h) {
        const float x = xs[(size_t)sl(h) * T];
        const long long o = ALONE ? (long long)i * H + h : ((long long)h * a.per_cls + mem) * a.nu + cls;
        if (MPPI_IN_RANGE(o, a.out_n)) a.out[o] = x - xp;
        xp = x;
    }
}

namespace {

template <int C>
int launch_c(const QPArgs& a, const QPClass* c, const QPTable* table, cudaStream_t s) {
    const int rs = a.H | 1;
    if (table) {
        const int seqs = QP_THREADS / a.L;
        const size_t sm = (size_t)a.tab_size * sizeof(float4) + (size_t)seqs * rs * sizeof(float);
        qp_project_kernel<C><<<(int)(((long long)a.n + seqs - 1) / seqs), QP_THREADS, sm, s>>>(a, *c, *table);
        return cudaGetLastError() == cudaSuccess ? MPPI_OK : MPPI_ERR_CUDA;
    }
    const int S = QP_MAX_L / a.L;
    const size_t normals = (size_t)S * a.H * ((a.nu + 3) / 4), tabs = (size_t)a.n_tab * a.tab_size;
    const size_t sm = ((size_t)(S * a.nu * rs + 3) / 4 + std::max(normals, tabs)) * sizeof(float4);
    if (sm > 48 * 1024) {
        cudaError_t e = open_shared_memory(qp_sample_kernel<C>);
        if (e != cudaSuccess) return MPPI_ERR_CUDA;
    }
    qp_sample_kernel<C><<<(a.per_cls + S - 1) / S, QP_MAX_L * a.nu, sm, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? MPPI_OK : MPPI_ERR_CUDA;
}

// 24 H bytes of shared memory per thread: 64 threads while they stay within
// 100 KB (two CTAs per SM), else one warp.
template <bool ALONE>
int launch_long(const QPArgs& a, const QPClass* c, const QPTable* table, cudaStream_t s) {
    const size_t per = (size_t)a.H * (sizeof(float4) + 2 * sizeof(float));
    const int T = 64 * per <= 100 * 1024 ? 64 : 32;
    const size_t sm = T * per;
    if (sm > 227 * 1024) return MPPI_ERR_UNSUPPORTED;
    static const QPClass no_class{};
    static const QPTable no_table{};
    if (sm > 48 * 1024) {
        cudaError_t e = open_shared_memory(qp_long_kernel<ALONE>);
        if (e != cudaSuccess) return MPPI_ERR_CUDA;
    }
    qp_long_kernel<ALONE>
        <<<(int)(((long long)a.n + T - 1) / T), T, sm, s>>>(a, c ? *c : no_class, table ? *table : no_table);
    return cudaGetLastError() == cudaSuccess ? MPPI_OK : MPPI_ERR_CUDA;
}

int launch_any(const QPArgs& a, const QPClass* c, const QPTable* table, cudaStream_t s) {
    if (a.L == 0) return table ? launch_long<true>(a, c, table, s) : launch_long<false>(a, c, table, s);
    switch ((a.H + a.L - 1) / a.L) {
        case 1: return launch_c<1>(a, c, table, s);
        case 2: return launch_c<2>(a, c, table, s);
        case 3: return launch_c<3>(a, c, table, s);
        case 4: return launch_c<4>(a, c, table, s);
        case 5: return launch_c<5>(a, c, table, s);
        case 6: return launch_c<6>(a, c, table, s);
        case 7: return launch_c<7>(a, c, table, s);
        case 8: return launch_c<8>(a, c, table, s);
        case 9: return launch_c<9>(a, c, table, s);
        case 10: return launch_c<10>(a, c, table, s);
        case 11: return launch_c<11>(a, c, table, s);
        case 12: return launch_c<12>(a, c, table, s);
        case 13: return launch_c<13>(a, c, table, s);
        case 14: return launch_c<14>(a, c, table, s);
        case 15: return launch_c<15>(a, c, table, s);
        case 16: return launch_c<16>(a, c, table, s);
        default: return MPPI_ERR_UNSUPPORTED;
    }
}

}  // namespace

int launch_qp(const QPArgs& a, cudaStream_t s) {
    if (a.n <= 0) return MPPI_OK;
    if (a.nu > 14 || a.n != a.per_cls * a.nu) return MPPI_ERR_UNSUPPORTED;
    return launch_any(a, nullptr, nullptr, s);
}

MPPI_BOUNDS_READER(bounds_word_qp)

}  // namespace mppi

using namespace mppi;

extern "C" int mppi_qp_project(int n, int H, float dt, const float* bounds, int iters, float rho, const float* scales,
                               const float* q0, const float* qd0, const float* v_in, float* v_out, void* stream) {
    static const float kDefault[4] = {MPPI_QP_SCALE_POSITION, MPPI_QP_SCALE_VELOCITY, MPPI_QP_SCALE_ACCELERATION,
                                      MPPI_QP_SCALE_JERK};
    const float* sc = scales ? scales : kDefault;
    if (n < 0 || H < 1 || H > MPPI_QP_MAX_H || iters < 0 || !(dt > 0.0f) || !bounds) return MPPI_ERR_INVALID_ARG;
    if (n > 0 && (!q0 || !qd0 || !v_in || !v_out)) return MPPI_ERR_INVALID_ARG;
    int rc = qp_validate(bounds, sc, rho);
    if (rc != MPPI_OK) return rc;
    if (n == 0) return MPPI_OK;
    // class record and table travel as kernel parameters: no allocation, no copy
    QPClass c;
    qp_make_class(bounds, sc, rho, &c);
    QPArgs a{};
    a.n = n;
    a.H = H;
    a.iters = iters;
    a.dt = dt;
    a.L = qp_lanes(n, H, false);
    a.tab_size = qp_table_size(H, a.L);
    a.n_tab = 1;
    QPTable table;
    const double scd[4] = {c.s[0], c.s[1], c.s[2], c.s[3]};
    rc = qp_table(H, a.L, rho, scd, table.v);
    if (rc != MPPI_OK) return rc;
    a.q0 = q0;
    a.qd0 = qd0;
    a.vin = v_in;
    a.out = v_out;
    a.in_n = a.out_n = (long long)n * H;
    return launch_any(a, &c, &table, (cudaStream_t)stream);
}
