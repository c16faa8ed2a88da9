// a5, a8: FP64 deformation-gradient fits (Section 2, Eq. 2-5 and Eq. 12).
//
// Eq. 2 maps a reference point r (lifted to (x - xpc, y - ypc, Z*)) to the
// test point Z* F r / ((F r).k).  Eq. 3 fits F to N point pairs by least
// squares.  The objective is invariant under F -> lambda F, so the fit runs
// in the gauge F_33 = 1: a linear start from the cross-multiplied equations
// Z* (F r)_a - r'_a (F r)_3 = 0 (8 unknowns, normal equations), then
// Gauss-Newton on the projected residuals; last, det F = 1.  The rotation is
// the polar factor R = P Q^T of F = P D Q^T (Eq. 4-5), computed with the
// Newton iteration X <- (X + X^-T)/2, which converges to the same orthogonal
// factor as the SVD.
//
// FP64 runs at 2 FMAs per clock and SM here, and a dependent FP64 instruction
// takes tens of cycles, so both the operation count and the length of the
// serial chain matter.  A group of lanes owns one pair: the lanes share the
// ROIs, the normal equations use the block structure of the Jacobian (27 sums
// instead of 72) and are solved through a 2x2 Schur complement.  Launch times
// against one thread per pair, first pass / second pass: 2,500 pairs of 25
// ROIs 142 / 150 us (was 1,557 / 1,317), one pair of 25 ROIs 87 / 85 us (was
// 1,381 / 1,311), 16 pairs of 100 ROIs 85 / 111 us (was 3,089 / 3,956).
#include <math.h>

#include "internal.cuh"

namespace {

constexpr int kMaxRoi = 512;

// Solve the n x n system A x = b (row-major, destroyed) by Gaussian
// elimination with partial pivoting.  Returns false if singular.
__device__ bool gauss_solve(double *A, double *b, int n, double *x)
{
    for (int c = 0; c < n; ++c) {
        int piv = c;
        double best = fabs(A[c * n + c]);
        for (int r = c + 1; r < n; ++r)
            if (fabs(A[r * n + c]) > best) { best = fabs(A[r * n + c]); piv = r; }
        if (!(best > 1e-300)) return false;
        if (piv != c) {
            for (int k = 0; k < n; ++k) { double t = A[c * n + k]; A[c * n + k] = A[piv * n + k]; A[piv * n + k] = t; }
            double t = b[c]; b[c] = b[piv]; b[piv] = t;
        }
        for (int r = c + 1; r < n; ++r) {
            double f = A[r * n + c] / A[c * n + c];
            if (f == 0.0) continue;
            for (int k = c; k < n; ++k) A[r * n + k] -= f * A[c * n + k];
            b[r] -= f * b[c];
        }
    }
    for (int r = n - 1; r >= 0; --r) {
        double s = b[r];
        for (int k = r + 1; k < n; ++k) s -= A[r * n + k] * x[k];
        x[r] = s / A[r * n + r];
    }
    return true;
}

__device__ double det3(const double *F)
{
    return F[0] * (F[4] * F[8] - F[5] * F[7]) - F[1] * (F[3] * F[8] - F[5] * F[6]) + F[2] * (F[3] * F[7] - F[4] * F[6]);
}

// The point pairs of one fit, relative to the pattern centre: the ROI centres
// (the same for every pair) and the measured points.  FIELD (first pass): the
// reference points are measured, r_i = c_i - u(c_i), r'_i = c_i; otherwise
// (second pass) the test points are, r_i = c_i, r'_i = c_i + q_i.
template <bool FIELD>
struct Points {
    const double2 *centre, *measured;
    __device__ void operator()(int i, double *pt) const
    {
        const double2 r = FIELD ? measured[i] : centre[i], t = FIELD ? centre[i] : measured[i];
        pt[0] = r.x;
        pt[1] = r.y;
        pt[2] = t.x;
        pt[3] = t.y;
    }
};

// Fit F (det 1) to N point pairs by one thread: pts(i, p) fills p = {rx, ry,
// tx, ty}.  The general form (full 8x8 systems, partial pivoting) for the
// nearly singular systems that fit_group leaves.  Returns false on a singular
// system.
template <class Pts>
__device__ __noinline__ bool fit_F(Pts pts, int N, double zs, double *F)
{
    double A[64], b[8], x[8];
    // linear start, F_33 = 1: Z* (F r)_a - t_a (F r)_3 = 0
    for (int i = 0; i < 64; ++i) A[i] = 0.0;
    for (int i = 0; i < 8; ++i) b[i] = 0.0;
    for (int i = 0; i < N; ++i) {
        double pt[4];
        pts(i, pt);
        const double r[3] = {pt[0], pt[1], zs};
        const double t[2] = {pt[2], pt[3]};
        for (int a = 0; a < 2; ++a) {
            double row[8];
            for (int k = 0; k < 8; ++k) row[k] = 0.0;
            for (int c = 0; c < 3; ++c) row[a * 3 + c] = zs * r[c];
            row[6] = -t[a] * r[0];
            row[7] = -t[a] * r[1];
            const double rhs = t[a] * zs;   // moves -t_a F_33 r_3 = -t_a Z* to the right
            for (int p = 0; p < 8; ++p) {
                b[p] += row[p] * rhs;
                for (int q = 0; q < 8; ++q) A[p * 8 + q] += row[p] * row[q];
            }
        }
    }
    if (!gauss_solve(A, b, 8, x)) return false;
    for (int k = 0; k < 8; ++k) F[k] = x[k];
    F[8] = 1.0;
    // Gauss-Newton on the Eq. 3 residuals Z* (F r)_a / (F r)_3 - t_a
    for (int it = 0; it < 60; ++it) {
        for (int i = 0; i < 64; ++i) A[i] = 0.0;
        for (int i = 0; i < 8; ++i) b[i] = 0.0;
        for (int i = 0; i < N; ++i) {
            double pt[4];
            pts(i, pt);
            const double r[3] = {pt[0], pt[1], zs};
            double v[3];
            for (int a = 0; a < 3; ++a) v[a] = F[a * 3] * r[0] + F[a * 3 + 1] * r[1] + F[a * 3 + 2] * r[2];
            const double iv = 1.0 / v[2];
            const double t[2] = {pt[2], pt[3]};
            for (int a = 0; a < 2; ++a) {
                const double res = zs * v[a] * iv - t[a];
                double J[8];
                for (int k = 0; k < 8; ++k) J[k] = 0.0;
                for (int c = 0; c < 3; ++c) J[a * 3 + c] = zs * r[c] * iv;
                J[6] = -zs * v[a] * r[0] * iv * iv;
                J[7] = -zs * v[a] * r[1] * iv * iv;
                for (int p = 0; p < 8; ++p) {
                    b[p] -= J[p] * res;
                    for (int q = 0; q < 8; ++q) A[p * 8 + q] += J[p] * J[q];
                }
            }
        }
        if (!gauss_solve(A, b, 8, x)) return false;
        double sn = 0.0, fn = 0.0;
        for (int k = 0; k < 8; ++k) {
            F[k] += x[k];
            sn += x[k] * x[k];
            fn += F[k] * F[k];
        }
        if (sqrt(sn) <= 1e-15 * sqrt(fn + 1.0)) break;
    }
    const double d = det3(F);
    if (!(d > 0.0)) return false;
    const double sc = cbrt(d);
    for (int k = 0; k < 9; ++k) F[k] /= sc;
    return true;
}

// ---------------------------------------------------------------- lane groups
// Sums over a pair's point pairs, in the order of the normal equations' blocks.
// With r = (r0, r1, Z*), g = Z*/v3, h_a = Z* v_a / v3^2 and the residuals e_a the
// Jacobian rows are J_a = (g r at F's row a, -h_a r0, -h_a r1), so that the matrix
// is [[P, 0, C_0], [0, P, C_1], [C_0^T, C_1^T, D]] with one P for both rows:
constexpr int S_P = 0;      // 6: sum g^2 (r0 r0, r0 r1, r1 r1, r0 Z*, r1 Z*, Z* Z*)
constexpr int S_C = 6;      // 2 x 5: sum g h_a (r0 r0, r0 r1, r1 r1, r0 Z*, r1 Z*)   (C_a negated)
constexpr int S_D = 16;     // 3: sum (h_0^2 + h_1^2) (r0 r0, r0 r1, r1 r1)
constexpr int S_B = 19;     // 2 x 3: sum -g e_a (r0, r1, Z*)
constexpr int S_E = 25;     // 2: sum (h_0 e_0 + h_1 e_1) (r0, r1)
constexpr int S_N = 27, S_PAD = 32;

__device__ __forceinline__ void add_point(double *s, double r0, double r1, double zs, double g, double h0, double h1,
                                          double e0, double e1)
{
    const double r00 = r0 * r0, r01 = r0 * r1, r11 = r1 * r1, r0z = r0 * zs, r1z = r1 * zs;
    const double gg = g * g, gh0 = g * h0, gh1 = g * h1, hh = fma(h0, h0, h1 * h1);
    const double ge0 = -g * e0, ge1 = -g * e1, he = fma(h0, e0, h1 * e1);
    s[S_P] = fma(gg, r00, s[S_P]);
    s[S_P + 1] = fma(gg, r01, s[S_P + 1]);
    s[S_P + 2] = fma(gg, r11, s[S_P + 2]);
    s[S_P + 3] = fma(gg, r0z, s[S_P + 3]);
    s[S_P + 4] = fma(gg, r1z, s[S_P + 4]);
    s[S_P + 5] = fma(gg, zs * zs, s[S_P + 5]);
    s[S_C] = fma(gh0, r00, s[S_C]);
    s[S_C + 1] = fma(gh0, r01, s[S_C + 1]);
    s[S_C + 2] = fma(gh0, r11, s[S_C + 2]);
    s[S_C + 3] = fma(gh0, r0z, s[S_C + 3]);
    s[S_C + 4] = fma(gh0, r1z, s[S_C + 4]);
    s[S_C + 5] = fma(gh1, r00, s[S_C + 5]);
    s[S_C + 6] = fma(gh1, r01, s[S_C + 6]);
    s[S_C + 7] = fma(gh1, r11, s[S_C + 7]);
    s[S_C + 8] = fma(gh1, r0z, s[S_C + 8]);
    s[S_C + 9] = fma(gh1, r1z, s[S_C + 9]);
    s[S_D] = fma(hh, r00, s[S_D]);
    s[S_D + 1] = fma(hh, r01, s[S_D + 1]);
    s[S_D + 2] = fma(hh, r11, s[S_D + 2]);
    s[S_B] = fma(ge0, r0, s[S_B]);
    s[S_B + 1] = fma(ge0, r1, s[S_B + 1]);
    s[S_B + 2] = fma(ge0, zs, s[S_B + 2]);
    s[S_B + 3] = fma(ge1, r0, s[S_B + 3]);
    s[S_B + 4] = fma(ge1, r1, s[S_B + 4]);
    s[S_B + 5] = fma(ge1, zs, s[S_B + 5]);
    s[S_E] = fma(he, r0, s[S_E]);
    s[S_E + 1] = fma(he, r1, s[S_E + 1]);
}

// Sum s over the G lanes of a group (every lane of the warp calls it): each
// exchange halves the values a lane still carries, so a lane adds 31 (G = 32)
// or 24 (G = 4) values instead of 27 per exchange; the sums meet in `ex`
// (shared memory of the group) and every lane reads all of them.
template <int G>
__device__ __forceinline__ void group_sum(double *s, double *ex, int sub)
{
    int n = S_PAD, base = 0;
#pragma unroll
    for (int off = G / 2; off > 0; off /= 2) {
        n /= 2;
        const bool up = (sub & off) != 0;
#pragma unroll
        for (int j = 0; j < S_PAD / 2; ++j)
            if (j < n) {
                const double give = up ? s[j] : s[j + n], keep = up ? s[j + n] : s[j];
                s[j] = keep + __shfl_xor_sync(0xffffffffu, give, off);
            }
        base += up ? n : 0;
    }
    constexpr int PER = S_PAD / G;
#pragma unroll
    for (int j = 0; j < PER; ++j) ex[base + j] = s[j];
    __syncwarp();
#pragma unroll
    for (int j = 0; j < S_N; ++j) s[j] = ex[j];
    __syncwarp();
}

// The step x (8 unknowns, F's rows 0 and 1, then F_31 and F_32) of the summed
// system.  False where a pivot lost more than 10 digits against its diagonal.
__device__ __forceinline__ bool solve_sums(const double *s, double *x)
{
    constexpr double TINY = 1e-10;
    const double p00 = s[S_P], p01 = s[S_P + 1], p11 = s[S_P + 2], p0z = s[S_P + 3], p1z = s[S_P + 4], pzz = s[S_P + 5];
    // P = L diag(d) L^T
    const double i0 = 1.0 / p00, l1 = p01 * i0, l2 = p0z * i0;
    const double d1 = fma(-l1, p01, p11), i1 = 1.0 / d1;
    const double m21 = fma(-l2, p01, p1z), l21 = m21 * i1;
    const double d2 = fma(-l21, m21, fma(-l2, p0z, pzz)), i2 = 1.0 / d2;
    auto solve3 = [&](double c0, double c1, double c2, double *y) {
        const double y1 = fma(-l1, c0, c1), y2 = fma(-l21, y1, fma(-l2, c0, c2));
        y[2] = y2 * i2;
        y[1] = fma(-l21, y[2], y1 * i1);
        y[0] = fma(-l1, y[1], fma(-l2, y[2], c0 * i0));
    };
    double S0 = s[S_D], S1 = s[S_D + 1], S2 = s[S_D + 2], e0 = s[S_E], e1 = s[S_E + 1];
    double ya[2][3], yb[2][3], yc[2][3];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        const double *c = s + S_C + 5 * a, *b = s + S_B + 3 * a;   // C_a = -c
        solve3(c[0], c[1], c[3], ya[a]);   // P^-1 (-C_a's column of F_31)
        solve3(c[1], c[2], c[4], yb[a]);   // ... of F_32
        solve3(b[0], b[1], b[2], yc[a]);
        S0 = fma(-c[3], ya[a][2], fma(-c[1], ya[a][1], fma(-c[0], ya[a][0], S0)));
        S1 = fma(-c[3], yb[a][2], fma(-c[1], yb[a][1], fma(-c[0], yb[a][0], S1)));
        S2 = fma(-c[4], yb[a][2], fma(-c[2], yb[a][1], fma(-c[1], yb[a][0], S2)));
        // right-hand side e - C_a^T y = e + c^T y
        e0 = fma(c[3], yc[a][2], fma(c[1], yc[a][1], fma(c[0], yc[a][0], e0)));
        e1 = fma(c[4], yc[a][2], fma(c[2], yc[a][1], fma(c[1], yc[a][0], e1)));
    }
    const double q0 = 1.0 / S0, q = S1 * q0, d3 = fma(-q, S1, S2);
    x[7] = fma(-q, e0, e1) / d3;
    x[6] = fma(-q, x[7], e0 * q0);
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int c = 0; c < 3; ++c) x[3 * a + c] = fma(yb[a][c], x[7], fma(ya[a][c], x[6], yc[a][c]));
    return p00 > 0.0 && d1 > TINY * p11 && d2 > TINY * pzz && S0 > TINY * s[S_D] && d3 > TINY * s[S_D + 2];
}

// Fit F (det 1) by the G lanes of a group; every lane of the warp takes part
// (groups with `live` false only in the exchanges).  Returns false where the
// system is nearly singular or the iteration does not settle (the caller then
// takes fit_F).  The last step's size times the contraction of the steps bounds
// what a further one would change; 1e-15 relative ends the iteration.
template <int G, bool FIELD>
__device__ bool fit_group(const Points<FIELD> &pts, int N, double zs, double *ex, int sub, bool live, double *F)
{
    double s[S_PAD], x[8];
    bool ok = live, done = !live;
#pragma unroll
    for (int k = 0; k < S_PAD; ++k) s[k] = 0.0;
    if (live)
        for (int i = sub; i < N; i += G) {   // linear start: the rows Z* (F r)_a - t_a (F r)_3 = 0 with F_33 = 1
            double pt[4];
            pts(i, pt);
            add_point(s, pt[0], pt[1], zs, zs, pt[2], pt[3], -pt[2] * zs, -pt[3] * zs);
        }
    group_sum<G>(s, ex, sub);
    ok = ok && solve_sums(s, x);
#pragma unroll
    for (int k = 0; k < 8; ++k) F[k] = x[k];
    F[8] = 1.0;
    done = done || !ok;
    double last = 0.0;
    for (int it = 0; it < 60; ++it) {
        if (__all_sync(0xffffffffu, done)) break;
#pragma unroll
        for (int k = 0; k < S_PAD; ++k) s[k] = 0.0;
        if (!done)
            for (int i = sub; i < N; i += G) {
                double pt[4];
                pts(i, pt);
                const double v0 = fma(F[0], pt[0], fma(F[1], pt[1], F[2] * zs));
                const double v1 = fma(F[3], pt[0], fma(F[4], pt[1], F[5] * zs));
                const double v2 = fma(F[6], pt[0], fma(F[7], pt[1], zs));
                const double iv = 1.0 / v2, g = zs * iv, w0 = g * v0, w1 = g * v1;
                add_point(s, pt[0], pt[1], zs, g, w0 * iv, w1 * iv, w0 - pt[2], w1 - pt[3]);
            }
        group_sum<G>(s, ex, sub);
        if (done) continue;
        ok = solve_sums(s, x);
        double sn = 0.0, fn = 1.0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            F[k] += x[k];
            sn = fma(x[k], x[k], sn);
            fn = fma(F[k], F[k], fn);
        }
        const double step = sqrt(sn), rate = it > 0 && step < 0.1 * last ? 2.0 * step / last : 1.0;
        last = step;
        done = !ok || step * rate <= 1e-15 * sqrt(fn);
    }
    ok = ok && done;
    const double d = det3(F);
    if (!(ok && d > 0.0)) return false;
    const double sc = 1.0 / cbrt(d);
#pragma unroll
    for (int k = 0; k < 9; ++k) F[k] *= sc;
    return true;
}

// Polar factor by Newton's iteration X <- (X + X^-T)/2 (Higham), FP64.  It
// converges quadratically: a relative step of 1e-10 leaves an error of 1e-20.
__device__ void polar_newton(const double *F, double *R)
{
    double X[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) X[k] = F[k];
    for (int it = 0; it < 100; ++it) {
        // X^-T = cof(X) / det(X)
        double C[9];
        C[0] = X[4] * X[8] - X[5] * X[7];
        C[1] = X[5] * X[6] - X[3] * X[8];
        C[2] = X[3] * X[7] - X[4] * X[6];
        C[3] = X[2] * X[7] - X[1] * X[8];
        C[4] = X[0] * X[8] - X[2] * X[6];
        C[5] = X[1] * X[6] - X[0] * X[7];
        C[6] = X[1] * X[5] - X[2] * X[4];
        C[7] = X[2] * X[3] - X[0] * X[5];
        C[8] = X[0] * X[4] - X[1] * X[3];
        const double hd = 0.5 / (X[0] * C[0] + X[1] * C[1] + X[2] * C[2]);
        double diff = 0.0, nrm = 0.0;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const double nx = fma(C[k], hd, 0.5 * X[k]);
            diff += (nx - X[k]) * (nx - X[k]);
            nrm += nx * nx;
            X[k] = nx;
        }
        if (diff <= 1e-20 * nrm) break;
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) R[k] = X[k];
}

__device__ float bilinear_clamped(const float *M, int h, int w, float x, float y)
{
    x = fminf(fmaxf(x, 0.0f), (float)(w - 1));
    y = fminf(fmaxf(y, 0.0f), (float)(h - 1));
    int x0 = min((int)floorf(x), w - 2);
    int y0 = min((int)floorf(y), h - 2);
    float fx = x - (float)x0, fy = y - (float)y0;
    const float *p = M + (size_t)y0 * w + x0;
    float top = fmaf(fx, p[1], (1.0f - fx) * p[0]);
    float bot = fmaf(fx, p[w + 1], (1.0f - fx) * p[w]);
    return fmaf(fy, bot, (1.0f - fy) * top);
}

__device__ void set_identity(double *M)
{
    for (int k = 0; k < 9; ++k) M[k] = (k % 4 == 0) ? 1.0 : 0.0;
}

constexpr int kFitThreads = 64;

// Shared memory of a CTA of the fit kernels: the ROI centres, every group's measured points and sums.
constexpr size_t fit_smem(int G, int N)
{
    return (size_t)N * 16 + (size_t)(kFitThreads / G) * ((size_t)N * 16 + S_PAD * 8);
}

// The Eq. 3 fit of G lanes per pair, kFitThreads / G pairs per CTA.  `measure(i, cx, cy)` gives the
// measured point of ROI i (relative to the pattern centre); `write(b, F, ok)` stores the result and
// runs on the group's first lane.
template <int G, bool FIELD, class Measure, class Write>
__device__ __forceinline__ void fit_pairs(int B, const int32_t *roi, int N, double xpc, double ypc, double zs,
                                          int32_t *status, Measure measure, Write write)
{
    extern __shared__ __align__(16) unsigned char fit_raw[];
    double2 *centre = reinterpret_cast<double2 *>(fit_raw);
    const int grp = threadIdx.x / G, sub = threadIdx.x % G;
    double2 *meas = centre + N + (size_t)grp * N;
    double *ex = reinterpret_cast<double *>(centre + N + (size_t)(kFitThreads / G) * N) + grp * S_PAD;
    const int b = blockIdx.x * (kFitThreads / G) + grp;
    const bool in = b < B;
    for (int i = threadIdx.x; i < N; i += kFitThreads)
        centre[i] = make_double2((double)roi[2 * i] - xpc, (double)roi[2 * i + 1] - ypc);
    bool finite = true;
    if (in)
        for (int i = sub; i < N; i += G) {
            const double2 m = measure(b, i, (double)roi[2 * i], (double)roi[2 * i + 1]);
            meas[i] = m;
            finite = finite && isfinite(m.x) && isfinite(m.y);
        }
    __syncthreads();
    const unsigned mine = (G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u) << ((threadIdx.x & 31) / G * G));
    finite = (__ballot_sync(0xffffffffu, finite) & mine) == mine;
    const Points<FIELD> pts{centre, meas};
    double F[9];
    bool ok = fit_group<G, FIELD>(pts, N, zs, ex, sub, in && finite, F);
    if (!in || sub != 0) return;
    if (!ok && finite) ok = fit_F(pts, N, zs, F);
    if (!ok && status)
        atomicOr(status + b, finite ? HREBSD_PAIR_FIT_FAILED : (HREBSD_PAIR_FIT_FAILED | HREBSD_PAIR_NONFINITE));
    write(b, F, ok);
}

// First pass: the field at the ROI centres (index coordinates c - 0.5).
template <int G>
__global__ void __launch_bounds__(kFitThreads) fit_rotation_kernel(const float *__restrict__ field, int B, int H, int W,
                                                                   const int32_t *__restrict__ roi, int N, double xpc,
                                                                   double ypc, double zs, double *F_first,
                                                                   double *R_finite, int32_t *status)
{
    fit_pairs<G, true>(B, roi, N, xpc, ypc, zs, status,
        [&](int b, int i, double cx, double cy) {
            const float *fx = field + (size_t)b * 2 * H * W, *fy = fx + (size_t)H * W;
            const float ux = bilinear_clamped(fx, H, W, (float)(cx - 0.5), (float)(cy - 0.5));
            const float uy = bilinear_clamped(fy, H, W, (float)(cx - 0.5), (float)(cy - 0.5));
            return make_double2(cx - (double)ux - xpc, cy - (double)uy - ypc);
        },
        [&](int b, double *F, bool ok) {
            double R[9];
            if (ok) {
                polar_newton(F, R);
            } else {
                set_identity(F);
                set_identity(R);
            }
            for (int k = 0; k < 9; ++k) {
                F_first[(size_t)b * 9 + k] = F[k];
                R_finite[(size_t)b * 9 + k] = R[k];
            }
        });
}

// Second pass: the ROI shifts, then F = F_inf R_finite (Eq. 12).
template <int G>
__global__ void __launch_bounds__(kFitThreads) solve_F_kernel(const float *__restrict__ q,
                                                              const int32_t *__restrict__ roi, int N, int B,
                                                              double xpc, double ypc, double zs,
                                                              const double *R_finite, double *Fout, int32_t *status)
{
    fit_pairs<G, false>(B, roi, N, xpc, ypc, zs, status,
        [&](int b, int i, double cx, double cy) {
            const float qx = q[((size_t)b * N + i) * 2], qy = q[((size_t)b * N + i) * 2 + 1];
            return make_double2(cx + (double)qx - xpc, cy + (double)qy - ypc);
        },
        [&](int b, double *Fi, bool ok) {
            if (!ok) set_identity(Fi);
            double F[9];
            if (R_finite) {
                const double *Rf = R_finite + (size_t)b * 9;
                for (int i = 0; i < 3; ++i)
                    for (int j = 0; j < 3; ++j)
                        F[i * 3 + j] = Fi[i * 3] * Rf[j] + Fi[i * 3 + 1] * Rf[3 + j] + Fi[i * 3 + 2] * Rf[6 + j];
            } else {
                for (int k = 0; k < 9; ++k) F[k] = Fi[k];
            }
            for (int k = 0; k < 9; ++k) Fout[(size_t)b * 9 + k] = F[k];
        });
}

// Lanes per pair.  A whole warp where there are too few pairs to fill the SMs otherwise (the chain of
// one fit is then the time) or where the ROIs of 16 pairs would not fit the static shared-memory
// limit; else 4 lanes, which share the exchanges and the 8x8 solve among 8 pairs of a warp.
bool fit_whole_warp(const hrebsd_ctx *ctx, int B, int N) { return B <= 2 * ctx->num_sms || N > 64; }

// Rotation part of arbitrary F (Eq. 4-5), one thread per pair.
__global__ void polar_kernel(const double *__restrict__ F, int B, double *R)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    double Fb[9], Rb[9];
    for (int k = 0; k < 9; ++k) Fb[k] = F[(size_t)b * 9 + k];
    polar_newton(Fb, Rb);
    for (int k = 0; k < 9; ++k) R[(size_t)b * 9 + k] = Rb[k];
}

// Quality of an Eq. 3 fit (Section 3.1, Fig. 3).  Point pairs: from the XCF
// shifts (r = c, r' = c + q) or from the demons field (r = c - u(c), r' = c).
// Model F_m = F R^T when R is given (the second pass, Eq. 12), else F.
// MAE = mean over ROIs of the angle between the measured test direction
// (r' - PC, Z*) and F_m (r - PC, Z*); PH = mean of the peak heights.
__global__ void fit_quality_kernel(const double *__restrict__ F, const double *__restrict__ R,
                                   const float *__restrict__ q, const float *__restrict__ field,
                                   const float *__restrict__ ph, int B, int H, int W, const int32_t *__restrict__ roi,
                                   int N, double xpc, double ypc, double zs, double *mae, double *ph_mean)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    double Fm[9];
    const double *Fb = F + (size_t)b * 9;
    if (R) {
        const double *Rb = R + (size_t)b * 9;
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j)
                Fm[i * 3 + j] = Fb[i * 3] * Rb[j * 3] + Fb[i * 3 + 1] * Rb[j * 3 + 1] + Fb[i * 3 + 2] * Rb[j * 3 + 2];
    } else {
        for (int k = 0; k < 9; ++k) Fm[k] = Fb[k];
    }
    const float *fx = field ? field + (size_t)b * 2 * H * W : nullptr;
    double sum = 0.0, phs = 0.0;
    for (int i = 0; i < N; ++i) {
        const double cx = roi[2 * i], cy = roi[2 * i + 1];
        double r[2], rp[2];
        if (q) {
            r[0] = cx;
            r[1] = cy;
            rp[0] = cx + (double)q[((size_t)b * N + i) * 2];
            rp[1] = cy + (double)q[((size_t)b * N + i) * 2 + 1];
        } else {
            const float ux = bilinear_clamped(fx, H, W, (float)(cx - 0.5), (float)(cy - 0.5));
            const float uy = bilinear_clamped(fx + (size_t)H * W, H, W, (float)(cx - 0.5), (float)(cy - 0.5));
            r[0] = cx - (double)ux;
            r[1] = cy - (double)uy;
            rp[0] = cx;
            rp[1] = cy;
        }
        const double v[3] = {r[0] - xpc, r[1] - ypc, zs};
        double p[3];
        for (int a = 0; a < 3; ++a) p[a] = Fm[a * 3] * v[0] + Fm[a * 3 + 1] * v[1] + Fm[a * 3 + 2] * v[2];
        const double m[3] = {rp[0] - xpc, rp[1] - ypc, zs};
        const double cr[3] = {p[1] * m[2] - p[2] * m[1], p[2] * m[0] - p[0] * m[2], p[0] * m[1] - p[1] * m[0]};
        sum += atan2(sqrt(cr[0] * cr[0] + cr[1] * cr[1] + cr[2] * cr[2]), p[0] * m[0] + p[1] * m[1] + p[2] * m[2]);
        if (ph) phs += (double)ph[(size_t)b * N + i];
    }
    mae[b] = sum / N;
    if (ph_mean) ph_mean[b] = ph ? phs / N : 0.0;
}

}  // namespace

extern "C" int hrebsd_fit_rotation(hrebsd_ctx *ctx, const float *field, int B, int H, int W, const int32_t *roi_xy,
                                   int N, const hrebsd_geometry *g, double *F_first, double *R_finite,
                                   int32_t *pair_status, void *stream)
{
    if (!ctx || !g || B < 0 || H < 2 || W < 2 || N < 4 || N > kMaxRoi) return HREBSD_EINVAL;
    if (B == 0) return HREBSD_OK;
    if (!field || !roi_xy || !F_first || !R_finite) return HREBSD_EINVAL;
    int e = hr_set_device(ctx);
    if (e) return e;
    hr_prof_begin(ctx, hr_stream(stream));
    const bool whole = fit_whole_warp(ctx, B, N);
    const int G = whole ? 32 : 4, per = kFitThreads / G;
    (whole ? fit_rotation_kernel<32> : fit_rotation_kernel<4>)<<<(B + per - 1) / per, kFitThreads, fit_smem(G, N),
                                                                 hr_stream(stream)>>>(
        field, B, H, W, roi_xy, N, g->xstar * W, g->ystar * H, g->zstar * W, F_first, R_finite, pair_status);
    hr_prof_end(ctx, PROF_FIT, hr_stream(stream));
    HR_LAUNCHED(ctx);
    return HREBSD_OK;
}

extern "C" int hrebsd_solve_F(hrebsd_ctx *ctx, const float *q, const int32_t *roi_xy, int N, int B, int H, int W,
                              const hrebsd_geometry *g, const double *R_finite, int normalization,
                              const hrebsd_elastic *elastic, double *F, int32_t *pair_status, void *stream)
{
    if (!ctx || !g || B < 0 || H < 2 || W < 2 || N < 4 || N > kMaxRoi) return HREBSD_EINVAL;
    if (normalization != HREBSD_NORM_DET1 && normalization != HREBSD_NORM_TRACTION_FREE) return HREBSD_EINVAL;
    if (normalization == HREBSD_NORM_TRACTION_FREE && (!elastic || !elastic->g || elastic->R < 1))
        return HREBSD_EINVAL;
    if (B == 0) return HREBSD_OK;
    if (!q || !roi_xy || !F) return HREBSD_EINVAL;
    int e = hr_set_device(ctx);
    if (e) return e;
    cudaStream_t st = hr_stream(stream);
    hr_prof_begin(ctx, st);
    const bool whole = fit_whole_warp(ctx, B, N);
    const int G = whole ? 32 : 4, per = kFitThreads / G;
    (whole ? solve_F_kernel<32> : solve_F_kernel<4>)<<<(B + per - 1) / per, kFitThreads, fit_smem(G, N), st>>>(
        q, roi_xy, N, B, g->xstar * W, g->ystar * H, g->zstar * W, R_finite, F, pair_status);
    hr_prof_end(ctx, PROF_SOLVE, st);
    HR_LAUNCHED(ctx);
    if (normalization == HREBSD_NORM_TRACTION_FREE) return hr_launch_traction_scale(ctx, F, elastic, B, pair_status, st);
    return HREBSD_OK;
}

extern "C" int hrebsd_polar_batch(hrebsd_ctx *ctx, const double *F, int B, double *R, void *stream)
{
    if (!ctx || B < 0) return HREBSD_EINVAL;
    if (B == 0) return HREBSD_OK;
    if (!F || !R) return HREBSD_EINVAL;
    int e = hr_set_device(ctx);
    if (e) return e;
    hr_prof_begin(ctx, hr_stream(stream));
    polar_kernel<<<(B + 63) / 64, 64, 0, hr_stream(stream)>>>(F, B, R);
    hr_prof_end(ctx, PROF_FIT, hr_stream(stream));
    HR_LAUNCHED(ctx);
    return HREBSD_OK;
}

extern "C" int hrebsd_fit_quality(hrebsd_ctx *ctx, const double *F, const double *R, const float *q, const float *field,
                                  const float *ph, int B, int H, int W, const int32_t *roi_xy, int N,
                                  const hrebsd_geometry *g, double *mae, double *ph_mean, void *stream)
{
    if (!ctx || !g || B < 0 || H < 2 || W < 2 || N < 1 || N > kMaxRoi) return HREBSD_EINVAL;
    if (B == 0) return HREBSD_OK;
    if (!F || !roi_xy || !mae || (!q) == (!field)) return HREBSD_EINVAL;
    int e = hr_set_device(ctx);
    if (e) return e;
    hr_prof_begin(ctx, hr_stream(stream));
    fit_quality_kernel<<<(B + 63) / 64, 64, 0, hr_stream(stream)>>>(F, R, q, field, ph, B, H, W, roi_xy, N,
                                                                    g->xstar * W, g->ystar * H, g->zstar * W, mae,
                                                                    ph_mean);
    hr_prof_end(ctx, PROF_SOLVE, hr_stream(stream));
    HR_LAUNCHED(ctx);
    return HREBSD_OK;
}
