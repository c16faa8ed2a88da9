// a1: static background correction + normalisation, and the 2x2 pyramid.
//
// Section 2 normalises every pattern to zero mean before correlation and
// Section 3.3 corrects the background before registration.  One CTA (a cluster
// of them where there are few patterns) owns one
// pattern: it reads it for the background moments, divides it by the fitted
// quadric once (float-float) writing the quotient less a constant to the
// output, then reads that back for the variance and the normalised output.
// The pattern stays in L2 between the passes as far as the patterns in work fit
// together; what is read or written for the last time is marked to leave first
// (HBM sees 2.2 reads and 1.5 writes a pixel, 3.3 and 1.9 without the marks).
// 4,096 patterns of 256 x 256: 1.02 ms, bound by the latency of the passes' loads
// (L2 and HBM, 46 % of the issue slots used, 86 instructions a pixel); 1.23 ms
// without the marks, 1.59 ms with scalar float-float arithmetic, index
// arithmetic for every pixel and a pass over the fit's sign (188 instructions),
// 2.40 ms with one load in flight per thread, an integer division per pixel
// and pass and the chunk sums in FP64.
#include <math.h>
#include <string.h>

#include <type_traits>

#include "internal.cuh"

namespace {

constexpr int kPreThreads = 512, kPreChunk = 8;
constexpr int kSmallThreads = 128, kSmallDim = 128, kSmallPixels = 4096;   // small patterns (see preprocess_kernel)

struct QuadricInverse {
    double ginv[36];   // inverse Gram matrix of the basis {1, x, y, x^2, xy, y^2}
    unsigned mw;       // ceil(2^32 / W): p / W = umulhi(p, mw) while p W < 2^32
};

__device__ __forceinline__ void basis6(float x, float y, float *phi)
{
    phi[0] = 1.0f;
    phi[1] = x;
    phi[2] = y;
    phi[3] = x * x;
    phi[4] = x * y;
    phi[5] = y * y;
}

// Block-wide sum of NV doubles per thread (NV <= 8); result broadcast.  Each exchange of the warp tree
// halves the values a lane carries (the pairs that are added stay those of a butterfly), so that six
// values cost 9 FP64 additions instead of 30.
template <int NV>
__device__ void block_sum(double (&v)[NV], double *red /* [32][NV] */)
{
    constexpr int P2 = NV > 4 ? 8 : NV > 2 ? 4 : NV;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    // sums over the warp; lane 32 k / P2 ends with value k
    auto warp_sum = [&](double (&x)[P2]) {
        int n = P2;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const bool up = (lane & o) != 0;
            if (n > 1) {
                n /= 2;
#pragma unroll
                for (int k = 0; k < P2 / 2; ++k)
                    if (k < n) {
                        const double give = up ? x[k] : x[k + n], keep = up ? x[k + n] : x[k];
                        x[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                    }
            } else {
                x[0] += __shfl_xor_sync(0xffffffffu, x[0], o);
            }
        }
    };
    const int mine = lane * P2 / 32;   // the value that this lane ends with
    const bool owner = lane % (32 / P2) == 0 && mine < NV;
    double x[P2];
#pragma unroll
    for (int k = 0; k < P2; ++k) x[k] = k < NV ? v[k] : 0.0;
    warp_sum(x);
    if (owner) red[wid * NV + mine] = x[0];
    __syncthreads();
    if (wid == 0) {
#pragma unroll
        for (int k = 0; k < P2; ++k) x[k] = k < NV && lane < nw ? red[lane * NV + k] : 0.0;
        __syncwarp();
        warp_sum(x);
        if (owner) red[mine] = x[0];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = red[k];
    __syncthreads();
}

// Unevaluated sums hi + lo of two FP32 values ("float-float", ~48 bits): the
// background quadric and the quotient pattern / quadric are evaluated in this
// precision, because the normalised output is a difference of two numbers near
// one divided by a standard deviation near 0.1, so plain FP32 would carry a
// smooth error pattern of ~10 units in the last place of the output.
struct ff {
    float hi, lo;
};

__device__ __forceinline__ ff ff_from_double(double v)
{
    const float h = (float)v;
    return {h, (float)(v - (double)h)};
}

// exact sum of two floats (Knuth's two-sum)
__device__ __forceinline__ ff two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}

// The same where a is zero or a multiple of the last place of b, or |a| >= |b| (Dekker's fast two-sum):
// three operations, the same pair.
__device__ __forceinline__ ff fast_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

// Two pixels' float-float numbers at a time, in packed FP32x2 arithmetic (a - b as fma(b, -1, a)); every
// rounding step is the scalar one.
struct ff2 {
    float2 hi, lo;
};
__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, both(-1.0f), a); }
__device__ __forceinline__ ff2 two_sum(float2 a, float2 b)
{
    const float2 s = __fadd2_rn(a, b), bb = sub2(s, a);
    return {s, __fadd2_rn(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ ff2 fast_two_sum(float2 a, float2 b)
{
    const float2 s = __fadd2_rn(a, b);
    return {s, sub2(b, sub2(s, a))};
}

// The last step of a sum: s.hi is a multiple of the smaller last place of a.hi and b.hi; where that is not
// one of lo's, one of them is 2^20 times the other and |s.hi| > |lo|.
__device__ __forceinline__ ff2 ff_add(ff2 a, ff2 b)
{
    const ff2 s = two_sum(a.hi, b.hi);
    return fast_two_sum(s.hi, __fadd2_rn(s.lo, __fadd2_rn(a.lo, b.lo)));
}

// a b, na = -a.hi.  (The error term of a product is at most a few of its last places.)
__device__ __forceinline__ ff2 ff_mul(ff2 a, float2 na, ff2 b)
{
    const float2 np = __fmul2_rn(na, b.hi);                // minus the product
    float2 e = __ffma2_rn(a.hi, b.hi, np);                 // its exact error
    e = __ffma2_rn(a.hi, b.lo, __ffma2_rn(a.lo, b.hi, e));
    const float2 s = sub2(e, np);                          // fast_two_sum(-np, e)
    return {s, sub2(e, __fadd2_rn(s, np))};
}

// A running sum of FP32 terms in three parts with exact carries (~72 bits): what a sum in FP64 holds,
// without the FP64 pipe (2 lanes per clock and SM), which bounded this kernel when every chunk's sums
// were converted and added there.
struct Sum3 {
    float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f;
    __device__ __forceinline__ void add(float v)
    {
        const ff a = two_sum(s0, v);
        s0 = a.hi;
        const ff b = two_sum(s1, a.lo);
        s1 = b.hi;
        s2 = __fadd_rn(s2, b.lo);
    }
};
struct Sum3x2 {   // two of them
    float2 s0 = {0.0f, 0.0f}, s1 = {0.0f, 0.0f}, s2 = {0.0f, 0.0f};
    __device__ __forceinline__ void add(float2 v)
    {
        const ff2 a = two_sum(s0, v);
        s0 = a.hi;
        const ff2 b = two_sum(s1, a.lo);
        s1 = b.hi;
        s2 = __fadd2_rn(s2, b.lo);
    }
};

// coordinate (2 k + 1 - n) / n in [-1, 1] of pixel k of n as hi + lo
__device__ __forceinline__ ff pixel_coord(int k, int n)
{
    const float num = (float)(2 * k + 1 - n), den = (float)n;   // exact integers
    const float h = __fdiv_rn(num, den);
    const float l = __fdiv_rn(__fmaf_rn(-h, den, num), den);   // the residual num - h n is exact
    return {h, l};
}

constexpr int kMaxDim = 1536;   // largest H and W of the background fit (per-row and per-column terms in shared memory)

__device__ __forceinline__ unsigned cluster_reg(bool size)
{
    unsigned r;
    if (size) asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    else asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Value at the shared-memory address `p` of this CTA in the CTA of rank `r`.
template <class T>
__device__ __forceinline__ T remote(const T *p, unsigned r)
{
    static_assert(sizeof(T) == 4 || sizeof(T) == 8, "float or double");
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm volatile("mapa.shared::cluster.u32 %0, %0, %1;" : "+r"(a) : "r"(r));
    T v;
    if constexpr (sizeof(T) == 4) asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    else asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}

// COL: the width divides the CTA's threads, so that a thread's pixels lie in one column.
// NT threads on patterns of at most DIM rows and columns.  Patterns of up to 4,096 pixels take 128 threads: 512 of
// them have little to do each and only three such CTAs fit an SM: 20,000 of 8 x 8 1,967 -> 568 us (without the fit
// 1,444 -> 382), 2,000 of 64 x 64 219 -> 69, one of 64 x 64 22 -> 14.
// CL: a cluster of CTAs shares the pattern, the chunks dealt out in turn.  The threads' partial sums of the
// ranks are added exactly (Sum3), thread by thread, in rank 0, so that they are the sums of one CTA.
template <bool COL, bool CL, int NT = kPreThreads, int DIM = kMaxDim>
__global__ void __launch_bounds__(NT, CL ? 2 : NT == kPreThreads ? 3 : 8) preprocess_kernel(const float *__restrict__ in, float *out, int H,
                                                                 int W, int flat, QuadricInverse qi)
{
    extern __shared__ float sums[];   // CL: the threads' partial sums [18][kPreThreads]
    const unsigned csize = CL ? cluster_reg(true) : 1, rank = CL ? cluster_reg(false) : 0;
    __shared__ double red[32 * 6];
    __shared__ double coef[7];   // the quadric's coefficients, the pattern's sum
    __shared__ float2 rowA[DIM], rowB[DIM];   // per row: c0 + c2 y + c5 y^2 and c1 + c4 y (hi, lo)
    __shared__ float2 colX[COL ? 1 : DIM];        // per column: x (hi, lo)
    __shared__ float rowY[DIM];                   // per row: y (the correctly rounded FP32 coordinate)
    const size_t base = (size_t)(CL ? blockIdx.x / csize : blockIdx.x) * H * W;
    const float *img = in + base;
    constexpr int bd = NT, cs = kPreThreads;   // threads; pixels between two of a chunk (whatever the threads: same sums)
    const int t = threadIdx.x;
    auto row_of = [&](int p) { return (int)__umulhi((unsigned)p, qi.mw); };
    const int n = H * W, rstep = COL ? cs / W : 0;   // COL: rows between a chunk's pixels

    // Sums are taken in FP32 over chunks of kChunk pixels of one thread, the chunk sums added exactly and
    // the threads' sums in FP64: the quadric's coefficients come out of a poorly conditioned 6 x 6 system, and plain FP32
    // sums of ~128 terms would move the output by ~1e-4.
    constexpr int kChunk = kPreChunk;
    ff xt{0.0f, 0.0f};   // COL: the thread's column
    if (flat) {   // the pixel coordinates, once per row and column
        if (COL) xt = pixel_coord(t % W, W);
        else
            for (int j = t; j < W; j += bd) {
                const ff x = pixel_coord(j, W);
                colX[j] = make_float2(x.hi, x.lo);
            }
        for (int i = t; i < H; i += bd) rowY[i] = pixel_coord(i, H).hi;
        __syncthreads();
    }
    // f(p0, whole) for this thread's chunks of the pixels p0, p0 + cs, ...; whole: every pixel is inside (else f counts
    // the others as 0).  A chunk's pixels are loaded before any of them is used, so that a thread has kChunk
    // loads in flight: the passes are bound by memory latency otherwise.
    auto chunks = [&](auto f) {
        auto from = [&](int q) {
            int p0 = q + (int)rank * (kChunk * cs);
            for (; p0 + (kChunk - 1) * cs < n; p0 += (int)csize * (kChunk * cs)) f(p0, std::true_type());
            if (p0 < n) f(p0, std::false_type());
        };
        if constexpr (bd == cs) from(t);
        else
#pragma unroll 1
            for (int q = t; q < cs; q += bd) from(q);
    };
    // false for pixels c of a chunk that are past the end for every thread (small patterns)
    auto any = [&](int c, auto whole) { return bd == cs || whole || c * cs < n; };
    // last: read for the last time (the line is the first to leave L2)
    auto load = [&](const float *src, int p0, auto whole, float (&v)[kChunk], auto last) {
#pragma unroll
        for (int c = 0; c < kChunk; ++c)
            v[c] = whole || p0 + c * cs < n ? (last ? __ldcs(src + p0 + c * cs) : src[p0 + c * cs]) : 0.0f;
    };
    // row and column of a chunk's pixel c (past the end: the last row); i0 = row_of(p0)
    auto cell = [&](int p0, int i0, int c, auto whole, int &i, int &j) {
        if (COL) {
            i = i0 + c * rstep;
            if (!whole) i = min(i, H - 1);
            j = 0;
        } else {
            const int p = whole ? p0 + c * cs : min(p0 + c * cs, n - 1);
            i = c == 0 ? i0 : row_of(p);
            j = p - i * W;
        }
    };
    // CL: thread t's parts x[0 .. NF) (three per sum) of all ranks added in rank 0; the caller meets once more
    // before `sums` is written again
    auto merge = [&](auto *x, auto nf) {
        constexpr int NF = decltype(nf)::value;
        if (!CL) return;
#pragma unroll
        for (int k = 0; k < NF; ++k) sums[k * bd + t] = x[k];
        cluster_sync();
        if (rank == 0)
            for (unsigned r = 1; r < csize; ++r) {
                float y[NF];
#pragma unroll
                for (int k = 0; k < NF; ++k) y[k] = remote(sums + k * bd + t, r);
#pragma unroll
                for (int k = 0; k < NF; k += 3) {
                    Sum3 s{x[k], x[k + 1], x[k + 2]};
                    s.add(y[k]);
                    s.add(y[k + 1]);
                    s.add(y[k + 2]);
                    x[k] = s.s0;
                    x[k + 1] = s.s1;
                    x[k + 2] = s.s2;
                }
            }
    };
    auto value3 = [](const float *x) { return (double)x[0] + ((double)x[1] + (double)x[2]); };
    // one sum over the pattern, in every thread of the cluster
    auto total_of = [&](const Sum3 &part) {
        float x[3] = {part.s0, part.s1, part.s2};
        merge(x, std::integral_constant<int, 3>());
        double s[1] = {value3(x)};
        block_sum<1>(s, red);
        if (CL) {
            if (t == 0) coef[0] = s[0];
            cluster_sync();
            if (rank) s[0] = remote(coef, 0);
            cluster_sync();
        }
        return s[0];
    };
    // pass 1: quadric moments b_k = sum phi_k I (basis at the correctly rounded pixel coordinates);
    // b_0 is the pattern's sum
    double total = 0.0;
    if (flat) {
        Sum3x2 part[3];
        chunks([&](int p0, auto whole) {
            float acc[6] = {0, 0, 0, 0, 0, 0}, v[kChunk];
            load(img, p0, whole, v, std::false_type());
            const int i0 = row_of(p0);
#pragma unroll
            for (int c = 0; c < kChunk; ++c) {
                if (!any(c, whole)) break;
                int i, j;
                cell(p0, i0, c, whole, i, j);
                float phi[6];
                basis6(COL ? xt.hi : colX[j].x, rowY[i], phi);
#pragma unroll
                for (int k = 0; k < 6; ++k) acc[k] = fmaf(phi[k], v[c], acc[k]);
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) part[k].add(make_float2(acc[2 * k], acc[2 * k + 1]));
        });
        float x[18];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            x[3 * k] = k % 2 ? part[k / 2].s0.y : part[k / 2].s0.x;
            x[3 * k + 1] = k % 2 ? part[k / 2].s1.y : part[k / 2].s1.x;
            x[3 * k + 2] = k % 2 ? part[k / 2].s2.y : part[k / 2].s2.x;
        }
        merge(x, std::integral_constant<int, 18>());
        double d[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) d[k] = value3(x + 3 * k);
        block_sum<6>(d, red);
        if (t == 0) {
            for (int r = 0; r < 6; ++r) {
                double c = 0.0;
                for (int k = 0; k < 6; ++k) c += qi.ginv[r * 6 + k] * d[k];
                coef[r] = c;
            }
            coef[6] = d[0];
        }
        if (CL) {   // rank 0's coefficients and sum in every CTA
            cluster_sync();
            double c = 0.0;
            if (rank && t < 7) c = remote(coef + t, 0);
            cluster_sync();
            if (rank && t < 7) coef[t] = c;
        }
        __syncthreads();
        total = coef[6];
        // per-row parts of the quadric in FP64, kept as hi + lo
        for (int i = t; i < H; i += bd) {
            const double y = (2.0 * i + 1.0 - H) / H;
            const ff A = ff_from_double(coef[0] + y * (coef[2] + y * coef[5]));
            const ff Bc = ff_from_double(coef[1] + y * coef[4]);
            rowA[i] = make_float2(A.hi, A.lo);
            rowB[i] = make_float2(Bc.hi, Bc.lo);
        }
        __syncthreads();
    }
    const ff C = flat ? ff_from_double(coef[3]) : ff{0.0f, 0.0f};

    // the division is skipped when the fitted surface is not positive at every pixel (checked on the
    // FP32 value of the quadric, whose sign differs from the hi + lo one only within rounding of zero);
    // no pixel needs a look where every row's lower bound is clear of the rounding (3 x 2^-24 of its terms)
    bool use_fit = flat;
    if (flat) {
        bool bad = false;
        for (int i = t; i < H; i += bd) {
            const float a = rowA[i].x, b = fabsf(rowB[i].x), low = a - b - fmaxf(-C.hi, 0.0f);
            bad |= !(low > 1e-5f * (a + b + fabsf(C.hi)));
        }
        if (__syncthreads_or(bad)) {
            bad = false;
#pragma unroll 4
            for (int p = t; p < n; p += bd) {
                const int i = row_of(p);
                const float x = COL ? xt.hi : colX[p - i * W].x;
                bad |= !(fmaf(x, fmaf(x, C.hi, rowB[i].x), rowA[i].x) > 0.0f);
            }
            use_fit = !__syncthreads_or(bad);
        }
    }

    // pass 2: the pattern divided by the quadric A(y) + x (B(y) + x c3), as hi + lo: q ~ v / f (within 2 units
    // of the last place, from the correctly rounded reciprocal), the remainder v - q f.hi exact by fma, then the
    // correction (remainder - q f.lo) / f; with the division by f.hi a product with the same
    // reciprocal (its error lands ~2^-24 below the correction, itself ~2^-24 below q).  Of it the quotient
    // less K (1 for the background-divided pattern, whose values lie near one;
    // the mean intensity, rounded, for the raw one), d = (q.hi - K) + q.lo in FP32: the leading part
    // cancels before rounding, so d keeps the float-float accuracy of q and the mean of d is small; d
    // is stored in the output (the pattern is read before it is overwritten, by the same thread) and
    // summed for the mean
    if (!flat) {   // the raw pattern's sum for K
        Sum3 part;
        chunks([&](int p0, auto whole) {
            float sv = 0.0f, v[kChunk];
            load(img, p0, whole, v, std::false_type());
#pragma unroll
            for (int c = 0; c < kChunk; ++c) sv += v[c];
            part.add(sv);
        });
        total = total_of(part);
    }
    const float K = use_fit ? 1.0f : (float)(total / n);
    float *o = out + base;
    Sum3 sum_d;
    if (use_fit) {
        const ff2 C2 = {both(C.hi), both(C.lo)};
        const ff2 x1 = {both(xt.hi), both(xt.lo)}, xC1 = ff_mul(x1, both(-xt.hi), C2);
        chunks([&](int p0, auto whole) {
            float sd = 0.0f, v[kChunk];
            load(img, p0, whole, v, std::true_type());
            const int i0 = row_of(p0);
#pragma unroll
            for (int c = 0; c < kChunk; c += 2) {   // two pixels at a time
                if (!any(c, whole)) break;
                int i, j, i2, j2;
                cell(p0, i0, c, whole, i, j);
                cell(p0, i0, c + 1, whole, i2, j2);
                const float2 a = rowA[i], a2 = rowA[i2], b = rowB[i], b2 = rowB[i2];
                ff2 x = x1, xC = xC1;
                float2 nx = both(-xt.hi);
                if (!COL) {
                    const float2 xa = colX[j], xb = colX[j2];
                    x = {make_float2(xa.x, xb.x), make_float2(xa.y, xb.y)};
                    nx = __fmul2_rn(x.hi, both(-1.0f));
                    xC = ff_mul(x, nx, C2);
                }
                const ff2 A = {make_float2(a.x, a2.x), make_float2(a.y, a2.y)}, Bc = {make_float2(b.x, b2.x), make_float2(b.y, b2.y)};
                const ff2 f = ff_add(A, ff_mul(x, nx, ff_add(Bc, xC)));
                const float2 vv = make_float2(v[c], v[c + 1]);
                const float2 rf = make_float2(__frcp_rn(f.hi.x), __frcp_rn(f.hi.y));
                const float2 q = __fmul2_rn(vv, rf), nq = __fmul2_rn(q, both(-1.0f));
                const float2 r = __ffma2_rn(nq, f.lo, __ffma2_rn(nq, f.hi, vv));
                const ff2 e = fast_two_sum(q, __fmul2_rn(r, rf));
                const float2 d = __fadd2_rn(__fadd2_rn(e.hi, both(-K)), e.lo);
                if (whole || p0 + c * cs < n) o[p0 + c * cs] = d.x;
                if (whole || p0 + (c + 1) * cs < n) o[p0 + (c + 1) * cs] = d.y;
                sd += whole || p0 + c * cs < n ? d.x : 0.0f;
                sd += whole || p0 + (c + 1) * cs < n ? d.y : 0.0f;
            }
            sum_d.add(sd);
        });
    } else {
        chunks([&](int p0, auto whole) {
            float sd = 0.0f, v[kChunk];
            load(img, p0, whole, v, std::true_type());
#pragma unroll
            for (int c = 0; c < kChunk; ++c) {
                const float d = __fadd_rn(__fsub_rn(v[c], K), 0.0f);
                if (whole || p0 + c * cs < n) {
                    o[p0 + c * cs] = d;
                    sd += d;
                }
            }
            sum_d.add(sd);
        });
    }
    const double mean_d = total_of(sum_d) / n, mean = mean_d + (double)K;
    const float md = (float)mean_d;
    // pass 3: variance about the mean
    Sum3 sum_v;
    chunks([&](int p0, auto whole) {
        float ss = 0.0f, v[kChunk];
        load(o, p0, whole, v, std::false_type());
#pragma unroll
        for (int c = 0; c < kChunk; ++c) {
            const float d = whole || p0 + c * cs < n ? __fsub_rn(v[c], md) : 0.0f;
            ss = fmaf(d, d, ss);
        }
        sum_v.add(ss);
    });
    const double sdv = sqrt(total_of(sum_v) / n);
    const float inv = (sdv > 0.0 && sdv > 1e-6 * fabs(mean)) ? (float)(1.0 / sdv) : 0.0f;
    // pass 4: output
    chunks([&](int p0, auto whole) {
        float v[kChunk];
        load(o, p0, whole, v, std::true_type());
#pragma unroll
        for (int c = 0; c < kChunk; ++c)
            if (whole || p0 + c * cs < n) __stcs(o + p0 + c * cs, __fsub_rn(v[c], md) * inv);
    });
}

// One pyramid level down: the 2x2 box mean, floor(H/2) x floor(W/2) (an odd
// last row or column takes no part).  VEC: H and W even, so every pair of
// neighbours starts on an 8-byte boundary and is read as one float2.
template <bool VEC>
__global__ void reduce2_kernel(const float *__restrict__ in, float *__restrict__ out, int n, int H, int W)
{
    const int h = H >> 1, w = W >> 1;
    const size_t total = (size_t)n * h * w;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (size_t)gridDim.x * blockDim.x) {
        size_t img = idx / ((size_t)h * w);
        int rem = (int)(idx - img * h * w);
        int i = rem / w, j = rem - i * w;
        const float *p = in + img * H * W + (size_t)(2 * i) * W + 2 * j;
        float2 a, b;
        if (VEC) {
            a = *reinterpret_cast<const float2 *>(p);
            b = *reinterpret_cast<const float2 *>(p + W);
        } else {
            a = make_float2(p[0], p[1]);
            b = make_float2(p[W], p[W + 1]);
        }
        out[idx] = 0.25f * ((a.x + a.y) + (b.x + b.y));
    }
}

int quadric_inverse(int H, int W, QuadricInverse *qi)
{
    double G[36] = {0};
    for (int i = 0; i < H; ++i)
        for (int j = 0; j < W; ++j) {
            double x = (j + 0.5) / W * 2.0 - 1.0, y = (i + 0.5) / H * 2.0 - 1.0;
            double phi[6] = {1.0, x, y, x * x, x * y, y * y};
            for (int k = 0; k < 6; ++k)
                for (int l = k; l < 6; ++l) G[k * 6 + l] += phi[k] * phi[l];
        }
    for (int k = 0; k < 6; ++k)
        for (int l = 0; l < k; ++l) G[k * 6 + l] = G[l * 6 + k];
    // Gauss-Jordan inversion with partial pivoting
    double A[6][12];
    for (int r = 0; r < 6; ++r)
        for (int c = 0; c < 12; ++c) A[r][c] = c < 6 ? G[r * 6 + c] : (c - 6 == r);
    for (int c = 0; c < 6; ++c) {
        int piv = c;
        for (int r = c + 1; r < 6; ++r)
            if (fabs(A[r][c]) > fabs(A[piv][c])) piv = r;
        if (fabs(A[piv][c]) < 1e-300) return -1;
        for (int k = 0; k < 12; ++k) {
            double t = A[c][k];
            A[c][k] = A[piv][k];
            A[piv][k] = t;
        }
        double d = A[c][c];
        for (int k = 0; k < 12; ++k) A[c][k] /= d;
        for (int r = 0; r < 6; ++r)
            if (r != c) {
                double f = A[r][c];
                for (int k = 0; k < 12; ++k) A[r][k] -= f * A[c][k];
            }
    }
    for (int r = 0; r < 6; ++r)
        for (int c = 0; c < 6; ++c) qi->ginv[r * 6 + c] = A[r][c + 6];
    return 0;
}

// The inverse for a pattern size, from the context's few latest sizes: summing the Gram matrix over the
// pixels takes the host 0.2 ms at 128 x 128 and 15 ms at 1244 x 1024, more than the kernel on few patterns.
int quadric_plan(hrebsd_ctx *ctx, int H, int W, QuadricInverse *qi)
{
    for (auto &q : ctx->quadrics)
        if (q.H == H && q.W == W) {
            memcpy(qi->ginv, q.ginv, sizeof qi->ginv);
            return 0;
        }
    if (quadric_inverse(H, W, qi)) return -1;
    if (ctx->quadrics.size() >= 8) ctx->quadrics.erase(ctx->quadrics.begin());
    hr_quadric q{H, W, {}};
    memcpy(q.ginv, qi->ginv, sizeof q.ginv);
    ctx->quadrics.push_back(q);
    return 0;
}

}  // namespace

// Launch the 2x2 box-mean reduction of n images [n][H][W] -> [n][H/2][W/2].
int hr_launch_reduce2(hrebsd_ctx *ctx, const float *in, float *out, int n, int H, int W, cudaStream_t st)
{
    size_t total = (size_t)n * (H / 2) * (W / 2);
    if (total == 0) return HREBSD_OK;
    int blocks = (int)((total + 255) / 256);
    int cap = ctx->num_sms * 16;
    if (blocks > cap) blocks = cap;
    hr_prof_begin(ctx, st);
    if (H % 2 == 0 && W % 2 == 0 && ((uintptr_t)in & 7) == 0)
        reduce2_kernel<true><<<blocks, 256, 0, st>>>(in, out, n, H, W);
    else
        reduce2_kernel<false><<<blocks, 256, 0, st>>>(in, out, n, H, W);
    hr_prof_end(ctx, PROF_DEMONS_AUX, st);
    HR_LAUNCHED(ctx);
    return HREBSD_OK;
}

extern "C" int hrebsd_preprocess_batch(hrebsd_ctx *ctx, const float *in, int n, int H, int W, int flat, float *out,
                                       void *stream)
{
    if (!ctx || n < 0 || H < 2 || W < 2) return HREBSD_EINVAL;
    if (n == 0) return HREBSD_OK;
    if (!in || !out) return HREBSD_EINVAL;
    int st = hr_set_device(ctx);
    if (st) return st;
    if (flat && (H > kMaxDim || W > kMaxDim)) return HREBSD_EINVAL;
    QuadricInverse qi;
    if (flat && quadric_plan(ctx, H, W, &qi)) return HREBSD_EINVAL;
    qi.mw = (unsigned)(((1ull << 32) + W - 1) / W);
    if (!flat)
        for (double &g : qi.ginv) g = 0.0;
    hr_prof_begin(ctx, hr_stream(stream));
    // few patterns: a cluster of up to 8 CTAs on each, while two CTAs per SM hold them all and each has at least
    // four chunks.  One CTA -> cluster: one 1244 x 1024 908 -> 137 us, 60 of them 1,556 -> 492 us, 10 of 640 x 480
    // 239 -> 62 us, one 256 x 256 63 -> 38 us.  Beyond the rule: 200 of 256 x 256, which keep the SMs busy without,
    // 103 -> 98 us in pairs and 147 us in fours; one 128 x 128, of four chunks, 30 -> 32 us
    int C = 8;
    while (C > 1 && ((long long)n * C > 2 * ctx->num_sms || (long long)H * W < 4LL * C * kPreChunk * kPreThreads)) C /= 2;
    const bool small = C == 1 && H <= kSmallDim && W <= kSmallDim && H * W <= kSmallPixels;
    const int threads = small ? kSmallThreads : kPreThreads;
    // widths that divide the CTA (64, 128, 256 ...): the column's terms once per thread
    const bool col = threads % W == 0;
    auto k = small ? (col ? preprocess_kernel<true, false, kSmallThreads, kSmallDim> : preprocess_kernel<false, false, kSmallThreads, kSmallDim>)
           : C > 1 ? (col ? preprocess_kernel<true, true> : preprocess_kernel<false, true>)
                   : (col ? preprocess_kernel<true, false> : preprocess_kernel<false, false>);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n * C));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = hr_stream(stream);
    cudaLaunchAttribute at;
    if (C > 1) {
        cfg.dynamicSmemBytes = 18 * kPreThreads * sizeof(float);
        HR_CHECK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes));
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = (unsigned)C;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
    }
    HR_CHECK(cudaLaunchKernelEx(&cfg, k, in, out, H, W, flat, qi));
    hr_prof_end(ctx, PROF_PRE, hr_stream(stream));
    HR_LAUNCHED(ctx);
    return HREBSD_OK;
}

// Box mean of f x f blocks: [n][H][W] -> [n][H/f][W/f] (the pyramid level
// log2(f) in one pass; used to build the inputs and targets of the learned
// initialiser at the 64x64 level).
namespace {
__global__ void downsample_kernel(const float *__restrict__ in, float *__restrict__ out, int n, int H, int W, int f)
{
    const int h = H / f, w = W / f;
    const size_t total = (size_t)n * h * w;
    const float s = 1.0f / (float)(f * f);
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (size_t)gridDim.x * blockDim.x) {
        const size_t img = idx / ((size_t)h * w);
        const int rem = (int)(idx - img * h * w), i = rem / w, j = rem - i * w;
        const float *p = in + img * H * W + (size_t)(i * f) * W + j * f;
        float acc = 0.0f;
        for (int a = 0; a < f; ++a)
            for (int b = 0; b < f; ++b) acc += p[(size_t)a * W + b];
        out[idx] = acc * s;
    }
}
}  // namespace

extern "C" int hrebsd_downsample_batch(hrebsd_ctx *ctx, const float *in, int n, int H, int W, int f, float *out,
                                       void *stream)
{
    if (!ctx || n < 0 || f < 1 || H % f || W % f) return HREBSD_EINVAL;
    if (n == 0) return HREBSD_OK;
    if (!in || !out) return HREBSD_EINVAL;
    int e = hr_set_device(ctx);
    if (e) return e;
    size_t total = (size_t)n * (H / f) * (W / f);
    int grid = (int)((total + 255) / 256);
    if (grid > ctx->num_sms * 16) grid = ctx->num_sms * 16;
    hr_prof_begin(ctx, hr_stream(stream));
    downsample_kernel<<<grid, 256, 0, hr_stream(stream)>>>(in, out, n, H, W, f);
    hr_prof_end(ctx, PROF_PRE, hr_stream(stream));
    HR_LAUNCHED(ctx);
    return HREBSD_OK;
}

// Displacement field between pyramid resolutions (learned initialiser): planar
// [B][2][h][w] -> [B][2][h2][w2], values rescaled to the new pixel unit.
// Shrinking by f: box mean of f x f blocks / f.  Growing by f: bilinear sample
// at x_c = (x_f + 0.5) / f - 0.5 (clamped to the image) times f, which for f = 2
// is the prolongation between registration levels (Section 1).
namespace {
__device__ __forceinline__ float bilinear_plane(const float *__restrict__ M, int h, int w, float x, float y)
{
    x = fminf(fmaxf(x, 0.0f), (float)(w - 1));
    y = fminf(fmaxf(y, 0.0f), (float)(h - 1));
    const int x0 = min((int)x, max(w - 2, 0)), y0 = min((int)y, max(h - 2, 0));
    const int x1 = min(x0 + 1, w - 1), y1 = min(y0 + 1, h - 1);
    const float fx = x - (float)x0, fy = y - (float)y0;
    const float a = M[y0 * w + x0], b = M[y0 * w + x1], c = M[y1 * w + x0], d = M[y1 * w + x1];
    const float top = fmaf(fx, b, (1.0f - fx) * a), bot = fmaf(fx, d, (1.0f - fx) * c);
    return fmaf(fy, bot, (1.0f - fy) * top);
}

__global__ void field_resample_kernel(const float *__restrict__ in, int B, int h, int w, float *__restrict__ out,
                                      int h2, int w2)
{
    const size_t total = (size_t)B * 2 * h2 * w2;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (size_t)gridDim.x * blockDim.x) {
        const size_t plane = idx / ((size_t)h2 * w2);   // b * 2 + component
        const int rem = (int)(idx - plane * h2 * w2), i = rem / w2, j = rem - i * w2;
        const float *src = in + plane * h * w;
        float v;
        if (h2 <= h) {
            const int f = h / h2;
            float acc = 0.0f;
            for (int a = 0; a < f; ++a)
                for (int b = 0; b < f; ++b) acc += src[(size_t)(i * f + a) * w + j * f + b];
            v = acc / (float)(f * f) / (float)f;
        } else {
            const int f = h2 / h;
            const float inv = 1.0f / (float)f;
            v = (float)f * bilinear_plane(src, h, w, ((float)j + 0.5f) * inv - 0.5f, ((float)i + 0.5f) * inv - 0.5f);
        }
        out[idx] = v;
    }
}

bool pow2_ratio(int a, int b)   // a = b * 2^k, k >= 0
{
    if (a < b || a % b) return false;
    const int r = a / b;
    return (r & (r - 1)) == 0;
}
}  // namespace

extern "C" int hrebsd_field_resample(hrebsd_ctx *ctx, const float *in, int B, int h, int w, float *out, int h2, int w2,
                                     void *stream)
{
    if (!ctx || B < 0 || h < 1 || w < 1 || h2 < 1 || w2 < 1) return HREBSD_EINVAL;
    const bool shrink = h2 <= h;
    if (shrink ? !(pow2_ratio(h, h2) && pow2_ratio(w, w2) && h / h2 == w / w2)
               : !(pow2_ratio(h2, h) && pow2_ratio(w2, w) && h2 / h == w2 / w))
        return HREBSD_EINVAL;
    if (B == 0) return HREBSD_OK;
    if (!in || !out) return HREBSD_EINVAL;
    int e = hr_set_device(ctx);
    if (e) return e;
    const size_t total = (size_t)B * 2 * h2 * w2;
    int grid = (int)((total + 255) / 256);
    if (grid > ctx->num_sms * 16) grid = ctx->num_sms * 16;
    hr_prof_begin(ctx, hr_stream(stream));
    field_resample_kernel<<<grid, 256, 0, hr_stream(stream)>>>(in, B, h, w, out, h2, w2);
    hr_prof_end(ctx, PROF_CNN, hr_stream(stream));
    HR_LAUNCHED(ctx);
    return HREBSD_OK;
}
