// f2: pattern preprocessing for real scans (Section 3.2-3.3): Gaussian
// low-/high-pass filtering, static and dynamic background correction, and the
// shift and zoom/shrink correction about the pattern centre.  The paper names
// these steps without their kernels; the library uses Gaussian filters of
// radius ceil(3 sigma) with normalised weights and replicated borders (the
// family of the demons smoothing), division by the scan's mean pattern
// (static) and by the pattern's own blur (dynamic), and a Keys cubic resample
// for the affine correction.  Everything is FP32 with FP32 accumulation (the
// mean over the scan in three FP32 parts with exact carries, combined in FP64).
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "internal.cuh"

namespace {

constexpr int kMaxFilterRadius = 96;

struct FilterTaps {
    int r;
    float t[2 * kMaxFilterRadius + 1];
};

bool make_taps(float sigma, FilterTaps *f)
{
    if (!(sigma >= 0.0f)) return false;
    if (sigma == 0.0f) {
        f->r = 0;
        f->t[0] = 1.0f;
        return true;
    }
    const int r = (int)ceil(3.0 * (double)sigma);
    if (r > kMaxFilterRadius) return false;
    double s = 0.0, w[2 * kMaxFilterRadius + 1];
    for (int k = -r; k <= r; ++k) s += (w[k + r] = exp(-(double)k * k / (2.0 * (double)sigma * sigma)));
    f->r = r;
    for (int k = 0; k <= 2 * r; ++k) f->t[k] = (float)(w[k] / s);
    return true;
}

// a / d, 0 where |d| < 1e-12
__device__ __forceinline__ float guarded_div(float a, float d) { return fabsf(d) >= 1e-12f ? a / d : 0.0f; }

// One direction of the separable blur (AXIS 0: along x, 1: along y), replicated borders.
//
// A CTA takes 32 lines (rows for x, columns for y, of all images one after the other) and a segment of at most 256 outputs along them; the
// lines lie in shared memory with their halo, two neighbouring lines interleaved as one float2.  Thread
// (pair, run) computes RUN consecutive outputs of its two lines: the window of RUN inputs sits in
// registers (input j in slot j mod RUN, so nothing moves), a tap is one shared-memory load and RUN packed
// FMAs.  Every output sums its taps in the order k = -r .. r, as one thread per output would.  Bound by
// the FP32 FMAs from radius ~20 up (2r + 1 per pixel), by HBM below.  1000 patterns of 256 x 256:
// radius 3 101 us each direction (one thread per output and tap: 350), radius 60 373 us along x and 341
// along y (was 2,900 each), the whole dynamic correction (radius 36) 730 us (was 4,000).
//
// The passes carry the element-wise steps around them, so that no intermediate image is written for
// them: PRE divides the input by the background bg as it is loaded; POST divides the input of the
// whole blur (src, by bg too if given) by the blurred value, or subtracts that from src.
enum { POST_NONE = 0, POST_DIV, POST_SUB };
constexpr int RUN = 16, LINES = 32, PAIRS = LINES / 2, MAX_SEG = 256;
// Shared memory of the largest tile.  The limit set on a kernel holds for the whole device, other handles and
// threads included, so it is this constant and not the call's own need.
constexpr int MAX_SMEM = PAIRS * ((MAX_SEG + 2 * kMaxFilterRadius) | 1) * (int)sizeof(float2);

struct BlurArgs {
    const float *in;    // input of this pass
    const float *src;   // POST: the image the result is combined with
    const float *bg;    // [H][W] static background (nullable)
    float *out;
    unsigned lines;     // rows (x) or columns (y; an odd width counts one more, so that a pair is of one image) of all images
    int H, W, segs, seg, stride, vec;   // segments per line, outputs per segment, float2 stride of a line pair
};

template <int AXIS, bool PRE, int POST>
__global__ void __launch_bounds__(256, 3) blur_pass_kernel(BlurArgs a, const __grid_constant__ FilterTaps f)
{
    extern __shared__ __align__(16) float2 blur_smem[];
    const int H = a.H, W = a.W, r = f.r, len = AXIS ? H : W;
    const size_t plane = (size_t)H * W;
    const int s0 = (int)(blockIdx.x % a.segs) * a.seg;        // first output of the segment
    const unsigned l0 = blockIdx.x / a.segs * LINES;          // first line
    const int n_out = min(a.seg, len - s0), n_in = a.seg + 2 * r;
    float *sm = reinterpret_cast<float *>(blur_smem);
    auto slot = [&](int line, int j) { return sm + 2 * ((line >> 1) * a.stride + j) + (line & 1); };
    // asynchronous copies: every load of the tile is in flight at once
    auto copy = [&](float *dst, const float *src) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                     : "memory");
    };
    if (AXIS) {   // lanes on columns: coalesced loads, conflict-free stores
        const int line = threadIdx.x & 31;
        const unsigned col = l0 + line, We = (W + 1) & ~1u, image = col / We;
        const int x = (int)(col - image * We);
        const float *img = a.in + image * plane + x;
        if (col < a.lines && x < W)
#pragma unroll 4
            for (int j = threadIdx.x >> 5; j < n_in; j += (int)blockDim.x >> 5)
                copy(slot(line, j), img + (size_t)min(max(s0 - r + j, 0), H - 1) * W);
    } else {
        for (int line = threadIdx.x >> 5; line < LINES; line += (int)blockDim.x >> 5) {
            const unsigned row = l0 + line;
            if (row >= a.lines) break;
            const float *p = a.in + (size_t)row * W;
#pragma unroll 4
            for (int j = threadIdx.x & 31; j < n_in; j += 32)
                copy(slot(line, j), p + min(max(s0 - r + j, 0), W - 1));
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (PRE)   // every thread divides what it copied
        for (int line = threadIdx.x >> 5; line < LINES; line += (int)blockDim.x >> 5) {
            const unsigned row = l0 + line;
            if (row >= a.lines) break;
            const float *bg = a.bg + (size_t)(row % H) * W;
#pragma unroll 4
            for (int j = threadIdx.x & 31; j < n_in; j += 32) {
                float *p = slot(line, j);
                *p = guarded_div(*p, __ldg(bg + min(max(s0 - r + j, 0), W - 1)));
            }
        }
    __syncthreads();
    // an odd number of runs leaves half a warp over: it repeats the last run and stores nothing
    const int pr = threadIdx.x % PAIRS, o0 = min((int)threadIdx.x / PAIRS * RUN, a.seg - RUN);
    const bool live = (int)threadIdx.x / PAIRS * RUN < a.seg;
    const float2 *q = blur_smem + pr * a.stride + o0;
    float2 acc[RUN], win[RUN];
#pragma unroll
    for (int i = 0; i < RUN; ++i) {
        acc[i] = make_float2(0.0f, 0.0f);
        win[i] = q[i];
    }
    auto taps = [&](int k, int u) {   // tap k = base + u, u = k mod RUN
        const float2 t = make_float2(f.t[k], f.t[k]);
#pragma unroll
        for (int i = 0; i < RUN; ++i) acc[i] = __ffma2_rn(t, win[(i + u) % RUN], acc[i]);
    };
    int k = 0;
    for (; k + RUN <= 2 * r + 1; k += RUN)
#pragma unroll
        for (int u = 0; u < RUN; ++u) {
            taps(k + u, u);
            if (k + u < 2 * r) win[u] = q[k + u + RUN];   // input of tap k + u + 1's last output
        }
#pragma unroll
    for (int u = 0; u < RUN; ++u) {
        if (k + u > 2 * r) break;
        taps(k + u, u);
        if (k + u < 2 * r) win[u] = q[k + u + RUN];
    }
    if (AXIS) {
        const unsigned col = l0 + 2 * pr, We = (W + 1) & ~1u, image = col / We;
        const int x = (int)(col - image * We), rows = live && col < a.lines ? n_out - o0 : 0;   // this thread's outputs
        const bool two = x + 1 < W;
        const size_t p0 = (size_t)(s0 + o0) * W + x, at0 = image * plane + p0;
        if (POST != POST_NONE) {   // all loads of the run before any use (src may be out: read here, written below)
            float2 c[RUN];
#pragma unroll
            for (int i = 0; i < RUN; ++i)
                c[i] = i < rows ? make_float2(a.src[at0 + (size_t)i * W], two ? a.src[at0 + (size_t)i * W + 1] : 0.0f)
                                : make_float2(0.0f, 0.0f);
            if (POST == POST_DIV && a.bg)
#pragma unroll
                for (int i = 0; i < RUN; ++i)
                    if (i < rows) {
                        c[i].x = guarded_div(c[i].x, __ldg(a.bg + p0 + (size_t)i * W));
                        if (two) c[i].y = guarded_div(c[i].y, __ldg(a.bg + p0 + (size_t)i * W + 1));
                    }
#pragma unroll
            for (int i = 0; i < RUN; ++i)
                acc[i] = POST == POST_DIV ? make_float2(guarded_div(c[i].x, acc[i].x), guarded_div(c[i].y, acc[i].y))
                                          : make_float2(c[i].x - acc[i].x, c[i].y - acc[i].y);
        }
#pragma unroll
        for (int i = 0; i < RUN; ++i) {
            if (i >= rows) break;
            float *o = a.out + at0 + (size_t)i * W;
            if (a.vec) {
                *reinterpret_cast<float2 *>(o) = acc[i];
            } else {
                o[0] = acc[i].x;
                if (two) o[1] = acc[i].y;
            }
        }
    } else {   // through shared memory, so that rows are written whole
        __syncthreads();
        if (live)
#pragma unroll
            for (int i = 0; i < RUN; ++i) blur_smem[pr * a.stride + o0 + i] = acc[i];
        __syncthreads();
        for (int line = threadIdx.x >> 5; line < LINES; line += (int)blockDim.x >> 5) {
            const unsigned row = l0 + line;
            if (row >= a.lines) break;
            for (int j = threadIdx.x & 31; j < n_out; j += 32)
                a.out[(size_t)row * W + s0 + j] = sm[2 * ((line >> 1) * a.stride + j) + (line & 1)];
        }
    }
}

// The same pass with one thread per output (no PRE), the same sums in the same order: few or small images, where
// the chain of a thread's 32 outputs in the kernel above is the time.
template <int AXIS, int POST>
__global__ void __launch_bounds__(256) blur_point_kernel(const float *__restrict__ in, const float *src, float *out, size_t total,
                                                         int H, int W, const __grid_constant__ FilterTaps f)
{
    const size_t plane = (size_t)H * W;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const size_t image = i / plane;
        const int p = (int)(i - image * plane), y = p / W, x = p - y * W, at = AXIS ? y : x, last = (AXIS ? H : W) - 1;
        const float *line = in + image * plane + (AXIS ? (size_t)x : (size_t)y * W);
        float acc = 0.0f;
#pragma unroll 4
        for (int k = -f.r; k <= f.r; ++k) acc = fmaf(f.t[k + f.r], __ldg(line + (size_t)min(max(at + k, 0), last) * (AXIS ? W : 1)), acc);
        out[i] = POST == POST_DIV ? guarded_div(src[i], acc) : POST == POST_SUB ? src[i] - acc : acc;
    }
}

// out = a / d, the [H][W] plane d broadcast over the images
__global__ void div_kernel(const float *a, const float *d, float *out, size_t total, size_t plane)
{
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x)
        out[i] = guarded_div(a[i], d[i % plane]);
}

// s + v exactly as s + e (Knuth's two-sum)
__device__ __forceinline__ void two_sum(float &s, float v, float &e)
{
    const float t = s + v, b = t - s;
    e = (s - (t - b)) + (v - b);
    s = t;
}

// Mean over the n images: GROUPS groups of images x 256 / GROUPS pixels per CTA.  FP64 additions and conversions
// would bound it (1000 patterns of 256 x 256: 289 us with one thread per pixel, 261 us in eight groups), so a
// group sums in three FP32 parts with exact carries, which hold more bits than one FP64 sum, and only the
// parts and the groups' sums are added in FP64 (49 us; the read alone takes 39).  Sums that leave the range of
// FP32 (or are not finite) are repeated in FP64.
template <int GROUPS>
__global__ void __launch_bounds__(256) mean_pattern_kernel(const float *__restrict__ in, int n, size_t plane, float *out)
{
    constexpr int PX = 256 / GROUPS;
    __shared__ double part[GROUPS][PX];
    const int lane = threadIdx.x % PX, grp = threadIdx.x / PX;
    const size_t p = (size_t)blockIdx.x * PX + lane;
    double s = 0.0;
    if (GROUPS == 1 && n <= 2) {   // fewer FP64 operations than the parts' combination
        if (p < plane)
            for (int i = 0; i < n; ++i) s += __ldg(in + p + (size_t)i * plane);
    } else if (p < plane) {
        const float *q = in + p;
        float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f, e;
        auto add = [&](float v) {
            two_sum(s0, v, e);
            two_sum(s1, e, e);
            s2 += e;
        };
        int i = grp;
        for (; i + 7 * GROUPS < n; i += 8 * GROUPS) {
            float v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = __ldg(q + (size_t)(i + GROUPS * j) * plane);
#pragma unroll
            for (int j = 0; j < 8; ++j) add(v[j]);
        }
        for (; i < n; i += GROUPS) add(__ldg(q + (size_t)i * plane));
        s = (double)s0 + ((double)s1 + (double)s2);
        if (!isfinite(s)) {
            s = 0.0;
            for (i = grp; i < n; i += GROUPS) s += __ldg(q + (size_t)i * plane);
        }
    }
    if (GROUPS > 1) {
        part[grp][lane] = s;
        __syncthreads();
    }
    if (grp == 0 && p < plane) {
#pragma unroll
        for (int g = 1; g < GROUPS; ++g) s += part[g][lane];
        out[p] = (float)(s / n);
    }
}

__device__ __forceinline__ void keys4(float t, float *wt)
{
    const float a = -0.5f;
    const float s0 = t + 1.0f, s1 = t, s2 = 1.0f - t, s3 = 2.0f - t;
    wt[0] = ((a * s0 - 5.0f * a) * s0 + 8.0f * a) * s0 - 4.0f * a;
    wt[1] = ((a + 2.0f) * s1 - (a + 3.0f)) * s1 * s1 + 1.0f;
    wt[2] = ((a + 2.0f) * s2 - (a + 3.0f)) * s2 * s2 + 1.0f;
    wt[3] = ((a * s3 - 5.0f * a) * s3 + 8.0f * a) * s3 - 4.0f * a;
}

// out(x) = in(pc + (x - pc - t) / s), index coordinates, Keys cubic, replicated borders
__global__ void shift_zoom_kernel(const float *__restrict__ in, int n, int H, int W, const float *__restrict__ shift,
                                  const float *__restrict__ zoom, float pcx, float pcy, float *__restrict__ out)
{
    const size_t plane = (size_t)H * W, total = (size_t)n * plane;
    for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (size_t)gridDim.x * blockDim.x) {
        const size_t img = idx / plane;
        const int rem = (int)(idx - img * plane), yo = rem / W, xo = rem - yo * W;
        const float tx = shift ? shift[img * 2] : 0.0f, ty = shift ? shift[img * 2 + 1] : 0.0f;
        const float s = zoom ? zoom[img] : 1.0f;
        const float x = pcx + ((float)xo - pcx - tx) / s, y = pcy + ((float)yo - pcy - ty) / s;
        const float fx0 = floorf(x), fy0 = floorf(y);
        const int x0 = (int)fx0, y0 = (int)fy0;
        float wx[4], wy[4];
        keys4(x - fx0, wx);
        keys4(y - fy0, wy);
        const float *M = in + img * plane;
        float acc = 0.0f;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const float *row = M + (size_t)min(max(y0 - 1 + m, 0), H - 1) * W;
            float r = 0.0f;
#pragma unroll
            for (int k = 0; k < 4; ++k) r = fmaf(wx[k], __ldg(row + min(max(x0 - 1 + k, 0), W - 1)), r);
            acc = fmaf(wy[m], r, acc);
        }
        out[idx] = acc;
    }
}

int grid_of(hrebsd_ctx *ctx, size_t total)
{
    size_t g = (total + 255) / 256, cap = (size_t)ctx->num_sms * 16;
    return (int)(g < cap ? (g ? g : 1) : cap);
}

// One thread per output while a pass holds little: a tile of the other kernel takes 4 us however little it holds,
// 10 with divisions, and longer the more taps its threads add in turn; the points take 1.6 us, 0.2 us per million
// taps and what they move.  The line was drawn through measured times of 1 to 20,000 images of 8 x 8 to
// 1024 x 1244 (within 25 % of the better one).  Lines shorter than 32 leave most of a tile empty.  Static and
// dynamic correction, sigma 5, tiles -> points: one image of 92 x 100 30.1 -> 7.8 us, four of 256 x 256 24.3 -> 13.9,
// 20,000 of 8 x 8 163 -> 44; 30 of 256 x 256 stay with the tiles (29 us, points 74).
bool by_points(int n, int H, int W, const FilterTaps &f, bool divides)
{
    const double px = 1e-6 * n * H * W, taps = 2 * f.r + 1, narrow = std::max(1.0, 32.0 / std::min(H, W));
    return 0.5 * px * taps + 4.5 * px <= (divides ? (7.9 + 0.06 * taps) * narrow : 1.7 + 0.05 * taps) * narrow;
}

template <int AXIS, int POST>
int launch_points(hrebsd_ctx *ctx, const float *in, const float *src, float *out, int n, int H, int W, const FilterTaps &f,
                  cudaStream_t st)
{
    const size_t total = (size_t)n * H * W;
    blur_point_kernel<AXIS, POST><<<grid_of(ctx, total), 256, 0, st>>>(in, src, out, total, H, W, f);
    HR_LAUNCHED(ctx);
    return HREBSD_OK;
}

template <int AXIS, bool PRE, int POST>
int launch_pass(hrebsd_ctx *ctx, const float *in, const float *src, const float *bg, float *out, int n, int H, int W,
                const FilterTaps &f, cudaStream_t st)
{
    BlurArgs a;
    a.in = in;
    a.src = src;
    a.bg = bg;
    a.out = out;
    a.H = H;
    a.W = W;
    const int len = AXIS ? H : W, per_image = AXIS ? (W + 1) / 2 * 2 : H;   // lines of an image
    a.segs = (len + MAX_SEG - 1) / MAX_SEG;
    const int runs = ((len + a.segs - 1) / a.segs + RUN - 1) / RUN;   // at most 16
    a.seg = runs * RUN;
    a.stride = (a.seg + 2 * f.r) | 1;   // odd: 16 lanes on 16 line pairs hit distinct banks
    a.vec = (W % 2 == 0) && (reinterpret_cast<uintptr_t>(out) % 8 == 0);
    const size_t smem = (size_t)PAIRS * a.stride * sizeof(float2);
    auto k = blur_pass_kernel<AXIS, PRE, POST>;
    if (smem > 48 * 1024) HR_CHECK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_SMEM));
    // (lines are counted in 32 bits: more images than that go in parts)
    const int part = (int)std::min<long long>(n, std::max(1LL, (1LL << 30) / ((long long)per_image * a.segs)));
    for (int i0 = 0; i0 < n; i0 += part) {
        const size_t off = (size_t)i0 * H * W;
        BlurArgs c = a;
        c.in += off;
        c.out += off;
        if (c.src) c.src += off;
        c.lines = (unsigned)std::min(part, n - i0) * (unsigned)per_image;
        const unsigned tiles = (c.lines + LINES - 1) / LINES * (unsigned)a.segs;
        const int threads = (runs * PAIRS + 31) / 32 * 32;   // whole warps
        k<<<tiles, threads, smem, st>>>(c, f);
        HR_LAUNCHED(ctx);
    }
    return HREBSD_OK;
}

enum { WS_F0 = 16, WS_F1 = 17 };

}  // namespace

extern "C" int hrebsd_bandpass_batch(hrebsd_ctx *ctx, const float *in, int n, int H, int W, float sigma_lp,
                                     float sigma_hp, float *out, void *stream)
{
    FilterTaps lp, hp;
    if (!ctx || n < 0 || H < 1 || W < 1 || !make_taps(sigma_lp, &lp) || !make_taps(sigma_hp, &hp))
        return HREBSD_EINVAL;
    if (n == 0) return HREBSD_OK;
    if (!in || !out) return HREBSD_EINVAL;
    int e = hr_set_device(ctx);
    if (e) return e;
    const size_t total = (size_t)n * H * W;
    void *t0, *t1;
    if ((e = hr_ws(ctx, WS_F0, total * 4, &t0)) || (e = hr_ws(ctx, WS_F1, total * 4, &t1))) return e;
    cudaStream_t st = hr_stream(stream);
    hr_prof_begin(ctx, st);
    float *x = (float *)t0, *y = (float *)t1;
    // a blur of `in` into dst (in may be dst: read by the x pass only); POST: dst = src - blur
    auto blur = [&](const FilterTaps &f, const float *src, float *dst, auto post) {
        constexpr int POST = decltype(post)::value;
        const bool points = by_points(n, H, W, f, false);
        const int e2 = points ? launch_points<0, POST_NONE>(ctx, in, nullptr, x, n, H, W, f, st)
                              : launch_pass<0, false, POST_NONE>(ctx, in, nullptr, nullptr, x, n, H, W, f, st);
        if (e2) return e2;
        return points ? launch_points<1, POST>(ctx, x, src, dst, n, H, W, f, st)
                      : launch_pass<1, false, POST>(ctx, x, src, nullptr, dst, n, H, W, f, st);
    };
    using None = std::integral_constant<int, POST_NONE>;
    if (hp.r > 0 || sigma_hp > 0.0f) {   // out = G_lp * in - G_hp * in
        if ((e = blur(lp, nullptr, y, None()))) return e;
        if ((e = blur(hp, y, out, std::integral_constant<int, POST_SUB>()))) return e;
    } else {
        if ((e = blur(lp, nullptr, out, None()))) return e;
    }
    hr_prof_end(ctx, PROF_PRE, st);
    return HREBSD_OK;
}

extern "C" int hrebsd_mean_pattern(hrebsd_ctx *ctx, const float *in, int n, int H, int W, float *out, void *stream)
{
    if (!ctx || n < 1 || H < 1 || W < 1 || !in || !out) return HREBSD_EINVAL;
    int e = hr_set_device(ctx);
    if (e) return e;
    cudaStream_t st = hr_stream(stream);
    hr_prof_begin(ctx, st);
    const size_t plane = (size_t)H * W;
    // few images leave the groups little to share, and 32 pixels are little work for a CTA: 1024 x 1244, one image
    // 156 us in groups, 28 without, 16 images 158 and 99; from 32 images (small planes: 8) the groups are as fast
    const int groups = n < 8 || (n < 32 && plane >= 32768) ? 1 : 8;
    const unsigned ctas = (unsigned)((plane * groups + 255) / 256);
    (groups == 1 ? mean_pattern_kernel<1> : mean_pattern_kernel<8>)<<<ctas, 256, 0, st>>>(in, n, plane, out);
    hr_prof_end(ctx, PROF_PRE, st);
    HR_LAUNCHED(ctx);
    return HREBSD_OK;
}

extern "C" int hrebsd_background_batch(hrebsd_ctx *ctx, const float *in, int n, int H, int W, const float *static_bg,
                                       float sigma_dyn, float *out, void *stream)
{
    FilterTaps f;
    if (!ctx || n < 0 || H < 1 || W < 1 || !make_taps(sigma_dyn, &f)) return HREBSD_EINVAL;
    if (n == 0) return HREBSD_OK;
    if (!in || !out) return HREBSD_EINVAL;
    int e = hr_set_device(ctx);
    if (e) return e;
    const size_t total = (size_t)n * H * W, plane = (size_t)H * W;
    cudaStream_t st = hr_stream(stream);
    void *t0 = nullptr;
    if (sigma_dyn > 0.0f && (e = hr_ws(ctx, WS_F0, total * 4, &t0))) return e;
    float *x = (float *)t0;
    hr_prof_begin(ctx, st);
    if (sigma_dyn > 0.0f && by_points(n, H, W, f, true)) {   // the divided images in out (which may be in)
        if (static_bg) {
            div_kernel<<<grid_of(ctx, total), 256, 0, st>>>(in, static_bg, out, total, plane);
            HR_LAUNCHED(ctx);
        }
        const float *cur = static_bg ? out : in;
        if ((e = launch_points<0, POST_NONE>(ctx, cur, nullptr, x, n, H, W, f, st))) return e;
        if ((e = launch_points<1, POST_DIV>(ctx, x, cur, out, n, H, W, f, st))) return e;
    } else if (sigma_dyn > 0.0f) {   // out may be in: the y pass reads each of its pixels just before it writes it
        e = static_bg ? launch_pass<0, true, POST_NONE>(ctx, in, nullptr, static_bg, x, n, H, W, f, st)
                      : launch_pass<0, false, POST_NONE>(ctx, in, nullptr, nullptr, x, n, H, W, f, st);
        if (e) return e;
        if ((e = launch_pass<1, false, POST_DIV>(ctx, x, in, static_bg, out, n, H, W, f, st))) return e;
    } else if (static_bg) {
        div_kernel<<<grid_of(ctx, total), 256, 0, st>>>(in, static_bg, out, total, plane);
        HR_LAUNCHED(ctx);
    } else if (in != out) {
        HR_CHECK(cudaMemcpyAsync(out, in, total * 4, cudaMemcpyDeviceToDevice, st));
    }
    hr_prof_end(ctx, PROF_PRE, st);
    return HREBSD_OK;
}

extern "C" int hrebsd_shift_zoom_batch(hrebsd_ctx *ctx, const float *in, int n, int H, int W, const float *shift,
                                       const float *zoom, const hrebsd_geometry *g, float *out, void *stream)
{
    if (!ctx || !g || n < 0 || H < 1 || W < 1) return HREBSD_EINVAL;
    if (n == 0) return HREBSD_OK;
    if (!in || !out || in == out) return HREBSD_EINVAL;
    int e = hr_set_device(ctx);
    if (e) return e;
    const size_t total = (size_t)n * H * W;
    cudaStream_t st = hr_stream(stream);
    hr_prof_begin(ctx, st);
    shift_zoom_kernel<<<grid_of(ctx, total), 256, 0, st>>>(in, n, H, W, shift, zoom, (float)(g->xstar * W - 0.5),
                                                           (float)(g->ystar * H - 0.5), out);
    hr_prof_end(ctx, PROF_PRE, st);
    HR_LAUNCHED(ctx);
    return HREBSD_OK;
}
