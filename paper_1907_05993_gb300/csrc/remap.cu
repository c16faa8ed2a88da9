// a6: remap of the reference pattern by R_finite (Section 2, Eq. 12).
//
// Output pixel x' (test frame) looks up the reference at the gnomonic
// projection of R^T r', r' = (x' - xpc, y' - ypc, Z*): the reference point
// that Eq. 2 maps onto x' under the pure rotation R.  The value is a Keys
// (1981) cubic convolution (a = -0.5) over 4x4 reference pixels with
// replicated borders.  The references (a few grains) are gathered through the
// read-only path and stay in L2, so HBM traffic is the 4 B written per pixel;
// the kernel is bound by instruction issue (16 loads, the weights and 20 FMAs
// per pixel).  A thread computes ROWS output rows of its column, so that what
// depends on the pair, the column or the row group is worked out once for
// them: 2,500 pairs of 256 x 256 1,030 us, one row at a time 1,204 us.  Few
// pairs take one row per thread: a thread's rows are then the time (one pair
// of 128 x 128 2.8 us, four rows 4.4).
#include "internal.cuh"

namespace {

__device__ __forceinline__ void keys_weights(float t, float *wt)
{
    // taps at offsets -1, 0, 1, 2 of the floor sample; t in [0, 1)
    const float a = -0.5f;
    const float s0 = t + 1.0f, s1 = t, s2 = 1.0f - t, s3 = 2.0f - t;
    wt[0] = ((a * s0 - 5.0f * a) * s0 + 8.0f * a) * s0 - 4.0f * a;
    wt[1] = ((a + 2.0f) * s1 - (a + 3.0f)) * s1 * s1 + 1.0f;
    wt[2] = ((a + 2.0f) * s2 - (a + 3.0f)) * s2 * s2 + 1.0f;
    wt[3] = ((a * s3 - 5.0f * a) * s3 + 8.0f * a) * s3 - 4.0f * a;
}

// A CTA walks a contiguous run of row groups (ROWS consecutive rows of one pair; all index arithmetic
// 32-bit), threads along the rows; R^T of a pair is converted to FP32 registers once, when the run enters
// the pair.  Pixels whose 4 x 4 footprint lies inside the reference read it without clamping; the others
// clamp every tap (the same values, since the clamp only acts outside).
template <int ROWS>
__global__ void __launch_bounds__(256) remap_kernel(const float *__restrict__ ref, const int32_t *__restrict__ ref_idx,
                                                    const double *__restrict__ Rf, int B, int H, int W, float xpc,
                                                    float ypc, float zs, unsigned groups_per_cta, float *__restrict__ out)
{
    const unsigned per_pair = (unsigned)(H + ROWS - 1) / ROWS, total = (unsigned)B * per_pair;
    const unsigned g0 = blockIdx.x * groups_per_cta;
    const unsigned g1 = min(total, g0 + groups_per_cta);
    const size_t plane = (size_t)H * W;
    int bcur = -1;
    float r[9], c0 = 0.0f, c1 = 0.0f, c2 = 0.0f;
    const float *M = ref;
    for (unsigned g = g0; g < g1; ++g) {
        const int b = (int)(g / per_pair), i0 = (int)(g - (unsigned)b * per_pair) * ROWS;
        if (b != bcur) {   // uniform across the CTA
            const double *R = Rf + (size_t)b * 9;
#pragma unroll
            for (int k = 0; k < 9; ++k) r[k] = (float)__ldg(R + k);
            c0 = r[6] * zs;
            c1 = r[7] * zs;
            c2 = r[8] * zs;
            M = ref + (size_t)__ldg(ref_idx + b) * plane;
            bcur = b;
        }
        for (int j = threadIdx.x; j < W; j += blockDim.x) {
            float *o = out + (size_t)b * plane + (size_t)i0 * W + j;
            const float dx = (float)j + 0.5f - xpc;
#pragma unroll
            for (int u = 0; u < ROWS; ++u) {
                if (i0 + u >= H) break;
                const float dy = (float)(i0 + u) + 0.5f - ypc;
                // v = R^T r'
                const float v0 = fmaf(r[0], dx, fmaf(r[3], dy, c0));
                const float v1 = fmaf(r[1], dx, fmaf(r[4], dy, c1));
                const float v2 = fmaf(r[2], dx, fmaf(r[5], dy, c2));
                const float iv = zs / v2;
                const float x = fmaf(v0, iv, xpc - 0.5f), y = fmaf(v1, iv, ypc - 0.5f);
                const float fx0 = floorf(x), fy0 = floorf(y);
                const int x0 = (int)fx0, y0 = (int)fy0;
                float wx[4], wy[4];
                keys_weights(x - fx0, wx);
                keys_weights(y - fy0, wy);
                float acc = 0.0f;
                if ((unsigned)(x0 - 1) < (unsigned)(W - 3) && (unsigned)(y0 - 1) < (unsigned)(H - 3) && W > 3 && H > 3) {
                    const float *p0 = M + ((y0 - 1) * W + (x0 - 1)), *p1 = p0 + W, *p2 = p1 + W, *p3 = p2 + W;
                    const float *p[4] = {p0, p1, p2, p3};
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        float rr = 0.0f;
#pragma unroll
                        for (int k = 0; k < 4; ++k) rr = fmaf(wx[k], __ldg(p[m] + k), rr);
                        acc = fmaf(wy[m], rr, acc);
                    }
                } else {
                    int cx[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) cx[k] = min(max(x0 - 1 + k, 0), W - 1);
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        const float *rowp = M + min(max(y0 - 1 + m, 0), H - 1) * W;
                        float rr = 0.0f;
#pragma unroll
                        for (int k = 0; k < 4; ++k) rr = fmaf(wx[k], __ldg(rowp + cx[k]), rr);
                        acc = fmaf(wy[m], rr, acc);
                    }
                }
                o[u * W] = acc;
            }
        }
    }
}

}  // namespace

extern "C" int hrebsd_remap(hrebsd_ctx *ctx, const float *ref, const int32_t *ref_idx, const double *R_finite, int B,
                            int H, int W, const hrebsd_geometry *g, float *remapped, void *stream)
{
    if (!ctx || !g || B < 0 || H < 2 || W < 2) return HREBSD_EINVAL;
    if (B == 0) return HREBSD_OK;
    if (!ref || !ref_idx || !R_finite || !remapped) return HREBSD_EINVAL;
    int e = hr_set_device(ctx);
    if (e) return e;
    const long long rows = (long long)B * H;
    if (rows > 0x7fffffffLL || (long long)H * W > 0x7fffffffLL) return HREBSD_EINVAL;
    const int threads = W >= 256 ? 256 : (W + 31) / 32 * 32;
    const long long cap = (long long)ctx->num_sms * (2048 / threads);   // resident CTAs
    hr_prof_begin(ctx, hr_stream(stream));
    // rows of a thread: one where the rows fill at most half the chip (four are 4 units of a CTA's time in turn),
    // four while their groups are resident at once, and then what takes less in whole rounds (four rows take 3.4
    // times one row's time): 24 pairs of 240 x 320, 1.2 rounds of four rows, 18.7 us by single rows, 23.2 by fours
    const long long fours = (long long)B * ((H + 3) / 4);
    auto rounds = [&](long long n) { return (n + cap - 1) / cap; };
    const bool single = 2 * rows <= cap || (fours > cap && 10 * rounds(rows) < 34 * rounds(fours));
    const int group = single ? 1 : 4;
    const long long groups = (long long)B * ((H + group - 1) / group);
    const unsigned grid = (unsigned)(groups < cap ? groups : cap);
    const unsigned per = (unsigned)((groups + grid - 1) / grid);   // row groups of one CTA's run
    (group == 1 ? remap_kernel<1> : remap_kernel<4>)<<<grid, threads, 0, hr_stream(stream)>>>(
        ref, ref_idx, R_finite, B, H, W, (float)(g->xstar * W), (float)(g->ystar * H), (float)(g->zstar * W), per, remapped);
    hr_prof_end(ctx, PROF_REMAP, hr_stream(stream));
    HR_LAUNCHED(ctx);
    return HREBSD_OK;
}
