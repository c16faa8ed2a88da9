// Demons iteration as a row sweep over strips of columns and bands of rows (included by demons.cu), for level
// widths that the row sweep of whole rows does not cover: the same step as demons_strip.cuh (see there), on
// NT columns of which the outer ones are a halo, so that nothing depends on the width or on its alignment.
//
// An item is a strip of at most NT - 15 output columns and a band of rows of one active pair.  Thread t owns
// the image column xl + t of the strip's loaded columns; u is exact from 3 columns inside, du's x pass from 6.
// The three columns past an image edge stand for the edge column: their threads read its x-pass rows, so that
// they form the same u and du (the last strip's origin is shifted so that they lie in the edge column's
// warp; see demons_wide_columns.cuh).  A band starts 6 rows early (rows that are only pushed through the
// windows) unless it starts at the top, where the first row fills the windows.  The rows of a step are copied
// by cp.async, each thread its own column (8 and 4 bytes: no alignment needed), completion on an mbarrier.
//
// Every pixel gets the operations of the other shapes in their order: bit-identical fields.  The SSD partials
// are one per item; where a stop rule can act on them, d is stored as well and ssd_group_kernel forms the
// partials of the tile shape that runs otherwise, term by term.
//
// Bound like the row sweep by its warps' latency (four warps per scheduler, 128 registers a thread), with 12
// to 40 % of the columns and rows computed twice; the texture gathers of the moving image give 8 %
// (16 pairs of 1244 x 1024 in two bands: an iteration 252 us with plain loads, 233 us with gathers; three
// bands, which fill the chip, 194 us).  Microseconds of an
// iteration, tiles -> sweep, and with the stop rule's regrouped SSD: 2,000 pairs of 200 x 200 1,386 -> 751
// (975); 16 of 1244 x 1024 209 -> 194 (251, not taken); 16 of 622 x 512 97 -> 56 (76); 152 of 311 x 300
// 255 -> 140 (189); 600 of 100 x 92 87 -> 61 (78).  For few pairs the bands' extra rows and the latency of a
// step outweigh it (one pair of 640 x 480 10 -> 17).
namespace wide {

constexpr int R = 7, RAD = 3;

#include "demons_wide_columns.cuh"

template <int NT>
struct Geo {
    static constexpr int HO = 4, HST = NT + 10, XST = NT + 10, FR_ = R + 2, FST = NT;   // as the row sweep
    static constexpr size_t S_OFF = 0;
    static constexpr size_t F_OFF = S_OFF + (size_t)2 * R * HST * 8;
    static constexpr size_t D_OFF = F_OFF + (size_t)2 * FR_ * FST * 4;
    static constexpr size_t X_OFF = D_OFF + (size_t)2 * R * HST * 8;
    static constexpr size_t Y_OFF = X_OFF + (size_t)R * XST * 8;
    static constexpr size_t BYTES = Y_OFF + (size_t)R * XST * 8;
    static_assert((HST / 2) % 8 == 5 && S_OFF % 16 == 0 && F_OFF % 16 == 0 && D_OFF % 16 == 0 && X_OFF % 16 == 0 && Y_OFF % 16 == 0,
                  "the x-pass lane map and 16-byte regions");
};

struct WideArgs {
    int strips, sw, bands, bh;   // strips of sw columns, bands of bh rows (bh >= 7 when there are several)
    float *dbuf;                 // [B][h][w] d (null unless the SSD is regrouped)
};

__device__ __forceinline__ void cp_async8(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(hr_tma::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(hr_tma::smem_u32(dst)), "l"(src) : "memory");
}
// Arrive on the barrier when this thread's copies so far have landed.
__device__ __forceinline__ void cp_async_arrive(uint64_t *bar)
{
    asm volatile("cp.async.mbarrier.arrive.noinc.shared.b64 [%0];" ::"r"(hr_tma::smem_u32(bar)) : "memory");
}

template <int NT, bool IN_S, bool TEX>
__global__ void __launch_bounds__(NT, 512 / NT) demons_wide_kernel(IterArgs a, WideArgs wa)
{
    using G = Geo<NT>;
    extern __shared__ __align__(16) unsigned char smraw[];
    float2 *sS0 = reinterpret_cast<float2 *>(smraw + G::S_OFF);
    float *sF0 = reinterpret_cast<float *>(smraw + G::F_OFF);
    float2 *sD0 = reinterpret_cast<float2 *>(smraw + G::D_OFF);
    float2 *sRX = reinterpret_cast<float2 *>(smraw + G::X_OFF);
    float2 *sDX = reinterpret_cast<float2 *>(smraw + G::Y_OFF);
    __shared__ float red[NT / 32];
    __shared__ __align__(8) uint64_t bar[2], dbar;
    const int t = threadIdx.x, lane = t & 31, warp = __shfl_sync(0xffffffffu, t >> 5, 0);
    constexpr int NWARP = NT / 32;
    float2 tf[2 * RAD + 1], tu[2 * RAD + 1];   // (symmetric: half of them in registers)
#pragma unroll
    for (int k = 0; k <= 2 * RAD; ++k) {
        const int j = k <= RAD ? k : 2 * RAD - k;
        tf[k] = make_float2(a.taps.f[j], a.taps.f[j]);
        tu[k] = make_float2(a.taps.up[j], a.taps.up[j]);
    }
    const int n_active = *a.n_active;
    if (blockIdx.x == 0 && t == 0) {
        *a.n_next_reset = 0;
        if (a.px_count) atomicAdd(a.px_count, (unsigned long long)n_active * a.h * a.w);
    }
    if (t == 0) {
        hr_tma::mbar_init(&bar[0], NT);
        hr_tma::mbar_init(&bar[1], NT);
        hr_tma::mbar_init(&dbar, NWARP);
        hr_tma::fence_mbar_init();
    }
    __syncthreads();
    const int h = a.h, w = a.w, per = wa.strips * wa.bands;
    const size_t plane = (size_t)h * w;
    const long long work = (long long)n_active * per;
    const float mx2 = (float)(w - 2), my2 = (float)(h - 2), wf = (float)w, al2 = a.alpha2;
    // the x-pass lane map of the row sweep
    const int xp = lane >> 3, xq_ = lane & 7;
    const bool xlane = xq_ != 7;
    const int xi = xp < 2 ? (xq_ < 6 ? xq_ >> 1 : 3) : (xq_ == 0 ? 3 : 4 + ((xq_ - 1) >> 1));
    const int xs = xp < 2 ? (xq_ < 6 ? (xq_ & 1) + 2 * xp : xp) : (xq_ == 0 ? xp : ((xq_ - 1) & 1) + 2 * (xp - 2));
    const int xc0 = (4 * warp + xs) * RUN;

    struct Item {
        int pair, x0, x1, xl, yb, ye, ys, nsteps;   // columns [x0, x1), first loaded column, rows [yb, ye), first row, steps
    };
    auto item_of = [&](long long i) {
        Item m;
        const int slot = (int)(i / per), r = (int)(i - (long long)slot * per), s = r / wa.bands, b = r - s * wa.bands;
        m.pair = a.active[slot];
        m.x0 = s * wa.sw;
        m.x1 = min(w, m.x0 + wa.sw);
        m.xl = strip_origin(m.x0, m.x1, w);
        m.yb = b * wa.bh;
        m.ye = min(h, m.yb + wa.bh);
        m.ys = m.yb > 0 ? m.yb - 2 * RAD : 0;
        m.nsteps = (m.ye + 2 * RAD - m.ys + R - 1) / R;
        return m;
    };
    // the copies of step k of an item into buffer gg & 1, this thread's column
    auto issue = [&](const Item &m, int k, uint32_t gg) {
        const int b = gg & 1, x = clampi(m.xl + t, 0, w - 1), y0 = m.ys + R * k;
        const float *fp = a.Ftest + (size_t)m.pair * plane + x;
        float *fd = sF0 + b * G::FR_ * G::FST + t;
        float2 *sd = sS0 + b * R * G::HST + G::HO + t;
        if (y0 - RAD - 1 >= 0 && y0 + R <= h) {
            if (IN_S) {
                const float2 *sp = a.in + (size_t)m.pair * plane + (size_t)y0 * w + x;
#pragma unroll
                for (int i = 0; i < R; ++i, sp += w) cp_async8(sd + i * G::HST, sp);
            }
            fp += (size_t)(y0 - RAD - 1) * w;
#pragma unroll
            for (int i = 0; i < G::FR_; ++i, fp += w) cp_async4(fd + i * G::FST, fp);
        } else {
            if (IN_S)
                for (int i = 0; i < R; ++i)
                    cp_async8(sd + i * G::HST, a.in + (size_t)m.pair * plane + (size_t)clampi(y0 + i, 0, h - 1) * w + x);
            for (int i = 0; i < G::FR_; ++i)
                cp_async4(fd + i * G::FST, fp + (size_t)clampi(y0 - RAD - 1 + i, 0, h - 1) * w);
        }
        cp_async_arrive(&bar[b]);
    };
    // step gg's rows: wait for the copies (bounded), x pass of G_f on the warp's own columns
    auto stage = [&](uint32_t gg) {
        const bool ok = hr_tma::mbar_wait(&bar[gg & 1], (gg >> 1) & 1u);
        if (IN_S) {
            float2 *sS = sS0 + (gg & 1) * R * G::HST;
            if (xlane) strip::run_x_halo<RAD>(sS + xi * G::HST, xc0, sRX + xi * G::XST + xc0, tf);
            __syncwarp();
        }
        return ok;
    };

    long long item = blockIdx.x;
    if (item >= work) return;
    uint32_t g = 0;
    bool primed = false;
    Item m = item_of(item);
    issue(m, 0, 0);
    issue(m, 1, 1);   // (every item has at least two steps)
    for (;;) {
        const bool has_next = item + gridDim.x < work;
        const Item nm = has_next ? item_of(item + gridDim.x) : m;
        const int ref = __ldg(a.ref_idx + m.pair);
        const float *M = a.Mref + (size_t)ref * plane;
        const float yt = (float)(ref * h) + 1.0f;   // TEX: as the row sweep
        const float2 *u0 = a.in + (size_t)m.pair * plane;
        float2 *dst = a.out + (size_t)m.pair * plane;
        const int x = m.xl + t, xq = clampi(x, 0, w - 1);
        const int tc = edge_column(m.xl, t, w);   // this thread's column of the rows
        const int tl = clampi(clampi(xq - 1, 0, w - 1) - m.xl, 0, NT - 1), tr = clampi(clampi(xq + 1, 0, w - 1) - m.xl, 0, NT - 1);
        const float tf_ = (float)xq, sx = (xq == 0 || xq == w - 1) ? 1.0f : 0.5f;
        const bool col = x >= m.x0 && x < m.x1;   // an output column
        const int ub = m.yb > 0 ? m.yb - RAD : 0;   // first du row
        // a step whose du rows are all inside, none at an image edge, from ub on, and whose outputs lie in the band
        auto interior_step = [&](int k) {
            const int y = m.ys + R * k;
            return y - RAD >= max(ub, 1) && y + RAD <= h - 2 && y - 2 * RAD >= m.yb && y < m.ye;
        };
        float2 rxw[R], dxw[R], ucur[R], uprev[RAD], last_dx = make_float2(0.0f, 0.0f);
        float ssd = 0.0f;
        bool ok = true;
        if (!primed) ok = stage(g);
        for (int k = 0; k < m.nsteps; ++k) {
            const int b = g & 1, yk0 = m.ys + R * k;
            float *sF = sF0 + b * G::FR_ * G::FST;
            float2 *sD = sD0 + b * R * G::HST;
            const float yk = (float)(yk0 - RAD);
            auto force_rows = [&](auto interior) {
                constexpr bool IN = decltype(interior)::value;
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const int y = yk0 + i, yu = y - RAD;
                    float2 u;
                    if (IN_S) {
                        const float2 v = sRX[i * G::XST + tc];
                        rxw[i] = v;
                        if (!IN && y == 0) {
#pragma unroll
                            for (int j = 0; j < R; ++j) rxw[j] = v;
                        }
                        u = __fmul2_rn(tf[0], rxw[(i + R - 2 * RAD) % R]);
#pragma unroll
                        for (int j = 1; j < R; ++j) u = ffma2(tf[j], rxw[(i + R - 2 * RAD + j) % R], u);
                    } else {
                        u = (IN || (yu >= 0 && yu < h)) ? u0[(size_t)yu * w + xq] : make_float2(0.0f, 0.0f);
                    }
                    ucur[i] = u;
                }
                float4 mv[R];
                float fxv[R], fyv[R];
                float2 q = make_float2(tf_, yk);
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    if (!IN) q.y = (float)clampi(yk0 + i - RAD, 0, h - 1);
                    float2 c, f;
                    warp_cell2(q, ucur[i], make_float2(mx2, my2), c, f);
                    if (IN) q = __fadd2_rn(q, make_float2(0.0f, 1.0f));
                    fxv[i] = f.x;
                    fyv[i] = f.y;
                    if constexpr (TEX) {
                        const float2 tg = __fadd2_rn(c, make_float2(1.0f, yt));
                        mv[i] = tex2Dgather<float4>(a.mtex, tg.x, tg.y, 0);
                    } else {   // (levels below 2^24 pixels)
                        const float *p = M + (int)fmaf(c.y, wf, c.x);
                        const float *p2 = p + w;
                        mv[i] = make_float4(__ldg(p2), __ldg(p2 + 1), __ldg(p + 1), __ldg(p));
                    }
                }
                auto put = [&](int i, int yu, float tt, float gx, float gy, float d) {
                    sD[i * G::HST + G::HO + t] = make_float2(tt * gx, tt * gy);
                    if (col && (IN || yu >= m.yb) && yu < m.ye) {
                        ssd = fmaf(d, d, ssd);
                        if (wa.dbuf) wa.dbuf[(size_t)m.pair * plane + (size_t)yu * w + x] = d;
                    }
                };
                float fa = sF[tc], fb = sF[G::FST + tc];
                if (IN) {
                    const float2 n1 = make_float2(-1.0f, -1.0f), one = make_float2(1.0f, 1.0f), a2 = make_float2(al2, al2);
#pragma unroll
                    for (int i = 0; i + 1 < R; i += 2) {   // row pairs in packed arithmetic, as the row sweep
                        const float *fr_ = sF + (i + 1) * G::FST;
                        const float f2 = fr_[G::FST + tc], f3 = fr_[2 * G::FST + tc];
                        const float2 fl = make_float2(fr_[tl], fr_[G::FST + tl]), frt = make_float2(fr_[tr], fr_[G::FST + tr]);
                        const float2 fx = make_float2(fxv[i], fxv[i + 1]), fy = make_float2(fyv[i], fyv[i + 1]);
                        const float2 omx = __ffma2_rn(fx, n1, one), omy = __ffma2_rn(fy, n1, one);
                        const float2 top = make_float2(fmaf(fx.x, mv[i].z, omx.x * mv[i].w), fmaf(fx.y, mv[i + 1].z, omx.y * mv[i + 1].w));
                        const float2 bot = make_float2(fmaf(fx.x, mv[i].y, omx.x * mv[i].x), fmaf(fx.y, mv[i + 1].y, omx.y * mv[i + 1].x));
                        const float2 mw = __ffma2_rn(fy, bot, __fmul2_rn(omy, top));
                        const float2 gx = __fmul2_rn(make_float2(sx, sx), __ffma2_rn(fl, n1, frt));
                        const float2 gy = __fmul2_rn(make_float2(0.5f, 0.5f), __ffma2_rn(make_float2(fa, fb), n1, make_float2(f2, f3)));
                        const float2 d = make_float2(fmaf(fb, -1.0f, mw.x), fmaf(f2, -1.0f, mw.y));
                        const float2 den = __ffma2_rn(gx, gx, __ffma2_rn(gy, gy, __fmul2_rn(__fmul2_rn(a2, d), d)));
                        put(i, yk0 + i - RAD, force_quot(d.x, den.x), gx.x, gy.x, d.x);
                        put(i + 1, yk0 + i + 1 - RAD, force_quot(d.y, den.y), gx.y, gy.y, d.y);
                        fa = f2;
                        fb = f3;
                    }
                }
#pragma unroll
                for (int i = IN ? R - 1 : 0; i < R; ++i) {
                    const int yu = yk0 + i - RAD;
                    const float *fr_ = sF + (i + 1) * G::FST;
                    const float fn = fr_[G::FST + tc];
                    if (IN || (yu >= ub && yu < h)) {
                        const float fl = fr_[tl], frt = fr_[tr], sy = (!IN && (yu == 0 || yu == h - 1)) ? 1.0f : 0.5f;
                        const float fx = fxv[i], fy = fyv[i];
                        const float omx = fmaf(fx, -1.0f, 1.0f), omy = fmaf(fy, -1.0f, 1.0f);
                        const float top = fmaf(fx, mv[i].z, omx * mv[i].w), bot = fmaf(fx, mv[i].y, omx * mv[i].x);
                        const float mw = fmaf(fy, bot, omy * top);
                        const float gx = sx * fmaf(fl, -1.0f, frt), gy = sy * fmaf(fa, -1.0f, fn);
                        const float d = fmaf(fb, -1.0f, mw);
                        put(i, yu, force_quot(d, fmaf(gx, gx, fmaf(gy, gy, (al2 * d) * d))), gx, gy, d);
                    }
                    fa = fb;
                    fb = fn;
                }
            };
            if (interior_step(k)) force_rows(std::true_type());
            else force_rows(std::false_type());
            __syncwarp();
            if (lane == 0) hr_tma::mbar_arrive(&dbar);
            const bool more = k + 1 < m.nsteps || has_next;
            if (more) ok = stage(g + 1) && ok;
            ok = hr_tma::mbar_wait(&dbar, g & 1u) && ok;
            if (!__all_sync(0xffffffffu, ok)) {   // a wait gave up: report, let this thread's copies land, stop
                if (t == 0) atomicExch(a.err, 1);
                asm volatile("cp.async.wait_all;" ::: "memory");
                return;
            }
            if (k + 2 < m.nsteps) issue(m, k + 2, g);
            else if (has_next) issue(nm, k + 2 - m.nsteps, g);
            // x pass of G_u on the du rows that exist
            if (xlane) {
                const int yu = yk0 + xi - RAD;
                if (yu >= ub && yu < h) strip::run_x_halo<RAD>(sD + xi * G::HST, xc0, sDX + xi * G::XST + xc0, tu);
            }
            __syncwarp();
            auto outputs = [&](auto interior) {
                constexpr bool IN = decltype(interior)::value;
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const int yu = yk0 + i - RAD, yo = yu - RAD;
                    if (IN || yu >= ub) {
                        const float2 v = (IN || yu < h) ? sDX[i * G::XST + t] : last_dx;
                        if (!IN && yu < h) last_dx = v;
                        dxw[(i + R - RAD) % R] = v;
                        if (!IN && yu == 0) {
#pragma unroll
                            for (int j = 0; j < R; ++j) dxw[j] = v;
                        }
                    }
                    if (IN || (yo >= m.yb && yo < m.ye)) {
                        float2 acc = __fmul2_rn(tu[0], dxw[(i + 2 * R - 3 * RAD) % R]);
#pragma unroll
                        for (int j = 1; j < R; ++j) acc = ffma2(tu[j], dxw[(i + 2 * R - 3 * RAD + j) % R], acc);
                        const float2 uo = i >= RAD ? ucur[i - RAD] : uprev[i];
                        if (col) dst[(size_t)yo * w + x] = __fadd2_rn(uo, acc);
                    }
                }
            };
            if (interior_step(k)) outputs(std::true_type());
            else outputs(std::false_type());
#pragma unroll
            for (int i = 0; i < RAD; ++i) uprev[i] = ucur[R - RAD + i];
            ++g;
        }
        // SSD of the item
        for (int o = 16; o > 0; o >>= 1) ssd += __shfl_xor_sync(0xffffffffu, ssd, o);
        if (lane == 0) red[warp] = ssd;
        __syncthreads();
        if (t == 0 && !wa.dbuf) {
            float s = 0.0f;
            for (int j = 0; j < NWARP; ++j) s += red[j];
            a.part[(size_t)m.pair * per + (int)(item % per)] = s;
        }
        if (!has_next) return;
        primed = true;
        item += gridDim.x;
        m = nm;
    }
}

// The SSD partials of tiles tx x ty as their kernel sums them (plain: the plain-load tiles, two points at a
// time; else the TMA-fed tiles, vertical runs of 4) from the stored d: a CTA of nt threads per (active pair,
// tile), each thread the terms of that kernel's thread.
__global__ void ssd_group_kernel(IterArgs a, const float *__restrict__ dbuf, int tx, int ty, int plain)
{
    __shared__ float red[32];
    const int nt = blockDim.x, t = threadIdx.x, lane = t & 31, warp = t >> 5, h = a.h, w = a.w;
    const int BW = tx + 2 * RAD;
    const long long work = (long long)*a.n_active * a.tiles;
    for (long long item = blockIdx.x; item < work; item += gridDim.x) {
        const int pair = a.active[item / a.tiles], tile = (int)(item % a.tiles);
        const int x0 = (tile % a.tiles_x) * tx, y0 = (tile / a.tiles_x) * ty;
        const float *D = dbuf + (size_t)pair * h * w;
        float s = 0.0f;
        // every term's load first (12 for each of these shapes), then the sum in order
        float d[12];
        if (plain) {   // 256 threads, 64 x 32: six pairs of points
#pragma unroll
            for (int k = 0; k < 12; ++k) {
                const int i = t + k * nt, r = i / BW - RAD, c = i % BW - RAD;
                d[k] = (unsigned)r < (unsigned)min(ty, h - y0) && (unsigned)c < (unsigned)min(tx, w - x0)
                           ? __ldg(D + (size_t)(y0 + r) * w + x0 + c) : 0.0f;
            }
#pragma unroll
            for (int k = 0; k < 12; k += 2) s = __fadd_rn(s, __fadd_rn(__fmul_rn(d[k], d[k]), __fmul_rn(d[k + 1], d[k + 1])));
        } else {   // at most three runs of 4 rows a thread
            const int rows_in = min(ty, h - y0);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int it = t + k * nt, g = it / BW, c = it - g * BW, vx = x0 - RAD + c;
                const bool in = c >= RAD && c < RAD + tx && vx < w;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = 4 * g + i - RAD;
                    d[4 * k + i] = in && (unsigned)r < (unsigned)rows_in ? __ldg(D + (size_t)(y0 + r) * w + vx) : 0.0f;
                }
            }
#pragma unroll
            for (int k = 0; k < 12; ++k) s = fmaf(d[k], d[k], s);
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) red[warp] = s;
        __syncthreads();
        if (t == 0) {
            float p = 0.0f;
            for (int i = 0; i < nt / 32; ++i) p += red[i];
            a.part[(size_t)pair * a.tiles + tile] = p;
        }
        __syncthreads();
    }
}

}  // namespace wide
