// Demons level resident in the shared memory of a thread-block cluster (included by demons.cu): the rows
// of a pair are cut into equal bands, one per CTA of the cluster, and the whole level -- every iteration,
// the stop rule and the final field -- runs in one launch without touching HBM in between.  For few pairs
// (one pair's latency is then the time, and a launch per iteration or one CTA per pair leave most of the
// chip idle) and for level sizes that the row sweep does not cover.
//
// Each output pixel gets the same operations in the same order as in the other shapes, so the field is
// bit-identical to theirs.  Per iteration k and CTA:
//   x pass of G_f on the band's s rows -> X (k > 0); the three rows at either end of the band are also
//     stored into the neighbouring CTAs' halo rows (distributed shared memory);
//   cluster barrier;
//   per column in vertical runs of 4 rows: y pass of G_f -> u, the moving image at x - u, the force of
//     Eq. 1 -> du;
//   CTA barrier; x pass of G_u -> Y, halo rows stored as above; cluster barrier;
//   y pass of G_u, plus u -> s_{k+1}; CTA barrier.
// So an iteration costs two cluster barriers whatever its size (3 to 4 us with the latencies between
// them); the rest is bound by instruction issue like the row sweep.  Levels of 20 iterations: one pair of
// 128 x 128 88 us (row sweep 682), of 256 x 256 158 us (1,407), 150 pairs of 92 x 100 334 us (64 x 32 tiles
// and a control launch per iteration 670), 458 us with the stop rule (686).
//
// The SSD of the stop rule.  Without a stop rule the SSD only tells whether the field stayed finite, and
// each CTA sums its own pixels.  With one, an SSD that differs in the last FP32 bit can end a level an
// iteration earlier or later, so the tiles' sums are formed exactly as the shape that would run otherwise
// forms them (`group`): d is kept in shared memory, and warps of the cluster stand in for the warps of that
// shape's tiles, adding the same pixels in the same order with the same warp tree.  The tiles are added in
// FP64, by 32 lanes and a tree where the control kernel takes fewer lanes: the sum of up to 1,024 FP32 values is
// exact in FP64, so the same in any order, unless they differ by more than a factor of 2^19.
namespace clu {

constexpr int NT = 512, RAD = 3, VR = 4, MAXC = 16, MAX_TASKS = 1024;

// Whose grouping the SSD follows: G_FREE any; G_TILE the TMA-fed tiles (tx x ty, nt threads); G_PLAIN the
// plain-load tiles (64 x 32, 256 threads); G_STRIP the row sweep; G_LEVEL the level in one CTA.
enum Group { G_FREE = 0, G_TILE, G_PLAIN, G_STRIP, G_LEVEL };

struct ClusterArgs {
    const float *Ftest;          // [B][h][w] test images of the level
    const float *Mref;           // [R][h][w] reference images of the level
    const int *ref_idx;          // [B]
    const float2 *u0;            // [B][h][w] the level's initial field
    float *uout;                 // final field: planar [B][2][h][w] (planar) or [B][h][w] float2
    double *hist;                // [B][hist_stride]
    int32_t *iters;              // [B][levels]
    int32_t *status;             // [B]
    unsigned long long *px_count;   // tracing: pixel-iterations (NULL = off)
    int B, h, w, hist_stride, cap, window, level, levels, planar;
    int C, hb, st;               // CTAs per cluster, rows per band, row stride of A, X, Y (float2)
    int group, tx, ty, nt, tiles_x, tiles, tasks;   // the SSD's grouping
    unsigned mw, mhb, mbw;       // ceil(2^32 / n) for n = w, hb and a tile's columns tx + 2 r
    float tol, alpha2;
    Taps taps;
};

// Row stride of the x passes' buffers: 4 columns of halo on either side of the row rounded up to whole runs
// (16-byte accesses), an odd number of 16-byte slots (lanes on consecutive rows hit distinct banks).
__host__ __device__ constexpr int HO = 4;
__host__ __device__ constexpr int row_stride(int w)
{
    const int n = round_up(w, RUN) + 2 * HO;
    return n % 4 == 2 ? n : n + 2;
}
// Shared memory of a CTA: A (s / du), X and Y (x-pass rows of G_f and of G_u, with 3 halo rows on either
// side), U (u), the test image's rows (with one on either side; a run of VR rows may read past the band),
// and d where the SSD is regrouped.
__host__ __device__ constexpr size_t bytes(int hb, int w, bool keep_d)
{
    return (size_t)row_stride(w) * 8 * (3 * hb + 12) + (size_t)w * 8 * hb + (size_t)w * 4 * (hb + 2 + VR) +
           (keep_d ? (size_t)w * 4 * hb : 0);
}

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Shared-memory address `p` of this CTA in the CTA of rank `r`.
__device__ __forceinline__ uint32_t remote(const void *p, unsigned r)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(hr_tma::smem_u32(p)), "r"(r));
    return a;
}
__device__ __forceinline__ void st_remote(uint32_t a, float4 v)
{
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}
__device__ __forceinline__ void st_remote(uint32_t a, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ float ld_remote(uint32_t a)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ int div_by(int n, unsigned magic) { return (int)__umulhi((unsigned)n, magic); }   // n, divisor < 2^16

__global__ void __launch_bounds__(NT, 1) demons_cluster_kernel(const __grid_constant__ ClusterArgs a)
{
    extern __shared__ __align__(16) unsigned char clu_smem[];
    const int h = a.h, w = a.w, hb = a.hb, st = a.st, C = a.C;
    const unsigned rank = C > 1 ? cluster_rank() : 0u;
    const int lo = (int)rank * hb, hi = min(h, lo + hb), rows = hi - lo;
    float2 *A = reinterpret_cast<float2 *>(clu_smem);   // [hb] s_k, then du; column x at HO + x, replicated halo columns
    float2 *X = A + (size_t)hb * st;                     // [hb + 6] row y at y - lo + 3
    float2 *Y = X + (size_t)(hb + 6) * st;               // [hb + 6]
    float2 *U = Y + (size_t)(hb + 6) * st;               // [hb][w] u_k
    float *F = reinterpret_cast<float *>(U + (size_t)hb * w);   // [hb + 2 + VR][w] row y at y - lo + 1
    float *D = F + (size_t)(hb + 2 + VR) * w;            // [hb][w] d (regrouped SSD)
    __shared__ float red[NT / 32], esum[MAXC], wsum[MAX_TASKS];
    __shared__ int s_state;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const unsigned mrows = rows > 1 ? (unsigned)(((1ull << 32) + rows - 1) / rows) : 0u;
    const int ymax = min(h - 1, hi + RAD - 1);   // last row that X and Y hold
    const float al2 = a.alpha2, mx2 = (float)(w - 2), my2 = (float)(h - 2);
    const size_t plane = (size_t)h * w;
    const bool regroup = a.group != G_FREE;
    enum { CONTINUE = 0, STOP = 1, CAPPED = 2 };
    auto sync_all = [&]() {
        if (C > 1) cluster_sync();
        else __syncthreads();
    };

    // row y of A, column x: the first and last column fill the halo columns with their value
    auto put_A = [&](int y, int x, float2 v) {
        float2 *p = A + y * st + HO + x;
        *p = v;
        if (x == 0) p[-1] = p[-2] = p[-3] = v;
        if (x == w - 1) p[1] = p[2] = p[3] = v;
    };
    // x pass of the band's rows of A into the rows of out, and into the neighbours' halo rows
    auto xpass = [&](float2 *out, const float *taps) {
        const int nseg = (w + RUN - 1) / RUN;
        const uint32_t up = rank > 0 ? remote(out, rank - 1) : 0u;
        const uint32_t down = (int)rank + 1 < C ? remote(out, rank + 1) : 0u;
        float2 tp[2 * RAD + 1];
#pragma unroll
        for (int k = 0; k <= 2 * RAD; ++k) tp[k] = make_float2(taps[k], taps[k]);
        for (int j = t; j < rows * nseg; j += NT) {
            const int seg = rows > 1 ? div_by(j, mrows) : j, y = j - seg * rows, x0 = seg * RUN;   // y: row of the band
            float2 *row = out + (y + RAD) * st + x0;
            strip::run_x_halo<RAD>(A + y * st, x0, row, tp);   // (columns past w: unused)
            const bool to_up = y < RAD && up, to_down = y >= rows - RAD && down;
            // the neighbour above holds row lo + y at its row hb + 3 + y, the one below at y - rows + 3
            if (to_up || to_down) {
                const uint32_t pu = up + (uint32_t)((hb + RAD + y) * st + x0) * 8u;
                const uint32_t pd = down + (uint32_t)((y - rows + RAD) * st + x0) * 8u;
#pragma unroll
                for (int o = 0; o < RUN; o += 2) {
                    const float4 v = *reinterpret_cast<const float4 *>(row + o);
                    if (to_up) st_remote(pu + 8u * o, v);
                    if (to_down) st_remote(pd + 8u * o, v);
                }
            }
        }
    };
    // y pass of a run of VR rows of column x starting at the image row y0
    auto ypass = [&](const float2 *in, const float *taps, int y0, int x, float2 (&acc)[VR]) {
        float2 win[VR + 2 * RAD];
#pragma unroll
        for (int q = 0; q < VR + 2 * RAD; ++q) win[q] = in[(clampi(y0 - RAD + q, 0, ymax) - lo + RAD) * st + x];
#pragma unroll
        for (int o = 0; o < VR; ++o) acc[o] = __fmul2_rn(make_float2(taps[0], taps[0]), win[o]);
#pragma unroll
        for (int k = 1; k <= 2 * RAD; ++k)
#pragma unroll
            for (int o = 0; o < VR; ++o) acc[o] = ffma2(make_float2(taps[k], taps[k]), win[o + k], acc[o]);
    };
    const int nitems = (rows + VR - 1) / VR * w;
    // d at an image position, wherever its band lies
    auto read_d = [&](int y, int x) {
        const int r = C > 1 ? div_by(y, a.mhb) : 0;
        const float *p = D + (y - r * hb) * w + x;
        return r == (int)rank ? *p : ld_remote(remote(p, r));
    };
    // the share of `lane` of virtual warp `vw` of tile `tile`, as the shape named by a.group sums it (the
    // loads of several terms in flight, the sums in that shape's order)
    auto lane_sum = [&](int tile, int vw) {
        const int vt = vw * 32 + lane;
        const int ty_ = tile / a.tiles_x, x0 = (tile - ty_ * a.tiles_x) * a.tx, y0 = ty_ * a.ty;
        float s = 0.0f;
        if (a.group == G_STRIP) {
            int y = 0;
            for (; y + 8 <= h; y += 8) {
                float d[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) d[i] = read_d(y + i, vt);
#pragma unroll
                for (int i = 0; i < 8; ++i) s = fmaf(d[i], d[i], s);
            }
            for (; y < h; ++y) {
                const float d = read_d(y, vt);
                s = fmaf(d, d, s);
            }
        } else if (a.group == G_LEVEL) {
            for (int p = vt; p < h * w; p += a.nt) {
                const int y = div_by(p, a.mw);
                const float d = read_d(y, p - y * w);
                s = fmaf(d, d, s);
            }
        } else if (a.group == G_TILE) {
            const int BW = a.tx + 2 * RAD, NG = (a.ty + 2 * RAD + 3) / 4, rows_in = min(a.ty, h - y0);
            for (int it = vt; it < NG * BW; it += a.nt) {
                const int g = div_by(it, a.mbw), c = it - g * BW, vx = x0 - RAD + c;
                if (c < RAD || c >= RAD + a.tx || vx >= w) continue;
                float d[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = 4 * g + i - RAD;   // row of the tile
                    d[i] = (unsigned)r < (unsigned)rows_in ? read_d(y0 + r, vx) : 0.0f;   // (+ 0 * 0: no change)
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) s = fmaf(d[i], d[i], s);
            }
        } else {   // G_PLAIN: two points at a time
            const int BW = a.tx + 2 * RAD, npts = BW * (a.ty + 2 * RAD);
            auto point = [&](int i) {
                const int rr = div_by(i, a.mbw), r = rr - RAD, c = i - rr * BW - RAD;
                if (i >= npts || (unsigned)r >= (unsigned)a.ty || (unsigned)c >= (unsigned)a.tx || y0 + r >= h || x0 + c >= w)
                    return 0.0f;
                return read_d(y0 + r, x0 + c);
            };
            for (int i0 = vt; i0 < npts; i0 += 4 * a.nt) {
                const float d0 = point(i0), d1 = point(i0 + a.nt), d2 = point(i0 + 2 * a.nt), d3 = point(i0 + 3 * a.nt);
                s = __fadd_rn(s, __fadd_rn(__fmul_rn(d0, d0), __fmul_rn(d1, d1)));
                s = __fadd_rn(s, __fadd_rn(__fmul_rn(d2, d2), __fmul_rn(d3, d3)));   // (past the end: + 0)
            }
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        return s;
    };

    const int nclusters = (int)gridDim.x / C;
    for (int pair = (int)blockIdx.x / C; pair < a.B; pair += nclusters) {
        const float *Fg = a.Ftest + (size_t)pair * plane;
        const float2 *ug = a.u0 + (size_t)pair * plane;
        const float *M = a.Mref + (size_t)__ldg(a.ref_idx + pair) * plane;
        double *hh = a.hist + (size_t)pair * a.hist_stride;
        // the stop rule of the control kernel after iteration k (one thread; every CTA computes the same)
        auto decide = [&](int k, double E) {
            int next = CONTINUE;
            int it = 0;
            bool bad = false;
            if (rank == 0 || a.window > 0) {
                if (!isfinite(E)) {
                    next = STOP;
                    it = k;
                    bad = true;
                } else if (a.window > 0 && k >= a.window && (hh[k - a.window] - E) < (double)a.tol * hh[k - a.window]) {
                    next = STOP;
                    it = k;
                } else if (k + 1 >= a.cap) {
                    next = CAPPED;
                    it = a.cap;
                }
            } else {
                next = !isfinite(E) ? STOP : k + 1 >= a.cap ? CAPPED : CONTINUE;
            }
            hh[k] = E;   // (the same value from every CTA of the cluster)
            if (rank == 0) {
                if (next != CONTINUE) {
                    a.iters[(size_t)pair * a.levels + a.level] = it;
                    if (bad) a.status[pair] |= HREBSD_PAIR_NONFINITE;
                    else if (next == CAPPED) a.status[pair] |= HREBSD_PAIR_CAPPED;
                }
                if (a.px_count) atomicAdd(a.px_count, (unsigned long long)plane);
            }
            s_state = next;
        };
        for (int p = t; p < rows * w; p += NT) {
            const int y = div_by(p, a.mw), x = p - y * w;
            U[p] = ug[(size_t)(lo + y) * w + x];
        }
        for (int p = t; p < (rows + 2) * w; p += NT) {
            const int y = div_by(p, a.mw), x = p - y * w;
            F[p] = Fg[(size_t)clampi(lo + y - 1, 0, h - 1) * w + x];
        }
        if (t == 0) s_state = CONTINUE;
        // the whole cluster, not only this CTA: iteration 0 stores into the neighbours' shared memory without
        // a barrier in between, which is defined only once every CTA of the cluster runs
        sync_all();
        for (int k = 0;; ++k) {
            bool final_pass = false;
            if (k > 0) {
                xpass(X, a.taps.f);
                sync_all();
                if (regroup) {   // the tiles' sums are complete: the stop rule after iteration k - 1
                    if (warp == 0) {
                        double E = 0.0;
                        const int nvw = a.nt / 32;
                        for (int i = lane; i < a.tiles; i += 32) {
                            float s = 0.0f;
                            for (int j = 0; j < nvw; ++j) s += wsum[i * nvw + j];
                            E += (double)s;
                        }
                        for (int o = 16; o > 0; o >>= 1) E += __shfl_xor_sync(0xffffffffu, E, o);
                        if (lane == 0) decide(k - 1, E);
                    }
                    __syncthreads();
                }
                if (s_state == STOP) break;   // the final field is u_{k-1}, in U
                final_pass = s_state == CAPPED;   // ... or G_f * s_cap
            }
            // ---- y pass of G_f, the force of Eq. 1
            float ssd = 0.0f;
            for (int j = t; j < nitems; j += NT) {
                const int g = div_by(j, a.mw), x = j - g * w, yl = VR * g, y0 = lo + yl;
                float2 u[VR];
                if (k > 0) {
                    ypass(X, a.taps.f, y0, x, u);
#pragma unroll
                    for (int i = 0; i < VR; ++i)
                        if (yl + i < rows) U[(yl + i) * w + x] = u[i];
                    if (final_pass) continue;
                } else {
#pragma unroll
                    for (int i = 0; i < VR; ++i) u[i] = U[min(yl + i, rows - 1) * w + x];
                }
                float4 m[VR];
                float2 f[VR];
                float2 q = make_float2((float)x, (float)y0);
#pragma unroll
                for (int i = 0; i < VR; ++i) {   // (rows past the band: a valid cell, unused)
                    float2 c;
                    warp_cell2(q, u[i], make_float2(mx2, my2), c, f[i]);
                    q.y += 1.0f;
                    const float *p = M + (int)fmaf(c.y, (float)w, c.x);
                    m[i] = make_float4(__ldg(p + w), __ldg(p + w + 1), __ldg(p + 1), __ldg(p));
                }
                // the force of row pairs in packed arithmetic, as in the row sweep (rows past the band are
                // computed from whatever lies there and not used)
                const float *fc = F + yl * w + x;   // row y0 - 1
                const int xl = x > 0 ? -1 : 0, xr = x < w - 1 ? 1 : 0;
                const float sx = (x == 0 || x == w - 1) ? 1.0f : 0.5f;
                const float2 n1 = make_float2(-1.0f, -1.0f), one = make_float2(1.0f, 1.0f), a2 = make_float2(al2, al2);
                float fa = fc[0], fb = fc[w];
#pragma unroll
                for (int i = 0; i < VR; i += 2) {
                    const float *fr_ = fc + (i + 1) * w;
                    const float f2 = fr_[w], f3 = fr_[2 * w];
                    const float2 fl = make_float2(fr_[xl], fr_[w + xl]), frt = make_float2(fr_[xr], fr_[w + xr]);
                    const int ya = y0 + i;
                    const float2 sy = make_float2((ya == 0 || ya == h - 1) ? 1.0f : 0.5f, ya + 1 == h - 1 ? 1.0f : 0.5f);
                    const float2 fx = make_float2(f[i].x, f[i + 1].x), fy = make_float2(f[i].y, f[i + 1].y);
                    const float2 omx = __ffma2_rn(fx, n1, one), omy = __ffma2_rn(fy, n1, one);
                    const float2 top = make_float2(fmaf(fx.x, m[i].z, omx.x * m[i].w), fmaf(fx.y, m[i + 1].z, omx.y * m[i + 1].w));
                    const float2 bot = make_float2(fmaf(fx.x, m[i].y, omx.x * m[i].x), fmaf(fx.y, m[i + 1].y, omx.y * m[i + 1].x));
                    const float2 mw = __ffma2_rn(fy, bot, __fmul2_rn(omy, top));
                    const float2 gx = __fmul2_rn(make_float2(sx, sx), __ffma2_rn(fl, n1, frt));
                    const float2 gy = __fmul2_rn(sy, __ffma2_rn(make_float2(fa, fb), n1, make_float2(f2, f3)));
                    const float2 d = make_float2(fmaf(fb, -1.0f, mw.x), fmaf(f2, -1.0f, mw.y));
                    const float2 den = __ffma2_rn(gx, gx, __ffma2_rn(gy, gy, __fmul2_rn(__fmul2_rn(a2, d), d)));
                    const float t0 = force_quot(d.x, den.x), t1 = force_quot(d.y, den.y);
                    if (yl + i < rows) {
                        put_A(yl + i, x, make_float2(t0 * gx.x, t0 * gy.x));
                        if (regroup) D[(yl + i) * w + x] = d.x;
                        else ssd = fmaf(d.x, d.x, ssd);
                    }
                    if (yl + i + 1 < rows) {
                        put_A(yl + i + 1, x, make_float2(t1 * gx.y, t1 * gy.y));
                        if (regroup) D[(yl + i + 1) * w + x] = d.y;
                        else ssd = fmaf(d.y, d.y, ssd);
                    }
                    fa = f2;
                    fb = f3;
                }
            }
            if (final_pass) {
                __syncthreads();
                break;
            }
            if (!regroup) {
                for (int o = 16; o > 0; o >>= 1) ssd += __shfl_xor_sync(0xffffffffu, ssd, o);
                if (lane == 0) red[warp] = ssd;
            }
            __syncthreads();
            if (!regroup && warp == 0) {   // this CTA's sum to every CTA
                float s = lane < NT / 32 ? red[lane] : 0.0f;
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (C > 1) {
                    if (lane < C) st_remote(remote(esum + rank, lane), s);
                } else if (lane == 0) {
                    esum[0] = s;
                }
            }
            xpass(Y, a.taps.up);
            sync_all();
            if (regroup) {   // d of the whole pair is in place
                for (int task = (int)rank * (NT / 32) + warp; task < a.tasks; task += C * (NT / 32)) {
                    const int nvw = a.nt / 32, tile = task / nvw;
                    const float s = lane_sum(tile, task - tile * nvw);
                    if (C > 1) {
                        if (lane < C) st_remote(remote(wsum + task, lane), s);
                    } else if (lane == 0) {
                        wsum[task] = s;
                    }
                }
            } else if (warp == 0) {
                double E = lane < C ? (double)esum[lane] : 0.0;
                for (int o = MAXC / 2; o > 0; o >>= 1) E += __shfl_xor_sync(0xffffffffu, E, o);
                if (lane == 0) decide(k, E);
            }
            // ---- s_{k+1} = u_k + G_u * du
            for (int j = t; j < nitems; j += NT) {
                const int g = div_by(j, a.mw), x = j - g * w, yl = VR * g;
                float2 acc[VR];
                ypass(Y, a.taps.up, lo + yl, x, acc);
#pragma unroll
                for (int i = 0; i < VR; ++i)
                    if (yl + i < rows) put_A(yl + i, x, __fadd2_rn(U[(yl + i) * w + x], acc[i]));
            }
            __syncthreads();
        }
        for (int p = t; p < rows * w; p += NT) {
            const int y = div_by(p, a.mw), x = p - y * w;
            const float2 v = U[p];
            const size_t at = (size_t)(lo + y) * w + x;
            if (a.planar) {
                a.uout[(size_t)pair * 2 * plane + at] = v.x;
                a.uout[(size_t)pair * 2 * plane + plane + at] = v.y;
            } else {
                reinterpret_cast<float2 *>(a.uout)[(size_t)pair * plane + at] = v;
            }
        }
        sync_all();   // no CTA is still stored into or read from when the next pair begins or it exits
    }
}

}  // namespace clu
