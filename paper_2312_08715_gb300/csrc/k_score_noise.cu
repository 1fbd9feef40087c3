// k_score_noise.cu - scoring under a grid of noise settings (the hierarchical noise of
// Alg. 1): each hypothesis is rendered once (render_tiles of the fused kernel)
// and every scored pixel's window is evaluated under all n_radius x n_pout settings, with
// the per-setting background terms of the fixed objects subtracted as in the single-setting
// kernel (the same per-pixel routine builds the background tables, so unchanged pixels
// cancel bit for bit). A marginal over the grid (log-sum-exp with the settings' prior log
// weights) is formed per hypothesis.
//
// Kind 0: a setting's term depends on the pixel only through its inlier count at the setting's
// radius, so the background tables hold each pixel's counts (a byte per radius, 4 B a pixel
// instead of a float per setting) and a scored pixel reads one word; only where a count
// differs are the terms of its settings looked up, four outlier probabilities per 16-byte
// load. Measured on a GB300 (ncu), 8,192 hypotheses of a 160x120 tabletop stage under 4 x 4
// settings: 687 us with a float per setting and pixel and the marginal formed by one thread,
// 252 us now (a single setting of the plain kernel: about 160).
#include <cuda_runtime.h>
#include <math.h>

#include "k_score.cuh"

namespace b3d {

__device__ __forceinline__ f32x2_t add2(f32x2_t a, f32x2_t b) {
    f32x2_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// Inlier counts of a pixel (kind 0), a byte per radius.
__device__ __forceinline__ unsigned pack_counts(const int *n) {
    return (unsigned)n[0] | ((unsigned)n[1] << 8) | ((unsigned)n[2] << 16) | ((unsigned)n[3] << 24);
}

// l_g for every setting g = 4 i + j (internal layout; i < nr radii, j < np outlier
// probabilities) of observed point q at pixel (xi, yi), the window's rendered depths given
// by fetch (negative: no point). The window is visited in pixel_ell's order and each pair's
// squared distance is formed by pixel_ell's expression; lut holds kNoiseLut entries per g.
// WT: the half window compiled in (1, 2; 0: runtime N.w). Every window element is
// evaluated and its terms predicated (a branch on a missing point costs more than the
// element: the lanes' pixels diverge); a predicated-off element adds nothing, so the sums
// are those of the element-skipping loop.
template <int WT, class Fetch>
__device__ __forceinline__ void noise_pixel_w(const NoiseLik &N, const float *lut, const Cam &c, float4 q, int xi, int yi,
                                              Fetch fetch, float *l, unsigned *counts) {
    const int w = WT > 0 ? WT : N.w;
    int n[kMaxNoiseR];
    float S[kMaxNoiseR];
#pragma unroll
    for (int i = 0; i < kMaxNoiseR; ++i) { n[i] = 0; S[i] = 0.f; }
#pragma unroll
    for (int dy = -w; dy <= w; ++dy) {
        const int yj = yi + dy;
        const bool rowok = yj >= 0 && yj < c.H;
        const float ry = ((float)yj + 0.5f - c.cy) * c.inv_fy;
#pragma unroll
        for (int dx = -w; dx <= w; ++dx) {
            const int xj = xi + dx;
            const float z = (rowok && xj >= 0 && xj < c.W) ? fetch(xj, yj) : -1.f;
            const bool valid = z >= 0.f;
            const float rx = ((float)xj + 0.5f - c.cx) * c.inv_fx;
            const float ex = fmaf(-z, rx, q.x), ey = fmaf(-z, ry, q.y), ez = q.z - z;
            const float d2 = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
#pragma unroll
            for (int i = 0; i < kMaxNoiseR; ++i) {
                if (i >= N.nr) break;
                if (N.kind == 0) n[i] += (valid & (d2 <= N.r2[i])) ? 1 : 0;
                else if (valid) S[i] += __expf(-d2 * N.inv2s2[i]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < kMaxNoiseR; ++i)
#pragma unroll
        for (int j = 0; j < kMaxNoiseP; ++j) {
            const int g = i * kMaxNoiseP + j;
            l[g] = 0.f;
            if (i < N.nr && j < N.np)
                l[g] = N.kind == 0 ? lut[g * kNoiseLut + n[i]] : __logf(fmaf(N.bg[g], S[i], N.a[j]));
        }
    *counts = pack_counts(n);
}

// noise_pixel_w for the runtime half window; counts: the pixel's inlier counts (kind 0).
template <class Fetch>
__device__ __forceinline__ void noise_pixel(const NoiseLik &N, const float *lut, const Cam &c, float4 q, int xi, int yi,
                                            Fetch fetch, float *l, unsigned *counts) {
    if (N.w == 1) noise_pixel_w<1>(N, lut, c, q, xi, yi, fetch, l, counts);
    else if (N.w == 2) noise_pixel_w<2>(N, lut, c, q, xi, yi, fetch, l, counts);
    else noise_pixel_w<0>(N, lut, c, q, xi, yi, fetch, l, counts);
}

// The inlier counts (kind 0, every radius below half a metre, so a window slot without a point
// (depth -1) fails every test by itself) of pixel column x, rows [ya, yb], against the
// background's counts: acc[g] += l_g - l_g(bg) where a count differs. The window slides down
// the column in registers; the distances are pixel_ell's (in packed pairs, each lane rounded
// as the scalar operation). Even radii count on the FMA pipe (see score_column), odd ones by
// comparison on the ALU pipe, so neither holds the other up. NR: radii compiled in (those
// past N.nr have r2 = -1, which nothing meets). lut4[i * kNoiseLut + n]: the terms of radius
// i and count n for the four outlier probabilities.
template <int W, int NR>
__device__ __forceinline__ void noise_column(const SceneView &S, const float *r2, const float4 *lut4, const unsigned *bgn,
                                             const Cam &c, const float *zd, int zx0, int zy0, int zw, int x, int ya, int yb,
                                             f32x2_t (*acc)[2]) {
    constexpr int D = 2 * W + 1;
    float nrx[D], nry[D], win[D][D], r2b[(NR + 1) / 2];
    bool colok[D];
#pragma unroll
    for (int i = 0; i < NR; i += 2) r2b[i / 2] = __int_as_float(__float_as_int(r2[i]) + (r2[i] > 0.f ? 1 : 0)) * 0x1p100f;
#pragma unroll
    for (int d = 0; d < D; ++d) {
        const int xj = x + d - W;
        colok[d] = xj >= 0 && xj < c.W;
        nrx[d] = -(((float)xj + 0.5f - c.cx) * c.inv_fx);
    }
    auto load_row = [&](int yj, float *row) {
        const bool rowok = yj >= 0 && yj < c.H;
#pragma unroll
        for (int d = 0; d < D; ++d) row[d] = (rowok && colok[d]) ? zd[(yj - zy0) * zw + (x + d - W - zx0)] : -1.f;
    };
#pragma unroll
    for (int r = 1; r < D; ++r) {
        load_row(ya - W + r - 1, win[r]);
        nry[r] = -(((float)(ya - W + r - 1) + 0.5f - c.cy) * c.inv_fy);
    }
    for (int y = ya; y <= yb; ++y) {
#pragma unroll
        for (int r = 0; r + 1 < D; ++r) {
            nry[r] = nry[r + 1];
#pragma unroll
            for (int d = 0; d < D; ++d) win[r][d] = win[r + 1][d];
        }
        load_row(y + W, win[D - 1]);
        nry[D - 1] = -(((float)(y + W) + 0.5f - c.cy) * c.inv_fy);
        const int gi = y * c.W + x;  // an image has at most 2^26 pixels
        const float4 q = S.obs[gi];
        const unsigned nb = bgn[gi];
        float nf[(NR + 1) / 2];
        int ni[NR / 2];
#pragma unroll
        for (int i = 0; i < (NR + 1) / 2; ++i) nf[i] = 0.f;
#pragma unroll
        for (int i = 0; i < NR / 2; ++i) ni[i] = 0;
        auto count = [&](float d2) {
#pragma unroll
            for (int i = 0; i < NR; ++i) {
                if (i & 1) ni[i / 2] += d2 <= r2[i] ? 1 : 0;
                else nf[i / 2] += __saturatef(fmaf(-d2, 0x1p100f, r2b[i / 2]));
            }
        };
        const f32x2_t qx2 = pk2(q.x, q.x), qy2 = pk2(q.y, q.y), qz2 = pk2(q.z, q.z);
#pragma unroll
        for (int r = 0; r < D; ++r) {
#pragma unroll
            for (int d = 0; d + 1 < D; d += 2) {
                const f32x2_t z2 = pk2(win[r][d], win[r][d + 1]);
                const f32x2_t ex = fma2(z2, pk2(nrx[d], nrx[d + 1]), qx2), ey = fma2(z2, pk2(nry[r], nry[r]), qy2);
                const f32x2_t ez = sub2(qz2, z2);
                float da, db;
                upk2(fma2(ex, ex, fma2(ey, ey, mul2(ez, ez))), da, db);
                count(da);
                count(db);
            }
            const float z = win[r][D - 1];
            const float ex = fmaf(z, nrx[D - 1], q.x), ey = fmaf(z, nry[r], q.y), ez = q.z - z;
            count(fmaf(ex, ex, fmaf(ey, ey, ez * ez)));
        }
        int n[kMaxNoiseR] = {0, 0, 0, 0};
#pragma unroll
        for (int i = 0; i < NR; ++i) n[i] = (i & 1) ? ni[i / 2] : (int)nf[i / 2];
        if (q.w == 0.f || pack_counts(n) == nb) continue;
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const float4 a = lut4[i * kNoiseLut + n[i]], b = lut4[i * kNoiseLut + (int)((nb >> (8 * i)) & 255u)];
            acc[i][0] = add2(acc[i][0], sub2(pk2(a.x, a.y), pk2(b.x, b.y)));
            acc[i][1] = add2(acc[i][1], sub2(pk2(a.z, a.w), pk2(b.z, b.w)));
        }
    }
}

__device__ __forceinline__ void load_noise_lut(const NoiseLik &N, float *s_lut) {
    for (int k = threadIdx.x; k < kMaxNoise * kNoiseLut; k += blockDim.x) s_lut[k] = N.lut[k];
}

// Kind 0 takes the count form when every radius is below half a metre and its square large
// enough for the scaled comparison of noise_column.
__host__ __device__ inline bool noise_counts(const NoiseLik &N) {
    if (N.kind != 0) return false;
    for (int i = 0; i < N.nr; ++i)
        if (!(N.r2[i] < 0.25f && N.r2[i] > 1e-20f)) return false;
    return true;
}

// Per-pixel background terms of every setting (count form: the packed inlier counts, in
// nell's first n words) and the terms' double-precision sums (fixed order: block partials,
// then the last block adds them in block order).
__global__ void __launch_bounds__(256) k_bg_noise_tables(SceneView S, NoiseLik N, float *nell, double *part,
                                                         unsigned *counter, double *sums) {
    __shared__ float s_lut[kMaxNoise * kNoiseLut];
    __shared__ double s_red[kMaxNoise][256 / 32];
    __shared__ bool s_last;
    load_noise_lut(N, s_lut);
    __syncthreads();
    const Cam &c = S.cam;
    const int64_t n = (int64_t)c.W * c.H;
    const bool by_count = noise_counts(N);
    double acc[kMaxNoise];
#pragma unroll
    for (int g = 0; g < kMaxNoise; ++g) acc[g] = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 q = S.obs[i];
        const int x = (int)(i % c.W), y = (int)(i / c.W);
        float l[kMaxNoise];
        unsigned counts = 0;
#pragma unroll
        for (int g = 0; g < kMaxNoise; ++g) l[g] = 0.f;
        if (q.w != 0.f)
            noise_pixel(N, s_lut, c, q, x, y,
                        [&](int xj, int yj) { return key_depth(S.bg[(int64_t)yj * c.W + xj], N.miss_mode, c.far_z); }, l,
                        &counts);
        if (by_count) reinterpret_cast<unsigned *>(nell)[i] = counts;
#pragma unroll
        for (int g = 0; g < kMaxNoise; ++g) {
            if ((g >> 2) < N.nr && (g & 3) < N.np) {
                if (!by_count) nell[(int64_t)g * n + i] = l[g];
                acc[g] += (double)l[g];
            }
        }
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int g = 0; g < kMaxNoise; ++g) {
        double v = acc[g];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) s_red[g][wid] = v;
    }
    __syncthreads();
    if (threadIdx.x < kMaxNoise) {
        double v = 0.0;
        for (int w = 0; w < nw; ++w) v += s_red[threadIdx.x][w];
        part[kMaxNoise * blockIdx.x + threadIdx.x] = v;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (threadIdx.x < kMaxNoise) {
        const volatile double *vp = part;
        double v = 0.0;
        for (unsigned b = 0; b < gridDim.x; ++b) v += vp[kMaxNoise * b + threadIdx.x];
        sums[threadIdx.x] = v;
    }
    if (threadIdx.x == 0) *counter = 0u;
}

// One hypothesis per CTA iteration: render, then the noise-grid terms of the scored pixels.
// out_ll [n_hyp, nr * np] (may be NULL) in the public layout g = i * np + j; out_marg
// [n_hyp] = log sum_g exp(ll_g + logw_g).
// CW, CR: the count form (kind 0) with half window CW and CR radii compiled in; CR = 0: the
// general form.
template <int NT, int MINB, int CW, int CR>
__global__ void __launch_bounds__(NT, MINB)
    k_score_noise(SceneView S, NoiseLik N, PoseList P, int64_t n_hyp, const float *nell, const double *nsums,
                  float *out_ll, float *out_marg) {
    constexpr int REG = score_region<NT>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned *zb = reinterpret_cast<unsigned *>(smem_raw);
    float4 *lat = reinterpret_cast<float4 *>(smem_raw + REG * sizeof(unsigned));
    __shared__ __align__(16) float s_lut[kMaxNoise * kNoiseLut];
    __shared__ ScoreShared<NT> sh;
    __shared__ float4 s_stage[NT * kStageStride];
    __shared__ float s_red[kMaxNoise][NT / 32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (CR > 0) {  // [radius][count][outlier probability]
        for (int k = tid; k < kMaxNoise * kNoiseLut; k += NT) {
            const int j = k & 3, in = k >> 2, i = in / kNoiseLut, n = in - i * kNoiseLut;
            s_lut[k] = N.lut[(i * kMaxNoiseP + j) * kNoiseLut + n];
        }
    } else {
        load_noise_lut(N, s_lut);
    }
    float r2[CR > 0 ? CR : 1];
#pragma unroll
    for (int i = 0; i < CR; ++i) r2[i] = i < N.nr ? N.r2[i] : -1.f;
    const Cam &c = S.cam;
    const int64_t npx = (int64_t)c.W * c.H;
    const int G = N.nr * N.np;
    __shared__ long long s_next;
    lattice_coords(S.mesh, lat);
    int64_t h = blockIdx.x, h_done;  // then from the counter S.work, as in the single-setting kernel
    __syncthreads();
    while (h < n_hyp) {
        long long nxt = h + gridDim.x;
        if (tid == 0) {
            if (S.work) nxt = (long long)gridDim.x + (long long)atomicAdd(S.work, 1ull);
            pose12(P, h, sh.pose);
        }
        float acc[kMaxNoise];
        f32x2_t acc2[CR > 0 ? CR : 1][2];
#pragma unroll
        for (int g = 0; g < kMaxNoise; ++g) acc[g] = 0.f;
#pragma unroll
        for (int i = 0; i < (CR > 0 ? CR : 1); ++i) acc2[i][0] = acc2[i][1] = pk2(0.f, 0.f);
        render_tiles<false, NT>(
            S, CR > 0 ? CW : N.w, N.miss_mode, sh, s_stage, zb, lat, nullptr,
            [&](const float *zd, int zx0, int zy0, int zw, int qx0, int qx1, int qy0, int qy1, int, int, int, int) {
                const int tww = qx1 - qx0 + 1, thh = qy1 - qy0 + 1;
                if constexpr (CR > 0) {  // thread -> (column, run of rows), as score_body
                    const int nseg = max(1, NT / tww);
                    const int rps = (thh + nseg - 1) / nseg;
                    const int seg = tid / tww;
                    for (int col = tid - seg * tww; seg < nseg && col < tww; col += NT) {
                        const int ya = qy0 + seg * rps, yb = min(ya + rps - 1, qy1);
                        if (ya <= yb)
                            noise_column<CW, CR>(S, r2, reinterpret_cast<const float4 *>(s_lut),
                                                 reinterpret_cast<const unsigned *>(nell), c, zd, zx0, zy0, zw, qx0 + col, ya,
                                                 yb, acc2);
                    }
                    return;
                }
                const int n_tile = tww * thh;
                const int dq = NT / tww, dr = NT - dq * tww;
                int y = tid / tww, x = tid - y * tww;
                for (int k = tid; k < n_tile; k += NT) {
                    const int gx = qx0 + x, gy = qy0 + y;
                    const int64_t gi = (int64_t)gy * c.W + gx;
                    const float4 q = S.obs[gi];
                    if (q.w != 0.f) {
                        float l[kMaxNoise];
                        unsigned counts;
                        noise_pixel(N, s_lut, c, q, gx, gy,
                                    [&](int xj, int yj) { return zd[(yj - zy0) * zw + (xj - zx0)]; }, l, &counts);
#pragma unroll
                        for (int g = 0; g < kMaxNoise; ++g)
                            if ((g >> 2) < N.nr && (g & 3) < N.np) acc[g] += minus_bg(l[g], nell[(int64_t)g * npx + gi]);
                    }
                    x += dr;
                    y += dq;
                    if (x >= tww) { x -= tww; ++y; }
                }
            });
#pragma unroll
        for (int i = 0; i < CR; ++i) {
            upk2(acc2[i][0], acc[4 * i], acc[4 * i + 1]);
            upk2(acc2[i][1], acc[4 * i + 2], acc[4 * i + 3]);
        }
        // block sums of the per-setting deltas, then ll_g = LL_bg_g + delta_g
#pragma unroll
        for (int g = 0; g < kMaxNoise; ++g) {
            if (CR > 0 && g >= 4 * CR) break;
            const float v = warp_sum(acc[g]);
            if (lane == 0) s_red[g][wid] = v;
        }
        if (tid == 0) s_next = nxt;
        __syncthreads();
        h_done = h;
        h = s_next;
        // the last warp finishes this hypothesis (a setting per lane, its exponential and the
        // logarithm in double precision) while the others set up the next: s_red is written
        // again only after that one's barriers, which the last warp joins
        if (wid == NT / 32 - 1) {
            const bool on = lane < kMaxNoise && (lane >> 2) < N.nr && (lane & 3) < N.np;
            double t = -INFINITY;
            if (on) {
                float v = 0.f;
                for (int w = 0; w < NT / 32; ++w) v += s_red[lane][w];
                const float ll = (float)(nsums[lane] + (double)v);
                if (out_ll) out_ll[h_done * G + (lane >> 2) * N.np + (lane & 3)] = ll;
                t = ll + (double)N.logw[lane];
            }
            double m = t;
            for (int o = 8; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
            double sum = on ? exp(t - m) : 0.0;
            for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (lane == 0) out_marg[h_done] = (float)(m + log(sum));
        }
    }
}

int launch_bg_noise_tables(const SceneView &sv, const NoiseLik &N, float *nell, double *part, unsigned *counter,
                           double *sums, cudaStream_t s) {
    const int64_t n = (int64_t)sv.cam.W * sv.cam.H;
    const int blocks = bg_table_blocks(n);
    k_bg_noise_tables<<<blocks, 256, 0, s>>>(sv, N, nell, part, counter, sums);
    return blocks;
}

void launch_score_noise(const SceneView &sv, const NoiseLik &N, const float *poses, int64_t n_hyp, const float *nell,
                        const double *nsums, float *out_ll, float *out_marg, cudaStream_t s) {
    // count form, CTAs per SM the registers are capped for: 6 with windows up to 3x3 (8,192
    // hypotheses under 4 x 4 settings 252 us; 4: 265, 5: 254, 7: 253), 4 with 5x5, whose window
    // takes the registers
    constexpr int NT = 128;
    const int n_lat = sv.mesh.nc[0] + sv.mesh.nc[1] + sv.mesh.nc[2];
    const int smem = score_region<NT>() * (int)sizeof(unsigned) + n_lat * (int)sizeof(float4);
    auto kern = k_score_noise<NT, 4, 0, 0>;
    if (noise_counts(N)) {
        const bool two = N.nr <= 2;
        kern = N.w == 1 ? (two ? k_score_noise<NT, 6, 1, 2> : k_score_noise<NT, 6, 1, 4>)
                        : (N.w == 2 ? (two ? k_score_noise<NT, 4, 2, 2> : k_score_noise<NT, 4, 2, 4>)
                                    : (two ? k_score_noise<NT, 6, 0, 2> : k_score_noise<NT, 6, 0, 4>));
    }
    const int per_sm = kernel_ctas_per_sm(kern, NT, smem);
    const int g = (int)std::min<int64_t>((int64_t)per_sm * score_sm_count(), std::max<int64_t>(n_hyp, 1));
    if (sv.work) cudaMemsetAsync(sv.work, 0, sizeof(unsigned long long), s);
    kern<<<g, NT, smem, s>>>(sv, N, PoseList{poses}, n_hyp, nell, nsums, out_ll, out_marg);
}

}  // namespace b3d
