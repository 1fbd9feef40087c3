// k_materialised.cu - the render-then-score form of libb3d: depth (and triangle-id) images
// of every hypothesis written to device memory, and the windowed likelihood of such images.
// Each direction is one pass over the images at close to memory bandwidth; the per-pixel
// work is confined to where an image differs from the scene's background, and the CTAs of a
// persistent grid overlap one hypothesis's streaming with another's raster or scoring.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "k_score.cuh"
#include "k_tris.cuh"

namespace b3d {

// ------------------------------------------------------------------------------------------
// materialised render
// ------------------------------------------------------------------------------------------
// Depth only (k_render_fused), one hypothesis per CTA iteration: the background depths
// (misses at the far plane) are streamed into the whole image, then the object is drawn by
// the fused score kernel's renderer (merged voxel rectangles, cooperative raster, 32-bit
// depth bits) and each tile's composited depths overwrite its fragment box.
// With triangle ids (k_render_obj): every pixel gets the background key's depth and id, then
// the object's triangles over its screen box, with 64-bit atomicMin on packed (depth bits,
// triangle id) (the nearest fragment wins, equal depths go to the smaller id), overwrite the
// pixels where they are nearer. The CTA that draws an image also streams its background: the
// stores (8 bytes a pixel, the bytes the call cannot do without) run beside other CTAs'
// rasterising, which is bound by instruction issue, instead of in a launch of their own
// (2,048 images of 160x120: 171 -> 150 us, 321x241: 1,439 -> 1,312; 450 of 160x120: 45 -> 35).
// Few large images are filled by a launch over all SMs first (k_fill_bg: a band of kBandPx
// background keys stays in shared memory while the CTA streams that band of the images).
constexpr int kBandPx = 4096;

inline int n_bands(int64_t npx) { return (int)((npx + kBandPx - 1) / kBandPx); }

// V = 4: 16-byte vector stores (the image size a multiple of 4 pixels and both outputs
// 16-byte aligned), else 1.
template <int V>
__global__ void __launch_bounds__(256) k_fill_bg(Cam c, const unsigned long long *bg, int64_t n_hyp, float *out_depth,
                                                 int *out_tid) {
    __shared__ __align__(16) float s_d[kBandPx];
    __shared__ __align__(16) int s_t[kBandPx];
    const int64_t npx = (int64_t)c.W * c.H, b0 = (int64_t)blockIdx.y * kBandPx;
    const int n = (int)min((int64_t)kBandPx, npx - b0);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const unsigned long long key = bg[b0 + i];
        s_d[i] = key_depth(key, 0, c.far_z);
        s_t[i] = key == kEmptyKey ? -1 : (int)(unsigned)(key & 0xffffffffu);
    }
    __syncthreads();
    for (int64_t h = blockIdx.x; h < n_hyp; h += gridDim.x) {
        float *dst = out_depth + h * npx + b0;
        int *tdst = out_tid ? out_tid + h * npx + b0 : nullptr;
        if (V == 4) {
            for (int k = threadIdx.x; k < n / 4; k += blockDim.x) {
                __stcs(reinterpret_cast<float4 *>(dst) + k, reinterpret_cast<const float4 *>(s_d)[k]);
                if (tdst) __stcs(reinterpret_cast<int4 *>(tdst) + k, reinterpret_cast<const int4 *>(s_t)[k]);
            }
        } else {
            for (int k = threadIdx.x; k < n; k += blockDim.x) {
                __stcs(dst + k, s_d[k]);
                if (tdst) __stcs(tdst + k, s_t[k]);
            }
        }
    }
}

// Pixels of an image of n 4-byte values before its first 16-byte boundary.
__device__ __forceinline__ int align_head(const void *image, int64_t n) {
    return (int)min((int64_t)((16u - ((uintptr_t)image & 15u)) & 15u) >> 2, n);
}

// The background keys' depths and ids into one image, by the CTA. FILL = 4: 16-byte stores
// between the image's first and last 16-byte boundaries (both outputs at the same offset from
// one), else 1: pixel by pixel.
template <int FILL>
__device__ __forceinline__ void fill_image(const unsigned long long *bg, float *depth, int *tri, int64_t npx, float far_z) {
    const int tid = threadIdx.x;
    auto dep = [&](unsigned hi) { return hi == 0xffffffffu ? far_z : __uint_as_float(hi); };
    // the low word of an empty key is its id, -1
    auto one = [&](int64_t i) {
        const unsigned long long key = __ldg(bg + i);
        __stcs(depth + i, dep((unsigned)(key >> 32)));
        __stcs(tri + i, (int)(unsigned)key);
    };
    if (FILL == 1) {
        for (int64_t i = tid; i < npx; i += kThreads) one(i);
        return;
    }
    const int head = align_head(depth, npx), n4 = (int)((npx - head) / 4), rest = (int)(npx - head) & 3;
    if (tid < head + rest) one(tid < head ? tid : npx - rest + (tid - head));  // before and after the vectors
    float4 *d4 = reinterpret_cast<float4 *>(depth + head);
    int4 *t4 = reinterpret_cast<int4 *>(tri + head);
    const unsigned long long *src = bg + head;
    const bool even = (head & 1) == 0;  // two 8-byte keys to a load
    auto get = [&](int k, uint4 &a, uint4 &b) {
        if (even) {
            a = __ldg(reinterpret_cast<const uint4 *>(src) + 2 * k);
            b = __ldg(reinterpret_cast<const uint4 *>(src) + 2 * k + 1);
        } else {
            const uint2 *p = reinterpret_cast<const uint2 *>(src) + 4 * k;
            const uint2 u0 = __ldg(p), u1 = __ldg(p + 1), u2 = __ldg(p + 2), u3 = __ldg(p + 3);
            a = make_uint4(u0.x, u0.y, u1.x, u1.y);
            b = make_uint4(u2.x, u2.y, u3.x, u3.y);
        }
    };
    auto put = [&](int k, const uint4 &a, const uint4 &b) {
        __stcs(d4 + k, make_float4(dep(a.y), dep(a.w), dep(b.y), dep(b.w)));
        __stcs(t4 + k, make_int4((int)a.x, (int)a.z, (int)b.x, (int)b.z));
    };
    int k = tid;
    for (; k + kThreads < n4; k += 2 * kThreads) {  // two vectors' loads in flight (four: slower, registers)
        uint4 a0, b0, a1, b1;
        get(k, a0, b0);
        get(k + kThreads, a1, b1);
        put(k, a0, b0);
        put(k + kThreads, a1, b1);
    }
    if (k < n4) {
        uint4 a0, b0;
        get(k, a0, b0);
        put(k, a0, b0);
    }
}

// FILL: of fill_image; 0: the images hold the background already.
template <class PS, int FILL>
__global__ void __launch_bounds__(kThreads, 3) k_render_obj(SceneView S, PS P, int64_t n_hyp, float *out_depth,
                                                         int *out_tid) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned long long *zb = reinterpret_cast<unsigned long long *>(smem_raw);  // [kRegionPx]
    __shared__ float s_pose[12];
    __shared__ int s_bb[4];
    __shared__ int s_flags;
    __shared__ TriRanges s_rg;
    __shared__ HugeQueue s_hq;
    const Cam &c = S.cam;
    const MeshView &m = S.mesh;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5;
    const int64_t npx = (int64_t)c.W * c.H;
    for (int64_t h = blockIdx.x; h < n_hyp; h += gridDim.x) {
        __syncthreads();
        if (wid == 0) {
            if (lane == 0) pose12(P, h, s_pose);
            __syncwarp();
            tri_view_warp(m, s_pose, c, lane, s_bb, &s_flags, &s_rg);
        }
        // the barriers below order these stores before the object's
        if (FILL) fill_image<FILL>(S.bg, out_depth + h * npx, out_tid + h * npx, npx, c.far_z);
        __syncthreads();
        if (!(s_flags & 1)) continue;
        const int bx0 = s_bb[0], bx1 = s_bb[1], by0 = s_bb[2], by1 = s_bb[3];
        const int tw = min(bx1 - bx0 + 1, kRegionPx);
        const int th = max(1, kRegionPx / tw);
        for (int ty0 = by0; ty0 <= by1; ty0 += th) {
            for (int tx0 = bx0; tx0 <= bx1; tx0 += tw) {
                const int tx1 = min(tx0 + tw - 1, bx1), ty1 = min(ty0 + th - 1, by1);
                const int zw = tx1 - tx0 + 1, nz = zw * (ty1 - ty0 + 1);
                for (int i = tid; i < nz; i += nt) zb[i] = kEmptyKey;
                if (tid == 0) s_hq.n = 0;
                __syncthreads();
                auto store = [&](int x, int y, float z, unsigned gid) {
                    atomicMin(&zb[(y - ty0) * zw + (x - tx0)], pack_key(z, gid));
                };
                for (int base = wid * 32; base < s_rg.total; base += nt)
                    tri_batch(m, s_rg, s_flags, s_pose, S.tri_base, c, base, 32, tx0, tx1, ty0, ty1, &s_hq, store);
                __syncthreads();
                if (s_hq.n > 0) {
                    tri_huge<kThreads>(s_hq, c, store);
                    __syncthreads();
                }
                const int dq = nt / zw, dr = nt - dq * zw;
                int y = tid / zw, x = tid - y * zw;
                for (int i = tid; i < nz; i += nt) {
                    const unsigned long long key = zb[i];
                    if (key != kEmptyKey) {
                        const int64_t gi = (int64_t)(ty0 + y) * c.W + (tx0 + x);
                        if (key < S.bg[gi]) {
                            out_depth[h * npx + gi] = key_depth(key, 0, c.far_z);
                            out_tid[h * npx + gi] = (int)(unsigned)(key & 0xffffffffu);
                        }
                    }
                    x += dr;
                    y += dq;
                    if (x >= zw) { x -= zw; ++y; }
                }
                __syncthreads();  // the next tile clears the z-buffer this one was read from
            }
        }
    }
}

template <int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_render_fused(SceneView S, PoseList P, int64_t n_hyp, float *out_depth) {
    constexpr int REG = score_region<NT>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned *zb = reinterpret_cast<unsigned *>(smem_raw);
    float4 *lat = reinterpret_cast<float4 *>(smem_raw + REG * sizeof(unsigned));
    __shared__ ScoreShared<NT> sh;
    __shared__ float4 s_stage[NT * kStageStride];
    const Cam &c = S.cam;
    const int tid = threadIdx.x;
    const int64_t npx = (int64_t)c.W * c.H;
    __shared__ long long s_next;
    lattice_coords(S.mesh, lat);  // ordered before use by the loop's first barrier
    int64_t h = blockIdx.x;  // then from the counter S.work when given
    while (h < n_hyp) {
        __syncthreads();
        long long nxt = h + gridDim.x;
        if (tid == 0) {
            if (S.work) nxt = (long long)gridDim.x + (long long)atomicAdd(S.work, 1ull);
            pose12(P, h, sh.pose);
        }
        float *dst = out_depth + h * npx;
        // the background first; render_tiles' barriers order these stores before the tiles'
        {  // 16-byte stores between the image's 16-byte boundaries, four loads in flight per thread.
            // An image of 161x121 starts at any offset from one: pixel by pixel its stores held
            // the CTA up (10,000 images, rendered and scored: 564 us against 433 for 160x120; now
            // 480 and 422)
            const int head = align_head(dst, npx);
            const int n4 = (int)((npx - head) / 4), rest = (int)(npx - head) & 3;
            float4 *d4 = reinterpret_cast<float4 *>(dst + head);
            auto stream = [&](auto get) {
                int k = tid;
                for (; k + 3 * NT < n4; k += 4 * NT) {
                    const float4 a0 = get(k), a1 = get(k + NT), a2 = get(k + 2 * NT), a3 = get(k + 3 * NT);
                    __stcs(d4 + k, a0); __stcs(d4 + k + NT, a1); __stcs(d4 + k + 2 * NT, a2); __stcs(d4 + k + 3 * NT, a3);
                }
                for (; k < n4; k += NT) __stcs(d4 + k, get(k));
            };
            if (head == 0) {
                stream([&](int k) { return __ldg(reinterpret_cast<const float4 *>(S.bgd) + k); });
            } else {
                const float *src = S.bgd + head;
                stream([&](int k) {
                    const float *p = src + 4 * k;
                    return make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
                });
                if (tid < head) dst[tid] = __ldg(S.bgd + tid);
            }
            if (tid < rest) dst[npx - rest + tid] = __ldg(S.bgd + (npx - rest + tid));
        }
        render_tiles<false, NT>(S, 0, 0, sh, s_stage, zb, lat, nullptr,
                                [&](const float *zd, int zx0, int zy0, int zw, int qx0, int qx1, int qy0, int qy1, int, int, int, int) {
                                    const int tww = qx1 - qx0 + 1, n = tww * (qy1 - qy0 + 1);
                                    const int dq = NT / tww, dr = NT - dq * tww;
                                    int y = tid / tww, x = tid - y * tww;
                                    for (int k = tid; k < n; k += NT) {
                                        const int gx = qx0 + x, gy = qy0 + y;
                                        dst[(int64_t)gy * c.W + gx] = zd[(gy - zy0) * zw + (gx - zx0)];
                                        x += dr;
                                        y += dq;
                                        if (x >= tww) { x -= tww; ++y; }
                                    }
                                });
        if (tid == 0) s_next = nxt;
        __syncthreads();
        h = s_next;
    }
}

// ------------------------------------------------------------------------------------------
// scoring of materialised depth images [n, H, W]
// ------------------------------------------------------------------------------------------
// The windowed likelihood of pixel i depends only on the depths in its window, so where an
// image's window holds the same bits as the background image (the scene's fixed objects,
// misses mapped as the likelihood maps them), l_i equals the background term exactly. One
// image per CTA iteration:
//  1. stream the image, comparing each depth's bits with the background's: the box of
//     pixels that differ;
//  2. score the pixels of box + w against their background terms (the depths of box + 2w,
//     read back through the cache, tile by tile in shared memory), with the sliding-window
//     column scorer of the fused kernel (WT = 1, 2) or pixel_ell (WT = 0):
//       LL_h = LL_bg + sum_{i in box + w} (l_i - l_i(bg)).
// MM = 1: miss mode 1 (pixels with id -1 carry no point). V = 4: step 1 reads 16-byte vectors
// between the image's 16-byte boundaries (with MM the ids' too), else 1: pixel by pixel.
// WHOLE: the images have no object slot (a moved camera's): they are scored in many tiles, and
// the next tile's depths are copied to shared memory while one is scored (without ids to look
// up on the way). The copies of one tile at a time were waited for in full (long scoreboard
// 4.9 of 12 stall cycles): 2,048 images of 200x200, rendered and scored, 1,476 -> 1,446 us.
__device__ __forceinline__ void box_note(int i, int W, int &x0, int &x1, int &y0, int &y1) {
    const int y = i / W, x = i - y * W;
    x0 = min(x0, x); x1 = max(x1, x); y0 = min(y0, y); y1 = max(y1, y);
}

// The pixels of a vector of four (starting at pixel i) whose bit is set in mask: one division
// for the vector when it lies in one row.
__device__ __forceinline__ void box_note4(int i, unsigned mask, int W, int &x0, int &x1, int &y0, int &y1) {
    const int y = i / W, x = i - y * W;
    if (x + 3 < W) {
        x0 = min(x0, x + __ffs(mask) - 1); x1 = max(x1, x + 31 - __clz(mask)); y0 = min(y0, y); y1 = max(y1, y);
    } else {
        for (int v = 0; v < 4; ++v)
            if ((mask >> v) & 1u) box_note(i + v, W, x0, x1, y0, y1);
    }
}

// score_column for the 3x3 inlier ball whose window slots without a point need no test of
// their own (r below half a metre), for the long columns of whole images: the window's three
// rows stay in fixed registers, each new row replacing the oldest, so nothing is shifted;
// addresses and row rays advance by one addition; the count accumulates on 2^23, whose low
// bits are the term's index. The nine 0/1 terms add up exactly in any order, so the count, and
// the sum, are score_column's. It takes 18% off the scoring of 200x200 images (2,048 images,
// 0.73 -> 0.61 ms); in the fused kernel, whose columns are a few rows long, it is 0.5% slower.
__device__ __forceinline__ float score_column_ball3(const SceneView &S, const Lik &L, const float *lut, const Cam &c,
                                                    const float *zd, int zx0, int zy0, int zw, int x, int ya, int yb) {
    const bool c0 = x > 0, c2 = x + 1 < c.W;
    const float rx0 = ((float)(x - 1) + 0.5f - c.cx) * c.inv_fx, rx1 = ((float)x + 0.5f - c.cx) * c.inv_fx;
    const float rx2 = ((float)(x + 1) + 0.5f - c.cx) * c.inv_fx;
    const f32x2_t nrx01 = pk2(-rx0, -rx1), nrx22 = pk2(-rx2, -rx2);
    const float r2b = __int_as_float(__float_as_int(L.r2) + 1) * 0x1p100f;  // (next float above r2) 2^100
    const float *zp = zd + (ya - 1 - zy0) * zw + (x - 1 - zx0);
    const float2 *qp = S.qe + ((int64_t)ya * c.W + x);
    int yj = ya - 1;
    float yf = (float)yj + 0.5f;  // exact, as are its increments
    auto load = [&](f32x2_t &z01, float &z2, float &nry) {
        const bool ok = (unsigned)yj < (unsigned)c.H;
        const float a = ok && c0 ? zp[0] : -1.f, b = ok ? zp[1] : -1.f;
        z2 = ok && c2 ? zp[2] : -1.f;
        z01 = pk2(a, b);
        nry = -((yf - c.cy) * c.inv_fy);
        zp += zw;
        yf += 1.f;
        ++yj;
    };
    f32x2_t pa, pb, pc;
    float sa, sb, sc, na, nb, nc;
    load(pa, sa, na);
    load(pb, sb, nb);
    float acc = 0.f;
    int left = yb - ya + 1;
    float2 next = *qp;  // the row's inputs are loaded a row ahead of their use
    auto score = [&](float nmid) {
        const float2 qe = next;  // observed depth (0: no point) and the background's term
        qp += c.W;
        if (--left > 0) next = *qp;
        // the observed point, formed from its depth as the observation kernel forms it
        const float qx = __fmul_rn(qe.x, rx1), qy = __fmul_rn(qe.x, -nmid);
        const f32x2_t qx2 = pk2(qx, qx), qy2 = pk2(qy, qy), qz2 = pk2(qe.x, qe.x);
        // (r2+ - d2) 2^100, saturated to [0, 1], is 1 exactly when d2 <= r2 (see score_column)
        float nf = 8388608.f;
        auto pair = [&](f32x2_t z2, f32x2_t nrx, f32x2_t nry) {
            const f32x2_t ex = fma2(z2, nrx, qx2), ey = fma2(z2, nry, qy2), ez = sub2(qz2, z2);
            float d2a, d2b;
            upk2(fma2(ex, ex, fma2(ey, ey, mul2(ez, ez))), d2a, d2b);
            nf += __saturatef(fmaf(-d2a, 0x1p100f, r2b));
            nf += __saturatef(fmaf(-d2b, 0x1p100f, r2b));
        };
        pair(pa, nrx01, pk2(na, na));
        pair(pb, nrx01, pk2(nb, nb));
        pair(pc, nrx01, pk2(nc, nc));
        pair(pk2(sa, sb), nrx22, pk2(na, nb));
        const float ex = fmaf(sc, -rx2, qx), ey = fmaf(sc, nc, qy), ez = qe.x - sc;
        nf += __saturatef(fmaf(-fmaf(ex, ex, fmaf(ey, ey, ez * ez)), 0x1p100f, r2b));
        const float l = lut[__float_as_int(nf) & 15];
        if (qe.x != 0.f) acc += l - qe.y;
    };
    for (;;) {
        load(pc, sc, nc);
        score(nb);
        if (left == 0) break;
        load(pa, sa, na);
        score(nc);
        if (left == 0) break;
        load(pb, sb, nb);
        score(na);
        if (left == 0) break;
    }
    return acc;
}

__device__ __forceinline__ void async_copy4(float *dst, const float *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <int WT, int NT, int MINB, int V, int MM, bool WHOLE>
__global__ void __launch_bounds__(NT, MINB) k_score_fused(SceneView S, Lik L, const float *depth, const int *tid_in,
                                                          int64_t n_hyp, float *out_ll) {
    constexpr int REG = score_region<NT>();
    constexpr int U = 4;  // vector loads in flight per thread in the streaming pass
    constexpr bool PIPE = WHOLE && MM == 0;
    __shared__ __align__(16) float zbuf[(PIPE ? 2 : 1) * REG];  // depths of the tile + w; PIPE: and of the next
    __shared__ float s_lut[kMaxLut];
    __shared__ float s_red[NT / 32];
    __shared__ int s_box[NT / 32][4];
    const Cam &c = S.cam;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int i = tid; i < L.n_lut; i += NT) s_lut[i] = L.lut[i];
    const int w = WT > 0 ? WT : L.w;
    const bool ball3 = WT == 1 && L.kind == 0 && L.r2 < 0.25f;
    const int64_t npx = (int64_t)c.W * c.H;
    const float *bgd = S.bgd + (MM ? npx : 0);
    __shared__ long long s_next;
    int64_t h = blockIdx.x;  // then from the counter S.work when given
    while (h < n_hyp) {
        __syncthreads();
        long long nxt = h + gridDim.x;
        if (tid == 0 && S.work) nxt = (long long)gridDim.x + (long long)atomicAdd(S.work, 1ull);
        const float *img = depth + h * npx;
        const int *tim = MM ? tid_in + h * npx : nullptr;
        // 1. the box of pixels whose depth bits differ from the background's
        int x0 = INT32_MAX, x1 = -1, y0 = INT32_MAX, y1 = -1;
        auto differs = [&](int64_t i) {
            float d = __ldg(img + i);
            if (MM && __ldg(tim + i) < 0) d = -1.f;
            return __float_as_uint(d) != __float_as_uint(__ldg(bgd + i));
        };
        // An image that differs from the background in its first row, last row and both outer
        // columns (a moved camera) has the whole image as its box, and needs no pass to find it.
        bool whole = false;
        {
            bool e = false;
            for (int x = tid; x < c.W; x += NT) e |= differs(x);
            if (__syncthreads_or(e)) {
                unsigned s = 0;
                for (int x = tid; x < c.W; x += NT) s |= differs(npx - c.W + x) ? 1u : 0u;
                for (int y = tid; y < c.H; y += NT) {
                    s |= differs((int64_t)y * c.W) ? 2u : 0u;
                    s |= differs((int64_t)y * c.W + c.W - 1) ? 4u : 0u;
                }
                whole = __syncthreads_or(s & 1u) && __syncthreads_or(s & 2u) && __syncthreads_or(s & 4u);
            }
        }
        if (whole) {
            x0 = 0; x1 = c.W - 1; y0 = 0; y1 = c.H - 1;
        } else if (V == 4) {
            const int head = align_head(img, npx), n4 = (int)((npx - head) / 4), rest = (int)(npx - head) & 3;
            const float4 *src = reinterpret_cast<const float4 *>(img + head);
            const int4 *tsrc = reinterpret_cast<const int4 *>(MM ? tim + head : nullptr);
            const float *gsrc = bgd + head;
            const bool galigned = ((uintptr_t)gsrc & 15u) == 0;
            auto get_g = [&](int k) {
                const float *p = gsrc + 4 * k;
                return galigned ? __ldg(reinterpret_cast<const float4 *>(p))
                                : make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
            };
            if (tid < head + rest) {  // the pixels before and after the vectors
                const int i = tid < head ? tid : (int)npx - rest + (tid - head);
                if (differs(i)) box_note(i, c.W, x0, x1, y0, y1);
            }
            for (int k0 = tid; k0 < n4; k0 += U * NT) {
                float4 d[U], g[U];
                int4 t[U];
#pragma unroll
                for (int j = 0; j < U; ++j) {
                    const int k = k0 + j * NT;
                    const bool ok = k < n4;
                    d[j] = ok ? __ldg(src + k) : make_float4(0.f, 0.f, 0.f, 0.f);
                    g[j] = ok ? get_g(k) : make_float4(0.f, 0.f, 0.f, 0.f);
                    t[j] = (MM && ok) ? __ldg(tsrc + k) : make_int4(0, 0, 0, 0);
                }
#pragma unroll
                for (int j = 0; j < U; ++j) {
                    const int k = k0 + j * NT;
                    const float e[4] = {t[j].x < 0 ? -1.f : d[j].x, t[j].y < 0 ? -1.f : d[j].y,
                                        t[j].z < 0 ? -1.f : d[j].z, t[j].w < 0 ? -1.f : d[j].w};
                    const float b[4] = {g[j].x, g[j].y, g[j].z, g[j].w};
                    unsigned mask = 0;
#pragma unroll
                    for (int v = 0; v < 4; ++v) mask |= __float_as_uint(e[v]) != __float_as_uint(b[v]) ? 1u << v : 0u;
                    if (mask) box_note4(head + 4 * k, mask, c.W, x0, x1, y0, y1);
                }
            }
        } else {
            for (int64_t k = tid; k < npx; k += NT)
                if (differs(k)) box_note((int)k, c.W, x0, x1, y0, y1);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            x0 = min(x0, __shfl_xor_sync(0xffffffffu, x0, o));
            x1 = max(x1, __shfl_xor_sync(0xffffffffu, x1, o));
            y0 = min(y0, __shfl_xor_sync(0xffffffffu, y0, o));
            y1 = max(y1, __shfl_xor_sync(0xffffffffu, y1, o));
        }
        if (lane == 0) { s_box[wid][0] = x0; s_box[wid][1] = x1; s_box[wid][2] = y0; s_box[wid][3] = y1; }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < NT / 32; ++k) {
            x0 = min(x0, s_box[k][0]); x1 = max(x1, s_box[k][1]);
            y0 = min(y0, s_box[k][2]); y1 = max(y1, s_box[k][3]);
        }
        // 2. score box + w
        float acc = 0.f;
        if (x1 >= 0) {
            const int sx0 = max(x0 - w, 0), sx1 = min(x1 + w, c.W - 1);
            const int sy0 = max(y0 - w, 0), sy1 = min(y1 + w, c.H - 1);
            // the column scorers give each column of a tile a thread
            const int tw = min(min(sx1 - sx0 + 1, WT > 0 ? min(S.tile_w, NT) : S.tile_w), REG / (1 + 2 * w) - 2 * w);
            const int th = max(1, REG / (tw + 2 * w) - 2 * w);
            // the depths of the tile at (tx0, ty0) + w into dst
            auto stage = [&](int tx0, int ty0, float *dst) {
                const int zx0 = max(tx0 - w, 0), zw = min(min(tx0 + tw - 1, sx1) + w, c.W - 1) - zx0 + 1;
                const int zy0 = max(ty0 - w, 0), nz = zw * (min(min(ty0 + th - 1, sy1) + w, c.H - 1) - zy0 + 1);
                const int dq = div_small(NT, zw), dr = NT - dq * zw;
                int y = div_small(tid, zw), x = tid - y * zw;
                for (int i = tid; i < nz; i += U * NT) {
                    float d[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        d[u] = 0.f;
                        if (i + u * NT < nz) {
                            const int gi = (zy0 + y) * c.W + (zx0 + x);  // an image has at most 2^26 pixels
                            if (PIPE) {
                                async_copy4(dst + i + u * NT, img + gi);
                            } else {
                                d[u] = __ldg(img + gi);
                                if (MM && __ldg(tim + gi) < 0) d[u] = -1.f;
                            }
                        }
                        x += dr;
                        y += dq;
                        if (x >= zw) { x -= zw; ++y; }
                    }
                    if (!PIPE) {
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if (i + u * NT < nz) dst[i + u * NT] = d[u];
                    }
                }
                if (PIPE) async_commit();
            };
            if (PIPE) stage(sx0, sy0, zbuf);
            int buf = 0;
            for (int ty0 = sy0; ty0 <= sy1; ty0 += th) {
                for (int tx0 = sx0; tx0 <= sx1; tx0 += tw) {
                    const int tx1 = min(tx0 + tw - 1, sx1), ty1 = min(ty0 + th - 1, sy1);
                    const int zx0 = max(tx0 - w, 0), zx1 = min(tx1 + w, c.W - 1), zy0 = max(ty0 - w, 0);
                    const int zw = zx1 - zx0 + 1;
                    const float *zd = zbuf + buf * REG;
                    if (PIPE) {
                        const bool wrap = tx0 + tw > sx1;
                        const int nx = wrap ? sx0 : tx0 + tw, ny = wrap ? ty0 + th : ty0;
                        buf ^= 1;
                        if (ny <= sy1) {
                            stage(nx, ny, zbuf + buf * REG);
                            async_wait<1>();
                        } else {
                            async_wait<0>();
                        }
                    } else {
                        stage(tx0, ty0, zbuf);
                    }
                    __syncthreads();
                    const int tww = tx1 - tx0 + 1, thh = ty1 - ty0 + 1;
                    if (WT > 0) {
                        // thread -> (column, run of rows)
                        const int nseg = max(1, div_small(NT, tww));
                        const int rps = div_small(thh + nseg - 1, nseg);
                        const int seg = div_small(tid, tww), col = tid - seg * tww;
                        if (seg < nseg && col < tww) {
                            const int ya = ty0 + seg * rps, yb = min(ya + rps - 1, ty1);
                            if (ya <= yb) {
                                FloatSum sum;
                                if (WT == 1 && ball3) sum.v = score_column_ball3(S, L, s_lut, c, zd, zx0, zy0, zw, tx0 + col, ya, yb);
                                else score_column<WT, !WHOLE>(S, L, s_lut, c, zd, zx0, zy0, zw, tx0 + col, ya, yb, sum, nullptr, nullptr);
                                acc += sum.v;
                            }
                        }
                    } else {
                        const int n_t = tww * thh;
                        const int dq = NT / tww, dr = NT - dq * tww;
                        int y = tid / tww, x = tid - y * tww;
                        for (int k = tid; k < n_t; k += NT) {
                            const int gx = tx0 + x, gy = ty0 + y;
                            const int64_t gi = (int64_t)gy * c.W + gx;
                            const float4 q = S.obs[gi];
                            if (q.w != 0.f)
                                acc += minus_bg(pixel_ell(L, s_lut, c, q, gx, gy,
                                                          [&](int xj, int yj) { return zd[(yj - zy0) * zw + (xj - zx0)]; }),
                                                S.ell_bg[gi]);
                            x += dr;
                            y += dq;
                            if (x >= tww) { x -= tww; ++y; }
                        }
                    }
                    __syncthreads();
                }
            }
        }
        const float tot = block_sum(acc, s_red);
        if (tid == 0) {
            out_ll[h] = (float)(*S.ll_bg + (double)tot);
            s_next = nxt;
        }
        __syncthreads();
        h = s_next;
    }
}

// ------------------------------------------------------------------------------------------
// launchers
// ------------------------------------------------------------------------------------------
static bool aligned16p(const void *p) { return ((uintptr_t)p & 15u) == 0; }
// two images of 4-byte values whose 16-byte boundaries fall on the same pixels
static bool same_offset16(const void *a, const void *b) { return (((uintptr_t)a ^ (uintptr_t)b) & 15u) == 0; }

// persistent grid: as many CTAs as fit (or `grid` when > 0), at most one per item
template <class K>
static int persistent_grid(K kernel, int threads, int smem, int64_t n, int grid) {
    if (grid > 0) return (int)std::min<int64_t>(grid, std::max<int64_t>(n, 1));
    const int per_sm = kernel_ctas_per_sm(kernel, threads, smem);
    return (int)std::min<int64_t>((int64_t)per_sm * score_sm_count(), std::max<int64_t>(n, 1));
}

// Launch shape of the fused materialised kernels: 128-thread CTAs; register caps from
// launch-bound sweeps: the renderer at 8 CTAs per SM on the 160x120 tabletop stage (145,800
// images; 64 registers; 3.64 against 3.77 ms at 6). The 3x3 scorer of images that differ from
// the reference around one object streams most of its pixels and wants 8 CTAs (render and
// score of 20,000 images 795 us; 10: 799, 7: 809); images of the whole scene moved (no object
// slot: a camera's) are scored everywhere and want registers: 7 (camera call of 2,048 images
// of 200x200 1,638 us; 8: 1,735, 10: 1,755, 6: 1,637).
constexpr int kMatNT = 128, kRenderMinB = 8;
template <int WT>
constexpr int score_fused_minb(bool whole) { return WT == 1 ? (whole ? 7 : 8) : 6; }

// Renders with ids of fewer than kFillFew images of more than kFillPx pixels fill them in a
// launch of their own: a CTA needs 10 us to stream an image of 76,800 pixels, the device less
// than 2 for 16 of them (16 images of 320x240: 90 us, 95 when each CTA fills its own; 150:
// 121 and 115; 16 of 160x120: 33 and 29).
constexpr int kFillFew = 100, kFillPx = 40000;

int launch_render_list(const SceneView &sv, PoseList P, int64_t n, float *depth, int *tid, int grid, cudaStream_t s) {
    if (n <= 0) return 0;
    const int64_t npx = (int64_t)sv.cam.W * sv.cam.H;
    if (tid) {
        const int smem = kRegionPx * (int)sizeof(unsigned long long);
        if (n < kFillFew && npx > kFillPx) {
            const bool vec = npx % 4 == 0 && aligned16p(depth) && aligned16p(tid);
            auto fill = vec ? k_fill_bg<4> : k_fill_bg<1>;
            const int nb = n_bands(npx);
            const int per_sm = kernel_ctas_per_sm(fill, 256, 0);
            const int64_t x = std::max<int64_t>(1, ((int64_t)per_sm * score_sm_count() + nb - 1) / nb);
            fill<<<dim3((unsigned)std::min<int64_t>(x, n), (unsigned)nb), 256, 0, s>>>(sv.cam, sv.bg, n, depth, tid);
            auto kern = k_render_obj<PoseList, 0>;
            kern<<<persistent_grid(kern, kThreads, smem, n, grid), kThreads, smem, s>>>(sv, P, n, depth, tid);
            return 2;
        }
        auto kern = same_offset16(depth, tid) ? k_render_obj<PoseList, 4> : k_render_obj<PoseList, 1>;
        kern<<<persistent_grid(kern, kThreads, smem, n, grid), kThreads, smem, s>>>(sv, P, n, depth, tid);
        return 1;
    }
    const int n_lat = sv.mesh.nc[0] + sv.mesh.nc[1] + sv.mesh.nc[2];
    const int smem = score_region<kMatNT>() * (int)sizeof(unsigned) + n_lat * (int)sizeof(float4);
    auto kern = k_render_fused<kMatNT, kRenderMinB>;
    if (sv.work) cudaMemsetAsync(sv.work, 0, sizeof(unsigned long long), s);
    kern<<<persistent_grid(kern, kMatNT, smem, n, grid), kMatNT, smem, s>>>(sv, P, n, depth);
    return 1;
}

template <int WT, bool WHOLE>
static void launch_score_fused(const SceneView &sv, const Lik &L, const float *depth, const int *tid, int64_t n,
                               float *ll, int grid, cudaStream_t s) {
    const bool mm = L.miss_mode == 1;
    constexpr int MB = score_fused_minb<WT>(WHOLE);
    auto kern = !mm ? k_score_fused<WT, kMatNT, MB, 4, 0, WHOLE>
                    : (same_offset16(depth, tid) ? k_score_fused<WT, kMatNT, MB, 4, 1, WHOLE> : k_score_fused<WT, kMatNT, MB, 1, 1, WHOLE>);
    if (sv.work) cudaMemsetAsync(sv.work, 0, sizeof(unsigned long long), s);
    kern<<<persistent_grid(kern, kMatNT, 0, n, grid), kMatNT, 0, s>>>(sv, L, depth, tid, n, ll);
}

int launch_score_depth(const SceneView &sv, const Lik &L, const float *depth, const int *tid, int64_t n, float *ll,
                       int grid, cudaStream_t s) {
    if (n <= 0) return 0;
    const bool whole = sv.mesh.n_full <= 0;  // no object slot
    if (L.w == 1 && whole) launch_score_fused<1, true>(sv, L, depth, tid, n, ll, grid, s);
    else if (L.w == 1) launch_score_fused<1, false>(sv, L, depth, tid, n, ll, grid, s);
    else if (L.w == 2 && whole) launch_score_fused<2, true>(sv, L, depth, tid, n, ll, grid, s);
    else if (L.w == 2) launch_score_fused<2, false>(sv, L, depth, tid, n, ll, grid, s);
    else launch_score_fused<0, false>(sv, L, depth, tid, n, ll, grid, s);
    return 1;
}

}  // namespace b3d
