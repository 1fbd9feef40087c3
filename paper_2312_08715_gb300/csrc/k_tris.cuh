// k_tris.cuh - triangle rasteriser shared by the renderers that need exact triangle ids or
// depths (materialised renders with ids, camera hypotheses). Per fragment it evaluates the
// expressions of raster_tri (b3d_device.cuh) on the same inputs, so it produces the same
// coverage and depth bits; what differs is how the work is shared out:
//  - a closed voxel mesh's surface triangles are stored by face class and lattice plane (as
//    its rectangles are), so only the contiguous ranges of the classes turned towards the
//    camera are set up: about half of the triangles;
//  - a warp takes 32 triangles, each lane sets one up; a triangle with a few candidate pixels
//    is tested by its lane, a larger one by the whole warp (its record broadcast), and one of
//    hundreds of pixels is queued for the whole CTA. With a thread per triangle a box face of
//    a thousand pixels held its CTA up on one lane (200x200 camera render, 2,048 hypotheses:
//    10 of 32 threads active, 15 of 19 stall cycles at barriers).
// Measured on a GB300 (ncu): camera render of 2,048 hypotheses at 200x200 (10k-voxel object,
// two boxes, 800-triangle table) 3.78 -> 1.16 ms, 794k -> 326k warp instructions a hypothesis;
// object render with ids, 2,048 poses at 160x120, 0.306 -> 0.119 ms, 75k -> 34k instructions.
// What is left is instruction issue (set-up and pixel tests): with large triangles in batches
// of 8 the camera render takes 0.93 to 1.0 ms at 69% of the issue rate. Pixels two at a time in packed
// arithmetic, by a lane for its own triangle or by the warp, were no faster.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "b3d_device.cuh"
#include "b3d_internal.h"

namespace b3d {

// A triangle set up for its pixel tests: the canonical edges with the orientation sign folded
// in (see stage_edge), the vertices' 1/z, the absolute area and the pixel box.
struct TriRec {
    float4 e0, e1, e2;
    float az, bz, cz, area;
    int x0, y0, bw, n;  // box origin, width, pixel count (0: nothing to draw)
    unsigned gid;
};

__device__ __forceinline__ int tri_setup(TriRec &T, const float4 &A, const float4 &B, const float4 &C, int cull, int rx0,
                                         int rx1, int ry0, int ry1) {
    T.n = 0;
    if (A.z < 0.f || B.z < 0.f || C.z < 0.f) return 0;
    const float area = edge_fn(A.x, A.y, B.x, B.y, C.x, C.y);
    if (cull ? !(area < 0.f) : !(area != 0.f)) return 0;
    const float umin = fminf(A.x, fminf(B.x, C.x)), umax = fmaxf(A.x, fmaxf(B.x, C.x));
    const float vmin = fminf(A.y, fminf(B.y, C.y)), vmax = fmaxf(A.y, fmaxf(B.y, C.y));
    const int x0 = (int)ceilf(fmaxf(umin - 0.5f, (float)rx0)), x1 = (int)floorf(fminf(umax - 0.5f, (float)rx1));
    const int y0 = (int)ceilf(fmaxf(vmin - 0.5f, (float)ry0)), y1 = (int)floorf(fminf(vmax - 0.5f, (float)ry1));
    if (x0 > x1 || y0 > y1) return 0;
    const float s = area > 0.f ? 1.f : -1.f;
    T.e0 = stage_edge(A.x, A.y, B.x, B.y, s);
    T.e1 = stage_edge(B.x, B.y, C.x, C.y, s);
    T.e2 = stage_edge(C.x, C.y, A.x, A.y, s);
    T.az = A.z; T.bz = B.z; T.cz = C.z;
    T.area = s * area;
    T.x0 = x0; T.y0 = y0;
    T.bw = x1 - x0 + 1;
    T.n = T.bw * (y1 - y0 + 1);
    return T.n;
}

// One candidate pixel: every test evaluated, one predicated store (see raster_block in
// k_score.cuh). With the sign folded into the edges, s e_k, s den and s area are formed
// exactly (negation is exact), so the depth is raster_tri's area / den.
template <class Store>
__device__ __forceinline__ void tri_pixel(const TriRec &T, int x, int y, bool valid, float far_z, Store &&store) {
    const float px = (float)x + 0.5f, py = (float)y + 0.5f;
    const float e0 = fmaf(T.e0.z, py - T.e0.y, -(T.e0.w * (px - T.e0.x)));
    const float e1 = fmaf(T.e1.z, py - T.e1.y, -(T.e1.w * (px - T.e1.x)));
    const float e2 = fmaf(T.e2.z, py - T.e2.y, -(T.e2.w * (px - T.e2.x)));
    if (valid & !(e0 < 0.f) & !(e1 < 0.f) & !(e2 < 0.f)) {
        const float z = T.area / fmaf(e1, T.az, fmaf(e2, T.bz, e0 * T.cz));
        if (z <= far_z) store(x, y, z, T.gid);
    }
}

// Up to 6 contiguous ranges of triangles: first triangle of range c, exclusive prefix of the
// range lengths, total.
struct TriRanges {
    int first[6];
    int pre[6];
    int total;
};

// How far (in object units) the camera must be inside a plane of a face class for the screen area of
// every triangle there to have the sign of a triangle turned away, whatever its rounding: 2 mm for
// 5 mm cells at 0.8 m in an image of 160x120. (With a fixed 0.1 mm + 0.01% instead, 18 of 30,000
// edge-on poses of 2 mm cells at 3 to 8 m, the principal point 6,000 pixels away, lost a pixel.)
// A triangle of legs e_b, e_c on a plane that the camera is d inside has twice the screen area
// f^2 e_b e_c d / (z_a z_b z_c). What is computed differs by the rounding of its vertices, each
// coordinate by E <= 2^-24 (3 f S / z + 3 V (1 + S / z)) with S the largest sum in the transform and
// V the largest screen coordinate (beyond the image too, with the principal point's), so by
// 2 sqrt(2) E (f + V) (e_b + e_c) / z + 8 E^2, and by 3 2^-24 of the squared leg (f + V) e / z in the
// products. With the smallest gap e of the lattice, K = 1 + V / f and r = E z / (f e) the sign is
// certain beyond d = z (5.7 K r + 8 r^2 + 3 2^-24 K^2), which grows with z: the farthest corner's is
// taken, and a third more for poses that are rigid to some percent only. kFaceMargin covers the
// rounding of the camera's position.
constexpr float kFaceMargin = 1e-4f;
__device__ __forceinline__ float face_margin(const MeshView &m, const Cam &c, float dist, float z, float screen) {
    const float rx = fmaxf(fabsf(m.lo[0]), fabsf(m.hi[0])), ry = fmaxf(fabsf(m.lo[1]), fabsf(m.hi[1]));
    const float rad = sqrtf(rx * rx + ry * ry + fmaxf(m.lo[2] * m.lo[2], m.hi[2] * m.hi[2]));  // of the box's corners
    const float S = dist + 2.f * rad, zf = 1.05f * (z + rad), f = fminf(c.fx, c.fy), fm = fmaxf(c.fx, c.fy);
    const float V = screen + fmaxf(fabsf(c.cx), fabsf(c.cy)), K = (fm + V) / f;
    const float r = 0x1p-24f * 3.f * (fm * S + V * (zf + S)) / (f * m.gap);  // E z / (f e)
    return kFaceMargin * (1.f + dist) + 1.34f * zf * (r * fmaf(8.f, r, 5.7f * K) + 3.f * 0x1p-24f * K * K);
}

// Screen box, flags (bit 0: on screen, bit 2: whole object beyond the near plane) and triangle
// ranges of one object under pose P (shared memory), by one warp. The ranges of a mesh whose
// surface triangles are stored by class hold every triangle of a class whose plane has the
// camera on its outer side or is within face_margin of it; the screen-area test of tri_setup
// decides on those, as it does without ranges. A pose that is not rigid to some percent, and a
// margin that is not a number, take every triangle.
__device__ __forceinline__ void tri_view_warp(const MeshView &m, const float *P, const Cam &c, int lane, int *bb,
                                              int *flags, TriRanges *rg) {
    float umin = INFINITY, umax = -INFINITY, vmin = INFINITY, vmax = -INFINITY;
    bool cfront = true;
    const bool has = m.n_full > 0;
    if (has && lane < 8) {  // the arithmetic of object_bbox, one corner per lane
        const float ox = (lane & 1) ? m.hi[0] : m.lo[0], oy = (lane & 2) ? m.hi[1] : m.lo[1];
        const float oz = (lane & 4) ? m.hi[2] : m.lo[2];
        float x, y, z;
        xform(P, ox, oy, oz, x, y, z);
        if (!(z >= c.near_z)) {
            cfront = false;
        } else {
            umin = umax = fmaf(c.fx, x / z, c.cx);
            vmin = vmax = fmaf(c.fy, y / z, c.cy);
        }
    }
    const bool front = has && __all_sync(0xffffffffu, cfront);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        umin = fminf(umin, __shfl_xor_sync(0xffffffffu, umin, o));
        umax = fmaxf(umax, __shfl_xor_sync(0xffffffffu, umax, o));
        vmin = fminf(vmin, __shfl_xor_sync(0xffffffffu, vmin, o));
        vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
    }
    const bool classes = front && m.tri_off != nullptr;
    int b = 0, cnt = 0;
    if (classes && lane < 6) {
        const int a = lane >> 1;
        // camera position in the object frame along axis a, by the adjugate of the linear part
        const int i = (a + 1) % 3, j = (a + 2) % 3;
        const float cx = P[3 + i] * P[6 + j] - P[6 + i] * P[3 + j], cy = P[6 + i] * P[j] - P[i] * P[6 + j],
                    cz = P[i] * P[3 + j] - P[3 + i] * P[j];
        const float det = fmaf(P[a], cx, fmaf(P[3 + a], cy, P[6 + a] * cz));
        const float t2 = fmaf(P[9], P[9], fmaf(P[10], P[10], P[11] * P[11]));
        const float oa = -fmaf(cx, P[9], fmaf(cy, P[10], cz * P[11])) / det;
        const float marg = face_margin(m, c, sqrtf(t2), P[11],
                                       fmaxf(fmaxf(fabsf(umin), fabsf(umax)), fmaxf(fabsf(vmin), fabsf(vmax))));
        // squared lengths of the rotation's columns
        float col = 0.f;
#pragma unroll
        for (int k = 0; k < 3; ++k) col = fmaxf(col, fmaf(P[k], P[k], fmaf(P[3 + k], P[3 + k], P[6 + k] * P[6 + k])));
        const int *off = m.tri_off + lane * m.np1;
        const int n = m.nc[a];
        const float *cd = m.coords + (a == 0 ? 0 : (a == 1 ? m.nc[0] : m.nc[0] + m.nc[1]));
        int lo = 0, hi = n;
        if (!(det > 0.95f && det < 1.05f && col < 1.05f)) {
            b = off[0];
            cnt = off[n] - b;
        } else if (lane & 1) {  // outward +axis: planes below the camera
            while (lo < hi) { const int mid = (lo + hi) >> 1; if (!(cd[mid] >= oa + marg)) lo = mid + 1; else hi = mid; }
            b = off[0];
            cnt = off[lo] - b;
        } else {  // outward -axis: planes above it
            while (lo < hi) { const int mid = (lo + hi) >> 1; if (cd[mid] <= oa - marg) lo = mid + 1; else hi = mid; }
            b = off[lo];
            cnt = off[n] - b;
        }
    } else if (!classes && lane == 0) {
        cnt = front ? m.n_surf : m.n_full;
    }
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += up;
    }
    if (lane < 6) {
        rg->first[lane] = b;
        rg->pre[lane] = incl - cnt;
    }
    if (lane == 5) rg->total = incl;
    if (lane == 0) {
        int b0 = 0, b1 = c.W - 1, b2 = 0, b3 = c.H - 1;
        if (front) {
            const float lo_u = fmaxf(umin - 0.5f, -2.f), hi_u = fminf(umax - 0.5f, (float)c.W + 1.f);
            const float lo_v = fmaxf(vmin - 0.5f, -2.f), hi_v = fminf(vmax - 0.5f, (float)c.H + 1.f);
            b0 = max((int)ceilf(lo_u) - 1, 0);
            b1 = min((int)floorf(hi_u) + 1, c.W - 1);
            b2 = max((int)ceilf(lo_v) - 1, 0);
            b3 = min((int)floorf(hi_v) + 1, c.H - 1);
        }
        bb[0] = b0; bb[1] = b1; bb[2] = b2; bb[3] = b3;
        *flags = (has && b0 <= b1 && b2 <= b3 ? 1 : 0) | (front ? 4 : 0);
    }
}

// Triangles whose pixel box exceeds kTriHuge wait in a CTA-wide queue (a full queue leaves
// them to their warp).
// A lane testing n pixels alone costs the warp n passes of ~35 instructions; sharing a triangle
// costs ~60 for its record and the index arithmetic: the lines lie where the two meet and where
// one warp would hold the CTA up.
constexpr int kTriOwn = 10;    // candidate pixels a lane tests for its own triangle
constexpr int kTriHuge = 384;  // and above which a triangle is queued for the whole CTA
constexpr int kHugeQueue = 48;
struct HugeQueue {
    TriRec rec[kHugeQueue];
    int n;
};

// Triangles [base, base + cnt) of the ranges, cnt at most 32, by one warp (all lanes call it).
template <class Store>
__device__ __forceinline__ void tri_batch(const MeshView &m, const TriRanges &rg, int flags, const float *pose, int tri_base,
                                          const Cam &c, int base, int cnt, int rx0, int rx1, int ry0, int ry1, HugeQueue *hq,
                                          Store &&store) {
    const int lane = threadIdx.x & 31;
    const bool front = (flags & 4) != 0;
    const int k = base + lane;
    TriRec T;
    T.n = 0;
    if (lane < cnt && k < rg.total) {
        int cls = 0;
#pragma unroll
        for (int j = 1; j < 6; ++j) cls += k >= rg.pre[j] ? 1 : 0;
        // ranges past the last hold nothing: their prefix is the total, above every k
        const int4 tr = (front ? m.tris_surf : m.tris_full)[rg.first[cls] + (k - rg.pre[cls])];
        float4 A, B, C;
        tri_screen(m, tr, pose, c, A, B, C);
        tri_setup(T, A, B, C, front ? m.closed : 0, rx0, rx1, ry0, ry1);
        T.gid = (unsigned)(tri_base + tr.w);
    }
    bool shared = T.n > kTriOwn;
    if (hq && T.n > kTriHuge) {
        const int slot = atomicAdd(&hq->n, 1);
        if (slot < kHugeQueue) {
            hq->rec[slot] = T;
            shared = false;
            T.n = 0;
        }
    }
    {  // a lane's own few pixels
        const int n_own = shared ? 0 : T.n;
        int x = T.x0, y = T.y0;
        for (int i = 0; i < n_own; ++i) {
            tri_pixel(T, x, y, true, c.far_z, store);
            if (++x >= T.x0 + T.bw) { x = T.x0; ++y; }
        }
    }
    // larger boxes: the warp's lanes share one triangle's pixels at a time
    for (unsigned big = __ballot_sync(0xffffffffu, shared); big; big &= big - 1) {
        const int src = __ffs(big) - 1;
        auto bc = [&](float v) { return __shfl_sync(0xffffffffu, v, src); };
        auto bi = [&](int v) { return __shfl_sync(0xffffffffu, v, src); };
        TriRec S;
        S.e0 = make_float4(bc(T.e0.x), bc(T.e0.y), bc(T.e0.z), bc(T.e0.w));
        S.e1 = make_float4(bc(T.e1.x), bc(T.e1.y), bc(T.e1.z), bc(T.e1.w));
        S.e2 = make_float4(bc(T.e2.x), bc(T.e2.y), bc(T.e2.z), bc(T.e2.w));
        S.az = bc(T.az); S.bz = bc(T.bz); S.cz = bc(T.cz); S.area = bc(T.area);
        S.x0 = bi(T.x0); S.y0 = bi(T.y0); S.bw = bi(T.bw); S.n = bi(T.n);
        S.gid = (unsigned)bi((int)T.gid);
        // quotients of numbers up to 32: an approximate reciprocal is exact after the half
        const float rb = __fdividef(1.f, (float)S.bw);
        const int dq = (int)(32.5f * rb), dr = 32 - dq * S.bw;
        int y = (int)(((float)lane + 0.5f) * rb), x = lane - y * S.bw;
        for (int i = lane; i < S.n; i += 32) {
            tri_pixel(S, S.x0 + x, S.y0 + y, true, c.far_z, store);
            x += dr;
            y += dq;
            if (x >= S.bw) { x -= S.bw; ++y; }
        }
    }
}

// The queued triangles, the CTA's NT threads sharing each one's pixels (after a barrier that
// follows the last tri_batch).
template <int NT, class Store>
__device__ __forceinline__ void tri_huge(const HugeQueue &hq, const Cam &c, Store &&store) {
    const int n = min(hq.n, kHugeQueue);
    for (int k = 0; k < n; ++k) {
        const TriRec &T = hq.rec[k];
        const int bw = T.bw, dq = NT / bw, dr = NT - dq * bw;
        int y = (int)threadIdx.x / bw, x = (int)threadIdx.x - y * bw;
        for (int i = threadIdx.x; i < T.n; i += NT) {
            tri_pixel(T, T.x0 + x, T.y0 + y, true, c.far_z, store);
            x += dr;
            y += dq;
            if (x >= bw) { x -= bw; ++y; }
        }
    }
}

}  // namespace b3d
