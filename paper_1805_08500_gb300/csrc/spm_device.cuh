// spm_device.cuh -- exact geometric predicates used by the SPM kernels.
//
// All predicate inputs are points of the integer lattice whose span is at most
// 32767 units, so every coordinate difference fits in 16 signed bits, every
// product of two differences in 31 bits, and an orientation determinant
// (difference of two such products) in a signed 32-bit int: the int32
// arithmetic below is exact. Products that involve a squared segment length
// are done in int64.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "spm_internal.h"

namespace spm {

// Programmatic dependent launch along the chains of small kernels: a kernel
// launched with programmatic stream serialization may be scheduled while its
// predecessor in the stream still runs. Each chain kernel first lets its own
// successor be scheduled (launch_dependents), then waits (griddepcontrol.wait)
// until its predecessor has completed and that grid's memory is visible,
// before it reads anything. Launched the ordinary way, both instructions do
// nothing.
__device__ __forceinline__ void chain_start() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Launches a kernel of a chain with programmatic stream
// serialization (it may be scheduled while its predecessor runs and waits
// for it in chain_start); an ordinary launch if the attribute is refused.
template <typename... KArgs, typename... Args>
static void launch_chained(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                           Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kern, args...) != cudaSuccess) {
        cudaGetLastError();
        kern<<<grid, block, smem, st>>>(args...);
    }
}


// Work counters of an instrumentation build (-DSPM_COUNT); compiled out otherwise.
#ifdef SPM_COUNT
static __device__ unsigned long long g_count[32];  // one copy per translation unit
#define SPM_CNT(i, v) atomicAdd(&::spm::g_count[i], (unsigned long long)(v))
#define SPM_CNT_MAX(i, v) atomicMax(&::spm::g_count[i], (unsigned long long)(v))
#else
#define SPM_CNT(i, v) ((void)0)
#define SPM_CNT_MAX(i, v) ((void)0)
#endif

__device__ __forceinline__ int orient32(int ax, int ay, int bx, int by, int cx, int cy) {
    return (bx - ax) * (cy - ay) - (by - ay) * (cx - ax);
}
__device__ __forceinline__ int cross32(int ax, int ay, int bx, int by) { return ax * by - ay * bx; }

// The same test with q = perpendicular foot of p on segment source A->B = seg
// (Sec. 4), f = A + (num/den)(B - A), 0 < num < den: orient(e_i, f) has the
// sign of (den - num) * orient(e_i, A) + num * orient(e_i, B) (int64). The
// line p->f is parallel to perp(B - A).
__device__ __forceinline__ bool foot_meets_poly(const int2 *V, int m, int4 seg, int px, int py, long long num,
                                                long long den) {
    const int nx = -(seg.w - seg.y), ny = seg.z - seg.x;
    bool pos = false, neg = false, apart = false;
    int2 a = __ldg(V + m - 1);
#pragma unroll 1
    for (int i = 0; i < m; ++i) {
        const int2 b = __ldg(V + i);
        const int s = nx * (b.y - py) - ny * (b.x - px);
        pos |= s > 0;
        neg |= s < 0;
        apart |= orient32(a.x, a.y, b.x, b.y, px, py) <= 0 &&
                 (den - num) * (long long)orient32(a.x, a.y, b.x, b.y, seg.x, seg.y) +
                         num * (long long)orient32(a.x, a.y, b.x, b.y, seg.z, seg.w) <= 0;
        a = b;
    }
    return pos && neg && !apart;
}

// Cone membership of direction w for a vertex generator: wedge cones are the
// closed CCW sector from c1 to c2 (angle < pi); ray cones the closed ray c1.
__device__ __forceinline__ bool in_cone(int ctype, int4 c, int wx, int wy) {
    if (ctype == kConeNone) return true;
    if (ctype == kConeWedge) return cross32(c.x, c.y, wx, wy) >= 0 && cross32(wx, wy, c.z, c.w) >= 0;
    if (ctype == kConeRay) return cross32(c.x, c.y, wx, wy) == 0 && c.x * wx + c.y * wy >= 0;
    return false;
}

// Shadow cone of vertex generator v with obstacle wedge (ws, we) (CCW) when
// reached along arrival direction d: the path wraps around the obstacle, so
// departures lie between d and the first wedge edge met when rotating from d
// toward the obstacle; empty when d points into the wedge.
__device__ __forceinline__ int make_cone(int4 wedge, int dx, int dy, int4 &c) {
    int a = cross32(dx, dy, wedge.x, wedge.y), b = cross32(dx, dy, wedge.z, wedge.w);
    if (a >= 0 && b >= 0 && (a | b)) {  // wedge on the left: turn counter-clockwise
        if (a == 0) { c = make_int4(dx, dy, dx, dy); return kConeRay; }
        c = make_int4(dx, dy, wedge.x, wedge.y);
        return kConeWedge;
    }
    if (a <= 0 && b <= 0 && (a | b)) {  // wedge on the right: turn clockwise
        if (b == 0) { c = make_int4(dx, dy, dx, dy); return kConeRay; }
        c = make_int4(wedge.z, wedge.w, dx, dy);
        return kConeWedge;
    }
    c = make_int4(0, 0, 0, 0);
    return kConeEmpty;
}

// in_cone(make_cone(wedge, d), w) written without branches (selects only):
// the same closed sector, ray or empty set. For tight loops where divergent
// branches cost more than the arithmetic.
__device__ __forceinline__ bool in_shadow_cone(int dx, int dy, short4 wedge, int wx, int wy) {
    const int a = cross32(dx, dy, wedge.x, wedge.y), b = cross32(dx, dy, wedge.z, wedge.w);
    const bool nz = (a | b) != 0;
    const bool left = (a >= 0) & (b >= 0) & nz, right = (a <= 0) & (b <= 0) & nz;
    const int cdw = cross32(dx, dy, wx, wy), dot = dx * wx + dy * wy;
    const bool ray_in = (cdw == 0) & (dot >= 0);
    const bool left_in = (cdw >= 0) & (cross32(wx, wy, wedge.x, wedge.y) >= 0);   // from d to the wedge start
    const bool right_in = (cdw <= 0) & (cross32(wedge.z, wedge.w, wx, wy) >= 0);  // from the wedge end to d
    return (left & ((a == 0) ? ray_in : left_in)) | (right & ((b == 0) ? ray_in : right_in));
}

// Arrival direction at generator v whose parent is u (lattice).
__device__ __forceinline__ void arrival_dir(const DevScene &ds, int u, int2 vl, int &dx, int &dy) {
    if (ds.gen_kind[u] == kSegI) {
        int4 L = ds.seg_lat[ds.gen_aux[u]];
        int ux = L.z - L.x, uy = L.w - L.y;
        int side = cross32(ux, uy, vl.x - L.x, vl.y - L.y);
        dx = side > 0 ? -uy : uy;
        dy = side > 0 ? ux : -ux;
        return;
    }
    int2 ul = ds.gen_lat[u];
    dx = vl.x - ul.x;
    dy = vl.y - ul.y;
}

// Does the open segment p->q meet the open interior of convex CCW polygon
// V[0..m)? Separating-axis test on the segment and the polygon (both convex):
// they are disjoint in the interiors iff some outward edge normal of the
// polygon or the normal of the segment weakly separates them, i.e. (a) all
// polygon vertices lie on one closed side of the line pq, or (b) both endpoints
// lie on the closed outer side of one edge line. One short loop: the pixel
// kernel's speed hangs on its code staying in the instruction caches.
__device__ __forceinline__ bool segment_meets_poly(const int2 *V, int m, int px, int py, int qx, int qy) {
    const int dx = qx - px, dy = qy - py;
    bool pos = false, neg = false, apart = false;
    int2 a = __ldg(V + m - 1);
#pragma unroll 2
    for (int i = 0; i < m; ++i) {
        const int2 b = __ldg(V + i);
        const int s = dx * (b.y - py) - dy * (b.x - px);
        pos |= s > 0;
        neg |= s < 0;
        const int ex = b.x - a.x, ey = b.y - a.y;
        apart |= ex * (py - a.y) - ey * (px - a.x) <= 0 && ex * (qy - a.y) - ey * (qx - a.x) <= 0;
        a = b;
    }
    return pos && neg && !apart;
}

// Calls f(bin) for the bins that the segment from (x, y) by (dx, dy) (lattice
// units) crosses, cell to cell, until f returns true; returns whether it did.
// The float steps are off by far less than the unit the polygons' boxes are
// grown by when they are binned. (A walk by columns with both their row
// ranges, grown by a margin, took four divisions a column and visited more
// bins: vertex phase of the 1024^2 polygons 0.106 -> 0.092 ms.)
template <class F>
__device__ __forceinline__ bool walk_cells(const DevScene &ds, float x, float y, float dx, float dy, F &&f) {
    const float u = (x - (float)ds.bin_x0) * ds.bin_inv, v = (y - (float)ds.bin_y0) * ds.bin_inv;
    const float du = dx * ds.bin_inv, dv = dy * ds.bin_inv;
    auto cell = [](float w, int n) { return min(max((int)floorf(w), 0), n - 1); };
    int cx = cell(u, ds.bin_nx), cy = cell(v, ds.bin_ny);
    const int ex = cell(u + du, ds.bin_nx), ey = cell(v + dv, ds.bin_ny);
    const int sx = ex >= cx ? 1 : -1, sy = ey >= cy ? 1 : -1;
    // segment parameter of the next crossing of a column / row border
    const float ix = __fdividef(1.f, fabsf(du)), iy = __fdividef(1.f, fabsf(dv));
    float nx = (float)(sx > 0 ? cx + 1 : cx), ny = (float)(sy > 0 ? cy + 1 : cy);
    float tx = ex == cx ? INFINITY : fabsf(nx - u) * ix, ty = ey == cy ? INFINITY : fabsf(ny - v) * iy;
    for (int left = abs(ex - cx) + abs(ey - cy);; --left) {
        SPM_CNT(24, 1);  // a bin walked
        if (f(cy * ds.bin_nx + cx)) return true;
        if (left <= 0) return false;
        if (tx < ty) {
            cx += sx;
            nx += (float)sx;
            tx = cx == ex ? INFINITY : fabsf(nx - u) * ix;
        } else {
            cy += sy;
            ny += (float)sy;
            ty = cy == ey ? INFINITY : fabsf(ny - v) * iy;
        }
    }
}

// Calls f(V, m) for every polygon that blocks the open segment between lattice
// points p and q (its open interior meets it) until f returns true; returns
// whether one did. One thread.
template <class F>
__device__ __forceinline__ bool walk_blockers(const DevScene &ds, int px, int py, int qx, int qy, F &&f) {
    const float dx = (float)(qx - px), dy = (float)(qy - py);
    const int bx0 = min(px, qx), bx1 = max(px, qx), by0 = min(py, qy), by1 = max(py, qy);
    return walk_cells(ds, (float)px, (float)py, dx, dy, [&](int bin) {
        const int end = __ldg(ds.bin_start + bin + 1);
        for (int it = __ldg(ds.bin_start + bin); it < end; ++it) {
            const int4 *rp = reinterpret_cast<const int4 *>(ds.bin_recs + it);
            const int4 bx = __ldg(rp);
            if (bx.z < bx0 || bx.x > bx1 || bx.w < by0 || bx.y > by1) continue;
            // the segment's line against the box, with half a unit of slack
            // (the float roundings are below 2^-8 of a unit)
            const float hx = 0.5f * (float)(bx.z - bx.x), hy = 0.5f * (float)(bx.w - bx.y);
            const float mx = 0.5f * (float)(bx.x + bx.z) - (float)px, my = 0.5f * (float)(bx.y + bx.w) - (float)py;
            const float reach = fabsf(dx) * (hy + 0.5f) + fabsf(dy) * (hx + 0.5f);
            if (fabsf(dx * my - dy * mx) > reach) continue;
            const int4 rec = __ldg(rp + 1);
            SPM_CNT(25, 1);  // a polygon tested
            if (segment_meets_poly(ds.poly_v + rec.y, rec.z, px, py, qx, qy) && f(ds.poly_v + rec.y, rec.z)) return true;
        }
        return false;
    });
}

// Exact visibility between lattice point p and generator target q (a point),
// one thread.
__device__ __forceinline__ bool visible_points(const DevScene &ds, int px, int py, int qx, int qy) {
    if (px == qx && py == qy) return true;
    return !walk_blockers(ds, px, py, qx, qy, [](const int2 *, int) { return true; });
}

// Does one polygon hide every point of the box from the point generator at
// lattice point g? The set of points whose open segment to g meets a convex
// polygon's interior is convex, so it suffices that it hides the four corners;
// such a polygon also blocks any one point of the box, here one near its centre.
__device__ __forceinline__ bool box_hidden(const DevScene &ds, int4 box, int2 g) {
    const int cx = (box.x + box.z) >> 1, cy = (box.y + box.w) >> 1;
    if (cx == g.x && cy == g.y) return false;
    return walk_blockers(ds, cx, cy, g.x, g.y, [&](const int2 *V, int m) {
        bool all = true;
#pragma unroll 1
        for (int k = 0; k < 4 && all; ++k)
            all = segment_meets_poly(V, m, k & 1 ? box.z : box.x, k & 2 ? box.w : box.y, g.x, g.y);
        return all;
    });
}

// Exact visibility between lattice point p and its perpendicular foot on
// segment source s (0 < num < den), one thread.
__device__ __forceinline__ bool visible_foot(const DevScene &ds, int s, int px, int py, long long num, long long den) {
    const int4 L = ds.seg_lat[s];
    const int ux = L.z - L.x, uy = L.w - L.y;
    if (cross32(ux, uy, px - L.x, py - L.y) == 0) return true;
    // the foot, to a hundredth of a unit: it only chooses bins and boxes to test
    const float t = __fdividef((float)num, (float)den);
    const float fx = (float)L.x + t * (float)ux, fy = (float)L.y + t * (float)uy;
    const int4 sb = make_int4((int)floorf(fminf((float)px, fx)) - 1, (int)floorf(fminf((float)py, fy)) - 1,
                              (int)ceilf(fmaxf((float)px, fx)) + 1, (int)ceilf(fmaxf((float)py, fy)) + 1);
    const float dx = (float)px - fx, dy = (float)py - fy;
    return !walk_cells(ds, fx, fy, dx, dy, [&](int bin) {
        const int end = __ldg(ds.bin_start + bin + 1);
        for (int it = __ldg(ds.bin_start + bin); it < end; ++it) {
            const int4 *rp = reinterpret_cast<const int4 *>(ds.bin_recs + it);
            const int4 bx = __ldg(rp);
            if (bx.z < sb.x || bx.x > sb.z || bx.w < sb.y || bx.y > sb.w) continue;
            const int4 rec = __ldg(rp + 1);
            if (foot_meets_poly(ds.poly_v + rec.y, rec.z, L, px, py, num, den)) return true;
        }
        return false;
    });
}

// Does test(rec) hold for a polygon (its record's second half: id, first vertex,
// vertices) whose box the segment from (x, y) by (dx, dy) comes near? One warp,
// every lane with the same arguments: a lane takes a bin the segment crosses,
// then the bins' records are dealt to the lanes evenly, so that a whole walk is
// three loads deep where a lane's own would be a hundred instructions and
// three loads a polygon.
template <class F>
__device__ __forceinline__ bool any_poly_near_warp(const DevScene &ds, float x, float y, float dx, float dy, F &&test) {
    const int lane = threadIdx.x & 31;
    constexpr float m = 1.f;  // slack of the float steps
    const float bs = (float)ds.bin_size, ibs = ds.bin_inv;
    auto col_of = [&](float v) { return min(max((int)floorf((v - (float)ds.bin_x0) * ibs), 0), ds.bin_nx - 1); };
    auto row_of = [&](float v) { return min(max((int)floorf((v - (float)ds.bin_y0) * ibs), 0), ds.bin_ny - 1); };
    const int c0 = col_of(fminf(x, x + dx) - m), c1 = col_of(fmaxf(x, x + dx) + m);
    const bool steep = fabsf(dx) < 0.5f;
    const float idx = steep ? 0.f : __fdividef(1.0f, dx);
    const float span = (steep ? fabsf(dy) : fminf(fabsf(dy * idx) * (bs + 2.f * m), fabsf(dy))) + 2.f * m;
    const int K = min((int)(span * ibs) + 3, ds.bin_ny), items = (c1 - c0 + 1) * K;  // an upper bound of a column's rows
    for (int j0 = 0; j0 < items; j0 += 32) {
        int first = 0, cnt = 0;
        if (j0 + lane < items) {
            const int c = (j0 + lane) / K, kr = j0 + lane - c * K;
            float ylo = fminf(0.f, dy), yhi = fmaxf(0.f, dy);
            if (!steep) {
                const float xa = (float)(ds.bin_x0 + (c0 + c) * ds.bin_size) - x;
                const float ta = (xa - m) * idx, tb = (xa + bs + m) * idx;
                const float ya = __saturatef(fminf(ta, tb)) * dy, yb = __saturatef(fmaxf(ta, tb)) * dy;
                ylo = fminf(ya, yb);
                yhi = fmaxf(ya, yb);
            }
            const int row = row_of(y + ylo - m) + kr;
            if (row <= row_of(y + yhi + m)) {
                const int bin = row * ds.bin_nx + c0 + c;
                first = __ldg(ds.bin_start + bin);
                cnt = __ldg(ds.bin_start + bin + 1) - first;
            }
        }
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int up = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += up;
        }
        const int recs = __shfl_sync(0xffffffffu, incl, 31);
        for (int r0 = 0; r0 < recs; r0 += 32) {
            const int r = r0 + lane;
            int own = 0;  // the first lane whose records end beyond r
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(0xffffffffu, incl, (own + o - 1) & 31) <= r) own += o;
            own &= 31;
            const int it = r + __shfl_sync(0xffffffffu, first - incl + cnt, own);
            bool hit = false;
            if (r < recs) {
                const int4 *rp = reinterpret_cast<const int4 *>(ds.bin_recs + it);
                const int4 bx = __ldg(rp), rec = __ldg(rp + 1);
                const float hx = 0.5f * (float)(bx.z - bx.x) + m, hy = 0.5f * (float)(bx.w - bx.y) + m;
                const float qx = 0.5f * (float)(bx.x + bx.z) - x, qy = 0.5f * (float)(bx.y + bx.w) - y;
                hit = fabsf(dx * qy - dy * qx) <= fabsf(dx) * hy + fabsf(dy) * hx &&
                      fabsf(qx - 0.5f * dx) <= 0.5f * fabsf(dx) + hx && fabsf(qy - 0.5f * dy) <= 0.5f * fabsf(dy) + hy &&
                      test(rec);
            }
            if (__any_sync(0xffffffffu, hit)) return true;
        }
    }
    return false;
}

// Pseudo-angle of direction (x, y) != 0: monotone in the true angle, [0, 4),
// opposite directions differ by exactly 2. The angular depth maps of the
// flood and the pixel pass bin directions by it (kAngBins bins of width
// kAngW; kAngEps covers its float error, about 1e-6).
constexpr float kAngW = 4.0f / kAngBins;
constexpr float kAngEps = 1e-4f;
__device__ __forceinline__ float pang(float x, float y) {
    const float r = __fdividef(fabsf(y), fabsf(x) + fabsf(y));
    if (y >= 0.f) return x >= 0.f ? r : 2.f - r;
    return x < 0.f ? 2.f + r : 4.f - r;
}

// Counter-clockwise pseudo-angle from lo to hi, the ends of an edge seen from
// its outer side: less than half a turn, so that a difference below -1 has
// passed 4. One that is merely negative is rounding (an edge in line with the
// viewer spans less than pang resolves: 1e-9 to 1e-7 where the lattice unit is
// the world's) and the edge covers nothing. Taken for a turn, it covered the
// whole circle at its line's distance, often below a unit, and hid everything.
__device__ __forceinline__ float pang_span(float lo, float hi) {
    const float d = hi - lo;
    return d < -1.f ? d + 4.f : fmaxf(d, 0.f);
}

// Exclusive prefix sum of one value per thread over a CTA of blockDim.x
// threads (a multiple of 32, at most 1024); every thread must call it.
// wsum: 32 shared slots. Returns the sum of the values of lower threads.
__device__ __forceinline__ long long cta_exclusive_scan(long long x, long long *wsum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    long long inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const long long w = lane < nwarp ? wsum[lane] : 0;
        long long wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < nwarp) wsum[lane] = wi - w;
    }
    __syncthreads();
    const long long r = wsum[warp] + inc - x;
    __syncthreads();  // wsum may be reused right after
    return r;
}


// Phase clocks of an instrumentation build (-DSPM_TIME); compiled out otherwise.
#ifdef SPM_TIME
// phase clocks of thread 0 (CTA wall time, barriers included), kept in
// registers and added to the global totals once at the end
static __device__ unsigned long long g_time[8];
#define SPM_T0()                                 \
    long long spm_t_ = clock64();                \
    unsigned long long spm_acc_[8] = {0, 0, 0, 0, 0, 0, 0, 0}
#define SPM_LAP(i)                                              \
    do {                                                        \
        const long long n_ = clock64();                         \
        spm_acc_[i] += (unsigned long long)(n_ - spm_t_);       \
        spm_t_ = n_;                                            \
    } while (0)
#define SPM_TFLUSH()                                                          \
    do {                                                                      \
        if (threadIdx.x == 0)                                                 \
            for (int i_ = 0; i_ < 8; ++i_) atomicAdd(&::spm::g_time[i_], spm_acc_[i_]); \
    } while (0)
#else
#define SPM_T0() ((void)0)
#define SPM_LAP(i) ((void)0)
#define SPM_TFLUSH() ((void)0)
#endif

}  // namespace spm
