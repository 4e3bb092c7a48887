// spm_flood.cu -- per-tile candidate lists by flooding each generator's
// potentially visible tiles (the per-tile culling step of the pixel pass).
//
// For a point generator g (point source, segment endpoint, obstacle vertex),
// the pixels that see g and lie in its shadow cone form a region that is
// star-shaped from g: the segment from g to any such pixel stays inside the
// cone and sees g all along. Every tile that segment crosses therefore holds
// visible points. A breadth-first flood over tiles from g's tile, expanding a
// tile only when it meets the cone and is not provably hidden from g (by the
// angular depth map below), thus reaches every tile where g can win (tiles
// are closed rectangles that tile the plane; 8-neighbour steps follow any
// segment). Each reached tile gets g in its candidate list. One CTA floods one
// generator, a breadth-first level at a time. Segment interiors, points
// outside the tile grid and floods whose level outgrows the frontier go to a
// global list that every tile scans. Any failure of the lists (pair capacity)
// sets a flag and the pixel pass falls back to scanning every generator.
#include <cuda_runtime.h>

#include <algorithm>

#include "spm_device.cuh"
#include "spm_internal.h"

namespace spm {
namespace {

constexpr int kFloodThreads = 256;  // one CTA floods one generator at a time
constexpr int kFront = 1024;        // frontier tiles per breadth-first level
constexpr int kFloodPolyBits = 65536;  // polygons tracked for insertion (beyond: inserted again, harmless)

// Full area of tile (tx, ty) in lattice units: closed rectangle, neighbours
// share edges. Pixel i covers [i * pitch, (i + 1) * pitch].
__device__ __forceinline__ int4 tile_area(const DevScene &ds, int tx, int ty) {
    const int px = ds.S * ds.Wx / ds.Nx, py = ds.S * ds.Wy / ds.Ny;
    const int T = ds.tile;
    return make_int4(tx * T * px, ty * T * py, min((tx + 1) * T, ds.Nx) * px, min((ty + 1) * T, ds.Ny) * py);
}

__device__ __forceinline__ bool cone_meets_box(int ct, int4 c, int2 v, int4 box) {
    if (ct == kConeNone) return true;
    if (ct == kConeEmpty) return false;
    const int cx[4] = {box.x, box.z, box.x, box.z}, cy[4] = {box.y, box.y, box.w, box.w};
    bool out1 = true, out2 = true;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int wx = cx[k] - v.x, wy = cy[k] - v.y;
        out1 &= cross32(c.x, c.y, wx, wy) < 0;
        out2 &= cross32(wx, wy, c.z, c.w) < 0;
    }
    return !(out1 || out2);
}

// What the kept part of the obstacle vertices is built for. Whoever overwrites
// it clears the tag in flood_counts; its last kernel sets it. A build whose
// kernels get the tag as `unless` does nothing when the device has that part
// already: recorded computes are replayed in whatever order the caller likes,
// between computes of other tunings.
__host__ __device__ __forceinline__ int kept_tag(const DevScene &ds) {
    return 4 | (ds.tile == kTile ? 2 : 0) | (ds.use_maps && ds.gen_maps ? 1 : 0);
}
__device__ __forceinline__ bool kept_already(const DevScene &ds, int unless) {
    return unless && ds.flood_counts[kKeptTag] == unless;
}

// Before the obstacle vertices' flood: no counts, no bits or tile counts.
__global__ void k_kept_reset(const __grid_constant__ DevScene ds, int unless) {
    if (kept_already(ds, unless)) return;
    const size_t i0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x, step = (size_t)gridDim.x * blockDim.x;
    const size_t ntiles = (size_t)ds.tiles_x * ds.tiles_y;
    if (i0 < 4) ds.flood_counts[i0] = 0;
    if (ds.vert_bits)
        for (size_t i = i0; i < ntiles * ds.vert_words; i += step) ds.vert_mask[i] = 0u;
    else
        for (size_t i = i0; i < ntiles; i += step) ds.tile_count[i] = 0;
}

__device__ __forceinline__ void push_global(const DevScene &ds, int g) {
    ds.glob_list[atomicAdd(&ds.flood_counts[1], 1)] = g;
}

// Angular depth map of one generator g (shadow volumes, in the spirit of the
// shadow construction of Sec. 3.1): directions around g are cut into kAng
// bins of a pseudo-angle; depth2[b] is an upper bound on the squared distance
// from g at which every ray of bin b has crossed a front-facing obstacle edge
// (g strictly on its outer side), i.e. entered an obstacle interior. A tile is
// hidden from g when every bin its corners span has depth2 at most the tile's
// squared nearest distance: each of its points lies beyond an obstacle
// interior on its ray. Along an edge's line the crossing distance is convex in
// the ray angle, so over a bin it peaks at one of the two boundary rays; the
// boundary directions are exact multiples of 1/512, which makes the dot
// products exact in integers and leaves a few float roundings (covered by a
// 1e-5 relative margin). Polygons enter the map as the flood reaches their
// tiles, so every test is conservative; unions of polygons (walls that
// overlap at posts) hide tiles that no single polygon hides.
constexpr int kAng = kAngBins;      // pseudo-angle bins over [0, 4)
constexpr int kAngQ = kAng / 4;     // bins per quadrant (boundary m is pseudo-angle m / kAngQ)
constexpr int kInsCap = 1024;       // polygons inserted per level

// Pseudo-angle difference b - a wrapped into (-2, 2].
__device__ __forceinline__ float pang_diff(float a, float b) {
    float d = b - a;
    if (d > 2.f) d -= 4.f;
    if (d <= -2.f) d += 4.f;
    return d;
}

// Direction of bin boundary m, scaled by kAngQ: integer components.
__device__ __forceinline__ int2 boundary_dir(int m) {
    const int mm = m & (kAng - 1), f = mm & (kAngQ - 1);
    switch (mm / kAngQ) {
        case 0: return make_int2(kAngQ - f, f);
        case 1: return make_int2(-f, kAngQ - f);
        case 2: return make_int2(-(kAngQ - f), -f);
        default: return make_int2(f, -(kAngQ - f));
    }
}

struct FloodSmem {
    float depth2[kAng];
    int front[2][kFront];  // current / next breadth-first level
    int flag[kFront];      // 0 visible, 1 hidden, 2 outside the cone
    int ins[kInsCap];      // polygons to insert before this level's tests
    int cnt[2];
    int n_ins;
    int overflow;
    int ins_dropped;       // a polygon was left out of the map (insertion list full)
};

// Is the closed box hidden from g (lattice point, not inside the box) by the
// depth map? A group of G lanes (lane gl of mask gmask) tests G of the
// spanned bins at a time (a tile near g spans hundreds of bins, a far one a
// few).
template <int G>
__device__ bool box_hidden_ang(const float *depth2, int2 g, int4 box, int gl, unsigned gmask, int stride) {
    const long long dx = max(max(box.x - g.x, g.x - box.z), 0), dy = max(max(box.y - g.y, g.y - box.w), 0);
    const float mind2 = (float)(dx * dx + dy * dy) * (1.f - 1e-6f);
    const float c0 = pang(0.5f * (float)(box.x + box.z) - (float)g.x, 0.5f * (float)(box.y + box.w) - (float)g.y);
    float lo = 0.f, hi = 0.f;
    const int cx[4] = {box.x, box.z, box.x, box.z}, cy[4] = {box.y, box.y, box.w, box.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float d = pang_diff(c0, pang((float)(cx[k] - g.x), (float)(cy[k] - g.y)));
        lo = fminf(lo, d);
        hi = fmaxf(hi, d);
    }
    const int k0 = (int)floorf((c0 + lo - kAngEps) / kAngW), k1 = (int)floorf((c0 + hi + kAngEps) / kAngW);
    for (int k = k0; k <= k1; k += G) {
        const int kk = k + gl;
        const bool h = kk > k1 || depth2[stride * ((kk + 2 * kAng) & (kAng - 1))] <= mind2;
        if (!__all_sync(gmask, h)) return false;
    }
    return true;
}
__device__ __forceinline__ bool box_hidden_ang_warp(const float *depth2, int2 g, int4 box, int lane, int stride = 1) {
    return box_hidden_ang<32>(depth2, g, box, lane, 0xffffffffu, stride);
}

// A front-facing edge a -> c (g strictly on its outer side) as seen from g.
// Its angle range goes counter-clockwise from c to a; n is its line's normal,
// with n . (a - g) = N > 0 and n . u > 0 for every ray u that meets the edge.
struct EdgeView {
    int nx, ny, ex, ey;  // normal, direction a -> c
    float N2, h2;        // N^2; the line's squared distance, rounded down
    float lo, hi;        // pseudo-angles of c and a, hi unwrapped past lo
    float c2, a2;        // their squared distances
    float sc, sa;        // and their places along the line, 0 at the foot of g
    int k0, k1;          // bins its closed angle range touches
};
__device__ __forceinline__ bool edge_view(int2 g, int4 e, EdgeView &v) {
    const int ax = e.x - g.x, ay = e.y - g.y, cx = e.z - g.x, cy = e.w - g.y;
    const int N = cross32(cx, cy, ax, ay);  // = -orient(a, c, g)
    if (N <= 0) return false;
    v.ex = e.z - e.x;
    v.ey = e.w - e.y;
    v.nx = -v.ey;
    v.ny = v.ex;
    v.N2 = (float)N * (float)N;
    v.h2 = __fdividef(v.N2, (float)v.ex * (float)v.ex + (float)v.ey * (float)v.ey) * (1.f - 1e-5f);
    v.lo = pang((float)cx, (float)cy);
    v.hi = v.lo + pang_span(v.lo, pang((float)ax, (float)ay));
    v.c2 = (float)cx * (float)cx + (float)cy * (float)cy;
    v.a2 = (float)ax * (float)ax + (float)ay * (float)ay;
    v.sc = (float)v.ex * (float)cx + (float)v.ey * (float)cy;
    v.sa = (float)v.ex * (float)ax + (float)v.ey * (float)ay;
    v.k0 = (int)floorf((v.lo - kAngEps) / kAngW);
    v.k1 = (int)floorf((v.hi + kAngEps) / kAngW);
    return true;
}

// Edge v enters bin k. The crossing distance along the line is convex in the
// ray's angle, so over the rays of the bin that meet the edge it is largest at
// an end of their range, and smallest there too unless the foot of g lies
// between. A bin wholly inside the edge's range takes the larger end as its
// full-blocking bound; every bin the range touches takes the smallest distance
// as a lower bound of where a ray can first meet an obstacle: a ray enters an
// obstacle through a front-facing edge or a vertex of one. Boundary rays are
// exact multiples of 1/kAngQ, so their products with n are exact in integers;
// a 1e-5 margin covers the few float roundings of the distances, kAngEps those
// of the range's ends (whose order pang_span keeps).
// check: read a bin first and leave it when the edge does not lower it (saves
// the atomic, costs the load's latency).
template <bool MAPS>
__device__ __forceinline__ void edge_into_bin(const EdgeView &v, int k, float *up, float *low, int stride, bool check) {
    auto at = [&](int mb, float &s) {  // squared crossing distance and place along the line at boundary mb
        const int2 u = boundary_dir(mb);
        const float D = (float)(v.nx * u.x + v.ny * u.y);  // |n| < 2^16, |u| <= kAngQ
        s = (float)(v.ex * u.x + v.ey * u.y);
        return __fdividef(v.N2 * (float)(u.x * u.x + u.y * u.y), D * D);
    };
    const float b0 = (float)k * kAngW, b1 = (float)(k + 1) * kAngW;
    float s0 = v.sc, s1 = v.sa;
    const float f0 = b0 <= v.lo ? v.c2 : at(k, s0), f1 = b1 >= v.hi ? v.a2 : at(k + 1, s1);
    const int slot = stride * ((k + kAng) & (kAng - 1));
    if (b0 >= v.lo + kAngEps && b1 <= v.hi - kAngEps) {
        const float d = fmaxf(f0, f1) * (1.f + 1e-5f);
        if (!check || up[slot] > d) atomicMin((int *)up + slot, __float_as_int(d));  // non-negative floats order as ints
    }
    if (MAPS) {
        const float f = (s0 > 0.f) != (s1 > 0.f) ? v.h2 : fminf(f0, f1);
        const float d = fmaxf(f * (1.f - 2e-5f) - 0.05f, 0.f);
        if (!check || low[slot] > d) atomicMin((int *)low + slot, __float_as_int(d));
    }
}

// Edges e0 .. min(e0 + kSrcEdges, end) - 1 into the map of a generator at g, one warp: a
// lane views an edge, then the bins they span are dealt to the lanes evenly (a
// wall next to the generator spans hundreds, a far one two or three). With up
// to check_most bins in all, they are read before they are written (far edges
// lower few bins; the wide ones are near and lower most).
constexpr int kSrcEdges = 16;
template <bool MAPS>
__device__ __forceinline__ void insert_edges_warp(const DevScene &ds, float *up, float *low, int2 g, int e0, int end,
                                                  int stride, int check_most) {
    const int lane = threadIdx.x & 31;
    EdgeView v = {};
    int span = 0;
    if (lane < kSrcEdges && e0 + lane < end && edge_view(g, __ldg(ds.edges + e0 + lane), v))
        span = v.k1 - v.k0 + 1;
    int incl = span;
#pragma unroll
    for (int o = 1; o < kSrcEdges; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(0xffffffffu, incl, kSrcEdges - 1);
    for (int r0 = 0; r0 < total; r0 += 32) {
        const int r = r0 + lane;
        int own = 0;  // the first edge whose bins end beyond r
#pragma unroll
        for (int o = kSrcEdges / 2; o > 0; o >>= 1)
            if (__shfl_sync(0xffffffffu, incl, own + o - 1) <= r) own += o;
        own = min(own, kSrcEdges - 1);
        EdgeView o;
        auto take = [&](float x) { return __shfl_sync(0xffffffffu, x, own); };
        o.ex = __shfl_sync(0xffffffffu, v.ex, own);
        o.ey = __shfl_sync(0xffffffffu, v.ey, own);
        o.nx = -o.ey;
        o.ny = o.ex;
        o.N2 = take(v.N2);
        o.h2 = take(v.h2);
        o.lo = take(v.lo);
        o.hi = take(v.hi);
        o.c2 = take(v.c2);
        o.a2 = take(v.a2);
        o.sc = take(v.sc);
        o.sa = take(v.sa);
        const int k = r - __shfl_sync(0xffffffffu, incl - span - v.k0, own);
        if (r < total) edge_into_bin<MAPS>(o, k, up, low, stride, total <= check_most);
    }
}

// One warp inserts polygon q's front-facing edges into the depth map: up to four
// edges one after another, every lane with all of them, the bins spread over the
// lanes; more are dealt (flood of the 3400 polygons, five edges each on average,
// 3150 us one after another, 2420 dealt; of the 160 x 160 maze 756 and 815).
template <bool MAPS>
__device__ void insert_polygon_warp(const DevScene &ds, float *depth2, float *lo2, int2 g, int q, int lane) {
    const int e0 = ds.poly_off[q], e1 = ds.poly_off[q + 1];
    static_assert(kMaxPolyVerts <= kSrcEdges, "a warp takes a polygon's edges at once");
    if (e1 - e0 > 4) {
        insert_edges_warp<MAPS>(ds, depth2, lo2, g, e0, e1, 1, 1 << 30);
        return;
    }
    for (int e = e0; e < e1; ++e) {
        EdgeView v;
        if (!edge_view(g, __ldg(ds.edges + e), v)) continue;
        for (int k = v.k0 + lane; k <= v.k1; k += 32) edge_into_bin<MAPS>(v, k, depth2, lo2, 1, true);
    }
}

// Floods generator g of scene ds: one CTA, a breadth-first level at a time.
// MAPS: also keep g's depth map (with the lower-bound bins) for the pixel pass.
template <bool MAPS>
__device__ void flood_one(const DevScene &ds, FloodSmem &sm, unsigned *fdyn, int g) {
    const int tid = threadIdx.x;
    const int ntiles = ds.tiles_x * ds.tiles_y, words = (ntiles + 31) / 32;
    const int pwords = ds.n_poly <= kFloodPolyBits ? (ds.n_poly + 31) / 32 : 0;
    unsigned *visited = fdyn, *seen = fdyn + words;  // tiles reached; polygons inserted
    // with maps: lower bound of the squared distance at which a ray of each
    // bin can first meet an obstacle (after the bitmaps in dynamic smem)
    float *lo2 = reinterpret_cast<float *>(fdyn + words + pwords);
    const int tpx = ds.tile * (ds.S * ds.Wx / ds.Nx), tpy = ds.tile * (ds.S * ds.Wy / ds.Ny);
    // mode 3 floods from geometry alone (every generator, no cone): it runs
    // before the vertex costs exist, and the pixel pass applies cost and cone
    const bool geometric = ds.flood_mode == 3;
    constexpr bool maps = MAPS;
    if (ds.gen_map_ok && tid == 0) ds.gen_map_ok[g] = 0;  // set again when the map is complete
    SPM_T0();
    if (!geometric && !(ds.gen_costf[g] < INFINITY)) return;
    const int kind = ds.gen_kind[g];
    const int ct = kind == kVert && !geometric ? ds.gen_ctype[g] : kConeNone;
    if (ct == kConeEmpty) return;
    if (kind == kSegI) {
        if (tid == 0) push_global(ds, g);
        return;
    }
    const int2 gl = ds.gen_lat[g];
    const int4 cone = ct != kConeNone ? ds.gen_cone[g] : make_int4(0, 0, 0, 0);
    const int tx = gl.x >= 0 ? gl.x / tpx : -1, ty = gl.y >= 0 ? gl.y / tpy : -1;
    __syncthreads();  // the previous generator is done with smem
    for (int w = tid; w < words + pwords; w += kFloodThreads) fdyn[w] = 0u;
    for (int k = tid; k < kAng; k += kFloodThreads) sm.depth2[k] = INFINITY;
    if (maps)
        for (int k = tid; k < kAng; k += kFloodThreads) lo2[k] = INFINITY;
    if (tid == 0) {
        sm.cnt[0] = 0;
        sm.overflow = 0;
        sm.n_ins = 0;
        sm.ins_dropped = 0;
    }
    __syncthreads();
    // seeds: every tile whose closed area contains g (up to 4 when g lies on tile edges)
    if (tid < 4) {
        const int sx = tx - (tid & 1), sy = ty - ((tid >> 1) & 1);
        if (tx >= 0 && ty >= 0 && sx >= 0 && sy >= 0 && sx < ds.tiles_x && sy < ds.tiles_y) {
            const int4 a4 = tile_area(ds, sx, sy);
            if (gl.x >= a4.x && gl.x <= a4.z && gl.y >= a4.y && gl.y <= a4.w) {
                const int t0 = sy * ds.tiles_x + sx;
                if (!(atomicOr(&visited[t0 >> 5], 1u << (t0 & 31)) & (1u << (t0 & 31))))
                    sm.front[0][atomicAdd(&sm.cnt[0], 1)] = t0;
            }
        }
    }
    __syncthreads();
    SPM_LAP(0);
    if (sm.cnt[0] == 0) {  // g outside every tile: scanned by all tiles instead
        if (tid == 0) push_global(ds, g);
        return;
    }
#ifdef SPM_COUNT
    int n_tests = 0, n_levels = 0;
#endif
    int p = 0;
    for (;;) {
        if (sm.overflow) {  // a level outgrew the frontier: every tile scans g instead
            if (tid == 0) {
                push_global(ds, g);
                SPM_CNT(13, 1);
            }
            break;
        }
        const int nc = min(sm.cnt[p], kFront);
        if (nc == 0) break;
        const int *cur = sm.front[p];
        // A: the polygons in the frontier tiles' bins enter the depth map
        for (int q = tid; q < nc * 16; q += kFloodThreads) {  // (tile, one of its first 16 bins)
            const int i = q >> 4, j = q & 15;
            const int t = cur[i];
            const int4 area = tile_area(ds, t % ds.tiles_x, t / ds.tiles_x);
            const int bx0 = max(0, (area.x - ds.bin_x0) / ds.bin_size), by0 = max(0, (area.y - ds.bin_y0) / ds.bin_size);
            const int bx1 = min(ds.bin_nx - 1, (area.z - ds.bin_x0) / ds.bin_size);
            const int by1 = min(ds.bin_ny - 1, (area.w - ds.bin_y0) / ds.bin_size);
            const int nbx = bx1 - bx0 + 1, nby = by1 - by0 + 1;
            for (int jj = j; jj < nbx * nby; jj += 16) {
                const int bin = (by0 + jj / nbx) * ds.bin_nx + bx0 + jj % nbx;
                const int e = __ldg(ds.bin_start + bin + 1);
                for (int it = __ldg(ds.bin_start + bin); it < e; ++it) {
                    const int poly = __ldg(reinterpret_cast<const int *>(ds.bin_recs + it) + 4);
                    if (pwords) {
                        const unsigned bit = 1u << (poly & 31);
                        if (atomicOr(&seen[poly >> 5], bit) & bit) continue;
                    }
                    const int slot = atomicAdd(&sm.n_ins, 1);
                    if (slot < kInsCap) sm.ins[slot] = poly;  // beyond the cap: left out of the map
                    else sm.ins_dropped = 1;
                }
            }
        }
        __syncthreads();
        SPM_LAP(1);
        const int ni = min(sm.n_ins, kInsCap);
        for (int q = tid >> 5; q < ni; q += kFloodThreads / 32)
            insert_polygon_warp<MAPS>(ds, sm.depth2, lo2, gl, sm.ins[q], tid & 31);
        __syncthreads();
        SPM_LAP(2);
#ifdef SPM_TIME
        spm_acc_[6] += 1;   // levels
        spm_acc_[7] += ni;  // polygons inserted
#endif
        // B: cone and depth-map test per frontier tile, a warp per tile
        for (int i = tid >> 5; i < nc; i += kFloodThreads / 32) {
            const int t = cur[i];
            const int4 area = tile_area(ds, t % ds.tiles_x, t / ds.tiles_x);
            int f = 2;
            if (cone_meets_box(ct, cone, gl, area)) {
                const bool inside = gl.x >= area.x && gl.x <= area.z && gl.y >= area.y && gl.y <= area.w;
                f = !inside && box_hidden_ang_warp(sm.depth2, gl, area, tid & 31) ? 1 : 0;
            }
            if ((tid & 31) == 0) sm.flag[i] = f;
        }
        if (tid == 0) {
            sm.cnt[p ^ 1] = 0;
            sm.n_ins = 0;
        }
        __syncthreads();
        SPM_LAP(3);
        // C: emit visible tiles, queue their fresh 8-neighbours
        int *nxt = sm.front[p ^ 1];
        for (int q = tid; q < nc * 9; q += kFloodThreads) {
            const int i = q / 9, k = q - 9 * i;
            const int f = sm.flag[i];
#ifdef SPM_COUNT
            if (k == 4 && f != 2) {
                SPM_CNT(11, 1);
                SPM_CNT(12, f == 0 ? 1 : 0);
            }
#endif
            if (f) continue;
            const int t = cur[i];
            if (k == 4) {
                const int slot = atomicAdd(&ds.flood_counts[0], 1);
                if (slot < ds.pair_cap) {
                    ds.pairs[slot] = make_int2(t, g);
                    atomicAdd(&ds.tile_count[t], 1);
                } else {
                    atomicOr(&ds.flood_counts[2], 1);
                }
                continue;
            }
            const int nx = t % ds.tiles_x + k % 3 - 1, ny = t / ds.tiles_x + k / 3 - 1;
            if (nx < 0 || ny < 0 || nx >= ds.tiles_x || ny >= ds.tiles_y) continue;
            const int nt = ny * ds.tiles_x + nx;
            if (atomicOr(&visited[nt >> 5], 1u << (nt & 31)) & (1u << (nt & 31))) continue;
            const int slot = atomicAdd(&sm.cnt[p ^ 1], 1);
            if (slot < kFront) nxt[slot] = nt;
            else sm.overflow = 1;
        }
#ifdef SPM_COUNT
        if (tid == 0) {
            ++n_levels;
            for (int i = 0; i < nc; ++i) n_tests += sm.flag[i] != 2;
        }
#endif
        __syncthreads();
        SPM_LAP(4);
        p ^= 1;
    }
#ifdef SPM_COUNT
    if (tid == 0) {
        SPM_CNT_MAX(14, n_tests);
        SPM_CNT_MAX(15, n_levels);
    }
#endif
    // keep the depth map for the pixel pass when it holds every polygon of
    // the reached tiles (no frontier overflow, nothing left out)
    if (maps && !sm.overflow && !sm.ins_dropped) {
        float2 *mp = ds.gen_maps + (size_t)g * kAng;
        for (int k = tid; k < kAng; k += kFloodThreads) mp[k] = make_float2(sm.depth2[k], lo2[k]);
        if (tid == 0) ds.gen_map_ok[g] = 1;
    }
    SPM_LAP(5);
    SPM_TFLUSH();
}

// Geometric culling of generator g without the walk: one CTA enters every
// polygon edge into its map and tests every tile against the complete map. In
// an open scene a generator reaches much of the grid, and the walk's levels
// (four barriers each, the whole grid's width deep) cost far more: first
// compute of the 1024^2 polygons, 1188 generators, 1.2 ms of walks.
// The result is a bit per tile and vertex (a superset of what the walk
// reaches), turned into the kept lists where they fit: with bits alone there is
// no capacity to outgrow (8836 tiles of the 1501^2 polygons hold 5 M pairs,
// over the lists' 4 M: every block scanned), with lists a tile's culling skips
// what it does not see (batch of 64: 1.6 ms of pixel pass against 1.9).
template <bool MAPS>
__device__ void flood_direct(const DevScene &ds, float *up, float *low, int g) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gl8 = lane & 7;
    const int ntiles = ds.tiles_x * ds.tiles_y, v = g - ds.n_src;
    const int2 gl = ds.gen_lat[g];
    __syncthreads();  // the previous generator is done with smem
    for (int k = tid; k < kAng; k += kFloodThreads) up[k] = low[k] = INFINITY;
    __syncthreads();
    for (int e = warp * kSrcEdges; e < ds.n_edge; e += kFloodThreads / 32 * kSrcEdges)
        insert_edges_warp<MAPS>(ds, up, low, gl, e, ds.n_edge, 1, 1 << 30);
    __syncthreads();
    const unsigned gmask = 0xffu << (lane & 24);
    for (int t0 = warp * 4; t0 < ntiles; t0 += kFloodThreads / 32 * 4) {
        const int t = t0 + (lane >> 3);
        if (t >= ntiles) continue;  // whole groups
        const int4 area = tile_area(ds, t % ds.tiles_x, t / ds.tiles_x);
        const bool inside = gl.x >= area.x && gl.x <= area.z && gl.y >= area.y && gl.y <= area.w;
        const bool seen = inside || !box_hidden_ang<8>(up, gl, area, gl8, gmask, 1);
        if (seen && gl8 == 0) atomicOr(&ds.vert_mask[(size_t)t * ds.vert_words + (v >> 5)], 1u << (v & 31));
    }
    if (MAPS) {
        float2 *mp = ds.gen_maps + (size_t)g * kAng;
        for (int k = tid; k < kAng; k += kFloodThreads) mp[k] = make_float2(up[k], low[k]);
    }
    if (tid == 0 && ds.gen_map_ok) ds.gen_map_ok[g] = MAPS ? 1 : 0;
}

// Resident CTAs take the obstacle vertices [g0, g1) from the work counter.
template <bool MAPS>
__global__ void __launch_bounds__(kFloodThreads, 6) k_flood_direct(const __grid_constant__ DevScene ds, int g0, int g1,
                                                                   int unless) {
    __shared__ float up[kAng], low[kAng];
    __shared__ int next_g;
    if (kept_already(ds, unless)) return;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) next_g = g0 + atomicAdd(&ds.flood_counts[3], 1);
        __syncthreads();
        if (next_g >= g1) break;
        flood_direct<MAPS>(ds, up, low, next_g);
    }
}

// The kept lists from the bits: a warp a tile counts them, and after the scan
// (static_tile_start) writes the list, in order; static_counts[3] says whether
// they fit. Up to kBitsOnly words a tile they would save a block nothing -- it
// takes 32 entries at a time -- and the first compute does without them (and
// saves the counts in the sources' first kernel: rectangles 256^2 130 -> 120 us).
constexpr int kBitsOnly = 2;
__global__ void k_bits_count(const __grid_constant__ DevScene ds, int unless) {
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (t >= ds.tiles_x * ds.tiles_y || kept_already(ds, unless)) return;  // whole warps
    int n = 0;
    for (int w = lane; w < ds.vert_words; w += 32) n += __popc(ds.vert_mask[(size_t)t * ds.vert_words + w]);
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0) ds.tile_count[t] = n;
}

__global__ void k_bits_fill(const __grid_constant__ DevScene ds, int unless) {
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    const int ntiles = ds.tiles_x * ds.tiles_y;
    if (t >= ntiles || kept_already(ds, unless)) return;  // whole warps
    const bool fit = ds.static_tile_start[ntiles] <= ds.pair_cap;
    if (t == 0 && lane == 0) ds.static_counts[3] = fit;
    if (!fit) return;
    int at = ds.static_tile_start[t];
    for (int w0 = 0; w0 < ds.vert_words; w0 += 32) {
        const int w = w0 + lane;
        const uint32_t bits = w < ds.vert_words ? ds.vert_mask[(size_t)t * ds.vert_words + w] : 0u;
        int incl = __popc(bits);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        int slot = at + incl - __popc(bits);
        for (uint32_t m = bits; m; m &= m - 1) ds.static_tile_items[slot++] = ds.n_src + 32 * w + __ffs(m) - 1;
        at += __shfl_sync(0xffffffffu, incl, 31);
    }
}

// Direct culling of the sources (generators [0, n_src)) in the geometric
// mode: few generators, each reaching much of the grid, which one CTA per
// generator would walk a breadth-first level at a time. Instead every
// polygon edge enters each source's depth map at once (a warp per source and
// sixteen edges, atomics into the source's map in global memory), and then every tile
// is tested against the complete maps at once (a warp a tile), which gives the
// tile a bit per source. That is a superset of what the walk reaches -- the
// walk also stops at tiles cut off by hidden ones -- and every tile where the
// source can win is still in it: the map only hides points that lie beyond an
// obstacle interior on their ray. With every polygon in it the map is
// complete, and the pixel pass may use it.
__device__ __forceinline__ bool src_on_grid(const DevScene &ds, int g) {
    const int2 gl = ds.gen_lat[g];
    return ds.gen_kind[g] != kSegI && gl.x >= 0 && gl.y >= 0 && gl.x <= ds.Nx * ds.pitch_x && gl.y <= ds.Ny * ds.pitch_y;
}

// The obstacle vertices' flood is done (keep = 1, 2: as bits alone; 0: some
// time ago): its counts are saved and its tag is set. restore: the counts a
// compute's sources start from, the global list and the overflow flag as that
// flood left them. One whole warp.
__device__ __forceinline__ void kept_counts(const DevScene &ds, int keep, int unless, bool restore) {
    const int k = threadIdx.x & 31;
    const bool built = keep && !kept_already(ds, unless);
    __syncwarp();  // every lane has read the tag
    if (k < 3 && built) ds.static_counts[k] = ds.flood_counts[k];
    if (k == 3 && built && keep == 2) ds.static_counts[3] = 0;
    if (k == kKeptTag && built) ds.flood_counts[k] = kept_tag(ds);
    if (k < 4 && restore) ds.flood_counts[k] = k == 1 || k == 2 ? ds.static_counts[k] : 0;
}

// Before the sources' culling: empty maps and the counts they start from.
__device__ __forceinline__ void src_prep(const DevScene &ds, int i0, int stride, int keep, int unless) {
    const bool maps = ds.use_maps && ds.gen_maps;
    for (int i = i0; i < ds.n_src * kAng; i += stride) {
        ds.gen_maps[i] = make_float2(INFINITY, INFINITY);
        if (i < ds.n_src) ds.gen_map_ok[i] = maps && src_on_grid(ds, i);  // complete by the time the pixel pass reads it
    }
    if (i0 < 32) kept_counts(ds, keep, unless, true);
}

template <bool MAPS>
__device__ __forceinline__ void src_insert(const DevScene &ds, int g, int e0) {
    if (!src_on_grid(ds, g)) return;  // the same for the whole warp
    float *mp = reinterpret_cast<float *>(ds.gen_maps + (size_t)g * kAng);
    insert_edges_warp<MAPS>(ds, mp, mp + 1, ds.gen_lat[g], e0, ds.n_edge, 2, 64);
}

// Word w of tile t's bits: a warp, its groups of kSrcGrp lanes a source each
// (most tiles span few bins). Segment interiors and sources off the grid are
// candidates of every tile. (A warp that went through all of a tile's words took
// 2.9 ms for 4000 sources on the 64 tiles of 256^2 rectangles.)
constexpr int kSrcGrp = 8;
__device__ __forceinline__ void src_tile(const DevScene &ds, int t, int w) {
    const int lane = threadIdx.x & 31, gl8 = lane % kSrcGrp, grp = lane / kSrcGrp;
    const unsigned gmask = ((1u << kSrcGrp) - 1u) << (grp * kSrcGrp);
    const int4 area = tile_area(ds, t % ds.tiles_x, t / ds.tiles_x);
    const int mine = 32 * w + lane;  // one load for the word's sources
    const int2 lat = mine < ds.n_src ? ds.gen_lat[mine] : make_int2(0, 0);
    const bool on = mine < ds.n_src && src_on_grid(ds, mine);
    const bool inside = lat.x >= area.x && lat.x <= area.z && lat.y >= area.y && lat.y <= area.w;
    const unsigned every = __ballot_sync(0xffffffffu, mine < ds.n_src && (inside || !on));
    uint32_t bits = every;
    const int n = min(32, ds.n_src - 32 * w);
#pragma unroll 2
    for (int j0 = 0; j0 < n; j0 += 32 / kSrcGrp) {
        const int j = j0 + grp;
        const int2 gl = make_int2(__shfl_sync(0xffffffffu, lat.x, j & 31), __shfl_sync(0xffffffffu, lat.y, j & 31));
        bool seen = false;
        if (j < n && !(every >> j & 1u))
            seen = !box_hidden_ang<kSrcGrp>(reinterpret_cast<const float *>(ds.gen_maps + (size_t)(32 * w + j) * kAng),
                                            gl, area, gl8, gmask, 2);
        const unsigned bal = __ballot_sync(0xffffffffu, seen && gl8 == 0);
#pragma unroll
        for (int q = 0; q < 32 / kSrcGrp; ++q)
            if (bal >> (q * kSrcGrp) & 1u) bits |= 1u << (j0 + q);
    }
    if (lane == 0) ds.src_mask[(size_t)t * ds.src_words + w] = bits;
}

__global__ void k_src_prep(const __grid_constant__ DevScene ds, int keep, int unless) {
    src_prep(ds, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, keep, unless);
}

template <bool MAPS>
__global__ void k_src_insert(const __grid_constant__ DevScene ds) {  // grid: (edges, sources)
    const int e0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kSrcEdges;
    for (int g = blockIdx.y; g < ds.n_src; g += gridDim.y) src_insert<MAPS>(ds, g, e0);
}

__global__ void k_src_tiles(const __grid_constant__ DevScene ds) {
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t < ds.tiles_x * ds.tiles_y) src_tile(ds, t, blockIdx.y);  // whole warps
}

// Automatic mode: flood only sparse visibility graphs (mazes); a dense one
// marks the lists unavailable and every tile scans every generator.
__device__ __forceinline__ bool flood_declined(const DevScene &ds) {
    if (ds.flood_mode != 0) return false;
    const double pairs = (double)ds.n_gen * (double)max(ds.n_vert, 1);
    return (double)ds.in_start[ds.n_vert] > 0.01 * pairs;
}

// Resident CTAs take generators from a work counter (flood_counts[3]) as
// they finish: flood depths vary widely, so a fixed stride would leave the
// kernel waiting for the CTAs that drew several deep generators.
// Generators [g0, g1) are flooded.
template <bool MAPS>
__global__ void __launch_bounds__(kFloodThreads, MAPS ? 6 : 8) k_flood(DevScene ds, int g0, int g1, int unless) {
    extern __shared__ unsigned fdyn[];
    __shared__ FloodSmem sm;
    __shared__ int next_g;
    if (kept_already(ds, unless)) return;
    if (flood_declined(ds)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) ds.flood_counts[2] = 1;
        return;
    }
    for (;;) {
        if (threadIdx.x == 0) next_g = g0 + atomicAdd(&ds.flood_counts[3], 1);
        __syncthreads();
        const int g = next_g;
        __syncthreads();  // next_g is rewritten for the next generator
        if (g >= g1) break;
        flood_one<MAPS>(ds, sm, fdyn, g);
    }
}

// After the obstacle vertices' flood (keep) its counts are saved; before the
// sources' flood (keep = 0) the lists start empty, the global list after the
// vertices' entries, the overflow flag as the vertices' flood left it, and the
// work counter from zero.
__global__ void k_flood_static(DevScene ds, int keep, int unless) {
    const int ntiles = ds.tiles_x * ds.tiles_y;
    if (!keep)
        for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < ntiles; t += gridDim.x * blockDim.x) ds.tile_count[t] = 0;
    if (blockIdx.x == 0 && threadIdx.x < 32) kept_counts(ds, keep, unless, !keep);
}



// Batched form: every (scene, generator) of the batch, one CTA each.
template <class T>
__device__ __forceinline__ int scene_of_b(const T *off, int n, T x) {
    int lo = 0, hi = n;  // last scene with off[s] <= x
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= x) lo = mid;
        else hi = mid;
    }
    return lo;
}

template <bool ANY_MAPS>  // some scene of the batch keeps depth maps
__global__ void __launch_bounds__(kFloodThreads, ANY_MAPS ? 6 : 8) k_flood_b(const __grid_constant__ BatchDev b) {
    extern __shared__ unsigned fdyn[];
    __shared__ FloodSmem sm;
    const int total = b.flood_off[b.n];
    for (int i = blockIdx.x; i < total; i += gridDim.x) {  // (scene, generator) tasks: sources only when reusing
        const int sc = scene_of_b(b.flood_off, b.n, i);
        const DevScene &ds = b.scenes[sc];
        if (!ds.use_flood || ds.flood_mode == 2) continue;
        if (flood_declined(ds)) {
            if (threadIdx.x == 0) ds.flood_counts[2] = 1;
            continue;
        }
        if (ANY_MAPS && ds.use_maps && ds.gen_maps) flood_one<true>(ds, sm, fdyn, i - b.flood_off[sc]);
        else flood_one<false>(ds, sm, fdyn, i - b.flood_off[sc]);
    }
}

// Per-scene list state before a batched flood: counts zeroed, or the lists
// marked unavailable for scenes that scan; the depth maps of directly culled
// sources emptied.
__global__ void k_flood_reset_b(const __grid_constant__ BatchDev b) {
    const int total = b.tile_off[b.n];
    const long long nmap = b.src_map_off[b.n];
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total + b.n + nmap;
         i += gridDim.x * (long long)blockDim.x) {
        if (i >= total + b.n) {
            const long long m = i - total - b.n;
            const int sc = scene_of_b(b.src_map_off, b.n, m);
            const DevScene &ds = b.scenes[sc];
            const long long e = m - b.src_map_off[sc];
            ds.gen_maps[e] = make_float2(INFINITY, INFINITY);
            if (e % kAng == 0) ds.gen_map_ok[e / kAng] = ds.use_maps && src_on_grid(ds, (int)(e / kAng));
        } else if (i < total) {
            const int oi = scene_of_b(b.tile_off, b.n, (int32_t)i), sc = b.order[oi];
            b.scenes[sc].tile_count[i - b.tile_off[oi]] = 0;
        } else {  // reusing scenes: the global list after the vertices' entries
            const DevScene &ds = b.scenes[(int)(i - total)];
            const bool on = ds.use_flood && ds.flood_mode != 2;
            // a kept part of another tuning (only a batch recorded in its
            // caller's graph meets one): the scene scans every generator
            // (all three loads at once)
            const int tag = ds.flood_reuse ? ds.flood_counts[kKeptTag] : 0;
            const int globals = ds.flood_reuse ? ds.static_counts[1] : 0, over = ds.flood_reuse ? ds.static_counts[2] : 0;
            const bool kept = tag == kept_tag(ds);
            ds.flood_counts[0] = 0;
            ds.flood_counts[1] = kept ? globals : 0;
            ds.flood_counts[2] = kept ? over : (on && !ds.flood_reuse ? 0 : 1);
            ds.flood_counts[3] = 0;
            if (on && !ds.flood_reuse) ds.flood_counts[kKeptTag] = 0;  // its flood overwrites the kept part
        }
    }
}

// Batched direct culling of sources: (scene, source, edges) and then
// (scene, tile) warp tasks over the scenes with src_direct.
template <bool ANY_MAPS>
__global__ void k_src_insert_b(const __grid_constant__ BatchDev b) {
    const long long n = b.src_ins_off[b.n];
    for (long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; w < n;
         w += (gridDim.x * (long long)blockDim.x) >> 5) {
        const int sc = scene_of_b(b.src_ins_off, b.n, w);
        const DevScene &ds = b.scenes[sc];
        const int i = (int)(w - b.src_ins_off[sc]), per = (ds.n_edge + kSrcEdges - 1) / kSrcEdges;
        if (ANY_MAPS && ds.use_maps) src_insert<true>(ds, i / per, i % per * kSrcEdges);
        else src_insert<false>(ds, i / per, i % per * kSrcEdges);
    }
}

__global__ void k_src_tiles_b(const __grid_constant__ BatchDev b) {
    const long long n = b.src_tile_off[b.n];
    for (long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; w < n;
         w += (gridDim.x * (long long)blockDim.x) >> 5) {
        const int sc = scene_of_b(b.src_tile_off, b.n, w);
        const DevScene &ds = b.scenes[sc];
        const long long i = w - b.src_tile_off[sc];
        src_tile(ds, (int)(i / ds.src_words), (int)(i % ds.src_words));
    }
}

// Exclusive scan of tile_count into tile_start (one CTA), then fill.
// The per-tile CSR of the pairs: the scene's lists, or (to_static) the kept
// lists of the obstacle vertices' flood.
// Each thread scans a run of consecutive tiles, a multiple of four long so
// that a full run moves by 16-byte loads and stores (runs of 16 on the
// 4096^2 maze: four loads instead of sixteen strided ones).
__device__ void tiles_scan_block(const DevScene &ds, bool to_static = false) {
    __shared__ long long wsum[32];
    int32_t *start = to_static ? ds.static_tile_start : ds.tile_start;
    const int n = ds.tiles_x * ds.tiles_y;
    constexpr int kRun = 16;  // vector path: runs of exactly kRun (4 x int4)
    const int per = ((n + blockDim.x - 1) / blockDim.x + 3) & ~3;
    const int lo = threadIdx.x * per, hi = min(n, lo + per);
    const bool vec = per == kRun && hi - lo == kRun;
    int4 c[kRun / 4];
    long long s = 0;
    if (vec) {
#pragma unroll
        for (int k = 0; k < kRun / 4; ++k) {
            c[k] = reinterpret_cast<const int4 *>(ds.tile_count + lo)[k];
            s += (long long)c[k].x + c[k].y + c[k].z + c[k].w;
        }
    } else {
        for (int i = lo; i < hi; ++i) s += ds.tile_count[i];
    }
    long long run = cta_exclusive_scan(s, wsum);  // every thread, once
    if (vec) {
#pragma unroll
        for (int k = 0; k < kRun / 4; ++k) {
            int4 o;
            o.x = (int32_t)run;
            run += c[k].x;
            o.y = (int32_t)run;
            run += c[k].y;
            o.z = (int32_t)run;
            run += c[k].z;
            o.w = (int32_t)run;
            run += c[k].w;
            reinterpret_cast<int4 *>(start + lo)[k] = o;
            reinterpret_cast<int4 *>(ds.tile_count + lo)[k] = make_int4(0, 0, 0, 0);  // reused as fill cursors
        }
    } else {
        for (int i = lo; i < hi; ++i) {
            start[i] = (int32_t)run;
            run += ds.tile_count[i];
            ds.tile_count[i] = 0;  // reused as fill cursor
        }
    }
    if (hi == n && lo < hi) start[n] = (int32_t)run;
    if (threadIdx.x == 0 && n == 0) start[0] = 0;
}

__device__ __forceinline__ void tiles_fill(const DevScene &ds, int i0, int stride, bool to_static = false) {
    const int32_t *start = to_static ? ds.static_tile_start : ds.tile_start;
    int32_t *items = to_static ? ds.static_tile_items : ds.tile_items;
    const int np = min(ds.flood_counts[0], ds.pair_cap);
    for (int i = i0; i < np; i += stride) {
        const int2 pr = ds.pairs[i];
        const int slot = atomicAdd(&ds.tile_count[pr.x], 1);
        items[start[pr.x] + slot] = pr.y;
    }
}

__global__ void __launch_bounds__(1024) k_tiles_scan(DevScene ds, int to_static, int unless) {
    if (!kept_already(ds, unless)) tiles_scan_block(ds, to_static);
}

__global__ void k_tiles_fill(DevScene ds, int to_static, int unless) {
    if (kept_already(ds, unless)) return;
    tiles_fill(ds, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, to_static);
}

// batched: one CTA per scene for the scan, a row of CTAs per scene for the fill
__global__ void __launch_bounds__(1024) k_tiles_scan_b(const __grid_constant__ BatchDev b) {
    const DevScene &ds = b.scenes[blockIdx.x];
    if (ds.use_flood && ds.flood_mode != 2 && !ds.src_direct) tiles_scan_block(ds);
}

__global__ void k_tiles_fill_b(const __grid_constant__ BatchDev b) {
    const DevScene &ds = b.scenes[blockIdx.y];
    if (ds.use_flood && ds.flood_mode != 2 && !ds.src_direct)
        tiles_fill(ds, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

}  // namespace

// dynamic part: visited tiles, inserted polygons, and with maps the lower-bound bins
size_t flood_smem_bytes(int tiles, int polys, bool maps) {
    return sizeof(unsigned) * (size_t)((tiles + 31) / 32 + (polys <= kFloodPolyBits ? (polys + 31) / 32 : 0) +
                                       (maps ? kAng : 0));
}

bool flood_possible(int tiles, int polys) {
    return flood_smem_bytes(tiles, polys, true) + sizeof(FloodSmem) <= 200 * 1024;
}

// Generators [g0, g1) walked by resident CTAs.
static void flood_walk(const DevScene &ds, cudaStream_t st, int g0, int g1, int unless) {
    if (g1 <= g0) return;
    const bool maps = ds.use_maps && ds.gen_maps;
    const size_t smem = flood_smem_bytes(ds.tiles_x * ds.tiles_y, ds.n_poly, maps);
    int per_sm = 0, dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, maps ? k_flood<true> : k_flood<false>, kFloodThreads, smem);
    const int blocks = max(1, min(max(sms, 1) * max(per_sm, 1), g1 - g0));
    if (maps) k_flood<true><<<blocks, kFloodThreads, smem, st>>>(ds, g0, g1, unless);
    else k_flood<false><<<blocks, kFloodThreads, smem, st>>>(ds, g0, g1, unless);
}

// The obstacle vertices' lists, kept for every later compute, up to their
// counts and tag: kept_counts(keep) is what is left to do, with what this
// returns. unless: kept_already's.
static int flood_kept(const DevScene &scene, cudaStream_t st, int unless) {
    DevScene ds = scene;
    ds.vert_bits = flood_verts_direct(ds) ? 1 : 0;
    const int ntiles = ds.tiles_x * ds.tiles_y;
    const size_t clear = (size_t)ntiles * (ds.vert_bits ? ds.vert_words : 1);
    k_kept_reset<<<(int)std::max<size_t>(1, std::min<size_t>((clear + 255) / 256, 152 * 8)), 256, 0, st>>>(ds, unless);
    if (!ds.vert_bits) {
        flood_walk(ds, st, ds.n_src, ds.n_gen, unless);
        k_tiles_scan<<<1, 1024, 0, st>>>(ds, 1, unless);
        k_tiles_fill<<<152 * 4, 256, 0, st>>>(ds, 1, unless);
        return 1;
    }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int blocks = std::min(max(sms, 1) * 6, ds.n_vert);
    if (ds.use_maps && ds.gen_maps) k_flood_direct<true><<<blocks, kFloodThreads, 0, st>>>(ds, ds.n_src, ds.n_gen, unless);
    else k_flood_direct<false><<<blocks, kFloodThreads, 0, st>>>(ds, ds.n_src, ds.n_gen, unless);
    if (ds.vert_words <= kBitsOnly) return 2;
    k_bits_count<<<(ntiles + 7) / 8, 256, 0, st>>>(ds, unless);
    k_tiles_scan<<<1, 1024, 0, st>>>(ds, 1, unless);
    k_bits_fill<<<(ntiles + 7) / 8, 256, 0, st>>>(ds, unless);
    return 1;
}

int flood_kept_tag(const DevScene &ds) { return kept_tag(ds); }

int flood_kept_kernels(const DevScene &ds) {
    const int build = !flood_verts_direct(ds) ? 3 + (ds.n_vert > 0) : ds.vert_words <= kBitsOnly ? 2 : 5;
    return build + (flood_sources_direct(ds) ? 0 : 1);
}

void launch_flood_kept(const DevScene &ds, cudaStream_t st) {
    const int tag = kept_tag(ds), keep = flood_kept(ds, st, tag);
    k_flood_static<<<1, 32, 0, st>>>(ds, keep, tag);
}

void launch_flood(const DevScene &ds, cudaStream_t st, FloodStatic how) {
    const int ntiles = ds.tiles_x * ds.tiles_y;
    if (ds.flood_mode == 2) {  // never: the pixel pass scans every generator
        static const int32_t off[4] = {0, 0, 1, 0};
        cudaMemcpyAsync(ds.flood_counts, off, sizeof off, cudaMemcpyHostToDevice, st);
        return;
    }
    const bool maps = ds.use_maps && ds.gen_maps;
    const int sblocks = max(1, min((ntiles + 255) / 256, 152));
    if (how == FloodStatic::kNone) {
        cudaMemsetAsync(ds.tile_count, 0, sizeof(int32_t) * ntiles, st);
        cudaMemsetAsync(ds.flood_counts, 0, sizeof(int32_t) * kFloodCounts, st);  // the tag too: the kept part goes
        flood_walk(ds, st, 0, ds.n_gen, 0);
    } else {
        const int unless = how == FloodStatic::kEnsure ? kept_tag(ds) : 0;
        const int keep = how == FloodStatic::kReuse ? 0 : flood_kept(ds, st, unless);
        if (flood_sources_direct(ds)) {  // a bit per source and tile: nothing to sort
            k_src_prep<<<std::min((ds.n_src * kAng + 255) / 256, 152 * 8), 256, 0, st>>>(ds, keep, unless);
            // ordinary launches: a dependent one would hold SMs, waiting, that
            // the vertex phase beside it needs
            const dim3 grid((ds.n_edge + 4 * kSrcEdges - 1) / (4 * kSrcEdges), std::min(ds.n_src, 65535));
            if (ds.n_edge > 0 && maps) k_src_insert<true><<<grid, 128, 0, st>>>(ds);
            else if (ds.n_edge > 0) k_src_insert<false><<<grid, 128, 0, st>>>(ds);
            k_src_tiles<<<dim3((ntiles + 7) / 8, ds.src_words), 256, 0, st>>>(ds);
            return;
        }
        if (keep) k_flood_static<<<1, 32, 0, st>>>(ds, keep, unless);
        k_flood_static<<<sblocks, 256, 0, st>>>(ds, 0, 0);
        flood_walk(ds, st, 0, ds.n_src, 0);
    }
    k_tiles_scan<<<1, 1024, 0, st>>>(ds, 0, 0);
    k_tiles_fill<<<152 * 4, 256, 0, st>>>(ds, 0, 0);
}

bool flood_sources_fit(const DevScene &ds) {
    const long long ntiles = (long long)ds.tiles_x * ds.tiles_y;
    return ds.gen_maps && ds.n_src > 0 && (long long)ds.n_src * (ds.n_poly + ntiles) <= (1LL << 24);
}
bool flood_sources_direct(const DevScene &ds) { return ds.src_mask && flood_sources_fit(ds); }

// The obstacle vertices without the walk: in open scenes, where a vertex sees
// many others (mazes: 3 tangent edges a vertex, polygon scenes: 8 to 45), and
// while a generator's edges and tiles stay a few thousand.
bool flood_verts_fit(const DevScene &ds) {
    const long long ntiles = (long long)ds.tiles_x * ds.tiles_y;
    return ds.n_vert > 0 && (ds.open_scene || ds.n_edge + ntiles <= 1024) && ds.n_edge + ntiles <= (1 << 17);
}
bool flood_verts_direct(const DevScene &ds) { return ds.vert_mask && flood_verts_fit(ds); }

int src_edge_warps(int n_edge) { return (n_edge + kSrcEdges - 1) / kSrcEdges; }

int flood_smem_attr() {
    const int dyn = 200 * 1024 - (int)sizeof(FloodSmem);
    return cudaFuncSetAttribute(k_flood<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn) == cudaSuccess &&
           cudaFuncSetAttribute(k_flood<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn) == cudaSuccess &&
           cudaFuncSetAttribute(k_flood_b<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn) == cudaSuccess &&
           cudaFuncSetAttribute(k_flood_b<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn) == cudaSuccess;
}

bool flood_batched_direct(const BatchDev &b) { return b.flood_smem > 0 && b.walk_tasks <= 0 && !b.any_lists; }

void launch_flood_batched(const BatchDev &b, cudaStream_t st, long long src_ins, long long src_tiles) {
    k_flood_reset_b<<<152 * 4, 256, 0, st>>>(b);
    if (b.flood_smem <= 0) return;  // every scene scans
    if (b.walk_tasks > 0) {
        if (b.any_maps) k_flood_b<true><<<152 * 8, kFloodThreads, b.flood_smem, st>>>(b);
        else k_flood_b<false><<<152 * 8, kFloodThreads, b.flood_smem, st>>>(b);
    }
    auto wblocks = [](long long warps) { return (int)std::max(1LL, std::min((warps + 7) / 8, 152LL * 16)); };
    if (src_ins > 0) {
        if (b.any_maps) k_src_insert_b<true><<<wblocks(src_ins), 256, 0, st>>>(b);
        else k_src_insert_b<false><<<wblocks(src_ins), 256, 0, st>>>(b);
    }
    if (src_tiles > 0) k_src_tiles_b<<<wblocks(src_tiles), 256, 0, st>>>(b);
    if (!b.any_lists) return;  // no lists but the kept ones
    k_tiles_scan_b<<<b.n, 1024, 0, st>>>(b);
    k_tiles_fill_b<<<dim3(16, b.n), 256, 0, st>>>(b);
}

}  // namespace spm

#ifdef SPM_TIME
// Instrumentation build only: reads and clears the flood's phase clocks.
extern "C" int spm_debug_times_flood(unsigned long long *out8) {
    cudaDeviceSynchronize();
    if (cudaMemcpyFromSymbol(out8, spm::g_time, sizeof(unsigned long long) * 8) != cudaSuccess) return 1;
    unsigned long long z[8] = {0};
    cudaMemcpyToSymbol(spm::g_time, z, sizeof z);
    return 0;
}
#endif

#ifdef SPM_COUNT
// Instrumentation build only: reads and clears this unit's work counters.
extern "C" int spm_debug_counters_flood(unsigned long long *out32) {
    cudaDeviceSynchronize();
    if (cudaMemcpyFromSymbol(out32, spm::g_count, sizeof(unsigned long long) * 32) != cudaSuccess) return 1;
    unsigned long long z[32] = {0};
    cudaMemcpyToSymbol(spm::g_count, z, sizeof z);
    return 0;
}
#endif
