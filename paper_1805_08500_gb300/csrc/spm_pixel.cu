// spm_pixel.cu -- pixel phase of the shortest-path map.
//
// arxiv 1805.08500 Sec. 3.1, Procedure 3 ("Cone"): a pixel that sees generator
// g takes cost(g) + |p - g| when that is smaller than what it holds; Sec. 4:
// a segment interior reaches p through its perpendicular foot. Instead of one
// full-screen pass per generator, one warp owns a block of 16 x 16 pixels and
// gathers only the generators that can win somewhere in it:
//   * free space: the pixels inside obstacles come from the scene's
//     free-space mask (built once, one bit per pixel);
//   * candidates: the list of the block's tile from the flood, or every
//     generator;
//   * cull: finite cost, shadow cone (or perpendicular strip) meets the block,
//     lower bound lb = cost + dist(g, block) below the block's current worst;
//   * order: candidates in order of lb; the warp stops once every pixel's best
//     is <= lb (no later candidate can win);
//   * depth maps (when the flood kept them): a pixel nearer than the lower
//     bound of its bin sees the candidate, one beyond the full-blocking upper
//     bound does not, and only the pixels in between take the exact test below
//     (deciding whole blocks from the bins they span first cost as much as it
//     saved: half of the blocks are neither);
//   * visibility: the warp lists the polygons whose interior may meet the hull
//     of (block, g), and every undecided pixel runs the exact integer
//     separating-axis test against that list (none when the list is empty);
//   * argmin: smaller distance, then smaller id;
//   * output: each lane writes four consecutive pixels of a row with one
//     16-byte store per plane (dist, parent).
#include <cuda_runtime.h>

#include <algorithm>

#include "spm_device.cuh"
#include "spm_internal.h"

namespace spm {
namespace {

constexpr int NT = kPixelThreads;  // threads of the free-space mask's CTAs

// Lower bound of the distance from segment source s's interior to any pixel of
// the box (lattice box, world fbox), or -1 when no pixel's perpendicular foot
// lies strictly inside the segment.
__device__ __forceinline__ float segment_lower_bound(const DevScene &ds, int s, int4 box, float4 fbox) {
    const int4 L = ds.seg_lat[s];
    const long long ux = L.z - L.x, uy = L.w - L.y, den = ux * ux + uy * uy;
    bool all_lo = true, all_hi = true, pos = false, neg = false;
    const float4 F = ds.seg_pos[s];
    const float fx = F.z - F.x, fy = F.w - F.y, il = rsqrtf(fx * fx + fy * fy);
    float mn = INFINITY;
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {  // the box's corners
        const long long num = ((k & 1 ? box.z : box.x) - L.x) * ux + ((k & 2 ? box.w : box.y) - L.y) * uy;
        all_lo &= num <= 0;
        all_hi &= num >= den;
        const float sd = (fx * ((k & 2 ? fbox.w : fbox.y) - F.y) - fy * ((k & 1 ? fbox.z : fbox.x) - F.x)) * il;
        pos |= sd > 0.f;
        neg |= sd < 0.f;
        mn = fminf(mn, fabsf(sd));
    }
    if (all_lo || all_hi) return -1.f;
    return (pos && neg) ? 0.f : mn * 0.999999f;
}

// ---------------------------------------------------------------------------
// One warp, one block of pixels (16 x 16, smaller on small grids), no barrier.
// ---------------------------------------------------------------------------
constexpr int kWarpCand = 160;   // candidates a warp holds before it works them off: nearly every block's at once
                                 // (in parts, a block's true generators may come last: 50 processed where 16 would do)
constexpr int kWarpPoly = 64;    // blocker polygons a warp lists at a time
constexpr int kBlocked = 1 << 15; // an undecided pixel found blocked

// A candidate's flags, above its generator id (below 2^20).
constexpr int kCandId = (1 << 20) - 1;
constexpr int kCandInCone = 1 << 20;  // the whole block lies in the shadow cone (or there is none)
constexpr int kCandMap = 1 << 21;     // its depth map is complete

// The pixels' state lives in shared memory (a lane's eight pixels at
// k * 32 + lane), not in registers: the loops over them stay rolled, nothing
// spills around the exact tests, and more warps are resident.
template <int PX, int PY, int ROW = PX == 1 ? 8 : 4>
struct Shape {                       // a lane's pixels: PX consecutive ones of PY rows
    static constexpr int kPix = PX * PY;
    static constexpr int kRow = ROW;                              // lanes across the block
    static constexpr int kW = PX * kRow, kH = PY * (32 / kRow);   // block size in pixels
};

template <int N>  // pixels a lane
struct WarpSmem {
    float bd[32 * N];            // best distance so far (-inf: not a free pixel of the grid)
    int bi[32 * N];              // and its generator
    float d[32 * N];             // the candidate's distances
    float lb[kWarpCand];         // candidates: least cost + distance over the block
    int cand[kWarpCand];         // generator id and flags
    int3 poly[kWarpPoly];        // blocker polygons: id, first vertex, vertices
    unsigned short item[32 * N]; // undecided pixels, lane * N + k, and kBlocked
};

// One warp's block of pixels. A lane holds PX consecutive pixels (k % PX) of
// PY rows, 32 / kRow apart (k / PX).
struct Block {
    int4 box;    // lattice box of its pixel centres
    int i0, j0;  // its first pixel
    int i1, j1;  // its last pixel within the grid
    int i, j;    // the lane's first pixel
    float worst; // largest best distance of the lane's pixels
    bool lists;  // the candidates come from flooded lists
};

__device__ __forceinline__ float point_dist(float cf, float dx, float dy) { return cf + sqrtf(dx * dx + dy * dy); }
__device__ __forceinline__ float pixel_x(const DevScene &ds, int i) { return ((float)i + 0.5f) * ds.hx; }
__device__ __forceinline__ float pixel_y(const DevScene &ds, int j) { return ((float)j + 0.5f) * ds.hy; }

// The candidates of a tile's pixels: the list culled for the tile, or the kept
// list of obstacle vertices and this compute's entries (each a list, or a bit
// per vertex or source) and the global list, or every generator.
struct TileList {
    const int32_t *a, *l, *gl;       // entries [0, na), [na, nl) and [nl, total)
    const uint32_t *abits, *lbits;   // or the first two parts' bits
    int na, nl, total;
    bool lists;
    __device__ __forceinline__ TileList(const DevScene &ds, int tile, bool culled) {
        lists = ds.use_flood && ds.flood_counts[2] == 0;
        a = l = gl = ds.glob_list;
        abits = lbits = nullptr;
        na = nl = 0;
        total = ds.n_gen;
        if (!lists) return;
        if (culled && ds.cull_on) {
            na = nl = total = ds.cull_count[tile];
            a = ds.cull_items + (size_t)tile * cull_cap(ds.tile);
            if (total >= 0) return;
            na = 0;
        }
        if (ds.static_lists && ds.vert_bits && !ds.static_counts[3]) {
            abits = ds.vert_mask + (size_t)tile * ds.vert_words;
            na = ds.n_vert;
        } else if (ds.static_lists) {
            const int s0 = ds.static_tile_start[tile];
            na = ds.static_tile_start[tile + 1] - s0;
            a = ds.static_tile_items + s0;
        }
        if (ds.static_lists && ds.src_direct) {
            lbits = ds.src_mask + (size_t)tile * ds.src_words;
            nl = na + ds.n_src;
        } else {
            const int l0 = ds.tile_start[tile];
            nl = na + ds.tile_start[tile + 1] - l0;
            l = ds.tile_items + l0;
        }
        total = nl + ds.flood_counts[1];
    }
    // entry e's generator, or false when there is none
    __device__ __forceinline__ bool entry(const DevScene &ds, int e, int &g) const {
        if (e >= total) return false;
        g = e;
        if (!lists) return true;
        const bool first = e < na, second = !first && e < nl;
        const int r = first ? e : second ? e - na : e - nl;
        const uint32_t *bits = first ? abits : second ? lbits : nullptr;
        if (bits) {
            g = first ? r + ds.n_src : r;
            return __ldg(bits + (r >> 5)) >> (r & 31) & 1u;
        }
        g = __ldg((first ? a : second ? l : gl) + r);
        return true;
    }
};

// Generator g as a candidate of the block: its lower bound and flags; false
// when it cannot win anywhere in the block. Most entries of a list go by their
// cost or cone, one 16-byte load.
__device__ __forceinline__ bool block_candidate(const DevScene &ds, int g, const Block &b, float ub, bool maps,
                                                float &lb, int &cand) {
    const int4 q = __ldg(ds.gen_cull + g);
    const float cost = __int_as_float(q.w);
    const int4 box = b.box;
    cand = g;
    if (cost < 0.f) {  // a segment interior
        const float4 fbox = make_float4(pixel_x(ds, b.i0), pixel_y(ds, b.j0), pixel_x(ds, b.i1), pixel_y(ds, b.j1));
        lb = segment_lower_bound(ds, ds.gen_aux[g], box, fbox);
        return lb >= 0.f && lb <= ub;
    }
    const int2 l = make_int2((short)q.x, q.x >> 16);
    const int x0 = box.x - l.x, x1 = box.z - l.x, y0 = box.y - l.y, y1 = box.w - l.y;
    const float dx = (float)max(max(x0, -x1), 0), dy = (float)max(max(y0, -y1), 0);
    // a source lies within a lattice unit of its lattice point, a vertex on it
    const float d2 = fmaf(dx, dx, dy * dy);
    const float d = d2 * rsqrtf(fmaxf(d2, 1e-20f)) - (g < ds.n_src ? 1.f : 0.f);
    lb = (cost + fmaxf(d, 0.f) * ds.inv_S) * 0.999999f;
    // cross(c1, w) and cross(w, c2) are linear in w: their extremes over the
    // box lie at the corners their signs choose (no cone: all zero)
    const int kx = (short)q.y, ky = q.y >> 16, kz = (short)q.z, kw = q.z >> 16;
    const int hi1 = kx * (kx > 0 ? y1 : y0) - ky * (ky > 0 ? x0 : x1);
    const int hi2 = kw * (kw > 0 ? x1 : x0) - kz * (kz > 0 ? y0 : y1);
    if (!(lb <= ub) || !(cost < INFINITY) || (hi1 | hi2) < 0) return false;
    const int lo1 = kx * (kx > 0 ? y0 : y1) - ky * (ky > 0 ? x1 : x0);
    const int lo2 = kw * (kw > 0 ? x0 : x1) - kz * (kz > 0 ? y1 : y0);
    // a ray's two directions are the same: the box would lie on its line
    if ((lo1 | lo2) >= 0 && (q.y != q.z || q.y == 0)) cand |= kCandInCone;
    if (maps && ds.gen_map_ok[g]) cand |= kCandMap;
    return true;
}

// Depth-map bins a pixel at offset (rx, ry) != 0 may lie in.
__device__ __forceinline__ int2 pixel_bins(float rx, float ry) {
    const float a = pang(rx, ry);
    return make_int2(((int)floorf((a - kAngEps) / kAngW) + kAngBins) & (kAngBins - 1),
                     (int)floorf((a + kAngEps) / kAngW) & (kAngBins - 1));
}

// The undecided pixels of a candidate (bit k of und: the lane's pixel k)
// tested exactly; returns the lane's visible ones. gl: a point generator's
// lattice position; seg_id: a segment interior's source, else -1. clear (with
// a depth map): no obstacle is met nearer than that to the generator on any of
// their segments.
// The polygons that may block one of them are those whose boxes meet the thick
// segment from the block's centre to the generator (or to the centre's foot on
// the segment source: the other pixels' segments are its translates) and, for
// a point, that no edge of theirs separates from the hull of the block's box
// and the generator. They are listed kWarpPoly at a time, and each list is
// tested against the undecided pixels, packed a lane each.
// Every step is one load deep for the whole warp: a lane takes a bin of the
// segment, then the bins' records are dealt to the lanes evenly, then a lane
// takes a listed polygon. (Lanes walking bins of their own, record by record
// and vertex by vertex, waited on some 80 loads in a row: 57k cycles a list on
// the 2048^2 maze.)
template <int PX, int PY, int ROW>
__device__ __forceinline__ unsigned resolve_pixels(const DevScene &ds, WarpSmem<PX * PY> &ws, const Block &b, int2 gl, int seg_id,
                                                   float clear, unsigned und) {
    using S = Shape<PX, PY, ROW>;
    constexpr int N = S::kPix;
    const int lane = threadIdx.x & 31;
    if (lane == 0) SPM_CNT(5, 1);
    SPM_CNT(7, __popc(und));
    // the undecided pixels, packed
    const int mine = __popc(und);
    int at = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, at, o);
        if (lane >= o) at += y;
    }
    const int n_item = __shfl_sync(0xffffffffu, at, 31);
    at -= mine;
    __syncwarp();
    {
        int p = at;
        for (unsigned m = und; m; m &= m - 1) ws.item[p++] = (unsigned short)(lane * N + __ffs(m) - 1);
    }
    const int4 box = b.box;
    const float cx = 0.5f * ((float)box.x + (float)box.z), cy = 0.5f * ((float)box.y + (float)box.w);
    float dx = (float)gl.x - cx, dy = (float)gl.y - cy;
    if (seg_id >= 0) {
        const int4 seg = ds.seg_lat[seg_id];
        const float fux = (float)(seg.z - seg.x), fuy = (float)(seg.w - seg.y);
        const float t = __fdividef((cx - seg.x) * fux + (cy - seg.y) * fuy, fux * fux + fuy * fuy);
        dx = seg.x + t * fux - cx;
        dy = seg.y + t * fuy - cy;
    } else {
        // the block's segments shrink toward the generator alike: what lies
        // nearer than `clear` to it is the same last share of each
        const float fx = fmaxf(fabsf((float)(box.x - gl.x)), fabsf((float)(box.z - gl.x)));
        const float fy = fmaxf(fabsf((float)(box.y - gl.y)), fabsf((float)(box.w - gl.y)));
        const float part = fmaxf(1.f - fmaxf(clear - 2.f, 0.f) * rsqrtf(fmaf(fx, fx, fy * fy)), 0.f);
        dx *= part;
        dy *= part;
    }
    const float ex = (float)(box.z - box.x), ey = (float)(box.w - box.y);
    const float m = 0.5f * (ex * ex + ey * ey) * rsqrtf(fmaxf(ex * ex + ey * ey, 1.f)) + 2.0f;  // half the segment's thickness
    const float bs = (float)ds.bin_size, ibs = ds.bin_inv;
    auto col_of = [&](float v) { return min(max((int)floorf((v - (float)ds.bin_x0) * ibs), 0), ds.bin_nx - 1); };
    auto row_of = [&](float v) { return min(max((int)floorf((v - (float)ds.bin_y0) * ibs), 0), ds.bin_ny - 1); };
    const int c0 = col_of(fminf(cx, cx + dx) - m), c1 = col_of(fmaxf(cx, cx + dx) + m);
    const bool steep = fabsf(dx) < 0.5f;
    const float idx = steep ? 0.f : __fdividef(1.0f, dx);
    // rows a column's share of the segment may span: an upper bound, so that
    // every (column, row) of it is an item of its own
    const float span = (steep ? fabsf(dy) : fminf(fabsf(dy * idx) * (bs + 2.f * m), fabsf(dy))) + 2.f * m;
    const int K = min((int)(span * ibs) + 3, ds.bin_ny), items = (c1 - c0 + 1) * K;
    int n = 0, first = 0, cnt = 0, incl = 0, recs = 0, r0 = 0;
    for (int j0 = 0;;) {
        while (r0 >= recs && j0 < items) {  // the next 32 bins
            cnt = 0;
            if (j0 + lane < items) {
                const int c = (j0 + lane) / K, kr = j0 + lane - c * K;
                float ylo = fminf(0.f, dy), yhi = fmaxf(0.f, dy);
                if (!steep) {
                    const float xa = (float)(ds.bin_x0 + (c0 + c) * ds.bin_size) - cx;
                    const float ta = (xa - m) * idx, tb = (xa + bs + m) * idx;
                    const float ya = __saturatef(fminf(ta, tb)) * dy, yb = __saturatef(fmaxf(ta, tb)) * dy;
                    ylo = fminf(ya, yb);
                    yhi = fmaxf(ya, yb);
                }
                const int row = row_of(cy + ylo - m) + kr;
                if (row <= row_of(cy + yhi + m)) {
                    const int bin = row * ds.bin_nx + c0 + c;
                    first = __ldg(ds.bin_start + bin);
                    cnt = __ldg(ds.bin_start + bin + 1) - first;
                }
            }
            incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            recs = __shfl_sync(0xffffffffu, incl, 31);
            r0 = 0;
            j0 += 32;
        }
        if (r0 < recs) {  // 32 of their records
            const int r = r0 + lane;
            int own = 0;  // the first lane whose records end beyond r
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(0xffffffffu, incl, (own + o - 1) & 31) <= r) own += o;
            own &= 31;
            const int it = __shfl_sync(0xffffffffu, first, own) + r -
                           (__shfl_sync(0xffffffffu, incl, own) - __shfl_sync(0xffffffffu, cnt, own));
            int4 rec = make_int4(-1 - lane, 0, 0, 0);
            bool hit = false;
            if (r < recs) {
                const int4 *rp = reinterpret_cast<const int4 *>(ds.bin_recs + it);
                const int4 bx = __ldg(rp);
                rec = __ldg(rp + 1);
                // its box against the thick segment: the line, then the extent
                const float hx = 0.5f * (float)(bx.z - bx.x) + m, hy = 0.5f * (float)(bx.w - bx.y) + m;
                const float qx = 0.5f * (float)(bx.x + bx.z) - cx, qy = 0.5f * (float)(bx.y + bx.w) - cy;
                hit = fabsf(dx * qy - dy * qx) <= fabsf(dx) * hy + fabsf(dy) * hx &&
                      fabsf(qx - 0.5f * dx) <= 0.5f * fabsf(dx) + hx && fabsf(qy - 0.5f * dy) <= 0.5f * fabsf(dy) + hy;
            }
            // a polygon lies in several bins: its first record here counts
            const unsigned same = __match_any_sync(0xffffffffu, rec.x);
            hit = hit && (same & ((1u << lane) - 1u)) == 0;
            for (int q = 0; q < n; ++q) hit = hit && ws.poly[q].x != rec.x;
            const unsigned bal = __ballot_sync(0xffffffffu, hit);
            if (hit) ws.poly[n + __popc(bal & ((1u << lane) - 1u))] = make_int3(rec.x, rec.y, rec.z);
            n += __popc(bal);
            r0 += 32;
            __syncwarp();
        }
        const bool done = r0 >= recs && j0 >= items;
        if (!done && n <= kWarpPoly - 32) continue;
        if (lane == 0) SPM_CNT(6, n);
        // the listed polygons against the undecided pixels
        if (seg_id < 0) {
            int kept = 0;
            for (int q0 = 0; q0 < n; q0 += 32) {
                bool keep = false;
                int3 pl = make_int3(0, 0, 0);
                if (q0 + lane < n) {
                    pl = ws.poly[q0 + lane];
                    const int2 *V = ds.poly_v + pl.y;
                    bool apart = false;
                    int2 a = __ldg(V + pl.z - 1);
#pragma unroll 2
                    for (int i = 0; i < pl.z; ++i) {
                        const int2 e = __ldg(V + i);
                        const int nx = -(e.y - a.y), ny = e.x - a.x;  // orient(a, e, p) = n . (p - a)
                        const int far = nx * ((nx > 0 ? box.z : box.x) - a.x) + ny * ((ny > 0 ? box.w : box.y) - a.y);
                        apart |= far <= 0 && nx * (gl.x - a.x) + ny * (gl.y - a.y) <= 0;
                        a = e;
                    }
                    keep = !apart;
                }
                const unsigned bal = __ballot_sync(0xffffffffu, keep);
                __syncwarp();
                if (keep) ws.poly[kept + __popc(bal & ((1u << lane) - 1u))] = pl;
                kept += __popc(bal);
                __syncwarp();
            }
            n = kept;
        }
        for (int e = lane; e < n_item && n > 0; e += 32) {
            const int it = ws.item[e], l = it / N, k = it % N;
            if (it & kBlocked) continue;
            const int px = ds.pitch_x * (b.i0 + l % S::kRow * PX + k % PX) + ds.pitch_x / 2;
            const int py = ds.pitch_y * (b.j0 + l / S::kRow + k / PX * (32 / S::kRow)) + ds.pitch_y / 2;
            bool v = true;
            if (seg_id < 0) {
                if (px != gl.x || py != gl.y)
                    for (int q = 0; q < n && v; ++q) {
                        SPM_CNT(10, 1);
                        v = !segment_meets_poly(ds.poly_v + ws.poly[q].y, ws.poly[q].z, px, py, gl.x, gl.y);
                    }
            } else {
                const int4 seg = ds.seg_lat[seg_id];
                const long long ux = seg.z - seg.x, uy = seg.w - seg.y, den = ux * ux + uy * uy;
                const long long num = (px - seg.x) * ux + (py - seg.y) * uy;
                if (cross32((int)ux, (int)uy, px - seg.x, py - seg.y) != 0)
                    for (int q = 0; q < n && v; ++q)
                        v = !foot_meets_poly(ds.poly_v + ws.poly[q].y, ws.poly[q].z, seg, px, py, num, den);
            }
            if (!v) ws.item[e] = (unsigned short)(it | kBlocked);
        }
        __syncwarp();
        n = 0;
        if (done) break;
    }
    unsigned vis = 0;
    for (unsigned w = und; w; w &= w - 1)
        if (!(ws.item[at++] & kBlocked)) vis |= w & -w;
    return vis;
}

// Candidate c against the block's pixels.
template <int PX, int PY, int ROW>
__device__ __forceinline__ void apply_candidate(const DevScene &ds, WarpSmem<PX * PY> &ws, Block &b, int c) {
    constexpr int kStep = 32 / ROW;  // rows between a lane's pixels
    const int lane = threadIdx.x & 31, g = c & kCandId;
    const float4 rec = __ldg(ds.gen_rec + g);
    const int4 q = __ldg(ds.gen_cull + g);
    const int2 gl = make_int2((short)q.x, q.x >> 16);
    const bool seg = (__float_as_int(rec.w) & 7) == kSegI;
    const int seg_id = seg ? ds.gen_aux[g] : -1;
    const float2 *map = c & kCandMap ? ds.gen_maps + (size_t)g * kAngBins : nullptr;
    float4 sf = make_float4(0.f, 0.f, 0.f, 0.f);
    float il = 0.f;
    if (seg) {
        sf = ds.seg_pos[seg_id];
        const float fux = sf.z - sf.x, fuy = sf.w - sf.y;
        il = 1.0f / sqrtf(fux * fux + fuy * fuy);
    }
    unsigned want = 0;
#pragma unroll 1
    for (int h = 0; h < PY; ++h) {
#pragma unroll 2
        for (int k4 = 0; k4 < PX; ++k4) {
            const int k = PX * h + k4, at = k * 32 + lane;
            const float d = point_dist(rec.z, pixel_x(ds, b.i + k4) - rec.x, pixel_y(ds, b.j + h * kStep) - rec.y);
            const float old = ws.bd[at];
            bool better = d < old;
            if (d == old) better = g < ws.bi[at];
            if (better) want |= 1u << k;
            ws.d[at] = d;
        }
    }
    if (seg) {
        want = 0;
#pragma unroll 1
        for (int k = 0; k < PX * PY; ++k) {
            const float fx = pixel_x(ds, b.i + k % PX), fy = pixel_y(ds, b.j + k / PX * kStep);
            // the roundings named: which product is contracted is otherwise the compiler's choice
            const float cross = fmaf(-(sf.w - sf.y), fx - sf.x, __fmul_rn(sf.z - sf.x, fy - sf.y));
            const float d = fabsf(cross) * il, old = ws.bd[k * 32 + lane];
            ws.d[k * 32 + lane] = d;
            if (d < old || (d == old && g < ws.bi[k * 32 + lane])) want |= 1u << k;
        }
    }
    SPM_CNT(14, __popc(want));
    if (!__any_sync(0xffffffffu, want)) return;
    unsigned vis = 0, und = 0;
    float clear = INFINITY;
    const int rx0 = ds.pitch_x * b.i + ds.pitch_x / 2 - gl.x, ry0 = ds.pitch_y * b.j + ds.pitch_y / 2 - gl.y;
    if (seg) {  // the perpendicular foot strictly inside the segment
        const int4 L = ds.seg_lat[seg_id];
        const long long ux = L.z - L.x, uy = L.w - L.y, den = ux * ux + uy * uy;
#pragma unroll 1
        for (unsigned m = want; m; m &= m - 1) {
            const int k = __ffs(m) - 1;
            const int px = ds.pitch_x * (b.i + k % PX) + ds.pitch_x / 2;
            const int py = ds.pitch_y * (b.j + k / PX * kStep) + ds.pitch_y / 2;
            const long long nm = (px - L.x) * ux + (py - L.y) * uy;
            if (nm > 0 && nm < den) und |= m & -m;
        }
    } else {
        const int4 cone = make_int4((short)q.y, q.y >> 16, (short)q.z, q.z >> 16);
        const int ct = (__float_as_int(rec.w) >> 3) & 3;
#pragma unroll 1
        for (int h = 0; h < PY; ++h) {
#pragma unroll
            for (int k4 = 0; k4 < PX; ++k4) {
                const unsigned bit = 1u << (PX * h + k4);
                if (!(want & bit)) continue;
                const int ix = rx0 + k4 * ds.pitch_x, iy = ry0 + h * kStep * ds.pitch_y;
                if (!(c & kCandInCone) && !in_cone(ct, cone, ix, iy)) continue;
                if (!map) {
                    und |= bit;
                } else {
                    const float rx = (float)ix, ry = (float)iy, r2 = fmaf(rx, rx, ry * ry);
                    const int2 bin = pixel_bins(rx, ry);
                    const float2 m0 = __ldg(map + bin.x), m1 = __ldg(map + bin.y);
                    const float low = fminf(m0.y, m1.y);
                    if (r2 == 0.f || r2 * (1.f + 1e-5f) < low) {  // visible (or the generator's own pixel)
                        SPM_CNT(12, 1);
                        vis |= bit;
                    } else if (r2 * (1.f - 1e-5f) < fmaxf(m0.x, m1.x)) {
                        und |= bit;
                        clear = fminf(clear, low);
                    } else {  // hidden
                        SPM_CNT(13, 1);
                    }
                }
            }
        }
    }
    if (__any_sync(0xffffffffu, und)) {
        // squared distances are non-negative: they order as their bits
        const float near = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(clear)));
        vis |= resolve_pixels<PX, PY, ROW>(ds, ws, b, gl, seg_id, map ? sqrtf(near) : 0.f, und);
    }
    float worst = -INFINITY;
#pragma unroll
    for (int k = 0; k < PX * PY; ++k) {
        const int at = k * 32 + lane;
        float d = ws.bd[at];
        if (vis >> k & 1u) {
            d = ws.d[at];
            ws.bd[at] = d;
            ws.bi[at] = g;
        }
        worst = fmaxf(worst, d);
    }
    b.worst = worst;
}

// A scan's candidates that one polygon hides from the block go before their turn
// (flooded lists were tested on the tile's area): the next 32 or so in order of
// their bounds, a lane each. l: the lane's bounds as bits, ~0: none. Returns the
// bound up to which they are tested. (All 160 at once, five a lane, most of them
// far ones that are never reached: 1024^2 polygons with 30 sources 805 us of
// pixel pass.)
template <int N>
__device__ __forceinline__ unsigned drop_hidden(const DevScene &ds, WarpSmem<N> &ws, const Block &b,
                                                unsigned (&l)[kWarpCand / 32], unsigned least, unsigned most) {
    const int lane = threadIdx.x & 31;
    auto within = [&](unsigned x) {
        int c = 0;
#pragma unroll
        for (int k = 0; k < kWarpCand / 32; ++k) c += l[k] <= x;
        return __reduce_add_sync(0xffffffffu, c);
    };
    unsigned upto = max(least, most - 1u);  // beyond `most` none can win
    if (within(upto) > 32) {
        unsigned lo = least;
#pragma unroll 1
        for (int it = 0; it < 12; ++it) {
            const unsigned mid = lo + (upto - lo) / 2;
            if (within(mid) <= 32) lo = mid;
            else upto = mid;
        }
        upto = lo;
    }
    int n = 0;
#pragma unroll
    for (int k = 0; k < kWarpCand / 32; ++k) {
        const unsigned bal = __ballot_sync(0xffffffffu, l[k] <= upto);
        const int at = n + __popc(bal & ((1u << lane) - 1u));
        if (l[k] <= upto && at < 32) ws.item[at] = (unsigned short)(lane + 32 * k);
        n += __popc(bal);
    }
    __syncwarp();
    if (lane < n) {
        const int slot = ws.item[lane];
        const int4 q = __ldg(ds.gen_cull + (ws.cand[slot] & kCandId));
        if (!(__int_as_float(q.w) < 0.f) && box_hidden(ds, b.box, make_int2((short)q.x, q.x >> 16))) ws.lb[slot] = -1.f;
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < kWarpCand / 32; ++k)
        if (l[k] <= upto && ws.lb[lane + 32 * k] < 0.f) l[k] = 0xffffffffu;
    return upto;
}

// The n candidates the warp holds, in order of their lower bounds, until none
// can improve a pixel.
template <int PX, int PY, int ROW, bool SCAN>
__device__ __forceinline__ void apply_candidates(const DevScene &ds, WarpSmem<PX * PY> &ws, int n, Block &b) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    unsigned l[kWarpCand / 32];
#pragma unroll
    for (int k = 0; k < kWarpCand / 32; ++k)
        l[k] = lane + 32 * k < n ? __float_as_uint(ws.lb[lane + 32 * k]) : 0xffffffffu;
    bool first = true;   // a scan's first candidate sets a bound to what the rest are good for
    unsigned tested = 0;
    for (;;) {
        unsigned mine = l[0];
#pragma unroll
        for (int k = 1; k < kWarpCand / 32; ++k) mine = min(mine, l[k]);
        const unsigned least = __reduce_min_sync(0xffffffffu, mine);
        if (least == 0xffffffffu) break;
        if (!__any_sync(0xffffffffu, b.worst > __uint_as_float(least))) break;
        if (SCAN && !b.lists && !first && least > tested) {
            tested = drop_hidden(ds, ws, b, l, least, __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(b.worst, 0.f))));
            continue;
        }
        first = false;
        const int from = __ffs(__ballot_sync(0xffffffffu, mine == least)) - 1;
        int c = 0;
        if (lane == from) {
#pragma unroll
            for (int k = kWarpCand / 32 - 1; k >= 0; --k)
                if (l[k] == least) c = k;
#pragma unroll
            for (int k = 0; k < kWarpCand / 32; ++k)
                if (k == c) l[k] = 0xffffffffu;
        }
        c = __shfl_sync(0xffffffffu, c, from);
        if (lane == 0) SPM_CNT(4, 1);
        apply_candidate<PX, PY, ROW>(ds, ws, b, ws.cand[32 * c + from]);
    }
    __syncwarp();
}

template <int PX, int PY, int ROW, bool SCAN>
__device__ __forceinline__ void pixel_block(const DevScene &ds, const int i0, const int j0, float *__restrict__ dist,
                                            int32_t *__restrict__ parent, WarpSmem<PX * PY> &ws) {
    using S = Shape<PX, PY, ROW>;
    constexpr int kStep = 32 / S::kRow;
    const int lane = threadIdx.x & 31;
    SPM_T0();
    Block b;
    b.i0 = i0;
    b.j0 = j0;
    b.i = b.i0 + lane % S::kRow * PX;
    b.j = b.j0 + lane / S::kRow;
    unsigned live = 0;
#pragma unroll
    for (int h = 0; h < PY; ++h)
        if (b.j + kStep * h < ds.Ny)  // the scene's free-space mask: outside every obstacle's open interior, inside the grid
            live |= ((__ldg(ds.free_bits + (size_t)(b.j + kStep * h) * ds.free_words + (b.i >> 5)) >> (b.i & 31)) &
                     ((1u << PX) - 1u)) << (PX * h);
#pragma unroll
    for (int k = 0; k < S::kPix; ++k) {
        ws.bd[k * 32 + lane] = (live >> k) & 1u ? INFINITY : -INFINITY;
        ws.bi[k * 32 + lane] = -1;
    }
    b.worst = live ? INFINITY : -INFINITY;
    if (lane == 0) SPM_CNT(0, 1);
    if (__any_sync(0xffffffffu, live)) {
        b.i1 = min(b.i0 + S::kW, ds.Nx) - 1;
        b.j1 = min(b.j0 + S::kH, ds.Ny) - 1;
        b.box = make_int4(ds.pitch_x * b.i0 + ds.pitch_x / 2, ds.pitch_y * b.j0 + ds.pitch_y / 2,
                          ds.pitch_x * b.i1 + ds.pitch_x / 2, ds.pitch_y * b.j1 + ds.pitch_y / 2);
        const int sh = ds.tile == kTile ? 5 : 4, tile = (j0 >> sh) * ds.tiles_x + (i0 >> sh);  // tiles of 32 or 16 pixels
        const TileList tl(ds, tile, true);
        b.lists = tl.lists;
        const bool maps = b.lists && ds.use_maps && ds.gen_maps;
        SPM_LAP(0);
        float ub = INFINITY;  // no pixel of the block can take more
        int n = 0;
        // A scan of more generators than the warp holds first takes every
        // lane's nearest one of the first kNearest: in the order of their ids,
        // hundreds of sources were tested before the near ones bounded the rest
        // (1024^2 polygons with 300 sources: pixel pass 551 -> 289 us).
        constexpr int kNearest = 2048;
        bool nearest = SCAN && !tl.lists && tl.total > kWarpCand;
        unsigned near_lb = 0xffffffffu;
        int near_c = 0, near_g = -1;
        for (int e0 = 0; e0 < tl.total;) {
            bool keep = false;
            float lb = 0.f;
            int c = 0, g = 0;
            const bool in = tl.entry(ds, e0 + lane, g);
            if (in) keep = block_candidate(ds, g, b, ub, maps, lb, c);
            e0 += 32;
            const bool last = e0 >= (SCAN && nearest ? min(tl.total, kNearest) : tl.total);
            if (SCAN) {
                if (nearest) {
                    if (keep && __float_as_uint(lb) < near_lb) {  // bounds are non-negative
                        near_lb = __float_as_uint(lb);
                        near_c = c;
                        near_g = g;
                    }
                    if (!last) continue;
                    keep = near_g >= 0;
                    lb = __uint_as_float(near_lb);
                    c = near_c;
                } else {
                    keep = keep && g != near_g;  // taken (an entry comes to the same lane)
                }
            }
            const unsigned bal = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                const int slot = n + __popc(bal & ((1u << lane) - 1u));
                ws.lb[slot] = lb;
                ws.cand[slot] = c;
            }
            n += __popc(bal);
            if (n > kWarpCand - 32 || (last && n > 0)) {
                if (lane == 0) SPM_CNT(1, n);
                SPM_LAP(1);
                apply_candidates<PX, PY, ROW, SCAN>(ds, ws, n, b);
                SPM_LAP(2);
                n = 0;
                if (!last || (SCAN && nearest)) {
                    float w = b.worst;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) w = fmaxf(w, __shfl_xor_sync(0xffffffffu, w, o));
                    ub = w;
                }
            }
            if (SCAN && nearest) {
                nearest = false;
                e0 = 0;
            }
        }
    }
    // 16-byte stores where every row of both planes starts on such a boundary
    const bool vec = PX == 4 && (ds.Nx & 3) == 0 &&
                     ((reinterpret_cast<size_t>(dist) | reinterpret_cast<size_t>(parent)) & 15) == 0;
#pragma unroll
    for (int h = 0; h < PY; ++h) {
        if (b.j + kStep * h >= ds.Ny) continue;
        float od[PX];
        int op[PX];
#pragma unroll
        for (int k = 0; k < PX; ++k) {
            op[k] = ws.bi[(PX * h + k) * 32 + lane];
            od[k] = op[k] >= 0 ? ws.bd[(PX * h + k) * 32 + lane] : INFINITY;
        }
        const size_t base = (size_t)(b.j + kStep * h) * ds.Nx + b.i;
        if (vec) {
            if (b.i < ds.Nx) {
                *reinterpret_cast<float4 *>(dist + base) = make_float4(od[0], od[1 % PX], od[2 % PX], od[3 % PX]);
                *reinterpret_cast<int4 *>(parent + base) = make_int4(op[0], op[1 % PX], op[2 % PX], op[3 % PX]);
            }
        } else {
#pragma unroll
            for (int k = 0; k < PX; ++k)
                if (b.i + k < ds.Nx) {
                    dist[base + k] = od[k];
                    parent[base + k] = op[k];
                }
        }
    }
    SPM_LAP(3);
    SPM_TFLUSH();
}

// Open scenes: most of a tile's list (every obstacle vertex that sees some of
// it) goes by its shadow cone, alike for the tile's blocks: one CTA culls the
// list for the tile. (Each block culling the whole list was half of the pixel
// pass of the differentiable scene, 900 entries a tile.)
constexpr int kCullThreads = 128;
__device__ __forceinline__ void cull_tile(const DevScene &ds, int tile) {
    __shared__ int n;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x == 0) n = 0;
    __syncthreads();
    Block b;
    b.i0 = tile % ds.tiles_x * ds.tile;
    b.j0 = tile / ds.tiles_x * ds.tile;
    b.i1 = min(b.i0 + ds.tile, ds.Nx) - 1;
    b.j1 = min(b.j0 + ds.tile, ds.Ny) - 1;
    b.box = make_int4(ds.pitch_x * b.i0 + ds.pitch_x / 2, ds.pitch_y * b.j0 + ds.pitch_y / 2,
                      ds.pitch_x * b.i1 + ds.pitch_x / 2, ds.pitch_y * b.j1 + ds.pitch_y / 2);
    const TileList tl(ds, tile, false);
    int32_t *out = ds.cull_items + (size_t)tile * cull_cap(ds.tile);
    for (int e0 = threadIdx.x & ~31; tl.lists && e0 < tl.total; e0 += kCullThreads) {
        int g = 0, c;
        float lb;
        const bool keep = tl.entry(ds, e0 + lane, g) && block_candidate(ds, g, b, INFINITY, false, lb, c);
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        int at = 0;
        if (lane == 0 && bal) at = atomicAdd(&n, __popc(bal));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(bal & ((1u << lane) - 1u));
        if (keep && at < cull_cap(ds.tile)) out[at] = g;
    }
    __syncthreads();
    if (threadIdx.x == 0) ds.cull_count[tile] = n <= cull_cap(ds.tile) ? n : -1;
}

__global__ void __launch_bounds__(kCullThreads) k_tile_cull(const __grid_constant__ DevScene ds, int tile0) {
    chain_start();
    cull_tile(ds, tile0 + blockIdx.x);
}

__global__ void __launch_bounds__(kCullThreads) k_tile_cull_b(const __grid_constant__ BatchDev b) {
    for (int t = blockIdx.x; t < b.total_tiles; t += gridDim.x) {
        int lo = 0, hi = b.n;  // last order index with tile_off <= t
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (__ldg(b.tile_off + mid) <= t) lo = mid;
            else hi = mid;
        }
        const DevScene &ds = b.scenes[b.order[lo]];
        if (ds.cull_on) cull_tile(ds, t - b.tile_off[lo]);  // the same for the whole CTA
        __syncthreads();
    }
}

constexpr long long kFourWaves = 4 * 152 * 28;  // GB300: 152 SMs
#ifndef SPM_BLK_MINB
#define SPM_BLK_MINB 28  // warps per SM the kernels are compiled for
#endif
// One warp a CTA, so that a finished block's place is taken at once: with four
// warps a CTA (sharing nothing) the early ones waited for the slowest, 15 %
// on the 4096^2 maze.
template <int PX, int PY, int ROW, bool SCAN>
__global__ void __launch_bounds__(32, SPM_BLK_MINB) k_pixel_blocks(const __grid_constant__ DevScene ds,
                                                                   float *__restrict__ dist,
                                                                   int32_t *__restrict__ parent, int row0) {
    __shared__ WarpSmem<PX * PY> sm;
    using S = Shape<PX, PY, ROW>;
    chain_start();
    pixel_block<PX, PY, ROW, SCAN>(ds, blockIdx.x * S::kW, row0 + blockIdx.y * S::kH, dist, parent, sm);
}

// Persistent form over a batch of scenes: each warp takes the next
// (scene, block) from a global counter (costliest tiles first), copies that
// scene's descriptor into shared memory and runs the same code. Blocks of
// 16 x 8: a batch's grids are coarse, and a larger block evaluates generators
// for pixels they cannot win (64 polygon scenes, 22.4 Mpixel: 16 x 16 1674 us,
// 16 x 8 1220, 8 x 8 1306). 24 warps an SM (1206 us; 28: 1220, 32: 1293, more
// of them contend for L1), four a CTA (one to sixteen: within 2 %).
constexpr int kBatchWarps = 4, kBatchSm = 24;
template <bool SCAN>  // some scene of many sources may scan
__global__ void __launch_bounds__(32 * kBatchWarps, kBatchSm / kBatchWarps) k_pixel_blocks_b(const __grid_constant__ BatchDev b) {
    using S = Shape<4, 1>;
    static_assert(S::kW == kBatchBlkW && S::kH == kBatchBlkH, "the batch counts these blocks");
    __shared__ WarpSmem<S::kPix> sm[kBatchWarps];
    __shared__ DevScene sds[kBatchWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    DevScene &ds = sds[warp];
    int held = -1;
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(b.tile_counter, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= b.total_blocks) break;
        int lo = 0, hi = b.n;  // last order index with blk_off <= t
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (__ldg(b.blk_off + mid) <= t) lo = mid;
            else hi = mid;
        }
        const int sc = __ldg(b.order + lo), blk = t - __ldg(b.blk_off + lo);
        if (sc != held) {
            __syncwarp();
            for (int w = lane; w < (int)(sizeof(DevScene) / 4); w += 32)
                reinterpret_cast<int *>(&ds)[w] = __ldg(reinterpret_cast<const int *>(&b.scenes[sc]) + w);
            __syncwarp();
            held = sc;
        }
        const int across = (ds.Nx + S::kW - 1) / S::kW;
        pixel_block<4, 1, 4, SCAN>(ds, blk % across * S::kW, blk / across * S::kH, b.dist[sc], b.parent[sc], sm[warp]);
        __syncwarp();
    }
}

}  // namespace

// Exact point query (Sec. 6, Discussion: a point on a region border may take
// a parent up to half a pixel's diagonal off; comparing the parents of the
// neighbouring pixels at the point itself removes the error). One warp: lane
// k < 9 evaluates the parent of pixel (i + k % 3 - 1, j + k / 3 - 1) at the
// lattice point q (world coordinates qf) with the exact predicates, FP64 keys
// in the same operation order as the distance definition; the smallest key
// (then id) wins.
__global__ void k_query_exact(const __grid_constant__ DevScene ds, const int32_t *__restrict__ field_parent, int i,
                              int j, int2 q, double2 qf, int32_t *out_par, double *out_dist) {
    const int lane = threadIdx.x;
    int g = -1;
    if (lane < 9) {
        const int ii = i + lane % 3 - 1, jj = j + lane / 3 - 1;
        if (ii >= 0 && jj >= 0 && ii < ds.Nx && jj < ds.Ny) g = field_parent[(size_t)jj * ds.Nx + ii];
    }
    double key = INFINITY;
    if (g >= 0 && ds.gen_cost[g] < INFINITY) {
        const int kind = ds.gen_kind[g];
        if (kind == kSegI) {
            const int s = ds.gen_aux[g];
            const int4 L = ds.seg_lat[s];
            const long long ux = L.z - L.x, uy = L.w - L.y;
            const long long num = (q.x - L.x) * ux + (q.y - L.y) * uy, den = ux * ux + uy * uy;
            if (num > 0 && num < den && visible_foot(ds, s, q.x, q.y, num, den)) {
                const float4 F = ds.seg_pos[s];
                const double fx = __dsub_rn((double)F.z, (double)F.x), fy = __dsub_rn((double)F.w, (double)F.y);
                const double c = __dsub_rn(__dmul_rn(fx, __dsub_rn(qf.y, (double)F.y)), __dmul_rn(fy, __dsub_rn(qf.x, (double)F.x)));
                key = __ddiv_rn(fabs(c), __dsqrt_rn(__dadd_rn(__dmul_rn(fx, fx), __dmul_rn(fy, fy))));
            }
        } else {
            const int2 gl = ds.gen_lat[g];
            const bool cone_ok = kind != kVert || in_cone(ds.gen_ctype[g], ds.gen_cone[g], q.x - gl.x, q.y - gl.y);
            if (cone_ok && visible_points(ds, q.x, q.y, gl.x, gl.y)) {
                const float2 gp = ds.gen_pos[g];
                const double dx = __dsub_rn(qf.x, (double)gp.x), dy = __dsub_rn(qf.y, (double)gp.y);
                key = __dadd_rn(ds.gen_cost[g], __dsqrt_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy))));
            }
        }
    }
    int best = key < INFINITY ? g : -1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double ok = __shfl_xor_sync(0xffffffffu, key, o);
        const int og = __shfl_xor_sync(0xffffffffu, best, o);
        if (ok < key || (ok == key && og >= 0 && (best < 0 || og < best))) {
            key = ok;
            best = og;
        }
    }
    if (lane == 0) {
        *out_par = best;
        *out_dist = key;
    }
}

// Parent chain of a pixel (Sec. 1), one thread: a few dependent loads, written
// straight to the host's page-locked buffer, so that a path costs one launch
// and one wait (three copies and a wait, one of them of the whole parent
// table, took 33 us a path).
__global__ void k_path(const __grid_constant__ DevScene ds, const int32_t *__restrict__ field_parent, size_t idx,
                       int room, PathOut *out) {
    int g = field_parent[idx], n = 0, seg = 0, more = 0;
    out->parent = g;
    for (int guard = 0; g >= 0 && guard <= ds.n_gen + 1; ++guard) {
        if (n >= room || g >= ds.n_gen) {
            more = g >= ds.n_gen ? 2 : 1;  // 2: the plane no longer holds this scene's map
            break;
        }
        const int kind = ds.gen_kind[g], next = ds.gen_par[g];
        if (kind == kSegI) {
            out->f = ds.seg_pos[ds.gen_aux[g]];
            seg = 1;
            break;
        }
        out->pt[n++] = ds.gen_pos[g];
        if (kind != kVert) break;
        g = next;
    }
    out->n = n;
    out->seg = seg;
    out->more = more;
}

void launch_path(const DevScene &ds, cudaStream_t st, const int32_t *field_parent, size_t idx, int room, PathOut *out) {
    k_path<<<1, 1, 0, st>>>(ds, field_parent, idx, room, out);
}

void launch_query_exact(const DevScene &ds, cudaStream_t st, const int32_t *field_parent, int i, int j, int qx,
                        int qy, double fx, double fy, int32_t *out_par, double *out_dist) {
    k_query_exact<<<1, 32, 0, st>>>(ds, field_parent, i, j, make_int2(qx, qy), make_double2(fx, fy), out_par,
                                    out_dist);
}

namespace {

// Lattice point inside the open interior of an obstacle?
__device__ bool centre_in_obstacle(const DevScene &ds, int px, int py) {
    const int bx = (px - ds.bin_x0) / ds.bin_size, by = (py - ds.bin_y0) / ds.bin_size;
    if (bx < 0 || by < 0 || bx >= ds.bin_nx || by >= ds.bin_ny) return false;
    const int bin = by * ds.bin_nx + bx;
    for (int it = ds.bin_start[bin]; it < ds.bin_start[bin + 1]; ++it) {
        const BinRec rec = ds.bin_recs[it];
        const int4 b4 = rec.box;
        if (px <= b4.x || px >= b4.z || py <= b4.y || py >= b4.w) continue;
        bool inside = true;
        for (int e = 0; e < rec.m && inside; ++e) {
            const int2 a = ds.poly_v[rec.voff + e], c = ds.poly_v[rec.voff + (e + 1 == rec.m ? 0 : e + 1)];
            inside = orient32(a.x, a.y, c.x, c.y, px, py) > 0;
        }
        if (inside) return true;
    }
    return false;
}

// Free-space mask of the pixel centres: bit (i % 32) of word j * free_words +
// i / 32 is set when pixel (i, j)'s centre lies outside the open interior of
// every obstacle. The obstacles are fixed for the scene's lifetime, so it is
// built once, one warp per word.
__global__ void k_free_mask(const __grid_constant__ DevScene ds, uint32_t *bits) {
    const long long w = (long long)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    if (w >= (long long)ds.Ny * ds.free_words) return;  // whole warps
    const int lane = threadIdx.x & 31;
    const int j = (int)(w / ds.free_words), i = (int)(w % ds.free_words) * 32 + lane;
    const int pitch_x = ds.S * ds.Wx / ds.Nx, pitch_y = ds.S * ds.Wy / ds.Ny;
    const bool is_free = i < ds.Nx && !centre_in_obstacle(ds, pitch_x * i + pitch_x / 2, pitch_y * j + pitch_y / 2);
    const unsigned m = __ballot_sync(0xffffffffu, is_free);
    if (lane == 0) bits[w] = m;
}

}  // namespace

void launch_free_mask(const DevScene &ds, cudaStream_t st, uint32_t *bits) {
    const long long words = (long long)ds.Ny * ds.free_words;
    const int per_block = NT / 32;
    k_free_mask<<<(unsigned)((words + per_block - 1) / per_block), NT, 0, st>>>(ds, bits);
}

// Every generator may be scanned: no flood, or the device decides, or lists
// that may outgrow their buffer, as an open scene's do (200 polygons, 2000
// sources, 4096^2, mode 1: 8.4 ms in the kernel for lists alone, 1.6 in the
// other, which takes 0 to 5 % longer where there are lists).
bool pixels_may_scan(const DevScene &ds) {
    const long long pairs = (long long)(ds.flood_mode == 3 && ds.static_lists
                                            ? std::max(ds.vert_bits ? 0 : ds.n_vert, ds.src_direct ? 0 : ds.n_src)
                                            : ds.n_gen) * ds.tiles_x * ds.tiles_y;
    return !ds.use_flood || ds.flood_mode == 2 || ds.flood_mode == 0 || (ds.open_scene && pairs > ds.pair_cap);
}

bool tiles_culled(const DevScene &ds) {
    return ds.cull_items && ds.use_flood && ds.flood_mode == 3 && flood_verts_direct(ds);
}

void launch_pixel_phase(const DevScene &scene, cudaStream_t st, float *dist, int32_t *parent, int row0, int row1,
                        bool to_host) {
    DevScene ds = scene;
    const int rows = row1 - row0;
    if (rows <= 0) return;
    ds.cull_on = tiles_culled(ds) ? 1 : 0;
    if (ds.cull_on) {
        const int t0 = row0 / ds.tile, t1 = (row1 + ds.tile - 1) / ds.tile;
        k_tile_cull<<<ds.tiles_x * (t1 - t0), kCullThreads, 0, st>>>(ds, t0 * ds.tiles_x);
    }
    auto run = [&](auto shape, auto kern) {
        const dim3 grid((ds.Nx + shape.kW - 1) / shape.kW, (rows + shape.kH - 1) / shape.kH);
        if (ds.cull_on) launch_chained(kern, grid, dim3(32), 0, st, ds, dist, parent, row0);
        else kern<<<grid, 32, 0, st>>>(ds, dist, parent, row0);
    };
    // The smallest blocks that make at most four waves of warps (28 an SM):
    // large blocks cull and order their candidates for more pixels at once, but
    // a grid of few blocks waits for its slowest. Pixel pass in us with one /
    // two / four / eight waves for the line: squares 1000^2 109 / 84 / 72 / 70,
    // 512^2 polygons 37 / 35 / 35 / 35, 1024^2 79 / 70 / 70 / 76, 1501^2 127 /
    // 127 / 127 / 123, maze 2048^2 80 / 80 / 80 / 90, differentiable 112 / 112 /
    // 113 / 124. Halving a 16 x 16 block costs the least work, and pays up to six
    // waves (four / six: 1560^2 polygons 120 / 113, 1700^2 150 / 138, maze 1536^2
    // 68 / 64).
    const bool scan = pixels_may_scan(ds);
    auto pick = [&](auto shape, auto lists, auto scans) {
        if (scan) run(shape, scans);
        else run(shape, lists);
    };
    const long long blocks = (long long)((ds.Nx + 15) / 16) * ((rows + 15) / 16);
    // A large grid's planes in the host's memory: blocks 32 wide, within a tile,
    // whose rows are whole 128-byte lines. The link takes 193 GB/s of those, as
    // of copies, but 172 of a 16 x 16 block's 64-byte rows, and such a map waits
    // for it (16 x 16 or 16 x 8 / 32 x 4, wall clock of spm_compute_host alone:
    // maze 4096^2 934 / 845 us, differentiable 2048^2 328 / 303, maze 2048^2 318
    // / 314; a host move of the sources before it is another 70 to 90). Smaller
    // grids wait for their slowest block (1024^2 polygons 194 / 205).
    if (to_host && !scan && ds.tile == kTile && blocks * 4 > kFourWaves) {
        run(Shape<4, 1, 8>(), k_pixel_blocks<4, 1, 8, false>);
        return;
    }
    // Without depth maps every undecided pixel is tested exactly, and a block that
    // spans the obstacles' spacing evaluates and tests generators for pixels that
    // they cannot win: blocks of at most a quarter of it (3400 polygons, no room
    // for maps, 18 pixels apart at 1024^2: pixel pass 4750 us in blocks of 8 x 8,
    // 4157 of 8 x 4; 35 apart at 2048^2: 4471 of 16 x 16, 3044 of 8 x 8).
    const double apart = ds.use_maps && ds.gen_maps || ds.n_poly == 0 ? 1e9 : (double)ds.Nx * ds.Ny / ds.n_poly;
    if (blocks * 8 <= kFourWaves || apart < 20. * 20.) pick(Shape<1, 1>(), k_pixel_blocks<1, 1, 8, false>, k_pixel_blocks<1, 1, 8, true>);
    else if (blocks * 4 <= kFourWaves || apart < 40. * 40.) pick(Shape<2, 1>(), k_pixel_blocks<2, 1, 4, false>, k_pixel_blocks<2, 1, 4, true>);
    else if (blocks * 2 <= kFourWaves / 2 * 3) pick(Shape<4, 1>(), k_pixel_blocks<4, 1, 4, false>, k_pixel_blocks<4, 1, 4, true>);
    else pick(Shape<4, 2>(), k_pixel_blocks<4, 2, 4, false>, k_pixel_blocks<4, 2, 4, true>);
}

void launch_pixel_phase_batched(const BatchDev &b, cudaStream_t st) {
    cudaMemsetAsync(b.tile_counter, 0, sizeof(int32_t), st);
    int per_sm = 0, dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const auto kern = b.any_scan ? k_pixel_blocks_b<true> : k_pixel_blocks_b<false>;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * kBatchWarps, 0);
    const int grid = max(1, min((b.total_blocks + kBatchWarps - 1) / kBatchWarps, sms * max(per_sm, 1)));
    if (b.any_cull) k_tile_cull_b<<<std::min(b.total_tiles, sms * 16), kCullThreads, 0, st>>>(b);
    kern<<<grid, 32 * kBatchWarps, 0, st>>>(b);
}

int count_kernel_launches_pixel() { return 1; }

}  // namespace spm

#ifdef SPM_COUNT
// Instrumentation build only: reads and clears the work counters.
extern "C" int spm_debug_counters(unsigned long long *out32) {
    cudaDeviceSynchronize();
    if (cudaMemcpyFromSymbol(out32, spm::g_count, sizeof(unsigned long long) * 32) != cudaSuccess) return 1;
    unsigned long long z[32] = {0};
    cudaMemcpyToSymbol(spm::g_count, z, sizeof z);
    return 0;
}
#endif

#ifdef SPM_TIME
// Instrumentation build only: reads and clears the pixel kernel's phase clocks
// (0 set-up, 1 candidates, 2 their pixels, 3 output; of each CTA's first warp).
extern "C" int spm_debug_times(unsigned long long *out8) {
    cudaDeviceSynchronize();
    if (cudaMemcpyFromSymbol(out8, spm::g_time, sizeof(unsigned long long) * 8) != cudaSuccess) return 1;
    unsigned long long z[8] = {0};
    cudaMemcpyToSymbol(spm::g_time, z, sizeof z);
    return 0;
}
#endif
