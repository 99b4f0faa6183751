// Beam pass: the beam optimisation of ESVO (Laine and Karras; Aokana Sec. 2
// names ESVO as the traversal it builds on), recast so that it cannot change
// a single output record.
//
// ESVO casts a coarse ray per pixel block first and starts the block's rays
// near the surface the coarse ray found.  Here the coarse pass computes, for
// every 8 x 4 pixel tile (one casting warp), a lower bound Dn on the
// L-infinity distance from the camera origin of every solid voxel of the
// frame's LOD-cut scene that the tile's rays can meet.  A ray's L-infinity
// distance from the origin at parameter t is t |d|_max, so the casting
// kernel restarts each ray's march at the last integer plane of its dominant
// axis crossed before that distance: every cell the ray passes before it is
// empty for this ray, the cell holding the restart point is empty, and every
// hit is entered later through the planes the full march crosses -- the same
// first hit, entry plane and distance, without the traversal in front of it.
//
// The bound is a minimum over nodes of the selected DAGs, scattered to the
// tiles their screen rectangle covers:
//   * level 0 takes every chunk region of the frame table with its DAG root,
//     the box being the region's AABB of valid voxels;
//   * a node is projected in FP32 to a rectangle of tiles (box_rect, with
//     margins that cover its rounding); if the rectangle spans more tiles
//     than the refinement threshold and the node is not a 4^3 leaf, it goes to
//     the next level's queue, where its children are projected in its place;
//     otherwise atomicMin(Dn[tile], its L-inf distance) over the rectangle.
//     A leaf uses the bounding box of its set voxels;
//   * a box that comes closer to the origin than 2/16 of the largest |d|
//     component covers every tile (rays reach it before camera depth 1/16);
//     any other box is projected from its part at depth >= 1/16, and dropped
//     if it has none or it lies beyond the view distance (a hit there is
//     reported as a miss anyway);
//   * a full queue makes the node scatter itself instead of its children.
// Every solid voxel a pixel ray meets lies in one scattered node whose
// rectangle holds that pixel's tile, so Dn[tile] is at most its distance.
//
// The bounds live in a pyramid (level 0: the tiles; level L: cells of
// 2^L x 2^L tiles): a node writes the finest level at which its rectangle
// spans at most 16 cells, and the casting kernel takes each tile's minimum
// over its cells.  Entries are 64-bit, (pass tag << 32) | bound, written by a
// non-returning atomic minimum; the tag counts down from pass to pass, so an
// entry of this pass always beats one left by an earlier pass, and readers
// take entries of another tag as "nothing solid": the pyramid is never reset.
#include <cuda_runtime.h>

#include <climits>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <mutex>

#include <cooperative_groups.h>

#include "aok_internal.h"
#include "aok_ptx.cuh"
#include "aok_select.cuh"

namespace cg = cooperative_groups;
using namespace aok;

namespace {

constexpr int kBeamThreads = 256;      // block size of the cooperative walk
constexpr int kBeamBlocksPerSM = 2;    // blocks per SM of the grid: 45 us against 50 with one, 48 with three (city 1080p)
constexpr uint32_t kWideWalkRegions = 4096;  // a pass beside a running cast takes one block per SM, which can start
                                             // there sooner, unless it walks more regions than this
constexpr double kNearS = 1.0 / 16.0;  // camera-depth plane the projection clips at
constexpr uint32_t kNoItem = 0xFFFFFFFFu;  // an empty queue slot
constexpr int kMaxBeamDevices = 128;

// Screen rectangle [x, z) x [y, w) of tiles a box (relative to the origin)
// can cover from its part at camera depth s >= kNearS; false if none.
// A corner's q = Af p is the first corner's plus the edges' steps; with
// u = 2^-24 it errs by at most dl = 16 u max_i sum_j |Af_ij| max |p_j| (2u M
// from the rounding of p and Af, 3u M from the first corner, 6u M from the
// three steps, each of an edge of up to 2 max |p_j|, 3u M from adding them).
// A box wholly in front of the plane is bounded by its corners' projections
// (their hull holds the box's), widened by the error that dl and the
// approximate reciprocal (2u) carry; a box that straddles it by u = q_x / q_s
// over q_x in [X0, X1] and q_s in [kNearS, S1], each widened by dl.  Then a 0.5
// pixel margin for the FP32 pixel rays.
__device__ bool box_rect(const BeamView& K, const float lo[3], const float hi[3], int4& rc) {
    float M = 0.0f;
    float q[3][8];
    const float pm0 = fmaxf(fabsf(lo[0]), fabsf(hi[0])), pm1 = fmaxf(fabsf(lo[1]), fabsf(hi[1])),
                pm2 = fmaxf(fabsf(lo[2]), fabsf(hi[2]));
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const float a0 = K.Af[3 * i], a1 = K.Af[3 * i + 1], a2 = K.Af[3 * i + 2];
        M = fmaxf(M, __fmaf_rn(fabsf(a0), pm0, __fmaf_rn(fabsf(a1), pm1, fabsf(a2) * pm2)));
        const float d0 = a0 * (hi[0] - lo[0]), d1 = a1 * (hi[1] - lo[1]), d2 = a2 * (hi[2] - lo[2]);
        q[i][0] = __fmaf_rn(a0, lo[0], __fmaf_rn(a1, lo[1], a2 * lo[2]));
        q[i][1] = q[i][0] + d0;
        q[i][2] = q[i][0] + d1;
        q[i][3] = q[i][1] + d1;
#pragma unroll
        for (int k = 0; k < 4; k++) q[i][4 + k] = q[i][k] + d2;
    }
    const float dl = M * 9.7e-7f + 1e-6f;
    float S0 = 3e38f, S1 = -3e38f;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        S0 = fminf(S0, q[2][k]);
        S1 = fmaxf(S1, q[2][k]);
    }
    const float near_s = (float)kNearS;
    if (S1 + dl < near_s) return false;  // wholly behind the plane: only the near rule can reach it
    float a0, a1, b0, b1;
    if (S0 - dl >= near_s) {
        float u0 = 3e38f, u1 = -3e38f, v0 = 3e38f, v1 = -3e38f;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const float r = rcp_approx(q[2][k]);
            u0 = fminf(u0, q[0][k] * r); u1 = fmaxf(u1, q[0][k] * r);
            v0 = fminf(v0, q[1][k] * r); v1 = fmaxf(v1, q[1][k] * r);
        }
        const float um = fmaxf(fabsf(u0), fabsf(u1)) * 1.001f, vm = fmaxf(fabsf(v0), fabsf(v1)) * 1.001f;
        const float rs = dl * rcp_approx(S0 - dl) * 1.00001f;
        const float mu = __fmaf_rn(rs, 1.0f + um, um * 4.8e-7f);
        const float mv = __fmaf_rn(rs, 1.0f + vm, vm * 4.8e-7f);
        a0 = u0 - mu; a1 = u1 + mu;
        b0 = v0 - mv; b1 = v1 + mv;
    } else {
        float X0 = 3e38f, X1 = -3e38f, Y0 = 3e38f, Y1 = -3e38f;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            X0 = fminf(X0, q[0][k]); X1 = fmaxf(X1, q[0][k]);
            Y0 = fminf(Y0, q[1][k]); Y1 = fmaxf(Y1, q[1][k]);
        }
        const float Xl = X0 - dl, Xh = X1 + dl, Yl = Y0 - dl, Yh = Y1 + dl;
        const float in = 1.0f / near_s, is = rcp_approx(S1 + dl);
        a0 = fminf(Xl * in, Xl * is); a1 = fmaxf(Xh * in, Xh * is);
        b0 = fminf(Yl * in, Yl * is); b1 = fmaxf(Yh * in, Yh * is);
        a0 -= fabsf(a0) * 1e-6f; a1 += fabsf(a1) * 1e-6f;
        b0 -= fabsf(b0) * 1e-6f; b1 += fabsf(b1) * 1e-6f;
    }
    // pixel-centre coordinates of the pixel rays (the inverse of ray_dir), 0.5 pixel margin
    const float hw = 0.5f * (float)K.W, hh = 0.5f * (float)K.H;
    const float x0 = (a0 * K.iU + 1.0f) * hw - 1.0f, x1 = (a1 * K.iU + 1.0f) * hw;
    const float y0 = (1.0f - b1 * K.iV) * hh - 1.0f, y1 = (1.0f - b0 * K.iV) * hh;
    if (!(x1 >= 0.0f) || !(y1 >= 0.0f) || !(x0 < (float)K.W) || !(y0 < (float)K.H)) return false;
    rc.x = (int)fmaxf(floorf(x0 * (1.0f / kBeamTileW)), 0.0f);
    rc.y = (int)fmaxf(floorf(y0 * (1.0f / kBeamTileH)), 0.0f);
    rc.z = (int)fminf(floorf(x1 * (1.0f / kBeamTileW)) + 1.0f, (float)K.tiles_x);
    rc.w = (int)fminf(floorf(y1 * (1.0f / kBeamTileH)) + 1.0f, (float)K.tiles_y);
    return rc.z > rc.x && rc.w > rc.y;
}

// Occupied extent [lo, hi) of a 4^3 leaf mask along each axis (bit = x + 4y + 16z).
__device__ __forceinline__ void leaf_extent(uint64_t m, int lo[3], int hi[3]) {
    uint64_t t = m | (m >> 32);
    t |= t >> 16;
    const uint64_t tz = t;  // z folded
    t |= t >> 8;
    t |= t >> 4;
    const uint32_t xo = (uint32_t)(t & 0xFu);
    uint64_t ty = tz | (tz >> 2);
    ty |= ty >> 1;
    const uint32_t yo = (uint32_t)((ty & 1u) | ((ty >> 3) & 2u) | ((ty >> 6) & 4u) | ((ty >> 9) & 8u));
    uint64_t q = m | (m >> 8);
    q |= q >> 4;
    q |= q >> 2;
    q |= q >> 1;
    const uint32_t zo = (uint32_t)((q & 1u) | ((q >> 15) & 2u) | ((q >> 30) & 4u) | ((q >> 45) & 8u));
    const uint32_t o[3] = {xo, yo, zo};
#pragma unroll
    for (int a = 0; a < 3; a++) {
        lo[a] = __ffs(o[a]) - 1;
        hi[a] = 32 - __clz(o[a]);
    }
}

// A node's box (the box of its solid voxels the device header carries, in
// 16ths of the cell, or a leaf's set voxels), its L-inf distance from the
// origin and screen rectangle.  A region root's box is also clipped to the
// region's AABB (clip, ref: the region's entry; below the roots a node's
// solid voxels lie in that AABB already, so the clip would only trim the
// rounding to 16ths).  hdr: the
// interior node's header word, loaded here.  Returns false if the node cannot
// meet any pixel ray.
__device__ __forceinline__ bool node_bound(const BeamView& V, int lod, bool clip, const ChunkRef& ref, uint32_t chunk,
                                           uint32_t node, uint32_t packed_cell, int s, int4& rc, int32_t& D,
                                           uint32_t& hdr) {
    const SceneDev& S = V.scene;
    const bool leaf = s == lod + 2;
    int32_t u[3];
    u[0] = (int32_t)(chunk % (uint32_t)S.grid[0]);
    u[1] = (int32_t)((chunk / (uint32_t)S.grid[0]) % (uint32_t)S.grid[1]);
    u[2] = (int32_t)(chunk / ((uint32_t)S.grid[0] * (uint32_t)S.grid[1]));
    const int32_t cell[3] = {(int32_t)(packed_cell & 1023u), (int32_t)((packed_cell >> 10) & 1023u),
                             (int32_t)((packed_cell >> 20) & 1023u)};
    int32_t blo[3], bhi[3];
    if (leaf) {
        int l[3], h[3];
        leaf_extent(S.leaves[node], l, h);
#pragma unroll
        for (int a = 0; a < 3; a++) {
            blo[a] = cell[a] + (l[a] << lod);
            bhi[a] = cell[a] + (h[a] << lod);
        }
    } else {
        hdr = __ldg(S.nodes + node);
        const uint32_t q = hdr >> 8;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const int32_t ql = (int32_t)((q >> (8 * a)) & 15u), qh = (int32_t)((q >> (8 * a + 4)) & 15u) + 1;
            blo[a] = cell[a] + ((ql << s) >> 4);
            bhi[a] = cell[a] + (((qh << s) + 15) >> 4);
            if (clip) {
                blo[a] = max(blo[a], (int32_t)ref.aabb[a]);
                bhi[a] = min(bhi[a], (int32_t)ref.aabb[3 + a]);
            }
        }
    }
    // L-inf distance from the origin (exact, numerator units: |values| < 2^30)
    int32_t wl[3], wh[3];
    int32_t dmax = 0;
    float e2 = 0.0f;
    bool empty = false;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        empty = empty || blo[a] >= bhi[a];
        wl[a] = (((u[a] << S.mlog) + blo[a]) << kFix) - V.O[a];
        wh[a] = (((u[a] << S.mlog) + bhi[a]) << kFix) - V.O[a];
        const int32_t da = wl[a] > 0 ? wl[a] : (wh[a] < 0 ? -wh[a] : 0);
        dmax = max(dmax, da);
        e2 += (float)da * (float)da;
    }
    D = dmax;
    if (empty || (V.view_num > 0.0f && sqrtf(e2) > V.view_num)) return false;
    if ((float)D < V.near_dn) {
        rc = make_int4(0, 0, V.tiles_x, V.tiles_y);
        return true;
    }
    const float sc = 1.0f / (1 << kFix);
    const float lf[3] = {(float)wl[0] * sc, (float)wl[1] * sc, (float)wl[2] * sc};
    const float hf[3] = {(float)wh[0] * sc, (float)wh[1] * sc, (float)wh[2] * sc};
    return box_rect(V, lf, hf, rc);
}

// D into the finest level L of the view's bound pyramid (level 0: the tiles;
// level L: cells of 2^L x 2^L tiles) at which the rectangle spans at most 16
// cells (or the coarsest); the casting kernels take each tile's minimum over
// its cells.
__device__ __forceinline__ void scatter_bound(const BeamView& V, uint32_t tag, const int4& rc, int32_t D) {
    int L = 0;
    int x0 = rc.x, y0 = rc.y, x1 = rc.z - 1, y1 = rc.w - 1;
    while (L < kBeamPyr - 1 && (x1 - x0 + 1) * (y1 - y0 + 1) > 16) {
        L++;
        x0 >>= 1; y0 >>= 1; x1 >>= 1; y1 >>= 1;
    }
    unsigned long long* lv = V.bounds + beam_level_offset((uint32_t)V.tiles_x, (uint32_t)V.tiles_y, L);
    const int wl = (V.tiles_x + (1 << L) - 1) >> L;
    const unsigned long long v = ((unsigned long long)tag << 32) | (uint32_t)D;
    for (int y = y0; y <= y1; y++)
        for (int x = x0; x <= x1; x++) red_min_u64(&lv[(size_t)y * wl + x], v);
}

// A checked pass (ck.err set) that meets a node or leaf index outside its
// pool: the error code goes into the error word and the view is bounded by 0
// (no ray of it skips anything), in place of the loads.
__device__ __noinline__ void bad_index(const BeamHead& P, const BeamView& V, uint32_t code) {
    atomicOr(P.ck.err, code);
    scatter_bound(V, P.tag, make_int4(0, 0, V.tiles_x, V.tiles_y), 0);
}

// The whole pass in one cooperative launch (every block resident): the
// levels of the walk over all views with a grid-wide barrier after each,
// ending at the first level that queued nothing.  Level 0 takes every view's
// chunk regions, one lane each; a later level takes the queued nodes, eight
// lanes each, a lane projecting the child of its octant.  A projected node is
// scattered or queued to be refined; one whose rectangle is so large that its
// children will be refined as well (a child's is about a quarter of it) queues
// them at once, unprojected, so that about half the levels remain, and with
// them half the chains of dependent loads and barriers that bound the pass.
// (City 1920x1080, three views: 71 / 51 / 77 us for the pass that projected
// every level, one lane a node, refining above 8 tiles; 45 / 37 / 49 for this
// one above 16.  Above 8 it gains nothing: its levels hold too many nodes.)
// Every lane of a warp runs the same iterations (the queue reservation is
// warp-wide), and a level's warps are dealt over the SMs first.  A queued item
// carries what its children's bounds need (region, node, cell, side, view,
// LOD, child mask), so a level's chain of dependent loads starts at the item
// itself; each lane loads its first item beside the level's count and the
// next one while it works on the current one.  Queues are read through L2
// (written by other SMs before the barrier).  Bounds carry the pass's tag, so
// nothing has to be reset before the walk or folded after it; the queue
// counters are zeroed behind the walk, a level after their last reader.
template <class PB>
__device__ __forceinline__ void beam_walk(const PB& P) {
    cg::grid_group g = cg::this_grid();
    __shared__ uint32_t hist[kBeamLevels];
    const int lane = (int)(threadIdx.x & 31u);
    const uint32_t warp = (threadIdx.x >> 5) * gridDim.x + blockIdx.x, warps = (blockDim.x >> 5) * gridDim.x;
    const bool checked = P.ck.err != nullptr;
    if (threadIdx.x < kBeamLevels) {
        hist[threadIdx.x] = 0;
        if (blockIdx.x == 0) P.hist[threadIdx.x] = 0;  // (added to after the first barrier)
    }
    __syncthreads();
    for (int level = 0; level < kBeamLevels - 1; level++) {
        const uint4* qin = P.q[level & 1];
        uint4* qout = P.q[(level + 1) & 1];
        const uint32_t per = level == 0 ? 32u : 4u;  // items a warp takes at a time
        const uint32_t mine = level == 0 ? (uint32_t)lane : (uint32_t)lane >> 3;
        const uint32_t first = warp * per, stride = warps * per;
        uint4 nxt = make_uint4(kNoItem, 0u, 0u, 0u);
        if (level > 0 && first + mine < P.cap) nxt = __ldcg(qin + first + mine);
        const uint32_t n = level == 0 ? P.n_regions : min(*(volatile uint32_t*)&P.cnt[level], P.cap);
        if (level > 0 && blockIdx.x == 0 && threadIdx.x == 0) P.cnt[level - 1] = 0;
        if (n == 0) break;  // the same value in every thread after the barrier
        for (uint32_t base = first; base < n; base += stride) {
            const uint32_t i = base + mine;
            uint32_t kids = 0, ch[8], cm[8];
            uint32_t chunk = kNoItem, node = 0, cell = 0, vi = 0;  // the node this lane projects
            int s = 0, lod = 0;
            ChunkRef ref;
            if (level == 0) {
                if (i < n) {
                    // the view holding region item i: the last with region_begin <= i
                    uint32_t lo = 0, hi = P.n_views - 1;
                    while (lo < hi) {
                        const uint32_t mid = (lo + hi + 1) >> 1;
                        if (P.v[mid].region_begin <= i) lo = mid;
                        else hi = mid - 1;
                    }
                    const uint32_t r = i - P.v[lo].region_begin;
                    // a pass that selects first writes the region's frame entry here
                    ref = P.select ? select_one(P.v[lo].scene, P.cam, const_cast<ChunkRef*>(P.v[lo].frame), nullptr,
                                                nullptr, nullptr, (int)r)
                                   : P.v[lo].frame[r];
                    vi = lo;
                    if (ref.root != kNone) {
                        chunk = r;
                        node = ref.root;
                        s = P.v[lo].scene.mlog;
                        lod = (int)ref.lod;
                    }
                }
            } else {
                const uint4 it = nxt;
                nxt = make_uint4(kNoItem, 0u, 0u, 0u);
                if (i + stride < n) nxt = __ldcg(qin + i + stride);
                const uint32_t mask = it.w >> 24, o = (uint32_t)lane & 7u;
                if (i < n && it.x != kNoItem && ((mask >> o) & 1u)) {
                    vi = (it.w >> 8) & 0xFFu;
                    const uint64_t at = (uint64_t)it.y + 2 + 2 * __popc(mask & ((1u << o) - 1u));
                    if (checked && at + 2 > P.ck.n_nodes) {
                        bad_index(P, P.v[vi], 1u);
                    } else {
                        chunk = it.x;
                        node = __ldg(P.v[vi].scene.nodes + at);
                        s = (int)(it.w & 0xFFu) - 1;
                        lod = (int)((it.w >> 16) & 0xFFu);
                        const uint32_t h = 1u << s;
                        cell = it.z + ((o & 1u) ? h : 0u) + ((o & 2u) ? h << 10 : 0u) + ((o & 4u) ? h << 20 : 0u);
                    }
                }
            }
            const BeamView& V = P.v[vi];
            int4 rc;
            int32_t D = 0;
            int sk = s;  // side of the nodes this lane queues
            uint32_t mk = 0;
            if (chunk != kNoItem) {
                atomicAdd(&hist[min(V.scene.mlog - s, kBeamLevels - 1)], 1u);
                const bool leaf = s == lod + 2;
                uint32_t hdr = 0;
                if (checked && (leaf ? node >= P.ck.n_leaves : (uint64_t)node + 2 > P.ck.n_nodes)) {
                    bad_index(P, V, leaf ? 2u : 1u);
                } else if (node_bound(V, lod, level == 0, ref, chunk, node, cell, s, rc, D, hdr)) {
                    const uint32_t area = (uint32_t)(rc.z - rc.x) * (uint32_t)(rc.w - rc.y);
                    mk = hdr & 0xFFu;
                    const uint32_t k = (uint32_t)__popc(mk);
                    if (leaf || area <= P.expand || s <= P.smin) {
                        scatter_bound(V, P.tag, rc, D);
                    } else if (checked && (uint64_t)node + 2 + 2 * k > P.ck.n_nodes) {
                        bad_index(P, V, 1u);
                    } else if (area / 4u > P.expand && s - 1 > lod + 2 && s - 1 > P.smin) {
                        // its children, to be refined without a projection of their own
                        kids = k;
                        sk = s - 1;
#pragma unroll
                        for (int j = 0; j < 8; j++) {
                            uint2 w = make_uint2(0u, 0u);
                            if ((uint32_t)j < k) w = __ldg(reinterpret_cast<const uint2*>(V.scene.nodes + node + 2 + 2 * j));
                            ch[j] = w.x;
                            cm[j] = w.y >> 24;
                        }
                        if (s - lod == kWideLevel) {  // no child masks beside the pointers
#pragma unroll
                            for (int j = 0; j < 8; j++) {
                                if ((uint32_t)j < k && checked && (uint64_t)ch[j] + 2 > P.ck.n_nodes) {
                                    bad_index(P, V, 1u);
                                    ch[j] = node;  // (an index within the pool; the view skips nothing)
                                }
                                if ((uint32_t)j < k) cm[j] = __ldg(V.scene.nodes + ch[j]) & 0xFFu;
                            }
                        }
                        atomicAdd(&hist[min(V.scene.mlog - sk, kBeamLevels - 1)], k);
                    } else {
                        kids = 1;
                    }
                }
            }
            // queue them: one reservation per warp
            uint32_t pre = kids;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, pre, o);
                if (lane >= o) pre += v;
            }
            const uint32_t total = __shfl_sync(0xFFFFFFFFu, pre, 31);
            uint32_t wbase = 0;
            if (total) {
                if (lane == 31) wbase = atomicAdd(&P.cnt[level + 1], total);
                wbase = __shfl_sync(0xFFFFFFFFu, wbase, 31);
            }
            if (kids) {
                const uint32_t at = wbase + pre - kids;
                const uint32_t w = (uint32_t)sk | (vi << 8) | ((uint32_t)lod << 16);
                if (at + kids > P.cap) {
                    // queue full: this node stands for its children; its slots
                    // below the capacity are marked empty
                    for (uint32_t q = at; q < P.cap && q < at + kids; q++) qout[q] = make_uint4(kNoItem, 0u, 0u, 0u);
                    scatter_bound(V, P.tag, rc, D);
                } else if (sk == s) {
                    qout[at] = make_uint4(chunk, node, cell, w | mk << 24);
                } else {
                    const uint32_t h = 1u << sk;
                    uint32_t m = mk;
#pragma unroll
                    for (int q = 0; q < 8; q++) {
                        const int o = m ? __ffs((int)m) - 1 : 0;
                        m &= m - 1u;
                        const uint32_t c = cell + ((o & 1) ? h : 0u) + ((o & 2) ? h << 10 : 0u) + ((o & 4) ? h << 20 : 0u);
                        if ((uint32_t)q < kids) qout[at + q] = make_uint4(chunk, ch[q], c, w | cm[q] << 24);
                    }
                }
            }
        }
        g.sync();
    }
    __syncthreads();
    if (threadIdx.x < kBeamLevels && hist[threadIdx.x]) atomicAdd(&P.hist[threadIdx.x], hist[threadIdx.x]);
}

template <class PB>
__global__ void __launch_bounds__(kBeamThreads) beam_kernel(const __grid_constant__ PB P) {
    beam_walk(P);
}

}  // namespace

extern "C" {

unsigned aokk_beam_grid(int sms) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, beam_kernel<BeamBatch>, kBeamThreads, 0) != cudaSuccess ||
        per_sm < 1)
        return 0;
    return (unsigned)(sms > 0 ? sms : 1) * (unsigned)(per_sm < kBeamBlocksPerSM ? per_sm : kBeamBlocksPerSM);
}

bool aokk_beam_view(const SceneDev* S, const CamDev* C, const ChunkRef* frame, unsigned long long* bounds,
                    BeamView* out) {
    // A = [c0, c1, -c2] with d_i = R[3i] u + R[3i+1] v - R[3i+2]
    double A[9];
    for (int i = 0; i < 3; i++) {
        A[3 * i + 0] = C->R[3 * i + 0];
        A[3 * i + 1] = C->R[3 * i + 1];
        A[3 * i + 2] = -(double)C->R[3 * i + 2];
    }
    const double det = A[0] * (A[4] * A[8] - A[5] * A[7]) - A[1] * (A[3] * A[8] - A[5] * A[6]) +
                       A[2] * (A[3] * A[7] - A[4] * A[6]);
    double nrm = 0.0;
    for (int i = 0; i < 9; i++) nrm = fmax(nrm, fabs(A[i]));
    if (!(std::isfinite(det) && fabs(det) > 1e-6 * nrm * nrm * nrm)) return false;
    const double U = (double)C->tan_half * (double)C->W / (double)C->H, V = (double)C->tan_half;
    // Pixel rays whose components reach the ends of binary32 lose the precision
    // the tile margin counts on.  Elsewhere only the ratios of the matrix matter:
    // its largest entry is brought to [1/2, 2), so that the projection stays
    // clear of those ends too (the approximate reciprocal flushes those of
    // numbers above 2^126 to zero).
    if (!(nrm > 0x1p-122 && nrm * (U + V + 1.0) < 0x1p126)) return false;
    int ex = 0;
    (void)std::frexp(nrm, &ex);
    const double sc = ex < 0 || ex > 1 ? std::ldexp(1.0, -ex) : 1.0;
    for (int i = 0; i < 9; i++) A[i] *= sc;
    const double id = 1.0 / (det * sc * sc * sc);
    double Ai[9];
    Ai[0] = (A[4] * A[8] - A[5] * A[7]) * id;
    Ai[1] = (A[2] * A[7] - A[1] * A[8]) * id;
    Ai[2] = (A[1] * A[5] - A[2] * A[4]) * id;
    Ai[3] = (A[5] * A[6] - A[3] * A[8]) * id;
    Ai[4] = (A[0] * A[8] - A[2] * A[6]) * id;
    Ai[5] = (A[2] * A[3] - A[0] * A[5]) * id;
    Ai[6] = (A[3] * A[7] - A[4] * A[6]) * id;
    Ai[7] = (A[1] * A[6] - A[0] * A[7]) * id;
    Ai[8] = (A[0] * A[4] - A[1] * A[3]) * id;
    BeamView& K = *out;
    std::memset(&K, 0, sizeof(K));
    K.scene = *S;
    K.frame = frame;
    K.bounds = bounds;
    for (int i = 0; i < 9; i++) K.Af[i] = (float)Ai[i];
    K.iU = (float)(1.0 / U);
    K.iV = (float)(1.0 / V);
    // largest |d| component over the screen, with slack for the FP32 ray arithmetic
    double dmax = 0.0;
    for (int i = 0; i < 3; i++) dmax = fmax(dmax, fabs(A[3 * i]) * U + fabs(A[3 * i + 1]) * V + fabs(A[3 * i + 2]));
    K.near_dn = (float)(2.0 * kNearS * dmax * 1.01 * (double)(1 << kFix));
    K.view_num = S->view_dist > 0.0f ? (float)(((double)S->view_dist * 1.00001 + 1.0) * (double)(1 << kFix)) : 0.0f;
    K.W = C->W;
    K.H = C->H;
    K.tiles_x = (C->W + kBeamTileW - 1) / kBeamTileW;
    K.tiles_y = (C->H + kBeamTileH - 1) / kBeamTileH;
    for (int a = 0; a < 3; a++) K.O[a] = C->O[a];
    return true;
}

// Beam passes of this process run one after another on each device: a pass
// waits for the previous one, whatever stream either was launched on, so that
// two cooperative launches that each fill the GPU never wait for each other's
// blocks.
static std::mutex g_beam_mu;
static cudaEvent_t g_beam_done[kMaxBeamDevices];
static unsigned long long g_beam_stream[kMaxBeamDevices];  // that pass's stream

extern "C++" {
// Whether a pass on `st` would wait for another stream's work (g_beam_mu held).
static bool pass_waits(int dev, cudaStream_t st) {
    unsigned long long id = 0;
    if (!g_beam_done[dev] || (cudaStreamGetId(st, &id) == cudaSuccess && id == g_beam_stream[dev])) return false;
    // (in the relaxed mode: a query would end another stream's capture)
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    const cudaError_t e = cudaEventQuery(g_beam_done[dev]);
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (e == cudaSuccess) return false;
    cudaGetLastError();  // "not ready" is no error of the next launch
    return true;
}

static cudaError_t pass_done(int dev, cudaStream_t st) {
    const cudaError_t e = cudaStreamGetId(st, &g_beam_stream[dev]);
    return e == cudaSuccess ? cudaEventRecord(g_beam_done[dev], st) : e;
}
}  // extern "C++"

// The pass as a node of a CUDA graph (aokk_batch_run), with the launch shape
// aokk_beam_run uses.  argp: one slot, valid until the node is set.
void aokk_beam_node(const BeamBatch* P, unsigned grid, void** argp, cudaKernelNodeParams* kp) {
    argp[0] = (void*)P;
    kp->func = (void*)beam_kernel<BeamBatch>;
    kp->gridDim = dim3(grid);
    kp->blockDim = dim3(kBeamThreads);
    kp->sharedMemBytes = 0;
    kp->kernelParams = argp;
    kp->extra = nullptr;
}

// The per-device order of beam passes for work that holds passes but is not
// launched by aokk_beam_run (a graph): before (record = 0) the stream waits
// for the previous pass; after (record = 1) the end of the stream's work so
// far becomes the point the next pass waits for.
int aokk_beam_order(void* stream, int record) {
    const cudaStream_t st = (cudaStream_t)stream;
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return aokk_status(e);
    if (dev < 0 || dev >= kMaxBeamDevices) return aokk_status(cudaErrorInvalidDevice);
    std::lock_guard<std::mutex> lk(g_beam_mu);
    if (!g_beam_done[dev]) e = cudaEventCreateWithFlags(&g_beam_done[dev], cudaEventDisableTiming);
    if (e == cudaSuccess) e = record ? pass_done(dev, st) : cudaStreamWaitEvent(st, g_beam_done[dev], 0);
    return aokk_status(e);
}

int aokk_beam_waits(void* stream) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxBeamDevices) return 1;
    std::lock_guard<std::mutex> lk(g_beam_mu);
    return pass_waits(dev, (cudaStream_t)stream);
}

extern "C++" {
template <class PB>
static int launch_pass(const PB* P, unsigned grid, void* stream, bool optional = false) {
    const cudaStream_t st = (cudaStream_t)stream;
    if (P->n_views == 0) return AOK_OK;
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return aokk_status(e);
    if (dev < 0 || dev >= kMaxBeamDevices) return aokk_status(cudaErrorInvalidDevice);
    std::lock_guard<std::mutex> lk(g_beam_mu);
    if (optional && pass_waits(dev, st)) return AOK_E_BUSY;
    if (!g_beam_done[dev]) e = cudaEventCreateWithFlags(&g_beam_done[dev], cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, g_beam_done[dev], 0);
    void* args[] = {(void*)P};
    if (e == cudaSuccess) e = cudaLaunchCooperativeKernel((const void*)beam_kernel<PB>, grid, kBeamThreads, args, 0, st);
    if (e == cudaSuccess) e = pass_done(dev, st);
    return aokk_status(e);
}
}  // extern "C++"

int aokk_beam_run_view(const BeamParams<1>* P, unsigned grid, void* stream, int beside, int optional) {
    return launch_pass(P, beside && P->n_regions <= kWideWalkRegions ? (grid + kBeamBlocksPerSM - 1) / kBeamBlocksPerSM : grid,
                       stream, optional != 0);
}

int aokk_beam_run(const BeamBatch* P, unsigned grid, void* stream) {
    if (P->n_views != 1) return launch_pass(P, grid, stream);
    BeamParams<1> one;
    static_cast<BeamHead&>(one) = *P;
    one.v[0] = P->v[0];
    return launch_pass(&one, grid, stream);
}

}  // extern "C"
