// Tile-chunk rendering pipeline (Aokana Sec. 3.5, Fig. 7): the paper's own
// organisation of the primary-ray pass, kept beside the per-ray chunk march
// (aok_kernels.cu) as an alternative with identical output.
//
//   1. tile selection: every chunk region selected and visible this frame
//      (select_kernel) projects its AABB of valid voxels to a rectangle of
//      8x8-pixel tiles; each (tile, chunk) in it is a pair, with the distance
//      from the camera to the AABB as the pair's depth (a lower bound of every
//      hit in it, which is what the paper's AABB depth is).
//   2. ray marching, pass 1: every pair whose depth is not beyond the tile's
//      depth in the previous frame's Hi-Z is marched: each pixel ray of the
//      tile is traced through that chunk's DAG only, and its hit goes into a
//      screen-sized 64-bit visibility buffer with an atomic minimum (the
//      paper's InterlockedMax on an inverted depth).
//   3. Hi-Z of this frame from the visibility buffer (per-tile maximum of an
//      upper bound of each pixel's distance so far).
//   4. ray marching, pass 2: the pairs pass 1 culled are tested again
//      against this frame's Hi-Z and the survivors marched.
//   5. resolve: each pixel decodes its visibility record and writes the same
//      output record as the march; the per-tile maximum of the final
//      distances becomes the next frame's Hi-Z.
//
// Pass 2 makes the result independent of the previous frame: a pair it culls
// lies beyond every pixel's current hit in that tile, so it cannot hold a
// nearer one.  With the beam pass (aok_beam.cu) a half tile (8 x 4 pixels,
// one beam tile) also skips the pairs whose chunk AABB lies wholly nearer
// than its bound -- no voxel there can be met -- and its rays start each
// remaining pair at the bound's restart plane, as in the march.  Differences
// from the paper: the pair list is implicit (a prefix sum over the chunks'
// rectangle areas, front to back, stepped through by the marching warps)
// instead of an appended TileInfo buffer with indirect dispatch; the key is
// the march order; each marching warp takes half a tile (32 pixels).
//
// Visibility record: 64 bits per pixel, installed by an atomic minimum.  From
// the top:
//   the place of the chunk region in the march order along the ray: the sum
//       of its mirrored grid coordinates, which grows by one from each region
//       of a ray's march to the next;
//   the region's grid coordinates along its two shorter axes (the third
//       follows from the order): at most 19 bits with the order for the 65,536
//       regions a scene may have;
//   40 bits of the hit: the voxel's index in the region's DAG (9 bits per
//       axis), its LOD (3), the entry axis (2; 3: origin inside), the material
//       (8) -- with the ray, everything the output record needs.
// The minimum is the hit of the first region along the ray that has one, the
// march's answer.  (The paper's record has the depth on top, which orders the
// hits of different chunks as the march does, but needs a division a hit, and
// here an FP64 one so that keys cannot misorder.)  City 1920x1080, changing
// views: 1236 us a frame with 32-bit depth keys and a 128-bit compare-and-swap
// of key and payload, exact 64-bit comparisons and regions in index order; 645
// with this record, the FP32 walk (aok_walk.cuh) and regions front to back.
#include <cuda_runtime.h>

#include <cstdint>

#include "aok_internal.h"
#include "aok_ptx.cuh"
#include "aok_trace.cuh"
#include "aok_walk.cuh"

using namespace aok;

namespace {

constexpr unsigned long long kNoKey = ~0ull;
constexpr int kHitBits = 40;  // a record's bits below the region's
enum { kStList = 0, kStTraced1, kStCulled1, kStTraced2, kStCulled2, kStPixelTraces, kStPixelSkips };

__device__ __forceinline__ void region_coords(const SceneDev& S, uint32_t chunk, int32_t u[3]) {
    u[0] = (int32_t)(chunk % (uint32_t)S.grid[0]);
    u[1] = (int32_t)((chunk / (uint32_t)S.grid[0]) % (uint32_t)S.grid[1]);
    u[2] = (int32_t)(chunk / ((uint32_t)S.grid[0] * (uint32_t)S.grid[1]));
}

// The record of a hit in region u (order: its place in the march order).
__device__ __forceinline__ unsigned long long pack_hit(const SceneDev& S, const TileDev& T, const int32_t u[3],
                                                       uint32_t order, uint32_t mir, int n, const HitRec& hit,
                                                       uint32_t mat) {
    const int32_t side = (1 << (S.mlog - n)) - 1;
    unsigned long long r = 0;
#pragma unroll
    for (int a = 0; a < 3; a++)
        r |= (unsigned long long)(uint32_t)(((mir >> a) & 1u) ? side - hit.c[a] : hit.c[a]) << (9 * a);
    r |= (unsigned long long)n << 27 | (unsigned long long)hit.e << 30 | (unsigned long long)mat << 32;
    const unsigned long long reg = ((unsigned long long)order << (T.ba + T.bb)) |
                                   ((unsigned long long)(uint32_t)sel3(T.ax[0], u[0], u[1], u[2]) << T.bb) |
                                   (uint32_t)sel3(T.ax[1], u[0], u[1], u[2]);
    return reg << kHitBits | r;
}

// A record decoded for its ray (direction d): voxel corner, LOD, entry axis,
// material and the hit distance, as emit_hit computes it.
struct VisHit {
    uint32_t c[3], mat;
    int n, e;
    uint32_t normal;
    float dist;
};
__device__ __forceinline__ VisHit unpack_hit(const SceneDev& S, const CamDev& C, const TileDev& T,
                                             unsigned long long key, const float d[3]) {
    const uint32_t mir = (d[0] < 0.0f ? 1u : 0u) | (d[1] < 0.0f ? 2u : 0u) | (d[2] < 0.0f ? 4u : 0u);
    const uint32_t reg = (uint32_t)(key >> kHitBits);
    const int32_t ua = (int32_t)((reg >> T.bb) & ((1u << T.ba) - 1u)), ub = (int32_t)(reg & ((1u << T.bb) - 1u));
    const int a0 = T.ax[0], a1 = T.ax[1], a2 = T.ax[2];
    auto mirrored = [&](int a, int32_t v) {
        return ((mir >> a) & 1u) ? sel3(a, S.grid[0], S.grid[1], S.grid[2]) - 1 - v : v;
    };
    const int32_t uc = mirrored(a2, (int32_t)(reg >> (T.ba + T.bb)) - mirrored(a0, ua) - mirrored(a1, ub));
    VisHit h;
    h.n = (int)((key >> 27) & 7u);
    h.e = (int)((key >> 30) & 3u);
    h.mat = (uint32_t)(key >> 32) & 0xFFu;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const int32_t u = a == a0 ? ua : (a == a1 ? ub : uc);
        h.c[a] = (uint32_t)((u << S.mlog) + (int32_t)(((uint32_t)(key >> (9 * a)) & 511u) << h.n));
    }
    h.dist = 0.0f;
    h.normal = 7u;
    if (h.e < 3) {
        // entry plane: the voxel's face the mirrored ray meets first, as a numerator
        const bool m = (mir >> h.e) & 1u;
        const int32_t we = (int32_t)sel3(h.e, h.c[0], h.c[1], h.c[2]), G = sel3(h.e, S.grid[0], S.grid[1], S.grid[2]),
                      O = sel3(h.e, C.O[0], C.O[1], C.O[2]);
        const int32_t face = m ? (G << S.mlog) - we - (1 << h.n) : we;
        const int32_t Ow = m ? (G << (S.mlog + kFix)) - O : O;
        const int32_t Ne = (int32_t)((uint32_t)face << kFix) - Ow;
        RayState r;
        r.d[0] = d[0];
        r.d[1] = d[1];
        r.d[2] = d[2];
        h.dist = __fdiv_rn((float)Ne * (1.0f / 4096.0f), fabsf(sel3(h.e, d[0], d[1], d[2]))) * ray_norm(r);
        h.normal = (uint32_t)(2 * h.e) + ((mir >> h.e) & 1u);
    }
    return h;
}

// How the march enters chunk region u: entry axis e (3: the origin lies in
// it), entry plane numerator Ne, mirrored local origin.  Returns false when
// the march does not visit the region.  A region the ray passes with positive
// length is visited; one it only touches (entry instant = exit instant, an
// edge or corner) is visited when every axis it is left through has a lower
// index than every axis it is entered through, because at a tie the march
// steps the axis of higher index first.  Rays that enter the world box
// exactly on an interior chunk plane are the one case decided differently
// (the march places them past the plane).
struct Entry {
    int e;
    int32_t Ne;
    int32_t Oloc[3];
    int32_t Hi[3];  // exit plane numerators of the region
    uint32_t order;
};

template <bool FAST>
__device__ __forceinline__ bool enter_region(const SceneDev& S, const CamDev& C, const RayState& r,
                                             const int32_t u[3], Entry& en) {
    const int cs = S.mlog + kFix;
    int32_t Lo[3], Hi[3];
    uint32_t order = 0;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const bool m = (r.mir >> a) & 1u;
        const int32_t Wfix = S.grid[a] << cs;
        const int32_t Ow = m ? Wfix - C.O[a] : C.O[a];
        const int32_t cc = m ? S.grid[a] - 1 - u[a] : u[a];
        order += (uint32_t)cc;
        Lo[a] = (cc << cs) - Ow;
        Hi[a] = ((cc + 1) << cs) - Ow;
        en.Oloc[a] = -Lo[a];
        en.Hi[a] = Hi[a];
    }
#pragma unroll
    for (int a = 0; a < 3; a++) {
        if (Hi[a] <= 0) return false;                      // behind the origin
        if (r.d[a] == 0.0f && Lo[a] > 0) return false;     // parallel slab missed
    }
    int e = 3;
    int32_t Ne = 0, me = 1, Ee = 0;
#pragma unroll
    for (int a = 0; a < 3; a++)  // latest entry plane; ties keep the lowest axis
        if (Lo[a] > 0 && (e == 3 || tltf<FAST>(Ne, me, Lo[a], r.m[a], r.E[a] - Ee))) {
            e = a; Ne = Lo[a]; me = r.m[a]; Ee = r.E[a];
        }
    if (e < 3) {
        int maxpre = -1;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            if (r.d[a] == 0.0f) continue;
            if (tltf<FAST>(Hi[a], r.m[a], Ne, me, Ee - r.E[a])) return false;  // left before entered
            if (!tltf<FAST>(Ne, me, Hi[a], r.m[a], r.E[a] - Ee)) maxpre = a;    // left at the entry instant
        }
        if (maxpre > e) return false;
    }
    en.e = e;
    en.Ne = Ne;
    en.order = order;
    return true;
}

// The march's skip of regions whose solid-voxel AABB (grown by 1/16 voxel)
// the ray misses, with the same FP32 arithmetic.
__device__ __forceinline__ bool aabb_pass(const SceneDev& S, const CamDev& C, const RayState& r, const ChunkRef& ref,
                                          const int32_t u[3]) {
    float tn = 0.0f, tf = 3.0e38f;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const float lo = (float)((u[a] << S.mlog) + ref.aabb[a]) - 0.0625f;
        const float hi = (float)((u[a] << S.mlog) + ref.aabb[3 + a]) + 0.0625f;
        if (r.d[a] == 0.0f) {
            if (C.of[a] < lo || C.of[a] > hi) return false;
        } else {
            const float inv = 1.0f / r.d[a];
            const float t1 = (lo - C.of[a]) * inv, t2 = (hi - C.of[a]) * inv;
            tn = fmaxf(tn, fminf(t1, t2));
            tf = fminf(tf, fmaxf(t1, t2));
        }
    }
    return tn <= tf;
}

// One pixel of a pair with exact comparisons throughout: 0 = region not
// entered, 1 = traced, 2 = skipped (the pixel already holds a hit of an earlier
// region, or the beam bound Dn puts every voxel the ray can meet past the
// region).  Dn > 0: the
// ray starts at the bound's restart plane when that lies later than the
// region's entry (trace_pixel_t's beam restart, within one region).
template <bool FAST, bool BEAM>
__device__ __forceinline__ int pair_pixel(const SceneDev& S, const CamDev& C, const ChunkRef& ref, uint32_t chunk,
                                          const RayState& r, size_t pix, const TileDev& T, int32_t Dn) {
    int32_t u[3];
    region_coords(S, chunk, u);
    Entry en;
    if (!enter_region<FAST>(S, C, r, u, en) || !aabb_pass(S, C, r, ref, u)) return 0;
    const unsigned long long cur = __ldcg(T.vis + pix);
    if (cur != kNoKey && (uint32_t)(cur >> kHitBits) >> (T.ba + T.bb) < en.order) return 2;
    int e = en.e;
    int32_t Ne = en.Ne;
    if (BEAM && Dn > 0) {
        // the last integer plane of the dominant axis crossed before the ray's
        // L-inf distance reaches Dn; at or past the region's exit: no hit here
        int as = 0;
        if (fabsf(r.d[1]) > fabsf(r.d[as])) as = 1;
        if (fabsf(r.d[2]) > fabsf(r.d[as])) as = 2;
        const int32_t Wf = S.grid[as] << (S.mlog + kFix);
        const int32_t Ow = ((r.mir >> as) & 1u) ? Wf - C.O[as] : C.O[as];
        const long long kp = ((long long)Dn - 1 + Ow) >> kFix;
        const long long Nl = (kp << kFix) - Ow;
        if (Nl >= (long long)en.Hi[as]) return 2;
        const int32_t me = e < 3 ? r.m[e] : 1, Ee = e < 3 ? r.E[e] : 0;
        if (Nl > 0 && (e == 3 || tltf<FAST>(Ne, me, (int32_t)Nl, r.m[as], r.E[as] - Ee))) {
#pragma unroll
            for (int a = 0; a < 3; a++)
                if (a != as && r.d[a] != 0.0f && !tltf<FAST>((int32_t)Nl, r.m[as], en.Hi[a], r.m[a], r.E[a] - r.E[as]))
                    return 2;  // the ray leaves the region no later than the restart point
            e = as;
            Ne = (int32_t)Nl;
        }
    }
    HitRec hit;
    Counters cnt = {0, 0, 0};
    if (trace_chunk<FAST, false, false, BEAM>(S, ref, r, en.Oloc, e, Ne, hit, cnt) &&
        (lowest_entry_face<FAST>(r, en.Oloc, (int)ref.lod, hit), within_view(S, r, hit))) {
        red_min_u64(T.vis + pix, pack_hit(S, T, u, en.order, r.mir, (int)ref.lod, hit, hit_material(S, ref, hit.idx)));
    }
    return 1;
}

// The exact version as the fallback of pair_walk (out of line: rare).
template <bool BEAM>
__device__ __noinline__ int pair_exact(const SceneDev& S, const CamDev& C, const ChunkRef* __restrict__ frame,
                                       uint32_t chunk, int px, int py, const TileDev& T, int32_t Dn) {
    const ChunkRef ref = frame[chunk];
    RayState r;
    const size_t pix = (size_t)py * C.W + px;
    return make_ray(C, px, py, r) ? pair_pixel<true, BEAM>(S, C, ref, chunk, r, pix, T, Dn)
                                  : pair_pixel<false, BEAM>(S, C, ref, chunk, r, pix, T, Dn);
}

// One pixel of a pair (results of pair_pixel): entry, skip tests and walk in
// FP32 as in walk_pixel, the exact version where a decision is left open.
// Called by all lanes of a warp for the same pair; `in`: the lane has a pixel.
template <bool BEAM>
__device__ __forceinline__ int pair_walk(const SceneDev& S, const CamDev& C, const ChunkRef* __restrict__ frame,
                                         uint32_t chunk, bool in, int px, int py, const TileDev& T, int32_t Dn) {
    const uint4* fr = reinterpret_cast<const uint4*>(frame + chunk);
    const uint4 ra = __ldg(fr), rb = __ldg(fr + 1);
    const size_t pix = (size_t)py * C.W + px;
    float d[3];
    ray_dir(C, px, py, d);
    const uint32_t mir = (d[0] < 0.0f ? 1u : 0u) | (d[1] < 0.0f ? 2u : 0u) | (d[2] < 0.0f ? 4u : 0u);
    WalkRay w;
    w.dmax = fmaxf(fmaxf(fabsf(d[0]), fabsf(d[1])), fabsf(d[2]));
    bool undecided = !(w.dmax > 0x1p-40f && w.dmax < 0x1p40f);
    w.gmax = 0.0f;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        w.ad[a] = fabsf(d[a]);
        w.inv[a] = w.ad[a] > 0.0f ? rcp_approx(w.ad[a]) : kZeroInv;
        if (w.ad[a] > 0.0f) w.gmax = fmaxf(w.gmax, w.inv[a]);
    }
    int32_t u[3], Ow[3], cc[3], Hi[3];
    region_coords(S, chunk, u);
    const int cs = S.mlog + kFix;
    const int32_t M = 1 << S.mlog;
    const int32_t alo[3] = {(int32_t)(rb.x & 0xFFFFu), (int32_t)(rb.x >> 16), (int32_t)(rb.y & 0xFFFFu)};
    const int32_t ahi[3] = {(int32_t)(rb.y >> 16), (int32_t)(rb.z & 0xFFFFu), (int32_t)(rb.z >> 16)};
    uint32_t order = 0;
    int e = 3;
    int32_t Ne = 0;
    bool enter = in;
    float tin = -1.0f, tin2 = -1.0f, tout = 3.0e38f, tn = 0.0f, tf = 3.0e38f;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const bool m = (mir >> a) & 1u;
        Ow[a] = m ? (S.grid[a] << cs) - C.O[a] : C.O[a];
        cc[a] = m ? S.grid[a] - 1 - u[a] : u[a];
        order += (uint32_t)cc[a];
        const int32_t Lo = (cc[a] << cs) - Ow[a];
        Hi[a] = Lo + (1 << cs);
        if (Hi[a] <= 0 || (w.ad[a] == 0.0f && Lo > 0)) enter = false;
        const float ti = Lo > 0 ? (float)Lo * w.inv[a] : -1.0f;
        tout = fminf(tout, (float)Hi[a] * w.inv[a]);
        if (ti > tin) { tin2 = tin; tin = ti; e = a; Ne = Lo; }
        else tin2 = fmaxf(tin2, ti);
        // the solid voxels' box grown by 1/16 voxel
        tn = fmaxf(tn, (float)(Lo + ((m ? M - ahi[a] : alo[a]) << kFix) - 256) * w.inv[a]);
        tf = fminf(tf, (float)(Lo + ((m ? M - alo[a] : ahi[a]) << kFix) + 256) * w.inv[a]);
    }
    if (!undecided && tin > tout * (1.0f + kWalkEps)) enter = false;
    else if (!(tin < tout * (1.0f - kWalkEps) && (e == 3 || tin2 < tin * (1.0f - kWalkEps)))) undecided = true;
    if (!undecided && tn > tf) enter = false;
    undecided = undecided && enter;
    int res = 0;
    bool traced = enter && !undecided;
    if (traced) {
        res = 1;
        const unsigned long long cur = __ldcg(T.vis + pix);
        if (cur != kNoKey && (uint32_t)(cur >> kHitBits) >> (T.ba + T.bb) < order) res = 2;
        if (BEAM && Dn > 0) {
            // the last integer plane of the dominant axis crossed before the ray's
            // L-inf distance reaches Dn; at or past the region's exit: no hit here
            int as = 0;
            if (w.ad[1] > w.ad[0]) as = 1;
            if (w.ad[2] > fmaxf(w.ad[0], w.ad[1])) as = 2;
            const int32_t O = sel3(as, Ow[0], Ow[1], Ow[2]);
            const long long Nl = ((((long long)Dn - 1 + O) >> kFix) << kFix) - O;
            if (Nl >= (long long)sel3(as, Hi[0], Hi[1], Hi[2])) {
                res = 2;
            } else if (Nl > 0) {
                const float ts = (float)(int32_t)Nl * sel3(as, w.inv[0], w.inv[1], w.inv[2]);
                if (ts > tout * (1.0f + kWalkEps)) {
                    res = 2;  // left the region before the restart point
                } else if (ts < tout * (1.0f - kWalkEps) && (e == 3 || ts > tin * (1.0f + kWalkEps))) {
                    e = as;
                    Ne = (int32_t)Nl;
                }
            }
        }
        traced = res == 1;
    }
    int32_t B[3];
    float x[3];
    int eb = 0;
    HitRec hit;
    if (traced && !walk_base<false>(w, Ow, e, Ne, B, x)) {
        undecided = true;
        traced = false;
    }
    bool found = false;
    if (__any_sync(0xFFFFFFFFu, traced))
        found = walk_chunk<false>(S, w, mir, Ow, cc, traced, true, ra.x, (int)ra.y, e, Ne, eb, B, x, undecided, hit);
    if (found) {
        const int n = (int)ra.y;
        RayState r;
        hit.Ne = 0;
        if (e < 3)
            hit.Ne = (((sel3(e, cc[0], cc[1], cc[2]) << S.mlog) + (sel3(e, hit.c[0], hit.c[1], hit.c[2]) << n)) << kFix) -
                     sel3(e, Ow[0], Ow[1], Ow[2]);
#pragma unroll
        for (int a = 0; a < 3; a++) r.d[a] = d[a];
        if (within_view(S, r, hit)) {
            ChunkRef ref;
            ref.mat_base = (uint64_t)ra.z | (uint64_t)ra.w << 32;
            ref.nblocks = rb.w;
            red_min_u64(T.vis + pix, pack_hit(S, T, u, order, mir, n, hit, hit_material(S, ref, hit.idx)));
        }
    }
    if (undecided) res = pair_exact<BEAM>(S, C, frame, chunk, px, py, T, Dn);
    return res;
}

// ---------------------------------------------------------------------------
// 1. tile selection: per chunk region, its tile rectangle and depth
// ---------------------------------------------------------------------------
// Eight lanes per region (lane k projects corner k of its AABB; FP64 is a
// slow pipe on this GPU, so the corners are spread over more SMs).
__global__ void __launch_bounds__(128) tc_rect_kernel(SceneDev S, CamDev C, const ChunkRef* __restrict__ frame,
                                                      TileDev T) {
    const int nch = S.grid[0] * S.grid[1] * S.grid[2];
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int chunk = tid >> 3, k = tid & 7;
    const bool valid = chunk < nch;
    const ChunkRef ref = valid ? frame[chunk] : ChunkRef{kNone, 0, 0, {0, 0, 0, 0, 0, 0}, 0};
    uint32_t area = 0;
    int4 rc = make_int4(0, 0, 0, 0);
    float dm = 0.0f;
    int32_t far = 0;
    // the group's lanes agree on every branch below (same region)
    const bool live = valid && ref.root != kNone;
    double lo[3] = {0.0, 0.0, 0.0}, hi[3] = {0.0, 0.0, 0.0};
    if (live) {
        int32_t u[3];
        region_coords(S, (uint32_t)chunk, u);
        double d2 = 0.0;
#pragma unroll
        for (int a = 0; a < 3; a++) {  // exact: |values| < 2^30
            const int32_t l = (((u[a] << S.mlog) + (int32_t)ref.aabb[a]) << kFix) - C.O[a];
            const int32_t h = (((u[a] << S.mlog) + (int32_t)ref.aabb[3 + a]) << kFix) - C.O[a];
            far = max(far, max(abs(l), abs(h)));
            lo[a] = (double)((u[a] << S.mlog) + ref.aabb[a]) - (double)C.of[a];
            hi[a] = (double)((u[a] << S.mlog) + ref.aabb[3 + a]) - (double)C.of[a];
            const double q = fmax(fmax(lo[a], -hi[a]), 0.0);
            d2 += q * q;
        }
        // every hit point of the region lies in the AABB: its distance is >= this
        if (k == 0) dm = __double2float_rd(sqrt(d2) * (1.0 - 1e-12));
    }
    dm = __shfl_sync(0xFFFFFFFFu, dm, 0, 8);
    const bool project = live && !(S.view_dist > 0.0f && dm > S.view_dist);
    // screen position of corner k (pixel-centre coordinates); a corner near or
    // behind the camera plane makes the rectangle the whole screen
    double px = 0.0, py = 0.0;
    bool full = false;
    if (project) {
        const double th = C.tan_half, asp = (double)C.W / (double)C.H;
        const double p0 = (k & 1) ? hi[0] : lo[0], p1 = (k & 2) ? hi[1] : lo[1], p2 = (k & 4) ? hi[2] : lo[2];
        const double xc = C.R[0] * p0 + C.R[3] * p1 + C.R[6] * p2;
        const double yc = C.R[1] * p0 + C.R[4] * p1 + C.R[7] * p2;
        const double zc = -(C.R[2] * p0 + C.R[5] * p1 + C.R[8] * p2);
        if (zc < 1e-3 * (fabs(p0) + fabs(p1) + fabs(p2) + 1.0)) {
            full = true;
        } else {
            px = (xc / zc / (th * asp) + 1.0) * 0.5 * C.W - 0.5;
            py = (1.0 - yc / zc / th) * 0.5 * C.H - 0.5;
        }
    }
    double x0 = full ? 1e300 : px, x1 = full ? -1e300 : px, y0 = full ? 1e300 : py, y1 = full ? -1e300 : py;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        x0 = fmin(x0, __shfl_xor_sync(0xFFFFFFFFu, x0, o, 8));
        x1 = fmax(x1, __shfl_xor_sync(0xFFFFFFFFu, x1, o, 8));
        y0 = fmin(y0, __shfl_xor_sync(0xFFFFFFFFu, y0, o, 8));
        y1 = fmax(y1, __shfl_xor_sync(0xFFFFFFFFu, y1, o, 8));
        const int fo = __shfl_xor_sync(0xFFFFFFFFu, (int)full, o, 8);  // every lane shuffles
        full = full || fo;
    }
    if (project) {
        if (full) {
            rc = make_int4(0, 0, T.tiles_x, T.tiles_y);
        } else {  // 2 px margin
            rc.x = (int)fmax(floor((x0 - 2.0) / 8.0), 0.0);
            rc.y = (int)fmax(floor((y0 - 2.0) / 8.0), 0.0);
            rc.z = (int)fmin(floor((x1 + 2.0) / 8.0) + 1.0, (double)T.tiles_x);
            rc.w = (int)fmin(floor((y1 + 2.0) / 8.0) + 1.0, (double)T.tiles_y);
        }
        if (rc.z > rc.x && rc.w > rc.y) area = (uint32_t)(rc.z - rc.x) * (uint32_t)(rc.w - rc.y);
    }
    if (valid && k == 0) {
        T.rect[chunk] = rc;
        T.dmin[chunk] = dm;
        T.dfar[chunk] = far;
        T.area[chunk] = area;
    }
}

// Lists the regions with pairs front to back -- by the leading bits of their
// depth, so that most of a pixel's farther pairs meet a record that ends them
// -- and their exclusive area prefix (one block); zeroes the frame's
// statistics.
constexpr int kDepthBuckets = 4096;  // exponent and 4 bits of the depth's mantissa
__device__ __forceinline__ uint32_t depth_bucket(float dm) {
    return min(__float_as_uint(fmaxf(dm, 0.0f)) >> 19, (uint32_t)kDepthBuckets - 1u);
}
__global__ void __launch_bounds__(1024) tc_scan_kernel(int nch, TileDev T) {
    __shared__ uint32_t s_hist[kDepthBuckets];
    __shared__ unsigned long long s_sum[1024];
    const int tid = threadIdx.x;
    // exclusive prefix over the block of one value per thread; the last entry is the total
    auto scan = [&](unsigned long long v) -> unsigned long long {
        s_sum[tid] = v;
        __syncthreads();
        for (int off = 1; off < 1024; off <<= 1) {
            const unsigned long long p = tid >= off ? s_sum[tid - off] : 0ull;
            __syncthreads();
            s_sum[tid] += p;
            __syncthreads();
        }
        return s_sum[tid] - v;
    };
    for (int i = tid; i < kDepthBuckets; i += 1024) s_hist[i] = 0;
    __syncthreads();
    for (int i = tid; i < nch; i += 1024)
        if (T.area[i]) atomicAdd(&s_hist[depth_bucket(T.dmin[i])], 1u);
    __syncthreads();
    uint32_t h[kDepthBuckets / 1024];
    uint32_t cnt = 0;
#pragma unroll
    for (int k = 0; k < kDepthBuckets / 1024; k++) {
        h[k] = cnt;
        cnt += s_hist[tid * (kDepthBuckets / 1024) + k];
    }
    const uint32_t at = (uint32_t)scan(cnt);
    const uint32_t n_list = (uint32_t)s_sum[1023];
#pragma unroll
    for (int k = 0; k < kDepthBuckets / 1024; k++) s_hist[tid * (kDepthBuckets / 1024) + k] = at + h[k];
    __syncthreads();
    for (int i = tid; i < nch; i += 1024)
        if (T.area[i]) T.list[atomicAdd(&s_hist[depth_bucket(T.dmin[i])], 1u)] = (uint32_t)i;
    __syncthreads();
    const uint32_t per = (n_list + 1023) / 1024;
    const uint32_t b = min((uint32_t)tid * per, n_list), e = min(b + per, n_list);
    unsigned long long sum = 0;
    for (uint32_t i = b; i < e; i++) sum += T.area[T.list[i]];
    unsigned long long base = scan(sum);
    for (uint32_t i = b; i < e; i++) {
        T.offs[i] = base;
        base += T.area[T.list[i]];
    }
    if (tid == 1023) {
        T.offs[n_list] = s_sum[1023];
        T.stats[kStList] = n_list;
    }
    if (tid > 0 && tid < kTileStats) T.stats[tid] = 0ull;
}

// ---------------------------------------------------------------------------
// 2./4. ray marching of the pairs: each warp takes half a tile (8 x 4 pixels)
// of one pair; warps stride over all 2 x pairs items.  PASS 1 marches the
// pairs the previous frame's Hi-Z keeps, PASS 2 those it culled and this
// frame's keeps.  A warp tests its next 32 items together, one per lane, and
// then marches those that are left: an item's test is a chain of five
// dependent loads, which the warp waited for item by item before (five views of
// city 1920x1080 637 / 372 / 630 / 470 / 483 -> 560 / 324 / 512 / 365 / 408 us a
// frame).  Items a warp takes are far apart on purpose: dear ones are neighbours
// (tickets of 4 / 8 / 16 items from a counter 628 / 675 / 757 us on the first view).
// ---------------------------------------------------------------------------
// The beam-pass bound of the 8 x 4 tile (x, y).
__device__ __forceinline__ int32_t tile_bound(const BeamLookup& b, uint32_t x, uint32_t y) {
    unsigned long long v = ~0ull;
#pragma unroll
    for (int L = 0; L < kBeamPyr; L++) v = min(v, __ldcg(b.bounds + b.off[L] + (y >> L) * b.wl[L] + (x >> L)));
    return (uint32_t)(v >> 32) == b.tag ? (int32_t)(uint32_t)v : INT_MAX;
}

template <int PASS, bool BEAM>
__global__ void __launch_bounds__(128, 7) tc_cast_kernel(const __grid_constant__ SceneDev S,
                                                      const __grid_constant__ CamDev C,
                                                      const ChunkRef* __restrict__ frame,
                                                      const __grid_constant__ TileDev T, const BeamLookup beam) {
    const uint32_t n_list = (uint32_t)T.stats[kStList];
    if (n_list == 0) return;
    const unsigned long long n_items = 2ull * T.offs[n_list];
    const int lane = threadIdx.x & 31;
    const unsigned long long nw = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
    __shared__ int4 s_item[4][32];  // {region, tile x, half tile y, bound}
    int4* items = s_item[threadIdx.x >> 5];
    uint32_t traced = 0, culled = 0, pix_traced = 0, pix_skipped = 0, lo = 0;
    for (unsigned long long first = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; first < n_items;
         first += 32 * nw) {
        const unsigned long long item = first + (unsigned)lane * nw;
        bool live = item < n_items;
        if (live) {
            const unsigned long long pair = item >> 1;
            while (lo + 1 < n_list && T.offs[lo + 1] <= pair) lo++;  // last listed region with offs <= pair
            const uint32_t chunk = T.list[lo];
            const uint32_t local = (uint32_t)(pair - T.offs[lo]);
            const int4 rc = T.rect[chunk];
            const int rw = rc.z - rc.x;
            const int tx = rc.x + (int)(local % (uint32_t)rw), ty = rc.y + (int)(local / (uint32_t)rw);
            const int tile = ty * T.tiles_x + tx;
            const float dm = T.dmin[chunk];
            const int by = ty * 2 + (int)(item & 1);  // the half tile: one beam tile
            bool cull;
            if (PASS == 1) {
                cull = dm > T.hiz_prev[tile];
            } else {
                live = dm > T.hiz_prev[tile];  // else marched in pass 1
                cull = live && dm > T.hiz[tile];
            }
            if (!cull && by * 4 >= C.H) live = false;  // below the last row
            int32_t Dn = 0;
            if (BEAM && live && !cull) {
                Dn = tile_bound(beam, (uint32_t)tx, (uint32_t)by);
                cull = Dn > T.dfar[chunk];  // wholly nearer than every voxel its rays meet
            }
            culled += cull;
            live = live && !cull;
            traced += live;
            items[lane] = make_int4((int)chunk, tx, by, Dn);
        }
        __syncwarp();
        for (uint32_t todo = __ballot_sync(0xFFFFFFFFu, live); todo; todo &= todo - 1u) {
            const int4 it = items[__ffs((int)todo) - 1];
            const int px = it.y * 8 + (lane & 7), py = it.z * 4 + (lane >> 3);
            const int res = pair_walk<BEAM>(S, C, frame, (uint32_t)it.x, px < C.W && py < C.H, px, py, T, it.w);
            pix_traced += res == 1;
            pix_skipped += res == 2;
            __syncwarp();
        }
    }
    traced = __reduce_add_sync(0xFFFFFFFFu, traced);
    culled = __reduce_add_sync(0xFFFFFFFFu, culled);
    pix_traced = __reduce_add_sync(0xFFFFFFFFu, pix_traced);
    pix_skipped = __reduce_add_sync(0xFFFFFFFFu, pix_skipped);
    if (lane == 0) {
        if (traced) atomicAdd(&T.stats[PASS == 1 ? kStTraced1 : kStTraced2], (unsigned long long)traced);
        if (culled) atomicAdd(&T.stats[PASS == 1 ? kStCulled1 : kStCulled2], (unsigned long long)culled);
        if (pix_traced) atomicAdd(&T.stats[kStPixelTraces], (unsigned long long)pix_traced);
        if (pix_skipped) atomicAdd(&T.stats[kStPixelSkips], (unsigned long long)pix_skipped);
    }
}

// ---------------------------------------------------------------------------
// 3. Hi-Z of this frame after pass 1: per tile, the maximum over its pixels of
// an upper bound of the distance of the pixel's hit so far (+inf: none yet).
// One warp per tile.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) tc_hiz_kernel(SceneDev S, CamDev C, TileDev T) {
    const int lane = threadIdx.x & 31;
    const int tile = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (tile >= T.tiles_x * T.tiles_y) return;
    const int tx = tile % T.tiles_x, ty = tile / T.tiles_x;
    float m = 0.0f;
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const int px = tx * 8 + (lane & 7), py = ty * 8 + k * 4 + (lane >> 3);
        if (px < C.W && py < C.H) {
            const unsigned long long key = __ldcg(T.vis + ((size_t)py * C.W + px));
            float dist = __int_as_float(0x7F800000);
            if (key != kNoKey) {
                float d[3];
                ray_dir(C, px, py, d);
                dist = __fmul_ru(unpack_hit(S, C, T, key, d).dist, 1.000001f);
            }
            m = fmaxf(m, dist);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
    if (lane == 0) T.hiz[tile] = m;
}

// ---------------------------------------------------------------------------
// 5. resolve: 16 x 8 pixel blocks (two tiles), warps of 8 x 4 pixels
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) tc_resolve_kernel(SceneDev S, CamDev C, const ChunkRef* __restrict__ frame,
                                                         TileDev T, uint4* __restrict__ out_hit,
                                                         float* __restrict__ out_t) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tx = blockIdx.x * 2 + (warp & 1), ty = blockIdx.y;
    const int px = tx * 8 + (lane & 7);
    const int py = ty * 8 + (warp >> 1) * 4 + (lane >> 3);
    float dist_up = 0.0f;
    if (px < C.W && py < C.H) {
        const size_t pix = (size_t)py * C.W + px;
        const unsigned long long key = __ldcg(T.vis + pix);
        if (key == kNoKey) {
            emit_miss(out_hit, out_t, pix);
            dist_up = __int_as_float(0x7F800000);
        } else {
            // the output record of emit_hit, rebuilt from the record and the ray
            float d[3];
            ray_dir(C, px, py, d);
            const VisHit h = unpack_hit(S, C, T, key, d);
            out_hit[pix] = make_uint4(h.c[0], h.c[1], h.c[2],
                                      (uint32_t)h.n | (h.mat << 8) | (h.normal << 16) | (1u << 19));
            out_t[pix] = h.dist;
            dist_up = __fmul_ru(h.dist, 1.000001f);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dist_up = fmaxf(dist_up, __shfl_xor_sync(0xFFFFFFFFu, dist_up, o));
    if (lane == 0 && tx < T.tiles_x && ty < T.tiles_y)
        atomicMax((int*)&T.hiz_next[ty * T.tiles_x + tx], __float_as_int(dist_up));
}

int tiles_status(cudaError_t e) { return aokk_status(e); }

}  // namespace

extern "C" {

int aokk_tiles_frame(const SceneDev* S, const CamDev* C, const ChunkRef* frame, const TileDev* T, uint4* hit, float* t,
                     int sms, void* stream, const BeamRead* beam) {
    const cudaStream_t s = (cudaStream_t)stream;
    const int nch = S->grid[0] * S->grid[1] * S->grid[2];
    const int tiles = T->tiles_x * T->tiles_y;
    static int per_sm[2] = {0, 0};
    if (!per_sm[0]) {
        int a = 0, b = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, tc_cast_kernel<1, true>, 128, 0);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, tc_cast_kernel<2, true>, 128, 0);
        per_sm[1] = b > 0 ? b : 1;
        per_sm[0] = a > 0 ? a : 1;
    }
    const BeamLookup bl = beam_lookup(beam && beam->bounds ? beam : nullptr, C->W, C->H);
    cudaError_t e = cudaMemsetAsync(T->hiz_next, 0, (size_t)tiles * sizeof(float), s);
    if (e != cudaSuccess) return AOK_E_CUDA;
    tc_rect_kernel<<<(8 * nch + 127) / 128, 128, 0, s>>>(*S, *C, frame, *T);
    tc_scan_kernel<<<1, 1024, 0, s>>>(nch, *T);
    if (bl.bounds) tc_cast_kernel<1, true><<<sms * per_sm[0], 128, 0, s>>>(*S, *C, frame, *T, bl);
    else tc_cast_kernel<1, false><<<sms * per_sm[0], 128, 0, s>>>(*S, *C, frame, *T, bl);
    tc_hiz_kernel<<<(tiles + 7) / 8, 256, 0, s>>>(*S, *C, *T);
    if (bl.bounds) tc_cast_kernel<2, true><<<sms * per_sm[1], 128, 0, s>>>(*S, *C, frame, *T, bl);
    else tc_cast_kernel<2, false><<<sms * per_sm[1], 128, 0, s>>>(*S, *C, frame, *T, bl);
    tc_resolve_kernel<<<dim3((C->W + 15) / 16, (C->H + 7) / 8), 128, 0, s>>>(*S, *C, frame, *T, hit, t);
    e = cudaMemsetAsync(T->vis, 0xFF, (size_t)C->W * C->H * 8, s);  // re-armed for the next frame
    if (e != cudaSuccess) return AOK_E_CUDA;
    return tiles_status(cudaGetLastError());
}

}  // extern "C"
