// The casting kernels' voxel walk: the march of aok_trace.cuh (chunk grid,
// then each chunk's sparse voxel DAG, Aokana Sec. 3.5) with every ordering
// decision made in FP32 together with a bound on its error.  A decision closer
// than its bound ends the fast walk, and the ray goes on in a second instance
// of the same walk that settles such decisions by exact comparisons, so that
// results stay those of the exact real ray.
//
// Why: the exact march spends two 32 x 32 -> 64-bit products (half-rate
// multiplies) and a 64-bit compare on every comparison of plane crossings, and
// compares again at every level it descends.  Here a crossing is one FMA, the
// nearest of three and its distance from the second one are the minimum and
// the median of three, and a cell's coordinates at all levels are found at once
// when an occupied cell is entered, so that descending costs no comparison.
// Bound: instruction issue (about 70% of it, the ALU pipe 67%) and the
// divergence of neighbour rays (17.5 of 32 lanes; 7 at the entry of a leaf
// block, 9 in its steps).  Frames, the exact march -> this walk (with what the
// march got beside it: bound, warp tiles, beam pass): city 1920x1080 485 -> 271
// us, overview 3840x2160 746 -> 411, open world 2560x1440 885 -> 511, 24 views
// 6301 -> 3263, 256x256 74 -> 38.
//
// Numbers.  The ray is taken in the frame mirrored so that d >= 0.  Its
// parameter t counts from a base point on the ray, known to 2^-24 of a voxel:
// an integer voxel B and a fraction x in [0, 1) per axis.  Plane j (in voxels
// of the chunk's LOD, from the base's voxel) is crossed at
// T = j g - x g, g = 1 / d.  With u = 2^-24: the approximate reciprocal is
// within 2u of 1 / d, x and the product x g within u each, the FMA within u
// of T, so |error of T| <= 3u T + 2u g; up to three steps T += g inside a
// leaf block add u T each.  Two crossings are told apart when they differ by
// more than eps T + 5u g_max, eps = 8u (14u in a leaf block): both errors, and
// the rounding of that sum.  A coordinate x + T d at the entry of a cell, used
// for its integer part, is within (4u T + 4u g_max) d_max (from T: 3u T d +
// 2u g d; from the FMA u T d, from x and x - 1/2 2u, and g_max d_max >= 1) and
// is used when it lies farther than 5u (T + g_max) d_max from every integer.
#pragma once
#include "aok_ptx.cuh"
#include "aok_trace.cuh"

namespace aok {

constexpr float kU = 0x1p-24f;
constexpr float kEpsT = 8.0f * kU, kEpsLeaf = 14.0f * kU, kEpsX = 5.0f * kU, kEpsG = 5.0f * kU;
constexpr float kWalkEps = 14.0f * kU;  // of the walk's start, where T is a product of two rounded factors
constexpr float kZeroInv = 1e35f;       // 1 / d of a zero component: its planes lie past every other crossing
constexpr uint32_t kMagicBits = 0x4B000000u;  // 2^23: kMagicBits | i is the float 2^23 + i for 0 <= i < 2^23
constexpr float kRound = 12582912.0f;   // 1.5 * 2^23: adding it rounds to an integer
// A base point farther back than this (voxels of the ray's largest component)
// is replaced when an occupied cell is entered, which keeps the bounds small:
// near when the cell is of level kNearLevel or below, where the ray is about to
// meet leaf blocks.
constexpr float kRebaseNear = 48.0f, kRebaseFar = 256.0f;
constexpr int kNearLevel = 4;

template <class T>
__device__ __forceinline__ T sel3(int e, T a, T b, T c) {
    return e == 0 ? a : (e == 1 ? b : c);
}

// 2^n, |n| < 127
__device__ __forceinline__ float pow2(int n) { return __int_as_float((127 + n) << 23); }

struct WalkRay {
    float ad[3], inv[3];  // |d|, 1 / |d|
    float gmax, dmax;     // largest 1 / |d| of a moving axis, largest |d|
};

// Where a walk goes on: the chunk cell and the plane (e, Ne) it is entered or
// continued at (e = 3: the origin; e < 0: the walk has not started).
struct WalkAt {
    int32_t cc[3], e, Ne;
};

// The decisions that FP32 leaves open, exactly (trace_chunk's comparisons and
// its rules for ties): Na / |da| < Nb / |db| ...
static __device__ __noinline__ bool exact_less(int32_t Na, float da, int32_t Nb, float db) {
    int32_t ma, Ea, mb, Eb;
    decompose(da, ma, Ea);
    decompose(db, mb, Eb);
    return tlt(Na, ma, Nb, mb, Eb - Ea);
}
// ... and the axis of the nearest of three exit planes, at a tie the higher one.
static __device__ __noinline__ int exact_nearest(int32_t N0, int32_t N1, int32_t N2, float d0, float d1, float d2) {
    const bool xy = exact_less(N0, d0, N1, d1);
    return exact_less(xy ? N0 : N1, xy ? d0 : d1, N2, d2) ? (xy ? 0 : 1) : 2;
}

// Base point of the ray where it crosses plane (e, Ne) (e = 3: the origin):
// voxel B and fraction x per axis of the mirrored world.  The quotient
// Ne / |d_e| is carried as a sum of two floats (residual by FMA), so that the
// point's error is below 2^-12 numerator units at any distance.  False if a
// coordinate lies within 2^-10 units (2^-22 voxels) of a voxel plane; EXACT
// then places it by comparison: a plane crossed no later than the base point
// is passed.
template <bool EXACT>
__device__ __forceinline__ bool walk_base(const WalkRay& w, const int32_t Ow[3], int e, int32_t Ne, int32_t B[3],
                                          float x[3]) {
    float q1 = 0.0f, q2 = 0.0f;
    const float ade = sel3(e, w.ad[0], w.ad[1], w.ad[2]);
    if (e < 3) {
        const float inv = sel3(e, w.inv[0], w.inv[1], w.inv[2]);
        const float Nf = (float)Ne, Nl = (float)(Ne - (int32_t)Nf);
        q1 = Nf * inv;
        q2 = (__fmaf_rn(-q1, ade, Nf) + Nl) * inv;
    }
    bool clear = true;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const float p1 = q1 * w.ad[a];
        const float p2 = __fmaf_rn(q2, w.ad[a], __fmaf_rn(q1, w.ad[a], -p1));
        const int32_t i1 = __float2int_rd(p1);
        float f = (p1 - (float)i1) + p2;
        const int32_t i2 = __float2int_rd(f);
        const bool plane = a == e;
        const int32_t I = (int32_t)((uint32_t)Ow[a] + (uint32_t)(plane ? Ne : i1 + i2));
        f = plane ? 0.0f : f - (float)i2;
        float lo = (float)(I & 4095) + f;
        B[a] = I >> kFix;
        // exact where nothing moved the coordinate off the origin's (e = 3, a zero component) or it is the plane itself
        if (!plane && e < 3 && w.ad[a] > 0.0f && !(fabsf(lo - 2048.0f) < 2048.0f - 0x1p-10f)) {
            clear = false;
            if (EXACT) {
                const int32_t P = lo < 2048.0f ? B[a] : B[a] + 1;
                const int32_t Np = (int32_t)(((uint32_t)P << kFix) - (uint32_t)Ow[a]);
                const int32_t Bn = exact_less(Ne, ade, Np, w.ad[a]) ? P - 1 : P;
                lo += 4096.0f * (float)(B[a] - Bn);
                B[a] = Bn;
            }
        }
        x[a] = lo * (1.0f / 4096.0f);
    }
    return clear;
}

// One chunk's part of a walk, called by all of a warp's lanes together, those
// with `traced` taking part: the traversal of the sparse voxel DAG `root` (LOD
// lod) of chunk cell cc from the ray's base point (based) or its crossing of
// plane (e, Ne).  True: a hit (c, e and idx of `hit`; e its entry axis).
// Otherwise, unless undecided, e is the axis the chunk is left through.
// (eb, Ne) follows the base point.
template <bool EXACT>
__device__ __forceinline__ bool walk_chunk(const SceneDev& S, const WalkRay& w, uint32_t mir, const int32_t (&Ow)[3],
                                           const int32_t (&cc)[3], bool traced, bool based, uint32_t root, int lod,
                                           int& e, int32_t& Ne, int& eb, int32_t (&B)[3], float (&x)[3],
                                           bool& undecided, HitRec& hit) {
    const uint32_t* __restrict__ nodes = S.nodes;
    // Voxel coordinates of the current cell at every level, in voxels
    // of the LOD, axis a shifted left by a: the octant of level k is
    // then bits k, k + 1, k + 2 of the three merged words.
    bool go = traced, occ = false;
    int n = 0, R = 3, k = 2;
    float gtol = 0.0f, dmaxn = 0.0f;
    uint32_t V0 = 0, V1 = 0, V2 = 0;
    float Kp[3], gs[3], hp[3], xm[3], dv[3];
    // {node, child mask | its place among its parent's children << 8}
    // of the path's interior levels R .. 3; an
    // EXACT walk keeps to the octree inside leaf blocks too (at a tie
    // the cells visited depend on it) and holds level 2 as well
    constexpr int kLow = EXACT ? 2 : 3;
    uint2 st[kMaxLevels - kLow];
    uint32_t pidx = 0, pm8 = 0, o = 0;
    uint64_t lmu = 0;
    // numerator of the plane at scaled coordinate P of axis a
    auto plane = [&](int a, uint32_t P) -> int32_t {
        return (((sel3(a, cc[0], cc[1], cc[2]) << S.mlog) + (int32_t)((P >> a) << n)) << kFix) -
               sel3(a, Ow[0], Ow[1], Ow[2]);
    };
    // crossing parameters and coordinates from the base point, the
    // latter kept within the cell of coordinates V with bits `low` free
    auto rebase = [&](uint32_t low) {
        const float up = pow2(n), down = pow2(-n);
        uint32_t J[3] = {V0, V1 >> 1, V2 >> 2};
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const int32_t l = B[a] - (cc[a] << S.mlog);
            // (a decided base point lies in the cell: only EXACT can meet its upper face, at a tie)
            J[a] = EXACT ? (uint32_t)max((int32_t)(J[a] & ~low), min(l >> n, (int32_t)(J[a] | low)))
                         : (J[a] & ~low) | ((uint32_t)(l >> n) & low);
            const int32_t below = EXACT ? l - (int32_t)(J[a] << n) : l & ((1 << n) - 1);
            const float xn = ((float)below + x[a]) * down;
            const float g = w.inv[a] * up;
            gs[a] = g * (1.0f / (float)(1 << a));
            hp[a] = __fmaf_rn(-xn, g, gs[a]);
            xm[a] = xn - 0.5f;
            dv[a] = w.ad[a] * down;
            Kp[a] = __uint_as_float(kMagicBits | (J[a] << a));
        }
        V0 = J[0];
        V1 = J[1] << 1;
        V2 = J[2] << 2;
    };
    // octant of the level-k cell in its parent, stored order: bits k,
    // k + 1, k + 2 of the three words merged (m = ~0 << k)
    uint32_t m = ~0u;
    auto octant = [&]() -> uint32_t {
        const uint32_t hi = (V2 & (m << 2)) | (V1 & ~(m << 2));
        return ((((hi & (m << 1)) | (V0 & ~(m << 1))) >> k) & 7u) ^ mir;
    };
    if (traced) {
        n = lod;
        R = S.mlog - n;
        gtol = kEpsG * w.gmax * pow2(n);
        dmaxn = w.dmax * pow2(-n);
        pidx = root;
        pm8 = nodes[pidx] & 0xFFu;
        if (!based) undecided = !walk_base<EXACT>(w, Ow, e, Ne, B, x) && !EXACT;
        eb = e;
        rebase((1u << R) - 1u);
        st[R - kLow] = make_uint2(pidx, pm8);
        k = R - 1;
        m = ~0u << k;
        o = octant();
        occ = (pm8 >> o) & 1u;
    }
    while (go) {
        while (occ && k > (EXACT ? 0 : 2)) {
            // into the occupied cell: its node and child mask
            if (EXACT && k == 1) {
                // the voxel bits of a leaf block's 2x2x2 group
                const uint64_t v = lmu >> ((o & 1u) * 2 + (o & 2u) * 4 + (o & 4u) * 8);
                pm8 = (uint32_t)((v & 3) | ((v >> 2) & 0xC) | ((v >> 12) & 0x30) | ((v >> 14) & 0xC0));
            } else {
                const uint32_t rank = __popc(pm8 & ~(~0u << o));
                const uint2 ch = __ldg(reinterpret_cast<const uint2*>(nodes + pidx + 2 + 2 * rank));
                pidx = ch.x;
                pm8 = ch.y >> 24;
                if (k == kWideLevel - 1) pm8 = nodes[pidx] & 0xFFu;
                if (EXACT && k == 2) {
                    lmu = __ldg(S.leaves + pidx);
                    uint64_t q = lmu | (lmu >> 1);
                    q |= q >> 4;
                    q |= q >> 16;  // the occupied groups
                    pm8 = (uint32_t)((q & 1) | ((q >> 1) & 2) | ((q >> 6) & 4) | ((q >> 7) & 8) |
                                     ((q >> 28) & 16) | ((q >> 29) & 32) | ((q >> 34) & 64) | ((q >> 35) & 128));
                }
                st[k - kLow] = make_uint2(pidx, pm8 | rank << 8);
            }
            k--;
            m = ~0u << k;
            o = octant();
            occ = (pm8 >> o) & 1u;
        }
        float tm = 0.0f;
        if (EXACT) {
            go = !occ;  // occupied at level 0: the hit
        } else if (occ) {
            // a 4^3 leaf block: voxel by voxel, to a set bit or out of
            // it; i: bit of the voxel in the mirrored frame
            lmu = __ldg(S.leaves + __ldg(nodes + pidx + 2 + 2 * __popc(pm8 & ~(~0u << o))));
            float T0 = __fmaf_rn(__uint_as_float(V0 | kMagicBits) - Kp[0], gs[0], hp[0]);
            float T1 = __fmaf_rn(__uint_as_float(V1 | 1u | kMagicBits) - Kp[1], gs[1], hp[1]);
            float T2 = __fmaf_rn(__uint_as_float(V2 | 3u | kMagicBits) - Kp[2], gs[2], hp[2]);
            uint32_t i = (V0 & 3u) | ((V1 & 6u) << 1) | ((V2 & 12u) << 2), inc = 0;
            const uint32_t mi = ((mir & 1u) | ((mir & 2u) << 1) | ((mir & 4u) << 2)) * 3u;
            for (;;) {
                const uint32_t j = i ^ mi;
                occ = (lmu >> j) & 1u;
                if (occ) break;
                // (decided when the second smallest, the median, lies past
                // thr; against three compares with thr and their logic, here
                // and below, 315 / 232 / 290 -> 307 / 229 / 282 us)
                const float lo01 = fminf(T0, T1), hi01 = fmaxf(T0, T1);
                tm = fminf(lo01, T2);
                const float thr = __fmaf_rn(tm, 1.0f + kEpsLeaf, gtol);
                undecided = undecided || !(fminf(hi01, fmaxf(lo01, T2)) > thr);
                const bool p2 = T2 < lo01, p0 = !p2 && T0 < T1, p1 = !p2 && !p0;
                if (p0) { T0 = T0 + gs[0]; inc = 1u; }
                else if (p1) { T1 = __fmaf_rn(gs[1], 2.0f, T1); inc = 4u; }
                else { T2 = __fmaf_rn(gs[2], 4.0f, T2); inc = 16u; }
                i += inc;
                if (!(i & (3u * inc))) break;  // left the block
            }
            if (occ) {
                if (inc) e = inc == 1u ? 0 : (inc == 4u ? 1 : 2);
                V0 = (V0 & ~3u) | (i & 3u);
                V1 = (V1 & ~6u) | ((i >> 1) & 6u);
                V2 = (V2 & ~12u) | ((i >> 2) & 12u);
                go = false;  // the hit
            }
        }
        // leave empty cells through their nearest exit face until an
        // occupied one or the chunk's end
        uint32_t m0 = m;
        while (!occ) {
            const uint32_t E0 = V0 | ~m | kMagicBits, E1 = V1 | ~(m << 1) | kMagicBits,
                           E2 = V2 | ~(m << 2) | kMagicBits;
            const float T0 = __fmaf_rn(__uint_as_float(E0) - Kp[0], gs[0], hp[0]);
            const float T1 = __fmaf_rn(__uint_as_float(E1) - Kp[1], gs[1], hp[1]);
            const float T2 = __fmaf_rn(__uint_as_float(E2) - Kp[2], gs[2], hp[2]);
            const float lo01 = fminf(T0, T1), hi01 = fmaxf(T0, T1);
            tm = fminf(lo01, T2);
            const float thr = __fmaf_rn(tm, 1.0f + kEpsT, gtol);
            const bool p2 = T2 < lo01;
            bool p0 = !p2 && T0 < T1, p1 = !p2 && !p0;
            const bool amb = !(fminf(hi01, fmaxf(lo01, T2)) > thr);
            if (EXACT) {
                if (amb) {
                    const int a = exact_nearest(plane(0, E0 + (1u - kMagicBits)), plane(1, E1 + (1u - kMagicBits)),
                                                plane(2, E2 + (1u - kMagicBits)), w.ad[0], w.ad[1], w.ad[2]);
                    p0 = a == 0;
                    p1 = a == 1;
                    tm = sel3(a, T0, T1, T2);
                }
            } else {
                undecided = undecided || amb;
            }
            e = p0 ? 0 : (p1 ? 1 : 2);
            const uint32_t nv = (p0 ? E0 : (p1 ? E1 : E2)) + (1u - kMagicBits);
            V0 = p0 ? nv : V0;
            V1 = p1 ? nv : V1;
            V2 = p0 || p1 ? V2 : nv;
            m0 = m;
            // the level of the cell entered: k for a sibling, else
            // that of the lowest set bit (the parent was left)
            const int K = __ffs((int)nv) - 1 - e;
            if (K >= R) { go = false; break; }  // left the chunk
            if (K != k) {
                const uint2 par = st[K + 1 - kLow];
                pidx = par.x;
                pm8 = par.y;
            }
            k = K;
            m = ~0u << k;
            o = octant();
            occ = (pm8 >> o) & 1u;
        }
        if (go) {
            // the entered cell's coordinates below the level it was
            // left at (the crossed axis' are zero: it is on a face);
            // at a tie, below the level it was entered at
            if (EXACT) m0 = m;
            const float lim = 0.5f - __fmaf_rn(tm, kEpsX, gtol) * dmaxn;
            const float x0 = __fmaf_rn(tm, dv[0], xm[0]), x1 = __fmaf_rn(tm, dv[1], xm[1]),
                        x2 = __fmaf_rn(tm, dv[2], xm[2]);
            const float r0 = (x0 + kRound) - kRound, r1 = (x1 + kRound) - kRound, r2 = (x2 + kRound) - kRound;
            const float f0 = e == 0 ? 0.0f : x0 - r0, f1 = e == 1 ? 0.0f : x1 - r1, f2 = e == 2 ? 0.0f : x2 - r2;
            const bool clear = fmaxf(fmaxf(fabsf(f0), fabsf(f1)), fabsf(f2)) < lim;
            if (tm * w.dmax > (k > kNearLevel ? kRebaseFar : kRebaseNear) || !clear) {
                // far from the base point, or next to a voxel plane: a new base here
                const int32_t Nt = plane(e, sel3(e, V0, V1, V2));
                if (!undecided) { eb = e; Ne = Nt; }
                undecided = (!walk_base<EXACT>(w, Ow, e, Nt, B, x) && !EXACT) || undecided;
                rebase(~m0);
            } else {
                const uint32_t k0 = e == 0 ? ~0u : m0, k1 = e == 1 ? ~0u : m0 << 1, k2 = e == 2 ? ~0u : m0 << 2;
                V0 = (V0 & k0) | (__float_as_uint(r0 + Kp[0]) & ~k0);
                V1 = (V1 & k1) | (__float_as_uint(__fmaf_rn(r1, 2.0f, Kp[1])) & ~k1);
                V2 = (V2 & k2) | (__float_as_uint(__fmaf_rn(r2, 4.0f, Kp[2])) & ~k2);
            }
        }
    }
    if ((!EXACT && undecided) || !traced || !occ) return false;
    hit.c[0] = (int32_t)V0;
    hit.c[1] = (int32_t)(V1 >> 1);
    hit.c[2] = (int32_t)(V2 >> 2);
    hit.e = e;
    // depth-first index (Sec. 3.3): the prefix beside each child
    // pointer of the path, then the leaf block's earlier voxels
    uint32_t idx;
    if (EXACT) {
        idx = nodes[st[1].x + 3 + 2 * (st[0].y >> 8)];
    } else {
        idx = nodes[pidx + 3 + 2 * __popc(pm8 & ~(~0u << o))];
    }
    idx &= kPrefixBits;
    for (int j = R; j > 3; j--)
        idx += nodes[st[j - kLow].x + 3 + 2 * (st[j - 1 - kLow].y >> 8)] & (j == kWideLevel ? ~0u : kPrefixBits);
    const uint32_t bit = ((V0 & 3u) | ((V1 & 6u) << 1) | ((V2 & 12u) << 2)) ^
                         (((mir & 1u) | ((mir & 2u) << 1) | ((mir & 4u) << 2)) * 3u);
    hit.idx = idx + (uint32_t)__popcll(lmu & ((1ull << bit) - 1ull));
    return true;
}

// Cast the pixel's ray and write its record.  BEAM: restart past the beam
// pass's bound Dn (0: none).  lanes: the warp's lanes that call it.  False
// (never with EXACT; nothing written): undecided at `at`, where an EXACT walk
// takes over.  The loops have one way out each, and the outer one is left by
// all lanes together: a return from inside them cost the warp its convergence
// (7 active lanes instead of 19, 2.5 times the time).
template <bool EXACT, bool BEAM>
__device__ __forceinline__ bool walk_pixel(const SceneDev& S, const CamDev& C, const ChunkRef* __restrict__ frame,
                                           int px, int py, uint4* __restrict__ out_hit, float* __restrict__ out_t,
                                           size_t pix, int32_t Dn, uint32_t lanes, WalkAt& at) {
    float d[3];
    ray_dir(C, px, py, d);
    const uint32_t mir = (d[0] < 0.0f ? 1u : 0u) | (d[1] < 0.0f ? 2u : 0u) | (d[2] < 0.0f ? 4u : 0u);
    bool undecided = false, miss = false, odd = false;
    // Only ratios of the components matter to the walk: EXACT brings an
    // unusual scale to a normal one, the fast walk leaves such a ray to it.
    WalkRay w;
    w.dmax = fmaxf(fmaxf(fabsf(d[0]), fabsf(d[1])), fabsf(d[2]));
    float scale = 1.0f;
    if (EXACT) {
        if (!(w.dmax > 0x1p-40f)) scale = 0x1p100f;
        if (w.dmax > 0x1p40f) scale = 0x1p-88f;
        w.dmax *= scale;
    } else {
        odd = !(w.dmax > 0x1p-40f && w.dmax < 0x1p40f);
    }
    w.gmax = 0.0f;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        w.ad[a] = EXACT ? fabsf(d[a]) * scale : fabsf(d[a]);
        w.inv[a] = w.ad[a] > 0.0f ? rcp_approx(w.ad[a]) : kZeroInv;
        if (w.ad[a] > 0.0f) w.gmax = fmaxf(w.gmax, w.inv[a]);
    }
    const int cs = S.mlog + kFix;
    int32_t Ow[3], Wfix[3];
    bool inside = true;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        Wfix[a] = S.grid[a] << cs;
        Ow[a] = ((mir >> a) & 1u) ? Wfix[a] - C.O[a] : C.O[a];
        inside = inside && Ow[a] >= 0 && Ow[a] < Wfix[a];
    }
    int e = 3;
    int32_t Ne = 0;
    const bool resumed = EXACT && at.e >= 0;
    if (resumed) {
        e = at.e;
        Ne = at.Ne;
    } else if (!inside) {
        // enter the world box: latest entry plane against the earliest exit plane
        float tin = -1.0f, tin2 = -1.0f, tout = 3.0e38f;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            if (Ow[a] >= Wfix[a] || (w.ad[a] == 0.0f && Ow[a] < 0)) miss = true;
            const float ti = Ow[a] < 0 ? (float)(-Ow[a]) * w.inv[a] : -1.0f;
            tout = fminf(tout, (float)(Wfix[a] - Ow[a]) * w.inv[a]);
            if (ti > tin) { tin2 = tin; tin = ti; e = a; }
            else tin2 = fmaxf(tin2, ti);
        }
        if (tin > tout * (1.0f + kWalkEps)) {
            miss = true;
        } else if (!miss && !(tin < tout * (1.0f - kWalkEps) && tin2 < tin * (1.0f - kWalkEps))) {
            undecided = true;
            if (EXACT) {
                e = -1;
                int ex = 0;
                for (int a = 0; a < 3; a++) {
                    const int32_t O = sel3(a, Ow[0], Ow[1], Ow[2]);
                    const float da = sel3(a, w.ad[0], w.ad[1], w.ad[2]);
                    if (O < 0 && (e < 0 || exact_less(-sel3(e, Ow[0], Ow[1], Ow[2]), sel3(e, w.ad[0], w.ad[1], w.ad[2]), -O, da)))
                        e = a;
                    if (a > 0 && exact_less(sel3(a, Wfix[0], Wfix[1], Wfix[2]) - O, da,
                                            sel3(ex, Wfix[0], Wfix[1], Wfix[2]) - sel3(ex, Ow[0], Ow[1], Ow[2]),
                                            sel3(ex, w.ad[0], w.ad[1], w.ad[2])))
                        ex = a;
                }
                miss = !exact_less(-sel3(e, Ow[0], Ow[1], Ow[2]), sel3(e, w.ad[0], w.ad[1], w.ad[2]),
                                   sel3(ex, Wfix[0], Wfix[1], Wfix[2]) - sel3(ex, Ow[0], Ow[1], Ow[2]),
                                   sel3(ex, w.ad[0], w.ad[1], w.ad[2]));
            }
        }
        Ne = -sel3(e, Ow[0], Ow[1], Ow[2]);
    }
    bool restarted = false;
    if (BEAM && Dn > 0 && !miss && !resumed) {
        // the beam restart of trace_pixel_t (from the box, if that order is undecided)
        int as = 0;
        if (w.ad[1] > w.ad[0]) as = 1;
        if (w.ad[2] > fmaxf(w.ad[0], w.ad[1])) as = 2;
        const int32_t O = sel3(as, Ow[0], Ow[1], Ow[2]);
        const int32_t Nl = (int32_t)(((uint32_t)(Dn - 1) + (uint32_t)O) & ~4095u) - O;
        if (Dn == INT_MAX || Nl >= (sel3(as, S.grid[0], S.grid[1], S.grid[2]) << cs) - O) {
            miss = true;  // nothing solid for this ray
        } else if (Nl > 0 && (e == 3 || (float)Nl * sel3(as, w.inv[0], w.inv[1], w.inv[2]) >
                                            (float)Ne * sel3(e, w.inv[0], w.inv[1], w.inv[2]) * (1.0f + kWalkEps))) {
            e = as;
            Ne = Nl;
            restarted = true;
        }
    }
    int eb = -1;  // base point's plane is (eb, Ne); < 0: the walk has not started
    int32_t B[3], cc[3];
    float x[3];
    const bool clear = walk_base<EXACT>(w, Ow, e, Ne, B, x);
    bool outside = false;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        cc[a] = resumed ? at.cc[a] : B[a] >> S.mlog;
        outside = outside || (uint32_t)cc[a] >= (uint32_t)S.grid[a];
        if (EXACT) cc[a] = max(0, min(cc[a], S.grid[a] - 1));  // (entered through an edge of the box)
    }
    if (restarted && outside && (EXACT || clear)) miss = true;  // left the world box before the restart point
    undecided = !EXACT && (odd || (!miss && (undecided || outside || !clear)));
    bool alive = !miss && !undecided, found = false;
    HitRec hit;
    // the current chunk cell's entry of the frame table
    auto chunk_entry = [&](int32_t u[3]) -> const uint4* {
#pragma unroll
        for (int a = 0; a < 3; a++) u[a] = ((mir >> a) & 1u) ? S.grid[a] - 1 - cc[a] : cc[a];
        return reinterpret_cast<const uint4*>(
            frame + ((uint32_t)u[0] + (uint32_t)S.grid[0] * ((uint32_t)u[1] + (uint32_t)S.grid[1] * (uint32_t)u[2])));
    };
    bool based = true;  // the base point lies on the entry of the current chunk
    while (EXACT ? alive : __any_sync(lanes, alive)) {
        bool traced = false;
        uint32_t root = kNone, lod = 0;
        if (alive) {
            int32_t u[3];
            const uint4* fr = chunk_entry(u);
            const uint4 ra = __ldg(fr), rb = __ldg(fr + 1);
            root = ra.x;
            lod = ra.y;
            if (S.view_dist > 0.0f && e < 3) {
                const float dn = sqrtf(w.ad[0] * w.ad[0] + w.ad[1] * w.ad[1] + w.ad[2] * w.ad[2]);
                const float tent = (float)Ne * (1.0f / 4096.0f) * sel3(e, w.inv[0], w.inv[1], w.inv[2]);
                if (tent * dn > S.view_dist * 1.00001f + 1.0f) alive = false;
            }
            if (BEAM && restarted) {
                traced = alive && root != kNone;  // restarted in this chunk, next to solid voxels: no use asking
            } else if (alive && root != kNone) {
                // skip chunks whose solid-voxel AABB (grown by 1/16 voxel) the ray misses
                const int32_t M = 1 << S.mlog;
                const int32_t lo[3] = {(int32_t)(rb.x & 0xFFFFu), (int32_t)(rb.x >> 16), (int32_t)(rb.y & 0xFFFFu)};
                const int32_t hi[3] = {(int32_t)(rb.y >> 16), (int32_t)(rb.z & 0xFFFFu), (int32_t)(rb.z >> 16)};
                float tn = 0.0f, tf = 3.0e38f;
#pragma unroll
                for (int a = 0; a < 3; a++) {
                    const bool m = (mir >> a) & 1u;
                    const int32_t off = (cc[a] << S.mlog) - B[a];
                    tn = fmaxf(tn, ((float)(off + (m ? M - hi[a] : lo[a])) - (x[a] + 0.0625f)) * w.inv[a]);
                    tf = fminf(tf, ((float)(off + (m ? M - lo[a] : hi[a])) - (x[a] - 0.0625f)) * w.inv[a]);
                }
                traced = tn <= tf;
            }
        }
        if (EXACT ? traced : __any_sync(lanes, traced)) {
            found = walk_chunk<EXACT>(S, w, mir, Ow, cc, traced, based, root, (int)lod, e, Ne, eb, B, x, undecided, hit) ||
                    found;
            if (found || (!EXACT && undecided)) alive = false;
        }
        if (alive && !traced) {
            // over this chunk cell: its nearest exit face
            float T[3];
#pragma unroll
            for (int a = 0; a < 3; a++)
                T[a] = __fmaf_rn((float)(((cc[a] + 1) << S.mlog) - B[a]), w.inv[a], -x[a] * w.inv[a]);
            const float thr = __fmaf_rn(fminf(fminf(T[0], T[1]), T[2]), 1.0f + kEpsT, kEpsG * w.gmax);
            const bool p0 = T[0] <= thr, p1 = T[1] <= thr, p2 = T[2] <= thr;
            const int en = p0 ? 0 : (p1 ? 1 : 2);
            if (p0 ? p1 || p2 : p1 == p2) {
                if (EXACT) {
                    e = exact_nearest(((cc[0] + 1) << cs) - Ow[0], ((cc[1] + 1) << cs) - Ow[1],
                                      ((cc[2] + 1) << cs) - Ow[2], w.ad[0], w.ad[1], w.ad[2]);
                } else {
                    eb = e;
                    undecided = true;
                    alive = false;
                }
            } else {
                e = en;
            }
        }
        if (alive) {
            based = false;
            restarted = false;
            cc[0] += e == 0;
            cc[1] += e == 1;
            cc[2] += e == 2;
            const int32_t ce = sel3(e, cc[0], cc[1], cc[2]);
            if (ce >= sel3(e, S.grid[0], S.grid[1], S.grid[2])) alive = false;
            Ne = (ce << cs) - sel3(e, Ow[0], Ow[1], Ow[2]);
        }
    }
    if (!EXACT && undecided) {
#pragma unroll
        for (int a = 0; a < 3; a++) at.cc[a] = cc[a];
        at.e = eb;
        at.Ne = Ne;
        return false;
    }
    if (found) {
        int32_t u[3];
        const uint4* fr = chunk_entry(u);
        const uint4 ra = __ldg(fr);
        const int n = (int)ra.y;
        hit.Ne = 0;
        if (e < 3)  // the voxel's face that the ray enters through
            hit.Ne = (((sel3(e, cc[0], cc[1], cc[2]) << S.mlog) + (sel3(e, hit.c[0], hit.c[1], hit.c[2]) << n)) << kFix) -
                     sel3(e, Ow[0], Ow[1], Ow[2]);
        if (EXACT && (e == 1 || e == 2)) {
            // entered through an edge or a corner: the lowest of its axes (lowest_entry_face)
            const int32_t Nh = hit.Ne;
            const float de = sel3(e, w.ad[0], w.ad[1], w.ad[2]);
            for (int b = e - 1; b >= 0; b--) {
                const float db = b ? w.ad[1] : w.ad[0];
                const int32_t Nb = ((((b ? cc[1] : cc[0]) << S.mlog) + ((b ? hit.c[1] : hit.c[0]) << n)) << kFix) -
                                   (b ? Ow[1] : Ow[0]);
                if (db > 0.0f && !exact_less(Nh, de, Nb, db) && !exact_less(Nb, db, Nh, de)) {
                    hit.e = b;
                    hit.Ne = Nb;
                }
            }
        }
        ChunkRef ref;
        ref.lod = ra.y;
        ref.mat_base = (uint64_t)ra.z | (uint64_t)ra.w << 32;
        ref.nblocks = __ldg(fr + 1).w;
        RayState r;
#pragma unroll
        for (int a = 0; a < 3; a++) r.d[a] = EXACT ? d[a] : w.ad[a];  // (their signs do not matter)
        r.mir = mir;
        found = emit_hit(S, r, ref, u, hit, ray_norm(r), out_hit, out_t, pix);
    }
    if (!found) emit_miss(out_hit, out_t, pix);
    return true;
}

// The rest of an undecided ray.  Out of line: about one ray in three thousand
// needs it, and inside the walk its comparisons cost every ray registers.
template <bool BEAM>
__device__ __noinline__ void walk_rest(const SceneDev& S, const CamDev& C, const ChunkRef* __restrict__ frame, int px,
                                       int py, uint4* __restrict__ out_hit, float* __restrict__ out_t, size_t pix,
                                       int32_t Dn, WalkAt at) {
    walk_pixel<true, BEAM>(S, C, frame, px, py, out_hit, out_t, pix, Dn, 0u, at);
}

template <bool BEAM>
__device__ __forceinline__ void cast_pixel(const SceneDev& S, const CamDev& C, const ChunkRef* __restrict__ frame,
                                           int px, int py, uint4* __restrict__ out_hit, float* __restrict__ out_t,
                                           size_t pix, int32_t Dn, uint32_t lanes) {
    WalkAt at;
    if (!walk_pixel<false, BEAM>(S, C, frame, px, py, out_hit, out_t, pix, Dn, lanes, at))
        walk_rest<BEAM>(S, C, frame, px, py, out_hit, out_t, pix, Dn, at);
}

}  // namespace aok
