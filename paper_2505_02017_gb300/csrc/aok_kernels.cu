// CUDA kernels (sm_103a): per-frame chunk LOD selection and visibility, and
// per-pixel primary-ray first-hit casting through the chunk grid and the
// selected sparse voxel DAGs (Aokana Sec. 3.4-3.5).  The exact traversal
// itself is in aok_trace.cuh.
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <climits>
#include <cstring>
#include <mutex>
#include <vector>

#include "aok_internal.h"
#include "aok_select.cuh"
#include "aok_trace.cuh"
#include "aok_walk.cuh"

using namespace aok;

namespace {

constexpr int kMaxDevices = 128;

// Programmatic dependent launch: the selection lets the cast after it on its
// stream be launched at once; the cast waits for it before anything else.
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_prerequisites() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__global__ void select_kernel(SceneDev S, CamDev C, ChunkRef* __restrict__ frame, int8_t* __restrict__ lod_out,
                              uint8_t* __restrict__ vis_out, uint32_t* __restrict__ n_visible) {
    const int nch = S.grid[0] * S.grid[1] * S.grid[2];
    const int chunk = blockIdx.x * blockDim.x + threadIdx.x;
    launch_dependents();
    if (chunk < nch) select_one(S, C, frame, lod_out, vis_out, n_visible, chunk);
}

// one launch for all views of a batch: blockIdx.y = view
__global__ void select_batch_kernel(const __grid_constant__ BatchParams P) {
    const ViewDev& v = P.v[blockIdx.y];
    const int nch = v.scene.grid[0] * v.scene.grid[1] * v.scene.grid[2];
    const int chunk = blockIdx.x * blockDim.x + threadIdx.x;
    if (chunk < nch) select_one(v.scene, v.cam, v.frame, nullptr, nullptr, nullptr, chunk);
}

// beam_bound (aok_trace.cuh) with the pyramid's level table; 0 (no restart)
// without bounds (a pass that found no usable projection for the view)
__device__ __forceinline__ int32_t beam_bound_lut(const BeamLookup& b, int px, int py) {
    if (!b.bounds) return 0;
    const uint32_t x = (uint32_t)px / kBeamTileW, y = (uint32_t)py / kBeamTileH;
    unsigned long long v = ~0ull;
#pragma unroll
    for (int L = 0; L < kBeamPyr; L++) v = min(v, __ldcg(b.bounds + b.off[L] + (y >> L) * b.wl[L] + (x >> L)));
    return (uint32_t)(v >> 32) == b.tag ? (int32_t)(uint32_t)v : INT_MAX;
}

// The same bound for the 8 x 4 tile whose first pixel is (px, py), called by all
// lanes of its warp: lane L reads level L of the pyramid, and
// the smallest bound of this pass's tag is one warp reduction (seven loads and
// 64-bit minima in every lane before: about 85 of 460 instructions of setup).
__device__ __forceinline__ int32_t beam_bound_warp(const BeamLookup& b, int px, int py, int lane) {
    if (!b.bounds) return 0;
    const int L = min(lane, kBeamPyr - 1);
    const uint32_t x = ((uint32_t)px / kBeamTileW) >> L, y = ((uint32_t)py / kBeamTileH) >> L;
    const unsigned long long v = __ldcg(b.bounds + b.off[L] + y * b.wl[L] + x);
    return (int32_t)__reduce_min_sync(0xFFFFFFFFu, (uint32_t)(v >> 32) == b.tag ? (uint32_t)v : (uint32_t)INT_MAX);
}

// The same for a view of a batch, whose pyramid's level offsets are not at hand.
__device__ __forceinline__ int32_t beam_bound_warp(const unsigned long long* __restrict__ b, uint32_t tag, int W, int H,
                                                   int px, int py, int lane) {
    if (!b) return 0;
    const uint32_t tx = (uint32_t)(W + kBeamTileW - 1) / kBeamTileW, ty = (uint32_t)(H + kBeamTileH - 1) / kBeamTileH;
    const int L = min(lane, kBeamPyr - 1);
    uint32_t off = 0;
#pragma unroll
    for (int l = 0; l < kBeamPyr - 1; l++) {
        const uint32_t n = ((tx + (1u << l) - 1) >> l) * ((ty + (1u << l) - 1) >> l);
        if (l < L) off += n;
    }
    const uint32_t x = ((uint32_t)px / kBeamTileW) >> L, y = ((uint32_t)py / kBeamTileH) >> L;
    const unsigned long long v = __ldcg(b + off + y * ((tx + (1u << L) - 1) >> L) + x);
    return (int32_t)__reduce_min_sync(0xFFFFFFFFu, (uint32_t)(v >> 32) == tag ? (uint32_t)v : (uint32_t)INT_MAX);
}

// 16 x 8 pixel tiles, warps of 8 x 4 pixels.  BEAM: the warp's 8 x 4 tile
// bound from the beam pass (aok_beam.cu) restarts its rays' march past the
// space in front of the nearest voxel they can meet.  At most 64 registers:
// 8 blocks per SM (over nine views of three scenes 7 blocks take 1.4% longer on
// average, 9 and 10 gain up to 2% on the overview and lose up to 5% in the open
// world).  A warp takes 12 to 20 us on average and up to 140, so a frame ends with few
// warps left; no other order of the rows or size of the blocks was shorter on
// all views.
//
// Without bounds a warp may take a smaller tile, wl and hl its sides' logs (3
// and 2: 8 x 4), in its first lanes: see cast_tile.
template <bool COUNT, bool BEAM = false>
__global__ void __launch_bounds__(128, 8) cast_kernel(const __grid_constant__ SceneDev S,
                                                   const __grid_constant__ CamDev C,
                                                   const ChunkRef* __restrict__ frame,
                                                   uint4* __restrict__ out_hit, float* __restrict__ out_t,
                                                   uint32_t* __restrict__ counts,
                                                   const __grid_constant__ BeamLookup beam, int wl, int hl) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (BEAM) { wl = 3; hl = 2; }
    const int wx = (blockIdx.x * 2 + (warp & 1)) << wl, wy = (blockIdx.y * 2 + (warp >> 1)) << hl;  // the warp's tile
    const int px = wx + (lane & ((1 << wl) - 1)), py = wy + (lane >> wl);
    const bool in = px < C.W && py < C.H && lane < 1 << (wl + hl);
    const uint32_t lanes = __ballot_sync(0xFFFFFFFFu, in);
    if (!lanes) return;
    if (!BEAM) wait_prerequisites();
    const int32_t Dn = BEAM ? beam_bound_warp(beam, wx, wy, lane) : 0;
    if (!in) return;
    const size_t pix = (size_t)py * C.W + px;
    // Nothing solid in the tile's view: the miss is written without setting the
    // ray up (overview 3840x2160 470 / 487 / 467 -> 418 / 439 / 418 us, walk
    // views 1920x1080 318 / 239 / 290 -> 316 / 236 / 290).
    if (BEAM && !COUNT && Dn == INT_MAX) {
        emit_miss(out_hit, out_t, pix);
        return;
    }
    if (COUNT) trace_pixel<true, false, BEAM>(S, C, frame, px, py, out_hit, out_t, counts, pix, nullptr, Dn);
    else cast_pixel<BEAM>(S, C, frame, px, py, out_hit, out_t, pix, Dn, lanes);
}

// Warp tile of a frame cast without bounds.  A frame of fewer pixels than the
// GPU holds threads ends when its slowest warp does, and a warp takes as long
// as the paths of all its rays together, step by step: with fewer rays a warp
// there are as many chains, each shorter, on schedulers that idle otherwise.
// So the smallest tile whose warps still fit one resident wave (8 blocks of 4
// warps per SM; 4,864 warps on 152 SMs): 16 rays up to 77,824 pixels, 8 up to
// 38,912, and so on to one.  Four city views each, 8 x 4 tiles -> this rule:
// 320x180 77 -> 70 us on average, 160x90 90 -> 61, 96x54 90 -> 47; past one wave
// it turns (480x270 with 16 rays a warp: two views 8% longer, two 9% shorter).
static void cast_tile(const CamDev& c, int& wl, int& hl) {
    static std::atomic<int> sms[kMaxDevices];
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = 0;
    n = sms[dev].load(std::memory_order_relaxed);
    if (!n) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 1;
        sms[dev].store(n, std::memory_order_relaxed);
    }
    wl = 3;
    hl = 2;
    const int64_t px = (int64_t)c.W * c.H, warps = (int64_t)n * 32;
    while (wl + hl > 0 && px <= warps << (wl + hl - 1)) {
        if (wl > hl) wl--;
        else hl--;
    }
}

// The same casting with every pool index checked (CheckDev); BEAM: with the
// beam pass's bounds.
template <bool BEAM>
__global__ void __launch_bounds__(128) cast_kernel_checked(SceneDev S, CamDev C, const ChunkRef* __restrict__ frame,
                                                           uint4* __restrict__ out_hit, float* __restrict__ out_t,
                                                           CheckDev ck, const BeamLookup beam) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int px = blockIdx.x * 16 + (warp & 1) * 8 + (lane & 7);
    const int py = blockIdx.y * 8 + (warp >> 1) * 4 + (lane >> 3);
    if (px >= C.W || py >= C.H) return;
    const int32_t Dn = BEAM ? beam_bound_lut(beam, px, py) : 0;
    trace_pixel<false, true, BEAM>(S, C, frame, px, py, out_hit, out_t, nullptr, (size_t)py * C.W + px, &ck, Dn);
}

// Persistent casting over a list of views (P.queue[0] = next tile, P.queue[1]
// = finished CTAs; both zero at launch).  Each warp pulls `per_fetch`
// consecutive warp tiles (2^tile_w_log x 32/2^tile_w_log pixels of one view)
// from a global counter until every tile of every view is done.
// P.v[v].tile_begin is the exclusive prefix sum of the views' tile counts.
__global__ void __launch_bounds__(256) cast_persistent(const __grid_constant__ BatchParams P) {
    const int lane = threadIdx.x & 31;
    const int tw = 1 << P.tile_w_log, th = 32 >> P.tile_w_log;
    uint32_t cur = 0;
    uint64_t vbeg = 0, vend = 0;
    int tiles_x = 1;
    for (;;) {
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(P.queue, (unsigned long long)P.per_fetch);
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
        if (base >= P.total_tiles) break;
        const uint64_t stop = min((uint64_t)base + P.per_fetch, P.total_tiles);
        for (uint64_t tile = base; tile < stop; tile++) {
            if (tile < vbeg || tile >= vend) {
                uint32_t lo = 0, hi = P.n_views - 1;  // last view with tile_begin <= tile
                while (lo < hi) {
                    const uint32_t mid = (lo + hi + 1) >> 1;
                    if (P.v[mid].tile_begin <= tile) lo = mid;
                    else hi = mid - 1;
                }
                cur = lo;
                vbeg = P.v[cur].tile_begin;
                vend = cur + 1 < P.n_views ? P.v[cur + 1].tile_begin : P.total_tiles;
                tiles_x = (P.v[cur].cam.W + tw - 1) >> P.tile_w_log;
            }
            const ViewDev& v = P.v[cur];
            const int32_t local = (int32_t)(tile - vbeg);
            const int px = (local % tiles_x) * tw + (lane & (tw - 1));
            const int py = (local / tiles_x) * th + (lane >> P.tile_w_log);
            const uint32_t lanes = __ballot_sync(0xFFFFFFFFu, px < v.cam.W && py < v.cam.H);
            if (px < v.cam.W && py < v.cam.H)
                cast_pixel<false>(v.scene, v.cam, v.frame, px, py, v.hit, v.t, (size_t)py * v.cam.W + px, 0, lanes);
        }
    }
    // the last CTA to finish re-arms the counters for the next launch
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&P.queue[1], 1ull) == (unsigned long long)gridDim.x - 1ull) {
            P.queue[0] = 0ull;
            P.queue[1] = 0ull;
            __threadfence();
        }
    }
}

// One launch over all views of a batch, scheduled by the hardware: block b
// covers block tile b of the concatenated views, a block tile being 2x2 warp
// tiles (2^tile_w_log x 32/2^tile_w_log pixels each); P.v[v].tile_begin is the
// exclusive prefix sum of the views' block-tile counts.  The view index derives
// from blockIdx only, so every per-view parameter load is block-uniform.  9
// blocks per SM (56 registers): 24 views take 1.3% less than with 8, 0.9% less
// than with 10 (one view's kernel gains nothing).
__global__ void __launch_bounds__(128, 9) cast_grid(const __grid_constant__ BatchParams P) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t blk = blockIdx.x;
    uint32_t lo = 0, hi = P.n_views - 1;  // last view with tile_begin <= blk
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (P.v[mid].tile_begin <= blk) lo = mid;
        else hi = mid - 1;
    }
    const ViewDev& v = P.v[lo];
    const int twl = P.tile_w_log, tw = 1 << twl, th = 32 >> twl;
    const int bw = (v.cam.W + 2 * tw - 1) / (2 * tw);
    const int32_t local = (int32_t)(blk - v.tile_begin);
    const int wx = ((local % bw) * 2 + (warp & 1)) * tw, wy = ((local / bw) * 2 + (warp >> 1)) * th;
    const int px = wx + (lane & (tw - 1)), py = wy + (lane >> twl);
    const uint32_t lanes = __ballot_sync(0xFFFFFFFFu, px < v.cam.W && py < v.cam.H);
    if (!lanes) return;
    // with a bound of 0 (no beam pass for this view) the march is the plain one
    const int32_t Dn = twl == 3 ? beam_bound_warp(v.beam, P.beam_tag, v.cam.W, v.cam.H, wx, wy, lane)
                                : beam_bound(v.beam, P.beam_tag, v.cam.W, v.cam.H, min(px, v.cam.W - 1), min(py, v.cam.H - 1));
    if (px >= v.cam.W || py >= v.cam.H) return;
    const size_t pix = (size_t)py * v.cam.W + px;
    if (twl == 3 && Dn == INT_MAX) emit_miss(v.hit, v.t, pix);  // nothing solid in the tile's view
    else cast_pixel<true>(v.scene, v.cam, v.frame, px, py, v.hit, v.t, pix, Dn, lanes);
}

// Descriptor patches in the order the host queued them (one thread: a later
// patch of the same descriptor must win, and there are at most kPatchMax).
__global__ void patch_desc_kernel(ChunkRef* __restrict__ desc, const __grid_constant__ DescPatches P) {
    if (threadIdx.x != 0) return;
    for (uint32_t i = 0; i < P.n; i++) desc[P.p[i].index] = P.p[i].ref;
}

__global__ void ray_dirs_kernel(CamDev C, float* __restrict__ dirs) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (size_t)C.W * (size_t)C.H) return;
    float d[3];
    ray_dir(C, (int)(i % (size_t)C.W), (int)(i / (size_t)C.W), d);
    dirs[3 * i] = d[0];
    dirs[3 * i + 1] = d[1];
    dirs[3 * i + 2] = d[2];
}

thread_local cudaError_t t_launch_error = cudaSuccess;

int status_of(cudaError_t e) { return aokk_status(e); }

}  // namespace

extern "C" {

int aokk_status(cudaError_t e) {
    if (e == cudaSuccess) return AOK_OK;
    t_launch_error = e;
    return AOK_E_CUDA;
}

cudaError_t aokk_take_launch_error() {
    cudaError_t e = t_launch_error;
    t_launch_error = cudaSuccess;
    if (e == cudaSuccess) e = cudaGetLastError();
    return e == cudaSuccess ? cudaErrorLaunchFailure : e;
}

int aokk_select(const SceneDev* s, const CamDev* c, ChunkRef* frame, int8_t* lod_out, uint8_t* vis_out,
                uint32_t* n_visible, void* stream) {
    const int nch = s->grid[0] * s->grid[1] * s->grid[2];
    select_kernel<<<(nch + 127) / 128, 128, 0, (cudaStream_t)stream>>>(*s, *c, frame, lod_out, vis_out, n_visible);
    return status_of(cudaGetLastError());
}

static cudaError_t cast_plain(const SceneDev* s, const CamDev* c, const ChunkRef* frame, uint4* hit, float* t,
                              cudaStream_t st) {
    int wl, hl;
    cast_tile(*c, wl, hl);
    dim3 grid((c->W + (2 << wl) - 1) >> (wl + 1), (c->H + (2 << hl) - 1) >> (hl + 1));
    // launched while the selection before it runs: 38 / 46 / 57 -> 36 / 44 / 55 us for 256x256 views, 63 / 71 / 86
    // -> 61 / 70 / 83 for 320x180 (behind a beam pass, whose SMs its blocks would crowd, frames got 1% longer)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(128);
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, cast_kernel<false>, *s, *c, frame, hit, t, (uint32_t*)nullptr,
                              beam_lookup(nullptr, 0, 0), wl, hl);
}

int aokk_cast(const SceneDev* s, const CamDev* c, const ChunkRef* frame, uint4* hit, float* t, uint32_t* counts,
              void* stream, const CheckDev* ck, const BeamRead* beam) {
    dim3 grid((c->W + 15) / 16, (c->H + 7) / 8);
    const cudaStream_t st = (cudaStream_t)stream;
    int wl = 3, hl = 2;
    const BeamLookup bl = beam_lookup(beam, c->W, c->H);
    if (ck && !counts && beam)
        cast_kernel_checked<true><<<grid, 128, 0, st>>>(*s, *c, frame, hit, t, *ck, bl);
    else if (ck && !counts)
        cast_kernel_checked<false><<<grid, 128, 0, st>>>(*s, *c, frame, hit, t, *ck, bl);
    else if (counts && beam)
        cast_kernel<true, true><<<grid, 128, 0, st>>>(*s, *c, frame, hit, t, counts, bl, wl, hl);
    else if (counts)
        cast_kernel<true><<<grid, 128, 0, st>>>(*s, *c, frame, hit, t, counts, bl, wl, hl);
    else if (beam)
        cast_kernel<false, true><<<grid, 128, 0, st>>>(*s, *c, frame, hit, t, nullptr, bl, wl, hl);
    else
        return status_of(cast_plain(s, c, frame, hit, t, st));
    return status_of(cudaGetLastError());
}

int aokk_select_batch(const BatchParams* p, void* stream) {
    dim3 grid((p->max_chunks + 127) / 128, p->n_views);
    select_batch_kernel<<<grid, 128, 0, (cudaStream_t)stream>>>(*p);
    return status_of(cudaGetLastError());
}

int aokk_cast_batch(const BatchParams* p, uint32_t ctas, uint32_t threads, void* stream) {
    if (ctas == 0)  // grid launch: one 128-thread block per block tile
        cast_grid<<<(unsigned)p->total_tiles, 128, 0, (cudaStream_t)stream>>>(*p);
    else
        cast_persistent<<<ctas, threads, 0, (cudaStream_t)stream>>>(*p);
    return status_of(cudaGetLastError());
}

// Run n_groups (select, cast) launch pairs on `stream`; with beams, each
// group's beam pass (beams[g], one cooperative launch) runs between its
// selection and its cast.  With a cache and no hand-off stream, the whole
// sequence is one CUDA graph built per shape (group sizes, launch dims, which
// groups hold a beam pass) -- select, cooperative beam
// kernel, cast per group, chained -- whose nodes are updated with the new
// parameters on every call; a graph holding beam passes keeps the per-device
// order of passes around its launch.
int aokk_batch_run(const BatchParams* groups, uint32_t n_groups, uint32_t ctas, uint32_t threads, void* stream,
                   const BeamBatch* beams, unsigned beam_grid, const BeamHandoff* handoff, GraphCache* gc) {
    const cudaStream_t st = (cudaStream_t)stream;
    auto has_beam = [&](uint32_t g) { return beams && beams[g].n_views > 0; };
    if (!gc || handoff) {
        for (uint32_t g = 0; g < n_groups; g++) {
            int r = aokk_select_batch(&groups[g], stream);
            if (!r && has_beam(g)) {
                if (handoff) {
                    const cudaStream_t bs = (cudaStream_t)handoff->stream;
                    cudaError_t e = cudaEventRecord(handoff->sel, st);
                    if (e == cudaSuccess) e = cudaStreamWaitEvent(bs, handoff->sel, 0);
                    r = aokk_status(e);
                    if (!r) r = aokk_beam_run(&beams[g], beam_grid, handoff->stream);
                    if (!r) {
                        e = cudaEventRecord(handoff->beam, bs);
                        if (e == cudaSuccess) e = cudaStreamWaitEvent(st, handoff->beam, 0);
                        r = aokk_status(e);
                    }
                } else {
                    r = aokk_beam_run(&beams[g], beam_grid, stream);
                }
            }
            if (!r) r = aokk_cast_batch(&groups[g], ctas, threads, stream);
            if (r) return r;
        }
        return AOK_OK;
    }
    bool any_beam = false;
    std::vector<uint64_t> key{n_groups, ctas, threads, beam_grid};
    for (uint32_t g = 0; g < n_groups; g++) {
        key.push_back(groups[g].n_views);
        key.push_back(groups[g].max_chunks);
        if (!ctas) key.push_back(groups[g].total_tiles);  // grid size of the casting node
        key.push_back(has_beam(g) ? 1u + beams[g].n_regions : 0u);  // the pass's grid depends on its regions
        any_beam |= has_beam(g);
    }
    auto params = [&](uint32_t g, bool sel, void** argp, cudaKernelNodeParams& kp) {
        argp[0] = (void*)&groups[g];
        kp.func = sel ? (void*)select_batch_kernel : (ctas ? (void*)cast_persistent : (void*)cast_grid);
        kp.gridDim = sel ? dim3((groups[g].max_chunks + 127) / 128, groups[g].n_views)
                         : dim3(ctas ? ctas : (unsigned)groups[g].total_tiles);
        kp.blockDim = sel ? dim3(128) : dim3(ctas ? threads : 128);
        kp.sharedMemBytes = 0;
        kp.kernelParams = argp;
        kp.extra = nullptr;
    };
    cudaError_t e = cudaSuccess;
    if (!gc->exec || gc->key != key) {
        aokk_graph_destroy(gc);
        e = cudaGraphCreate(&gc->graph, 0);
        cudaGraphNode_t prev = nullptr;
        auto add = [&](cudaGraphNode_t node) {
            gc->nodes.push_back(node);
            prev = node;
        };
        for (uint32_t g = 0; g < n_groups && e == cudaSuccess; g++) {
            void* argp[1];
            cudaKernelNodeParams kp;
            cudaGraphNode_t node;
            params(g, true, argp, kp);
            e = cudaGraphAddKernelNode(&node, gc->graph, prev ? &prev : nullptr, prev ? 1 : 0, &kp);
            if (e != cudaSuccess) break;
            add(node);
            if (has_beam(g)) {
                aokk_beam_node(&beams[g], beam_grid, argp, &kp);
                e = cudaGraphAddKernelNode(&node, gc->graph, &prev, 1, &kp);
                if (e != cudaSuccess) break;
                cudaLaunchAttributeValue coop;
                std::memset(&coop, 0, sizeof(coop));
                coop.cooperative = 1;
                e = cudaGraphKernelNodeSetAttribute(node, cudaLaunchAttributeCooperative, &coop);
                if (e != cudaSuccess) break;
                add(node);
            }
            params(g, false, argp, kp);
            e = cudaGraphAddKernelNode(&node, gc->graph, &prev, 1, &kp);
            if (e != cudaSuccess) break;
            add(node);
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&gc->exec, gc->graph, 0);
        if (e != cudaSuccess) {
            aokk_graph_destroy(gc);
            return aokk_status(e);
        }
        gc->key = key;
    } else {
        size_t i = 0;
        for (uint32_t g = 0; g < n_groups && e == cudaSuccess; g++) {
            void* argp[1];
            cudaKernelNodeParams kp;
            params(g, true, argp, kp);
            e = cudaGraphExecKernelNodeSetParams(gc->exec, gc->nodes[i++], &kp);
            if (e == cudaSuccess && has_beam(g)) {
                aokk_beam_node(&beams[g], beam_grid, argp, &kp);
                e = cudaGraphExecKernelNodeSetParams(gc->exec, gc->nodes[i++], &kp);
            }
            if (e == cudaSuccess) {
                params(g, false, argp, kp);
                e = cudaGraphExecKernelNodeSetParams(gc->exec, gc->nodes[i++], &kp);
            }
        }
        if (e != cudaSuccess) return aokk_status(e);
    }
    int r = any_beam ? aokk_beam_order(stream, 0) : AOK_OK;
    if (!r) r = status_of(cudaGraphLaunch(gc->exec, st));
    if (!r && any_beam) r = aokk_beam_order(stream, 1);
    return r;
}

void aokk_graph_destroy(GraphCache* gc) {
    if (gc->exec) cudaGraphExecDestroy(gc->exec);
    if (gc->graph) cudaGraphDestroy(gc->graph);
    gc->exec = nullptr;
    gc->graph = nullptr;
    gc->nodes.clear();
    gc->key.clear();
}

int aokk_max_ctas_per_sm(uint32_t threads) {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, cast_persistent, (int)threads, 0);
    return n;
}

int aokk_patch_desc(ChunkRef* desc, const DescPatches* p, void* stream) {
    if (p->n == 0) return AOK_OK;
    patch_desc_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(desc, *p);
    return status_of(cudaGetLastError());
}

int aokk_ray_dirs(const CamDev* c, float* dirs, void* stream) {
    const size_t n = (size_t)c->W * (size_t)c->H;
    ray_dirs_kernel<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream>>>(*c, dirs);
    return status_of(cudaGetLastError());
}

// ---------------------------------------------------------------------------
// Read bandwidth microbenchmark: one resident grid streams the buffer `passes`
// times in 16-byte words through L2 (ld.global.cg, L1 bypassed; volatile so
// that no pass is merged with another), four independent loads in flight per
// thread.  A buffer smaller than L2 measures L2 read bandwidth, a larger one
// HBM read bandwidth.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t ld_cg_xor(const uint4* p) {
    uint32_t a, b, c, d;
    asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(a), "=r"(b), "=r"(c), "=r"(d) : "l"(p));
    return a ^ b ^ c ^ d;
}

__global__ void __launch_bounds__(512) read_bw_kernel(const uint4* __restrict__ p, size_t n, int passes,
                                                      uint32_t* __restrict__ sink) {
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    uint32_t acc = 0;
    for (int r = 0; r < passes; r++) {
        size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
        for (; i + 3 * stride < n; i += 4 * stride)
            acc ^= ld_cg_xor(p + i) ^ ld_cg_xor(p + i + stride) ^ ld_cg_xor(p + i + 2 * stride) ^
                   ld_cg_xor(p + i + 3 * stride);
        for (; i < n; i += stride) acc ^= ld_cg_xor(p + i);
    }
    if (acc == 0x9E3779B9u) sink[0] = acc;  // data-dependent store keeps the loads
}

int aokk_read_bw(const void* buf, size_t n16, int passes, uint32_t* sink, int sms, void* stream) {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, read_bw_kernel, 512, 0);
    read_bw_kernel<<<sms * std::max(per_sm, 1), 512, 0, (cudaStream_t)stream>>>((const uint4*)buf, n16, passes, sink);
    return status_of(cudaGetLastError());
}

// ---------------------------------------------------------------------------
// Render without allocating: the per-frame chunk table lives in a file-scope
// device array instead of scene-owned memory.  The array is created when the
// module loads on a device and stays until the process exits.  Its device
// address is looked up once per device (with that device current) and
// cached; every call then reuses the same array, so calls that overlap on the
// GPU race on it.  select_kernel overwrites every entry of the scene's grid
// before cast_kernel reads it, so nothing needs clearing between calls.
// ---------------------------------------------------------------------------
static __device__ __align__(256) ChunkRef g_noalloc_frame[AOK_NOALLOC_MAX_CHUNKS];

static std::atomic<ChunkRef*> g_noalloc_ptr[kMaxDevices];
static std::mutex g_noalloc_mu;

int aokk_render_noalloc(const SceneDev* s, const CamDev* c, uint4* hit, float* t, void* stream, const CheckDev* ck) {
    const long long nch = (long long)s->grid[0] * s->grid[1] * s->grid[2];
    if (nch > AOK_NOALLOC_MAX_CHUNKS) return AOK_E_INVALID;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return AOK_E_CUDA;
    if (dev < 0 || dev >= kMaxDevices) return AOK_E_INVALID;
    ChunkRef* frame = g_noalloc_ptr[dev].load(std::memory_order_acquire);
    if (!frame) {
        std::lock_guard<std::mutex> g(g_noalloc_mu);
        frame = g_noalloc_ptr[dev].load(std::memory_order_relaxed);
        if (!frame) {
            void* p = nullptr;
            const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_frame);
            if (e != cudaSuccess || !p) return AOK_E_CUDA;
            frame = (ChunkRef*)p;
            g_noalloc_ptr[dev].store(frame, std::memory_order_release);
        }
    }
    const cudaStream_t st = (cudaStream_t)stream;
    select_kernel<<<(unsigned)((nch + 127) / 128), 128, 0, st>>>(*s, *c, frame, nullptr, nullptr, nullptr);
    dim3 grid((c->W + 15) / 16, (c->H + 7) / 8);
    if (ck)
        cast_kernel_checked<false><<<grid, 128, 0, st>>>(*s, *c, frame, hit, t, *ck, beam_lookup(nullptr, 0, 0));
    else
        return status_of(cast_plain(s, c, frame, hit, t, st));
    return status_of(cudaGetLastError());
}

int aokk_sm_count(int device) {
    int n = 0;
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, device);
    return n;
}

}  // extern "C"
