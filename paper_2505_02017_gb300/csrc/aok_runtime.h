// Host-side state of the runtime (not part of the C ABI).
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <condition_variable>
#include <cstdint>
#include <deque>
#include <map>
#include <memory>
#include <mutex>
#include <thread>
#include <unordered_map>
#include <utility>
#include <vector>

#include "aok_internal.h"

namespace aok {

constexpr uint64_t kNoRange = ~0ull;

struct Pool {  // units of the pool's element type
    uint64_t cap = 0, used = 0;
    std::vector<std::pair<uint64_t, uint64_t>> free_list;  // (offset, count)
    uint64_t alloc(uint64_t n);
    void release(uint64_t off, uint64_t n);
};

struct ChunkAlloc {
    uint64_t node_off = 0, node_n = 0, leaf_off = 0, leaf_n = 0, mat_off = 0, mat_n = 0;
};

struct Scene {
    aok_scene_desc desc{};
    double color_tol = -1.0;  // colour-block tolerance of later uploads (< 0: raw arrays)
    int mlog = 0;
    int64_t n_chunks = 0;
    uint32_t* d_nodes = nullptr;
    uint64_t* d_leaves = nullptr;
    uint8_t* d_mats = nullptr;
    ChunkRef* d_desc = nullptr;   // [chunk * n_lods + lod]
    ChunkRef* d_frame = nullptr;  // per-frame selection of aok_render
    uint64_t select_gen = 0;      // selections written into d_frame so far
    Pool nodes, leaves, mats;
    std::vector<ChunkRef> h_desc;
    std::vector<ChunkAlloc> alloc;
    std::mutex mu;
    std::vector<aok_stream*> streams;  // streamers of this scene (guarded by mu)
};

// Stop a streamer of a scene that is being destroyed: join its workers, free
// its loads and quarantined space; the object stays for aok_stream_destroy.
void stream_detach(aok_stream* s);

// A grow-only array of beam pyramid entries.
struct BoundBuf {
    unsigned long long* p = nullptr;
    size_t cap = 0;      // entries
    uint32_t epoch = 0;  // of the tags in it (beam_renew)
};

// Device arena of aok_render_batch: per-view frame tables, work counters and
// the CUDA graph of the last list shape.
struct BatchArena {
    ChunkRef* d_frames = nullptr;
    size_t frames_cap = 0;
    BoundBuf beam_bounds;                   // the views' bound pyramids
    unsigned long long* d_queue = nullptr;  // 2 per group, zero between launches
    size_t queue_cap = 0;
    GraphCache graph;
};

struct ServeState;

// Frames rendered into host memory through a pipeline: slot k's selection
// and beam pass (on `prep`, the highest stream priority) overlap slot k-1's
// cast (on `render`), which overlaps slot k-2's device-to-host copy (on
// `copy`).  Each slot has its own chunk table and bound pyramid.
constexpr int kHostSlots = 3;
struct HostSlot {
    void* hit = nullptr;
    float* t = nullptr;
    ChunkRef* frame = nullptr;  // the slot's chunk table
    size_t frame_cap = 0;       // entries
    BoundBuf bounds;            // the slot's bound pyramid
    cudaEvent_t prepped = nullptr, rendered = nullptr, copied = nullptr;
    uint64_t ticket = 0;  // frame in this slot (0: none yet)
};
struct HostPipe {
    cudaStream_t prep = nullptr, render = nullptr, copy = nullptr;
    HostSlot slot[kHostSlots];
    size_t px = 0;        // pixels each slot holds
    uint64_t next = 0;    // last ticket issued
};

// Buffers of the tile-chunk pipeline for one resolution and grid size (one
// device allocation carved into the TileDev arrays), and the scene whose
// Hi-Z history hiz_prev holds.
struct TileState {
    TileDev dev{};
    void* block = nullptr;
    size_t bytes = 0;
    int32_t W = 0, H = 0;
    int64_t n_chunks = 0;
    uint32_t scene = 0xFFFFFFFFu;
};

// A walk's queues of `cap` nodes a level, the counts per level and, of the
// last pass (not a single view's), the walk histogram.
struct BeamQueues {
    uint4* q[2] = {nullptr, nullptr};
    uint32_t *cnt = nullptr, *hist = nullptr;
    uint32_t cap = 0;
};

// The beam pass: the walk's queues and launch grid (shared by all passes of
// the context), the single-view bound pyramid and what its last pass was
// computed for.
struct BeamState {
    // The single-view passes' buffers and records, until a pass and the cast
    // that reads it are enqueued.  Frames without the pass don't take it, nor
    // do batches, host frames and the server, which have their own buffers.
    std::mutex view_mu;
    std::mutex mu;  // the queues' allocation and the pass counter (the serving thread shares them)
    void* qblock = nullptr;
    size_t qbytes = 0;
    BeamQueues q;              // of the passes that frames have to take
    unsigned grid = 0;         // blocks of the cooperative launch
    BoundBuf bounds;           // single-view pyramid
    // What the passes use that frames need not take: one block beside the
    // budget, allocated with the context (14 MB), so that such a frame needs
    // no memory of its own, in its first pass or later, and takes none from
    // what the budget is for.  Without it (opt_block == nullptr: the device
    // had no room) there are no such passes.
    void* opt_block = nullptr;
    BeamQueues opt_q;
    uint32_t* view_hist = nullptr;  // walk histogram of the last single view's pass
    BoundBuf opt, opt_host[kHostSlots], opt_batch;
    // the last cast that read `opt`: the next one may come on a stream that
    // nothing orders with it
    cudaEvent_t opt_read = nullptr;
    unsigned long long opt_stream = 0;  // that cast's stream
    uint32_t passes = 0;                   // passes run in this epoch (their tags count down)
    std::atomic<uint32_t> epoch{0};        // times the tags have started over
    std::atomic<uint64_t> total{0};        // passes run
    // the last single-view pass, for aok_beam_info
    bool ran = false;
    BeamRead last{nullptr, 0};
    int32_t W = 0, H = 0;
    // the last one kept for the cast of its selection: a scene, its selection, a camera
    bool valid = false;
    uint32_t scene = 0xFFFFFFFFu;
    uint64_t gen = 0;
    CamDev cam{};
    BeamRead read{nullptr, 0};
};

// The reachable nodes of a chunk blob by depth, found while it is validated
// and used to lay it out.  The vectors keep their storage from one blob to the
// next (a blob's would be fresh pages of several MB each time).
struct BlobPlan {
    std::vector<uint32_t> ord;    // [blob words] place of the node at this word in `node`, or kNoOrd
    std::vector<uint32_t> node;   // word index of every reachable node, by depth
    std::vector<uint32_t> level;  // [levels + 1] first place of each depth
    std::vector<uint32_t> off;    // device word offset of every reachable node
    std::vector<uint16_t> box;    // solid-voxel box of every reachable node: lo x, y, z, hi x, y, z
    uint64_t words = 0;           // device words of the nodes
    static constexpr uint32_t kNoOrd = 0xFFFFFFFFu;
};

struct aok_ctx_impl;

}  // namespace aok

struct aok_ctx {
    int device = 0;
    int sm_count = 0;
    size_t budget = 0, used = 0;
    std::mutex mem_mu;
    cudaError_t last_cuda = cudaSuccess;
    cudaStream_t copy_stream = nullptr;
    std::mutex scene_mu;
    std::map<uint32_t, aok::Scene*> scenes;
    uint32_t next_scene = 0;
    void* staging = nullptr;
    size_t staging_cap = 0;
    aok::BlobPlan upload_plan;  // (with the staging buffer, under upload_mu)
    uint32_t* pinned_word = nullptr;
    uint32_t* d_counter = nullptr;
    // persistent casting launch shape (0 = defaults) and single-view kernel choice
    uint32_t ctas_per_sm = 0, threads_per_cta = 0, packet_rays = 0, tile_w_log = 0;
    int single_persistent = 0;
    int batch_persistent = 0;  // 0: batches cast with one grid launch over block tiles
    int batch_graph = 1;       // 1: a batch's launches replay as one CUDA graph
    unsigned long long* d_single_queue = nullptr;  // counters of single-view persistent launches
    aok::BatchParams single_params;
    aok::BatchArena batch;
    // device frame of aok_render_host
    void* host_hit_dev = nullptr;
    float* host_t_dev = nullptr;
    size_t host_frame_px = 0;
    aok::ServeState* serve = nullptr;
    aok::TileState tiles;
    aok::BeamState beam;
    int beam_on = 1;  // single-view renders run the beam pass before casting
    uint32_t beam_refine = AOK_BEAM_REFINE;  // refine nodes spanning more tiles than this ...
    int beam_min_log2 = 2;     // ... whose side is above 2^this LOD-0 voxels
    // Frames of beam_min_pixels take the pass.  Those of beam_min_optional take it where it can run: not on a stream
    // that is being captured (the passes of a device wait for one another by events a capture can't hold) and not
    // beyond the room of its buffers.  Smaller ones cast without it (city views of 1120 x 630 break
    // even at 160-240 us, 1280 x 720 ones gain 12% on average with it, -29% to +12%, and 960 x 540 ones nothing).
    uint64_t beam_min_pixels = AOK_BEAM_MIN_PIXELS, beam_min_optional = AOK_BEAM_MIN_OPTIONAL;
    uint32_t beam_queue = 0;             // nodes a queue level may hold (0: the allocated 2^20)
    aok::HostPipe pipe;
    int checked = 0;  // single-view casts check every pool index (error word: d_counter[8])
    std::mutex upload_mu;  // the staging buffer and the copy stream: one upload at a time
};

namespace aok {
int cuda_status(aok_ctx* ctx, cudaError_t e);
// AOK_E_CUDA for a launcher that returned AOK_E_CUDA, with the error code it read.
int launch_failure(aok_ctx* ctx);
int charge(aok_ctx* ctx, size_t bytes);
void uncharge(aok_ctx* ctx, size_t bytes);
int dev_alloc(aok_ctx* ctx, void** p, size_t bytes);
void dev_free(aok_ctx* ctx, void* p, size_t bytes);
Scene* find_scene(aok_ctx* ctx, uint32_t id);
int make_cam(aok_ctx* ctx, const Scene* sc, const aok_camera* cam, double tau, CamDev* out);
SceneDev scene_dev(const Scene* sc);
void batch_release(aok_ctx* ctx);
void free_alloc(Scene* sc, ChunkAlloc& a);
// The beam passes of a batch (one per group) for its views of at least the
// context's beam frame size; sets the views' bounds, in the batch arena or,
// with view_bounds, in view_bounds[view] (nullptr: that view casts without).
// Leaves `out` empty if no view takes the pass.
// (arena: the buffer that some of view_bounds lie in; the others are cleared
// for every pass.  pass_stream: where those passes run.)
int beam_for_batch(aok_ctx* ctx, BatchParams* groups, uint32_t ngroups, std::vector<BeamBatch>& out, void* stream,
                   unsigned long long* const* view_bounds = nullptr, BoundBuf* arena = nullptr,
                   void* pass_stream = nullptr);
// Whether a frame of W x H pixels on `stream` takes the beam pass in this
// context, and whether it may also be cast without.
inline bool beam_required(const aok_ctx* ctx, int32_t W, int32_t H) {
    return ctx->beam_on && (uint64_t)W * (uint64_t)H >= ctx->beam_min_pixels;
}
enum BeamUse { kBeamNone, kBeamOptional, kBeamRequired };
BeamUse beam_use(const aok_ctx* ctx, int32_t W, int32_t H, void* stream);
// Lets this thread query an event while another one captures a stream in the
// global capture mode (whose capture the query would end).
struct RelaxedCapture {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
    ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};
// Pinned staging memory and the stream its copies go on.
struct Staging {
    void* buf = nullptr;
    size_t cap = 0;
    cudaStream_t stream = nullptr;
    size_t min_cap = (size_t)64 << 20;  // smallest buffer allocated when it grows
    BlobPlan plan;
};
int stage_chunk(aok_ctx* ctx, Scene* sc, int64_t di, uint32_t lod, const aok_chunk_blob* blob, bool evict_old_first,
                Staging* stg, std::mutex* pool_mu, ChunkAlloc* out_a, ChunkRef* out_ref);
int render_persistent(aok_ctx* ctx, Scene* sc, const CamDev& cd, const aok_frame* frame, void* stream, bool select);
}  // namespace aok
