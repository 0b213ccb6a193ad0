// Host side of the C ABI declared in include/mv.h: argument checks, allocation of the
// device-resident world store, and the kernel launches.  No rendering arithmetic runs here.
#define MV_ENABLE_TEST_HOOKS
#include "../../include/mv.h"
#include "mv_device.cuh"
#include "mv_pack.cuh"
#include "mv_merge.cuh"
#include "mv_render.cuh"
#include "mv_scene.cuh"

#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

using namespace mv;

namespace {

// Threads per CTA of the render kernel, by how many CTAs the staged blocks leave room for on an SM: three (or more) of 384 threads or
// two of 576, so that as many warps walk (2048 x 2 observations of 160x32x160 rooms, 104 KB a block: 342 us with 384, 308).
// (Blocks that would leave one alone are staged in small batches and under large images only, see mv_create_batch.)
constexpr int kRenderThreads = 384, kRenderThreadsTwo = 576;
constexpr int kRenderThreadsSmall = 192;       // CTAs with few tiles (small images): twice as many, shorter CTAs per SM
// Below this many tiles per CTA the small shape is faster when there are CTAs enough to fill the GPU with it and room for five on
// an SM (measured: 64x36 images +10 %; 128x72 -2 %; four CTAs alone on the GPU -20 %: fewer warps per CTA, longer CTA; 48x36
// with room for five 135.7 us, 140.2 with three of the ordinary shape).
constexpr int kSmallCtaTiles = 192;
constexpr int kHostChunks = 8;
// Staging and set-up of a CTA in tiles' worth of work, with the GPU full and with little to do (see pick_split).
constexpr double kSetupTiles = 28.0, kPartTiles = 8.0;
constexpr size_t kMergeScratchBytes = (size_t)1 << 30;         // bit arrays for the envs of one merge launch

inline uint32_t round_up(uint32_t v, uint32_t a) { return (v + a - 1) / a * a; }

}  // namespace

// The first `whole` CTAs of a render have agents_per_cta observations each, the other observations `parts` CTAs each.
struct Split { int64_t whole; int parts; };

struct mv_batch {
    mv_batch_desc desc;
    int num_obs = 0;
    size_t mat_bytes_per_env = 0;       // material store: one byte per voxel index (columns padded to 2^ysh)
    EnvLayout lay{};
    unsigned char *d_env_blocks = nullptr;
    uint8_t *d_mat = nullptr;
    CamRec *d_cams = nullptr;
    uint32_t *d_status = nullptr;
    int *d_acc = nullptr;               // [E][kPackAccInts] accumulators of the uploads in flight
    uint32_t *d_merge = nullptr;        // merge scratch: MergeLayout::env_words for merge_chunk envs
    MergeLayout merge{};
    int merge_chunk = 0;
    int4 *d_overlay = nullptr;          // [O][max_overlay_rects]
    int32_t *d_overlay_count = nullptr; // [O]
    int32_t *d_env_index = nullptr;     // [E] destination envs of a scattered upload (mv_upload_worlds_at)
    // host-side readiness tracking (per env)
    std::vector<uint8_t> has_grid, has_palette;
    int missing_grid = 0, missing_palette = 0;
    bool has_cams = false;
    double kr = 0, ku = 0;
    uint32_t sky_rgbx = 0;
    struct Smem { uint32_t tile_off, agent_off, agent_stride, agent_ov_off, agent_mask_off, misc_off, bytes; };
    Smem smem{};                        // shared-memory layout of the render kernel for agents_per_cta
    int agents_per_cta = 1;             // observations one CTA renders: 1, or every agent of its env
    int threads = kRenderThreads;       // threads per CTA of the render kernel (fewer for CTAs with few tiles)
    int sms = 0;
    int resident = 1;                   // CTAs of the render kernel that an SM holds
    int forced_parts = 0;               // test hooks: CTAs per observation (0: pick_split decides),
    bool forced_agents = false;         // agents_per_cta as the caller wants it, also in a small batch
    int tiles_x = 0, tiles_y = 0, mask_words = 0;
    int64_t launches = 0;
    int wait_polls = 1 << 18;
    bool occ_shared = true;             // occupancy staged in shared memory (else read from global)
    bool want_occ_shared = true;        // the same where it fits: the library's choice, or the caller's (a test hook)
    int smem_sm = 0;                    // shared memory of an SM
    int smem_max = 0;                   // opt-in shared memory per CTA of the device
    int auto_agents_per_cta = 1;        // the library's own choice (a test hook can override it)
    int skip_staging = 0;
    bool prefetch = false;              // occupancy in global memory is asked for in L2 (prefetch_pays, or a test hook)
    int last_cuda_error = 0;
    // mv_step_host resources (allocated on first use)
    uint8_t *d_rgb = nullptr;
    float *d_depth = nullptr;
    mv_camera *d_cam_in = nullptr;
    mv_box *d_box_in = nullptr;
    int32_t *d_count_in = nullptr;
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t ev_chunk[kHostChunks] = {};
    cudaEvent_t ev_done = nullptr;
    bool host_ready = false;
};

namespace {

int cuda_fail(mv_batch *b, cudaError_t e) {
    if (b) b->last_cuda_error = (int)e;
    return e == cudaErrorMemoryAllocation ? MV_ERR_OUT_OF_MEMORY : MV_ERR_CUDA;
}

#define MV_CUDA(b, call)                                   \
    do {                                                   \
        cudaError_t e_ = (call);                           \
        if (e_ != cudaSuccess) return cuda_fail((b), e_);  \
    } while (0)

struct DeviceGuard {
    int prev = -1;
    bool ok = false, changed = false;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) return;
        ok = prev == dev || (changed = cudaSetDevice(dev) == cudaSuccess);
    }
    ~DeviceGuard() { if (changed) cudaSetDevice(prev); }
};

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Shared-memory layout of the render kernel when one CTA renders `apc` observations of an env:
// staged env block (without the occupancy when that stays in global memory), tile table, then one block per agent (ray
// table, camera record, eye-relative boxes, overlay rectangles, per-tile masks of boxes and the GUI bit), then the barrier
// and flag words and the planes' guards.
mv_batch::Smem smem_layout(const mv_batch *b, int apc, bool occ_shared) {
    const mv_batch_desc &d = b->desc;
    const uint32_t ntiles = (uint32_t)(b->tiles_x * b->tiles_y);
    mv_batch::Smem m{};
    m.tile_off = round_up(b->lay.block_bytes - (occ_shared ? 0u : b->lay.occ_bytes), 16);
    m.agent_off = round_up(m.tile_off + ntiles * 16, kAgentAlign);
    m.agent_ov_off = kAgentRelOff + (uint32_t)d.max_boxes * 32;
    m.agent_mask_off = m.agent_ov_off + (uint32_t)d.max_overlay_rects * 32;
    // per tile: the box-mask words, preceded by a summary word when there is more than one
    const uint32_t words_per_tile = b->mask_words > 1 ? (uint32_t)b->mask_words + 1 : 1u;
    const uint32_t agent_bytes = m.agent_mask_off + round_up(ntiles * words_per_tile * 4, 16);
    m.agent_stride = apc > 1 ? round_up(agent_bytes, kAgentAlign) : agent_bytes;
    m.misc_off = m.agent_off + (uint32_t)apc * m.agent_stride;
    m.bytes = m.misc_off + 32;
    return m;
}

// Launch of a per-step kernel (see launch_dependents).
template <typename... Params, typename... Args>
cudaError_t launch_step(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const Args &...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute overlap{};
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &overlap;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

int pick_threads(const mv_batch *b, int apc) {
    const int per_sm = b->smem_sm / ((int)smem_layout(b, apc, b->occ_shared).bytes + 1024);        // (1 KB of every CTA is the system's)
    if (per_sm < 3) return kRenderThreadsTwo;
    const bool few_tiles = b->tiles_x * b->tiles_y * apc < kSmallCtaTiles;
    const bool fills = (int64_t)b->num_obs / apc >= (int64_t)6 * b->sms;
    return few_tiles && fills && per_sm >= 5 ? kRenderThreadsSmall : kRenderThreads;
}

// How a render of `obs` observations is dealt to CTAs; R = CTAs that are resident at once, costs in units of an observation's work.
// - Less than about a round of CTAs: every observation in parts, as many as cost least: a part's length while all parts run at
//   once (so few observations get as many parts as make a tile for every warp), with more the rounds it takes.
// - More: the observations of the last R / 2 CTAs one by one, and those of CTAs of one or two agents in up to three parts, fewer
//   for small images; the others whole.  Cost: the work of all CTAs, set-up included, over R, and some of the last one's length.
// Against three CTAs made to an SM of contiguous parts, and all whole from a round on: 300 observations of 128x32x128 columns 38.2
// us and 57.0, 1024 x 2 of 128x72 rooms 107.6 and 111.7, 4096 x 4 900.4 and 914.7.  The costs are rough: among small batches the
// number of parts can be off by one or two from the best, for 3 to 9 % (112 observations of 88x60: 10.4 us in four parts, 9.2 in three).
// `cost`: what the choice costs, for the choice between CTAs of one and of all agents.
Split pick_split(const mv_batch *b, int64_t obs, double *cost = nullptr) {
    const int ntiles = b->tiles_x * b->tiles_y, apc = b->agents_per_cta, most = ntiles / (b->threads / 32) > 1 ? ntiles / (b->threads / 32) : 1;
    const int64_t ctas = obs / apc;
    const double R = (double)b->resident * b->sms, setup = kSetupTiles / ntiles;
    double least = 0.0, unused;
    if (!cost) cost = &unused;
    *cost = 0.0;
    const double speed = (double)b->threads / kRenderThreads;              // of a CTA, with the GPU full
    if (b->forced_parts > 0) return {0, b->forced_parts > most ? most : b->forced_parts};
    if (ctas >= 0.9 * R) {
        int parts = (ntiles + 35) / 72;
        parts = (parts > 3 ? 3 : parts) - (apc - 1);
        if (parts < 1) parts = 1;
        const int64_t tail = parts * apc > 1 ? (int64_t)(R / 2) : 0;
        least = ((double)(ctas - tail) * (apc + setup) + (double)tail * apc * (1 + parts * setup)) / R + 0.6 * (tail ? 1.0 / parts + setup : apc + setup);
        *cost = least / speed;
        return {ctas - tail, parts};
    }
    if (b->forced_agents) return {ctas, 1};
    Split best{0, most};
    const double part_setup = kPartTiles / ntiles;
    auto cost_of = [&](int parts) {
        const double part = 1.0 / parts + part_setup, rounds = obs * (double)parts / R;
        return rounds > 1.0 ? part * (rounds + 0.15) : part;
    };
    least = cost_of(most);
    if ((double)obs * most > R) {
        // (the most parts that run at once, or about the least of (1 / parts + part_setup) (obs parts / R + 0.15))
        const int at_once = (int)(R / obs), even = (int)std::sqrt(0.15 * R / (part_setup * obs));
        for (int parts : {at_once, at_once + 1, even, even + 1}) {
            parts = parts < 1 ? 1 : parts > most ? most : parts;
            const double c = cost_of(parts);
            if (c < least) { least = c; best.parts = parts; }
        }
    }
    *cost = least / speed;
    return best;
}

// The instantiations of the render kernel: by the CTA's threads, and one plane of occupancy staged, several staged, or read from
// global memory.
using RenderFn = void (*)(const RenderParams);
template <int NT> RenderFn render_fn_of(const mv_batch *b, bool occ_shared) {
    if (!occ_shared) return render_kernel<NT, kOccGlobal>;
    return b->lay.planes == 1 ? render_kernel<NT, kOccWord> : render_kernel<NT, kOccPlanes>;
}
RenderFn render_fn(const mv_batch *b, int threads, bool occ_shared) {
    return threads == kRenderThreadsSmall ? render_fn_of<kRenderThreadsSmall>(b, occ_shared) : threads == kRenderThreads ? render_fn_of<kRenderThreads>(b, occ_shared)
           : render_fn_of<kRenderThreadsTwo>(b, occ_shared);
}
RenderFn render_fn(const mv_batch *b) { return render_fn(b, b->threads, b->occ_shared); }

// Is a plane of occupancy per environment asked for in L2 as a render begins, where it is read from global memory?  A render finds
// its lines in HBM if other work has pushed them out of L2 since the last one, or if the batch itself does; rendered again and again with
// nothing in between, a batch that L2 holds has no use for it, and lines that no ray sees push out what is used.  So, with figures in us
// without / with, first after other work, then again and again (images of 128x72 but where it says so):
// - few environments, whose planes and frames L2 holds side by side, so that asking pushes nothing out.  192x48x192 columns 64 of them 60.4 /
//   43.2, 28.4 / 28.3; 320: 120.1 / 93.0, 68.4 / 68.6; 128 with 4 agents 118.5 / 105.3, 86.4 / 86.7; rooms 148: 33.8 / 29.7, 21.0 / 21.3; 320 of 64x36
//   39.9 / 33.8, 21.5 / 21.7.  More lose: 512 columns 115 / 106 but 78 / 86, 640: 84 / 113, 300 of 256x144 126 / 145, 400 rooms (both planes) 41.8 / 46.9.
// - more frames than L2 holds, which push everything out in every step, as long as the planes are not much beside the frames and an
//   image has few rays to share their lines.  2048 columns 248.4 / 222.2, 243.4 / 217.1; rooms 158.9 / 155.2, 153.2 / 149.7; 512 with 4 agents 236.4 / 211.8,
//   230.7 / 206.8; 4096 of 128x48x128 360.8 / 348.9, 355.4 / 343.0.  Not: planes four times the frames (2048 rooms of 256x64x256 152.7 / 166.5);
//   2048 rooms of 64x36 (both planes) 55.9 / 82.7; 1024 of 256x144 (both) 240.7 / 243.0.
bool prefetch_pays(const mv_batch *b) {
    const int64_t px = (int64_t)b->desc.width * b->desc.height, frames = 7 * px * b->num_obs, planes = (int64_t)b->desc.num_envs * b->lay.occ_plane;
    constexpr int64_t MB = 1 << 20;
    return (planes <= 46 * MB && planes + frames <= 68 * MB) || (frames >= 120 * MB && 2 * planes <= 5 * frames && px <= 1 << 14);
}

bool fits_staged(const mv_batch *b, int apc) { return (int64_t)smem_layout(b, apc, true).bytes <= b->smem_max; }

// CTA shape of the render kernel when a CTA renders `apc` observations of an environment (which has to fit unstaged at least).
int choose_shape(mv_batch *b, int apc) {
    b->agents_per_cta = apc;
    b->occ_shared = b->want_occ_shared && fits_staged(b, apc);
    b->smem = smem_layout(b, apc, b->occ_shared);
    b->threads = pick_threads(b, apc);
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b->resident, render_fn(b), b->threads, b->smem.bytes);
    if (e == cudaSuccess && b->resident >= 1) return MV_OK;
    cudaGetLastError();
    b->resident = 1;
    return e == cudaSuccess ? MV_ERR_UNSUPPORTED : cuda_fail(b, e);
}

// The merge sweep keeps a layer number per column: a byte for grids less than 256 high.  Rows of up to 16 words (W) are held in
// registers, one lane a row.
using MergeFn = void (*)(const unsigned char *, const uint8_t *, EnvLayout, MergeLayout, int, uint32_t *, uint4 *, int32_t *, int);
template <typename Cov> MergeFn merge_sweep_of(int W) {
    return W <= 2 ? merge_sweep_kernel<Cov, 2> : W <= 4 ? merge_sweep_kernel<Cov, 4> : W <= 8 ? merge_sweep_kernel<Cov, 8>
           : W <= 16 ? merge_sweep_kernel<Cov, 16> : merge_sweep_kernel<Cov, 0>;
}
MergeFn merge_sweep(int grid_y, int W) { return grid_y < 256 ? merge_sweep_of<uint8_t>(W) : merge_sweep_of<uint16_t>(W); }

int launch_render(mv_batch *b, uint8_t *d_rgb, float *d_depth, int obs_begin, int obs_count, cudaStream_t s) {
    RenderParams p{};
    p.env_blocks = b->d_env_blocks;
    p.mat = b->d_mat; p.mat_stride = b->mat_bytes_per_env;
    p.cams = b->d_cams;
    p.rgb = d_rgb;
    p.depth = d_depth;
    p.status = b->d_status;
    p.lay = b->lay;
    p.obs_begin = obs_begin;
    p.agents = b->desc.agents_per_env;
    p.max_boxes = b->desc.max_boxes;
    p.palette = b->desc.palette_size;
    p.W = b->desc.width; p.H = b->desc.height; p.inv_W = 1.0f / (float)b->desc.width;
    p.tiles_x = b->tiles_x; p.tiles_y = b->tiles_y; p.mask_words = b->mask_words;
    p.sky_rgbx = b->sky_rgbx;
    p.miss_depth = b->desc.miss_depth;
    p.smem_tile_off = b->smem.tile_off; p.smem_agent_off = b->smem.agent_off; p.smem_misc_off = b->smem.misc_off;
    p.agent_stride = b->smem.agent_stride; p.agent_ov_off = b->smem.agent_ov_off;
    p.agent_mask_off = b->smem.agent_mask_off;
    p.agents_per_cta = b->agents_per_cta;
    // accumulated crossing times drift from the exact products by at most one rounding per step
    p.exit_scale = 1.0f - (float)(b->desc.grid_x + b->desc.grid_y + b->desc.grid_z + 3) * 1.1920929e-7f;
    p.overlay = b->d_overlay;
    p.overlay_count = b->d_overlay_count;
    p.max_overlay = b->desc.max_overlay_rects;
    p.wait_polls = b->wait_polls;
    p.skip_staging = b->skip_staging;
    p.prefetch = b->prefetch;
    const Split split = pick_split(b, obs_count);         // (callers pass whole environments when a CTA renders one)
    p.whole_ctas = (unsigned)split.whole; p.parts = (unsigned)split.parts;
    const int64_t ctas = split.whole + (obs_count - split.whole * b->agents_per_cta) * split.parts;
    MV_CUDA(b, launch_step(render_fn(b), dim3((unsigned)ctas), dim3((unsigned)b->threads), b->smem.bytes, s, p));
    b->launches++;
    return MV_OK;
}

int launch_cameras(mv_batch *b, const mv_camera *d_cams, cudaStream_t s) {
    const int n = b->num_obs;
    MV_CUDA(b, launch_step(camera_kernel, dim3((n + 127) / 128), dim3(128), 0, s, reinterpret_cast<const int32_t *>(d_cams), b->d_cams, n,
                           b->kr, b->ku, b->d_status));
    b->launches++;
    b->has_cams = true;
    return MV_OK;
}

// One launch for whatever the upload brings (null: not in this upload).
int launch_upload(mv_batch *b, int env_begin, const int32_t *d_env_index, int env_count, const uint8_t *d_grid,
                  const mv_box *d_boxes, const int32_t *d_count, const uint8_t *d_palette, cudaStream_t s) {
    const mv_batch_desc &d = b->desc;
    UploadArgs u{};
    u.grid = d_grid; u.boxes = reinterpret_cast<const uint4 *>(d_boxes); u.counts = d_count; u.palette_rgb = d_palette;
    u.env_blocks = b->d_env_blocks; u.mat = b->d_mat; u.mat_stride = b->mat_bytes_per_env; u.acc = b->d_acc; u.status = b->d_status;
    u.env_index = d_env_index; u.lay = b->lay; u.env_begin = env_begin; u.env_count = env_count;
    u.gx = d.grid_x; u.gy = d.grid_y; u.gz = d.grid_z; u.max_boxes = d.max_boxes; u.palette = d.palette_size;
    for (int c = 0; c < 3; ++c) u.light[c] = (double)d.light_dir[c];
    u.ambient = (double)d.ambient;
    auto ctas = [](size_t threads) { return (threads + kUploadThreads - 1) / kUploadThreads; };
    u.words = (d.grid_y + 31) / 32;
    u.tiles_per_env = (int)ctas((size_t)(d.grid_x / 4) * d.grid_z) * u.words;
    // tiles a CTA packs one after the other: one, until there are two CTAs for every slot of the GPU (164 / 512 envs of
    // 128x32x128: 62 / 119 us with three CTAs of 256 threads per SM and four for every slot, 53 / 114 like this)
    const int64_t per_slot = (int64_t)u.tiles_per_env * env_count / (12 * 2 * (int64_t)b->sms);
    u.tiles_per_cta = (int)(per_slot < 1 ? 1 : per_slot > 8 ? 8 : per_slot);
    u.pack_ctas_per_env = (u.tiles_per_env + u.tiles_per_cta - 1) / u.tiles_per_cta;
    const size_t pack = d_grid ? (size_t)u.pack_ctas_per_env * env_count : 0;
    const size_t lut = d_palette ? ctas((size_t)env_count * kFaces * d.palette_size) : 0;
    const size_t box = d_boxes ? ctas((size_t)env_count * (d.max_boxes + 1)) : 0;
    if (pack + lut + box == 0) return MV_OK;
    if (pack + lut + box > 0x7fffffffull) return MV_ERR_INVALID_ARG;
    u.pack_ctas = (unsigned)pack; u.lut_ctas = (unsigned)lut;
    u.wait_polls = b->wait_polls; u.skip_staging = b->skip_staging;
    MV_CUDA(b, launch_step(upload_kernel, dim3((unsigned)(pack + lut + box)), dim3(kUploadThreads), pack ? kUploadSmem : 0, s, u));
    b->launches++;
    return MV_OK;
}

// First-use resources of mv_step_host: all of them or none, so that a failed attempt can be retried.
void free_host_step(mv_batch *b) {
    cudaFree(b->d_rgb); cudaFree(b->d_depth); cudaFree(b->d_cam_in); cudaFree(b->d_box_in); cudaFree(b->d_count_in);
    b->d_rgb = nullptr; b->d_depth = nullptr; b->d_cam_in = nullptr; b->d_box_in = nullptr; b->d_count_in = nullptr;
    if (b->copy_stream) cudaStreamDestroy(b->copy_stream);
    b->copy_stream = nullptr;
    for (auto &ev : b->ev_chunk) { if (ev) cudaEventDestroy(ev); ev = nullptr; }
    if (b->ev_done) cudaEventDestroy(b->ev_done);
    b->ev_done = nullptr;
    b->host_ready = false;
}

int alloc_host_step(mv_batch *b) {
    const size_t px = (size_t)b->desc.width * b->desc.height;
    const size_t O = (size_t)b->num_obs, E = (size_t)b->desc.num_envs;
    cudaError_t e = cudaMalloc(&b->d_rgb, O * px * 3);
    if (e == cudaSuccess) e = cudaMalloc(&b->d_depth, O * px * 4);
    if (e == cudaSuccess) e = cudaMalloc(&b->d_cam_in, O * sizeof(mv_camera));
    if (e == cudaSuccess && b->desc.max_boxes > 0) {
        e = cudaMalloc(&b->d_box_in, E * b->desc.max_boxes * sizeof(mv_box));
        if (e == cudaSuccess) e = cudaMalloc(&b->d_count_in, E * sizeof(int32_t));
    }
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&b->copy_stream, cudaStreamNonBlocking);
    for (auto &ev : b->ev_chunk)
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->ev_done, cudaEventDisableTiming);
    if (e != cudaSuccess) {
        free_host_step(b);
        cudaGetLastError();
        return cuda_fail(b, e);
    }
    b->host_ready = true;
    return MV_OK;
}

// End of a synchronous host step: wait for the stream, then report a staging wait that ran out
// (the frames of such a step are not valid).
int finish_host_step(mv_batch *b, cudaStream_t s) {
    uint32_t word = 0;
    MV_CUDA(b, cudaMemcpyAsync(&word, b->d_status, 4, cudaMemcpyDeviceToHost, s));
    MV_CUDA(b, cudaStreamSynchronize(s));
    return (word & kFlagTimeout) ? MV_ERR_DEVICE_TIMEOUT : MV_OK;
}

}  // namespace

// ---- fixed scratch for mv_step_host_static -------------------------------------------------
// Lives in the library image: every GPU that loads the library holds these bytes until the
// process exits.  In host code the array's name is only a host-side stand-in, never a device
// address; the address a kernel or a copy may use comes from cudaGetSymbolAddress, taken once
// per device with that device current.
#define MV_STATIC_SCRATCH_BYTES (8u << 20)
static __device__ __align__(256) unsigned char g_static_scratch[MV_STATIC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
unsigned char *g_static_scratch_ptr[kMaxDevices] = {};

// Device address of the scratch array on `device` (which must be current).  First use on a
// device asks the runtime for the symbol's address; later uses return the cached pointer.
int static_scratch_for_device(mv_batch *b, int device, unsigned char **out) {
    if (device < 0 || device >= kMaxDevices) return MV_ERR_UNSUPPORTED;
    if (!g_static_scratch_ptr[device]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess || !p) return cuda_fail(b, e);
        g_static_scratch_ptr[device] = static_cast<unsigned char *>(p);
    }
    *out = g_static_scratch_ptr[device];
    return MV_OK;
}
}  // namespace

namespace {
// Checks a scene descriptor and spells it out for the kernels.
bool scene_args(const mv_scene_desc *d, const int64_t *d_env_ids, int env_count, SceneArgs *a) {
    auto dim_ok = [](int g) { return g >= 4 && g <= 1024 && (g % 4) == 0; };
    if (!d || !d_env_ids || env_count < 0 || d->world < 0 || d->world > 2 || !dim_ok(d->grid_x) || !dim_ok(d->grid_y) ||
        !dim_ok(d->grid_z) || d->palette_size < 1 || d->palette_size > 256 || d->count < 0 || d->count > (d->world == 1 ? 1024 : 1 << 24) ||
        d->line_pitch < 0 || d->line_pitch > 1024 || d->pillars < 0 || d->pillars > 1 << 24 || d->agents < 1 || d->agents > 1 << 16 ||
        d->movable_boxes < 0 || d->movable_boxes > 1 << 16 || d->step < 0 ||
        (int64_t)env_count * d->grid_x * d->grid_z / 4 > (1ll << 38) || (int64_t)env_count * (d->world == 1 ? 1 : d->count) > (1ll << 38))
        return false;
    *a = SceneArgs{};
    a->seed = d->seed; a->world = d->world; a->gx = d->grid_x; a->gy = d->grid_y; a->gz = d->grid_z; a->palette = d->palette_size;
    a->count = d->count; a->pitch = d->line_pitch; a->pillars = d->pillars; a->agents = d->agents; a->boxes = d->movable_boxes;
    a->bodies = d->body_boxes ? 1 : 0; a->max_boxes = d->movable_boxes + (d->body_boxes ? d->agents : 0); a->step = d->step;
    a->cam_y_is_fixed = d->cam_y_is_fixed ? 1 : 0; a->cam_y = d->cam_y; a->env_count = env_count; a->env = d_env_ids;
    return true;
}

// A cell for every agent's camera?  (Cells that nobody can stand in are dealt out last.)
bool cameras_fit(const SceneArgs &a) { return a.agents <= a.gx * a.gz; }

size_t ctas_of(size_t threads, int per_cta) { return (threads + per_cta - 1) / per_cta; }

// Height and material of every column, as keys.
cudaError_t launch_scene_keys(const SceneArgs &a, unsigned long long *keys, cudaStream_t s) {
    if (a.world == kWorldRooms) {
        scene_rooms_kernel<<<a.env_count, kSceneThreads, (4 * (size_t)a.count + a.gx + a.gz) * 4, s>>>(a, keys);
    } else {
        const cudaError_t e = cudaMemsetAsync(keys, 0, (size_t)a.env_count * a.gx * a.gz * 8, s);
        if (e != cudaSuccess) return e;
        if (a.count > 0) scene_rects_kernel<<<(unsigned)ctas_of((size_t)a.env_count * a.count, kSceneThreads), kSceneThreads, 0, s>>>(a, keys);
    }
    return cudaGetLastError();
}

// A list of destination environments has to be strictly increasing: in range and no environment written twice.
bool index_ok(const mv_batch *b, const int32_t *h_env_index, int env_count) {
    for (int i = 0; i < env_count; ++i)
        if (h_env_index[i] < 0 || h_env_index[i] >= b->desc.num_envs || (i > 0 && h_env_index[i] <= h_env_index[i - 1])) return false;
    return true;
}

// Notes that an environment has its grid (or its palette).
void mark(std::vector<uint8_t> &has, int &missing, int env) {
    if (!has[env]) { has[env] = 1; missing--; }
}

// Body of both upload entry points.  h_env_index: null for the contiguous range that starts at
// env_begin, else the (validated) destination env of each uploaded env.
int upload_worlds(mv_batch *b, int env_begin, const int32_t *h_env_index, int env_count, const uint8_t *d_grid,
                  const mv_box *d_boxes, const int32_t *d_box_count, const uint8_t *d_palette, cudaStream_t s) {
    if (d_boxes && !d_box_count) return MV_ERR_INVALID_ARG;
    if (d_boxes && b->desc.max_boxes == 0) return MV_ERR_INVALID_ARG;
    if ((d_grid && !aligned16(d_grid)) || (d_boxes && !aligned16(d_boxes))) return MV_ERR_INVALID_ARG;
    if (env_count == 0) return MV_OK;
    DeviceGuard g(b->desc.device);
    if (!g.ok) return MV_ERR_CUDA;
    const int32_t *d_index = nullptr;
    if (h_env_index) {
        // The list is copied in stream order into a buffer the batch owns; an earlier scattered upload
        // on another stream that has not finished would be overwritten (one stream at a time).
        MV_CUDA(b, cudaMemcpyAsync(b->d_env_index, h_env_index, (size_t)env_count * 4, cudaMemcpyHostToDevice, s));
        d_index = b->d_env_index;
    }
    int r = launch_upload(b, env_begin, d_index, env_count, d_grid, d_boxes, d_box_count, d_palette, s);
    if (r != MV_OK) return r;
    // (once every env has a grid and a palette there is nothing left to track)
    for (int i = 0; i < env_count && ((d_grid && b->missing_grid > 0) || (d_palette && b->missing_palette > 0)); ++i) {
        const int e = h_env_index ? h_env_index[i] : env_begin + i;
        if (d_grid) mark(b->has_grid, b->missing_grid, e);
        if (d_palette) mark(b->has_palette, b->missing_palette, e);
    }
    return MV_OK;
}
}  // namespace

extern "C" {

const char *mv_status_string(int status) {
    switch (status) {
        case MV_OK: return "ok";
        case MV_ERR_INVALID_ARG: return "invalid argument";
        case MV_ERR_OUT_OF_MEMORY: return "out of memory";
        case MV_ERR_CUDA: return "CUDA runtime error";
        case MV_ERR_NOT_READY: return "worlds or cameras not uploaded yet";
        case MV_ERR_DEVICE_TIMEOUT: return "device-side wait timed out";
        case MV_ERR_UNSUPPORTED: return "configuration exceeds a documented limit";
        default: return status > 0 ? "data-error flags set" : "unknown status";
    }
}

int mv_create_batch(const mv_batch_desc *desc, mv_batch **out) {
    if (!desc || !out) return MV_ERR_INVALID_ARG;
    *out = nullptr;
    const mv_batch_desc &d = *desc;
    auto dim_ok = [](int g) { return g >= 4 && g <= 1024 && (g % 4) == 0; };
    if (d.num_envs < 1 || d.agents_per_env < 1 || !dim_ok(d.grid_x) || !dim_ok(d.grid_y) || !dim_ok(d.grid_z) ||
        d.max_boxes < 0 || d.max_boxes > 256 || d.width < 8 || d.width > 4096 || (d.width % 8) != 0 ||
        d.height < 4 || d.height > 4096 || (d.height % 4) != 0 || d.palette_size < 1 || d.palette_size > 256 ||
        !(d.hfov_rad > 0.0f) || !(d.hfov_rad < 3.14159f) || !(d.ambient >= 0.0f) || !(d.ambient <= 1.0f) ||
        !std::isfinite(d.miss_depth) || d.device < 0 || d.max_overlay_rects < 0 || d.max_overlay_rects > 16)
        return MV_ERR_INVALID_ARG;
    const double ln = (double)d.light_dir[0] * d.light_dir[0] + (double)d.light_dir[1] * d.light_dir[1] +
                      (double)d.light_dir[2] * d.light_dir[2];
    if (!(ln > 0.0) || !std::isfinite(ln)) return MV_ERR_INVALID_ARG;
    if ((int64_t)d.num_envs * d.agents_per_env > (1 << 30)) return MV_ERR_INVALID_ARG;

    mv_batch *b = new (std::nothrow) mv_batch();
    if (!b) return MV_ERR_OUT_OF_MEMORY;
    b->desc = d;
    b->num_obs = d.num_envs * d.agents_per_env;
    b->has_grid.assign(d.num_envs, 0);
    b->has_palette.assign(d.num_envs, 0);
    b->missing_grid = b->missing_palette = d.num_envs;

    EnvLayout &L = b->lay;
    L.ysh = 5;                                              // material bytes per (x, z) column: a power of two >= grid_y, >= 32
    while ((1 << L.ysh) < d.grid_y) L.ysh++;
    L.pitch = (uint32_t)d.grid_x + 1;
    L.origin = L.pitch + 1;                                 // a fence row, and the fence column before x = 0
    const size_t columns = (size_t)L.pitch * (d.grid_z + 2) + 1;
    L.planes = d.grid_y <= 32 ? 1 : (uint32_t)((d.grid_y + kPlaneHeights - 1) / kPlaneHeights);
    L.occ_plane = round_up((uint32_t)columns * 4, 16);
    L.occ_bytes = L.planes * L.occ_plane;
    b->mat_bytes_per_env = (columns << L.ysh);
    L.lut_off = L.occ_bytes;
    L.box_off = L.lut_off + round_up(kFaces * d.palette_size * 4, 16);
    L.count_off = L.box_off + (uint32_t)d.max_boxes * 32;
    L.block_bytes = L.count_off + 32;
    L.stride = round_up(L.block_bytes, 128);

    b->tiles_x = d.width / 8;
    b->tiles_y = d.height / 4;
    // a bit per box, and one behind them for "a GUI rectangle touches the tile"
    b->mask_words = (d.max_boxes + (d.max_overlay_rects > 0 ? 1 : 0) + 31) / 32;
    if (b->mask_words < 1) b->mask_words = 1;

    // kr = tan(hfov/2)/W, ku = (tan(hfov/2)*H/W)/H in double (scalar set-up for the camera kernel)
    const double tx = std::tan((double)d.hfov_rad / 2.0);
    const double ty = tx * (double)d.height / (double)d.width;
    b->kr = tx / (double)d.width;
    b->ku = ty / (double)d.height;
    b->sky_rgbx = (uint32_t)d.sky_rgb[0] | ((uint32_t)d.sky_rgb[1] << 8) | ((uint32_t)d.sky_rgb[2] << 16);

    int ndev = 0;
    cudaError_t e = cudaGetDeviceCount(&ndev);
    if (e != cudaSuccess || d.device >= ndev) { delete b; return e != cudaSuccess ? MV_ERR_CUDA : MV_ERR_INVALID_ARG; }
    DeviceGuard g(d.device);
    if (!g.ok) { delete b; return MV_ERR_CUDA; }
    int smem_max = 0, sms = 0;
    e = cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, d.device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, d.device);
    if (e != cudaSuccess) { delete b; return MV_ERR_CUDA; }
    b->smem_max = smem_max;
    b->sms = sms;
    e = cudaDeviceGetAttribute(&b->smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, d.device);
    if (e != cudaSuccess) { delete b; return MV_ERR_CUDA; }
    // The occupancy normally rides in shared memory with the rest of the env block.  It stays in global memory where it does not
    // fit, and where staging it would leave one CTA on an SM, reading it would leave three, and there are more observations than
    // those hold at once: of such a grid the rays see a small part, which the cache holds, and with one CTA nobody works while
    // the next block is staged.  Up to then the parts of an observation are staged side by side.  In us, staged / from global memory:
    //   192x32x192  rooms 148: 25.7 / 24.2   300: 38.1 / 41.0   512: 64.5 / 54.5   2048: 216 / 183   columns 26.9 / 38.9   43.8 / 59.0   69.8 / 77.7   223 / 217
    //   128x48x128  rooms 148: 23.2 / 23.2   300: 36.2 / 34.3   512: 60.3 / 47.2   2048: 201 / 146   columns 31.6 / 37.5   53.1 / 50.8   65.3 / 73.6   238 / 190
    //   148x56x112  rooms 148: 26.6 / 21.8   300: 39.6 / 33.3   444: 50.9 / 55.3   512: 62.5 / 55.4   columns 32.5 / 38.8   46.7 / 48.5   62.0 / 66.2   71.5 / 70.0
    // (These again and again with nothing in between.  After other work 192x32x192 rooms take 33.8 / 33.7, 48.2 / 52.1, 70.7 / 68.7, 222 / 188, but columns,
    // whose rays look far, 34.0 / 59.7, 54.3 / 79.7, 74.8 / 116, 228 / 222.)
    // Where the tables of a large image leave room for one either way, staged is 13 to 33 % faster for any number (640x360 on 64x16x64
    // rooms, 300: 474 / 555), and no slower where they leave two (480x272 on 96x32x96 rooms, 300: 344 / 369, 1000: 1030 / 1024).
    const auto room = [&](bool staged) { return (int64_t)b->smem_sm / ((int64_t)smem_layout(b, 1, staged).bytes + 1024); };   // (CTAs on an SM)
    b->want_occ_shared = room(true) > 1 || room(false) < 3 || b->num_obs <= 3 * sms;
    b->occ_shared = b->want_occ_shared && fits_staged(b, 1);
    b->smem = smem_layout(b, 1, b->occ_shared);
    if ((int64_t)b->smem.bytes > smem_max) { delete b; return MV_ERR_UNSUPPORTED; }
    // The dynamic shared-memory cap is a property of the kernel function on this device, shared by
    // every batch: raise it to the device's maximum once, never to one batch's own size.
    for (int threads : {kRenderThreadsSmall, kRenderThreads, kRenderThreadsTwo})
        for (RenderFn f : {render_fn(b, threads, true), render_fn(b, threads, false)})
            if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(upload_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kUploadSmem);
    if (e != cudaSuccess) { delete b; return MV_ERR_CUDA; }
    b->prefetch = prefetch_pays(b);
    // A CTA per environment (block staged once for all its agents) or per observation, whichever is expected to take less.
    int shape = choose_shape(b, 1);
    if (shape == MV_OK && d.agents_per_env > 1 && (int64_t)smem_layout(b, d.agents_per_env, b->occ_shared).bytes <= smem_max) {   // (never give up staged occupancy for it)
        double one, all;
        pick_split(b, b->num_obs, &one);
        shape = choose_shape(b, d.agents_per_env);
        const bool whole = pick_split(b, b->num_obs, &all).whole > 0;      // (where all goes in parts there is nothing to share)
        if (shape == MV_OK && whole && all < one) b->auto_agents_per_cta = d.agents_per_env;
        else shape = choose_shape(b, 1);
    }
    if (shape != MV_OK) { delete b; return shape; }

    const size_t blocks_bytes = (size_t)d.num_envs * L.stride;
    bool ok = cudaMalloc(&b->d_env_blocks, blocks_bytes) == cudaSuccess &&
              cudaMalloc(&b->d_mat, (size_t)d.num_envs * b->mat_bytes_per_env) == cudaSuccess &&
              cudaMalloc(&b->d_cams, (size_t)b->num_obs * sizeof(CamRec)) == cudaSuccess &&
              cudaMalloc(&b->d_status, 16) == cudaSuccess &&
              cudaMalloc(&b->d_acc, (size_t)d.num_envs * kPackAccInts * 4) == cudaSuccess &&
              cudaMalloc(&b->d_env_index, (size_t)d.num_envs * 4) == cudaSuccess;
    if (ok && d.max_overlay_rects > 0)
        ok = cudaMalloc(&b->d_overlay, (size_t)b->num_obs * d.max_overlay_rects * 16) == cudaSuccess &&
             cudaMalloc(&b->d_overlay_count, (size_t)b->num_obs * 4) == cudaSuccess &&
             cudaMemset(b->d_overlay_count, 0, (size_t)b->num_obs * 4) == cudaSuccess;
    if (ok) ok = cudaMemset(b->d_env_blocks, 0, blocks_bytes) == cudaSuccess &&
                 cudaMemset(b->d_status, 0, 16) == cudaSuccess;
    if (ok) {
        const int n = d.num_envs * kPackAccInts;
        init_acc_kernel<<<(n + 255) / 256, 256>>>(b->d_acc, n);
        const size_t words = (size_t)d.num_envs * (L.occ_bytes / 4);
        fence_kernel<<<(unsigned)((words + 255) / 256), 256>>>(b->d_env_blocks, L, d.grid_x, d.grid_z, d.num_envs);
        ok = cudaGetLastError() == cudaSuccess && cudaStreamSynchronize(0) == cudaSuccess;
    }
    if (!ok) {
        cudaGetLastError();
        mv_destroy(b);
        return MV_ERR_OUT_OF_MEMORY;
    }
    *out = b;
    return MV_OK;
}

int mv_upload_worlds(mv_batch *b, int env_begin, int env_count, const uint8_t *d_grid, const mv_box *d_boxes,
                     const int32_t *d_box_count, const uint8_t *d_palette, void *cuda_stream) {
    if (!b || env_begin < 0 || env_count < 0 || (int64_t)env_begin + env_count > b->desc.num_envs)
        return MV_ERR_INVALID_ARG;
    return upload_worlds(b, env_begin, nullptr, env_count, d_grid, d_boxes, d_box_count, d_palette,
                         static_cast<cudaStream_t>(cuda_stream));
}

int mv_upload_worlds_at(mv_batch *b, int env_count, const int32_t *h_env_index, const uint8_t *d_grid,
                        const mv_box *d_boxes, const int32_t *d_box_count, const uint8_t *d_palette,
                        void *cuda_stream) {
    if (!b || env_count < 0 || env_count > b->desc.num_envs || (env_count > 0 && !h_env_index))
        return MV_ERR_INVALID_ARG;
    if (!index_ok(b, h_env_index, env_count)) return MV_ERR_INVALID_ARG;
    return upload_worlds(b, 0, h_env_index, env_count, d_grid, d_boxes, d_box_count, d_palette,
                         static_cast<cudaStream_t>(cuda_stream));
}

int mv_set_cameras(mv_batch *b, const mv_camera *d_cams, void *cuda_stream) {
    if (!b || !d_cams) return MV_ERR_INVALID_ARG;
    DeviceGuard g(b->desc.device);
    if (!g.ok) return MV_ERR_CUDA;
    return launch_cameras(b, d_cams, static_cast<cudaStream_t>(cuda_stream));
}

int mv_set_overlays(mv_batch *b, const mv_overlay_rect *d_rects, const int32_t *d_count, void *cuda_stream) {
    if (!b || (d_rects && !d_count)) return MV_ERR_INVALID_ARG;
    const int m = b->desc.max_overlay_rects;
    if (m == 0) return d_rects ? MV_ERR_INVALID_ARG : MV_OK;
    if (d_rects && !aligned16(d_rects)) return MV_ERR_INVALID_ARG;
    DeviceGuard g(b->desc.device);
    if (!g.ok) return MV_ERR_CUDA;
    const int64_t n = (int64_t)b->num_obs * (m + 1);
    MV_CUDA(b, launch_step(copy_overlays_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, static_cast<cudaStream_t>(cuda_stream),
                           reinterpret_cast<const int4 *>(d_rects), d_count, b->d_overlay, b->d_overlay_count, b->num_obs, m));
    b->launches++;
    return MV_OK;
}

int mv_move_agents(mv_batch *b, mv_camera *d_cams_inout, const mv_agent_move *d_moves, const mv_body_shape *shape,
                   void *cuda_stream) {
    if (!b || !d_cams_inout || !d_moves || !aligned16(d_moves)) return MV_ERR_INVALID_ARG;
    mv_body_shape sh = {0.25f, 0.75f, 0.25f, 1.0f};
    if (shape) sh = *shape;
    if (!(sh.half_width >= 0.0f) || !(sh.below_eye >= 0.0f) || !(sh.above_eye >= 0.0f) || !(sh.max_pitch >= 0.0f) ||
        !(sh.half_width < 16.0f) || !(sh.below_eye < 16.0f) || !(sh.above_eye < 16.0f))
        return MV_ERR_INVALID_ARG;
    if (b->missing_grid > 0) return MV_ERR_NOT_READY;
    DeviceGuard g(b->desc.device);
    if (!g.ok) return MV_ERR_CUDA;
    const int n = b->num_obs;
    MV_CUDA(b, launch_step(move_agents_kernel, dim3((n + 127) / 128), dim3(128), 0, static_cast<cudaStream_t>(cuda_stream),
                           reinterpret_cast<int32_t *>(d_cams_inout), reinterpret_cast<const float4 *>(d_moves), b->d_cams, b->d_env_blocks,
                           b->lay, n, b->desc.agents_per_env, b->desc.grid_x, b->desc.grid_y, b->desc.grid_z, b->desc.max_boxes,
                           sh.half_width, sh.below_eye, sh.above_eye, sh.max_pitch, b->kr, b->ku, b->d_status));
    b->launches++;
    b->has_cams = true;
    return MV_OK;
}

int mv_merge_voxels(mv_batch *b, int env_begin, int env_count, mv_box *d_boxes_out, int32_t *d_count_out,
                    int max_out, void *cuda_stream) {
    if (!b || env_begin < 0 || env_count < 0 || (int64_t)env_begin + env_count > b->desc.num_envs || !d_boxes_out ||
        !d_count_out || max_out < 1 || !aligned16(d_boxes_out))
        return MV_ERR_INVALID_ARG;
    for (int e = env_begin; e < env_begin + env_count; ++e)
        if (!b->has_grid[e]) return MV_ERR_NOT_READY;
    if (env_count == 0) return MV_OK;
    DeviceGuard g(b->desc.device);
    if (!g.ok) return MV_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    if (!b->d_merge) {
        const mv_batch_desc &d = b->desc;
        MergeLayout ml{};
        ml.gx = d.grid_x; ml.gy = d.grid_y; ml.gz = d.grid_z;
        ml.mat_stride = b->mat_bytes_per_env;
        ml.W = (d.grid_x + 31) / 32;
        ml.colw = 1 << (b->lay.ysh - 5);
        ml.mask_words = (uint32_t)d.grid_y * d.grid_z * ml.W;
        ml.slots = ml.W + 1;
        ml.work_bytes = (uint32_t)d.grid_z * ml.slots * 16 + (uint32_t)d.grid_x * d.grid_z * (d.grid_y < 256 ? 1 : 2);
        ml.work_off = (3 * ml.mask_words + (uint32_t)d.grid_x * d.grid_z * ml.colw + 3) / 4 * 4;
        cudaFuncAttributes fa{};
        const void *sweep = (const void *)merge_sweep(d.grid_y, ml.W);
        MV_CUDA(b, cudaFuncGetAttributes(&fa, sweep));
        ml.work_in_smem = ml.work_bytes + fa.sharedSizeBytes <= (size_t)b->smem_max;
        if (ml.work_in_smem)       // (to the device's maximum: the cap belongs to the function, not to this batch)
            MV_CUDA(b, cudaFuncSetAttribute(sweep, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            b->smem_max - (int)fa.sharedSizeBytes));
        ml.env_words = ((size_t)ml.work_off + (ml.work_in_smem ? 0 : ml.work_bytes / 4) + 3) / 4 * 4;
        size_t chunk = kMergeScratchBytes / (ml.env_words * 4);
        chunk = chunk < 1 ? 1 : (chunk > (size_t)d.num_envs ? (size_t)d.num_envs : chunk);
        MV_CUDA(b, cudaMalloc(&b->d_merge, chunk * ml.env_words * 4));
        b->merge = ml;
        b->merge_chunk = (int)chunk;
    }
    const MergeLayout &ml = b->merge;
    const int per_env = (ml.W + 3) / 4 * ((ml.gz + 7) / 8) * ml.colw;
    for (int e0 = 0; e0 < env_count; e0 += b->merge_chunk) {
        const int n = env_count - e0 < b->merge_chunk ? env_count - e0 : b->merge_chunk;
        (b->lay.planes > 1 ? merge_masks_kernel<true> : merge_masks_kernel<false>)<<<(unsigned)n * per_env, kMergeThreads, 0, s>>>(b->d_env_blocks, b->d_mat, b->lay, ml,
                                                                          env_begin + e0, b->d_merge);
        b->launches++;
        MV_CUDA(b, cudaGetLastError());
        merge_sweep(b->desc.grid_y, ml.W)<<<n, kMergeThreads, ml.work_in_smem ? ml.work_bytes : 0, s>>>(
            b->d_env_blocks, b->d_mat, b->lay, ml, env_begin + e0, b->d_merge,
            reinterpret_cast<uint4 *>(d_boxes_out + (size_t)e0 * max_out), d_count_out + e0, max_out);
        b->launches++;
        MV_CUDA(b, cudaGetLastError());
    }
    return MV_OK;
}

int mv_render_batch(mv_batch *b, uint8_t *d_rgb, float *d_depth, void *cuda_stream) {
    if (!b || !d_rgb || !d_depth || !aligned16(d_rgb) || !aligned16(d_depth)) return MV_ERR_INVALID_ARG;
    if (b->missing_grid > 0 || b->missing_palette > 0 || !b->has_cams) return MV_ERR_NOT_READY;
    DeviceGuard g(b->desc.device);
    if (!g.ok) return MV_ERR_CUDA;
    return launch_render(b, d_rgb, d_depth, 0, b->num_obs, static_cast<cudaStream_t>(cuda_stream));
}

int mv_step_host(mv_batch *b, const mv_camera *h_cams, const mv_box *h_boxes, const int32_t *h_box_count,
                 uint8_t *h_rgb, float *h_depth, void *cuda_stream) {
    if (!b || !h_cams || !h_rgb || !h_depth) return MV_ERR_INVALID_ARG;
    if (h_boxes && (!h_box_count || b->desc.max_boxes == 0)) return MV_ERR_INVALID_ARG;
    if (b->missing_grid > 0 || b->missing_palette > 0) return MV_ERR_NOT_READY;
    DeviceGuard g(b->desc.device);
    if (!g.ok) return MV_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    const size_t px = (size_t)b->desc.width * b->desc.height;
    const int E = b->desc.num_envs, O = b->num_obs;
    if (!b->host_ready) {
        int r = alloc_host_step(b);
        if (r != MV_OK) return r;
    }
    MV_CUDA(b, cudaMemcpyAsync(b->d_cam_in, h_cams, (size_t)O * sizeof(mv_camera), cudaMemcpyHostToDevice, s));
    if (h_boxes) {
        MV_CUDA(b, cudaMemcpyAsync(b->d_box_in, h_boxes, (size_t)E * b->desc.max_boxes * sizeof(mv_box),
                                   cudaMemcpyHostToDevice, s));
        MV_CUDA(b, cudaMemcpyAsync(b->d_count_in, h_box_count, (size_t)E * sizeof(int32_t), cudaMemcpyHostToDevice, s));
        int r = launch_upload(b, 0, nullptr, E, nullptr, b->d_box_in, b->d_count_in, nullptr, s);
        if (r != MV_OK) return r;
    }
    int r = launch_cameras(b, b->d_cam_in, s);
    if (r != MV_OK) return r;
    // render chunk by chunk; each chunk's frames start their trip to the host while the next renders
    // (chunks are whole environments, as the render launch wants when one CTA renders an env)
    const int A = b->desc.agents_per_env;
    const int chunks = E < kHostChunks ? 1 : kHostChunks;
    for (int c = 0; c < chunks; ++c) {
        const int o0 = (int)((int64_t)E * c / chunks) * A, o1 = (int)((int64_t)E * (c + 1) / chunks) * A;
        r = launch_render(b, b->d_rgb, b->d_depth, o0, o1 - o0, s);
        if (r != MV_OK) return r;
        MV_CUDA(b, cudaEventRecord(b->ev_chunk[c], s));
        MV_CUDA(b, cudaStreamWaitEvent(b->copy_stream, b->ev_chunk[c], 0));
        MV_CUDA(b, cudaMemcpyAsync(h_rgb + (size_t)o0 * px * 3, b->d_rgb + (size_t)o0 * px * 3,
                                   (size_t)(o1 - o0) * px * 3, cudaMemcpyDeviceToHost, b->copy_stream));
        MV_CUDA(b, cudaMemcpyAsync(h_depth + (size_t)o0 * px, b->d_depth + (size_t)o0 * px,
                                   (size_t)(o1 - o0) * px * 4, cudaMemcpyDeviceToHost, b->copy_stream));
    }
    MV_CUDA(b, cudaEventRecord(b->ev_done, b->copy_stream));
    MV_CUDA(b, cudaStreamWaitEvent(s, b->ev_done, 0));
    return finish_host_step(b, s);
}

int mv_step_host_static(mv_batch *b, const mv_camera *h_cams, uint8_t *h_rgb, float *h_depth,
                        void *cuda_stream) {
    if (!b || !h_cams || !h_rgb || !h_depth) return MV_ERR_INVALID_ARG;
    if (b->missing_grid > 0 || b->missing_palette > 0) return MV_ERR_NOT_READY;
    const size_t px = (size_t)b->desc.width * b->desc.height;
    const size_t O = (size_t)b->num_obs;
    // layout inside the scratch array: depth | rgb | cameras, each 256-byte aligned
    const size_t depth_bytes = (O * px * 4 + 255) / 256 * 256;
    const size_t rgb_bytes = (O * px * 3 + 255) / 256 * 256;
    const size_t cam_bytes = O * sizeof(mv_camera);
    if (depth_bytes + rgb_bytes + cam_bytes > (size_t)MV_STATIC_SCRATCH_BYTES) return MV_ERR_UNSUPPORTED;
    DeviceGuard g(b->desc.device);
    if (!g.ok) return MV_ERR_CUDA;
    unsigned char *scratch = nullptr;
    int r = static_scratch_for_device(b, b->desc.device, &scratch);
    if (r != MV_OK) return r;
    float *d_depth = reinterpret_cast<float *>(scratch);
    uint8_t *d_rgb = scratch + depth_bytes;
    mv_camera *d_cams = reinterpret_cast<mv_camera *>(scratch + depth_bytes + rgb_bytes);
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    // nothing in the scratch has to start at zero: the cameras are overwritten by the copy
    // below and the render kernel writes every byte of both frame buffers
    MV_CUDA(b, cudaMemcpyAsync(d_cams, h_cams, cam_bytes, cudaMemcpyHostToDevice, s));
    r = launch_cameras(b, d_cams, s);
    if (r != MV_OK) return r;
    r = launch_render(b, d_rgb, d_depth, 0, b->num_obs, s);
    if (r != MV_OK) return r;
    MV_CUDA(b, cudaMemcpyAsync(h_rgb, d_rgb, O * px * 3, cudaMemcpyDeviceToHost, s));
    MV_CUDA(b, cudaMemcpyAsync(h_depth, d_depth, O * px * 4, cudaMemcpyDeviceToHost, s));
    return finish_host_step(b, s);
}

int mv_scene_worlds(const mv_scene_desc *desc, const int64_t *d_env_ids, int env_count, uint8_t *d_grid,
                    uint8_t *d_palette, int64_t *d_height, int device, void *cuda_stream) {
    SceneArgs a;
    if (!scene_args(desc, d_env_ids, env_count, &a) || !d_grid || !d_palette || !d_height || !aligned16(d_height) || !aligned16(d_grid))
        return MV_ERR_INVALID_ARG;
    if (env_count == 0) return MV_OK;
    DeviceGuard g(device);
    if (!g.ok) return MV_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    const size_t cells = (size_t)a.gx * a.gz;
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(d_height);
    MV_CUDA(nullptr, launch_scene_keys(a, keys, s));
    const size_t columns = ctas_of(env_count * cells / 4, kSceneThreads), colours = ctas_of((size_t)env_count * 3 * a.palette, kSceneThreads);
    scene_expand_kernel<<<(unsigned)(columns + colours), kSceneThreads, 0, s>>>(a, keys, d_grid, d_palette, (long long)columns);
    MV_CUDA(nullptr, cudaGetLastError());
    return MV_OK;
}

int mv_scene_entities(const mv_scene_desc *desc, const int64_t *d_env_ids, int env_count, const int64_t *d_height,
                      const int32_t *d_slots, mv_box *d_boxes, int32_t *d_box_count, mv_camera *d_cams, int device,
                      void *cuda_stream) {
    SceneArgs a;
    if (!scene_args(desc, d_env_ids, env_count, &a) || !cameras_fit(a) || !d_height || !d_box_count || !d_cams || (a.max_boxes > 0 && !d_boxes))
        return MV_ERR_INVALID_ARG;
    if (env_count == 0) return MV_OK;
    DeviceGuard g(device);
    if (!g.ok) return MV_ERR_CUDA;
    scene_entities_kernel<<<env_count, kEntityThreads, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
        a, reinterpret_cast<const long long *>(d_height), d_slots, reinterpret_cast<uint32_t *>(d_boxes), d_box_count,
        reinterpret_cast<uint32_t *>(d_cams));
    MV_CUDA(nullptr, cudaGetLastError());
    return MV_OK;
}

int mv_scene_upload(mv_batch *b, const mv_scene_desc *desc, const int64_t *d_env_ids, int env_count, const int32_t *h_env_index,
                    mv_camera *d_cams, mv_box *d_boxes, int32_t *d_box_count, uint8_t *d_palette, int64_t *d_work, void *cuda_stream) {
    SceneArgs a;
    if (!b || !scene_args(desc, d_env_ids, env_count, &a) || !cameras_fit(a) || env_count > b->desc.num_envs || (env_count > 0 && !h_env_index) || !d_cams ||
        !d_box_count || !d_palette || !d_work || !aligned16(d_work) || (a.max_boxes > 0 && (!d_boxes || !aligned16(d_boxes))) ||
        a.gx != b->desc.grid_x || a.gy != b->desc.grid_y || a.gz != b->desc.grid_z || a.palette != b->desc.palette_size ||
        a.max_boxes != b->desc.max_boxes || a.agents != b->desc.agents_per_env || !index_ok(b, h_env_index, env_count))
        return MV_ERR_INVALID_ARG;
    if (env_count == 0) return MV_OK;
    DeviceGuard g(b->desc.device);
    if (!g.ok) return MV_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    const size_t columns = ctas_of((size_t)a.gx * a.gz / 4, kEntityThreads), colours = ctas_of((size_t)env_count * 3 * a.palette, kEntityThreads);
    // Few high worlds have few columns and many bytes, more than an SM writes in the time that boxes and cameras take: their heights are dealt to as
    // many CTAs as leave each one an SM of its own (more would share those that place boxes).  64x1024x64, 1 world: 89 -> 25 us (by its arrays
    // and an upload 61), 8: 90 -> 30; 64x256x64, 8: 39 -> 24; from 64 worlds on, and where grids are at most 32 high, nothing changes.
    const int64_t idle = (int64_t)b->sms - (int64_t)(env_count + colours), most = (a.gy + 31) / 32;
    int64_t slabs = idle / (int64_t)(columns * env_count);
    slabs = slabs < 1 ? 1 : slabs > most ? most : slabs;
    const size_t ctas = env_count * (columns * slabs + 1) + colours;
    if (ctas > 0x7fffffffull) return MV_ERR_INVALID_ARG;
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(d_work);
    MV_CUDA(b, cudaMemcpyAsync(b->d_env_index, h_env_index, (size_t)env_count * 4, cudaMemcpyHostToDevice, s));
    MV_CUDA(b, launch_scene_keys(a, keys, s));
    if (a.world == kWorldRooms || a.count > 0) b->launches++;
    const auto populate = slabs > 1 ? scene_populate_kernel<true> : scene_populate_kernel<false>;
    populate<<<(unsigned)ctas, kEntityThreads, 0, s>>>(
        a, keys, b->d_env_index, reinterpret_cast<uint32_t *>(d_boxes), d_box_count, reinterpret_cast<uint32_t *>(d_cams), d_palette, b->d_env_blocks,
        b->d_mat, b->mat_bytes_per_env, b->lay, b->d_acc, (int)columns, (int)slabs, b->d_status);
    MV_CUDA(b, cudaGetLastError());
    b->launches++;
    const int r = launch_upload(b, 0, b->d_env_index, env_count, nullptr, a.max_boxes > 0 ? d_boxes : nullptr, d_box_count, d_palette, s);
    if (r != MV_OK) return r;
    for (int i = 0; i < env_count && (b->missing_grid > 0 || b->missing_palette > 0); ++i) {
        mark(b->has_grid, b->missing_grid, h_env_index[i]);
        mark(b->has_palette, b->missing_palette, h_env_index[i]);
    }
    return MV_OK;
}

int mv_advance_episodes(mv_batch *b, int64_t *d_t, int64_t *d_episode, const int64_t *d_length, uint8_t *d_done, int advance,
                        int bar_rows, const uint8_t *bar_rgb, void *cuda_stream) {
    if (!b || !d_t || !d_episode || !d_length || (advance && !d_done) || bar_rows < 0 || bar_rows > 4096 ||
        (bar_rows > 0 && (!bar_rgb || b->desc.max_overlay_rects == 0)))
        return MV_ERR_INVALID_ARG;
    DeviceGuard g(b->desc.device);
    if (!g.ok) return MV_ERR_CUDA;
    const uint32_t rgb = bar_rows > 0 ? (uint32_t)bar_rgb[0] | (uint32_t)bar_rgb[1] << 8 | (uint32_t)bar_rgb[2] << 16 : 0u;
    episode_clocks_kernel<<<(b->desc.num_envs + 127) / 128, 128, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
        d_t, d_episode, d_length, d_done, b->desc.num_envs, b->desc.agents_per_env, advance ? 1 : 0, b->desc.width, bar_rows, rgb,
        bar_rows > 0 ? b->d_overlay : nullptr, b->d_overlay_count, b->desc.max_overlay_rects);
    b->launches++;
    MV_CUDA(b, cudaGetLastError());
    return MV_OK;
}

int mv_query_status(mv_batch *b, int clear, void *cuda_stream) {
    if (!b) return MV_ERR_INVALID_ARG;
    DeviceGuard g(b->desc.device);
    if (!g.ok) return MV_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    uint32_t word = 0;
    MV_CUDA(b, cudaMemcpyAsync(&word, b->d_status, 4, cudaMemcpyDeviceToHost, s));
    if (clear) MV_CUDA(b, cudaMemsetAsync(b->d_status, 0, 4, s));
    MV_CUDA(b, cudaStreamSynchronize(s));
    if (word & kFlagTimeout) return MV_ERR_DEVICE_TIMEOUT;
    return (int)word;
}

int64_t mv_launch_count(const mv_batch *b) { return b ? b->launches : 0; }

int mv_debug_occupancy_in_global(mv_batch *b, int on) {
    if (!b) return MV_ERR_INVALID_ARG;
    if (on < 0) return b->occ_shared ? 0 : 1;
    if (!on && !fits_staged(b, b->agents_per_cta)) return MV_ERR_UNSUPPORTED;
    DeviceGuard g(b->desc.device);
    if (!g.ok) return MV_ERR_CUDA;
    b->want_occ_shared = !on;
    return choose_shape(b, b->agents_per_cta);
}

int mv_debug_prefetch(mv_batch *b, int on) {
    if (!b || on > 2) return MV_ERR_INVALID_ARG;
    if (on >= 0) b->prefetch = on == 2 ? prefetch_pays(b) : on == 1;
    return b->prefetch && !b->occ_shared ? 1 : 0;
}

int mv_debug_parts(mv_batch *b, int parts) {
    if (!b || parts < 0) return MV_ERR_INVALID_ARG;
    b->forced_parts = parts;
    const Split split = pick_split(b, b->num_obs);
    return split.whole > 0 ? 1 : split.parts;
}

int mv_debug_agents_per_cta(mv_batch *b, int agents_per_cta) {
    if (!b) return MV_ERR_INVALID_ARG;
    const int A = b->desc.agents_per_env;
    int apc = agents_per_cta == 0 ? b->auto_agents_per_cta : agents_per_cta;
    if (apc != 1 && apc != A) return MV_ERR_INVALID_ARG;
    DeviceGuard g(b->desc.device);
    if (!g.ok) return MV_ERR_CUDA;
    if ((int64_t)smem_layout(b, apc, false).bytes > b->smem_max) return MV_ERR_UNSUPPORTED;
    const int shape = choose_shape(b, apc);
    if (shape != MV_OK) return shape;
    b->forced_agents = agents_per_cta != 0;
    return (int)pick_split(b, b->num_obs).whole;
}

int mv_debug_staging(mv_batch *b, int skip_staging, int wait_polls) {
    if (!b || wait_polls < 1 || wait_polls > (1 << 24)) return MV_ERR_INVALID_ARG;
    b->skip_staging = skip_staging ? 1 : 0;
    b->wait_polls = wait_polls;
    return MV_OK;
}

int mv_destroy(mv_batch *b) {
    if (!b) return MV_OK;
    int rc = MV_OK;
    {
        DeviceGuard g(b->desc.device);
        if (g.ok) {
            if (cudaDeviceSynchronize() != cudaSuccess) rc = MV_ERR_CUDA;
            cudaFree(b->d_env_blocks); cudaFree(b->d_mat); cudaFree(b->d_cams); cudaFree(b->d_status); cudaFree(b->d_acc);
            cudaFree(b->d_overlay); cudaFree(b->d_overlay_count); cudaFree(b->d_merge); cudaFree(b->d_env_index);
            free_host_step(b);
            cudaGetLastError();
        }
    }
    delete b;
    return rc;
}

}  // extern "C"
