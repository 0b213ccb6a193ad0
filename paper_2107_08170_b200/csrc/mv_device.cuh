// Device-side data layout shared by the pack, camera and render kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace mv {

// Face codes: 0..5 = -x,+x,-y,+y,-z,+z (outward normal), 6 = camera inside the solid.
constexpr int kFaces = 7;
constexpr int kFaceInside = 6;

constexpr uint32_t kFlagMaterial = 0x1u;
constexpr uint32_t kFlagBoxCount = 0x2u;
constexpr uint32_t kFlagBadCamera = 0x4u;
constexpr uint32_t kFlagTimeout = 0x8u;

// Per-observation ray basis written by the camera kernel (64 bytes, one 128-bit lane each).
struct __align__(16) CamRec {
    float P[3], F[3], Rs[3], Us[3];   // eye, unit forward, per-half-pixel right and up steps
    int32_t self_box;
    uint32_t flags;                   // kFlagBadCamera when a component was not finite
    uint32_t pad[2];
};
static_assert(sizeof(CamRec) == 64, "CamRec must be 64 bytes");

// One environment's render inputs, contiguous in HBM so that a single bulk copy stages them
// into shared memory:  [occupancy bits | shade LUT | boxes | box count + occupied bounds].
// Occupancy is packed along y: a word holds the lowest heights of an (x, z) column, a walk along x or z moves by whole words and
// a walk along y stays inside the word.  Grids of up to 32 heights are one plane of such words.  Higher ones are several, 31
// heights each, one plane behind the other: bit 31 of a plane is never a voxel, so a walk up or down that leaves the plane
// meets it (as it meets the fence) and goes on in the next one, and an environment filled only low down needs only its
// lowest planes.  Where the occupancy is not staged as a rule, the planes are the same.
// Materials are a byte per voxel at index u = (column << ysh) | y, 2^ysh >= grid_y, at least 32.
// The grid is fenced in: one column between each row and the next (pitch = grid_x + 1) and a row before the first and
// after the last are all ones, written once when the batch is made, so a walk in x and z that leaves the grid hits
// something at once instead of having to be stopped by a test at every step.
struct EnvLayout {
    uint32_t occ_bytes;     // planes * occ_plane
    uint32_t occ_plane;     // bytes of a plane: (pitch*(grid_z + 2) + 1) words, rounded up to 16
    uint32_t planes;        // 1, or ceil(grid_y / 31) for grids more than 32 high
    uint32_t lut_off;       // 7*palette_size RGBX words
    uint32_t box_off;       // max_boxes * 32 bytes
    uint32_t count_off;     // 32 bytes: {box count, lo x,y,z, hi x,y,z, pad}; [lo, hi) = cell box
                            // that contains every filled voxel (lo > hi when the grid is empty)
    uint32_t block_bytes;   // bytes staged per CTA (multiple of 16)
    uint32_t stride;        // distance between envs in HBM (multiple of 128)
    uint32_t ysh;           // log2 of the material bytes per (x, z) column
    uint32_t pitch, origin; // columns from one row to the next; column of (0, 0)
};

__host__ __device__ __forceinline__ uint32_t column_index(const EnvLayout &lay, int x, int z) {
    return lay.origin + (uint32_t)x + lay.pitch * (uint32_t)z;
}
__host__ __device__ __forceinline__ uint32_t voxel_index(const EnvLayout &lay, int x, int y, int z) {
    return (column_index(lay, x, z) << lay.ysh) | (uint32_t)y;
}

// Plane of height y, and the height at which a plane begins.
constexpr uint32_t kPlaneHeights = 31, kPlaneEnd = 0x80000000u;
__host__ __device__ __forceinline__ uint32_t plane_of(const EnvLayout &lay, int y) { return lay.planes == 1 ? 0u : (uint32_t)y / kPlaneHeights; }
__host__ __device__ __forceinline__ int plane_begin(uint32_t plane) { return (int)(plane * kPlaneHeights); }
// Is the voxel filled, by the occupancy at `occ` (an env block, or what is staged of it)?
__device__ __forceinline__ bool voxel_filled(const EnvLayout &lay, const unsigned char *occ, int x, int y, int z) {
    const uint32_t q = plane_of(lay, y);
    const uint32_t w = *reinterpret_cast<const uint32_t *>(occ + (size_t)q * lay.occ_plane + 4u * column_index(lay, x, z));
    return (w >> (y - plane_begin(q))) & 1u;
}
// Tiles that go to the same CTA when an observation's are shared out: 32 pixels, whose bytes of a row are whole sectors.
constexpr int kPartRun = 4;

struct RenderParams {
    const unsigned char *env_blocks;   // [E] EnvLayout blocks
    const uint8_t *mat;                // [E][mat_stride] material ids by voxel index (clamped at upload)
    size_t mat_stride;
    const CamRec *cams;                // [O]
    uint8_t *rgb;                      // [O][H][W][3]
    float *depth;                      // [O][H][W]
    uint32_t *status;
    EnvLayout lay;
    int obs_begin;
    int agents;
    int max_boxes, palette;
    int W, H, tiles_x, tiles_y, mask_words;
    float inv_W;                       // 1 / W
    uint32_t sky_rgbx;
    float miss_depth;
    int agents_per_cta;                // observations one of the first whole_ctas CTAs renders: 1, or all agents of its env
    unsigned whole_ctas;               // the CTAs behind those render a part of one observation each:
    unsigned parts;                    // every parts-th run of kPartRun tiles of it
    float exit_scale;                  // 1 - (bound on the rounding drift of accumulated crossing times)
    // shared-memory offsets after the staged env block: tile table, per-agent blocks (ray table, camera record,
    // eye-relative boxes, then overlay rectangles and per-tile box masks at the offsets below), barrier and flag words
    uint32_t smem_tile_off, smem_agent_off, smem_misc_off;
    uint32_t agent_stride, agent_ov_off, agent_mask_off;
    const int4 *overlay;               // [O][max_overlay] 16-byte records, or null
    const int32_t *overlay_count;      // [O]
    int max_overlay;
    int wait_polls;                    // bound of the staging wait
    int skip_staging;                  // test hook: the block copy is not issued, so the wait runs out
    int prefetch;                      // occupancy that is read from global memory is asked for in L2
};
// A launch takes the host 0.3 us less with parameters of 20 to 32 bytes beyond a multiple of 64 than with any other size (212 to
// 224: 1.75 us, 208 and 228: 2.05 to 2.1; as measured with driver 580.159), a tenth of a step of the smallest batches.
static_assert(sizeof(RenderParams) % 64 >= 20 && sizeof(RenderParams) % 64 <= 32, "see above");

// Bulk asynchronous copies into shared memory and the barrier that counts their bytes.
__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
// Plain (single-CTA) bulk copy global -> shared, completion counted on an mbarrier.
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait: gives up after `limit` polls instead of spinning forever.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity, int limit) {
    for (int i = 0; i < limit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}
constexpr int kDrainPolls = 1 << 26;               // bound of the wait for a copy known to be in flight

// Programmatic dependent launch.  Every per-step kernel waits for the previous kernel before it touches global memory, and
// every one but the render kernel begins with launch_dependents, which lets the next kernel of the stream that was launched
// with the attribute start once all CTAs of this one run; so launch latency and CTA set-up overlap with what is still
// running, and nothing else changes.  (Nothing starts before the end of a render.)
// A kernel launched like this is alive while the one before it still writes, so none of its global loads may promise
// read-only data: no __ldg or ld.global.nc, and no const __restrict__ parameter, from which the compiler infers one and
// which it may then move across the wait.  Ordinary loads stay behind the wait's memory clobber.
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

}  // namespace mv
