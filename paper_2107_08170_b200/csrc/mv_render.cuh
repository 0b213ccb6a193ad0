// The render kernel: ray generation, grid traversal, box tests, shading and frame store for
// every observation of the batch in one launch (paper Section 3.2, Eq. 2).
//
// The grid's first CTAs render whole observations: one each, or all agents of an environment.  Behind
// them come CTAs that render a part of one observation each: the last observations of a large batch, or
// all of a small one (pick_split in the host code says how many).  A single bulk asynchronous copy
// stages the environment's block (1-bit occupancy grid, shaded colour table, box list) into
// shared memory once for what the CTA renders; while it is in flight the other warps clear the per-tile box
// masks and write the tile table.  Each agent's boxes are then binned to 8x4-pixel screen tiles
// by the bounding rectangle of their projected corners (conservative, so every box that a
// pixel's ray can touch is tested for that pixel).  Tiles are dealt to warps round-robin; each
// lane owns one pixel of the tile: it walks the occupancy grid (packed along y: a column of up to
// 32 voxels is one word) with a predicated 3D-DDA in shared memory, tests the tile's candidate
// boxes with slab tests, looks the colour up in the shaded table and the warp writes 24-byte RGB
// row segments as packed 32-bit words and 32-byte depth row segments.  The common case runs in
// three blocks of PTX (ray set-up + walk, colour, stores); everything rarer is C++ around them.
// The walk is confined to the cell box that holds every filled voxel of the environment (built at
// upload), so rays that leave it stop at once; GUI rectangles, if any, are painted over the colour
// just before the store.
//
// Grids more than 32 high take the same path plane by plane (EnvLayout; a walk changes planes outside its loop): thirteen
// instructions a step where a walk by voxel index takes sixteen, and only the planes that hold anything are copied (4096
// observations of 64x36x64 rooms 260 us, 317 by voxel index; 6005 of 144x64x136 columns 197 and 496).
#pragma once
#include "mv_device.cuh"

namespace mv {

#define kInf (__int_as_float(0x7f800000))
constexpr uint32_t kNoRow = 0xffffffffu;           // "no surface" marker of the traversal

// Reciprocal to 1 ulp in one instruction; every use is inside toleranced intersection arithmetic.
__device__ __forceinline__ float fast_rcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// Makes a value opaque to the optimiser at this point, so that it is held in a register from
// here on instead of being recomputed at every use.
template <typename T> __device__ __forceinline__ void keep(T &v) { asm volatile("" : "+r"(reinterpret_cast<uint32_t &>(v))); }
// The same for the assembler, which would rebuild a cheap value at every use: a shuffle it has to take as it comes.
template <typename T> __device__ __forceinline__ void opaque(T &v, int lane) {
    uint32_t &u = reinterpret_cast<uint32_t &>(v);
    asm volatile("shfl.sync.idx.b32 %0, %0, %1, 31, 0xffffffff;" : "+r"(u) : "r"(lane));
}
// Two products, rounded as one by one, for one issue slot.
__device__ __forceinline__ void mul2(float &p, float &q, float a, float b, float c, float d) {
    asm("{\n .reg .b64 x, y;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n mul.rn.f32x2 x, x, y;\n mov.b64 {%0, %1}, x;\n}"
        : "=f"(p), "=f"(q) : "f"(a), "f"(b), "f"(c), "f"(d));
}
__device__ __forceinline__ float min3f(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float max3f(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// ---------------------------------------------------------------------------------------------
// The DDA loop.  Crossing times accumulate (t += dt) and the exit time handed in is pulled in by
// the rounding drift that can build up, which keeps the walk inside the occupied box; the loop is
// also bounded by a step budget.  One step: t = min(tx,ty,tz); leave when t >= exit time or when
// the cell entered by the previous step is filled (one branch for both); else the axis whose
// crossing time equals t (ties: x, then y, then z) advances.  Two registers alternate as t, so
// that after a hit the time at which the filled cell was entered is still there.
//
// Two flavours of the cell state:
//  * column-word (grids up to 32 voxels high, occupancy in shared memory): the state is the
//    shared-memory address `pos` of the (x, z) column's word and a one-bit mask `bit` of the height;
//    x and z steps add a byte stride to the address, a y step rotates the mask by 1 or 31, and the
//    test is one load and one AND.
//  * planes (any grid, see EnvLayout): the same within a plane, bit 31 counting as filled in every column; a walk that meets it
//    on the way up or down goes on in the next plane (MV_DDA_CROSS).  Where the occupancy is not staged, `pos` is the word's
//    byte offset in the environment's block and the load is a global one.
// Register names used by the macros (declared by the enclosing asm block): tx ty tz dtx dty dtz
// (f32), sx sy sz pos bit guard w a it q (b32), ta tb (f32), px py pz pq ph pf (pred), texit (f32), ag gbase (b64).
#define MV_DDA_HEAD(T, OUT)                          \
    " min.f32 " T ", tx, ty, tz;\n"                  \
    " setp.geu.or.f32 pq, " T ", texit, ph;\n"       \
    " @pq bra " OUT ";\n"                            \
    " setp.eq.f32 px, tx, " T ";\n"                  \
    " setp.eq.and.f32 py|pz, ty, " T ", !px;\n"      \
    " @px add.f32 tx, tx, dtx;\n"                    \
    " @py add.f32 ty, ty, dty;\n"                    \
    " @pz add.f32 tz, tz, dtz;\n"
#define MV_DDA_MOVE                                  \
    " @px add.s32 pos, pos, sx;\n"                   \
    " @pz add.s32 pos, pos, sz;\n"                   \
    " @py shf.l.wrap.b32 bit, bit, bit, sy;\n"
#define MV_DDA_LOAD_SHARED " ld.shared.u32 w, [pos];\n"
#define MV_DDA_LOAD_GLOBAL " mad.wide.u32 ag, pos, 1, gbase;\n ld.global.u32 w, [ag];\n"
#define MV_DDA_STEP_COLW(T, OUT) MV_DDA_HEAD(T, OUT) MV_DDA_MOVE MV_DDA_LOAD_SHARED \
    " lop3.or.b32 w|ph, w, bit, 0, 0xC0, pf;\n"
// (`guard` is the plane's end here)
#define MV_DDA_TEST " lop3.or.b32 a|ph, w, bit, guard, 0xC8, pf;\n"
#define MV_DDA_STEP_PLANE_SHARED(T, OUT) MV_DDA_HEAD(T, OUT) MV_DDA_MOVE MV_DDA_LOAD_SHARED MV_DDA_TEST
#define MV_DDA_STEP_PLANE_GLOBAL(T, OUT) MV_DDA_HEAD(T, OUT) MV_DDA_MOVE MV_DDA_LOAD_GLOBAL MV_DDA_TEST
// The common case's step: nothing but a filled cell stops it.  What lies outside the occupied box counts as filled here
// (the fence in x and z, `guard` = the heights outside it); afterwards w, the last column read, tells which it was.
// The fence keeps the walk in bounds, and with a guard bit in every column it ends by itself: it only ever moves on,
// along x, y and z, and each of them ends at something filled.
#define MV_DDA_SEALED_HEAD(T, OUT)                   \
    " min.f32 " T ", tx, ty, tz;\n"                  \
    " @ph bra " OUT ";\n"                            \
    " setp.eq.f32 px, tx, " T ";\n"                  \
    " setp.eq.and.f32 py|pz, ty, " T ", !px;\n"      \
    " @px add.f32 tx, tx, dtx;\n"                    \
    " @py add.f32 ty, ty, dty;\n"                    \
    " @pz add.f32 tz, tz, dtz;\n"
#define MV_DDA_STEP_SEALED(T, OUT) MV_DDA_SEALED_HEAD(T, OUT) MV_DDA_MOVE MV_DDA_LOAD_SHARED MV_DDA_TEST
#define MV_DDA_STEP_SEALED_GLOBAL(T, OUT) MV_DDA_SEALED_HEAD(T, OUT) MV_DDA_MOVE MV_DDA_LOAD_GLOBAL MV_DDA_TEST
// Loop around eight steps.  On leaving: ph = a filled cell was entered, thit = when, and px/py
// still say along which axis.
#define MV_DDA_LOOP(STEP)                            \
    " setp.ne.u32 pf, 0, 0;\n"                       \
    " setp.ne.u32 ph, 0, 0;\n"                       \
    "MV_DDA_LOOP_TOP:\n"                             \
    STEP("ta", "MV_DDA_OUT_A") STEP("tb", "MV_DDA_OUT_B") STEP("ta", "MV_DDA_OUT_A") STEP("tb", "MV_DDA_OUT_B") \
    STEP("ta", "MV_DDA_OUT_A") STEP("tb", "MV_DDA_OUT_B") STEP("ta", "MV_DDA_OUT_A") STEP("tb", "MV_DDA_OUT_B") \
    " sub.s32 it, it, 8;\n"                          \
    " setp.gt.s32 pq, it, 0;\n"                      \
    " @pq bra MV_DDA_LOOP_TOP;\n"                    \
    "MV_DDA_OUT_A:\n"                                \
    " @ph mov.f32 thit, tb;\n"                       \
    " bra MV_DDA_OUT;\n"                             \
    "MV_DDA_OUT_B:\n"                                \
    " @ph mov.f32 thit, ta;\n"                       \
    "MV_DDA_OUT:\n"
// Loop of the sealed walk.  On leaving: ph set, thit = when the filled cell was entered, px/py/pz say along which axis.
#define MV_DDA_SEALED(STEP)                          \
    " setp.ne.u32 pf, 0, 0;\n"                       \
    " setp.ne.u32 ph, 0, 0;\n"                       \
    "MV_DDA_LOOP_TOP:\n"                             \
    STEP("ta", "MV_DDA_OUT_A") STEP("tb", "MV_DDA_OUT_B") STEP("ta", "MV_DDA_OUT_A") STEP("tb", "MV_DDA_OUT_B") \
    STEP("ta", "MV_DDA_OUT_A") STEP("tb", "MV_DDA_OUT_B") STEP("ta", "MV_DDA_OUT_A") STEP("tb", "MV_DDA_OUT_B") \
    " bra MV_DDA_LOOP_TOP;\n"                        \
    "MV_DDA_OUT_A:\n"                                \
    " mov.f32 thit, tb;\n"                           \
    " bra MV_DDA_OUT;\n"                             \
    "MV_DDA_OUT_B:\n"                                \
    " mov.f32 thit, ta;\n"                           \
    "MV_DDA_OUT:\n"
// Behind either loop: a walk that met the end of its plane goes on in the next one up or down.  END: the plane's end (0 where
// there is one plane), PLANE: bytes from plane to plane, TAB: the shared-memory address of five words: the lowest and, << 16, the
// highest plane that anything is filled in, then the guards of the lowest, of those between (of the only one), of the highest, and
// all ones for those beyond, which nothing is filled in or which are not there.  BEYOND: what happens on meeting one of those;
// GUARD: which of the plane's heights count as filled from now on.
#define MV_DDA_CROSS(END, PLANE, TAB, BEYOND, GUARD, LOAD) \
    " setp.ne.b32 pq, bit, " END ";\n"               \
    " @pq bra MV_DDA_DONE;\n"                        \
    " setp.eq.s32 pq, sy, 1;\n"                      \
    " selp.s32 w, 1, -1, pq;\n"                      \
    " add.s32 q, q, w;\n"                            \
    " mad.lo.s32 pos, w, " PLANE ", pos;\n"          \
    " ld.shared.u32 a, [" TAB "];\n"                 \
    " and.b32 w, a, 0xffff;\n"                       \
    " sub.s32 w, q, w;\n"                            \
    " min.s32 w, w, 1;\n"                            \
    " shr.u32 a, a, 16;\n"                           \
    " sub.s32 a, q, a;\n"                            \
    " max.s32 a, a, -1;\n"                           \
    " add.s32 a, a, w;\n"                            \
    " add.s32 a, a, 1;\n"                            \
    " and.b32 a, a, 3;\n"                            \
    " mad.lo.s32 a, a, 4, " TAB ";\n"                \
    " ld.shared.u32 a, [a+4];\n"                     \
    " mov.b32 w, 0xffffffff;\n"                      \
    " setp.eq.u32 ph, a, 0xffffffff;\n"              \
    BEYOND                                           \
    " @ph bra MV_DDA_DONE;\n"                        \
    " selp.b32 bit, 1, 0x40000000, pq;\n"            \
    GUARD                                            \
    LOAD                                             \
    MV_DDA_TEST                                      \
    " @!ph bra MV_DDA_LOOP_TOP;\n"                   \
    "MV_DDA_DONE:\n"
#define MV_DDA_DECL                                  \
    " .reg .pred px, py, pz, pq, ph, pf;\n"          \
    " .reg .f32 tx, ty, tz, dtx, dty, dtz, ta, tb, texit, thit;\n" \
    " .reg .b32 sx, sy, sz, pos, bit, guard, w, a, it, q;\n"   \
    " .reg .b64 ag, gbase;\n"

// Threads resident per SM that the registers are laid out for: three CTAs of 384 with 56 registers (16384 observations
// 1.42 ms when two with 69 took 1.62).
constexpr int kThreadsPerSm = 3 * 384;

constexpr uint32_t kAgentInside = 1u;      // eye inside the occupied cell box
constexpr uint32_t kAgentBad = 2u;         // non-finite camera: sky frame
constexpr uint32_t kAgentFilled = 4u;      // the eye's own voxel is filled
constexpr uint32_t kAgentSealed = 8u;      // the common case: eye inside, not in a filled voxel, some height outside the box, not too large a grid
// Per-agent block in shared memory.  First the ray table, one 64-byte entry per combination of direction signs (x negative:
// +64, y: +128, z: +256; the block is 512-byte aligned, so an entry's address is the block's OR-ed with the sign bits):
//   {distance (>= 0) from the eye to the cell face met first, in x and z; what a step in x and z adds to the position}
//   {first stretch: from the eye to its end in x, z, y, a little less (kSkipMargin); start position, from which kSkipBias steps each way are taken off}
//   {first stretch: what is added to t |d| in x and z to give the crossings up to time t, rounded down; distance and step
//    in y (the step is a rotate count in the column-word flavour)}
//   {colour-table row of the face entered by an x, z, y step; -}
// then the record {Fx, Fy, Rx, Uy} {Ux, Uz, Fz, Rz} {start bit mask, heights outside the occupied box, flags, self box} {eye
// x, y, z, overlay count} {64-bit address of the env's material store, biased for the walk's positions; sky colour; miss
// depth} {lower corner of the occupied box, plane of the eye} {upper corner, -}, eye-relative boxes, overlay rectangles and per-tile box masks at offsets the host lays out.
constexpr uint32_t kAgentTabBytes = 512, kAgentAlign = 512;
constexpr uint32_t kAgentRecVecs = 7;
constexpr uint32_t kAgentRelOff = kAgentTabBytes + 16u * kAgentRecVecs;
// (as text, for the PTX blocks)
#define MV_TAB_SKIP "16"
#define MV_TAB_SKIP2 "32"
#define MV_TAB_ROW "48"
#define MV_REC_F "512"
#define MV_REC_U "528"
#define MV_REC_START "544"
#define MV_REC_MAT "576"
#define MV_REC_PLANE "604"
// a hit is looked at again if the ray leaves the cell within this factor of the time of the hit (1 - 2^-13)
#define MV_GRAZE "0f3F7FF800"
constexpr float kSealedScale = 1.0f - 1e-4f;       // least exit_scale for which that factor is wide enough
// hard bound of the traversal loop: no grid allows more steps than 3 x 1024 + 3
#define MV_STEP_BUDGET "3080"
// The empty box that a walk starts with (see the table's construction) grows by at most this many cells an axis.
constexpr int kSkipCells = 8, kSkipCellsY = 4;
// Crossings are counted up to a little less than the box's exit time: 2^-16 of the count, where rounding takes 2^-20 of
// it at most; one that falls in between is left to the walk.
constexpr float kSkipMargin = 1.0f - 1.52587890625e-5f;
// The count comes out of an addition of 2^23, whose float's bits are 0x4B000000 + count.
constexpr uint32_t kSkipBias = 0x4B000000u;
#define MV_SKIP_MAGIC "0f4B000000"
#define MV_SKIP_MAGIC2 "0x4B0000004B000000"       // the same, twice
#define MV_SKIP_UNMAGIC2 "0xCB000001CB000001"     // -(2^23 + 1), twice

// One thread's share of a sky frame (non-finite camera).
template <int NT>
__device__ __forceinline__ void write_sky(uint8_t *rgb_obs, float *depth_obs, int npx, uint32_t sky_rgbx, float miss_depth) {
    for (int i = threadIdx.x; i < npx; i += NT) depth_obs[i] = miss_depth;
    for (int i = threadIdx.x; i < npx * 3; i += NT) rgb_obs[i] = (uint8_t)(sky_rgbx >> (8 * (i % 3)));
}

// OCC: how the occupancy is walked.  kOccWord: staged in shared memory with the rest of the env block, one plane (the normal
// case).  kOccPlanes: staged, several planes, of which those up to the highest filled voxel are copied.  kOccGlobal: read from
// global memory, any number of planes; only the rest of the block is staged.
constexpr int kOccWord = 0, kOccPlanes = 1, kOccGlobal = 2;
template <int NT, int OCC>
__global__ void __launch_bounds__(NT, kThreadsPerSm / NT) render_kernel(const RenderParams p)
{
    constexpr bool COLW = OCC == kOccWord;
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kWarps = NT / 32;
    // The first CTAs of the grid render whole observations, those behind them every parts-th run of tiles of one (a batch with
    // few observations, or the end of the grid).  Neighbouring runs cost about the same, so the parts of an observation do too.
    // A part marks the boxes in all tiles' masks, like a whole; only its tile table is shorter.
    const bool whole = blockIdx.x < p.whole_ctas;
    const int apc = whole ? p.agents_per_cta : 1, parts = whole ? 1 : (int)p.parts;
    const int obs_in = whole ? (int)blockIdx.x * apc : (int)((blockIdx.x - p.whole_ctas) / p.parts);
    const int part = whole ? 0 : (int)(blockIdx.x - p.whole_ctas) - obs_in * parts;
    const int obs0 = p.obs_begin + obs_in + (whole ? 0 : (int)p.whole_ctas * p.agents_per_cta);
    const int env = p.agents == 1 ? obs0 : obs0 / p.agents;
    const int W = p.W, H = p.H;
    const int ntiles = p.tiles_x * p.tiles_y;
    // Box masks per tile: mw words of one bit per box.  With more than 32 boxes a summary word (the OR of
    // the others) comes first, so that the per-tile test reads one word whatever the box count.
    const int mw = p.mask_words;
    const int ms = mw > 1 ? mw + 1 : 1;              // words per tile
    const int m0 = mw > 1 ? 1 : 0;                   // position of the first real mask word

    const unsigned char *env_block = p.env_blocks + (size_t)env * p.lay.stride;
    // shared memory: room for the staged planes, then the rest of the block
    const uint32_t stage_occ = OCC == kOccGlobal ? 0u : p.lay.occ_bytes, unstaged = p.lay.occ_bytes - stage_occ;
    const unsigned char *s_lut = smem + (p.lay.lut_off - unstaged);
    const float4 *s_box = reinterpret_cast<const float4 *>(smem + (p.lay.box_off - unstaged));
    const int *s_count = reinterpret_cast<const int *>(smem + (p.lay.count_off - unstaged));
    float4 *s_tile = reinterpret_cast<float4 *>(smem + p.smem_tile_off);
    unsigned char *s_agents = smem + p.smem_agent_off;
    uint64_t *s_bar = reinterpret_cast<uint64_t *>(smem + p.smem_misc_off);
    uint32_t *s_flag = reinterpret_cast<uint32_t *>(smem + p.smem_misc_off + 8);
    uint32_t *s_guard = reinterpret_cast<uint32_t *>(smem + p.smem_misc_off + 12);       // (see MV_DDA_CROSS)
    auto agent_tab = [&](int ag) { return reinterpret_cast<float4 *>(s_agents + (size_t)ag * p.agent_stride); };
    auto agent_rec = [&](int ag) { return reinterpret_cast<float4 *>(s_agents + (size_t)ag * p.agent_stride + kAgentTabBytes); };
    auto agent_rel = [&](int ag) { return reinterpret_cast<float4 *>(s_agents + (size_t)ag * p.agent_stride + kAgentRelOff); };
    auto agent_ov = [&](int ag) { return reinterpret_cast<int4 *>(s_agents + (size_t)ag * p.agent_stride + p.agent_ov_off); };
    auto agent_mask = [&](int ag) { return reinterpret_cast<uint32_t *>(s_agents + (size_t)ag * p.agent_stride + p.agent_mask_off); };
    // how many tiles the CTA has
    const int runs = (ntiles + kPartRun - 1) / kPartRun, own_runs = (runs - part + parts - 1) / parts;
    const int mine = own_runs * kPartRun - ((runs - 1 - part) % parts == 0 ? runs * kPartRun - ntiles : 0);

    if (warp == 0) {
        // ---- The first warp asks for the environment block before all else, as the CTA waits longest for it, and for the cameras
        // (16384 of 128x32x128 1012 us; 1025 with the tile table written first).
        if (lane == 0) mbar_init(s_bar, 1);
        wait_for_previous();
        if (lane == 0 && !p.skip_staging) {
            if (COLW) {
                mbar_expect_tx(s_bar, p.lay.block_bytes);
                bulk_load(smem, env_block, p.lay.block_bytes, s_bar);
            } else {
                uint32_t bytes = 0;
                if (OCC == kOccPlanes) {
                    const int *bounds = reinterpret_cast<const int *>(env_block + p.lay.count_off);
                    bytes = bounds[2] < bounds[5] ? (plane_of(p.lay, bounds[5] - 1) + 1u) * p.lay.occ_plane : 0u;
                }
                mbar_expect_tx(s_bar, bytes + p.lay.block_bytes - p.lay.occ_bytes);
                if (bytes) bulk_load(smem, env_block, bytes, s_bar);
                bulk_load(smem + stage_occ, env_block + p.lay.occ_bytes, p.lay.block_bytes - p.lay.occ_bytes, s_bar);
            }
        }
        for (int ag = lane; ag < apc; ag += 32) {
            const float4 *cq = reinterpret_cast<const float4 *>(p.cams + obs0 + ag);
            const float4 c0 = cq[0], c1 = cq[1], c2 = cq[2], c3 = cq[3];   // P F | F R | R U | self, flags
            const int ovc = p.overlay ? min(max(p.overlay_count[obs0 + ag], 0), p.max_overlay) : 0;
            float4 *rec = agent_rec(ag);
            rec[0] = make_float4(c0.w, c1.x, c1.z, c2.z);
            rec[1] = make_float4(c2.y, c2.w, c1.y, c2.x);
            rec[2] = make_float4(0.0f, 0.0f, __uint_as_float((__float_as_uint(c3.y) & kFlagBadCamera) ? kAgentBad : 0u), c3.x);
            rec[3] = make_float4(c0.x, c0.y, c0.z, __int_as_float(ovc));
        }
    } else {
        // ---- the others write the tile table and clear the masks (this much needs nothing from the kernels before)
        for (int ag = 0; ag < apc; ++ag) {
            uint32_t *mk = agent_mask(ag);
            for (int i = tid - 32; i < ntiles * ms; i += NT - 32) mk[i] = 0u;
        }
        const float inv_tiles_x = 1.0f / (float)p.tiles_x;
        for (int j = tid - 32; j < mine; j += NT - 32) {
            const int i = parts == 1 ? j : (part + j / kPartRun * parts) * kPartRun + j % kPartRun;
            // (i + 0.5) / tiles_x is at least 1 / (2 tiles_x) away from an integer: exact in float for any image
            const int ty = (int)(((float)i + 0.5f) * inv_tiles_x), tx = i - ty * p.tiles_x;
            // a = 2px+1-W and b = H-1-2py of the tile's first pixel (small integers: exact as floats), its place in the image and in
            // an agent's block (the tile's box mask)
            s_tile[j] = make_float4((float)(16 * tx + 1 - W), (float)(H - 1 - 8 * ty), __int_as_float(ty * 4 * W + tx * 8),
                                    __int_as_float((int)p.agent_mask_off + 4 * i * ms));
        }
        wait_for_previous();
    }
    __syncthreads();
    // ---- meanwhile: occupancy that is not staged is asked for in L2 once per environment, the plane that the first agent's eye is in: rays
    // that look far touch a new line with every row, one after the other, and a line from HBM takes twice as long as one from L2.
    // (For which batches: see prefetch_pays.)
    if (OCC == kOccGlobal && p.prefetch && tid == 32 && part == 0 && obs0 == env * p.agents) {
        const int top = plane_begin(p.lay.planes) - 1, y = (int)fminf(fmaxf(agent_rec(0)[3].y, 0.0f), (float)top);
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;"
                     ::"l"(__cvta_generic_to_global(env_block + (size_t)(y / (int)kPlaneHeights) * p.lay.occ_plane)), "r"(p.lay.occ_plane) : "memory");
    }
    // ---- meanwhile: GUI rectangles
    if (p.overlay) {
        // GUI rectangles of each observation (unpacked to x0,y0,x1,y1 / colour in two slots); the tiles any of them touches
        // carry the bit behind the boxes'
        for (int i = tid; i < apc * p.max_overlay; i += NT) {
            const int ag = i / p.max_overlay, r = i - ag * p.max_overlay;
            const int ovc = min(max(p.overlay_count[obs0 + ag], 0), p.max_overlay);
            if (r >= ovc) continue;
            const int4 q = p.overlay[(size_t)(obs0 + ag) * p.max_overlay + r];
            const int x0 = (int)(short)(q.x & 0xffff), y0 = (int)(short)(q.x >> 16);
            const int x1 = (int)(short)(q.y & 0xffff), y1 = (int)(short)(q.y >> 16);
            agent_ov(ag)[2 * r] = make_int4(x0, y0, x1, y1);
            agent_ov(ag)[2 * r + 1] = make_int4(q.z & 0xffffff, 0, 0, 0);
            const int cx0 = max(x0, 0), cy0 = max(y0, 0), cx1 = min(x1, W), cy1 = min(y1, H);
            if (cx0 < cx1 && cy0 < cy1)
                for (int ty = cy0 >> 2; ty <= ((cy1 - 1) >> 2); ++ty)
                    for (int tx = cx0 >> 3; tx <= ((cx1 - 1) >> 3); ++tx) {
                        const int t = ty * p.tiles_x + tx;
                        uint32_t *tm = agent_mask(ag) + t * ms;
                        atomicOr(tm + m0 + (p.max_boxes >> 5), 1u << (p.max_boxes & 31));
                        if (mw > 1) *tm = 1u;
                    }
        }
    }

    // ---- wait for the block: one warp polls, the whole CTA takes the same decision
    if (warp == 0) {
        const bool ok = mbar_wait_bounded(s_bar, 0, p.wait_polls);
        if (lane == 0) *s_flag = ok ? 1u : 0u;
    }
    __syncthreads();
    if (*s_flag == 0u) {
        // The wait ran out.  Nothing of the frame is written.  If the copy was issued it is still
        // on its way into this CTA's shared memory, so one warp keeps the CTA alive until it lands.
        if (tid == 0) atomicOr(p.status, kFlagTimeout);
        if (warp == 0 && !p.skip_staging) mbar_wait_bounded(s_bar, 0, kDrainPolls);
        return;
    }
    mbar_try_wait(s_bar, 0);              // completed phase: makes the staged bytes visible to this thread

    // ---- per-agent traversal set-up and box binning
    const int pitch = (int)p.lay.pitch;
    // Traversal is confined to the cell box [lo, hi) that holds every filled voxel of this env
    // (nothing outside it can be hit), so rays that leave it, e.g. into the sky, stop there.
    const int lox = s_count[1], loy = s_count[2], loz = s_count[3];
    const int hix = s_count[4], hiy = s_count[5], hiz = s_count[6];
    const bool any_voxel = (lox < hix) && (loy < hiy) && (loz < hiz);
    const uint32_t used_planes = COLW ? 1u : any_voxel ? plane_of(p.lay, hiy - 1) + 1u : 0u;
    constexpr bool staged = OCC != kOccGlobal;
    const uint32_t occ_base = staged ? smem_addr(smem) : 0u;
    const unsigned char *occ = staged ? smem : env_block;
    const uint32_t plane_end = COLW || p.lay.planes == 1 ? 0u : kPlaneEnd;
    const int P_ = p.palette;
    const uint32_t lut_base = smem_addr(s_lut);
    const uint32_t inside_row = lut_base + (uint32_t)(kFaceInside * P_ * 4);
    // position of cell (cx, cy, cz) in the walk's own terms (see MV_DDA_*): its word, and the plane's heights that lie outside
    // the occupied box
    auto cell_plane = [&](int cy) -> uint32_t { return COLW ? 0u : plane_of(p.lay, cy); };
    auto cell_pos = [&](int cx, int cy, int cz) -> uint32_t {
        return occ_base + cell_plane(cy) * p.lay.occ_plane + 4u * column_index(p.lay, cx, cz);
    };
    auto plane_guard = [&](uint32_t q) -> uint32_t {
        const int lo = loy - plane_begin(q), hi = hiy - plane_begin(q);
        return ~(hi >= 32 ? 0xffffffffu : (1u << max(hi, 0)) - 1u) | ((1u << min(max(lo, 0), 31)) - 1u) | plane_end;
    };
    if (!COLW && tid < 5) {               // the planes' guards
        const uint32_t q_lo = any_voxel ? plane_of(p.lay, loy) : 0u, q_hi = any_voxel ? used_planes - 1u : 0u;
        const uint32_t q = tid == 1 || q_lo == q_hi ? q_lo : tid == 2 ? q_lo + 1u : q_hi;
        s_guard[tid] = tid == 0 ? q_lo | q_hi << 16 : tid == 4 || !any_voxel ? 0xffffffffu : plane_guard(q);
    }
    // Where the eye is, in the terms of the walk's tables.
    auto eye_cell = [&](const float4 &c0, int &cx, int &cy, int &cz) -> bool {
        const bool in = any_voxel && (c0.x >= (float)lox) && (c0.x < (float)hix) && (c0.y >= (float)loy) &&
                        (c0.y < (float)hiy) && (c0.z >= (float)loz) && (c0.z < (float)hiz);
        cx = cy = cz = 0;
        if (in) { cx = (int)floorf(c0.x); cy = (int)floorf(c0.y); cz = (int)floorf(c0.z); }
        return in;
    };
    // The ray tables but for the first stretch, and the state a walk starts in: a thread per combination of signs.
    for (int slot = tid; slot < 8 * apc; slot += NT) {
        const int ag = slot >> 3, signs = slot & 7;
        float4 *entry = agent_tab(ag) + 4 * signs, *rec = agent_rec(ag);
        const float4 c0 = rec[3];
        int cx, cy, cz;
        const bool cam_in = eye_cell(c0, cx, cy, cz);
        const int dx = (signs & 1) ? -1 : 1, dy = (signs & 2) ? -1 : 1, dz = (signs & 4) ? -1 : 1;
        const float qx = dx < 0 ? c0.x - (float)cx : (float)(cx + 1) - c0.x, qz = dz < 0 ? c0.z - (float)cz : (float)(cz + 1) - c0.z;
        const float qy = dy < 0 ? c0.y - (float)cy : (float)(cy + 1) - c0.y;
        const int sx = 4 * dx, sz = 4 * pitch * dz, sy = dy < 0 ? 31 : 1;
        entry[0] = make_float4(qx, qz, __int_as_float(sx), __int_as_float(sz));
        entry[2] = make_float4((1.0f - qx) * kSkipMargin, (1.0f - qz) * kSkipMargin, qy, __int_as_float(sy));
        entry[3] = make_float4(__uint_as_float(lut_base + (uint32_t)((dx < 0 ? 1 : 0) * P_ * 4)),
                               __uint_as_float(lut_base + (uint32_t)((4 + (dz < 0 ? 1 : 0)) * P_ * 4)),
                               __uint_as_float(lut_base + (uint32_t)((2 + (dy < 0 ? 1 : 0)) * P_ * 4)), 0.0f);
        if (signs == 0) {
            const bool filled = cam_in && voxel_filled(p.lay, occ, cx, cy, cz);
            const uint32_t q = cell_plane(cy), guard = plane_guard(q);
            rec[2].x = __uint_as_float(1u << ((cy - plane_begin(q)) & 31));
            rec[2].y = __uint_as_float(guard);                   // heights outside the occupied box
            rec[2].z = __uint_as_float(__float_as_uint(rec[2].z) | (cam_in ? kAgentInside : 0u) | (filled ? kAgentFilled : 0u) |
                                       (cam_in && !filled && guard && p.exit_scale > kSealedScale ? kAgentSealed : 0u));
            const unsigned long long mp = reinterpret_cast<unsigned long long>(p.mat + (size_t)env * p.mat_stride - ((size_t)occ_base << (p.lay.ysh - 2)));
            rec[4] = make_float4(__uint_as_float((uint32_t)mp), __uint_as_float((uint32_t)(mp >> 32)),
                                 __uint_as_float(p.sky_rgbx), p.miss_depth);
            rec[5] = make_float4((float)lox, (float)loy, (float)loz, __uint_as_float(q));
            rec[6] = make_float4((float)hix, (float)hiy, (float)hiz, 0.0f);
        }
    }
    // The first stretch of a walk.  For every combination of signs: a box of empty cells that begins at the eye's cell.  A ray
    // crosses nothing filled before it leaves that box, so it takes all its x and z crossings up to then at once, whatever
    // their order (three steps of seven on average; the vertical ones are too few to be worth it): 234 -> 220
    // instructions a tile on 128x32x128 columns, 1230 -> 1184 us for 16384 observations; 64x16x64 rooms with boxes
    // 1126 -> 1007 us.
    // A warp per agent, eight lanes per quadrant, each with a row of cells at the eye's height: the empty cells at its
    // beginning, the least of them over the rows up to it, and of those rectangles the one with the longest shorter side; then
    // as many layers above and below as are empty over all of it.  (Growing the boxes layer by layer gives the same ones
    // within 1 %, but ten rounds that depend on one another were the longest part of a CTA's set-up: 5000 to 7000 cycles.)
    for (int ag = (warp + kWarps - 2) % kWarps; ag < apc; ag += kWarps) {
        const int j = lane & 7, dx = (lane & 8) ? -1 : 1, dz = (lane & 16) ? -1 : 1;
        const float4 c0 = agent_rec(ag)[3];
        int cx, cy, cz;
        const bool cam_in = eye_cell(c0, cx, cy, cz);
        // (an eye exactly on a cell face and looking down the axis leaves its cell at once: the rectangle begins a cell
        // further on, so that mirrored views get mirrored boxes)
        const int on_x = dx < 0 && c0.x == (float)cx ? 1 : 0, on_z = dz < 0 && c0.z == (float)cz ? 1 : 0;
        const int bx = cx + dx * on_x, bz = cz + dz * on_z;
        const int lim_x = min(kSkipCells - 1, dx < 0 ? bx - lox : hix - 1 - bx), lim_z = dz < 0 ? bz - loz : hiz - 1 - bz;
        const uint32_t q = cell_plane(cy);
        const int yb = (cy - plane_begin(q)) & 31;
        const uint32_t *word = reinterpret_cast<const uint32_t *>(occ + (size_t)q * p.lay.occ_plane) + (int)column_index(p.lay, bx, bz + dz * j);
        const bool row_in = cam_in && j <= lim_z;
        uint32_t col[kSkipCells], filled = ~0u << kSkipCells, seen = plane_end;
#pragma unroll
        for (int i = 0; i < kSkipCells; ++i) {
            col[i] = row_in && i <= lim_x ? word[dx * i] : ~0u;
            filled |= ((col[i] >> yb) & 1u) << i;
        }
        int w = __ffs(filled) - 1;                               // empty cells at the row's beginning
#pragma unroll
        for (int s = 1; s < 8; s <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, w, s, 8);
            if (j >= s) w = min(w, o);
        }
        // longest shorter side first, then the longer one; the extents ride along
        int key = w > 0 ? min(w - 1, j) << 12 | max(w - 1, j) << 8 | (w - 1) << 4 | j : -1;
#pragma unroll
        for (int s = 1; s < 8; s <<= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, s));
        const bool any = key >= 0;
        const int rx = any ? (key >> 4) & 15 : 0, rz = any ? key & 15 : 0;
#pragma unroll
        for (int i = 0; i < kSkipCells; ++i)
            if (i <= rx && j <= rz) seen |= col[i];
#pragma unroll
        for (int s = 1; s < 8; s <<= 1) seen |= __shfl_xor_sync(0xffffffffu, seen, s);
        if (j < 2) {                                             // lane 0 of the quadrant: upward, lane 1: downward
            const int dy = j ? -1 : 1;
            // empty layers next to the eye's, from the columns or-ed together (the bit beyond the word counts as filled)
            const uint32_t beyond = dy > 0 ? (yb < 31 ? seen >> (yb + 1) | 0x80000000u >> yb : 1u)
                                           : (yb > 0 ? __brev(seen << (32 - yb)) | 1u << yb : 1u);
            const int ey = any ? min(min(kSkipCellsY, __ffs(beyond) - 1), dy < 0 ? cy - loy : hiy - 1 - cy) : 0;
            const int ex = any ? rx + on_x : 0, ez = any ? rz + on_z : 0;
            const int sx = 4 * dx, sz = 4 * pitch * dz;
            const int signs = (dx < 0 ? 1 : 0) | (dy < 0 ? 2 : 0) | (dz < 0 ? 4 : 0);
            const float qx = dx < 0 ? c0.x - (float)cx : (float)(cx + 1) - c0.x, qz = dz < 0 ? c0.z - (float)cz : (float)(cz + 1) - c0.z;
            const float qy = dy < 0 ? c0.y - (float)cy : (float)(cy + 1) - c0.y;
            agent_tab(ag)[4 * signs + 1] = make_float4(((float)ex + qx) * kSkipMargin, ((float)ez + qz) * kSkipMargin,
                                                       ((float)ey + qy) * kSkipMargin, __uint_as_float(cell_pos(cx, cy, cz) -
                                                       kSkipBias * (uint32_t)sx - kSkipBias * (uint32_t)sz));
        }
    }
    // Boxes: relative to the eye, and binned by the bounding rectangle of their projected corners (conservative, so every box
    // that a pixel's ray can touch is tested for that pixel).  Four lanes to a box, two corners and every fourth row of
    // tiles each; dealt from the last warp down, away from the warps that build the tables above.
    {
        const int nb = min(s_count[0], p.max_boxes), part = lane & 3;
        for (int i0 = 0; i0 < 4 * apc * p.max_boxes; i0 += NT) {
            const int i = (i0 + (kWarps - 1 - warp) * 32 + lane) >> 2;
            if ((i & ~7) >= apc * p.max_boxes) break;            // (the whole warp)
            const int ag = apc == 1 ? 0 : min(i / p.max_boxes, apc - 1), b = min(i - ag * p.max_boxes, p.max_boxes - 1);
            const float4 *rec = agent_rec(ag);
            const float4 c0 = rec[0], c1 = rec[1], P4 = rec[3];
            const float Px = P4.x, Py = P4.y, Pz = P4.z, Fx = c0.x, Fy = c0.y, Fz = c1.z;
            const float Rx = c0.z, Rz = c1.w, Ux = c1.x, Uy = c0.w, Uz = c1.y;       // (cameras do not roll: Ry = 0)
            const int self_box = __float_as_int(rec[2].w);
            const float ir2 = fast_rcp(Rx * Rx + Rz * Rz), iu2 = fast_rcp(Ux * Ux + Uy * Uy + Uz * Uz);
            const float4 A = s_box[2 * b], B = s_box[2 * b + 1];
            const float lx = A.x - Px, ly = A.y - Py, lz = A.z - Pz;
            const float hx = A.w - Px, hy = B.x - Py, hz = B.y - Pz;
            const bool valid = (b < nb) && (b != self_box) && (A.x < A.w) && (A.y < B.x) && (A.z < B.y) && i < apc * p.max_boxes;
            float tmin = kInf, tmax = -kInf, fxmin = kInf, fxmax = -kInf, fymin = kInf, fymax = -kInf;
            uint32_t beside = 15u;                            // a bit per side of the view that all corners lie beyond
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const float vx = (part & 1) ? hx : lx, vy = c ? hy : ly, vz = (part & 2) ? hz : lz;
                const float t = vx * Fx + vy * Fy + vz * Fz;
                const float u = (vx * Rx + vz * Rz) * ir2;
                const float w = (vx * Ux + vy * Uy + vz * Uz) * iu2;
                tmin = fminf(tmin, t); tmax = fmaxf(tmax, t);
                const float wide = ((float)W - 0.5f) * t, high = ((float)H - 0.5f) * t;      // (a quarter of a pixel beyond the outermost centres)
                beside &= (u > wide ? 1u : 0u) | (-u > wide ? 2u : 0u) | (w > high ? 4u : 0u) | (-w > high ? 8u : 0u);
                const float it = fast_rcp(fmaxf(t, 1e-3f));
                const float fx = (u * it + (float)(W - 1)) * 0.5f;     // pixel column of the projection
                const float fy = ((float)(H - 1) - w * it) * 0.5f;     // pixel row
                fxmin = fminf(fxmin, fx); fxmax = fmaxf(fxmax, fx);
                fymin = fminf(fymin, fy); fymax = fmaxf(fymax, fy);
            }
#pragma unroll
            for (int s = 1; s < 4; s <<= 1) {
                tmin = fminf(tmin, __shfl_xor_sync(0xffffffffu, tmin, s)); tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, s));
                fxmin = fminf(fxmin, __shfl_xor_sync(0xffffffffu, fxmin, s)); fxmax = fmaxf(fxmax, __shfl_xor_sync(0xffffffffu, fxmax, s));
                fymin = fminf(fymin, __shfl_xor_sync(0xffffffffu, fymin, s)); fymax = fmaxf(fymax, __shfl_xor_sync(0xffffffffu, fymax, s));
                beside &= __shfl_xor_sync(0xffffffffu, beside, s);
            }
            const bool front = tmin > 0.05f;                 // whole box safely in front of the eye plane
            if (part == 0 && valid) {
                agent_rel(ag)[2 * b] = make_float4(lx, ly, lz, front ? tmin * 0.9999f : 0.0f);
                agent_rel(ag)[2 * b + 1] = make_float4(hx, hy, hz, B.z);
            }
            // Ignored, wholly behind the eye, or wholly beside the view.  The last matters for boxes across the eye plane, which have no
            // bounding rectangle and go to every tile: nearly all of them are off to one side, half a box an agent among 32 in a
            // room of 64x64, and testing them in every tile is a sixth of the frame (8192 x 2 of 256x144 2591 us, 3040 with them).
            if (!valid || tmax < -1e-3f || beside) continue;
            int px0 = 0, px1 = W - 1, py0 = 0, py1 = H - 1;
            if (front) {
                px0 = (int)ceilf(fmaxf(fxmin - 0.25f, 0.0f));
                px1 = (int)floorf(fminf(fxmax + 0.25f, (float)(W - 1)));
                py0 = (int)ceilf(fmaxf(fymin - 0.25f, 0.0f));
                py1 = (int)floorf(fminf(fymax + 0.25f, (float)(H - 1)));
                if (px0 > px1 || py0 > py1) continue;
            }
            const uint32_t bit = 1u << (b & 31);
            uint32_t *mask = agent_mask(ag);
            for (int ty = (py0 >> 2) + part; ty <= (py1 >> 2); ty += 4)
                for (int tx = px0 >> 3; tx <= (px1 >> 3); ++tx) {
                    uint32_t *tm = mask + (ty * p.tiles_x + tx) * ms;
                    atomicOr(tm + m0 + (b >> 5), bit);
                    if (mw > 1) *tm = 1u;                           // the summary word only has to be non-zero
                }
        }
    }
    __syncthreads();

    uint32_t guards = smem_addr(s_guard);
    // Does the uncommon tile loop read the occupied box again, so that its bounds hold no registers while the common one runs?  As
    // compiled that is 1 % faster for one plane (8192 x 2 of 256x144: 3065 us, 3099 without), and slower for several (4096 of
    // 64x36x64 254 and 250) and in CTAs of 576 threads (2048 x 2 of 160x32x160 318 and 303).
    constexpr bool kReadBox = COLW && NT != 576;
    const float flox = (float)lox, floy = (float)loy, floz = (float)loz;
    const float fhix = (float)hix, fhiy = (float)hiy, fhiz = (float)hiz;

    // ---- per-lane constants of the 8 x 4 tile: pixel offsets and the store plan.  Depth goes to the
    // lane's own pixel.  A tile row's RGB is 24 bytes = six 32-bit words; word j starts inside pixel
    // q = j + j/3 of the row (at its byte j % 3) and ends inside pixel q + 1, so the lanes of pixels
    // 0, 1, 2, 4, 5, 6 of each row write one word each, picked by a byte permute from the lane's own
    // packed colour and its right neighbour's; the lanes of pixels 3 and 7 store no RGB word.  keep()
    // pins the constants in registers: recomputing them per tile costs more issue slots than the
    // registers are worth.
    float lane_a = (float)(2 * (lane & 7)), lane_b = -(float)(2 * (lane >> 3));
    const int st_r = lane >> 3, st_q = lane & 7, st_j = st_q - (st_q >> 2), st_byte = st_q & 3;
    // bytes st_byte.. of the own pixel (3 of them at most), then the neighbour's from its byte 0 (selector 4..)
    uint32_t st_sel = st_byte == 0 ? 0x4210u : (st_byte == 1 ? 0x5421u : (st_byte == 2 ? 0x6542u : 0xffffffffu));
    const int depth_lane_off = (lane >> 3) * W + (lane & 7);
    const int rgb_lane_off = st_r * W * 3 + st_j * 4;
    opaque(lane_a, lane); opaque(lane_b, lane); opaque(st_sel, lane);
    unsigned long long lane_ab;
    asm("mov.b64 %0, {%1, %2};" : "=l"(lane_ab) : "f"(lane_a), "f"(lane_b));
    const uint32_t tile_begin = smem_addr(s_tile) + 16u * (uint32_t)warp;
    uint32_t tile_end = smem_addr(s_tile) + 16u * (uint32_t)mine;
    opaque(tile_end, lane);

    for (int ag = 0; ag < apc; ++ag) {
        const int obs = obs0 + ag;
        uint8_t *rgb_obs = p.rgb + (size_t)obs * H * W * 3;
        float *depth_obs = p.depth + (size_t)obs * H * W;
        const uint32_t aflags = __float_as_uint(agent_rec(ag)[2].z);
        if (aflags & kAgentBad) {                   // non-finite camera: a sky frame
            write_sky<NT>(rgb_obs, depth_obs, W * H, p.sky_rgbx, p.miss_depth);
            continue;
        }
        uint32_t abase = smem_addr(agent_tab(ag));
        // (store addresses as global-space addresses for the PTX store block)
        unsigned long long depth_lane = (unsigned long long)__cvta_generic_to_global(depth_obs + depth_lane_off);
        unsigned long long rgb_lane = (unsigned long long)__cvta_generic_to_global(rgb_obs + rgb_lane_off);
        keep(abase);
        asm volatile("" : "+l"(depth_lane), "+l"(rgb_lane));

        // ---- tiles: warp w takes tiles w, w + nwarps, ... (8 x 4 pixels, one per lane).  Two loops, so
        // that the choice between the common case and the rest is taken per agent, not per tile; what
        // follows the walk is the same for both.  The warp-wide reduction and shuffle in it name all 32
        // lanes, so they wait by themselves for lanes whose walk ran longer.
        auto finish_tile = [&](uint32_t mask_p, int tile_px, uint32_t pos, uint32_t bit, uint32_t plane, uint32_t row,
                               uint32_t tab, uint32_t graze, float t_hit, float dtx, float dty, float dtz) {
            // ---- the hit voxel's material byte is asked for from global memory (its colour is looked up
            // in the shaded table only in the store block, after everything that does not need it), this
            // tile's first box-mask word is read, and the latest voxel hit of the warp is found (boxes wholly
            // behind it are skipped).  Predicated, not branched; sky colour and miss depth ride with the
            // material store's address in the agent block.  (The voxel index is rebuilt from the column's
            // address, the bit and the plane.)
            uint32_t rgbx, m, mat_id;
            float depth;
            {
                uint32_t y, vi;
                asm("bfind.u32 %0, %1;" : "=r"(y) : "r"(bit));
                vi = COLW ? (pos << 3) + y : (pos << (p.lay.ysh - 2)) + y + plane * (kPlaneHeights - (p.lay.occ_plane << (p.lay.ysh - 2)));
                asm volatile("{\n"
                    " .reg .pred pv;\n"
                    " .reg .b32 skyb, missb;\n"
                    " .reg .b64 mp, sm;\n"
                    " ld.shared.v2.b64 {mp, sm}, [%7+" MV_REC_MAT "];\n"
                    " ld.shared.u32 %2, [%8];\n"
                    " mov.b64 {skyb, missb}, sm;\n"
                    " mov.b32 %0, skyb;\n"
                    " mov.b32 %1, missb;\n"
                    " setp.ne.u32 pv, %4, 0xffffffff;\n"
                    " mad.wide.u32 mp, %5, 1, mp;\n"
                    " @pv ld.global.u8 %3, [mp];\n"
                    " @pv mov.f32 %1, %6;\n"
                    "}\n"
                    : "=&r"(rgbx), "=&f"(depth), "=&r"(m), "=&r"(mat_id)
                    : "r"(row), "r"(vi), "f"(t_hit), "r"(abase), "r"(mask_p)
                    : "memory");
            }

            // ---- the less common work, behind one test: boxes binned to this tile, and the GUI overlay (the bit behind the
            // boxes').  A box wins only with a strictly smaller time; boxes wholly behind the warp's latest voxel hit are skipped.
            if ((m | graze) != 0u) {
                // A voxel that the ray enters within the rounding of crossing times before it leaves the occupied box does not
                // count (see exit_scale).  The ray leaves the box no earlier than the voxel, so that can only be where it leaves
                // the voxel again almost at once: one ray in a thousand, and only for those the exit time is worked out.
                if (graze) {
                    const float4 eye = agent_rec(ag)[3], lo = agent_rec(ag)[5], hi = agent_rec(ag)[6];
                    const float t_exit = min3f(((tab & 64u) ? eye.x - lo.x : hi.x - eye.x) * dtx, ((tab & 128u) ? eye.y - lo.y : hi.y - eye.y) * dty,
                                               ((tab & 256u) ? eye.z - lo.z : hi.z - eye.z) * dtz) * p.exit_scale;
                    if (!(t_hit < t_exit)) { row = kNoRow; t_hit = kInf; rgbx = p.sky_rgbx; depth = p.miss_depth; }
                }
                if (m != 0u) {
                    const float wmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(t_hit)));
                    float tb = t_hit;
                    bool gui = false;
                    // (more than one word: m was the summary; start with the first real word)
                    if (mw > 1) asm volatile("ld.shared.u32 %0, [%1+4];" : "=r"(m) : "r"(mask_p));
                    // signed reciprocals again, from the signs in the table entry's address
                    const float ix = __uint_as_float(__float_as_uint(dtx) | ((tab & 64u) << 25));
                    const float iy = __uint_as_float(__float_as_uint(dty) | ((tab & 128u) << 24));
                    const float iz = __uint_as_float(__float_as_uint(dtz) | ((tab & 256u) << 23));
                    uint32_t baddr = 0;
                    for (int w = 0;;) {
                        if (p.overlay && w == (p.max_boxes >> 5)) {
                            gui = (m >> (p.max_boxes & 31)) & 1u;
                            m &= ~(1u << (p.max_boxes & 31));
                        }
                        while (m) {
                            const int b = (__ffs(m) - 1) + 32 * w;
                            m &= m - 1;
                            float4 lo, hi;
                            const uint32_t rel_p = abase + kAgentRelOff + 32u * (uint32_t)b;
                            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(lo.x), "=f"(lo.y), "=f"(lo.z), "=f"(lo.w) : "r"(rel_p));
                            if (lo.w > wmax) continue;
                            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4+16];" : "=f"(hi.x), "=f"(hi.y), "=f"(hi.z), "=f"(hi.w) : "r"(rel_p));
                            float x1, x2, y1, y2;
                            mul2(x1, y1, lo.x, lo.y, ix, iy);
                            mul2(x2, y2, hi.x, hi.y, ix, iy);
                            const float z1 = lo.z * iz, z2 = hi.z * iz;
                            const float nx = fminf(x1, x2), ny = fminf(y1, y2), nz = fminf(z1, z2);
                            const float tn = max3f(nx, ny, nz);
                            const float tf = min3f(fmaxf(x1, x2), fmaxf(y1, y2), fmaxf(z1, z2));
                            const float t = fmaxf(tn, 0.0f);
                            if ((tn <= tf) && (tf > 0.0f) && (t < tb)) {
                                tb = t;
                                uint32_t r = inside_row;
                                if (!(tn < 0.0f))
                                    asm volatile("ld.shared.u32 %0, [%1+" MV_TAB_ROW "];" : "=r"(r)
                                                 : "r"(tab + ((nx == tn) ? 0u : ((ny == tn) ? 8u : 4u))));
                                baddr = r + 4u * __float_as_uint(hi.w);
                            }
                        }
                        if (++w >= mw) break;
                        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(m) : "r"(mask_p + 4u * (uint32_t)(w + 1)));
                    }
                    if (baddr) {
                        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(rgbx) : "r"(baddr));
                        depth = tb + 0.0f;
                        row = kNoRow;                            // the voxel behind the box is not looked up
                    }
                    // GUI overlay: rectangles in list order, later ones on top; depth is left alone
                    if (gui) {
                        const int4 *ov = agent_ov(ag);
                        const int ov_count = __float_as_int(agent_rec(ag)[3].w);
                        // (tile_px / W, exact: tile rows begin at multiples of 4 W, so the quotient is 8 / W away from the next integer or more)
                        const int row0 = (int)(((float)tile_px + 4.0f) * p.inv_W);
                        const int px = tile_px - row0 * W + (lane & 7), py = row0 + (lane >> 3);
                        if (row != kNoRow) {                     // the rectangles go over the voxel colour: look it up now
                            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(rgbx) : "r"(row + 4u * mat_id));
                            row = kNoRow;
                        }
                        for (int r = 0; r < ov_count; ++r) {
                            const int4 q = ov[2 * r];
                            if (px >= q.x && px < q.z && py >= q.y && py < q.w) rgbx = (uint32_t)ov[2 * r + 1].x;
                        }
                    }
                }
            }

            // ---- store: depth rows are 32-byte segments; RGB rows are 24 bytes = 6 packed words
            asm volatile("{\n"
                " .reg .pred ps, pv;\n"
                " .reg .b32 ca, cb, cc;\n"
                " .reg .b64 ad;\n"
                " mad.wide.s32 ad, %2, 4, %3;\n"
                " st.global.f32 [ad], %1;\n"
                " setp.ne.u32 pv, %6, 0xffffffff;\n"
                " mad.lo.u32 ca, %7, 4, %6;\n"
                " mov.b32 cc, %0;\n"
                " @pv ld.shared.u32 cc, [ca];\n"
                " shfl.sync.down.b32 cb, cc, 1, 31, 0xffffffff;\n"
                " mad.wide.s32 ad, %2, 3, %4;\n"
                " prmt.b32 ca, cc, cb, %5;\n"
                " setp.ge.s32 ps, %5, 0;\n"
                " @ps st.global.u32 [ad], ca;\n"
                "}\n"
                :: "r"(rgbx), "f"(depth), "r"(tile_px), "l"(depth_lane), "l"(rgb_lane), "r"(st_sel), "r"(row), "r"(mat_id)
                : "memory");
        };
        if (aflags & kAgentSealed) {
            for (uint32_t tile_p = tile_begin; tile_p < tile_end; tile_p += 16u * kWarps) {
                int tile_px;
                uint32_t pos, bit = 0, plane = 0, row, tab, graze, mask_p;
                float t_hit, dtx, dty, dtz;
                // ---- the common case in one block of PTX: tile record, ray through the pixel centre
                // (d = F + a*Rs + b*Us, a = 2px+1-W, b = H-1-2py, two chained FMAs per component),
                // reciprocals, the table entry for the ray's signs, first crossing times, the first
                // stretch, then the walk.  The basis is re-read from shared memory per tile:
                // three broadcast loads cost less than nine registers held across the walk.
                // Where two components take the same operation and their operands lie side by side as loaded, one
                // instruction does both (f32x2: the same roundings, one issue slot): 1079 -> 1065 us for 16384
                // observations, 3194 -> 3118 for 16384 of 256x144.  Packing the products with dt as well is slower: the
                // pairs it wants do not outlive the walk's own use of the registers, and are moved.  (The end of the first
                // stretch as one product, packed: 3121 -> 3095.)
                // A direction component that is exactly zero needs no special case here: its reciprocal
                // is +-inf, so its crossing time is +inf (or NaN when the eye sits exactly on the face,
                // which min and the compares ignore) and that axis is never stepped, which is the rule
                // for such rays.
#define MV_SEALED_RAY(TILE, BASE, AB, MASK) \
                    MV_DDA_DECL \
                    " .reg .f32 Ta, Tb, Fx, Fy, Fz, Rx, Rz, Ux, Uy, Uz, ca, cb, dx, dy, dz, ix, iy, iz;\n" \
                    " .reg .f32 q0, q1, q2, q3, q4;\n" \
                    " .reg .b32 u, v;\n" \
                    " .reg .b64 T2, D2, Q2, C2, M2;\n" \
                    " ld.shared.v4.b32 {Ta, Tb, %0, " MASK "}, [" TILE "];\n" \
                    " ld.shared.v4.f32 {Fx, Fy, Rx, Uy}, [" BASE "+" MV_REC_F "];\n" \
                    " ld.shared.v4.f32 {Ux, Uz, Fz, Rz}, [" BASE "+" MV_REC_U "];\n" \
                    " ld.shared.v2.b32 {bit, guard}, [" BASE "+" MV_REC_START "];\n" \
                    " mov.b64 C2, {Ta, Tb};\n" \
                    " add.rn.f32x2 C2, C2, " AB ";\n" \
                    " mov.b64 {ca, cb}, C2;\n" \
                    " mov.b64 T2, {Fx, Fy};\n" \
                    " mov.b64 D2, {Rx, Uy};\n" \
                    " fma.rn.f32x2 T2, C2, D2, T2;\n" \
                    " mov.b64 {dx, dy}, T2;\n" \
                    " fma.rn.f32 dz, ca, Rz, Fz;\n" \
                    " fma.rn.f32 dx, cb, Ux, dx;\n" \
                    " fma.rn.f32 dz, cb, Uz, dz;\n" \
                    " abs.f32 ix, dx;\n" \
                    " abs.f32 iy, dy;\n" \
                    " abs.f32 iz, dz;\n" \
                    " rcp.approx.ftz.f32 dtx, ix;\n" \
                    " rcp.approx.ftz.f32 dty, iy;\n" \
                    " rcp.approx.ftz.f32 dtz, iz;\n" \
                    " mov.b32 u, dx;\n" \
                    " mov.b32 v, dz;\n" \
                    " prmt.b32 u, u, v, 0x00FB;\n"    /* byte 0: sign of dx, byte 1: sign of dz */ \
                    " lop3.b32 %8, u, 0x140, " BASE ", 0xEA;\n" \
                    " mov.b32 u, dy;\n" \
                    " shr.u32 u, u, 24;\n" \
                    " lop3.b32 %8, u, 0x80, %8, 0xEA;\n" \
                    " ld.shared.v4.b32 {tx, tz, sx, sz}, [%8];\n" \
                    " ld.shared.v4.b32 {q0, q1, q2, pos}, [%8+" MV_TAB_SKIP "];\n" \
                    " ld.shared.v4.b32 {q3, q4, ty, sy}, [%8+" MV_TAB_SKIP2 "];\n" \
                    " mul.f32 tx, tx, dtx;\n" \
                    " mul.f32 ty, ty, dty;\n" \
                    " mul.f32 tz, tz, dtz;\n" \
                    " mov.b64 Q2, {q0, q1};\n" \
                    " mov.b64 D2, {dtx, dtz};\n" \
                    " mul.rn.f32x2 Q2, Q2, D2;\n" \
                    " mov.b64 {q0, q1}, Q2;\n" \
                    " mul.f32 q2, q2, dty;\n" \
                    " min.f32 q0, q0, q1, q2;\n" \
                    " fma.rn.f32 q3, q0, ix, q3;\n" \
                    " fma.rn.f32 q4, q0, iz, q4;\n" \
                    " mov.b64 Q2, {q3, q4};\n" \
                    " mov.b64 M2, " MV_SKIP_MAGIC2 ";\n" \
                    " add.rm.f32x2 Q2, Q2, M2;\n" \
                    " mov.b64 {q3, q4}, Q2;\n" \
                    " mov.b32 u, q3;\n" \
                    " mad.lo.u32 pos, u, sx, pos;\n" \
                    " mov.b32 u, q4;\n" \
                    " mad.lo.u32 pos, u, sz, pos;\n" \
                    /* (the first crossing by an addition as in the walk and only the rest by a product, so that up to two crossings */ \
                    /* give the bits that the walk would give and ties between axes go the same way) */ \
                    " setp.gt.f32 px, q3, " MV_SKIP_MAGIC ";\n" \
                    " setp.gt.f32 pz, q4, " MV_SKIP_MAGIC ";\n" \
                    " mov.b64 Q2, {q3, q4};\n" \
                    " mov.b64 M2, " MV_SKIP_UNMAGIC2 ";\n" \
                    " add.rn.f32x2 Q2, Q2, M2;\n" \
                    " mov.b64 {q3, q4}, Q2;\n" \
                    " @px add.f32 tx, tx, dtx;\n" \
                    " @pz add.f32 tz, tz, dtz;\n" \
                    " @px fma.rn.f32 tx, q3, dtx, tx;\n" \
                    " @pz fma.rn.f32 tz, q4, dtz, tz;\n"
#define MV_SEALED_END \
                    /* a miss if the cell is fence (its guard bits are set) or lies at a height outside the box */ \
                    " or.b32 w, w, bit;\n" \
                    " and.b32 w, w, guard;\n" \
                    " setp.eq.u32 ph, w, 0;\n" \
                    /* (a hit that may be too close to the ray's exit from the box: see below) */ \
                    " min.f32 ta, tx, ty, tz;\n" \
                    " mul.f32 ta, ta, " MV_GRAZE ";\n" \
                    " setp.ge.and.f32 pq, thit, ta, ph;\n" \
                    " selp.u32 %9, 1, 0, pq;\n" \
                    " mov.b32 %4, 0xffffffff;\n" \
                    " @!ph mov.f32 thit, 0f7F800000;\n" \
                    " mov.b32 u, %8;\n" \
                    " @py add.u32 u, u, 8;\n" \
                    " @pz add.u32 u, u, 4;\n" \
                    " @ph ld.shared.u32 %4, [u+" MV_TAB_ROW "];\n" \
                    " mov.b32 %1, pos;\n" \
                    " mov.b32 %2, bit;\n" \
                    " mov.f32 %3, thit;\n" \
                    " mov.f32 %5, dtx;\n" \
                    " mov.f32 %6, dty;\n" \
                    " mov.f32 %7, dtz;\n"
                if constexpr (COLW) {
                    asm volatile("{\n" MV_SEALED_RAY("%11", "%12", "%13", "%10") MV_DDA_SEALED(MV_DDA_STEP_SEALED) MV_SEALED_END "}\n"
                        : "=&r"(tile_px), "=&r"(pos), "=&r"(bit), "=&f"(t_hit), "=&r"(row), "=&f"(dtx), "=&f"(dty), "=&f"(dtz), "=&r"(tab), "=&r"(graze), "=&r"(mask_p)
                        : "r"(tile_p), "r"(abase), "l"(lane_ab)
                        : "memory");
                } else {
#define MV_SEALED_PLANE " ld.shared.u32 q, [%13+" MV_REC_PLANE "];\n"
#define MV_SEALED_CROSS(LOAD) MV_DDA_CROSS("%15", "%16", "%17", "", " mov.b32 guard, a;\n", LOAD) " mov.b32 %11, q;\n"
#define MV_SEALED_IO                                                                                                \
                        : "=&r"(tile_px), "=&r"(pos), "=&r"(bit), "=&f"(t_hit), "=&r"(row), "=&f"(dtx), "=&f"(dty), "=&f"(dtz), "=&r"(tab), "=&r"(graze), \
                          "=&r"(mask_p), "=&r"(plane)                                               \
                        : "r"(tile_p), "r"(abase), "l"(lane_ab), "r"(plane_end), "r"(p.lay.occ_plane), "r"(guards), "l"(env_block)                                  \
                        : "memory"
                    if constexpr (staged)
                        asm volatile("{\n" MV_SEALED_RAY("%12", "%13", "%14", "%10") MV_SEALED_PLANE MV_DDA_SEALED(MV_DDA_STEP_SEALED) MV_SEALED_CROSS(MV_DDA_LOAD_SHARED) MV_SEALED_END "}\n" MV_SEALED_IO);
                    else
                        asm volatile("{\n" MV_SEALED_RAY("%12", "%13", "%14", "%10") MV_SEALED_PLANE " mov.b64 gbase, %18;\n" MV_DDA_SEALED(MV_DDA_STEP_SEALED_GLOBAL) MV_SEALED_CROSS(MV_DDA_LOAD_GLOBAL) MV_SEALED_END "}\n" MV_SEALED_IO);
#undef MV_SEALED_PLANE
#undef MV_SEALED_CROSS
#undef MV_SEALED_IO
                }
#undef MV_SEALED_RAY
#undef MV_SEALED_END
                finish_tile(abase + mask_p, tile_px, pos, bit, plane, row, tab, graze, t_hit, dtx, dty, dtz);
            }
        } else {
            const float4 P4 = agent_rec(ag)[3];
            const float Px = P4.x, Py = P4.y, Pz = P4.z;
            const bool cam_in = (aflags & kAgentInside) != 0;
            float4 lo = make_float4(flox, floy, floz, 0.0f), hi = make_float4(fhix, fhiy, fhiz, 0.0f);
            if constexpr (kReadBox) { lo = agent_rec(ag)[5]; hi = agent_rec(ag)[6]; }
            const int ilox = kReadBox ? (int)lo.x : lox, iloy = kReadBox ? (int)lo.y : loy, iloz = kReadBox ? (int)lo.z : loz;
            const int ihix = kReadBox ? (int)hi.x : hix, ihiy = kReadBox ? (int)hi.y : hiy, ihiz = kReadBox ? (int)hi.z : hiz;
            const bool any = kReadBox ? ilox < ihix && iloy < ihiy && iloz < ihiz : any_voxel;
            for (uint32_t tile_p = tile_begin; tile_p < tile_end; tile_p += 16u * kWarps) {
                int tile_px;
                uint32_t pos, bit = 0, plane = 0, row, tab, mask_p;
                float t_hit, dtx, dty, dtz;
                // ---- every other case: the same steps in C++, with the eye possibly outside the
                // occupied box and either flavour of the walk
                float Ta, Tb;
                asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=f"(Ta), "=f"(Tb), "=r"(tile_px), "=r"(mask_p) : "r"(tile_p));
                const float4 FR = agent_rec(ag)[0], UY = agent_rec(ag)[1];
                const uint32_t bit0 = __float_as_uint(agent_rec(ag)[2].x);
                const float a = Ta + lane_a, bb = Tb + lane_b;
                float dx = fmaf(bb, UY.x, fmaf(a, FR.z, FR.x));
                float dy = fmaf(bb, FR.w, FR.y);
                float dz = fmaf(bb, UY.y, fmaf(a, UY.w, UY.z));
                dx = dx == 0.0f ? 1e-30f : dx;
                dy = dy == 0.0f ? 1e-30f : dy;
                dz = dz == 0.0f ? 1e-30f : dz;
                const float ix = fast_rcp(dx), iy = fast_rcp(dy), iz = fast_rcp(dz);
                dtx = fabsf(ix); dty = fabsf(iy); dtz = fabsf(iz);
                tab = abase | ((__float_as_uint(dx) >> 25) & 64u) | ((__float_as_uint(dy) >> 24) & 128u) | ((__float_as_uint(dz) >> 23) & 256u);
                float qx, qy, qz, ex, ey, ez, kx, kz;
                int sx, sy, sz;
                uint32_t at;
                asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=f"(qx), "=f"(qz), "=r"(sx), "=r"(sz) : "r"(tab));
                asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4+" MV_TAB_SKIP "];" : "=f"(ex), "=f"(ez), "=f"(ey), "=r"(at) : "r"(tab));
                asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4+" MV_TAB_SKIP2 "];" : "=f"(kx), "=f"(kz), "=f"(qy), "=r"(sy) : "r"(tab));
                const bool ngx = dx < 0.0f, ngy = dy < 0.0f, ngz = dz < 0.0f;
                float t0x, t0y, t0z, t_exit;
                t_hit = 0.0f;
                pos = 0; bit = bit0; row = kNoRow;
                if (!COLW) plane = __float_as_uint(agent_rec(ag)[5].w);
                if (cam_in) {
                    // (crossing times are sums: the exit time is pulled in by the rounding that can pile up in them)
                    t0x = qx * dtx;
                    t0y = qy * dty;
                    t0z = qz * dtz;
                    const int cx = (int)floorf(Px), cy = (int)floorf(Py), cz = (int)floorf(Pz);
                    t_exit = min3f(fmaf((float)(ngx ? cx - ilox : ihix - 1 - cx), dtx, t0x), fmaf((float)(ngy ? cy - iloy : ihiy - 1 - cy), dty, t0y),
                                   fmaf((float)(ngz ? cz - iloz : ihiz - 1 - cz), dtz, t0z)) * p.exit_scale;
                    // the first stretch, as in the block above
                    const float ts = min3f(ex * dtx, ez * dtz, ey * dty);
                    const float nx = __fadd_rd(fmaf(ts, fabsf(dx), kx), 8388608.0f), nz = __fadd_rd(fmaf(ts, fabsf(dz), kz), 8388608.0f);
                    pos = at + __float_as_uint(nx) * (uint32_t)sx + __float_as_uint(nz) * (uint32_t)sz;
                    if (nx > 8388608.0f) t0x = fmaf(nx - 8388609.0f, dtx, t0x + dtx);
                    if (nz > 8388608.0f) t0z = fmaf(nz - 8388609.0f, dtz, t0z + dtz);
                    if (aflags & kAgentFilled) { row = inside_row; t_exit = -kInf; }
                } else {
                    // eye outside the occupied box: clip the ray to it, start in the entry cell
                    const float x1 = (lo.x - Px) * ix, x2 = (hi.x - Px) * ix;
                    const float y1 = (lo.y - Py) * iy, y2 = (hi.y - Py) * iy;
                    const float z1 = (lo.z - Pz) * iz, z2 = (hi.z - Pz) * iz;
                    const float nrx = fminf(x1, x2), nry = fminf(y1, y2), nrz = fminf(z1, z2);
                    const float tn = max3f(nrx, nry, nrz);
                    const float tf = min3f(fmaxf(x1, x2), fmaxf(y1, y2), fmaxf(z1, z2));
                    const bool alive = any && (tn <= tf) && (tf > 0.0f);
                    const int eaxis = tn < 0.0f ? -1 : (nrx == tn ? 0 : (nry == tn ? 1 : 2));
                    t_hit = alive ? fmaxf(tn, 0.0f) : 0.0f;
                    int cx = min(max((int)floorf(fmaf(t_hit, dx, Px)), ilox), ihix - 1);
                    int cy = min(max((int)floorf(fmaf(t_hit, dy, Py)), iloy), ihiy - 1);
                    int cz = min(max((int)floorf(fmaf(t_hit, dz, Pz)), iloz), ihiz - 1);
                    if (eaxis == 0) cx = ngx ? ihix - 1 : ilox;
                    if (eaxis == 1) cy = ngy ? ihiy - 1 : iloy;
                    if (eaxis == 2) cz = ngz ? ihiz - 1 : iloz;
                    if (!alive) { cx = cy = cz = 0; }
                    pos = cell_pos(cx, cy, cz);
                    plane = cell_plane(cy);
                    bit = 1u << (cy - plane_begin(plane));
                    t0x = ((float)(cx + (ngx ? 0 : 1)) - Px) * ix;
                    t0y = ((float)(cy + (ngy ? 0 : 1)) - Py) * iy;
                    t0z = ((float)(cz + (ngz ? 0 : 1)) - Pz) * iz;
                    t_exit = min3f(fmaf(ngx ? (float)(cx - ilox) : (float)(ihix - 1 - cx), dtx, t0x),
                                   fmaf(ngy ? (float)(cy - iloy) : (float)(ihiy - 1 - cy), dty, t0y),
                                   fmaf(ngz ? (float)(cz - iloz) : (float)(ihiz - 1 - cz), dtz, t0z)) * p.exit_scale;
                    const bool filled = alive && voxel_filled(p.lay, occ, cx, cy, cz);
                    // entered through the box face of axis eaxis, or the eye is inside a solid
                    if (filled) {
                        if (eaxis < 0) row = inside_row;
                        else asm volatile("ld.shared.u32 %0, [%1+" MV_TAB_ROW "];" : "=r"(row) : "r"(tab + (eaxis == 0 ? 0u : (eaxis == 1 ? 8u : 4u))));
                    }
                    if (!alive || filled) t_exit = -kInf;
                }
#define MV_DDA_IO                                                                                         \
                    : "+r"(pos), "+r"(bit), "+f"(t_hit), "+r"(row), "+r"(plane)                                     \
                    : "f"(t0x), "f"(t0y), "f"(t0z), "f"(dtx), "f"(dty), "f"(dtz), "r"(sx), "r"(sy), "r"(sz), "f"(t_exit), \
                      "r"(tab), "r"(plane_end), "r"(p.lay.occ_plane), "r"(guards), "l"(env_block)                     \
                    : "memory"
#define MV_DDA_IN                                                                                         \
                    " mov.b32 pos, %0;\n mov.b32 bit, %1;\n mov.f32 thit, %2;\n mov.b32 q, %4;\n"                  \
                    " mov.f32 tx, %5;\n mov.f32 ty, %6;\n mov.f32 tz, %7;\n mov.f32 dtx, %8;\n mov.f32 dty, %9;\n"   \
                    " mov.f32 dtz, %10;\n mov.b32 sx, %11;\n mov.b32 sy, %12;\n mov.b32 sz, %13;\n mov.f32 texit, %14;\n" \
                    " mov.b32 guard, %16;\n mov.s32 it, " MV_STEP_BUDGET ";\n mov.b64 gbase, %19;\n"
// (a walk that ran out or left the box may stand at a plane's end all the same: only one that entered it goes on)
#define MV_DDA_CROSS_GENERAL(LOAD)                                                                        \
                    " @!ph bra MV_DDA_DONE;\n"                                                                   \
                    MV_DDA_CROSS("%16", "%17", "%18", " @ph bra MV_DDA_BEYOND;\n", "", LOAD)                     \
                    " bra MV_DDA_END;\n"                                                                         \
                    "MV_DDA_BEYOND:\n"                                                                           \
                    " setp.ne.u32 ph, 0, 0;\n"                                                                   \
                    "MV_DDA_END:\n"
#define MV_DDA_OUTS                                                                                       \
                    " selp.u32 a, 8, 4, py;\n selp.u32 a, 0, a, px;\n add.u32 a, a, %15;\n"                        \
                    " @ph ld.shared.u32 %3, [a+" MV_TAB_ROW "];\n mov.b32 %0, pos;\n mov.b32 %1, bit;\n mov.f32 %2, thit;\n mov.b32 %4, q;\n"
                if constexpr (COLW) {
                    asm volatile("{\n" MV_DDA_DECL MV_DDA_IN MV_DDA_LOOP(MV_DDA_STEP_COLW) MV_DDA_OUTS "}\n" MV_DDA_IO);
                } else if constexpr (staged) {
                    asm volatile("{\n" MV_DDA_DECL MV_DDA_IN MV_DDA_LOOP(MV_DDA_STEP_PLANE_SHARED) MV_DDA_CROSS_GENERAL(MV_DDA_LOAD_SHARED) MV_DDA_OUTS "}\n" MV_DDA_IO);
                } else {
                    asm volatile("{\n" MV_DDA_DECL MV_DDA_IN MV_DDA_LOOP(MV_DDA_STEP_PLANE_GLOBAL) MV_DDA_CROSS_GENERAL(MV_DDA_LOAD_GLOBAL) MV_DDA_OUTS "}\n" MV_DDA_IO);
                }
#undef MV_DDA_IO
#undef MV_DDA_IN
#undef MV_DDA_CROSS_GENERAL
#undef MV_DDA_OUTS
                if (row == kNoRow) t_hit = kInf;          // no voxel hit
                finish_tile(abase + mask_p, tile_px, pos, bit, plane, row, tab, 0u, t_hit, dtx, dty, dtz);
            }
        }
    }
}

}  // namespace mv
