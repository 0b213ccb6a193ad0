// The seeded scene generators of the package's scenes.py on the device: the same arrays, bit for bit.  Values come from
// a counter-based integer hash, so every cell, box and camera is worked out on its own; what has an order there (the
// tallest rectangle of a cell, the last pillar, the highest scores) is a maximum here.  Floating point is the
// generator's: double, every operation rounded on its own, then one rounding to float.  Bound by the grid bytes written:
// 512 worlds of 128x32x128 (268 MB) with their boxes and cameras in 0.25 ms; as torch operations 7.2 ms, a hundred launches
// over 64-bit tensors of every rectangle's cells.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace mv {

constexpr int kSceneThreads = 256, kEntityThreads = 512;
constexpr int kWorldSegments = 0, kWorldRooms = 1, kWorldColumns = 2;

struct SceneArgs {
    unsigned long long seed;
    int world, gx, gy, gz, palette;
    int count, pitch, pillars;                         // rectangles, or wall lines with their pitch and pillars
    int agents, boxes, bodies, max_boxes, step;
    int cam_y_is_fixed;
    float cam_y;
    int env_count;
    const int64_t *env;                                // [env_count] seeded scene ids
};

__device__ __forceinline__ unsigned long long scene_mix(unsigned long long x)
{
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}

// One stream of the generator for one environment.
struct SceneRng {
    unsigned long long k;
    __device__ __forceinline__ SceneRng(unsigned long long seed, int stream, long long env)
    {
        const unsigned long long base = seed * 0x9E3779B97F4A7C15ull + (unsigned long long)stream * 0xD1B54A32D192ED03ull;
        k = scene_mix((unsigned long long)env * 0x9E3779B97F4A7C15ull + base) + (unsigned long long)stream;
    }
    __device__ __forceinline__ uint32_t bits(unsigned long long idx) const
    {
        return (uint32_t)(scene_mix(k + idx * 0x94D049BB133111EBull) >> 32);
    }
    __device__ __forceinline__ double uniform(unsigned long long idx) const { return __dmul_rn((double)bits(idx), 1.0 / 4294967296.0); }
    __device__ __forceinline__ int range(unsigned long long idx, int lo, int hi) const
    {
        return lo + (int)(((long long)bits(idx) * (long long)(hi - lo + 1)) >> 32);
    }
};

// Columns and wall segments: a thread per rectangle leaves height * 256 + material in every cell it covers, the largest
// wins.  `keys` (the height array, zeroed before) is rewritten as heights by scene_expand_kernel.
__global__ void __launch_bounds__(kSceneThreads) scene_rects_kernel(const SceneArgs a, unsigned long long *__restrict__ keys)
{
    const long long gid = (long long)blockIdx.x * kSceneThreads + threadIdx.x;
    const int e = (int)(gid / a.count), r = (int)(gid - (long long)e * a.count);
    if (e >= a.env_count) return;
    const long long env = a.env[e];
    const bool thin = a.world == kWorldSegments;
    const int side = thin ? 8 : 6, hmin = thin ? 2 : 1, hmax = thin ? a.gy - 2 : 12;
    auto pick = [&](int stream, int lo, int hi) { return SceneRng(a.seed, stream, env).range((unsigned long long)r, lo, hi); };
    const int x0 = pick(10, 0, a.gx - 1), z0 = pick(11, 0, a.gz - 1);
    int w = pick(12, 1, side), d = pick(13, 1, side);
    if (thin) { if (pick(16, 0, 1) == 1) d = 1; else w = 1; }
    const long long key = (long long)pick(14, hmin, hmax) * 256 + pick(15, 1, a.palette - 1);
    if (key <= 0) return;
    for (int z = z0; z < min(z0 + d, a.gz); ++z)
        for (int x = x0; x < min(x0 + w, a.gx); ++x)
            atomicMax(keys + ((size_t)e * a.gz + z) * a.gx + x, (unsigned long long)key);
}

// Rooms: floor plan of border, wall lines with doors, and pillars; one CTA per environment.  Shared memory: positions and
// materials of the lines (two axes), each axis sorted, and the materials by coordinate.
__global__ void __launch_bounds__(kSceneThreads) scene_rooms_kernel(const SceneArgs a, unsigned long long *__restrict__ keys)
{
    extern __shared__ int s_room[];
    const int e = blockIdx.x, n = a.count, gx = a.gx, gz = a.gz, tid = threadIdx.x;
    const long long env = a.env[e];
    int *s_pos = s_room, *s_sorted = s_room + 2 * n, *s_m = s_room + 4 * n;          // [axis][line]; s_m: by x, then by z
    unsigned long long *map = keys + (size_t)e * gx * gz;
    const int border = SceneRng(a.seed, 24, env).range(0, 1, a.palette - 1);
    for (int i = tid; i < gx + gz; i += kSceneThreads) s_m[i] = 0;
    for (int i = tid; i < 2 * n; i += kSceneThreads) {
        const int axis = i / n, l = i - axis * n, size = axis ? gz : gx;
        s_pos[i] = min(max(a.pitch * (l + 1) + SceneRng(a.seed, 20 + axis, env).range(l, -2, 2), 2), size - 3);
    }
    __syncthreads();
    for (int i = tid; i < 2 * n; i += kSceneThreads) {
        const int axis = i / n, l = i - axis * n, p = s_pos[i];
        int rank = 0;
        bool last = true;                                         // (of several lines in one place the last one's material counts)
        for (int j = 0; j < n; ++j) {
            const int q = s_pos[axis * n + j];
            rank += q < p || (q == p && j < l);
            if (q == p && j > l) last = false;
        }
        s_sorted[axis * n + rank] = p;
        if (last && p >= 0 && p < (axis ? gz : gx)) s_m[axis * gx + p] = SceneRng(a.seed, 22 + axis, env).range(l, 1, a.palette - 1);
    }
    __syncthreads();
    for (int c = tid; c < gx * gz; c += kSceneThreads) {
        const int z = c / gx, x = c - z * gx;
        int m = s_m[x] > 0 ? s_m[x] : s_m[gx + z];
        if (m == 0 && (x == 0 || x == gx - 1 || z == 0 || z == gz - 1)) m = border;
        map[c] = (unsigned long long)m;
    }
    __syncthreads();
    // doors: two cells of every stretch of a line between crossing lines, if it has two
    for (int i = tid; i < 2 * n * (n + 1); i += kSceneThreads) {
        const int axis = i / (n * (n + 1)), r = i - axis * n * (n + 1), l = r / (n + 1), seg = r - l * (n + 1);
        const int *cross = s_sorted + (1 - axis) * n;
        const int size = axis ? gx : gz, lo = seg ? cross[seg - 1] : 0, hi = seg < n ? cross[seg] : size - 1;
        const int room = max(hi - lo - 1, 0);
        if (room < 2) continue;
        const double u = SceneRng(a.seed, 26 + axis, env).uniform((unsigned long long)(l * 16 + seg));
        const int d0 = lo + 1 + (int)__dmul_rn(u, (double)max(room - 1, 1));
        const int line = s_pos[axis * n + l];
        for (int k = 0; k < 2; ++k) {
            const int along = min(d0 + k, size - 2);
            map[axis ? line * gx + along : along * gx + line] = 0;
        }
    }
    __syncthreads();
    if (tid == 0) map[0] = (unsigned long long)border;
    __syncthreads();
    for (int i = tid; i < a.pillars; i += kSceneThreads) {
        const int x = SceneRng(a.seed, 28, env).range(i, 1, gx - 2), z = SceneRng(a.seed, 29, env).range(i, 1, gz - 2);
        const int m = SceneRng(a.seed, 30, env).range(i, 1, a.palette - 1);
        atomicMax(map + z * gx + x, 1ull << 40 | (unsigned long long)i << 8 | (unsigned long long)m);
    }
    __syncthreads();
    for (int c = tid; c < gx * gz; c += kSceneThreads) {
        const unsigned long long m = map[c] & 255u;
        map[c] = m ? (unsigned long long)(a.gy - 1) << 8 | m : 0ull;
    }
}

// Keys to heights and to the grid: a thread writes four columns, a warp whole 128-byte runs of every layer.  The palettes
// ride in the same launch.
__global__ void __launch_bounds__(kSceneThreads) scene_expand_kernel(const SceneArgs a, unsigned long long *__restrict__ keys,
                                                                     uint8_t *__restrict__ grid, uint8_t *__restrict__ palette,
                                                                     long long column_ctas)
{
    if ((long long)blockIdx.x >= column_ctas) {
        const long long i = ((long long)blockIdx.x - column_ctas) * kSceneThreads + threadIdx.x;
        const int per = 3 * a.palette, e = (int)(i / per);
        if (e < a.env_count) palette[i] = (uint8_t)SceneRng(a.seed, 31, a.env[e]).range((unsigned long long)(i - (long long)e * per), 24, 255);
        return;
    }
    const int groups = a.gx / 4 * a.gz;
    const long long gid = (long long)blockIdx.x * kSceneThreads + threadIdx.x;
    const int e = (int)(gid / groups), r = (int)(gid - (long long)e * groups);
    if (e >= a.env_count) return;
    ulonglong2 *kp = reinterpret_cast<ulonglong2 *>(keys + (size_t)e * a.gx * a.gz) + 2 * (size_t)r;
    const ulonglong2 k01 = kp[0], k23 = kp[1];
    const unsigned long long k[4] = {k01.x, k01.y, k23.x, k23.y};
    kp[0] = make_ulonglong2(k[0] >> 8, k[1] >> 8);
    kp[1] = make_ulonglong2(k[2] >> 8, k[3] >> 8);
    int h[4];
    uint32_t m[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) { h[c] = (int)(k[c] >> 8); m[c] = (uint32_t)(k[c] & 255u) << (8 * c); }
    const uint32_t layer = (uint32_t)a.gx * a.gz / 4;
    uint32_t *dst = reinterpret_cast<uint32_t *>(grid + (size_t)e * a.gx * a.gy * a.gz) + r;
    dst[0] = (uint32_t)SceneRng(a.seed, 25, a.env[e]).range(0, 1, a.palette - 1) * 0x01010101u;
    for (int y = 1; y < a.gy; ++y) {
        uint32_t v = 0;
#pragma unroll
        for (int c = 0; c < 4; ++c) v |= y <= h[c] ? m[c] : 0u;
        dst[(size_t)y * layer] = v;
    }
}

// Movable boxes and cameras (and agents' bodies) of one environment per CTA; heights: [env_count][gz][gx].  Camera records go
// to cams[slot], slot = the position in the list or, if given, slots[position].  Few CTAs, so the pass over the columns would
// wait for one height after the other: eight are in flight per thread (164 worlds of 128x128 columns: 30 -> 20 us, with twice
// the threads).  KEYS: `heights` are still keys.
template <bool KEYS>
__device__ __forceinline__ void scene_entities(const SceneArgs &a, const long long *__restrict__ heights, const int32_t *__restrict__ slots,
                                               uint32_t *__restrict__ boxes, int32_t *__restrict__ counts, uint32_t *__restrict__ cams)
{
    __shared__ int s_n, s_ok[kEntityThreads / 32];
    __shared__ unsigned long long s_best[kEntityThreads / 32], s_pick;
    const int e = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int gx = a.gx, gy = a.gy, gz = a.gz, A = a.agents, cells = gx * gz;
    const long long env = a.env[e];
    const long long *of_env = heights + (size_t)e * cells;
    const auto height = [of_env](int c) { return KEYS ? of_env[c] >> 8 : of_env[c]; };
    uint32_t *out = boxes + (size_t)e * a.max_boxes * 8;
    auto bits_of = [](float f) { return __float_as_uint(f); };
    if (tid == 0) s_n = 0;
    for (int i = tid; i < a.max_boxes * 8; i += kEntityThreads) out[i] = 0u;
    __syncthreads();
    for (int b0 = 0; b0 < a.boxes; b0 += kEntityThreads) {             // the accepted boxes, in order
        const int b = b0 + tid;
        uint32_t rec[7];
        bool ok = false;
        if (b < a.boxes) {
            float size[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) size[c] = (float)__dadd_rn(0.3, __dmul_rn(0.7, SceneRng(a.seed, 40 + c, env).uniform(b)));
            const float cx = (float)__dadd_rn(0.5, __dmul_rn(SceneRng(a.seed, 43, env).uniform(b), (double)gx - 1.0));
            const float cz = (float)__dadd_rn(0.5, __dmul_rn(SceneRng(a.seed, 44, env).uniform(b), (double)gz - 1.0));
            const float hx = __fmul_rn(size[0], 0.5f), hz = __fmul_rn(size[2], 0.5f);
            const float lox = __fsub_rn(cx, hx), hix = __fadd_rn(cx, hx), loz = __fsub_rn(cz, hz), hiz = __fadd_rn(cz, hz);
            const int x0 = min(max((int)floorf(lox), 0), gx - 1), x1 = min(max((int)floorf(hix), 0), gx - 1);
            const int z0 = min(max((int)floorf(loz), 0), gz - 1), z1 = min(max((int)floorf(hiz), 0), gz - 1);
            const int top = 1 + (int)max(max(height(z0 * gx + x0), height(z0 * gx + x1)), max(height(z1 * gx + x0), height(z1 * gx + x1)));
            const float loy = (float)top, hiy = __fadd_rn(loy, size[1]);
            ok = top < gy - 1 && hiy <= (float)gy;
            rec[0] = bits_of(lox); rec[1] = bits_of(loy); rec[2] = bits_of(loz);
            rec[3] = bits_of(hix); rec[4] = bits_of(hiy); rec[5] = bits_of(hiz);
            rec[6] = (uint32_t)SceneRng(a.seed, 45, env).range(b, 1, a.palette - 1);
        }
        const unsigned vote = __ballot_sync(0xffffffffu, ok);
        if (lane == 0) s_ok[warp] = __popc(vote);
        __syncthreads();
        int at = s_n + __popc(vote & ((1u << lane) - 1u)), all = 0;
        for (int w = 0; w < kEntityThreads / 32; ++w) { if (w < warp) at += s_ok[w]; all += s_ok[w]; }
        if (ok)
#pragma unroll
            for (int i = 0; i < 7; ++i) out[at * 8 + i] = rec[i];
        __syncthreads();
        if (tid == 0) s_n += all;
        __syncthreads();
    }
    const int n_boxes = s_n;
    // cameras: the standable columns with the highest scores.  Key: score (0 where nobody can stand), then the lower cell.
    const SceneRng score(a.seed, 50 + 7 * a.step, env);
    const float inv_gx = 1.0f / (float)gx;                            // (exact below 2^21 cells: the row of c is never that close to the next)
    auto key_of = [&](int c, long long h) {
        const int z = (int)(((float)c + 0.5f) * inv_gx), x = c - z * gx;
        const bool stand = h + 1 < gy - 1 && x > 0 && x < gx - 1 && z > 0 && z < gz - 1;
        const unsigned long long s = stand ? 1ull + score.bits((unsigned long long)c) : 0ull;
        return s << 24 | (unsigned long long)(0xffffff - c);
    };
    auto block_max = [&](unsigned long long v) {
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) { const unsigned long long o = __shfl_xor_sync(0xffffffffu, v, s); v = o > v ? o : v; }
        if (lane == 0) s_best[warp] = v;
        __syncthreads();
        v = s_best[0];
#pragma unroll
        for (int w = 1; w < kEntityThreads / 32; ++w) v = s_best[w] > v ? s_best[w] : v;
        __syncthreads();
        return v;
    };
    unsigned long long head = 0;                                      // the best cell among those the thread owns
    for (int c0 = tid; c0 < cells; c0 += 8 * kEntityThreads) {
        long long h[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) h[i] = c0 + i * kEntityThreads < cells ? height(c0 + i * kEntityThreads) : 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int c = c0 + i * kEntityThreads;
            const unsigned long long k = c < cells ? key_of(c, h[i]) : 0ull;
            head = k > head ? k : head;
        }
    }
    for (int ag = 0; ag < A; ++ag) {
        const unsigned long long pick = block_max(head);
        if (head == pick) s_pick = (unsigned long long)tid;
        __syncthreads();
        const int owner = (int)s_pick, c = 0xffffff - (int)(pick & 0xffffffull);
        if (ag + 1 < A) {                                             // the owner's next best, looked for by everybody
            unsigned long long next = 0;
            for (int i = owner + tid * kEntityThreads; i < cells; i += kEntityThreads * kEntityThreads) {
                const unsigned long long k = key_of(i, height(i));
                if (k < pick && k > next) next = k;
            }
            next = block_max(next);
            if (tid == owner) head = next;
        }
        if (tid == 0) {
            const int cx = c % gx, cz = c / gx, cy = 1 + (int)height(c);
            const unsigned long long idx = (unsigned long long)(ag + 64 * a.step);
            double off[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) off[i] = __dadd_rn(0.1, __dmul_rn(0.8, SceneRng(a.seed, 60 + i, env).uniform(idx)));
            const float px = (float)__dadd_rn((double)cx, off[0]), pz = (float)__dadd_rn((double)cz, off[2]);
            const float py = a.cam_y_is_fixed ? __fadd_rn(a.cam_y, (float)(cy - 1)) : (float)__dadd_rn((double)cy, off[1]);
            const float yaw = (float)__dmul_rn(SceneRng(a.seed, 63, env).uniform(idx), 6.283185307179586);
            const float pitch = (float)__dmul_rn(__dsub_rn(SceneRng(a.seed, 64, env).uniform(idx), 0.5), 0.6);
            uint32_t *cam = cams + ((size_t)(slots ? slots[e] : e) * A + ag) * 6;
            cam[0] = bits_of(px); cam[1] = bits_of(py); cam[2] = bits_of(pz);
            cam[3] = bits_of(yaw); cam[4] = bits_of(pitch);
            cam[5] = (uint32_t)(a.bodies ? n_boxes + ag : -1);
            if (a.bodies) {
                uint32_t *o = out + (size_t)(n_boxes + ag) * 8;
                o[0] = bits_of(__fsub_rn(px, 0.25f)); o[1] = bits_of(__fsub_rn(py, 0.75f)); o[2] = bits_of(__fsub_rn(pz, 0.25f));
                o[3] = bits_of(__fadd_rn(px, 0.25f)); o[4] = bits_of(__fadd_rn(py, 0.25f)); o[5] = bits_of(__fadd_rn(pz, 0.25f));
                o[6] = (uint32_t)SceneRng(a.seed, 65, env).range((unsigned long long)ag, 1, a.palette - 1);
            }
        }
        __syncthreads();
    }
    if (tid == 0) counts[e] = n_boxes + (a.bodies ? A : 0);
}

__global__ void __launch_bounds__(kEntityThreads) scene_entities_kernel(const SceneArgs a, const long long *__restrict__ heights,
                                                                       const int32_t *__restrict__ slots, uint32_t *__restrict__ boxes,
                                                                       int32_t *__restrict__ counts, uint32_t *__restrict__ cams)
{
    scene_entities<false>(a, heights, slots, boxes, counts, cams);
}

// Worlds from their keys straight into a batch: what scene_expand_kernel, scene_entities_kernel and the packing of an upload leave, without
// the grid's bytes in between, in one launch.  First a CTA per environment for boxes and cameras, which takes longest, beside them those
// that write the world store, then the palettes.  A thread of the store takes four columns, floor and one stack each: their occupancy words
// and 32 bytes of material at a time as one store, whole sectors; the floor fills the whole grid, so of the cell box only the height
// is looked for.  SLABS: every CTA of columns is `slabs` ones, each with every slabs-th 32 heights and plane (few high worlds, see
// mv_scene_upload).  163 worlds of 128x32x128: 67 us with their keys, which before went through grid bytes and an upload: 111.
template <bool SLABS>
__global__ void __launch_bounds__(kEntityThreads) scene_populate_kernel(const SceneArgs a, const unsigned long long *__restrict__ keys,
                                                                       const int32_t *__restrict__ env_index, uint32_t *__restrict__ boxes,
                                                                       int32_t *__restrict__ counts, uint32_t *__restrict__ cams,
                                                                       uint8_t *__restrict__ palette, unsigned char *__restrict__ env_blocks,
                                                                       uint8_t *__restrict__ mat, size_t mat_stride, EnvLayout lay,
                                                                       int *__restrict__ acc_all, int column_ctas, int slabs, uint32_t *__restrict__ status)
{
    if ((int)blockIdx.x < a.env_count) {
        scene_entities<true>(a, reinterpret_cast<const long long *>(keys), env_index, boxes, counts, cams);
        return;
    }
    const int n_slabs = SLABS ? slabs : 1, ctas_per_env = column_ctas * n_slabs;
    const int cta = (int)blockIdx.x - a.env_count, store_ctas = a.env_count * ctas_per_env;
    if (cta >= store_ctas) {
        const long long i = (long long)(cta - store_ctas) * kEntityThreads + threadIdx.x;
        const int per = 3 * a.palette, e = (int)(i / per);
        if (e < a.env_count) palette[i] = (uint8_t)SceneRng(a.seed, 31, a.env[e]).range((unsigned long long)(i - (long long)e * per), 24, 255);
        return;
    }
    __shared__ int s_top;
    const int e = cta / ctas_per_env, part = cta - e * ctas_per_env, slab = SLABS ? part / column_ctas : 0;
    const int r = (part - slab * column_ctas) * kEntityThreads + (int)threadIdx.x, row_groups = a.gx / 4;
    const size_t env = (size_t)env_index[e];
    unsigned char *blk = env_blocks + env * lay.stride;
    if (threadIdx.x == 0) s_top = 0;
    __syncthreads();
    int top = 0;                                                 // (of threads without columns too)
    if (r < row_groups * a.gz) {
        const ulonglong2 *kp = reinterpret_cast<const ulonglong2 *>(keys + (size_t)e * a.gx * a.gz) + 2 * (size_t)r;
        const ulonglong2 k01 = kp[0], k23 = kp[1];
        const unsigned long long k[4] = {k01.x, k01.y, k23.x, k23.y};
        // (ids are clamped to the palette as by an upload: the generator's begin with 1, also where there is one colour)
        uint32_t floor_mat = (uint32_t)SceneRng(a.seed, 25, a.env[e]).range(0, 1, a.palette - 1);
        const uint32_t cap = (uint32_t)(a.palette - 1);
        bool clamped = floor_mat > cap;
        floor_mat = min(floor_mat, cap);
        const int z = r / row_groups, x = 4 * (r - z * row_groups);
        const uint32_t col0 = column_index(lay, x, z), words = lay.occ_plane / 4;
        uint32_t *occ = reinterpret_cast<uint32_t *>(blk) + col0;
        uint8_t *dst = mat + env * mat_stride + ((size_t)col0 << lay.ysh);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint32_t id = (uint32_t)(k[c] & 255u), m = min(id, cap);
            clamped |= id > cap;
            // filled cells of the column from the floor up (a stack without material is none)
            const int n = id ? 1 + (int)min(k[c] >> 8, (unsigned long long)(a.gy - 1)) : 1;
            top = max(top, n);
            for (uint32_t q = slab; q < lay.planes; q += n_slabs) {
                const int in = min(max(n - plane_begin(q), 0), lay.planes == 1 ? 32 : (int)kPlaneHeights);
                occ[(size_t)q * words + c] = in == 32 ? 0xffffffffu : (1u << in) - 1u;
            }
            for (int y0 = 32 * slab; y0 < a.gy; y0 += 32 * n_slabs) {
                uint32_t w[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int in = min(max(n - y0 - 4 * i, 0), 4);              // bytes of this word that are filled
                    w[i] = m * 0x01010101u & (uint32_t)((1ull << (8 * in)) - 1ull);
                }
                if (y0 == 0) w[0] = (w[0] & ~0xffu) | floor_mat;
                store32(dst + ((size_t)c << lay.ysh) + y0, w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]);
            }
        }
        if (clamped) atomicOr(status, kFlagMaterial);
    }
    top = __reduce_max_sync(0xffffffffu, top);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_top, top);
    __syncthreads();
    if (threadIdx.x == 0) {                                     // (the accumulators as an upload uses and leaves them)
        int *acc = acc_all + env * kPackAccInts;
        atomicMax(acc + 4, s_top);
        __threadfence();
        if (atomicAdd(acc + 6, 1) == ctas_per_env - 1) {
            __threadfence();
            int *box = reinterpret_cast<int *>(blk + lay.count_off) + 1;
            box[0] = box[1] = box[2] = 0;
            box[3] = a.gx; box[4] = __ldcg(acc + 4); box[5] = a.gz; box[6] = 0;
            acc[4] = -1; acc[6] = 0;
        }
    }
}

// One step of the episode clocks of a batch (advance = 0: none, only the bars): t and episode advance, done says whose
// episode ended, and each agent's time-left bar (bar_rows rows, as long as the share that is left, whole pixels) goes to
// the overlay table (null: no bars).
__global__ void episode_clocks_kernel(int64_t *__restrict__ t, int64_t *__restrict__ episode, const int64_t *__restrict__ len,
                                      uint8_t *__restrict__ done, int envs, int agents, int advance, int width, int bar_rows,
                                      uint32_t bar_rgb, int4 *__restrict__ overlay, int32_t *__restrict__ overlay_count, int max_rects)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= envs) return;
    const int64_t n = len[e];
    int64_t now = t[e];
    if (advance) {
        const bool over = ++now >= n;
        if (over) { now = 0; episode[e] += 1; }
        t[e] = now;
        done[e] = over ? 1 : 0;
    }
    if (!overlay) return;
    const int64_t x1 = min(max(((int64_t)width * (n - now)) / max(n, (int64_t)1), (int64_t)0), (int64_t)width);
    for (int ag = 0; ag < agents; ++ag) {
        const size_t o = (size_t)e * agents + ag;
        overlay[o * max_rects] = make_int4(0, (int)x1 | bar_rows << 16, (int)bar_rgb, 0);
        overlay_count[o] = 1;
    }
}

}  // namespace mv
