// World-store and camera kernels: everything that turns the caller's arrays into the
// device-resident layout the render kernel stages (paper Section 3.3: geometry is prepared
// once per episode; Section 3.2: objects and cameras are state that changes every step).
#pragma once
#include "mv_device.cuh"
#include <type_traits>

namespace mv {

// Four 0/non-zero bytes of a word -> 4 bits.
__device__ __forceinline__ uint32_t nz_bits4(uint32_t v) {
    const uint32_t ones = __vcmpne4(v, 0u) & 0x01010101u;
    return (ones * 0x01020408u) >> 24;
}

// Eight 0/non-zero bytes (two words) -> 8 bits: a non-zero byte leaves 0x80, and a dot product with powers of two
// collects them.
__device__ __forceinline__ uint32_t nz_bits8(uint32_t a, uint32_t b)
{
    const uint32_t n0 = (((a & 0x7f7f7f7fu) + 0x7f7f7f7fu) | a) & 0x80808080u;
    const uint32_t n1 = (((b & 0x7f7f7f7fu) + 0x7f7f7f7fu) | b) & 0x80808080u;
    return __dp4a(n1, 0x80402010u, __dp4a(n0, 0x08040201u, 0u)) >> 7;
}

// One 32-byte store (32-byte aligned).
__device__ __forceinline__ void store32(void *dst, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t e, uint32_t f,
                                        uint32_t g, uint32_t h)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(a), "r"(b), "r"(c), "r"(d),
                 "r"(e), "r"(f), "r"(g), "r"(h) : "memory");
}

// 4 x 4 byte transpose: in[i] holds byte c of column c at height i; out[c] the four heights of column c.
__device__ __forceinline__ void transpose4x4(const uint32_t in[4], uint32_t out[4]) {
    const uint32_t a = __byte_perm(in[0], in[1], 0x5140), b = __byte_perm(in[2], in[3], 0x5140);   // c0h0 c0h1 c1h0 c1h1 | ..h2 h3
    const uint32_t c = __byte_perm(in[0], in[1], 0x7362), d = __byte_perm(in[2], in[3], 0x7362);   // c2h0 c2h1 c3h0 c3h1 | ..h2 h3
    out[0] = __byte_perm(a, b, 0x5410); out[1] = __byte_perm(a, b, 0x7632);
    out[2] = __byte_perm(c, d, 0x5410); out[3] = __byte_perm(c, d, 0x7632);
}

// Destination env of the e-th env of an upload: a contiguous range, or an index list.
__device__ __forceinline__ size_t upload_env(const int32_t *env_index, int env_begin, size_t e) {
    return env_index ? (size_t)env_index[e] : (size_t)env_begin + e;
}

// Per-env accumulators of an upload in flight: lo x,y,z, hi x,y,z (inclusive), CTAs done, pad.  Idle between uploads:
// lo = 2^30, hi = -1, done = 0 (the CTA that finishes an env puts them back).
constexpr int kPackAccInts = 8;
constexpr int kUploadThreads = 64;
constexpr int kUploadStages = 2;
constexpr int kUploadSmem = kUploadStages * 32 * kUploadThreads * 4;

// The fence around the columns of every env (see EnvLayout); grid columns keep their zeros.
__global__ void fence_kernel(unsigned char *env_blocks, EnvLayout lay, int gx, int gz, int num_envs)
{
    const int words = (int)(lay.occ_bytes / 4);
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long e = gid / words;
    if (e >= num_envs) return;
    const int w = (int)(gid - e * words), c = w % (int)(lay.occ_plane / 4) - 1, z = c < 0 ? -1 : c / (int)lay.pitch - 1;
    const int x = c - (z + 1) * (int)lay.pitch;
    if (z < 0 || z >= gz || x < 0 || x >= gx) reinterpret_cast<uint32_t *>(env_blocks + (size_t)e * lay.stride)[w] = 0xffffffffu;
}

__global__ void init_acc_kernel(int *acc, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, k = i % kPackAccInts;
    if (i < n) acc[i] = k < 3 ? 1 << 30 : (k < 6 ? -1 : 0);
}

struct UploadArgs {
    const uint8_t *grid;               // null: no grid in this upload
    const uint4 *boxes;                // null: no boxes
    const int32_t *counts;
    const uint8_t *palette_rgb;        // null: no palettes
    unsigned char *env_blocks;
    uint8_t *mat;
    size_t mat_stride;
    int *acc;                          // [E][kPackAccInts]
    uint32_t *status;
    const int32_t *env_index;          // destination envs, or null for the range from env_begin
    EnvLayout lay;
    int env_begin, env_count;
    int gx, gy, gz, max_boxes, palette;
    int words, tiles_per_env, tiles_per_cta, pack_ctas_per_env;     // tiles of 256 columns x 32 heights, `words` of them one above the other
    // CTAs [0, pack_ctas) pack, the next lut_ctas shade, the rest copy boxes
    unsigned pack_ctas, lut_ctas;
    int wait_polls;                    // bound of the wait for a tile's copies
    int skip_staging;                  // test hook: the last CTA of every env issues no copies, so its wait runs out
    double light[3], ambient;
};

// A CTA packs a few tiles of one env, a tile being 256 consecutive columns, 32 heights of them: each height is 256 bytes of
// the grid in a row, fetched by one bulk copy into shared memory, the next tile's while this one is packed (two
// buffers, twelve small CTAs per SM: about 190 KB per SM on the way without holding a register, and loads, packing and stores of different CTAs overlap).  A thread takes four
// neighbouring columns: four occupancy words and four columns of material bytes (ids clamped to the palette; what
// is not filled is never read, but comes out as 0), a column's 32 bytes as one 32-byte store, a whole sector.  Also
// grows the cell box [lo, hi) that contains every filled voxel of the env; the last CTA of an env writes it next to
// the box count (an empty grid gives lo > hi).  A CTA whose wait runs out counts like the others, so that the env's
// accumulators are idle again for the next upload.  512 envs of 128x32x128 (268 MB in, 302 MB out): 150 us, then 42 us to
// read the bits back for the bounds, with four-byte loads into registers and 16-byte stores; 114 us now (5.0 TB/s).
template <bool TALL>
__device__ __forceinline__ void pack_columns(const UploadArgs &p)
{
    extern __shared__ __align__(128) uint32_t s_tile[];       // [kUploadStages][32][kUploadThreads]
    __shared__ uint64_t s_bar[kUploadStages];
    __shared__ int s_acc[6], s_last, s_bad;
    const int xg_n = p.gx / 4;                                // groups of four columns per row
    const int e = (int)(blockIdx.x / (unsigned)p.pack_ctas_per_env), part = (int)(blockIdx.x - (unsigned)e * p.pack_ctas_per_env);
    const size_t env = upload_env(p.env_index, p.env_begin, (size_t)e);
    unsigned char *blk = p.env_blocks + env * p.lay.stride;
    const int groups = xg_n * p.gz;                           // of four columns, per 32 heights
    const size_t layer = (size_t)p.gz * p.gx;
    const uint8_t *grid = p.grid + (size_t)e * layer * p.gy;
    const int tile_begin = part * p.tiles_per_cta, tile_end = min(tile_begin + p.tiles_per_cta, p.tiles_per_env);
    if (threadIdx.x < kUploadStages) mbar_init(&s_bar[threadIdx.x], 1);
    if (threadIdx.x < 6) s_acc[threadIdx.x] = threadIdx.x < 3 ? 1 << 30 : -1;
    if (threadIdx.x == 6) s_bad = 0;
    __syncthreads();
    const bool withheld = p.skip_staging && part == p.pack_ctas_per_env - 1;
    // the tile to pack next and the one to fetch next: which 32 heights of a column, and its first group of columns
    int wq = TALL ? tile_begin % p.words : 0, r0 = (TALL ? tile_begin / p.words : tile_begin) * kUploadThreads;
    int fetch_wq = wq, fetch_r0 = r0;
    auto advance = [&](int &w, int &r) { if (TALL && ++w < p.words) return; w = 0; r += kUploadThreads; };
    auto fetch = [&](int tile) {                              // one warp
        if (withheld) return;
        const int stage = (tile - tile_begin) % kUploadStages, heights = min(p.gy - 32 * fetch_wq, 32);
        const uint32_t bytes = 4u * (uint32_t)min(groups - fetch_r0, kUploadThreads);
        if (threadIdx.x == 0) mbar_expect_tx(&s_bar[stage], bytes * (uint32_t)heights);
        __syncwarp();
        if ((int)threadIdx.x < heights)
            bulk_load(s_tile + (size_t)(stage * 32 + (int)threadIdx.x) * kUploadThreads,
                      grid + (size_t)(32 * fetch_wq + (int)threadIdx.x) * layer + 4 * (size_t)fetch_r0, bytes, &s_bar[stage]);
        advance(fetch_wq, fetch_r0);
    };
    if (threadIdx.x < 32)
        for (int t = tile_begin; t < min(tile_begin + kUploadStages, tile_end); ++t) fetch(t);
    int lo[3] = {1 << 30, 1 << 30, 1 << 30}, hi[3] = {-1, -1, -1};
    uint32_t clamped = 0, below[4] = {0, 0, 0, 0};            // the columns' 32 heights below these
    // A plane's 31 heights begin q heights down in the tile below.  Where that tile is another CTA's, these heights are read here, too:
    // a load each, all in flight beside the copies.  (With all tiles of a column in one CTA a few tall worlds leave the GPU idle:
    // one of 16x1024x16 74 us, 7.1 like this; one of 64x64x64 8.6 and 6.5; 256 of 64x1024x64 659 and 458.)
    auto read_below = [&](auto most) {
        constexpr int N = decltype(most)::value;
        const uint8_t *src = grid + (size_t)(32 * wq - 1) * layer + 4 * (size_t)min(r0 + (int)threadIdx.x, groups - 1);
        uint32_t v[N], eight = 0;
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = i < wq ? *reinterpret_cast<const uint32_t *>(src - (size_t)i * layer) : 0u;
#pragma unroll
        for (int i = 0; i < N; ++i) {                         // byte c of `eight`: eight heights of column c, the highest in bit 7
            eight |= (((((v[i] & 0x7f7f7f7fu) + 0x7f7f7f7fu) | v[i]) & 0x80808080u) >> (i & 7));
            if ((i & 7) < 7) continue;
#pragma unroll
            for (int c = 0; c < 4; ++c) below[c] |= (eight >> (8 * c) & 0xffu) << (31 - i);
            eight = 0;
        }
    };
    if (TALL && wq > 8) read_below(std::integral_constant<int, 32>());
    else if (TALL && wq > 0) read_below(std::integral_constant<int, 8>());
    for (int tile = tile_begin; tile < tile_end; ++tile, advance(wq, r0)) {
        const int n = tile - tile_begin, stage = n % kUploadStages;
        const uint32_t parity = (uint32_t)(n / kUploadStages) & 1u;
        const uint32_t *mine = s_tile + (size_t)stage * 32 * kUploadThreads + threadIdx.x;
        if (!mbar_wait_bounded(&s_bar[stage], parity, p.wait_polls)) s_bad = 1;
        __syncthreads();
        if (s_bad) {                                          // (as in the render kernel: report, drain, pack no more)
            if (threadIdx.x == 0) {
                atomicOr(p.status, kFlagTimeout);
                for (int m = n; m < min(n + kUploadStages, tile_end - tile_begin) && !withheld; ++m)
                    mbar_wait_bounded(&s_bar[m % kUploadStages], (uint32_t)(m / kUploadStages) & 1u, kDrainPolls);
            }
            break;
        }
        const int r = r0 + (int)threadIdx.x, heights = min(p.gy - 32 * wq, 32);
        uint32_t col[4][8], bits[4] = {0, 0, 0, 0};
        const uint32_t cap = (uint32_t)(p.palette - 1);
        // a byte exceeds cap iff bit 7 of ((low seven bits + add) combined with the byte) is set
        const uint32_t add = (127u - (cap & 127u)) * 0x01010101u, big_cap = cap >= 128u ? 0xffffffffu : 0u;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            uint32_t v[16], over = 0;
#pragma unroll
            for (int i = 0; i < 16; ++i)
                v[i] = 16 * half + i < heights ? mine[(16 * half + i) * kUploadThreads] : 0u;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const uint32_t s = (v[i] & 0x7f7f7f7fu) + add;
                over |= big_cap ? (s & v[i]) : (s | v[i]);
            }
            // occupancy is decided before clamping (with one palette entry every id becomes 0)
            uint32_t q4[4][4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t t[4];
                transpose4x4(v + 4 * q, t);
#pragma unroll
                for (int c = 0; c < 4; ++c) q4[c][q] = t[c];
            }
#pragma unroll
            for (int c = 0; c < 4; ++c)
                bits[c] |= (nz_bits8(q4[c][0], q4[c][1]) | nz_bits8(q4[c][2], q4[c][3]) << 8) << (16 * half);
            if ((over & 0x80808080u) && r < groups) {          // (beyond the env the buffer holds whatever it held)
                clamped = 1u;
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int q = 0; q < 4; ++q) q4[c][q] = __vminu4(q4[c][q], cap * 0x01010101u);
            }
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int q = 0; q < 4; ++q) col[c][4 * half + q] = q4[c][q];
        }
        __syncthreads();                                      // the buffer has been read
        if (threadIdx.x < 32 && tile + kUploadStages < tile_end) fetch(tile + kUploadStages);
        if (r >= groups) continue;
        const int z = r / xg_n, xg = r - z * xg_n;
        const uint32_t col0 = column_index(p.lay, 4 * xg, z);
        uint8_t *mdst = p.mat + env * p.mat_stride + ((size_t)col0 << p.lay.ysh) + 32 * wq;
        uint32_t *occ = reinterpret_cast<uint32_t *>(blk);
#pragma unroll
        for (int c = 0; c < 4; ++c)
            store32(mdst + ((size_t)c << p.lay.ysh), col[c][0], col[c][1], col[c][2], col[c][3], col[c][4], col[c][5],
                    col[c][6], col[c][7]);
        // (the last tile also fills the planes above its own)
        const uint32_t words = p.lay.occ_plane / 4;
        if (!TALL) {
#pragma unroll
            for (int c = 0; c < 4; ++c) occ[col0 + c] = bits[c];
        } else {
            for (int q = wq; q == wq || (wq == p.words - 1 && q < (int)p.lay.planes); ++q)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const uint32_t off = (kPlaneHeights * (uint32_t)q) & 31u;
                    const uint32_t w = q == 0 ? bits[c] : q == wq ? __funnelshift_r(below[c], bits[c], off) : bits[c] >> off;
                    occ[(size_t)q * words + col0 + c] = w & ~kPlaneEnd;
                }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) below[c] = bits[c];
        const uint32_t any = bits[0] | bits[1] | bits[2] | bits[3];
        if (any) {
            lo[0] = min(lo[0], 4 * xg + (bits[0] ? 0 : bits[1] ? 1 : bits[2] ? 2 : 3));
            hi[0] = max(hi[0], 4 * xg + (bits[3] ? 3 : bits[2] ? 2 : bits[1] ? 1 : 0));
            lo[1] = min(lo[1], 32 * wq + __ffs(any) - 1); hi[1] = max(hi[1], 32 * wq + 31 - __clz(any));
            lo[2] = min(lo[2], z); hi[2] = max(hi[2], z);
        }
    }
    if (clamped) atomicOr(p.status, kFlagMaterial);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int l = __reduce_min_sync(0xffffffffu, lo[c]), h = __reduce_max_sync(0xffffffffu, hi[c]);
        if ((threadIdx.x & 31) == 0) { atomicMin(&s_acc[c], l); atomicMax(&s_acc[3 + c], h); }
    }
    __syncthreads();
    int *acc = p.acc + env * kPackAccInts;
    if (threadIdx.x < 3) atomicMin(acc + threadIdx.x, s_acc[threadIdx.x]);
    else if (threadIdx.x < 6) atomicMax(acc + threadIdx.x, s_acc[threadIdx.x]);
    if (threadIdx.x < 32) {
        __threadfence();
        __syncwarp();
        if (threadIdx.x == 0) s_last = atomicAdd(acc + 6, 1) == p.pack_ctas_per_env - 1;
        __syncwarp();
        if (s_last) {
            __threadfence();
            int *dst = reinterpret_cast<int *>(blk + p.lay.count_off);
            if (threadIdx.x < 6) {
                dst[1 + threadIdx.x] = __ldcg(acc + threadIdx.x) + (threadIdx.x < 3 ? 0 : 1);
                acc[threadIdx.x] = threadIdx.x < 3 ? 1 << 30 : -1;
            }
            if (threadIdx.x == 6) { dst[7] = 0; acc[6] = 0; }
        }
    }
}

// Shaded colour table per env: lut[face][m] = RGBX of floor(palette*I_face + 0.5), in double.
__device__ __forceinline__ void shade_palettes(const UploadArgs &p, unsigned cta)
{
    const long long gid = (long long)cta * kUploadThreads + threadIdx.x;     // (1.2 million envs of 256 colours are 2^31 entries)
    const int P = p.palette, e = (int)(gid / (kFaces * P)), r = (int)(gid - (long long)e * (kFaces * P));
    if (e >= p.env_count) return;
    const int f = r / P, m = r - f * P;
    double I = p.ambient;
    if (f < 6) {
        const double lx = p.light[0], ly = p.light[1], lz = p.light[2];
        const double n = sqrt(__dadd_rn(__dadd_rn(__dmul_rn(lx, lx), __dmul_rn(ly, ly)), __dmul_rn(lz, lz)));
        const double comp = (f >> 1) == 0 ? lx : ((f >> 1) == 1 ? ly : lz);
        double l = comp / n;
        if (!(f & 1)) l = -l;                       // even faces have the negative normal
        l = l > 0.0 ? l : 0.0;
        I = __dadd_rn(p.ambient, __dmul_rn(__dsub_rn(1.0, p.ambient), l));
    }
    const uint8_t *pc = p.palette_rgb + ((size_t)e * P + m) * 3;
    uint32_t out = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        double v = floor(__dadd_rn(__dmul_rn((double)pc[c], I), 0.5));
        v = v > 255.0 ? 255.0 : v;
        out |= (uint32_t)v << (8 * c);
    }
    uint32_t *lut = reinterpret_cast<uint32_t *>(p.env_blocks + upload_env(p.env_index, p.env_begin, (size_t)e) * p.lay.stride + p.lay.lut_off);
    lut[f * P + m] = out;
}

// Box lists into the env blocks; material ids and counts are clamped.
__device__ __forceinline__ void copy_boxes(const UploadArgs &p, unsigned cta)
{
    const long long gid = (long long)cta * kUploadThreads + threadIdx.x;
    const int per_env = p.max_boxes + 1, e = (int)(gid / per_env), b = (int)(gid - (long long)e * per_env);
    if (e >= p.env_count) return;
    unsigned char *blk = p.env_blocks + upload_env(p.env_index, p.env_begin, (size_t)e) * p.lay.stride;
    if (b == p.max_boxes) {
        int n = p.counts[e];
        if (n < 0 || n > p.max_boxes) { n = n < 0 ? 0 : p.max_boxes; atomicOr(p.status, kFlagBoxCount); }
        *reinterpret_cast<int *>(blk + p.lay.count_off) = n;
        return;
    }
    const uint4 *src = p.boxes + ((size_t)e * p.max_boxes + b) * 2;
    uint4 lo = src[0], hi = src[1];
    if (hi.z >= (uint32_t)p.palette) { hi.z = p.palette - 1; atomicOr(p.status, kFlagMaterial); }
    uint4 *dst = reinterpret_cast<uint4 *>(blk + p.lay.box_off) + 2 * b;
    dst[0] = lo;
    dst[1] = hi;
}

// Everything one upload brings, in one launch: the CTAs are dealt to the three jobs by number.
__global__ void __launch_bounds__(kUploadThreads, 12) upload_kernel(const UploadArgs p)
{
    launch_dependents();
    wait_for_previous();
    if (blockIdx.x < p.pack_ctas) p.words == 1 ? pack_columns<false>(p) : pack_columns<true>(p);
    else if (blockIdx.x < p.pack_ctas + p.lut_ctas) shade_palettes(p, blockIdx.x - p.pack_ctas);
    else copy_boxes(p, blockIdx.x - p.pack_ctas - p.lut_ctas);
}

// Camera -> ray basis, evaluated in double and rounded to float:
// F = (cp*sy, sp, cp*cy), R = (cy, 0, -sy), U = (-sp*sy, cp, -sp*cy); Rs = R*kr, Us = U*ku
// with kr = tan(hfov/2)/W and ku = (tan(hfov/2)*H/W)/H computed on the host in double.
__device__ __forceinline__ void write_camrec(CamRec *out, float px, float py, float pz, float yaw, float pitch,
                                             int self_box, double kr, double ku, uint32_t *status)
{
    CamRec r;
    r.self_box = self_box;
    r.pad[0] = r.pad[1] = 0;
    const bool ok = isfinite(px) && isfinite(py) && isfinite(pz) && isfinite(yaw) && isfinite(pitch);
    r.flags = ok ? 0u : kFlagBadCamera;
    double sy, cy, sp, cp;
    sincos((double)(ok ? yaw : 0.0f), &sy, &cy);
    sincos((double)(ok ? pitch : 0.0f), &sp, &cp);
    r.P[0] = px; r.P[1] = py; r.P[2] = pz;
    r.F[0] = (float)__dmul_rn(cp, sy); r.F[1] = (float)sp; r.F[2] = (float)__dmul_rn(cp, cy);
    r.Rs[0] = (float)__dmul_rn(cy, kr); r.Rs[1] = (float)__dmul_rn(0.0, kr); r.Rs[2] = (float)__dmul_rn(-sy, kr);
    r.Us[0] = (float)__dmul_rn(__dmul_rn(-sp, sy), ku); r.Us[1] = (float)__dmul_rn(cp, ku);
    r.Us[2] = (float)__dmul_rn(__dmul_rn(-sp, cy), ku);
    *out = r;
    if (!ok) atomicOr(status, kFlagBadCamera);
}

__global__ void camera_kernel(const int32_t *cams, CamRec *out, int num_obs,
                              double kr, double ku, uint32_t *status)
{
    launch_dependents();
    wait_for_previous();
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= num_obs) return;
    const int32_t *c = cams + (size_t)o * 6;
    write_camrec(out + o, __int_as_float(c[0]), __int_as_float(c[1]), __int_as_float(c[2]),
                 __int_as_float(c[3]), __int_as_float(c[4]), c[5], kr, ku, status);
}

// True iff the body box around (x, y, z) lies inside the grid and touches no filled voxel
// (cells floor(lo)..floor(hi) on every axis, ends included).
__device__ __forceinline__ bool body_free(const unsigned char *occ, const EnvLayout &lay, int gx, int gy, int gz, float x, float y,
                                          float z, float hw, float below, float above)
{
    const float lx = __fsub_rn(x, hw), hx = __fadd_rn(x, hw);
    const float ly = __fsub_rn(y, below), hy = __fadd_rn(y, above);
    const float lz = __fsub_rn(z, hw), hz = __fadd_rn(z, hw);
    if (!(lx >= 0.0f) || !(hx < (float)gx) || !(ly >= 0.0f) || !(hy < (float)gy) || !(lz >= 0.0f) ||
        !(hz < (float)gz))
        return false;
    const int i0 = (int)floorf(lx), i1 = (int)floorf(hx), j0 = (int)floorf(ly), j1 = (int)floorf(hy);
    const int k0 = (int)floorf(lz), k1 = (int)floorf(hz);
    for (int j = j0; j <= j1; ++j)
        for (int k = k0; k <= k1; ++k)
            for (int i = i0; i <= i1; ++i)
                if (voxel_filled(lay, occ, i, j, k)) return false;
    return true;
}

// Agent motion with voxel collision; one thread per agent.  Updates the caller's camera array,
// the ray-basis table and the agent's own body box inside its env block.
__global__ void move_agents_kernel(int32_t *cams, const float4 *moves, CamRec *recs, unsigned char *env_blocks,
                                   EnvLayout lay, int num_obs, int agents, int gx, int gy, int gz, int max_boxes,
                                   float hw, float below, float above, float max_pitch, double kr, double ku,
                                   uint32_t *status)
{
    launch_dependents();
    wait_for_previous();
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= num_obs) return;
    int32_t *c = cams + (size_t)o * 6;
    const float x = __int_as_float(c[0]), y = __int_as_float(c[1]), z = __int_as_float(c[2]);
    const float4 mv = moves[o];
    const float yaw = __fadd_rn(__int_as_float(c[3]), mv.z);
    float pitch = __fadd_rn(__int_as_float(c[4]), mv.w);
    pitch = pitch > max_pitch ? max_pitch : pitch;
    pitch = pitch < -max_pitch ? -max_pitch : pitch;
    double sy, cy;
    sincos((double)yaw, &sy, &cy);
    const double sxd = __dadd_rn(__dmul_rn((double)mv.x, sy), __dmul_rn((double)mv.y, cy));
    const double szd = __dsub_rn(__dmul_rn((double)mv.x, cy), __dmul_rn((double)mv.y, sy));
    const float x_try = (float)__dadd_rn((double)x, sxd);
    const float z_try = (float)__dadd_rn((double)z, szd);
    unsigned char *blk = env_blocks + (size_t)(o / agents) * lay.stride;
    float nx = x, nz = z;
    if (body_free(blk, lay, gx, gy, gz, x_try, y, nz, hw, below, above)) nx = x_try;
    if (body_free(blk, lay, gx, gy, gz, nx, y, z_try, hw, below, above)) nz = z_try;
    c[0] = __float_as_int(nx); c[2] = __float_as_int(nz);
    c[3] = __float_as_int(yaw); c[4] = __float_as_int(pitch);
    const int self_box = c[5];
    write_camrec(recs + o, nx, y, nz, yaw, pitch, self_box, kr, ku, status);
    const int count = *reinterpret_cast<const int *>(blk + lay.count_off);
    if (self_box >= 0 && self_box < min(count, max_boxes)) {
        float *b = reinterpret_cast<float *>(blk + lay.box_off) + 8 * self_box;
        b[0] = __fsub_rn(nx, hw); b[1] = __fsub_rn(y, below); b[2] = __fsub_rn(nz, hw);
        b[3] = __fadd_rn(nx, hw); b[4] = __fadd_rn(y, above); b[5] = __fadd_rn(nz, hw);
    }
}

// GUI rectangles into the library's table; counts clamped to 0..max_rects.
__global__ void copy_overlays_kernel(const int4 *rects, const int32_t *counts, int4 *out_rects, int32_t *out_counts,
                                     int num_obs, int max_rects)
{
    launch_dependents();
    wait_for_previous();
    const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int o = (int)(gid / (max_rects + 1)), r = (int)(gid - (long long)o * (max_rects + 1));
    if (o >= num_obs) return;
    if (r == max_rects) {
        const int n = rects ? counts[o] : 0;
        out_counts[o] = n < 0 ? 0 : (n > max_rects ? max_rects : n);
    } else if (rects) {
        out_rects[(size_t)o * max_rects + r] = rects[(size_t)o * max_rects + r];
    }
}

}  // namespace mv
