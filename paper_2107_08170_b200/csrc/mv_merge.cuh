// Greedy merging of an env's voxels into boxes (paper Section 3.3).  The result is that of a serial sweep
// in index order (x fastest, then z, then y): the first filled, uncovered voxel starts a box, which grows
// along +x, then +z, then +y while every cell of the new row / slab is filled, uncovered and of the same
// material.  That sweep is one long chain of dependent steps per box; here each row of a layer is one step.
//
// Why rows can be done at once.  Within a layer y = j call a cell open if it is filled and not covered by
// a box that began in a lower layer.  A box that began in an earlier row of the layer and covers cell
// (x, k) also covers (x, k-1), so: (1) the boxes that begin in row k are exactly the maximal runs of equal
// material among the cells of the row that are open and not covered by boxes reaching in from row k-1;
// (2) a box reaches row k+1 iff all its cells there are open and of its material (no other box of the layer
// can cover them); (3) likewise, since a box that covers (x, j+1, z) also covers (x, j, z), the height is the
// least run of equal material going up from the box's footprint, whatever other boxes do.  So a row is a
// handful of bit operations on x-packed words: which boxes end (a failing cell marks its whole segment, two
// carry-propagating additions), which begin; and the heights of a layer's boxes are independent of each other.
//
// Measured (512 envs of 128x32x128 with 1361 boxes each): 11.4 ms with one warp growing one box at a time (about
// 8 us a box, all of it latency); 0.44 ms with the rows of a layer one after the other in one warp; 0.25 ms with all rows at
// once (see sweep_layer), of which the bit arrays 0.1.
#pragma once
#include "mv_device.cuh"
#include "mv_pack.cuh"

namespace mv {

constexpr int kMergeThreads = 256;
constexpr int kMergeList = 768;           // boxes of a layer handled at a time
constexpr int kMergeSmallArea = 64;       // footprints up to this many cells go to four lanes, larger ones to the CTA

// Scratch of one env, in 32-bit words: three x-packed bit arrays [y][z][W] (filled; equal to the cell at
// x-1; equal to the cell at z-1), one y-packed array [z][x][colw] (equal to the cell above), and, where
// shared memory is too small for it, the work area of the sweep.
struct MergeLayout {
    int gx, gy, gz;
    int W;                    // words per x-row
    int colw;                 // words per (x, z) column
    uint32_t mask_words;      // words of one x-packed array
    int slots;                // records per row of the sweep's work area: the row's words and one more
    uint32_t work_bytes;      // 16 bytes per record of one layer + one Cov per column
    uint32_t work_off;        // word offset of the work area in the env's scratch
    int work_in_smem;
    size_t env_words;         // words between envs
    size_t mat_stride;        // bytes between envs in the material store
};

// 32 x 32 bit transpose over a warp: bit i of lane l becomes bit l of lane i.
__device__ __forceinline__ uint32_t transpose32(uint32_t v, int lane)
{
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        const uint32_t m = s == 16 ? 0x0000ffffu : s == 8 ? 0x00ff00ffu : s == 4 ? 0x0f0f0f0fu : s == 2 ? 0x33333333u : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(0xffffffffu, v, s);
        v = (lane & s) ? (((y >> s) & m) | (v & ~m)) : (((y << s) & ~m) | (v & m));
    }
    return v;
}

// The bit arrays of a launch's envs.  One CTA: 8 z-rows x 128 x x 32 heights of one env; a warp takes 32 columns of
// four rows, so that the column at z-1 is still in registers; the y-packed results are transposed in registers and
// leave through shared memory as runs of up to 128 bytes.  Bound by the material bytes it streams (one byte per
// voxel, the x-1 column from L1) and by instructions, once the upper 16 heights are left out where nothing is filled up there; then
// two rows also share a transpose (512 worlds of 128x32x128 287.5 -> 281.4 us, 1047 of 112x44x52 329.2 -> 306.6).
template <bool PLANES>
__global__ void __launch_bounds__(kMergeThreads) merge_masks_kernel(const unsigned char *__restrict__ env_blocks,
                                                                    const uint8_t *__restrict__ mat, EnvLayout lay,
                                                                    MergeLayout ml, int env_begin, uint32_t *__restrict__ scratch)
{
    const int nzb = (ml.gz + 7) / 8, nwb = (ml.W + 3) / 4;
    int r = blockIdx.x;
    const int wb = r % nwb; r /= nwb;
    const int zb = r % nzb; r /= nzb;
    const int wq = r % ml.colw, e = r / ml.colw;
    const unsigned char *blk = env_blocks + (size_t)(env_begin + e) * lay.stride;
    const int *bounds = reinterpret_cast<const int *>(blk + lay.count_off);
    const int loy = bounds[2], hiy = bounds[5];
    if (32 * wq >= hiy || 32 * wq + 32 <= loy) return;          // nothing filled at these heights (or an empty grid)
    __shared__ uint32_t s_out[3][32][8 * 4 + 1];     // (padded: the writes run down a column)
    const int lane = threadIdx.x & 31, wi = (threadIdx.x >> 5) & 3, half = threadIdx.x >> 7;
    const int w = 4 * wb + wi, x = 32 * w + lane, z0 = 8 * zb + 4 * half;
    const bool upper = hiy - 32 * wq > 16, higher = hiy - 32 * wq > 32, in_x = x < ml.gx;
    // 32 heights of a column, and the one above them (PLANES: of the two or three planes that they lie in, as far as anything is filled)
    const uint32_t plane = PLANES ? plane_of(lay, 32 * wq) : 0u, off = 32u * (uint32_t)wq - (uint32_t)plane_begin(plane), words = lay.occ_plane / 4;
    const uint32_t *occ = reinterpret_cast<const uint32_t *>(blk) + (size_t)plane * words + lay.origin + x;
    const bool second = PLANES && plane + 1 < lay.planes && hiy > plane_begin(plane + 1), third = second && off > 29 && plane + 2 < lay.planes;
    auto bits = [&](int at, uint32_t &above) {
        const uint32_t *w = occ + at;
        if (!PLANES) { above = 0u; return w[0]; }
        unsigned long long b = (w[0] & ~kPlaneEnd) >> off;
        if (second) b |= (unsigned long long)(w[words] & ~kPlaneEnd) << (kPlaneHeights - off);
        if (third) b |= (unsigned long long)w[2 * words] << (2 * kPlaneHeights - off);
        above = (uint32_t)(b >> 32);
        return (uint32_t)b;
    };
    const uint8_t *m_col = mat + (size_t)(env_begin + e) * ml.mat_stride + ((size_t)(lay.origin + x) << lay.ysh) + 32 * wq;
    uint32_t *ye = scratch + (size_t)e * ml.env_words + 3 * (size_t)ml.mask_words + x * ml.colw + wq;
    auto load_column = [&](const uint8_t *src, uint32_t out[8]) {
        const uint4 a = __ldg(reinterpret_cast<const uint4 *>(src));
        uint4 b = make_uint4(0, 0, 0, 0);
        if (upper) b = __ldg(reinterpret_cast<const uint4 *>(src) + 1);
        out[0] = a.x; out[1] = a.y; out[2] = a.z; out[3] = a.w;
        out[4] = b.x; out[5] = b.y; out[6] = b.z; out[7] = b.w;
    };
    // Bit per height at which two columns' material bytes are equal (bits above 16 are not wanted when !upper).
    // A differing byte leaves 0x80 in its place; a dot product with powers of two collects eight of them.
    auto equal_bits = [&](const uint32_t a[8], const uint32_t b[8]) {
        auto differ8 = [&](int q) {
            const uint32_t v0 = a[q] ^ b[q], v1 = a[q + 1] ^ b[q + 1];
            const uint32_t n0 = (((v0 & 0x7f7f7f7fu) + 0x7f7f7f7fu) | v0) & 0x80808080u;
            const uint32_t n1 = (((v1 & 0x7f7f7f7fu) + 0x7f7f7f7fu) | v1) & 0x80808080u;
            return __dp4a(n1, 0x80402010u, __dp4a(n0, 0x08040201u, 0u));          // 128 x the eight bits
        };
        uint32_t ne = (differ8(0) >> 7) | (differ8(2) << 1);
        if (upper) ne |= (differ8(4) << 9) | (differ8(6) << 17);
        return ~ne;
    };
    uint32_t own[8] = {}, back[8] = {}, f_back = 0, f_above = 0, f_even = 0, lx_even = 0, lz_even = 0;
    if (in_x && z0 > 0 && z0 < ml.gz) {
        f_back = bits((z0 - 1) * (int)lay.pitch, f_above);
        load_column(m_col + ((size_t)(z0 - 1) * lay.pitch << lay.ysh), back);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int z = z0 + i;
        uint32_t f = 0, lx = 0, lz = 0;
        if (z < ml.gz && in_x) {
            const int row = z * (int)lay.pitch;
            const uint8_t *src = m_col + ((size_t)row << lay.ysh);
            uint32_t other[8], f_left = 0, unused;
            f = bits(row, f_above);
            load_column(src, own);
            if (x > 0) {
                f_left = bits(row - 1, unused);
                load_column(src - (1u << lay.ysh), other);
            }
            lz = f & f_back & equal_bits(own, back);
            if (x > 0) lx = f & f_left & equal_bits(own, other);
            const uint32_t above = PLANES && higher ? src[32] : 0u;
#pragma unroll
            for (int q = 0; q < 7; ++q) other[q] = __funnelshift_r(own[q], own[q + 1], 8);     // one height up
            other[7] = (own[7] >> 8) | (above << 24);
            ye[(size_t)z * ml.gx * ml.colw] = f & ((f >> 1) | (f_above << 31)) & equal_bits(own, other);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) back[q] = own[q];
        f_back = f;
        if (upper) {
            s_out[0][lane][(4 * half + i) * 4 + wi] = transpose32(f, lane);
            s_out[1][lane][(4 * half + i) * 4 + wi] = transpose32(lx, lane);
            s_out[2][lane][(4 * half + i) * 4 + wi] = transpose32(lz, lane);
        } else if (i & 1) {                              // 16 heights of two rows in one transpose
            const int at = (4 * half + i - 1 + (lane >> 4)) * 4 + wi;
            s_out[0][lane & 15][at] = transpose32(f_even | f << 16, lane);
            s_out[1][lane & 15][at] = transpose32(lx_even | lx << 16, lane);
            s_out[2][lane & 15][at] = transpose32(lz_even | lz << 16, lane);
        } else {
            f_even = f & 0xffffu; lx_even = lx & 0xffffu; lz_even = lz & 0xffffu;
        }
    }
    __syncthreads();
    uint32_t *dst = scratch + (size_t)e * ml.env_words;
    for (int i = threadIdx.x; i < 3 * 32 * 32; i += kMergeThreads) {
        const int a = i >> 10, y = (i >> 5) & 31, zz = (i >> 2) & 7, wo = 4 * wb + (i & 3);
        const int j = 32 * wq + y, k = 8 * zb + zz;
        if (j >= loy && j < hiy && k < ml.gz && wo < ml.W)
            dst[(size_t)a * ml.mask_words + ((size_t)j * ml.gz + k) * ml.W + wo] = s_out[a][y][i & 31];
    }
}

// out = a + b over N words, least significant first.
template <int N> __device__ __forceinline__ void add_words(const uint32_t *a, const uint32_t *b, uint32_t *out)
{
    uint32_t carry = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const unsigned long long t = (unsigned long long)a[i] + b[i] + carry;
        out[i] = (uint32_t)t;
        carry = (uint32_t)(t >> 32);
    }
}

// A warp that has not settled its rows of a layer after kSweepTurns leaves the layer to sweep_rows, and the next layers go there at once:
// three, then seven and fifteen if the one after them does the same.  Where two boxes lie side by side every row of their edge
// takes a turn, and a turn of six words a row takes twice as long as a row in sweep_rows: one such layer of 192x192 75 us without
// a limit, 39 with it.  With 8 turns columns give up too (32 worlds of 192x32x192 333 us; 201 with 16, 200 without a limit).  Rows of
// up to two words have none: their turns are as short as a row in sweep_rows (16 worlds of 64x8x64 with such edges 110.7 us, 127.1).
constexpr int kSweepTurns = 16, kSweepPause = 15;
// What the sweep of a layer hands on when it has more rows than the CTA has threads, and the warps to each other.
template <int N> struct SweepEdges {
    uint32_t warp[2][kMergeThreads / 32][N];      // L of a warp's last row, by the parity of the round
    uint32_t open[N], link[N];                    // cells and L of the last row of the 256 before
};

// Carry chain along a row, one word a lane: gen | (prop & carry from the bit below), which is what an addition
// computes.  Whole lanes generate (G) or propagate (P) a carry; two votes and one more addition carry it across them, but out
// of no lane whose bit is missing in `out`.
__device__ __forceinline__ uint32_t fill(uint32_t gen, uint32_t prop, uint32_t lane_bit, uint32_t out = 0xffffffffu)
{
    const uint32_t a = gen | prop;
    uint32_t s = a + gen;
    const uint32_t G = __ballot_sync(0xffffffffu, s < a) & out, P = (__ballot_sync(0xffffffffu, s == 0xffffffffu) & out) | G;
    s += ((P + G) ^ P ^ G) & lane_bit ? 1u : 0u;
    return gen | (a & (s ^ a ^ gen));
}

// Part B of the sweep (see merge_sweep_kernel) for rows of up to N words, one after the other: one warp, a word of the row per lane.
// A box with a failing cell ends, so a fail has to spread both ways along its segment, and carries only run upward.  Rows are
// therefore held twice, in order in the lower lanes and mirrored (words and bits) from lane 16 on: the same instructions spread a
// fail upward in one half and downward in the other, and the halves then exchange what they found.  Per lane: S = open cells of the
// row before, L = those of them that are in the same box as the cell before them in the lane's own direction.  `before`: the row
// before the first one, or null.  About 240 cycles a row, all of them latency.
template <int N>
__device__ __forceinline__ void sweep_rows(uint4 *rows, int slots, int W, int nrows, int lane, const SweepEdges<N> *before)
{
    const bool mirror = lane >= 16;
    const int w = mirror ? W - 1 - (lane - 16) : lane;                  // the lane's word of the row
    const bool valid = w >= 0 && w < W;
    const int partner = !valid ? lane : mirror ? w : 16 + W - 1 - w;
    const uint32_t lane_bit = 1u << lane;
    auto turned = [&](uint32_t v) { return mirror ? __brev(v) : v; };
    auto turned_links = [&](uint32_t v, uint32_t next) { return mirror ? __brev(__funnelshift_r(v, next, 1)) : v; };
    // (idle lanes share the row's empty record, which is also what comes after its last word)
    const int at = valid ? w : W, behind = valid ? w + 1 : W;
    uint32_t S = before && valid ? turned(before->open[w]) : 0u;
    uint32_t L = before && valid ? turned_links(before->link[w], w + 1 < W ? before->link[w + 1] : 0u) : 0u;
    // a row's record is fetched two rows ahead and turned one row ahead, while the lanes wait for each other
    uint4 ahead = rows[at];
    uint32_t ahead_y = rows[behind].y, x = turned(ahead.x), lx = turned_links(ahead.y, ahead_y), fits = turned(ahead.x & ahead.z);
    const uint4 *p = rows + (nrows > 1 ? slots : 0);
    ahead = p[at]; ahead_y = p[behind].y;
#pragma unroll 4
    for (int k = 0; k < nrows; ++k, rows += slots) {
        p += k + 2 < nrows ? slots : 0;
        const uint4 next = p[at];
        const uint32_t next_y = p[behind].y;
        uint32_t D = fill(S & ~fits, L, lane_bit, 0xffff7fffu);
        D |= __brev(__shfl_sync(0xffffffffu, D, partner));
        const uint32_t A = x & ~(S & ~D);
        uint32_t prev = __shfl_up_sync(0xffffffffu, A, 1, 16);
        prev = (lane & 15) ? prev : 0u;
        const uint32_t link = A & __funnelshift_l(prev, A, 1) & lx;
        if (valid && !mirror) rows[w] = make_uint4(A, A & ~link, D & S & ~L, 0u);
        S = (S & ~D) | A;
        L = (L & ~D) | link;
        x = turned(ahead.x); lx = turned_links(ahead.y, ahead_y); fits = turned(ahead.x & ahead.z);
        ahead = next; ahead_y = next_y;
    }
}

// Part B of the sweep (see merge_sweep_kernel) for rows of up to N words: one lane a row.  A row is ml.slots records of
// {open cells, x links, z links, -}, which become {new cells, their first cells, first cells of boxes that end here, -}.
// What a row needs of the row before is its open cells (every one is in some box) and L: which of them are in the same box as
// their neighbour at x-1.  A box ends where one of its cells fails, and the fail takes its whole segment of L along: a carry
// chain upward and one downward, an addition each, the second on the reversed row.  So a row's L is a function of the L before,
// and instead of going down the rows one by one (230 cycles each, 195 us of the 290 that 512 worlds of 128x32x128 took) all
// rows begin with the L they have when no box reaches in, and apply the function until nothing changes: after i + 1 times row i
// is right whatever the guess was, so that ends.  What comes from above is forgotten where boxes end, and obstacles a few
// cells deep take a few times.  A warp settles its 32 rows with the row above them as it was last published (at first as that row
// itself begins; as if nothing reached in, a solid floor took 32 times a warp, one warp after the other: 32 worlds of 192x32x192
// columns 256 us, now 201); then the warps publish their last rows, until that changes nothing either.  False if the rows were left
// to sweep_rows.
template <int N>
__device__ __forceinline__ bool sweep_layer(uint4 *rows, int slots, int W, int nrows, SweepEdges<N> &edges)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int k0 = 0; k0 < nrows; k0 += kMergeThreads) {
        const int k = k0 + tid;
        uint4 *p = rows + (size_t)k * slots;
        const bool works = k0 + 32 * warp < nrows;
        uint32_t S[N], open[N], xl[N], fail[N], L[N], in[N], above[N];
#pragma unroll
        for (int w = 0; w < N; ++w) {
            const uint4 r = w < W && k < nrows ? p[w] : make_uint4(0, 0, 0, 0), up = w < W && k < nrows && tid > 0 ? p[w - slots] : make_uint4(0, 0, 0, 0);
            S[w] = tid > 0 ? up.x : k0 > 0 && k < nrows ? edges.open[w] : 0u;
            open[w] = r.x; xl[w] = r.y;
            fail[w] = S[w] & ~(r.x & r.z);
            above[w] = tid > 0 ? S[w] & __funnelshift_l(w ? S[w - 1] : 0u, S[w], 1) & up.y : k0 > 0 ? edges.link[w] : 0u;
        }
#pragma unroll
        for (int w = 0; w < N; ++w) L[w] = open[w] & __funnelshift_l(w ? open[w - 1] : 0u, open[w], 1) & xl[w];
        if (lane == 31)
#pragma unroll
            for (int w = 0; w < N; ++w) edges.warp[1][warp][w] = L[w];           // (what the next warp takes it for at first)
        // the cells of boxes that end with the row before, given what reaches in
        auto ended = [&](uint32_t *D) {
            uint32_t a[N], b[N], s[N];
#pragma unroll
            for (int w = 0; w < N; ++w) a[w] = fail[w] | in[w];
            add_words<N>(a, fail, s);
#pragma unroll
            for (int w = 0; w < N; ++w) D[w] = fail[w] | (a[w] & (s[w] ^ a[w] ^ fail[w]));
#pragma unroll
            for (int w = 0; w < N; ++w) {
                a[N - 1 - w] = __brev(fail[w] | __funnelshift_r(in[w], w + 1 < N ? in[w + 1] : 0u, 1));
                b[N - 1 - w] = __brev(fail[w]);
            }
            add_words<N>(a, b, s);
#pragma unroll
            for (int w = 0; w < N; ++w) D[w] |= __brev(a[N - 1 - w] & (s[N - 1 - w] ^ a[N - 1 - w] ^ b[N - 1 - w]));
        };
        for (int round = 0;; ++round) {
            bool news = false, gave_up = false;
            if (works) {
                for (int turn = 0;; ++turn) {
                    uint32_t D[N], A[N];
#pragma unroll
                    for (int w = 0; w < N; ++w) {
                        in[w] = __shfl_up_sync(0xffffffffu, L[w], 1);
                        if (lane == 0) in[w] = above[w];
                    }
                    ended(D);
#pragma unroll
                    for (int w = 0; w < N; ++w) A[w] = open[w] & ~(S[w] & ~D[w]);
                    bool changed = false;
#pragma unroll
                    for (int w = 0; w < N; ++w) {
                        const uint32_t l = (in[w] & ~D[w]) | (A[w] & __funnelshift_l(w ? A[w - 1] : 0u, A[w], 1) & xl[w]);
                        changed |= l != L[w];
                        L[w] = l;
                    }
                    if (!__any_sync(0xffffffffu, changed)) break;
                    if (N > 2 && turn == kSweepTurns) { gave_up = true; break; }
                }
                if (lane == 31)
#pragma unroll
                    for (int w = 0; w < N; ++w) {
                        news |= L[w] != edges.warp[~round & 1][warp][w];
                        edges.warp[round & 1][warp][w] = L[w];
                    }
            }
            const int votes = __syncthreads_count(gave_up || news);           // (news: a warp's last lane at most)
            if (N > 2 && votes >= 32) {
                if (warp == 0) sweep_rows<N>(rows + (size_t)k0 * slots, slots, W, nrows - k0, lane, k0 ? &edges : nullptr);
                return false;
            }
            if (votes == 0) break;
            if (lane == 0 && warp > 0)
#pragma unroll
                for (int w = 0; w < N; ++w) above[w] = edges.warp[round & 1][warp - 1][w];
        }
        uint32_t D[N];
        ended(D);
#pragma unroll
        for (int w = 0; w < N; ++w) {
            const uint32_t A = open[w] & ~(S[w] & ~D[w]);
            if (w < W && k < nrows) p[w] = make_uint4(A, A & ~L[w], D[w] & S[w] & ~in[w], 0u);
        }
        if (k0 + kMergeThreads < nrows) {
            if (tid == kMergeThreads - 1)
#pragma unroll
                for (int w = 0; w < N; ++w) { edges.open[w] = open[w]; edges.link[w] = L[w]; }
            __syncthreads();
        }
    }
    return true;
}

// The same for rows of more than 16 words: one warp, a word of the row per lane, the rows one after the other.
__device__ __forceinline__ void sweep_wide_rows(uint4 *rows, int slots, int W, int nrows, int lane)
{
    uint4 *p = rows + min(lane, W);
    const uint32_t lane_bit = 1u << lane;
    uint32_t S = 0, L = 0, Lup = 0;                                     // linked to x-1, linked to x+1
    for (int k = 0; k < nrows; ++k, p += slots) {
        const uint4 r = *p;
        const uint32_t fail = S & ~(r.x & r.z);
        uint32_t D = fill(fail, L, lane_bit);
        // downward: bits reversed, lanes exchanged end for end
        const uint32_t g = __brev(__shfl_xor_sync(0xffffffffu, fail, 31)), pr = __brev(__shfl_xor_sync(0xffffffffu, Lup, 31));
        D |= __brev(__shfl_xor_sync(0xffffffffu, fill(g, pr, lane_bit), 31));
        const uint32_t A = r.x & ~(S & ~D);
        uint32_t prev = __shfl_up_sync(0xffffffffu, A, 1);
        prev = lane ? prev : 0u;
        const uint32_t link = A & __funnelshift_l(prev, A, 1) & r.y;
        *p = make_uint4(A, A & ~link, D & S & ~L, 0u);
        S = (S & ~D) | A;
        L = (L & ~D) | link;
        uint32_t next = __shfl_down_sync(0xffffffffu, L, 1);
        next = lane < 31 ? next : 0u;
        Lup = __funnelshift_r(L, next, 1);
    }
}

// Height of the run of equal material that starts at layer j of a column; e = the column's word that holds bit j.
__device__ __forceinline__ int run_up(uint32_t e, const uint32_t *__restrict__ ye, int col, int colw, int j)
{
    int q = j >> 5, left = 32 - (j & 31);
    int ones = __ffs(~(e >> (j & 31))) - 1;
    ones = ones < 0 ? 32 : ones;
    int n = 1 + min(ones, left);
    while (ones >= left && ++q < colw) {
        e = __ldg(ye + (size_t)col * colw + q);
        left = 32;
        ones = __ffs(~e) - 1;
        ones = ones < 0 ? 32 : ones;
        n += ones;
    }
    return n;
}

// The sweep, one CTA per env, layer by layer: (A) all threads form the layer's open cells; (B) sweep_layer leaves, per row, the
// cells of new boxes, their first cells and the first cells of boxes that end there; (C) the new boxes are numbered in sweep
// order (a block-wide scan), measured, given their heights and the layers above marked as covered, in parallel.  Of the 240
// thousand cycles that 13 layers of a 128x32x128 world take, A has 40, B 62, numbering 13, sizes 36 and heights 74.  Cov holds a
// layer number: a byte where that is enough, so that four CTAs fit an SM at 128x128 columns.
template <typename Cov, int N>
__global__ void __launch_bounds__(kMergeThreads, N > 0 && N <= 4 ? 4 : N == 8 ? 3 : 1) merge_sweep_kernel(const unsigned char *__restrict__ env_blocks,
                                                                       const uint8_t *__restrict__ mat, EnvLayout lay, MergeLayout ml,
                                                                       int env_begin, uint32_t *__restrict__ scratch,
                                                                       uint4 *__restrict__ boxes_out, int32_t *__restrict__ count_out,
                                                                       int max_out)
{
    extern __shared__ __align__(16) unsigned char s_work[];
    __shared__ uint32_t s_list[kMergeList];          // first cell of a box: z << 16 | x
    __shared__ uint32_t s_size[kMergeList];          // its depth << 16 | width
    __shared__ uint16_t s_high[kMergeList], s_big[kMergeList];
    __shared__ uint8_t s_mat[kMergeList];
    __shared__ int s_nbig, s_part[kMergeThreads / 32];
    __shared__ SweepEdges<N ? N : 1> s_edges;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, e = blockIdx.x;
    const int gx = ml.gx, gz = ml.gz, W = ml.W, slots = ml.slots;
    const unsigned char *blk = env_blocks + (size_t)(env_begin + e) * lay.stride;
    const int *bounds = reinterpret_cast<const int *>(blk + lay.count_off);
    const int loy = bounds[2], loz = bounds[3], hiy = bounds[5], hiz = bounds[6];
    const uint8_t *m_env = mat + (size_t)(env_begin + e) * ml.mat_stride;
    uint32_t *mine = scratch + (size_t)e * ml.env_words;
    const uint32_t *masks = mine, *ye = mine + 3 * (size_t)ml.mask_words;
    uint4 *rows = reinterpret_cast<uint4 *>(ml.work_in_smem ? s_work : reinterpret_cast<unsigned char *>(mine + ml.work_off));
    Cov *cov = reinterpret_cast<Cov *>(rows + (size_t)gz * slots);      // per column: covered below this layer
    uint4 *out = boxes_out + (size_t)e * max_out * 2;
    for (int i = tid; i < gx * gz * (int)sizeof(Cov) / 4; i += kMergeThreads) reinterpret_cast<uint32_t *>(cov)[i] = 0u;
    for (int i = tid; i < gz; i += kMergeThreads) rows[i * slots + slots - 1] = make_uint4(0, 0, 0, 0);     // (idle lanes share it)
    __syncthreads();

    const int nt = (hiz - loz) * W;                  // words of the rows that hold anything
    const float inv_W = 1.0f / (float)W;
    auto row_of = [&](int t) { return (int)(((float)t + 0.5f) * inv_W); };        // exact: t < 2^15 is far from half a step
    int count = 0, rest = 0, pause = 1;
    for (int j = loy; j < hiy; ++j) {
        // ---- A
        bool any = false;
        for (int t = tid; t < nt; t += kMergeThreads) {
            const int q = row_of(t), k = loz + q, w = t - q * W, x0 = 32 * w;
            const uint32_t *m = masks + ((size_t)j * gz + k) * W + w;
            uint32_t u = m[0];
            const uint32_t lx = m[ml.mask_words], lz = m[2 * (size_t)ml.mask_words];
            uint32_t c = 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (x0 + 4 * i >= gx) break;
                if constexpr (sizeof(Cov) == 1) {
                    const uint32_t v = *reinterpret_cast<const uint32_t *>(cov + k * gx + x0 + 4 * i);
                    c |= nz_bits4(__vcmpgtu4(v, (uint32_t)j * 0x01010101u)) << (4 * i);
                } else {
                    const uint2 v = *reinterpret_cast<const uint2 *>(cov + k * gx + x0 + 4 * i);
                    c |= ((uint32_t)((v.x & 0xffffu) > (uint32_t)j) | (uint32_t)((v.x >> 16) > (uint32_t)j) << 1 |
                          (uint32_t)((v.y & 0xffffu) > (uint32_t)j) << 2 | (uint32_t)((v.y >> 16) > (uint32_t)j) << 3) << (4 * i);
                }
            }
            u &= ~c;
            rows[k * slots + w] = make_uint4(u, lx, lz, 0u);
            any |= u != 0u;
        }
        if (!__syncthreads_or(any)) continue;
        // ---- B
        if constexpr (N > 0) {
            if (N > 2 && rest > 0) {
                --rest;
                if (warp == 0) sweep_rows<N>(rows + loz * slots, slots, W, hiz - loz, lane, nullptr);
            } else {
                pause = sweep_layer<N>(rows + loz * slots, slots, W, hiz - loz, s_edges) ? 1 : min(2 * pause + 1, kSweepPause);
                rest = pause > 1 ? pause : 0;
            }
        } else if (warp == 0) sweep_wide_rows(rows + loz * slots, slots, W, hiz - loz, lane);
        __syncthreads();
        // ---- C: number the first cells in sweep order
        const int per = (nt + kMergeThreads - 1) / kMergeThreads;
        const int t_begin = min(tid * per, nt), t_end = min(t_begin + per, nt);
        int own = 0;
        for (int t = t_begin; t < t_end; ++t) { const int q = row_of(t); own += __popc(rows[(loz + q) * slots + t - q * W].y); }
        int incl = own;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, s);
            if (lane >= s) incl += v;
        }
        if (lane == 31) s_part[warp] = incl;
        __syncthreads();
        int total = 0, rank0 = incl - own;
#pragma unroll
        for (int v = 0; v < kMergeThreads / 32; ++v) {
            if (v < warp) rank0 += s_part[v];
            total += s_part[v];
        }
        for (int win = 0; win < total; win += kMergeList) {
            if (tid == 0) s_nbig = 0;
            if (own > 0 && rank0 < win + kMergeList && rank0 + own > win) {
                int r = rank0 - win;
                for (int t = t_begin; t < t_end; ++t) {
                    const int q = row_of(t), k = loz + q, w = t - q * W;
                    for (uint32_t m = rows[k * slots + w].y; m; m &= m - 1, ++r)
                        if (r >= 0 && r < kMergeList) s_list[r] = (uint32_t)k << 16 | (uint32_t)(32 * w + __ffs(m) - 1);
                }
            }
            __syncthreads();
            const int n = min(total - win, kMergeList);
            // a thread per box: the run in its first row, and the rows until its first cell is marked ended
            for (int b = tid; b < n; b += kMergeThreads) {
                const int x = (int)(s_list[b] & 0xffffu), k = (int)(s_list[b] >> 16);
                const uint8_t m = m_env[voxel_index(lay, x, j, k)];
                int wd = x >> 5;
                uint4 r = rows[k * slots + wd];
                uint32_t stop = (r.y | ~r.x) & ~((2u << (x & 31)) - 1u);
                while (stop == 0u && ++wd < W) { r = rows[k * slots + wd]; stop = r.y | ~r.x; }
                const int w = (stop ? 32 * wd + __ffs(stop) - 1 : gx) - x;
                int d = 1;
                while (k + d < hiz && !((rows[(k + d) * slots + (x >> 5)].z >> (x & 31)) & 1u)) ++d;
                s_size[b] = (uint32_t)d << 16 | (uint32_t)w;
                s_mat[b] = m;
                if (w * d > kMergeSmallArea) s_big[atomicAdd(&s_nbig, 1)] = (uint16_t)b;
            }
            __syncthreads();
            // heights and cover: four lanes per small footprint, four loads in flight each.  The whole warp stays
            // together (votes and shuffles among all lanes): groups that run apart would wait out each load one by one.
            const int g = lane & 3;
            for (int b0 = 8 * warp; b0 < n; b0 += kMergeThreads / 4) {
                const int b = min(b0 + (lane >> 2), n - 1);
                const int x = (int)(s_list[b] & 0xffffu), k = (int)(s_list[b] >> 16);
                const int w = (int)(s_size[b] & 0xffffu);
                int area = w * (int)(s_size[b] >> 16);
                if (area > kMergeSmallArea || b0 + (lane >> 2) >= n) area = 0;
                // cell c of the footprint; c / w by a reciprocal, exact for c < 64
                const float inv = 1.0f / (float)w;
                auto cell = [&](int c) { const int q = (int)(((float)c + 0.5f) * inv); return x + (c - q * w) + gx * (k + q); };
                int h = 1 << 20;
                for (int c0 = g; __any_sync(0xffffffffu, c0 < area); c0 += 16) {
                    uint32_t e4[4];
                    bool tall = false;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        e4[i] = c0 + 4 * i < area ? __ldg(ye + (size_t)cell(c0 + 4 * i) * ml.colw + (j >> 5)) : 0xffffffffu;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int ones = __ffs(~(e4[i] >> (j & 31))) - 1;          // (-1: all 32 of them)
                        h = min(h, c0 + 4 * i < area ? (ones < 0 ? 33 : ones + 1) : h);
                        tall |= c0 + 4 * i < area && (ones < 0 || ones + (j & 31) == 32);
                    }
                    if (ml.colw > 1 && tall && h + (j & 31) > 32) {                // the runs go on in the columns' next words
                        h = 1 << 20;
                        for (int c = g; c < min(area, c0 + 16); c += 4)
                            h = min(h, run_up(__ldg(ye + (size_t)cell(c) * ml.colw + (j >> 5)), ye, cell(c), ml.colw, j));
                    }
                }
                h = min(h, __shfl_xor_sync(0xffffffffu, h, 1));
                h = min(h, __shfl_xor_sync(0xffffffffu, h, 2));
                if (h > 1)
                    for (int c = g; c < area; c += 4) cov[cell(c)] = (Cov)(j + h);
                if (g == 0 && area > 0) s_high[b] = (uint16_t)h;
                __syncwarp();
            }
            __syncthreads();
            for (int i = 0; i < s_nbig; ++i) {
                const int b = s_big[i], x = (int)(s_list[b] & 0xffffu), k = (int)(s_list[b] >> 16);
                const int w = (int)(s_size[b] & 0xffffu), area = w * (int)(s_size[b] >> 16);
                int h = 1 << 20;
                for (int c = tid; c < area && h > 1; c += kMergeThreads) {
                    const int q = c / w;
                    const int col = x + (c - q * w) + gx * (k + q);
                    h = min(h, run_up(__ldg(ye + (size_t)col * ml.colw + (j >> 5)), ye, col, ml.colw, j));
                }
                h = __reduce_min_sync(0xffffffffu, h);
                if (lane == 0) s_part[warp] = h;
                __syncthreads();
#pragma unroll
                for (int v = 0; v < kMergeThreads / 32; ++v) h = min(h, s_part[v]);
                if (h > 1)
                    for (int c = tid; c < area; c += kMergeThreads) {
                        const int q = c / w;
                        cov[x + (c - q * w) + gx * (k + q)] = (Cov)(j + h);
                    }
                if (tid == 0) s_high[b] = (uint16_t)h;
                __syncthreads();
            }
            for (int b = tid; b < n && count + win + b < max_out; b += kMergeThreads) {
                const int x = (int)(s_list[b] & 0xffffu), k = (int)(s_list[b] >> 16), idx = count + win + b;
                const int w = (int)(s_size[b] & 0xffffu), d = (int)(s_size[b] >> 16), h = s_high[b];
                const uint32_t m = s_mat[b];
                out[2 * idx] = make_uint4(__float_as_uint((float)x), __float_as_uint((float)j), __float_as_uint((float)k),
                                          __float_as_uint((float)(x + w)));
                out[2 * idx + 1] = make_uint4(__float_as_uint((float)(j + h)), __float_as_uint((float)(k + d)), m, 0u);
            }
            __syncthreads();
        }
        count += total;
    }
    if (tid == 0) count_out[e] = count;
}

}  // namespace mv
