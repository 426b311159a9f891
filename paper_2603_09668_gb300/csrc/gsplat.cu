// Particle-bound 3D Gaussians: the covariance update under the MPM
// deformation gradient (Sec. 3.2, Sigma_p(t) = F_p Sigma_p F_p^T) and the
// alpha-blended splatting renderer of Eq. rendering (the 3D Gaussian
// representation: Sigma' = J W Sigma W^T J^T, C = sum T_i c_i alpha_i), with
// its reverse mode down to the particle positions and deformation gradients,
// so that an image loss differentiates through the MPM adjoint.
//
// Pipeline of gs_render (one camera), on 8 x 8 pixel tiles:
//   k_gs_preprocess  per Gaussian: Sigma, camera-space centre, projected
//                    centre mu', the inverse 2D covariance (conic), packed
//                    with its opacity and colour in 48 bytes; the pixel
//                    rectangle of the 3-sigma ellipse, and one count for
//                    every tile the rectangle meets;
//   k_gs_tile_scan   the tiles' ranges in the list;
//   k_gs_list        each Gaussian into the ranges of its tiles, as the 64-bit
//                    key (depth bits, index), in any order;
//   k_gs_tile_sort   each tile's keys sorted in shared memory: increasing
//                    depth, ties by index, so the list does not depend on the
//                    order it was filled in;
//   k_gs_render_fwd  one tile per block: its Gaussians are read front to back
//                    in batches of 64 into shared memory, then every pixel
//                    composites them.
// A tile with more Gaussians than the shared-memory sort holds sends the call
// through a stable LSD radix sort of all depths and a stable sort of the list
// by tile instead (the same lists). A list too long for 8 x 8 tiles (wide
// Gaussians: up to four times the entries) is made on 16 x 16 tiles.
// gs_render_backward walks the same ranges front to back again with the
// final colour known (dC/dalpha_i = T_i c_i - (C - C_<=i) / (1 - alpha_i)),
// reduces each Gaussian's pixel contributions per warp before one atomic,
// and k_gs_preprocess_bwd carries the 2D gradients back to x and F.
// Measured at 100,284 Gaussians, 512 x 512 (us, launches serialised), against
// 16 x 16 tiles with the radix sorts for every call: lists 200 -> 50, forward
// compositing 108 -> 59, backward 570 -> 70; two views with L1, D-SSIM and
// their gradients 2,187 -> 549.
#include <math.h>
#include <string.h>

#include <new>

#include <algorithm>

#include "common.cuh"

namespace dw {

// Tile edges are 2^ts pixels; a tile's block has a thread per pixel and takes
// its list in batches of as many entries. The path renders particles, whose
// Gaussians cover a few pixels: 8 pixels leave a warp (8 x 4 pixels) few idle
// lanes per Gaussian, and four times as many blocks as 16, with lists half as
// long (100,284 Gaussians of about 7 pixels at 512 x 512: 183,000 entries of 256
// pixels against 306,000 of 64). Wide Gaussians meet four times as many tiles of
// 8 as of 16: a list that would be longer than GS_LIST_MAX, what its indices
// hold, is made on 16 instead.
constexpr int GS_FINE = 3, GS_COARSE = 4;
__host__ __device__ constexpr int gs_threads(int ts) { return 1 << (2 * ts); }
constexpr int GS_SORT_MAX = 4096;   // keys of one tile k_gs_tile_sort holds
constexpr int GS_SORT_THREADS = 128;
constexpr int GS_BIG_CTAS = 608;    // four per SM
constexpr int GS_ROW = 12;          // floats per Gaussian of the packed rows and of the 2D gradients
constexpr int RS_THREADS = 256;
constexpr int RS_TILE = RS_THREADS * 16;  // keys per sort block
// Entries of a list: the sort's last block and a tile's last batch step past it
// by up to RS_TILE, in 32-bit indices.
constexpr int64_t GS_LIST_MAX = (1ll << 31) - RS_TILE;

struct GsCam {
    float R[9], T[3];
    float fx, fy, cx, cy;
    int width, height;
    float near_z;
};

// Per-Gaussian forward quantities recomputed identically by both passes.
struct GsProj {
    float S[6];       // Sigma = F Sigma0 F^T (xx, yy, zz, xy, xz, yz)
    float t[3];       // camera-space centre
    float J[6];       // rows (J00 J01 J02), (J10 J11 J12); J01 = J10 = 0
    float V[6];       // R Sigma R^T
    float s2[3];      // Sigma' (xx, xy, yy)
    float mu[2];
    float conic[3];   // inverse of Sigma' (a, b, c)
    bool visible;
};

__device__ __forceinline__ void sym_full(const float s[6], float M[3][3]) {
    M[0][0] = s[0];
    M[1][1] = s[1];
    M[2][2] = s[2];
    M[0][1] = M[1][0] = s[3];
    M[0][2] = M[2][0] = s[4];
    M[1][2] = M[2][1] = s[5];
}

__device__ __forceinline__ void load_F(const float *__restrict__ F, int64_t n, int64_t i,
                                       float Fm[3][3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) Fm[a][b] = F[(3 * a + b) * n + i];
}

__device__ __forceinline__ void cov_update(const float Fm[3][3], const float s0[6], float S[6]) {
    float S0[3][3], FS[3][3];
    sym_full(s0, S0);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            FS[a][b] = Fm[a][0] * S0[0][b] + Fm[a][1] * S0[1][b] + Fm[a][2] * S0[2][b];
    float M[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            M[a][b] = FS[a][0] * Fm[b][0] + FS[a][1] * Fm[b][1] + FS[a][2] * Fm[b][2];
    S[0] = M[0][0];
    S[1] = M[1][1];
    S[2] = M[2][2];
    S[3] = M[0][1];
    S[4] = M[0][2];
    S[5] = M[1][2];
}

__device__ __forceinline__ void gs_project(const GsCam &c, const float x[3], const float S[6],
                                           GsProj &p) {
#pragma unroll
    for (int k = 0; k < 6; ++k) p.S[k] = S[k];
#pragma unroll
    for (int a = 0; a < 3; ++a)
        p.t[a] = c.R[3 * a] * x[0] + c.R[3 * a + 1] * x[1] + c.R[3 * a + 2] * x[2] + c.T[a];
    p.visible = p.t[2] > c.near_z;
    const float tz = p.visible ? p.t[2] : 1.0f;
    const float iz = 1.0f / tz;
    p.J[0] = c.fx * iz;
    p.J[1] = 0.0f;
    p.J[2] = -c.fx * p.t[0] * iz * iz;
    p.J[3] = 0.0f;
    p.J[4] = c.fy * iz;
    p.J[5] = -c.fy * p.t[1] * iz * iz;
    float Sm[3][3], RS[3][3], Vm[3][3];
    sym_full(S, Sm);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            RS[a][b] = c.R[3 * a] * Sm[0][b] + c.R[3 * a + 1] * Sm[1][b] + c.R[3 * a + 2] * Sm[2][b];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            Vm[a][b] = RS[a][0] * c.R[3 * b] + RS[a][1] * c.R[3 * b + 1] + RS[a][2] * c.R[3 * b + 2];
    p.V[0] = Vm[0][0];
    p.V[1] = Vm[1][1];
    p.V[2] = Vm[2][2];
    p.V[3] = Vm[0][1];
    p.V[4] = Vm[0][2];
    p.V[5] = Vm[1][2];
    // Sigma' = J V J^T with J = [[j0, 0, j2], [0, j4, j5]]
    const float j0 = p.J[0], j2 = p.J[2], j4 = p.J[4], j5 = p.J[5];
    const float JV0[3] = {j0 * Vm[0][0] + j2 * Vm[2][0], j0 * Vm[0][1] + j2 * Vm[2][1],
                          j0 * Vm[0][2] + j2 * Vm[2][2]};
    const float JV1[3] = {j4 * Vm[1][0] + j5 * Vm[2][0], j4 * Vm[1][1] + j5 * Vm[2][1],
                          j4 * Vm[1][2] + j5 * Vm[2][2]};
    p.s2[0] = JV0[0] * j0 + JV0[2] * j2;  // xx
    p.s2[1] = JV0[1] * j4 + JV0[2] * j5;  // xy
    p.s2[2] = JV1[1] * j4 + JV1[2] * j5;  // yy
    const float det = p.s2[0] * p.s2[2] - p.s2[1] * p.s2[1];
    p.visible = p.visible && det > 0.0f;
    const float idet = p.visible ? 1.0f / det : 0.0f;
    p.conic[0] = p.s2[2] * idet;
    p.conic[1] = -p.s2[1] * idet;
    p.conic[2] = p.s2[0] * idet;
    p.mu[0] = c.fx * p.t[0] * iz + c.cx;
    p.mu[1] = c.fy * p.t[1] * iz + c.cy;
}

// ------------------------------------------------------------ covariance --

__global__ void k_gs_covariance(const float *__restrict__ F, const float *__restrict__ s0,
                                int64_t n, float *__restrict__ sigma) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float Fm[3][3], a[6], S[6];
    load_F(F, n, i, Fm);
#pragma unroll
    for (int k = 0; k < 6; ++k) a[k] = s0[k * n + i];
    cov_update(Fm, a, S);
#pragma unroll
    for (int k = 0; k < 6; ++k) sigma[k * n + i] = S[k];
}

// ------------------------------------------------------------ preprocess --

// Tiles met by a Gaussian with pixel rectangle r (drawn = false: none).
struct GsTiles {
    int first, nx, count;  // tile of the rectangle's corner, tiles per row, tiles
};

__device__ __forceinline__ GsTiles gs_tiles(int4 r, bool drawn, int tiles_x, int ts) {
    const int x0 = r.x >> ts, y0 = r.y >> ts;
    GsTiles t;
    t.first = y0 * tiles_x + x0;
    t.nx = drawn ? (r.z >> ts) - x0 + 1 : 0;
    t.count = drawn ? t.nx * ((r.w >> ts) - y0 + 1) : 0;
    return t;
}

// A Gaussian that meets more than GS_BIG of the fine tiles is queued (k_gs_big).
constexpr int GS_BIG = 16;

// f(tile, mask) for every tile of each lane's Gaussian that meets at most
// GS_BIG of them, called by whole warps with the mask of the lanes that call
// it together. Neighbouring particles' Gaussians meet the same tiles, so f
// combines equal tiles of the mask before its atomic.
template <typename Fn>
__device__ __forceinline__ void gs_for_tiles(const GsTiles &g, int tiles_x, Fn f) {
    const int cnt = g.count <= GS_BIG ? g.count : 0;
    const int most = __reduce_max_sync(0xffffffffu, cnt);
    for (int t = 0, tx = 0, tile = g.first; t < most; ++t) {
        const unsigned mask = __ballot_sync(0xffffffffu, t < cnt);
        if (t < cnt) f(tile, mask);
        __syncwarp();
        ++tile;
        if (++tx == g.nx) {
            tx = 0;
            tile += tiles_x - g.nx;
        }
    }
}

// One of the mask's lanes adds a tile's lanes to its count.
__device__ __forceinline__ void gs_count_tile(int tile, unsigned mask, uint32_t *__restrict__ tile_count) {
    const unsigned peers = __match_any_sync(mask, tile);
    if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&tile_count[tile], __popc(peers));
}

// Per Gaussian: row = (mu'(2), conic(3), opacity, colour(3)), the pixel
// rectangle [x0, x1] x [y0, y1] of the pixel centres inside the 3-sigma ellipse
// (empty when x1 < x0), the depth key (float bits of t_z, or all ones when not
// drawn), and one count for each tile met; a Gaussian that meets more than
// GS_BIG tiles goes to a queue instead (k_gs_big).
__global__ void __launch_bounds__(128) k_gs_preprocess(
    GsCam c, const float *__restrict__ x, const float *__restrict__ F, const float *__restrict__ s0,
    const float *__restrict__ color, const float *__restrict__ opacity, int n, int tiles_x,
    float4 *__restrict__ rows, int4 *__restrict__ rect, uint32_t *__restrict__ key,
    uint32_t *__restrict__ tile_count, uint32_t *__restrict__ big, uint32_t *__restrict__ big_count) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = min(t, n - 1);  // the last warp's spare lanes repeat the last Gaussian
    float Fm[3][3], a[6], S[6];
    load_F(F, n, i, Fm);
#pragma unroll
    for (int k = 0; k < 6; ++k) a[k] = s0[(int64_t)k * n + i];
    const float op = opacity[i], c0 = color[i], c1 = color[(int64_t)n + i], c2 = color[2 * (int64_t)n + i];
    cov_update(Fm, a, S);
    const float xp[3] = {x[i], x[(int64_t)n + i], x[2 * (int64_t)n + i]};
    GsProj p;
    gs_project(c, xp, S, p);
    int4 r = make_int4(0, 0, -1, -1);
    if (p.visible) {
        const float rx = 3.0f * sqrtf(p.s2[0]), ry = 3.0f * sqrtf(p.s2[2]);
        // pixel px has its centre at px + 1/2
        const float lx = ceilf(p.mu[0] - rx - 0.5f), hx = floorf(p.mu[0] + rx - 0.5f);
        const float ly = ceilf(p.mu[1] - ry - 0.5f), hy = floorf(p.mu[1] + ry - 0.5f);
        r.x = (int)fmaxf(lx, 0.0f);
        r.y = (int)fmaxf(ly, 0.0f);
        r.z = (int)fminf(hx, (float)(c.width - 1));
        r.w = (int)fminf(hy, (float)(c.height - 1));
        if (!(lx <= hx && ly <= hy)) r = make_int4(0, 0, -1, -1);  // also NaN
    }
    const bool drawn = r.z >= r.x && r.w >= r.y;
    const GsTiles g = gs_tiles(r, drawn && t < n, tiles_x, GS_FINE);
    gs_for_tiles(g, tiles_x, [&](int tile, unsigned mask) { gs_count_tile(tile, mask, tile_count); });
    if (t >= n) return;
    if (g.count > GS_BIG) big[atomicAdd(big_count, 1u)] = (uint32_t)i;
    rows[3 * (int64_t)i] = make_float4(p.mu[0], p.mu[1], p.conic[0], p.conic[1]);
    rows[3 * (int64_t)i + 1] = make_float4(p.conic[2], op, c0, c1);
    rows[3 * (int64_t)i + 2] = make_float4(c2, 0.0f, 0.0f, 0.0f);
    rect[i] = r;
    key[i] = drawn ? __float_as_uint(p.t[2]) : 0xffffffffu;  // t_z > 0: bits order as floats
}

// ------------------------------------------------------------ radix sort --

__global__ void __launch_bounds__(RS_THREADS) k_rs_hist(const uint32_t *__restrict__ key, int n,
                                                        int shift, int nblocks,
                                                        uint32_t *__restrict__ counts) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int base = blockIdx.x * RS_TILE;
    const int end = min(base + RS_TILE, n);
    for (int i = base + threadIdx.x; i < end; i += RS_THREADS)
        atomicAdd(&h[(key[i] >> shift) & 255u], 1u);
    __syncthreads();
    counts[threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

// Exclusive scan of counts[0..m) in one block (digit-major, block-minor, so
// the offsets keep the blocks' order within a digit).
__global__ void __launch_bounds__(1024) k_rs_scan(uint32_t *__restrict__ counts, int m) {
    __shared__ uint32_t part[1024];
    const int per = (m + 1023) / 1024;
    const int b = threadIdx.x * per, e = min(b + per, m);
    uint32_t s = 0;
    for (int i = b; i < e; ++i) s += counts[i];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        const uint32_t v = threadIdx.x >= off ? part[threadIdx.x - off] : 0u;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    uint32_t run = part[threadIdx.x] - s;  // exclusive prefix of this thread's range
    for (int i = b; i < e; ++i) {
        const uint32_t c = counts[i];
        counts[i] = run;
        run += c;
    }
}

// Stable scatter: each block walks its tile 256 keys at a time in order; a
// key's slot is its digit's running base in the block, plus the same-digit
// keys of earlier warps of the chunk, plus the same-digit lanes before it.
__global__ void __launch_bounds__(RS_THREADS) k_rs_scatter(const uint32_t *__restrict__ kin,
                                                           const uint32_t *__restrict__ vin,
                                                           uint32_t *__restrict__ kout,
                                                           uint32_t *__restrict__ vout, int n,
                                                           int shift, int nblocks,
                                                           const uint32_t *__restrict__ offsets) {
    constexpr int WARPS = RS_THREADS / 32;
    __shared__ uint32_t base[256];
    __shared__ uint32_t wcount[WARPS][257];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    base[threadIdx.x] = offsets[threadIdx.x * nblocks + blockIdx.x];
    const int tile0 = blockIdx.x * RS_TILE;
    const int tile1 = min(tile0 + RS_TILE, n);
    for (int c0 = tile0; c0 < tile1; c0 += RS_THREADS) {
        for (int k = threadIdx.x; k < WARPS * 257; k += RS_THREADS) (&wcount[0][0])[k] = 0u;
        __syncthreads();
        const int i = c0 + threadIdx.x;
        const bool valid = i < tile1;
        const uint32_t kv = valid ? kin[i] : 0u;
        const uint32_t d = valid ? ((kv >> shift) & 255u) : 256u;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const unsigned below = peers & ((1u << lane) - 1u);
        if (below == 0u) wcount[warp][d] = (uint32_t)__popc(peers);  // the lowest lane of a group
        __syncthreads();
        if (valid) {
            uint32_t pos = base[d] + (uint32_t)__popc(below);
            for (int w = 0; w < warp; ++w) pos += wcount[w][d];
            kout[pos] = kv;
            vout[pos] = vin[i];
        }
        __syncthreads();
        {  // advance every digit's base by its count in this chunk
            const int dd = threadIdx.x;
            uint32_t add = 0;
#pragma unroll
            for (int w = 0; w < WARPS; ++w) add += wcount[w][dd];
            base[dd] += add;
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------ tile lists --

// A scan word: entries in the high half, batches in the low one.
__device__ __forceinline__ uint32_t gs_batches(uint32_t entries, int ts) {
    return (entries + gs_threads(ts) - 1) >> (2 * ts);
}
__device__ __forceinline__ unsigned long long gs_word(uint32_t entries, int ts) {
    return ((unsigned long long)entries << 32) | gs_batches(entries, ts);
}

// What gs_render reads back: the list's length, its batches, the longest tile's
// list and the queue's length.
struct GsStat {
    unsigned long long total;
    uint32_t batches, most, big;
};

// Exclusive scan of the tiles' counts in one block: ranges[t].x = ranges[t].y
// = the tile's first entry (k_gs_list advances .y to its end), and of their
// batches: batch_off[t] = the tile's first batch.
__global__ void __launch_bounds__(1024) k_gs_tile_scan(const uint32_t *__restrict__ count,
                                                       int tiles, int ts, int2 *__restrict__ ranges,
                                                       uint32_t *__restrict__ batch_off,
                                                       GsStat *__restrict__ stat) {
    // Of a list that is accepted (below 2^31 entries) both sums of a word fit 32
    // bits: an image has at most 2^28 tiles. `all` holds any list's length.
    __shared__ unsigned long long wsum[32];
    __shared__ uint32_t wmax[32];
    __shared__ unsigned long long carry, wall[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    uint32_t mx = 0;
    unsigned long long all = 0;
    __syncthreads();
    for (int base = 0; base < tiles; base += 4096) {
        uint32_t v[4];
        unsigned long long t = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int i = base + (int)threadIdx.x * 4 + j;
            v[j] = i < tiles ? count[i] : 0u;
            mx = max(mx, v[j]);
            all += v[j];
            t += gs_word(v[j], ts);
        }
        unsigned long long incl = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            unsigned long long w = wsum[lane], wi = w;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long y = __shfl_up_sync(0xffffffffu, wi, o);
                if (lane >= o) wi += y;
            }
            wsum[lane] = wi - w + carry;
            __syncwarp();
            if (lane == 31) carry += wi;
        }
        __syncthreads();
        unsigned long long run = wsum[warp] + incl - t;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int i = base + (int)threadIdx.x * 4 + j;
            if (i < tiles) {
                const int at = (int)(run >> 32);
                ranges[i] = make_int2(at, at);
                batch_off[i] = (uint32_t)run;
            }
            run += gs_word(v[j], ts);
        }
        __syncthreads();
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) all += __shfl_xor_sync(0xffffffffu, all, o);
    if (lane == 0) {
        wmax[warp] = mx;
        wall[warp] = all;
    }
    __syncthreads();
    if (warp == 0) {
        mx = __reduce_max_sync(0xffffffffu, wmax[lane]);
        all = wall[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) all += __shfl_xor_sync(0xffffffffu, all, o);
        if (lane == 0) {
            stat->total = all;
            stat->batches = (uint32_t)carry;
            stat->most = mx;
        }
    }
}

__device__ __forceinline__ unsigned long long gs_key(const uint32_t *__restrict__ key, int i) {
    return ((unsigned long long)key[i] << 32) | (uint32_t)i;
}

// Each drawn Gaussian outside the queue counted in the tiles it meets, or (LIST)
// its key into their ranges.
template <bool LIST>
__global__ void __launch_bounds__(128) k_gs_list(const int4 *__restrict__ rect,
                                                 const uint32_t *__restrict__ key, int n,
                                                 int tiles_x, int ts, uint32_t *__restrict__ tile_count,
                                                 int2 *__restrict__ ranges,
                                                 unsigned long long *__restrict__ list) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x, i = min(t, n - 1);
    const int4 r = rect[i];
    const bool drawn = t < n && r.z >= r.x && r.w >= r.y;
    const bool queued = gs_tiles(r, drawn, tiles_x, GS_FINE).count > GS_BIG;
    const unsigned long long k = gs_key(key, i);
    const int lane = threadIdx.x & 31;
    gs_for_tiles(gs_tiles(r, drawn && !queued, tiles_x, ts), tiles_x, [&](int tile, unsigned mask) {
        if (!LIST) {
            gs_count_tile(tile, mask, tile_count);
            return;
        }
        const unsigned peers = __match_any_sync(mask, tile);
        const int leader = __ffs(peers) - 1;
        int at = 0;
        if (lane == leader) at = atomicAdd(&ranges[tile].y, __popc(peers));
        at = __shfl_sync(peers, at, leader);
        list[at + __popc(peers & ((1u << lane) - 1u))] = k;
    });
}

// The queued Gaussians' tiles, counted or (LIST) listed: as many warps per
// Gaussian as there are, up to sixteen, so that a few that cover the whole image
// do not leave a warp each with thousands of tiles. (Always sixteen: 100,000 of 45
// tiles each took 478 us to count, most warps without a tile.)
template <bool LIST>
__global__ void __launch_bounds__(256) k_gs_big(const uint32_t *__restrict__ big,
                                                const uint32_t *__restrict__ big_count,
                                                const int4 *__restrict__ rect,
                                                const uint32_t *__restrict__ key, int tiles_x, int ts,
                                                uint32_t *__restrict__ tile_count,
                                                int2 *__restrict__ ranges,
                                                unsigned long long *__restrict__ list,
                                                GsStat *__restrict__ stat) {
    const uint32_t queued = *big_count;
    if (!LIST && blockIdx.x == 0 && threadIdx.x == 0) stat->big = queued;
    if (queued == 0) return;
    const int lane = threadIdx.x & 31;
    const uint32_t warps = gridDim.x * 8, warp = blockIdx.x * 8 + (threadIdx.x >> 5);
    const uint32_t per = min(16u, max(1u, warps / queued)), groups = warps / per;
    const int slice = (int)(warp % per), step = 32 * (int)per;
    if (warp / per >= groups) return;
    for (uint32_t q = warp / per; q < queued; q += groups) {  // far below 2^32
        const int i = (int)big[q];
        const GsTiles g = gs_tiles(rect[i], true, tiles_x, ts);
        const unsigned long long k = LIST ? gs_key(key, i) : 0ull;
#pragma unroll 4
        for (int t = slice * 32 + lane; t < g.count; t += step) {
            const int tile = g.first + t / g.nx * tiles_x + t % g.nx;
            if (LIST)
                list[atomicAdd(&ranges[tile].y, 1)] = k;
            else
                atomicAdd(&tile_count[tile], 1u);
        }
    }
}

// The batches of tile t: batch k holds the entries from gs_threads k on of its
// range; batch_tile[batch_off[t] + k] = t.
__device__ __forceinline__ void gs_write_batches(int t, int cnt, int ts, const uint32_t *__restrict__ batch_off,
                                                 uint32_t *__restrict__ batch_tile) {
    const int nb = (int)gs_batches(cnt, ts);
    for (int k = threadIdx.x; k < nb; k += blockDim.x) batch_tile[batch_off[t] + k] = (uint32_t)t;
}

// Bitonic sort of each tile's keys (one tile per block, at most GS_SORT_MAX);
// the Gaussians' indices in order go to gid. A warp's threads compare within
// 64 consecutive keys while the distance is at most 32, so only the longer
// distances need the block's barrier.
template <int TS>
__global__ void __launch_bounds__(GS_SORT_THREADS) k_gs_tile_sort(
    const int2 *__restrict__ ranges, const unsigned long long *__restrict__ list,
    const uint32_t *__restrict__ batch_off, uint32_t *__restrict__ gid,
    uint32_t *__restrict__ batch_tile) {
    extern __shared__ unsigned long long k[];  // the longest list, rounded up to a power of two
    const int2 rg = ranges[blockIdx.x];
    const int cnt = rg.y - rg.x;
    if (cnt <= 0) return;
    gs_write_batches(blockIdx.x, cnt, TS, batch_off, batch_tile);
    int size = 2;
    while (size < cnt) size <<= 1;
    for (int i = threadIdx.x; i < size; i += GS_SORT_THREADS) k[i] = i < cnt ? list[rg.x + i] : ~0ull;
    __syncthreads();
    for (int len = 2; len <= size; len <<= 1) {
        for (int d = len >> 1; d > 0; d >>= 1) {
            for (int t = threadIdx.x; t < size / 2; t += GS_SORT_THREADS) {
                const int i = 2 * t - (t & (d - 1)), j = i + d;
                const unsigned long long a = k[i], b = k[j];
                if ((a > b) == ((i & len) == 0)) {
                    k[i] = b;
                    k[j] = a;
                }
            }
            if (d > 32)
                __syncthreads();
            else
                __syncwarp();
        }
        if (len >= 64) __syncthreads();  // the next distance is len
    }
    __syncthreads();
    for (int i = threadIdx.x; i < cnt; i += GS_SORT_THREADS) gid[rg.x + i] = (uint32_t)k[i];
}

// The end of every tile's range, and its batches (the radix path; one tile per
// block).
__global__ void __launch_bounds__(64) k_gs_batches(const uint32_t *__restrict__ count, int ts,
                                                   const uint32_t *__restrict__ batch_off,
                                                   int2 *__restrict__ ranges,
                                                   uint32_t *__restrict__ batch_tile) {
    const int cnt = (int)count[blockIdx.x];
    if (threadIdx.x == 0) ranges[blockIdx.x].y = ranges[blockIdx.x].x + cnt;
    gs_write_batches(blockIdx.x, cnt, ts, batch_off, batch_tile);
}

// The radix path: keys and indices of all Gaussians.
__global__ void k_gs_order_init(const uint32_t *__restrict__ key, int n, uint32_t *__restrict__ k,
                                uint32_t *__restrict__ v) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    k[i] = key[i];
    v[i] = (uint32_t)i;
}

// Tiles met by Gaussian order[k] (its pixel rectangle in tiles).
__global__ void k_gs_tile_count(const uint32_t *__restrict__ order, const int4 *__restrict__ rect,
                                int n, int ts, uint32_t *__restrict__ cnt) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int4 r = rect[order[k]];
    uint32_t c = 0;
    if (r.z >= r.x && r.w >= r.y)
        c = (uint32_t)(((r.z >> ts) - (r.x >> ts) + 1) * ((r.w >> ts) - (r.y >> ts) + 1));
    cnt[k] = c;
}

// Exclusive scan of 1024 values per block (256 threads x 4), block totals out; in
// and out may be the same array.
__global__ void __launch_bounds__(256) k_scan1024(const uint32_t *in, int n, uint32_t *out,
                                                  uint32_t *__restrict__ sums) {
    __shared__ uint32_t part[256];
    const int base = blockIdx.x * 1024 + threadIdx.x * 4;
    uint32_t v[4], t = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        v[j] = base + j < n ? in[base + j] : 0u;
        t += v[j];
    }
    part[threadIdx.x] = t;
    __syncthreads();
    for (int off = 1; off < 256; off <<= 1) {
        const uint32_t a = threadIdx.x >= off ? part[threadIdx.x - off] : 0u;
        __syncthreads();
        part[threadIdx.x] += a;
        __syncthreads();
    }
    uint32_t run = part[threadIdx.x] - t;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (base + j < n) out[base + j] = run;
        run += v[j];
    }
    if (threadIdx.x == 255) sums[blockIdx.x] = part[255];
}

// out += the scanned block offsets.
__global__ void k_scan_finish(uint32_t *__restrict__ out, int n, const uint32_t *__restrict__ block_off) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] += block_off[i / 1024];
}

// One entry (tile id, Gaussian) per tile met, written in depth order, a warp per
// Gaussian (20,000 of some 300 tiles: 15 us; a thread each took 181).
__global__ void __launch_bounds__(256) k_gs_duplicate(const uint32_t *__restrict__ order,
                                                      const int4 *__restrict__ rect,
                                                      const uint32_t *__restrict__ off, int n, int tiles_x,
                                                      int ts, uint32_t *__restrict__ tile_key,
                                                      uint32_t *__restrict__ gid) {
    const int k = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (k >= n) return;
    const uint32_t g = order[k], o = off[k];
    const int4 r = rect[g];
    const GsTiles t = gs_tiles(r, r.z >= r.x && r.w >= r.y, tiles_x, ts);
    for (int i = threadIdx.x & 31; i < t.count; i += 32) {
        tile_key[o + i] = (uint32_t)(t.first + i / t.nx * tiles_x + i % t.nx);
        gid[o + i] = g;
    }
}

// ---------------------------------------------------------------- render --

// A batch of the tile's range, from entry b0 on, in shared memory.
template <int TS>
struct GsBatch {
    float4 row[gs_threads(TS)][3];  // mu(2) conic(3) opacity color(3), 3 unused
    int id[gs_threads(TS)];
};

template <int TS>
__device__ __forceinline__ int gs_load_batch(int b0, int end, const uint32_t *__restrict__ list,
                                             const float4 *__restrict__ rows, GsBatch<TS> &s) {
    const int cnt = min(gs_threads(TS), end - b0);
    if ((int)threadIdx.x < cnt) {
        const int g = (int)list[b0 + threadIdx.x];
        s.id[threadIdx.x] = g;
#pragma unroll
        for (int k = 0; k < 3; ++k) s.row[threadIdx.x][k] = rows[3 * (int64_t)g + k];
    }
    __syncthreads();
    return cnt;
}

// KEEP: each batch's colour and transmittance in front of it go to `before`, for
// the backward, which takes each batch by itself (as a test of the pointer in the
// loop instead, 66 us against 59).
template <int TS, bool KEEP>
__global__ void __launch_bounds__(gs_threads(TS)) k_gs_render_fwd(
    GsCam c, unsigned tiles_x, const uint32_t *__restrict__ list, const int2 *__restrict__ ranges,
    const float4 *__restrict__ rows, float *__restrict__ image, float *__restrict__ image_keep,
    const uint32_t *__restrict__ batch_off, float4 *__restrict__ before) {
    constexpr int TILE = 1 << TS, THREADS = gs_threads(TS);
    __shared__ GsBatch<TS> s;
    const int tx0 = (int)(blockIdx.x % tiles_x) * TILE, ty0 = (int)(blockIdx.x / tiles_x) * TILE;
    const int px = tx0 + (threadIdx.x & (TILE - 1)), py = ty0 + threadIdx.x / TILE;
    const float fx = (float)px + 0.5f, fy = (float)py + 0.5f;
    const int2 rg = ranges[blockIdx.x];
    float T = 1.0f, C0 = 0.0f, C1 = 0.0f, C2 = 0.0f;
    float4 *keep = KEEP ? before + (size_t)batch_off[blockIdx.x] * THREADS + threadIdx.x : nullptr;
    for (int b0 = rg.x; b0 < rg.y; b0 += THREADS, keep += THREADS) {
        const int cnt = gs_load_batch(b0, rg.y, list, rows, s);
        if (KEEP) *keep = make_float4(C0, C1, C2, T);
#pragma unroll 4
        for (int k = 0; k < cnt; ++k) {
            const float4 r = s.row[k][0], u = s.row[k][1];
            const float dx = fx - r.x, dy = fy - r.y;
            const float q = r.z * dx * dx + 2.0f * r.w * dx * dy + u.x * dy * dy;
            if (q <= 9.0f) {
                const float a = u.y * expf(-0.5f * q);
                const float w = T * a;
                C0 += w * u.z;
                C1 += w * u.w;
                C2 += w * s.row[k][2].x;
                T *= 1.0f - a;
            }
        }
        __syncthreads();
    }
    if (px < c.width && py < c.height) {
        const int64_t hw = (int64_t)c.width * c.height, pix = (int64_t)py * c.width + px;
        image[pix] = C0;
        image[hw + pix] = C1;
        image[2 * hw + pix] = C2;
        image_keep[pix] = C0;
        image_keep[hw + pix] = C1;
        image_keep[2 * hw + pix] = C2;
    }
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sums of eight values over the warp: lane L receives the total of value
// (L >> 2) of v. Each of the first three steps halves the values a lane still
// carries (it sends one half and adds the other's counterpart), so 9 shuffles
// instead of 40.
__device__ __forceinline__ float warp_sum8(const float (&v)[8]) {
    const int lane = threadIdx.x & 31;
    float a[4], b[2], t;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const bool up = lane & 16;
        const float keep = up ? v[4 + j] : v[j], send = up ? v[j] : v[4 + j];
        a[j] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const bool up = lane & 8;
        const float keep = up ? a[2 + j] : a[j], send = up ? a[j] : a[2 + j];
        b[j] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
    {
        const bool up = lane & 4;
        const float keep = up ? b[1] : b[0], send = up ? b[0] : b[1];
        t = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    t += __shfl_xor_sync(0xffffffffu, t, 2);
    t += __shfl_xor_sync(0xffffffffu, t, 1);
    return t;
}

// One batch of a tile's list per block, from the colour and transmittance the
// forward pass kept in front of it: as one block per tile the longest list's
// serial walk was the kernel's time (235 entries on the 1,300 tiles that the
// 100,284-Gaussian sheet meets: 17 warps per SM). Per pixel, front to back:
// w = T alpha, dL/dc += g w, dL/dalpha = g . (T c - (C - C_<=i) / (1 - alpha)).
// With s = exp(-q/2) dL/dalpha, d = pixel - mu' and dL/dq = -s opacity / 2, all
// of a Gaussian's gradients are linear in the sums over pixels of s, s d and
// s d d^T, which k_gs_preprocess_bwd turns into dL/d(mu', conic). Each warp's
// nine sums go to the Gaussian's row of g2d (GS_ROW floats, so nine
// neighbouring words: two sectors) from nine lanes at once. WALK: without
// `before`, one tile per block, its batches one after the other.
template <int TS, bool WALK>
__global__ void __launch_bounds__(gs_threads(TS)) k_gs_render_bwd(
    GsCam c, unsigned tiles_x, const uint32_t *__restrict__ list, const int2 *__restrict__ ranges,
    const float4 *__restrict__ rows, const uint32_t *__restrict__ batch_tile,
    const uint32_t *__restrict__ batch_off, const float4 *__restrict__ before,
    const float *__restrict__ image_keep, const float *__restrict__ g_image,
    float *__restrict__ g2d) {
    constexpr int TILE = 1 << TS, THREADS = gs_threads(TS);
    __shared__ GsBatch<TS> s;
    const unsigned tile = WALK ? blockIdx.x : batch_tile[blockIdx.x];
    const int tx0 = (int)(tile % tiles_x) * TILE, ty0 = (int)(tile / tiles_x) * TILE;
    const int px = tx0 + (threadIdx.x & (TILE - 1)), py = ty0 + threadIdx.x / TILE;
    const bool inside = px < c.width && py < c.height;
    const float fx = (float)px + 0.5f, fy = (float)py + 0.5f;
    const int64_t hw = (int64_t)c.width * c.height, pix = (int64_t)py * c.width + px;
    float Cf[3] = {0.0f, 0.0f, 0.0f}, gC[3] = {0.0f, 0.0f, 0.0f};
    if (inside) {
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
            Cf[ch] = image_keep[ch * hw + pix];
            gC[ch] = g_image[ch * hw + pix];
        }
    }
    const float4 b4 = WALK ? make_float4(0.0f, 0.0f, 0.0f, 1.0f)
                           : before[(size_t)blockIdx.x * THREADS + threadIdx.x];
    float T = b4.w, Cl[3] = {b4.x, b4.y, b4.z};
    const int lane = threadIdx.x & 31;
    const int2 rg = ranges[tile];
    if (WALK && rg.x >= rg.y) return;
    int b0 = rg.x + (WALK ? 0 : (int)(blockIdx.x - batch_off[tile]) * THREADS);
    do {
        const int cnt = gs_load_batch(b0, rg.y, list, rows, s);
#pragma unroll 2
        for (int k = 0; k < cnt; ++k) {
            const float4 r = s.row[k][0], u = s.row[k][1];
            const float dx = fx - r.x, dy = fy - r.y;
            const float q = r.z * dx * dx + 2.0f * r.w * dx * dy + u.x * dy * dy;
            const bool hit = inside && q <= 9.0f;
            if (!__any_sync(0xffffffffu, hit)) continue;
            // s d (2), s d d^T (3), s, dL/dcolor (3)
            float v[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f}, v8 = 0.0f;
            if (hit) {
                const float col[3] = {u.z, u.w, s.row[k][2].x};
                const float e = expf(-0.5f * q);
                const float a = u.y * e;
                const float w = T * a, inv = 1.0f / (1.0f - a);
                float dA = 0.0f;
#pragma unroll
                for (int ch = 0; ch < 3; ++ch) {
                    Cl[ch] += w * col[ch];
                    dA += gC[ch] * (T * col[ch] - (Cf[ch] - Cl[ch]) * inv);
                }
                v[5] = dA * e;
                v[0] = v[5] * dx;
                v[1] = v[5] * dy;
                v[2] = v[0] * dx;
                v[3] = v[0] * dy;
                v[4] = v[1] * dy;
                v[6] = gC[0] * w;
                v[7] = gC[1] * w;
                v8 = gC[2] * w;
                T *= 1.0f - a;
            }
            const float t = warp_sum8(v), t8 = warp_sum(v8);
            // lane 4 j adds value j, lane 1 value 8
            const int j = (lane & 3) == 0 ? lane >> 2 : 8;
            const float mine = j == 8 ? t8 : t;
            if (((lane & 3) == 0 || lane == 1) && mine != 0.0f)
                atomicAdd(&g2d[(int64_t)s.id[k] * GS_ROW + j], mine);
        }
        if (WALK) __syncthreads();
        b0 += THREADS;
    } while (WALK && b0 < rg.y);
}

// The 2D gradients of each Gaussian (k_gs_render_bwd's sums) -> dL/dx, dL/dF (and the
// colour and opacity gradients), accumulated into the caller's buffers.
__global__ void k_gs_preprocess_bwd(GsCam c, const float *__restrict__ x,
                                    const float *__restrict__ F, const float *__restrict__ s0,
                                    const float *__restrict__ opacity, int n,
                                    const float *__restrict__ g2d, float *__restrict__ g_x,
                                    float *__restrict__ g_F, float *__restrict__ g_color,
                                    float *__restrict__ g_opacity) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t nn = n;
    const float4 *gr = reinterpret_cast<const float4 *>(g2d + (int64_t)i * GS_ROW);
    const float4 ga = gr[0], gb = gr[1];
    float gv[9] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y, gb.z, gb.w, gr[2].x};
    if (g_opacity) g_opacity[i] += gv[5];
    if (g_color) {
        g_color[i] += gv[6];
        g_color[nn + i] += gv[7];
        g_color[2 * nn + i] += gv[8];
    }
    float Fm[3][3], a6[6], S[6];
    load_F(F, nn, i, Fm);
#pragma unroll
    for (int k = 0; k < 6; ++k) a6[k] = s0[k * nn + i];
    cov_update(Fm, a6, S);
    const float xp[3] = {x[i], x[nn + i], x[2 * nn + i]};
    GsProj p;
    gs_project(c, xp, S, p);
    if (!p.visible) return;
    {  // dL/dmu' = -2 sum dL/dq A d, dL/dA = sum dL/dq d d^T, dL/dq = -s o / 2
        const float o = opacity[i], m0 = gv[0], m1 = gv[1];
        gv[0] = o * (p.conic[0] * m0 + p.conic[1] * m1);
        gv[1] = o * (p.conic[1] * m0 + p.conic[2] * m1);
        gv[2] *= -0.5f * o;
        gv[3] *= -o;
        gv[4] *= -0.5f * o;
    }
    // conic A = Sigma'^-1: dL/dSigma' = -A Abar A, Abar = [[ga, gb/2], [gb/2, gc]]
    const float A00 = p.conic[0], A01 = p.conic[1], A11 = p.conic[2];
    const float b00 = gv[2], b01 = 0.5f * gv[3], b11 = gv[4];
    const float M00 = b00 * A00 + b01 * A01, M01 = b00 * A01 + b01 * A11;  // Abar A
    const float M10 = b01 * A00 + b11 * A01, M11 = b01 * A01 + b11 * A11;
    const float G00 = -(A00 * M00 + A01 * M10), G01 = -(A00 * M01 + A01 * M11);
    const float G11 = -(A01 * M01 + A11 * M11);
    const float G[2][2] = {{G00, G01}, {G01, G11}};
    const float J[2][3] = {{p.J[0], p.J[1], p.J[2]}, {p.J[3], p.J[4], p.J[5]}};
    float V[3][3];
    sym_full(p.V, V);
    // dL/dV = J^T G J ; dL/dJ = 2 G J V
    float GJ[2][3];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int b = 0; b < 3; ++b) GJ[r][b] = G[r][0] * J[0][b] + G[r][1] * J[1][b];
    float dV[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) dV[a][b] = J[0][a] * GJ[0][b] + J[1][a] * GJ[1][b];
    float dJ[2][3];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            dJ[r][b] = 2.0f * (GJ[r][0] * V[0][b] + GJ[r][1] * V[1][b] + GJ[r][2] * V[2][b]);
    // dL/dSigma = R^T dV R
    float RtdV[3][3], dS[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            RtdV[a][b] = c.R[a] * dV[0][b] + c.R[3 + a] * dV[1][b] + c.R[6 + a] * dV[2][b];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            dS[a][b] = RtdV[a][0] * c.R[b] + RtdV[a][1] * c.R[3 + b] + RtdV[a][2] * c.R[6 + b];
    // dL/dF = 2 dS F Sigma0
    float S0[3][3], FS0[3][3];
    sym_full(a6, S0);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            FS0[a][b] = Fm[a][0] * S0[0][b] + Fm[a][1] * S0[1][b] + Fm[a][2] * S0[2][b];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
            g_F[(3 * a + b) * nn + i] +=
                2.0f * (dS[a][0] * FS0[0][b] + dS[a][1] * FS0[1][b] + dS[a][2] * FS0[2][b]);
    // camera-space centre: from mu' and from J
    const float iz = 1.0f / p.t[2], iz2 = iz * iz, iz3 = iz2 * iz;
    float gt[3];
    gt[0] = gv[0] * c.fx * iz + dJ[0][2] * (-c.fx * iz2);
    gt[1] = gv[1] * c.fy * iz + dJ[1][2] * (-c.fy * iz2);
    gt[2] = -gv[0] * c.fx * p.t[0] * iz2 - gv[1] * c.fy * p.t[1] * iz2 +
            dJ[0][0] * (-c.fx * iz2) + dJ[0][2] * (2.0f * c.fx * p.t[0] * iz3) +
            dJ[1][1] * (-c.fy * iz2) + dJ[1][2] * (2.0f * c.fy * p.t[1] * iz3);
#pragma unroll
    for (int b = 0; b < 3; ++b)
        g_x[b * nn + i] += c.R[b] * gt[0] + c.R[3 + b] * gt[1] + c.R[6 + b] * gt[2];
}

// Block sum of term, added to *loss times scale by one thread.
__device__ __forceinline__ void block_add(float term, float scale, float *loss, float bias = 0.0f) {
    __shared__ float red[8];
    const int t = threadIdx.y * blockDim.x + threadIdx.x;
    term = warp_sum(term);
    if ((t & 31) == 0) red[t >> 5] = term;
    __syncthreads();
    if (t < 32) {
        float s = t < 8 ? red[t] : 0.0f;
        s = warp_sum(s);
        if (t == 0) atomicAdd(loss, scale * s + bias);
    }
}

// Four values per thread, so that a block's one atomic on the loss stands for
// 1024 of them (the 3,072 atomics of a 3 x 512 x 512 image on one address took
// most of 7.4 us).
__global__ void __launch_bounds__(256) k_image_l1(const float *__restrict__ img,
                                                  const float *__restrict__ target, int64_t n,
                                                  float weight, float *__restrict__ loss,
                                                  float *__restrict__ g) {
    float term = 0.0f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int64_t i = ((int64_t)blockIdx.x * 4 + j) * 256 + threadIdx.x;
        if (i < n) {
            const float d = img[i] - target[i];
            term += fabsf(d);
            if (g) g[i] += weight * (d > 0.0f ? 1.0f : (d < 0.0f ? -1.0f : 0.0f));
        }
    }
    block_add(term, weight, loss);
}

// ----------------------------------------------------------------- D-SSIM --
// The structural term of L_render: 1 - mean SSIM with local statistics under
// an 11 x 11 Gaussian window (sigma 1.5, zero outside the image), computed as
// separable blurs within a 32 x 16 tile: the tile of both images with a halo of
// 5 in shared memory, horizontal sums of the five maps x, y, x^2, y^2, x y of
// its 26 rows, then vertical sums, so that the maps never reach memory. The
// gradient blurs the per-pixel partials back the same way (the window is
// symmetric, so the transposed blur is the blur). One launch each; as six
// launches over whole maps in memory the two took 125 us at 3 x 512 x 512.

struct SsimWin {
    float w[11];
};

constexpr int SS_X = 32, SS_Y = 16, SS_H = 5;  // tile and halo; 32 x 8 threads
constexpr int SS_RX = SS_X + 2 * SS_H, SS_RY = SS_Y + 2 * SS_H;
// Row strides in shared memory: a warp's horizontal sums read and write four
// columns apart in four rows, which strides of 42 and 32 put on the same banks
// two and four times (two views at 512 x 512, all kernels: 2.4% less).
constexpr int SS_LT = SS_RX + 1, SS_LH = SS_X + 1;

// First pixel of this block's tile, and the offset of its plane (blocks run over
// the tiles of all planes, x fastest).
__device__ __forceinline__ int2 ss_tile(int H, int W) {
    const unsigned tx = (W + SS_X - 1) / SS_X, ty = (H + SS_Y - 1) / SS_Y;
    return make_int2((int)(blockIdx.x % tx) * SS_X, (int)(blockIdx.x / tx % ty) * SS_Y);
}
__device__ __forceinline__ int64_t ss_plane(int H, int W) {
    const unsigned tx = (W + SS_X - 1) / SS_X, ty = (H + SS_Y - 1) / SS_Y;
    return (int64_t)(blockIdx.x / (tx * ty)) * H * W;
}

// The tile at (x0, y0) of a plane with its halo, zero outside the image.
__device__ __forceinline__ void ss_load(const float *__restrict__ plane, int H, int W, int x0, int y0,
                                        float (*t)[SS_LT]) {
    for (int i = threadIdx.y * SS_X + threadIdx.x; i < SS_RX * SS_RY; i += 256) {
        const int cx = i % SS_RX, cy = i / SS_RX, px = x0 + cx - SS_H, py = y0 + cy - SS_H;
        t[cy][cx] = px >= 0 && px < W && py >= 0 && py < H ? plane[(int64_t)py * W + px] : 0.0f;
    }
}

// SSIM per pixel from the blurred maps (mu_x, mu_y, <x^2>, <y^2>, <x y>);
// loss += weight (1 - mean SSIM); part = weight * dD/d(mu_x, <x^2>, <x y>).
__global__ void __launch_bounds__(256) k_ssim(const float *__restrict__ x,
                                              const float *__restrict__ y, int H, int W, int64_t n,
                                              SsimWin k, float weight, float *__restrict__ loss,
                                              float *__restrict__ part) {
    __shared__ float tx[SS_RY][SS_LT], ty[SS_RY][SS_LT];
    __shared__ float h[5][SS_RY][SS_LH];
    const int2 at = ss_tile(H, W);
    const int x0 = at.x, y0 = at.y;
    const int64_t plane = ss_plane(H, W);
    ss_load(x + plane, H, W, x0, y0, tx);
    ss_load(y + plane, H, W, x0, y0, ty);
    __syncthreads();
    // four neighbouring sums per thread from 14 values of its row
    const int tid = threadIdx.y * SS_X + threadIdx.x;
    if (tid < SS_RY * SS_X / 4) {
        const int r = tid / (SS_X / 4), c4 = tid % (SS_X / 4) * 4;
        float a[14], b[14];
#pragma unroll
        for (int i = 0; i < 14; ++i) {
            a[i] = tx[r][c4 + i];
            b[i] = ty[r][c4 + i];
        }
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            float s[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int d = 0; d < 11; ++d) {
                const float w = k.w[d];
                s[0] += w * a[o + d];
                s[1] += w * b[o + d];
                s[2] += w * a[o + d] * a[o + d];
                s[3] += w * b[o + d] * b[o + d];
                s[4] += w * a[o + d] * b[o + d];
            }
#pragma unroll
            for (int m = 0; m < 5; ++m) h[m][r][c4 + o] = s[m];
        }
    }
    __syncthreads();
    const float C1 = 0.01f * 0.01f, C2 = 0.03f * 0.03f;
    const float scale = -weight / (float)n;
    float term = 0.0f;
    float vv[2][5];  // two neighbouring rows per thread from 12 values of its column
#pragma unroll
    for (int m = 0; m < 5; ++m) {
        float t[12];
#pragma unroll
        for (int i = 0; i < 12; ++i) t[i] = h[m][2 * threadIdx.y + i][threadIdx.x];
#pragma unroll
        for (int o = 0; o < 2; ++o) {
            vv[o][m] = 0.0f;
#pragma unroll
            for (int d = 0; d < 11; ++d) vv[o][m] += k.w[d] * t[o + d];
        }
    }
#pragma unroll
    for (int o = 0; o < 2; ++o) {
        const int r = 2 * threadIdx.y + o;
        const float(&v)[5] = vv[o];
        const int px = x0 + threadIdx.x, py = y0 + r;
        if (px >= W || py >= H) continue;
        const float A = v[0], Ay = v[1], B = v[2], Byy = v[3], Cxy = v[4];
        const float n1 = 2.0f * A * Ay + C1, n2 = 2.0f * (Cxy - A * Ay) + C2;
        const float d1 = A * A + Ay * Ay + C1, d2 = (B - A * A) + (Byy - Ay * Ay) + C2;
        const float dd = d1 * d2;
        const float S = n1 * n2 / dd;
        term += S;
        if (part) {
            const int64_t i = plane + (int64_t)py * W + px;
            const float dA = 2.0f * Ay * (n2 - n1) / dd - 2.0f * A * n1 * n2 * (d2 - d1) / (dd * dd);
            const float dB = -S / d2;
            const float dC = 2.0f * n1 / dd;
            part[i] = scale * dA;
            part[n + i] = scale * dB;
            part[2 * n + i] = scale * dC;
        }
    }
    block_add(term, scale, loss, blockIdx.x == 0 ? weight : 0.0f);
}

// g += blur(p_mu) + 2 x blur(p_xx) + y blur(p_xy)
__global__ void __launch_bounds__(256) k_ssim_grad(const float *__restrict__ x,
                                                   const float *__restrict__ y,
                                                   const float *__restrict__ part, int H, int W,
                                                   int64_t n, SsimWin k, float *__restrict__ g) {
    __shared__ float t[3][SS_RY][SS_LT];
    __shared__ float h[3][SS_RY][SS_LH];
    const int2 at = ss_tile(H, W);
    const int x0 = at.x, y0 = at.y;
    const int64_t plane = ss_plane(H, W);
#pragma unroll
    for (int m = 0; m < 3; ++m) ss_load(part + m * n + plane, H, W, x0, y0, t[m]);
    __syncthreads();
    const int tid = threadIdx.y * SS_X + threadIdx.x;
    if (tid < SS_RY * SS_X / 4) {
        const int r = tid / (SS_X / 4), c4 = tid % (SS_X / 4) * 4;
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            float a[14];
#pragma unroll
            for (int i = 0; i < 14; ++i) a[i] = t[m][r][c4 + i];
#pragma unroll
            for (int o = 0; o < 4; ++o) {
                float s = 0.0f;
#pragma unroll
                for (int d = 0; d < 11; ++d) s += k.w[d] * a[o + d];
                h[m][r][c4 + o] = s;
            }
        }
    }
    __syncthreads();
    float b[2][3];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        float a[12];
#pragma unroll
        for (int i = 0; i < 12; ++i) a[i] = h[m][2 * threadIdx.y + i][threadIdx.x];
#pragma unroll
        for (int o = 0; o < 2; ++o) {
            b[o][m] = 0.0f;
#pragma unroll
            for (int d = 0; d < 11; ++d) b[o][m] += k.w[d] * a[o + d];
        }
    }
#pragma unroll
    for (int o = 0; o < 2; ++o) {
        const int px = x0 + threadIdx.x, py = y0 + 2 * threadIdx.y + o;
        if (px >= W || py >= H) continue;
        const int64_t i = plane + (int64_t)py * W + px;
        g[i] += b[o][0] + 2.0f * x[i] * b[o][1] + y[i] * b[o][2];
    }
}

static SsimWin ssim_window() {
    SsimWin k;
    double w[11], sum = 0.0;
    for (int i = 0; i < 11; ++i) {
        w[i] = exp(-((i - 5.0) * (i - 5.0)) / (2.0 * 1.5 * 1.5));
        sum += w[i];
    }
    for (int i = 0; i < 11; ++i) k.w[i] = (float)(w[i] / sum);
    return k;
}

// A device buffer of the handle that grows when a call needs it to.
template <typename T>
struct GsBuf {
    T *p = nullptr;
    int64_t cap = 0;

    void free() {
        cudaFree(p);
        p = nullptr;
        cap = 0;
    }
    // At least `need` elements, with half as much again as before when it grows
    // and that can be had.
    dw_status grow(int64_t need, const char *what) {
        if (need <= cap) return DW_OK;
        const int64_t more = cap / 2 * 3;
        free();
        cudaError_t e = cudaErrorMemoryAllocation;
        for (int64_t want : {std::max(need, more), need}) {
            e = cudaMalloc((void **)&p, sizeof(T) * (size_t)want);
            if (e == cudaSuccess) {
                cap = want;
                return DW_OK;
            }
            cudaGetLastError();
            p = nullptr;
            if (e != cudaErrorMemoryAllocation || want == need) break;
        }
        return cuda_fail(e, what);
    }
};

struct GsHandle {
    int64_t cap = 0;
    int width = 0, height = 0;
    float4 *rows = nullptr;          // [cap][3] packed projected Gaussians
    float *g2d = nullptr;            // [cap][GS_ROW] their gradients
    float *image = nullptr;
    int4 *rect = nullptr;
    uint32_t *key = nullptr;         // [cap] depth bits
    uint32_t *tile_count = nullptr;  // [tiles]
    int2 *ranges = nullptr;          // [tiles]
    uint32_t *batch_off = nullptr;   // [tiles] first batch of each tile
    uint32_t *big = nullptr;         // [cap + 1] queue of Gaussians meeting many tiles; [cap]: its length
    GsStat *stat = nullptr;
    // tile list: keys as filled (the shared-memory sort), Gaussians in order
    GsBuf<unsigned long long> lkey;
    GsBuf<uint32_t> lgid;
    // batches of the list: their tiles, and each pixel's colour and
    // transmittance in front of them (empty if there was no memory for it)
    GsBuf<uint32_t> batch_tile;
    GsBuf<float4> before;
    bool kept = false;               // the last gs_render filled `before`
    uint32_t batches = 0;            // of the last gs_render
    // the radix path's buffers: depth sort and tile-list sort in turn
    GsBuf<uint32_t> rk[2], rv[2], rcounts, tcnt, toff, bsum;
    const uint32_t *list = nullptr;  // the sorted Gaussian column of the last gs_render
    int ts = GS_FINE, tiles_x = 0, tiles_y = 0;  // tiles of the last gs_render
    int last_n = -1;  // Gaussians of the last gs_render
    // inputs and camera of the last gs_render (the backward must see the same)
    const void *last_in[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    dw_camera last_cam{};
};

static GsCam to_cam(const dw_camera &c) {
    GsCam g;
    for (int k = 0; k < 9; ++k) g.R[k] = c.R[k];
    for (int k = 0; k < 3; ++k) g.T[k] = c.T[k];
    g.fx = c.fx;
    g.fy = c.fy;
    g.cx = c.cx;
    g.cy = c.cy;
    g.width = c.width;
    g.height = c.height;
    g.near_z = c.near_z;
    return g;
}

// Exclusive scan of n values, in place with in = out; sums: one word per 1024.
// k_rs_scan alone, whose threads read their shares a word at a time, took 534 us
// for the sorts of a call with 100,000 Gaussians and 4.5 million entries; now 70.
static void gs_scan_counts(const uint32_t *in, int n, uint32_t *out, uint32_t *sums, cudaStream_t s) {
    if (n <= 4096 && in == out) {
        k_rs_scan<<<1, 1024, 0, s>>>(out, n);
        return;
    }
    const int nb = (n + 1023) / 1024;
    k_scan1024<<<nb, 256, 0, s>>>(in, n, out, sums);
    k_rs_scan<<<1, 1024, 0, s>>>(sums, nb);
    k_scan_finish<<<grid_for(n, 256), 256, 0, s>>>(out, n, sums);
}

// Stable LSD radix sort of (k, v) by the low 8 * passes bits of k; the
// result ends in (k, v) (the pointers are swapped as the passes alternate).
static void radix_sort(uint32_t *&k, uint32_t *&v, uint32_t *&k2, uint32_t *&v2, int n,
                       int passes, uint32_t *counts, uint32_t *sums, cudaStream_t s) {
    const int nb = (n + RS_TILE - 1) / RS_TILE;
    for (int p = 0; p < passes; ++p) {
        const int shift = 8 * p;
        k_rs_hist<<<nb, RS_THREADS, 0, s>>>(k, n, shift, nb, counts);
        gs_scan_counts(counts, 256 * nb, counts, sums, s);
        k_rs_scatter<<<nb, RS_THREADS, 0, s>>>(k, v, k2, v2, n, shift, nb, counts);
        std::swap(k, k2);
        std::swap(v, v2);
    }
}

}  // namespace dw

using namespace dw;

struct dw_gs_s : GsHandle {};

static void gs_set_tiles(dw_gs h, int ts) {
    h->ts = ts;
    h->tiles_x = ((h->width - 1) >> ts) + 1;
    h->tiles_y = ((h->height - 1) >> ts) + 1;
}

static void gs_list_free(dw_gs h) {
    h->lkey.free();
    h->lgid.free();
    h->batch_tile.free();
    h->before.free();
    for (int k = 0; k < 2; ++k) {
        h->rk[k].free();
        h->rv[k].free();
    }
    h->rcounts.free();
    h->tcnt.free();
    h->toff.free();
    h->bsum.free();
}

// Buffers for the counted list: 12 bytes per entry where the tiles are sorted
// in shared memory, 16 for the radix sorts, and 16 per entry (of full batches)
// of `before`, which is done without when it cannot be had.
static dw_status gs_list_reserve(dw_gs h, int64_t n, const GsStat &stat) {
    const int64_t m = (int64_t)stat.total, batch = stat.batches, both = std::max(n, m);
    dw_status st = h->lgid.grow(m, "gs_render (tile list)");
    if (stat.most <= GS_SORT_MAX) {
        if (st == DW_OK) st = h->lkey.grow(m, "gs_render (tile list)");
    } else {
        if (st == DW_OK) st = h->rk[0].grow(both, "gs_render (radix sort)");
        if (st == DW_OK) st = h->rk[1].grow(both, "gs_render (radix sort)");
        if (st == DW_OK) st = h->rv[0].grow(both, "gs_render (radix sort)");
        if (st == DW_OK) st = h->rv[1].grow(n, "gs_render (radix sort)");
        const int64_t counts = 256 * ((both - 1) / RS_TILE + 1);
        if (st == DW_OK) st = h->rcounts.grow(counts, "gs_render (radix sort)");
        if (st == DW_OK) st = h->tcnt.grow(n, "gs_render (radix sort)");
        if (st == DW_OK) st = h->toff.grow(n, "gs_render (radix sort)");
        if (st == DW_OK) st = h->bsum.grow((std::max(n, counts) - 1) / 1024 + 1, "gs_render (radix sort)");
    }
    if (st == DW_OK) st = h->batch_tile.grow(batch, "gs_render (list batches)");
    if (st == DW_OK) h->kept = h->before.grow(batch * gs_threads(h->ts), "gs_render (list batches)") == DW_OK;
    return st;
}

// The tile lists by two stable sorts: all Gaussians by depth, then the list,
// filled in that order, by tile.
static void gs_list_radix(dw_gs h, int n, int64_t m, cudaStream_t s) {
    uint32_t *ka = h->rk[0].p, *va = h->rv[0].p, *kb = h->rk[1].p, *vb = h->rv[1].p;
    uint32_t *tcnt = h->tcnt.p, *toff = h->toff.p, *bsum = h->bsum.p;
    k_gs_order_init<<<grid_for(n, 256), 256, 0, s>>>(h->key, n, ka, va);
    radix_sort(ka, va, kb, vb, n, 4, h->rcounts.p, bsum, s);  // depth order in va (an even number of passes)
    k_gs_tile_count<<<grid_for(n, 256), 256, 0, s>>>(va, h->rect, n, h->ts, tcnt);
    gs_scan_counts(tcnt, n, toff, bsum, s);
    // the list: tile keys to kb, Gaussians to lgid, then both sorted (the depth
    // order in va is read before the sort's second buffers overwrite it)
    k_gs_duplicate<<<grid_for(n, 8), 256, 0, s>>>(va, h->rect, toff, n, h->tiles_x, h->ts, kb,
                                                    h->lgid.p);
    int bits = 1;
    while ((1ll << bits) < (int64_t)h->tiles_x * h->tiles_y) ++bits;
    uint32_t *lk = kb, *lv = h->lgid.p, *lk2 = ka, *lv2 = va;
    radix_sort(lk, lv, lk2, lv2, (int)m, (bits + 7) / 8, h->rcounts.p, bsum, s);
    h->list = lv;
}

extern "C" dw_status gs_create(int64_t max_gaussians, int32_t width, int32_t height, dw_gs *out) {
    DW_REQUIRE(out, "out must not be NULL");
    *out = nullptr;
    DW_REQUIRE(max_gaussians >= 1 && max_gaussians < (1ll << 30), "max_gaussians must be in [1, 2^30)");
    DW_REQUIRE(width >= 1 && height >= 1 && (int64_t)width * height < (1ll << 31),
               "image size must be positive and below 2^31 pixels");
    dw_gs h = new (std::nothrow) dw_gs_s();
    if (!h) {
        set_error("out of host memory");
        return DW_ERR_OOM;
    }
    h->cap = max_gaussians;
    h->width = width;
    h->height = height;
    gs_set_tiles(h, GS_FINE);  // the coarse tiles are fewer
    const size_t n = (size_t)max_gaussians, tiles = (size_t)h->tiles_x * h->tiles_y;
    cudaError_t e = cudaMalloc((void **)&h->rows, sizeof(float4) * 3 * n);
    if (e == cudaSuccess) e = cudaMalloc((void **)&h->g2d, sizeof(float) * GS_ROW * n);
    if (e == cudaSuccess) e = cudaMalloc((void **)&h->rect, sizeof(int4) * n);
    if (e == cudaSuccess) e = cudaMalloc((void **)&h->key, sizeof(uint32_t) * n);
    if (e == cudaSuccess)
        e = cudaMalloc((void **)&h->image, sizeof(float) * 3 * (size_t)width * height);
    if (e == cudaSuccess) e = cudaMalloc((void **)&h->tile_count, sizeof(uint32_t) * tiles);
    if (e == cudaSuccess) e = cudaMalloc((void **)&h->ranges, sizeof(int2) * tiles);
    if (e == cudaSuccess) e = cudaMalloc((void **)&h->batch_off, sizeof(uint32_t) * tiles);
    if (e == cudaSuccess) e = cudaMalloc((void **)&h->big, sizeof(uint32_t) * (n + 1));
    if (e == cudaSuccess) e = cudaMalloc((void **)&h->stat, sizeof(GsStat));
    if (e != cudaSuccess) {
        dw_status st = cuda_fail(e, "gs_create");
        gs_destroy(h);
        return st;
    }
    *out = h;
    return DW_OK;
}

extern "C" dw_status gs_destroy(dw_gs h) {
    if (!h) return DW_OK;
    cudaFree(h->rows);
    cudaFree(h->g2d);
    cudaFree(h->rect);
    cudaFree(h->key);
    cudaFree(h->image);
    cudaFree(h->tile_count);
    cudaFree(h->ranges);
    cudaFree(h->batch_off);
    cudaFree(h->big);
    cudaFree(h->stat);
    gs_list_free(h);
    delete h;
    return DW_OK;
}

extern "C" dw_status gs_covariance(const float *F, const float *sigma0, int64_t n, float *sigma,
                                   dw_stream stream) {
    DW_REQUIRE(n >= 0, "n must be >= 0");
    if (n == 0) return DW_OK;
    DW_REQUIRE(F && sigma0 && sigma, "F, sigma0 and sigma must not be NULL");
    k_gs_covariance<<<grid_for(n, 256), 256, 0, as_stream(stream)>>>(F, sigma0, n, sigma);
    DW_LAUNCHED("k_gs_covariance");
    return DW_OK;
}

static dw_status gs_check(dw_gs h, const dw_camera *cam, const float *x, const float *F,
                          const float *sigma0, const float *color, const float *opacity,
                          int64_t n) {
    DW_REQUIRE(h && cam, "handle and camera must not be NULL");
    DW_REQUIRE(n >= 0 && n <= h->cap, "n must be in [0, max_gaussians]");
    DW_REQUIRE(cam->width == h->width && cam->height == h->height,
               "camera image size differs from the handle's");
    DW_REQUIRE(cam->fx > 0.0f && cam->fy > 0.0f && cam->near_z > 0.0f,
               "focal lengths and near must be > 0");
    DW_REQUIRE(n == 0 || (x && F && sigma0 && color && opacity), "inputs must not be NULL");
    return DW_OK;
}

// The scan of the tiles' counts, and what the host needs of it (waits for s).
static dw_status gs_scan(dw_gs h, GsStat &stat, cudaStream_t s) {
    k_gs_tile_scan<<<1, 1024, 0, s>>>(h->tile_count, h->tiles_x * h->tiles_y, h->ts, h->ranges,
                                      h->batch_off, h->stat);
    DW_CUDA(cudaMemcpyAsync(&stat, h->stat, sizeof stat, cudaMemcpyDeviceToHost, s));
    DW_CUDA(cudaStreamSynchronize(s));
    return DW_OK;
}

// The Gaussians projected and counted in the fine tiles they meet.
static dw_status gs_count(dw_gs h, const GsCam &c, const float *x, const float *F, const float *sigma0,
                          const float *color, const float *opacity, int n, GsStat &stat,
                          cudaStream_t s) {
    uint32_t *queued = h->big + h->cap;
    DW_CUDA(cudaMemsetAsync(h->tile_count, 0, sizeof(uint32_t) * (size_t)h->tiles_x * h->tiles_y, s));
    DW_CUDA(cudaMemsetAsync(queued, 0, sizeof(uint32_t), s));
    k_gs_preprocess<<<grid_for(n, 128), 128, 0, s>>>(c, x, F, sigma0, color, opacity, n, h->tiles_x,
                                                     h->rows, h->rect, h->key, h->tile_count, h->big,
                                                     queued);
    k_gs_big<false><<<GS_BIG_CTAS, 256, 0, s>>>(h->big, queued, h->rect, h->key, h->tiles_x, h->ts,
                                                h->tile_count, h->ranges, h->lkey.p, h->stat);
    return gs_scan(h, stat, s);
}

// The projected Gaussians counted again, in the tiles set now.
static dw_status gs_recount(dw_gs h, int n, GsStat &stat, cudaStream_t s) {
    DW_CUDA(cudaMemsetAsync(h->tile_count, 0, sizeof(uint32_t) * (size_t)h->tiles_x * h->tiles_y, s));
    k_gs_list<false><<<grid_for(n, 128), 128, 0, s>>>(h->rect, h->key, n, h->tiles_x, h->ts,
                                                      h->tile_count, h->ranges, h->lkey.p);
    k_gs_big<false><<<GS_BIG_CTAS, 256, 0, s>>>(h->big, h->big + h->cap, h->rect, h->key, h->tiles_x,
                                                h->ts, h->tile_count, h->ranges, h->lkey.p, h->stat);
    return gs_scan(h, stat, s);
}

// The counted tiles' lists in order, and their batches.
static dw_status gs_make_list(dw_gs h, int n, const GsStat &stat, cudaStream_t s) {
    const int ntiles = h->tiles_x * h->tiles_y;
    const dw_status st = gs_list_reserve(h, n, stat);
    if (st != DW_OK) return st;
    if (stat.most > GS_SORT_MAX) {
        gs_list_radix(h, n, (int64_t)stat.total, s);
        k_gs_batches<<<(unsigned)ntiles, 64, 0, s>>>(h->tile_count, h->ts, h->batch_off, h->ranges,
                                                     h->batch_tile.p);
        return DW_OK;
    }
    h->list = h->lgid.p;
    k_gs_list<true><<<grid_for(n, 128), 128, 0, s>>>(h->rect, h->key, n, h->tiles_x, h->ts,
                                                     h->tile_count, h->ranges, h->lkey.p);
    if (stat.big > 0)
        k_gs_big<true><<<GS_BIG_CTAS, 256, 0, s>>>(h->big, h->big + h->cap, h->rect, h->key, h->tiles_x,
                                                   h->ts, h->tile_count, h->ranges, h->lkey.p, h->stat);
    size_t len = 2;
    while (len < stat.most) len <<= 1;
    auto sort = h->ts == GS_FINE ? k_gs_tile_sort<GS_FINE> : k_gs_tile_sort<GS_COARSE>;
    sort<<<(unsigned)ntiles, GS_SORT_THREADS, len * sizeof(unsigned long long), s>>>(
        h->ranges, h->lkey.p, h->batch_off, h->lgid.p, h->batch_tile.p);
    return DW_OK;
}

extern "C" dw_status gs_render(dw_gs h, const dw_camera *cam, const float *x, const float *F,
                               const float *sigma0, const float *color, const float *opacity,
                               int64_t n, float *image, dw_stream stream) {
    dw_status st = gs_check(h, cam, x, F, sigma0, color, opacity, n);
    if (st != DW_OK) return st;
    DW_REQUIRE(image, "image must not be NULL");
    cudaStream_t s = as_stream(stream);
    const GsCam c = to_cam(*cam);
    const int nn = (int)n;
    h->last_n = -1;  // no picture to differentiate until this call has drawn one
    gs_set_tiles(h, GS_FINE);
    if (nn > 0) {
        GsStat stat{};
        st = gs_count(h, c, x, F, sigma0, color, opacity, nn, stat, s);
        bool fits = stat.total <= (unsigned long long)GS_LIST_MAX;
        if (st == DW_OK && fits && stat.total > 0) st = gs_make_list(h, nn, stat, s);
        if (st == DW_ERR_OOM || (st == DW_OK && !fits)) {
            if (st != DW_OK) gs_list_free(h);
            gs_set_tiles(h, GS_COARSE);
            st = gs_recount(h, nn, stat, s);
            if (st != DW_OK) return st;
            fits = stat.total <= (unsigned long long)GS_LIST_MAX;
            DW_REQUIRE(fits, "tile list too long (Gaussians x tiles met >= 2^31)");
            if (stat.total > 0) st = gs_make_list(h, nn, stat, s);
        }
        if (st != DW_OK) return st;
        h->batches = stat.batches;
    } else {
        const size_t ntiles = (size_t)h->tiles_x * h->tiles_y;
        DW_CUDA(cudaMemsetAsync(h->ranges, 0, sizeof(int2) * ntiles, s));
        DW_CUDA(cudaMemsetAsync(h->batch_off, 0, sizeof(uint32_t) * ntiles, s));
        h->batches = 0;
    }
    auto kern = h->kept ? (h->ts == GS_FINE ? k_gs_render_fwd<GS_FINE, true> : k_gs_render_fwd<GS_COARSE, true>)
                        : (h->ts == GS_FINE ? k_gs_render_fwd<GS_FINE, false> : k_gs_render_fwd<GS_COARSE, false>);
    kern<<<(unsigned)(h->tiles_x * h->tiles_y), gs_threads(h->ts), 0, s>>>(
        c, (unsigned)h->tiles_x, h->list, h->ranges, h->rows, image, h->image, h->batch_off,
        h->before.p);
    h->last_n = nn;
    const void *in[5] = {x, F, sigma0, color, opacity};
    memcpy(h->last_in, in, sizeof in);
    h->last_cam = *cam;
    DW_LAUNCHED("gs_render");
    return DW_OK;
}

extern "C" dw_status gs_render_backward(dw_gs h, const dw_camera *cam, const float *x,
                                        const float *F, const float *sigma0, const float *color,
                                        const float *opacity, int64_t n, const float *g_image,
                                        float *g_x, float *g_F, float *g_color, float *g_opacity,
                                        dw_stream stream) {
    dw_status st = gs_check(h, cam, x, F, sigma0, color, opacity, n);
    if (st != DW_OK) return st;
    DW_REQUIRE(g_image && g_x && g_F, "g_image, g_x and g_F must not be NULL");
    const void *in[5] = {x, F, sigma0, color, opacity};
    DW_REQUIRE(h->last_n == (int)n && memcmp(h->last_in, in, sizeof in) == 0 &&
                   memcmp(&h->last_cam, cam, sizeof *cam) == 0,
               "gs_render_backward must follow gs_render of the same Gaussians and camera");
    if (n == 0) return DW_OK;
    cudaStream_t s = as_stream(stream);
    const GsCam c = to_cam(*cam);
    const int nn = (int)n;
    DW_CUDA(cudaMemsetAsync(h->g2d, 0, sizeof(float) * GS_ROW * (size_t)nn, s));
    auto kern = h->kept ? (h->ts == GS_FINE ? k_gs_render_bwd<GS_FINE, false> : k_gs_render_bwd<GS_COARSE, false>)
                        : (h->ts == GS_FINE ? k_gs_render_bwd<GS_FINE, true> : k_gs_render_bwd<GS_COARSE, true>);
    if (h->batches > 0)
        kern<<<h->kept ? h->batches : (unsigned)(h->tiles_x * h->tiles_y), gs_threads(h->ts), 0, s>>>(
            c, (unsigned)h->tiles_x, h->list, h->ranges, h->rows, h->batch_tile.p, h->batch_off, h->before.p,
            h->image, g_image, h->g2d);
    k_gs_preprocess_bwd<<<grid_for(nn, 256), 256, 0, s>>>(c, x, F, sigma0, opacity, nn, h->g2d, g_x, g_F,
                                                           g_color, g_opacity);
    DW_LAUNCHED("gs_render_backward");
    return DW_OK;
}

extern "C" dw_status image_l1_loss(const float *image, const float *target, int64_t n,
                                   float weight, float *loss, float *g_image, dw_stream stream) {
    DW_REQUIRE(n >= 0, "n must be >= 0");
    if (n == 0) return DW_OK;
    DW_REQUIRE(image && target && loss, "image, target and loss must not be NULL");
    k_image_l1<<<grid_for(n, 1024), 256, 0, as_stream(stream)>>>(image, target, n, weight, loss,
                                                                 g_image);
    DW_LAUNCHED("k_image_l1");
    return DW_OK;
}

extern "C" dw_status image_dssim_loss(const float *image, const float *target, int32_t channels,
                                      int32_t height, int32_t width, float weight, float *loss,
                                      float *g_image, float *workspace, dw_stream stream) {
    DW_REQUIRE(channels >= 1 && height >= 1 && width >= 1, "image sizes must be >= 1");
    const int64_t n = (int64_t)channels * height * width;
    DW_REQUIRE(10 * n < (1ll << 31), "image too large (10 C H W must be < 2^31)");
    DW_REQUIRE(image && target && loss && workspace, "image, target, loss and workspace must not be NULL");
    cudaStream_t s = as_stream(stream);
    const SsimWin k = ssim_window();
    const unsigned grid = (unsigned)((width + SS_X - 1) / SS_X) * (unsigned)((height + SS_Y - 1) / SS_Y) *
                          (unsigned)channels;
    const dim3 block(SS_X, 8);
    float *part = g_image ? workspace : nullptr;
    k_ssim<<<grid, block, 0, s>>>(image, target, height, width, n, k, weight, loss, part);
    if (g_image)
        k_ssim_grad<<<grid, block, 0, s>>>(image, target, part, height, width, n, k, g_image);
    DW_LAUNCHED("image_dssim_loss");
    return DW_OK;
}
