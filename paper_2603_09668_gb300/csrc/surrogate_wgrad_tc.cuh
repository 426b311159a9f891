// Weight and bias gradients of the surrogate network's 3x3x3 convolutions on
// the fifth-generation tensor cores (tcgen05.mma kind::f16, BF16 operands,
// FP32 accumulators in tensor memory, operands loaded by TMA).
//
// dW[tap][co][ci] = sum_v g[v][co] in[v + d(tap)][ci] (zero padding) is a
// GEMM over voxels (K). A tile is 16 (x) x WG_TY (y) voxels of one slice z of
// the input; for each of its rows y and each dy one MMA computes
//   D_dy[(dx, ci)][(co, dz)] += sum_{16 x-voxels}
//            in[(x + dx - 1, y + dy - 1, z)][ci] g[(x, y, z - dz + 1)][co]
// with M = 128 rows = 4 dx slots x 32 input channels (the fourth slot, and
// for CIN = 16 the upper half of every slot, are rows whose results are not
// read), N = 3 COUT, K = 16 voxels. Both operands are MN-major: in the planar
// activation layout [C/8][n^3][8] a voxel's 8 channels are one 16-byte row,
// and 8 consecutive voxels of one 8-channel plane form a core matrix (8 K
// rows x 16 B). The input rows are loaded three times per tile, shifted by
// dx = 0, 1, 2 voxels (three TMA boxes, 16-byte aligned in x because a voxel
// record is 16 bytes), into consecutive slots, so that every 8-row group of
// M, (dx, 8 channels), is one plane further: a uniform stride-dimension
// offset, which is what lets the three dx taps share one MMA. The three g
// slices come as one box whose (plane, slice) order gives the 8-column groups
// of N the same property, so the three dz taps share it too. Slices outside
// the volume are zeros. The three dy accumulators (9 COUT columns of tensor
// memory) stay in tensor memory over all of a CTA's tiles; the epilogue
// writes the CTA's partial sums once.
//
// With one MMA of N = COUT per (dy, dz), on 16 x 4 tiles of g and the three
// input slices around them, 64 voxels took 36 MMAs and 58 KB of loads (now 12
// and 27 KB), and the bias gradient read g once more: a 32 -> 32 layer with
// its reductions took 66 us at 64^3 and 183 us at 96^3, now 20 and 46 us
// (without the MMAs 16 us at 64^3: launches, the loads' start and the
// partial sums' reduction are most of the rest). With WG_TY = 4 (six stages)
// 96^3 takes 54 us instead of 50: the halo rows are half of a plane's six.
//
// Roles: warp 5, lane 0 issues the TMA loads (a ring of WG_NST stages); warp
// 4, lane 0 the MMAs; warps 0-3 add up the g slice of each tile for the bias
// gradient, from the stage the MMAs read it from, and at the end read the
// accumulators (warp w: rows 32 w .. 32 w + 31). Every wait is bounded (about
// a second): the kernel then sets ERRBIT_TIMEOUT, drains its copies and frees
// the tensor memory.
#pragma once

#include "surrogate_tc.cuh"

namespace dw {

constexpr int WG_TX = 16, WG_TY = 8;   // tile: 16 x-voxels (one K step) x WG_TY rows, one z slice
constexpr int WG_HY = WG_TY + 2;       // halo rows
constexpr int WG_ROW = WG_TX * 16;     // bytes of one row of 16 voxel records
constexpr int WG_PLANE = WG_HY * WG_ROW;   // one 8-channel plane of a slot
constexpr int WG_GSLICE = WG_TY * WG_ROW;  // one 8-channel plane of a g slice
constexpr int WG_NST = 4;              // pipeline stages
constexpr int WG_EPI = 4;              // bias and epilogue warps: tensor-memory rows 0-127
constexpr int WG_MMA_WARP = WG_EPI, WG_LOAD_WARP = WG_EPI + 1;
constexpr int WG_THREADS = 32 * (WG_EPI + 2);

template <int CIN>
constexpr int wg_slot() { return (CIN / 8) * WG_PLANE; }
template <int CIN, int COUT>
constexpr int wg_stage() { return 3 * wg_slot<CIN>() + (COUT / 8) * 3 * WG_GSLICE; }
// The stages, plus what the M = 128 rows of the last stage's MMAs reach past
// it (an MMA's A operand ends within 16 planes of the stage start), plus
// alignment.
template <int CIN, int COUT>
constexpr size_t wg_smem() {
    constexpr int extra = 16 * WG_PLANE > wg_stage<CIN, COUT>() ? 16 * WG_PLANE - wg_stage<CIN, COUT>() : 0;
    return (size_t)WG_NST * wg_stage<CIN, COUT>() + extra + 1024;
}
template <int COUT>
constexpr int wg_tmem_cols() { return 9 * COUT <= 256 ? 256 : 512; }

// kind::f16 instruction descriptor: FP32 accumulator, BF16 A and B, both
// MN-major (bits 15 and 16), M = 128, N = n.
__host__ __device__ constexpr uint32_t wg_idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(128 >> 4) << 24);
}

struct WgPipe {
    uint64_t full[WG_NST], empty[WG_NST], done;
    uint32_t tmem_base;
    int abort_flag;
    float bias[WG_EPI][32];
};

// Tiles of this CTA: a contiguous range of the layer's (x, y, z) tiles (at
// least one: the grid has no more CTAs than there are tiles).
__device__ __forceinline__ void wg_range(int ntiles, int &t0, int &t1) {
    t0 = (int)((int64_t)ntiles * blockIdx.x / gridDim.x);
    t1 = (int)((int64_t)ntiles * (blockIdx.x + 1) / gridDim.x);
}

template <int CIN, int COUT>
__device__ __forceinline__ void wg_load(const CUtensorMap *tm_in, const CUtensorMap *tm_g,
                                        uint32_t stage, uint32_t bar, int n, int tile) {
    const int tx = n / WG_TX, ty = n / WG_TY;
    const int x0 = (tile % tx) * WG_TX, y0 = ((tile / tx) % ty) * WG_TY, z = tile / (tx * ty);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                 :: "r"(bar), "r"(wg_stage<CIN, COUT>()) : "memory");
#pragma unroll
    for (int d = 0; d < 3; ++d)
        asm volatile(
            "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
            " [%0], [%1, {%2, %3, %4, %5}], [%6];"
            :: "r"(stage + d * wg_slot<CIN>()), "l"((uint64_t)tm_in), "r"(8 * (x0 - 1 + d)),
               "r"(y0 - 1), "r"(z), "r"(0), "r"(bar)
            : "memory");
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];"
        :: "r"(stage + 3 * wg_slot<CIN>()), "l"((uint64_t)tm_g), "r"(8 * x0), "r"(y0), "r"(z - 1),
           "r"(0), "r"(bar)
        : "memory");
}

// Partial gradients of CTA b over its tiles: part[b][tap][co][ci] and
// part_b[b][co]. tm_in: the input activations as boxes {128, WG_HY, 1,
// CIN/8}; tm_g: the output gradients as boxes {128, WG_TY, 3, COUT/8} (both
// views [C/8][z][y][x * 8]).
template <int CIN, int COUT>
__global__ void __launch_bounds__(WG_THREADS, 1) k_wgrad_tc(const __grid_constant__ CUtensorMap tm_in,
                                                            const __grid_constant__ CUtensorMap tm_g,
                                                            int n, float *__restrict__ part,
                                                            float *__restrict__ part_b, int *err) {
    static_assert((CIN == 16 || CIN == 32) && (COUT == 16 || COUT == 32), "unsupported shape");
    constexpr int STAGE = wg_stage<CIN, COUT>(), GOFF = 3 * wg_slot<CIN>();
    constexpr int TCOLS = wg_tmem_cols<COUT>(), NW = 3 * COUT;
    constexpr uint32_t IDESC = wg_idesc(NW);
    extern __shared__ unsigned char smem_raw[];
    __shared__ WgPipe pp;
    unsigned char *smem = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        pp.abort_flag = 0;
        for (int i = 0; i < WG_NST; ++i) {
            mbar_init(smem_u32(&pp.full[i]), 1);
            mbar_init(smem_u32(&pp.empty[i]), 1 + WG_EPI);  // the MMAs, the bias warps
        }
        mbar_init(smem_u32(&pp.done), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&pp.tmem_base)), "r"(TCOLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_trigger();
    const uint32_t taddr = pp.tmem_base;
    volatile int *abort_p = &pp.abort_flag;
    const int ntiles = (n / WG_TX) * (n / WG_TY) * n;
    int t0, t1;
    wg_range(ntiles, t0, t1);
    const int cnt = t1 - t0;

    if (warp == WG_LOAD_WARP) {
        if (lane == 0) {
            pdl_wait();  // everything else in the kernel follows from the first load
            int j = 0;
            for (; j < cnt; ++j) {
                const int s = j % WG_NST;
                if (j >= WG_NST && !tc_wait(smem_u32(&pp.empty[s]), (j / WG_NST - 1) & 1, abort_p)) {
                    *abort_p = 1;
                    break;
                }
                wg_load<CIN, COUT>(&tm_in, &tm_g, sbase + s * STAGE, smem_u32(&pp.full[s]), n, t0 + j);
            }
            // drain (bounded): the last copies into every stage
            for (int i = max(0, j - WG_NST); i < j; ++i)
                tc_wait(smem_u32(&pp.full[i % WG_NST]), (i / WG_NST) & 1, nullptr);
        }
        __syncwarp();
    } else if (warp == WG_MMA_WARP) {
        if (lane == 0) {
            for (int j = 0; j < cnt; ++j) {
                const int s = j % WG_NST;
                if (!tc_wait(smem_u32(&pp.full[s]), (j / WG_NST) & 1, abort_p)) {
                    *abort_p = 1;
                    break;
                }
                tc_fence_after();
                const uint64_t a0 = tc_desc(sbase + s * STAGE, 128, WG_PLANE);
                const uint64_t b0 = tc_desc(sbase + s * STAGE + GOFF, 128, WG_GSLICE);
#pragma unroll
                for (int r = 0; r < WG_TY; ++r) {
#pragma unroll
                    for (int dy = 0; dy < 3; ++dy) {
                        const uint64_t ad = a0 + (uint32_t)((r + dy) * WG_ROW >> 4);
                        const uint64_t bd = b0 + (uint32_t)(r * WG_ROW >> 4);
                        const uint32_t d = taddr + (uint32_t)(dy * NW);
                        const uint32_t acc = (j | r) != 0;  // the CTA's first row starts each sum
                        asm volatile(
                            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
                            :: "r"(d), "l"(ad), "l"(bd), "r"(IDESC), "r"(acc)
                            : "memory");
                    }
                }
                tc_commit(smem_u32(&pp.empty[s]));
            }
            // all MMAs issued have ended when done completes (bounded)
            tc_commit(smem_u32(&pp.done));
            tc_wait(smem_u32(&pp.done), 0, nullptr);
        }
        __syncwarp();
    } else {
        // bias: the 16-byte records of the tile's own g slice, spread over the
        // threads by (row, x) within a plane, so that a thread's planes are fixed
        constexpr int PL = COUT / 8, REC = WG_TY * WG_TX, PPP = 32 * WG_EPI / REC;  // planes per pass
        static_assert(32 * WG_EPI % REC == 0 && PL % PPP == 0, "bias records do not split evenly");
        float acc[PL / PPP][8] = {};
        bool ok = true;
        for (int j = 0; j < cnt && ok; ++j) {
            const int s = j % WG_NST;
            ok = tc_wait(smem_u32(&pp.full[s]), (j / WG_NST) & 1, abort_p);
            if (ok) {
                const unsigned char *g = smem + s * STAGE + GOFF + WG_GSLICE + (tid % REC) * 16;
#pragma unroll
                for (int p = 0; p < PL / PPP; ++p) {
                    const uint4 q = *reinterpret_cast<const uint4 *>(g + (p * PPP + tid / REC) * 3 * WG_GSLICE);
                    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        acc[p][2 * c] += __uint_as_float(w[c] << 16);
                        acc[p][2 * c + 1] += __uint_as_float(w[c] & 0xffff0000u);
                    }
                }
            }
            ok = __all_sync(0xffffffffu, ok);
            if (lane == 0) mbar_arrive(smem_u32(&pp.empty[s]));
        }
        // the warp's sums of its planes (p PPP + its first thread's plane)
#pragma unroll
        for (int p = 0; p < PL / PPP; ++p)
#pragma unroll
            for (int c = 0; c < 8; ++c) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc[p][c] += __shfl_xor_sync(0xffffffffu, acc[p][c], o);
                if (lane == 0) pp.bias[warp][p * 8 + c] = acc[p][c];
            }
        asm volatile("bar.sync 1, %0;" :: "n"(32 * WG_EPI) : "memory");
        if (tid < COUT) {
            constexpr int WPP = WG_EPI / PPP;  // warps per plane
            const int pl = tid / 8, w0 = (pl % PPP) * WPP;
            float sum = 0.0f;
            for (int w = 0; w < WPP; ++w) sum += pp.bias[w0 + w][pl / PPP * 8 + (tid & 7)];
            part_b[(size_t)blockIdx.x * COUT + tid] = sum;
        }
        // rows 32 warp .. + 31: m = dx CIN + ci (rows from 3 CIN on are padding)
        const int m = 32 * warp + lane;
        ok = tc_wait(smem_u32(&pp.done), 0, abort_p) && !*abort_p;
        ok = __all_sync(0xffffffffu, ok);
        if (ok) {
            tc_fence_after();
            const uint32_t tq = taddr + ((uint32_t)(32 * warp) << 16);
            const int dx = m / CIN, ci = m % CIN;
            float *pc = part + (size_t)blockIdx.x * 27 * COUT * CIN + (size_t)dx * COUT * CIN + ci;
#pragma unroll 1
            for (int dy = 0; dy < 3; ++dy) {
#pragma unroll
                for (int c0 = 0; c0 < NW; c0 += 16) {
                    float r[16];
                    tc_ld<16>(tq + (uint32_t)(dy * NW + c0), r);
                    if (m < 3 * CIN) {
#pragma unroll
                        for (int cc = 0; cc < 16; ++cc) {
                            // 8-column group (plane, g slice z + 1 - dz)
                            const int grp = (c0 + cc) / 8, dz = 2 - grp % 3, co = grp / 3 * 8 + cc % 8;
                            pc[((size_t)(9 * dz + 3 * dy) * COUT + co) * CIN] = r[cc];
                        }
                    }
                }
            }
        } else if (lane == 0) {
            atomicOr(err, ERRBIT_TIMEOUT);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(taddr), "r"(TCOLS));
    }
}

}  // namespace dw
