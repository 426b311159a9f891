// The MPM particle kernels with a particle's work split over the three z
// layers of its stencil: a CTA of three warps holds 32 particles, warp k
// gathers and scatters the nine nodes of layer k, and warp 0 (the owner) does
// the per-particle algebra between them.
//
// Why: with a few thousand particles a kernel of one particle (or two) per
// thread puts a warp or less on each SM, and its time is that warp's
// dependent instruction stream (about 2,800 instructions for two particles
// per thread, most of them run once, so instruction fetch is not hidden
// either). Three warps of 32 particles run a third of the node work each, so
// the stream is a third as long and there are six times as many warps. The
// price is two exchanges through shared memory per kernel and the stencil
// computed three times, which loses once the SMs are full.
#pragma once

#include "mpm_adjoint.cuh"
#include "mpm_pair_warp.cuh"

namespace dw {

constexpr int LAYER_P = 32;        // particles per CTA
constexpr int LAYER_THREADS = 96;  // one warp per stencil layer

struct LayerSmem {
    float4 rows[3][33][P2G_ROW];  // per warp: node values of its layer (+ a zero row)
    float part[2][12][32];        // partial sums of warps 1 and 2, per particle
    float bc[12][32];             // the owner's A (9) and m v (3), for every warp
    float Pk[9][32];              // reverse: the owner's stress
    int keys[32];                 // base node of each particle's stencil, -1: adds nothing
};

__device__ __forceinline__ float sel3(const float w[3], int k) {
    return k == 0 ? w[0] : (k == 1 ? w[1] : w[2]);
}

__device__ __forceinline__ int stencil_node(const MpmParams &P, const Stencil &s) {
    return (s.base[2] * P.N + s.base[1]) * P.N + s.base[0];
}

// Layer k's part of the G2P sums (tensor-product evaluation as in
// g2p_update): B = sum W v, S0 = sum W o_x v, S1 = sum W o_y v; the z sum is
// k B.
__device__ __forceinline__ void layer_gather(const MpmParams &P, const Stencil &s, int k,
                                             const float4 *__restrict__ grid_v, float B[3],
                                             float S0[3], float S1[3]) {
    const float4 *g = grid_v + stencil_node(P, s) + k * P.N * P.N;
    float4 q[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) q[i] = g[(i / 3) * P.N + i % 3];
    const float wz = sel3(s.w[2], k);
#pragma unroll
    for (int c = 0; c < 3; ++c) B[c] = S0[c] = S1[c] = 0.0f;
#pragma unroll
    for (int oj = 0; oj < 3; ++oj) {
        const float wyz = s.w[1][oj] * wz;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float g0 = pr::comp(q[3 * oj], c), g1 = pr::comp(q[3 * oj + 1], c),
                        g2 = pr::comp(q[3 * oj + 2], c);
            const float a = s.w[0][0] * g0 + s.w[0][1] * g1 + s.w[0][2] * g2;
            const float bx = s.w[0][1] * g1 + 2.0f * s.w[0][2] * g2;
            B[c] += wyz * a;
            S0[c] += wyz * bx;
            if (oj == 1) S1[c] += wyz * a;
            if (oj == 2) S1[c] += 2.0f * wyz * a;
        }
    }
}

// C = A B, in the order of operations of the paired kernels (mul3_2).
__device__ __forceinline__ void layer_mul3(const float A[9], const float B[9], float C[9]) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            C[3 * i + j] = __fmaf_rn(A[3 * i + 2], B[6 + j],
                                     __fmaf_rn(A[3 * i + 1], B[3 + j], __fmul_rn(A[3 * i], B[j])));
}

// A particle's node value is W (m, r + ox sx + oy sy) in layer k, with
// r = m v - A fx dx + k sz and s the columns of A times dx.
struct LayerAffine {
    float r[3], sx[3], sy[3];
};

__device__ __forceinline__ LayerAffine layer_affine(const MpmParams &P, const Stencil &s,
                                                    const float A[9], const float mv[3], int k) {
    LayerAffine L;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float in = __fmaf_rn(A[3 * c + 2], s.fx[2],
                                   __fmaf_rn(A[3 * c + 1], s.fx[1], __fmul_rn(A[3 * c], s.fx[0])));
        const float r0 = __fmaf_rn(-in, P.dx, mv[c]), sz = __fmul_rn(A[3 * c + 2], P.dx);
        L.r[c] = k == 0 ? r0 : __fmaf_rn((float)k, sz, r0);
        L.sx[c] = __fmul_rn(A[3 * c], P.dx);
        L.sy[c] = __fmul_rn(A[3 * c + 1], P.dx);
    }
    return L;
}

// Adds layer k's node values of the warp's 32 particles (consecutive lanes of
// one base node form a run; `keys` holds the base nodes) to the grid: values
// into shared-memory rows, rows summed per run, one float4 atomic per node and
// run. mass = 0: no mass channel. All 32 lanes call it; a lane without a
// stencil passes key < 0 and zeros its row.
__device__ __forceinline__ void layer_scatter(const MpmParams &P, const Stencil &s,
                                              const LayerAffine &L, int k, float mass, int key,
                                              float4 (*rows)[P2G_ROW], const int *keys,
                                              float4 *__restrict__ grid) {
    const int lane = threadIdx.x & 31;
    const int prev = __shfl_up_sync(FULL, key, 1);
    const unsigned starts = __ballot_sync(FULL, lane == 0 || prev != key);
    const unsigned ends = (starts >> 1) | 0x80000000u;
    const float wz = sel3(s.w[2], k);
    if (lane < 9) rows[32][lane] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int oj = 0; oj < 3; ++oj) {
        const float wyz = s.w[1][oj] * wz;
        float b[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) b[c] = oj == 0 ? L.r[c] : __fmaf_rn((float)oj, L.sy[c], L.r[c]);
#pragma unroll
        for (int oi = 0; oi < 3; ++oi) {
            const float W = s.w[0][oi] * wyz;
            float4 val;
            val.x = W * mass;
            val.y = W * __fmaf_rn((float)oi, L.sx[0], b[0]);
            val.z = W * __fmaf_rn((float)oi, L.sx[1], b[1]);
            val.w = W * __fmaf_rn((float)oi, L.sx[2], b[2]);
            rows[lane][3 * oj + oi] = key >= 0 ? val : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    __syncwarp();
    if (ends == 0x80000000u) {
        rows_one_run(rows, key, k, P.N, grid);
    } else {
        const int r0 = 11 * (lane / 9), cnt = min(32, r0 + 11) - r0;
        const unsigned e = r0 < 32 ? ((ends >> r0) & 0x7ffu) | (1u << (cnt - 1)) : 0u;
        rows_walk<11>(rows, keys, r0, cnt, e, k, P.N, grid);
    }
}

// The blocks of the next grid's active list that warp k marks for a run's
// first particle (blocks k, k + 3 and k + 6 of the eight its stencil can
// touch): flags loaded here, tested after the scatter.
struct LayerMarks {
    int id[3], flag[3];
};

__device__ __forceinline__ LayerMarks layer_marks_load(const ActiveBlocks &ab, const Stencil &s,
                                                       int key, int k) {
    LayerMarks m;
    const int prev = __shfl_up_sync(FULL, key, 1);
    const bool start = key >= 0 && ((threadIdx.x & 31) == 0 || prev != key) && ab.flags;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int d = k + 3 * q;
        m.id[q] = start && d < 8 ? stencil_block(ab, s.base[0], s.base[1], s.base[2], d) : -1;
        m.flag[q] = m.id[q] >= 0 ? *(volatile int *)&ab.flags[m.id[q]] : 1;
    }
    return m;
}

__device__ __forceinline__ void layer_marks_store(const ActiveBlocks &ab, const LayerMarks &m) {
#pragma unroll
    for (int q = 0; q < 3; ++q)
        if (m.flag[q] == 0 && atomicExch(&ab.flags[m.id[q]], 1) == 0)
            ab.list[atomicAdd(ab.count, 1)] = ab.tag | m.id[q];
}

// P2G of the CTA's particles from the owner's A, m v and key (owner: warp 0,
// the particle at (x0, x1, x2) of every lane already known to all warps when
// s is their stencil). Called by all 96 threads with the owner's values in
// registers; the other warps' A, mv and key are ignored.
__device__ __forceinline__ void layer_p2g(const MpmParams &P, LayerSmem &sm, const Stencil &s,
                                          float A[9], float mv[3], int key, float mass,
                                          float4 *__restrict__ grid, const ActiveBlocks &ab) {
    const int w = threadIdx.x >> 5;
    const LayerMarks marks = layer_marks_load(ab, s, key, w);
    const LayerAffine L = layer_affine(P, s, A, mv, w);
    layer_scatter(P, s, L, w, mass, key, sm.rows[w], sm.keys, grid);
    layer_marks_store(ab, marks);
}

// The owner's A, m v and key to every warp (a CTA barrier inside).
__device__ __forceinline__ void layer_share(LayerSmem &sm, float A[9], float mv[3], int &key) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (w == 0) {
#pragma unroll
        for (int k = 0; k < 9; ++k) sm.bc[k][lane] = A[k];
#pragma unroll
        for (int c = 0; c < 3; ++c) sm.bc[9 + c][lane] = mv[c];
        sm.keys[lane] = key;
    }
    __syncthreads();
    if (w != 0) {
#pragma unroll
        for (int k = 0; k < 9; ++k) A[k] = sm.bc[k][lane];
#pragma unroll
        for (int c = 0; c < 3; ++c) mv[c] = sm.bc[9 + c][lane];
        key = sm.keys[lane];
    }
}

// The layers' partial sums v[0..M) of warps 1 and 2 to the owner (a CTA
// barrier inside): o1 and o2 receive them in warp 0.
template <int M>
__device__ __forceinline__ void layer_collect(LayerSmem &sm, const float (&v)[M], float (&o1)[M],
                                              float (&o2)[M]) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (w != 0) {
#pragma unroll
        for (int k = 0; k < M; ++k) sm.part[w - 1][k][lane] = v[k];
    }
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int k = 0; k < M; ++k) {
            o1[k] = sm.part[0][k][lane];
            o2[k] = sm.part[1][k][lane];
        }
    }
}

// The owner's G2P result from the three layers' sums: v_p and C_p.
__device__ __forceinline__ void layer_velocity(const MpmParams &P, const Stencil &s,
                                               const float (&v)[9], const float (&o1)[9],
                                               const float (&o2)[9], float vn[3], float Cn[9]) {
    const float Ddx = P.D * P.dx;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        vn[c] = v[c] + o1[c] + o2[c];
        const float S0 = v[3 + c] + o1[3 + c] + o2[3 + c], S1 = v[6 + c] + o1[6 + c] + o2[6 + c],
                    S2 = o1[c] + 2.0f * o2[c];
        Cn[3 * c] = Ddx * (S0 - vn[c] * s.fx[0]);
        Cn[3 * c + 1] = Ddx * (S1 - vn[c] * s.fx[1]);
        Cn[3 * c + 2] = Ddx * (S2 - vn[c] * s.fx[2]);
    }
}

// Layer k's part of a reverse gather over node quantities q = (q0, b): with
// the particle's node value W (mass, val) of LayerAffine L,
//   t_i = mass q0_i + val_i . b_i,   G_a = sum_i dW_i/dx_a t_i,
//   B = sum W b, S0 = sum W o_x b, S1 = sum W o_y b.
// out: B (3), Gx, Gy (in units of 1 / dx), M = sum over the layer of wx wy t
// (combined over the layers by the owner), then S0, S1 with MOMENTS. V3: the
// vector is in .xyz and q0 is not used (grid velocities); else q = (q0, b).
// Every b is taken relative to `ref`, the middle node's: the weights sum to
// one and reproduce x, so a constant b contributes nothing to sum W b (o - fx)
// and its parts of sum dW/dx t and of -A^T sum W b cancel; subtracting it
// cancels them before the rounding instead of after it. So does taking each
// derivative sum, whose weights sum to zero, over differences to the middle
// node. (dL/dx of an isolated particle, 24^3 grid, two substeps: 3.2e-4 off the
// float64 value without, see the reverse segment's test.)
template <bool V3, bool MOMENTS, int M>
__device__ __forceinline__ void layer_rev_gather(const MpmParams &P, const Stencil &s,
                                                 const LayerAffine &L, int k, float mass,
                                                 const float4 *__restrict__ grid, float (&out)[M],
                                                 float ref[3]) {
    const int N2 = P.N * P.N;
    const float4 *g = grid + stencil_node(P, s);
    const float4 mid = g[N2 + P.N + 1];
    g += k * N2;
    float4 q[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) q[i] = g[(i / 3) * P.N + i % 3];
    ref[0] = V3 ? mid.x : mid.y;
    ref[1] = V3 ? mid.y : mid.z;
    ref[2] = V3 ? mid.z : mid.w;
#pragma unroll
    for (int i = 0; i < 9; ++i) {  // (b, q0)
        const float4 n = q[i];
        q[i] = make_float4((V3 ? n.x : n.y) - ref[0], (V3 ? n.y : n.z) - ref[1],
                           (V3 ? n.z : n.w) - ref[2], V3 ? 0.0f : n.x);
    }
    const float wz = sel3(s.w[2], k);
    float B[3] = {0.f, 0.f, 0.f}, S0[3] = {0.f, 0.f, 0.f}, S1[3] = {0.f, 0.f, 0.f};
    float Gx = 0.0f, T[3];
#pragma unroll
    for (int oj = 0; oj < 3; ++oj) {
        float t[3];
#pragma unroll
        for (int oi = 0; oi < 3; ++oi) {
            float acc = V3 ? 0.0f : mass * q[3 * oj + oi].w;
#pragma unroll
            for (int c = 0; c < 3; ++c)
                acc += pr::comp(q[3 * oj + oi], c) * (L.r[c] + (float)oj * L.sy[c] + (float)oi * L.sx[c]);
            t[oi] = acc;
        }
        T[oj] = s.w[0][0] * t[0] + s.w[0][1] * t[1] + s.w[0][2] * t[2];
        Gx += s.w[1][oj] * (s.dw[0][0] * (t[0] - t[1]) + s.dw[0][2] * (t[2] - t[1]));
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float b0 = pr::comp(q[3 * oj], c), b1 = pr::comp(q[3 * oj + 1], c),
                        b2 = pr::comp(q[3 * oj + 2], c);
            const float a = s.w[0][0] * b0 + s.w[0][1] * b1 + s.w[0][2] * b2;
            B[c] += s.w[1][oj] * a;
            if (MOMENTS) {
                S0[c] += s.w[1][oj] * (s.w[0][1] * b1 + 2.0f * s.w[0][2] * b2);
                if (oj == 1) S1[c] += s.w[1][oj] * a;
                if (oj == 2) S1[c] += 2.0f * s.w[1][oj] * a;
            }
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) out[c] = wz * B[c];
    out[3] = wz * Gx;
    out[4] = wz * (s.dw[1][0] * (T[0] - T[1]) + s.dw[1][2] * (T[2] - T[1]));
    out[5] = s.w[1][0] * T[0] + s.w[1][1] * T[1] + s.w[1][2] * T[2];
    if (MOMENTS) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            out[6 + c] = wz * S0[c];
            out[9 + c] = wz * S1[c];
        }
    }
}

// The owner's sums over the layers of layer_rev_gather: B (without ref), and
// G = sum dW/dx t.
template <int M>
__device__ __forceinline__ void layer_rev_sums(const MpmParams &P, const Stencil &s,
                                               const float (&v)[M], const float (&o1)[M],
                                               const float (&o2)[M], float B[3], float G[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) B[c] = v[c] + o1[c] + o2[c];
    G[0] = P.inv_dx * (v[3] + o1[3] + o2[3]);
    G[1] = P.inv_dx * (v[4] + o1[4] + o2[4]);
    G[2] = P.inv_dx * (s.dw[2][0] * (v[5] - o1[5]) + s.dw[2][2] * (o2[5] - o1[5]));
}

// dx sum W b_c (o - fx)_b from the layers' moments (rows c, columns b).
__device__ __forceinline__ void layer_moments(const MpmParams &P, const Stencil &s,
                                              const float (&v)[12], const float (&o1)[12],
                                              const float (&o2)[12], const float B[3], float m[9]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float S0 = v[6 + c] + o1[6 + c] + o2[6 + c], S1 = v[9 + c] + o1[9 + c] + o2[9 + c],
                    S2 = o1[c] + 2.0f * o2[c];
        m[3 * c] = P.dx * (S0 - B[c] * s.fx[0]);
        m[3 * c + 1] = P.dx * (S1 - B[c] * s.fx[1]);
        m[3 * c + 2] = P.dx * (S2 - B[c] * s.fx[2]);
    }
}

}  // namespace dw
