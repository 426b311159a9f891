// Kernels on the layer split of mpm_layer.cuh: P2G, G2P, the fused G2P/P2G of
// a rollout, and the reverse substep of a checkpointed segment (fused across
// substeps), with their launchers.
#include "mpm_handle.cuh"
#include "mpm_layer.cuh"

namespace dw {

// Resident CTAs per SM the launch bounds ask for. Forward: 80 registers; ten
// CTAs (64 registers) gain 4% at 40,000 particles and lose 4% at 5,504.
// Reverse: 80 registers with 36 bytes spilled; a reverse substep of a segment
// with its recompute (us, 100,284 / 400,040 particles of a sheet): five CTAs
// 54.1 / 157.8, six 49.0 / 137.9, eight 45.9 / 127.3, nine 48.2 / 131.3. The
// kernels they replace took 59.4 / 146.4 (39.9 against 19.8 at 5,504).
constexpr int LAYER_FWD_CTAS = 8, LAYER_REV_CTAS = 8;

// ---------------------------------------------------------------- forward --

__global__ void __launch_bounds__(LAYER_THREADS) k_layer_p2g(
    MpmParams P, const float *__restrict__ x, const float *__restrict__ v,
    const float *__restrict__ C, const float *__restrict__ F, int64_t n, float4 *__restrict__ grid,
    int *err, ActiveBlocks ab) {
    __shared__ LayerSmem sm;
    pdl_wait();
    pdl_trigger();
    const int w = threadIdx.x >> 5;
    const int64_t p = (int64_t)blockIdx.x * LAYER_P + (threadIdx.x & 31);
    const bool live = p < n;
    float xp[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) xp[a] = live ? x[a * n + p] : 0.0f;
    Stencil s;
    const bool in = make_stencil(P, xp[0], xp[1], xp[2], s) && live;
    float A[9], mv[3];
    int key = -1;
    if (w == 0) {
#pragma unroll
        for (int k = 0; k < 9; ++k) A[k] = 0.0f;
        mv[0] = mv[1] = mv[2] = 0.0f;
        if (in) {
            float Cp[9], Fp[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                Cp[k] = C[k * n + p];
                Fp[k] = F[k * n + p];
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) mv[a] = P.p_mass * v[a * n + p];
            if (!p2g_affine(P, Fp, Cp, A)) atomicOr(err, ERRBIT_INVERTED);
            key = stencil_node(P, s);
        } else if (live) {
            atomicOr(err, ERRBIT_DOMAIN);
        }
    }
    layer_share(sm, A, mv, key);
    layer_p2g(P, sm, s, A, mv, key, P.p_mass, grid, ab);
}

// The fused G2P of substep k and P2G of substep k + 1 (SCATTER), or the G2P
// alone, from x and F to xo and Fo (which may be the same arrays); v and C are
// written when vo and Co are given. In a rollout x and F were last written two
// launches back by a kernel that has completed once this one runs, so they are
// read before the dependency wait, through L2 (ld.global.cg); EARLY = false
// reads them after it. KEYS: as in pair_warp.
template <bool SCATTER, bool EARLY, bool KEYS>
__global__ void __launch_bounds__(LAYER_THREADS, LAYER_FWD_CTAS) k_layer_g2p(
    MpmParams P, const float *x, const float *F, const uint8_t *__restrict__ pinned,
    const float4 *__restrict__ grid_v, float *xo, float *vo, float *Co, float *Fo,
    float4 *__restrict__ grid_next, int64_t n, int *err, ActiveBlocks ab_next, int *reset_count,
    int *keys_out, int *counts_out) {
    __shared__ LayerSmem sm;
    const int w = threadIdx.x >> 5;
    const int64_t p = (int64_t)blockIdx.x * LAYER_P + (threadIdx.x & 31);
    const bool live = p < n;
    if (!EARLY) {
        pdl_wait();
        pdl_trigger();
    }
    float xp[3], Fp[9];
    bool pin = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) xp[a] = live ? __ldcg(x + a * n + p) : 0.0f;
    if (w == 0) {
#pragma unroll
        for (int k = 0; k < 9; ++k) Fp[k] = live ? __ldcg(F + k * n + p) : 0.0f;
        pin = live && pinned && pinned[p];
    }
    Stencil s;
    const bool in = make_stencil(P, xp[0], xp[1], xp[2], s) && live;
    if (EARLY) {
        pdl_wait();
        pdl_trigger();
    }
    if (reset_count && blockIdx.x == 0 && threadIdx.x == 0) *reset_count = 0;
    float sums[9], o1[9], o2[9];
    layer_gather(P, s, w, grid_v, sums, sums + 3, sums + 6);
    layer_collect(sm, sums, o1, o2);
    float A[9], mv[3];
    int key = -1;
    if (w == 0) {
        float vn[3], Cn[9];
        layer_velocity(P, s, sums, o1, o2, vn, Cn);
        if (pin || !in) {  // a stencil off the grid: unchanged, v = C = 0
#pragma unroll
            for (int a = 0; a < 3; ++a) vn[a] = 0.0f;
#pragma unroll
            for (int k = 0; k < 9; ++k) Cn[k] = 0.0f;
        }
        float M[9], Fn[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) M[k] = __fadd_rn(__fmul_rn(P.dt, Cn[k]), k % 4 == 0 ? 1.0f : 0.0f);
        layer_mul3(M, Fp, Fn);
#pragma unroll
        for (int a = 0; a < 3; ++a) xp[a] += P.dt * vn[a];
        if (live) {
#pragma unroll
            for (int a = 0; a < 3; ++a) xo[a * n + p] = xp[a];
#pragma unroll
            for (int k = 0; k < 9; ++k) Fo[k * n + p] = Fn[k];
            if (vo) {
#pragma unroll
                for (int a = 0; a < 3; ++a) vo[a * n + p] = vn[a];
            }
            if (Co) {
#pragma unroll
                for (int k = 0; k < 9; ++k) Co[k * n + p] = Cn[k];
            }
            const bool fin = isfinite(xp[0]) && isfinite(xp[1]) && isfinite(xp[2]) && finite9(Fn);
            if (!fin) atomicOr(err, ERRBIT_NONFINITE);
        }
        if (KEYS) {
            const unsigned act = __ballot_sync(FULL, live);
            if (live) {
                const int ck = cell_key(P, ab_next.nb, xp[0], xp[1], xp[2]);
                keys_out[p] = ck;
                const unsigned peers = __match_any_sync(act, ck);
                if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&counts_out[ck], __popc(peers));
            }
            __syncwarp();
        }
        if (SCATTER) {
#pragma unroll
            for (int k = 0; k < 9; ++k) A[k] = 0.0f;
#pragma unroll
            for (int a = 0; a < 3; ++a) mv[a] = P.p_mass * vn[a];
            if (make_stencil(P, xp[0], xp[1], xp[2], s) && live) {
                if (!p2g_affine(P, Fn, Cn, A)) atomicOr(err, ERRBIT_INVERTED);
                key = stencil_node(P, s);
            } else if (live) {
                atomicOr(err, ERRBIT_DOMAIN);
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) sm.part[0][a][threadIdx.x] = xp[a];
        }
    }
    if (!SCATTER) return;
    layer_share(sm, A, mv, key);
    if (w != 0)
        make_stencil(P, sm.part[0][0][threadIdx.x & 31], sm.part[0][1][threadIdx.x & 31],
                     sm.part[0][2][threadIdx.x & 31], s);
    layer_p2g(P, sm, s, A, mv, key, P.p_mass, grid_next, ab_next);
}

dw_status launch_layer_p2g(const MpmParams &P, const float *x, const float *v, const float *C,
                           const float *F, int64_t n, float4 *grid, int *err,
                           const ActiveBlocks &ab, cudaStream_t st) {
    DW_CUDA(launch_pdl(k_layer_p2g, grid_for(n, LAYER_P), LAYER_THREADS, st, P, x, v, C, F, n, grid,
                       err, ab));
    return DW_OK;
}

dw_status launch_layer_g2p(const MpmParams &P, const float *x, const float *F,
                           const uint8_t *pinned, const float4 *grid_v, const dw_mpm_state &out,
                           int64_t n, int *err, int *reset_count, cudaStream_t st) {
    const ActiveBlocks none{nullptr, nullptr, nullptr, 0, 0};
    DW_CUDA(launch_pdl(k_layer_g2p<false, false, false>, grid_for(n, LAYER_P), LAYER_THREADS, st, P,
                       x, F, pinned, grid_v, out.x, out.v, out.C, out.F, (float4 *)nullptr, n, err,
                       none, reset_count, (int *)nullptr, (int *)nullptr));
    return DW_OK;
}

dw_status launch_layer_g2p2g(const MpmParams &P, const float *x, const float *F,
                             const uint8_t *pinned, const float4 *grid_v, const dw_mpm_state &out,
                             float4 *grid_next, int64_t n, int *err, const ActiveBlocks &ab_next,
                             int *reset_count, int *keys, int *counts, cudaStream_t st) {
    auto kern = keys ? k_layer_g2p<true, true, true> : k_layer_g2p<true, true, false>;
    DW_CUDA(launch_pdl(kern, grid_for(n, LAYER_P), LAYER_THREADS, st, P, x, F, pinned, grid_v, out.x,
                       out.v, out.C, out.F, grid_next, n, err, ab_next, reset_count, keys, counts));
    return DW_OK;
}

// ---------------------------------------------------------------- reverse --
//
// A segment's reverse pass alternates two kernels per substep j:
//   k_rev_nodes: the reverse grid update of substep j (its (m, p) read from
//     the grid tape) and, by the other half of the CTAs, the grid velocities
//     of substep j - 1, also from the tape;
//   k_layer_rev: the reverse P2G of substep j (dL/d(state j)), and from it,
//     without leaving the registers, the reverse G2P of substep j - 1.
// The first k_layer_rev of a segment has no reverse P2G, the last no reverse
// G2P. Per substep that is two launches instead of four (grid restore, reverse
// G2P, reverse grid, reverse P2G), the 24 gradient floats per particle stay in
// registers, and nothing restores the (m, p) grid; a chain of small kernels is
// bound by their latencies, a large one by its issue slots and occupancy.

// State j (the reverse P2G's input), state j - 1 (the reverse G2P's), both as
// rows of length n.
struct LayerRev {
    const float *xj, *vj, *Cj, *Fj;  // not read with FIRST
    const float *xi, *Fi;            // not read with LAST
    const uint8_t *pinned;
    const float4 *grid_bmp;  // substep j's (dL/dm_i, dL/dp_i)
    const float4 *grid_v;    // substep j - 1's velocities
    float4 *grid_bv;         // receives (0, dL/dv_i) of substep j - 1
    float *scratch;          // [12][cap]: partial dL/dx (3) and dL/dF (9) of the reverse G2P
    float *gx, *gv, *gC, *gF;  // dL/d(state after the segment) in (FIRST), dL/d(start) out (LAST)
    double *gE_part;         // [CTAs] dL/dE of the CTA's particles so far, or NULL
    int *reset_count;        // active-list count to clear (FIRST), or NULL
    int64_t n, cap;
};

template <bool FIRST, bool LAST>
__global__ void __launch_bounds__(LAYER_THREADS, LAYER_REV_CTAS) k_layer_rev(MpmParams P, LayerRev R) {
    __shared__ LayerSmem sm;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t n = R.n, p = (int64_t)blockIdx.x * LAYER_P + lane;
    const bool live = p < n;
    // dL/d(state j), complete in warp 0
    float gx[3], gv[3], gC[9], gF[9];
    float gE = 0.0f;
    if (FIRST) {
        pdl_wait();
        pdl_trigger();
        if (R.reset_count && blockIdx.x == 0 && threadIdx.x == 0) *R.reset_count = 0;
        if (w == 0) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                gx[a] = live ? R.gx[a * n + p] : 0.0f;
                gv[a] = live ? R.gv[a * n + p] : 0.0f;
            }
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                gC[k] = live ? R.gC[k * n + p] : 0.0f;
                gF[k] = live ? R.gF[k * n + p] : 0.0f;
            }
        }
    } else {
        // The state and the partial gradients come from launches before the
        // previous one, so the state's part of the work runs before the wait
        // (loads through L2). What the owner needs again after the gather is
        // kept in shared memory or loaded again: the gather holds 36 registers.
        float xj[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) xj[a] = live ? __ldcg(R.xj + a * n + p) : 0.0f;
        Stencil s;
        const bool in = make_stencil(P, xj[0], xj[1], xj[2], s) && live;
        LayerAffine L;
        {
            float A[9], mv[3];
            int key = -1;
            if (w == 0) {
                float Fj[9], Cj[9], Pk[9], PFt[9];
#pragma unroll
                for (int a = 0; a < 3; ++a) mv[a] = live ? P.p_mass * __ldcg(R.vj + a * n + p) : 0.0f;
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    Cj[k] = live ? __ldcg(R.Cj + k * n + p) : 0.0f;
                    Fj[k] = live ? __ldcg(R.Fj + k * n + p) : 0.0f;
                }
                stress_P(P, Fj, Pk);
                mul3_abt(Pk, Fj, PFt);
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    A[k] = -P.kappa * PFt[k] + P.p_mass * Cj[k];
                    sm.Pk[k][lane] = Pk[k];
                }
            }
            layer_share(sm, A, mv, key);
            L = layer_affine(P, s, A, mv, w);
        }
        pdl_wait();
        pdl_trigger();
        float v[12], o1[12], o2[12], ref[3];
        layer_rev_gather<false, true>(P, s, L, w, P.p_mass, R.grid_bmp, v, ref);
        float Fj[9];
        if (w == 0) {
#pragma unroll
            for (int a = 0; a < 3; ++a) gx[a] = live ? __ldcg(R.scratch + a * R.cap + p) : 0.0f;
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                Fj[k] = live ? __ldcg(R.Fj + k * n + p) : 0.0f;
                gF[k] = live ? __ldcg(R.scratch + (3 + k) * R.cap + p) : 0.0f;
            }
        }
        layer_collect(sm, v, o1, o2);
        if (w == 0) {
            float B[3], G[3], bA[9];
            layer_rev_sums(P, s, v, o1, o2, B, G);
            layer_moments(P, s, v, o1, o2, B, bA);
            if (!in) {
#pragma unroll
                for (int a = 0; a < 3; ++a) B[a] = G[a] = ref[a] = 0.0f;
#pragma unroll
                for (int k = 0; k < 9; ++k) bA[k] = 0.0f;
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (in)
                    gx[a] += G[a] - (sm.bc[a][lane] * B[0] + sm.bc[3 + a][lane] * B[1] +
                                     sm.bc[6 + a][lane] * B[2]);
                gv[a] = P.p_mass * (B[a] + ref[a]);
            }
            if (in) {
                float Pk[9], bAF[9], bAtP[9], bP[9];
#pragma unroll
                for (int k = 0; k < 9; ++k) Pk[k] = sm.Pk[k][lane];
                mul3(bA, Fj, bAF);
                mul3_atb(bA, Pk, bAtP);
                float pp = 0.0f;
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    bP[k] = -P.kappa * bAF[k];
                    gF[k] += -P.kappa * bAtP[k];
                    pp += bP[k] * Pk[k];
                }
                stress_P_adjoint(P, Fj, bP, gF);
                gE = pp / P.E;
            }
#pragma unroll
            for (int k = 0; k < 9; ++k) gC[k] = P.p_mass * bA[k];
        }
    }
    if (w == 0) {  // dL/dE: the CTA's sum over the segment (k_layer_gE adds them up)
        if (R.gE_part) {
            double sum = gE;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(FULL, sum, o);
            if (lane == 0) R.gE_part[blockIdx.x] = FIRST ? 0.0 : R.gE_part[blockIdx.x] + sum;
        }
        if (LAST && live) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                R.gx[a * n + p] = gx[a];
                R.gv[a * n + p] = gv[a];
            }
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                R.gC[k * n + p] = gC[k];
                R.gF[k * n + p] = gF[k];
            }
        }
    }
    if (LAST) return;
    float xi[3], Fi[9], CjDt[9];  // CjDt: dt C of state j, the C' of substep j - 1
    bool pin = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) xi[a] = live ? __ldcg(R.xi + a * n + p) : 0.0f;
    if (w == 0) {
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            Fi[k] = live ? __ldcg(R.Fi + k * n + p) : 0.0f;
            if (!FIRST) CjDt[k] = live ? P.dt * __ldcg(R.Cj + k * n + p) : 0.0f;
        }
        pin = live && R.pinned && R.pinned[p];
    }
    // reverse G2P of substep j - 1: F' = (I + dt C') F, x' = x + dt v
    Stencil s;
    const bool in = make_stencil(P, xi[0], xi[1], xi[2], s) && live;
    float A[9], mv[3], bF[9];
    int key = -1;
    if (w == 0) {
        float gFFt[9];
        mul3_abt(gF, Fi, gFFt);
#pragma unroll
        for (int k = 0; k < 9; ++k) A[k] = P.D * (gC[k] + P.dt * gFFt[k]);
#pragma unroll
        for (int a = 0; a < 3; ++a) mv[a] = gv[a] + P.dt * gx[a];
        if (in && !pin) key = stencil_node(P, s);
        if (!FIRST) {
            // a pinned particle's C' is zero, in the state as in G2P
#pragma unroll
            for (int k = 0; k < 9; ++k) CjDt[k] = (pin ? 0.0f : CjDt[k]) + (k % 4 == 0 ? 1.0f : 0.0f);
            mul3_atb(CjDt, gF, bF);
        }
    }
    layer_share(sm, A, mv, key);
    const LayerAffine L = layer_affine(P, s, A, mv, w);
    float v[FIRST ? 12 : 6], o1[FIRST ? 12 : 6], o2[FIRST ? 12 : 6], ref[3];
    layer_rev_gather<true, FIRST>(P, s, L, w, 0.0f, R.grid_v, v, ref);
    layer_scatter(P, s, L, w, 0.0f, key, sm.rows[w], sm.keys, R.grid_bv);
    layer_collect(sm, v, o1, o2);
    if (w == 0 && live) {
        float B[3], G[3];
        layer_rev_sums(P, s, v, o1, o2, B, G);
        if constexpr (FIRST) {  // C' = (4 / dx^2) sum W v (x_i - x_p)^T of the same gather
            float m[9];
            layer_moments(P, s, v, o1, o2, B, m);
#pragma unroll
            for (int k = 0; k < 9; ++k)
                m[k] = (key >= 0 ? P.dt * P.D * m[k] : 0.0f) + (k % 4 == 0 ? 1.0f : 0.0f);
            mul3_atb(m, gF, bF);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            float b = gx[a];
            if (key >= 0) b += G[a] - (A[a] * B[0] + A[3 + a] * B[1] + A[6 + a] * B[2]);
            R.scratch[a * R.cap + p] = in ? b : 0.0f;
        }
#pragma unroll
        for (int k = 0; k < 9; ++k) R.scratch[(3 + k) * R.cap + p] = in ? bF[k] : 0.0f;
    }
}

// *g_E += the sum of part[0..n) (one CTA of 256 threads).
__global__ void __launch_bounds__(256) k_layer_gE(const double *__restrict__ part, int n, float *g_E) {
    __shared__ double red[8];
    pdl_wait();
    pdl_trigger();
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += 256) s += part[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) s += red[w];
        atomicAdd(g_E, (float)s);  // handles on other streams may add to the same sum
    }
}

// One substep's grid in the tape: entry e of the list is block list[e], its
// 64 nodes' (m, p) at mp[64 e].
struct GridSlot {
    const float4 *mp;
    const int *list, *count;
};

// Even CTAs: the reverse grid update of the substep whose grid is `rev` (dL/dv_i
// in grid_bv, cleared here) into grid_bmp, with the wind gradient. Odd CTAs:
// the grid velocities of the substep before it, whose grid is `vel` (mp NULL:
// none).
__global__ void __launch_bounds__(GRID_THREADS) k_rev_nodes(MpmParams P, WindDev wind, float t_rev,
                                                            float t_vel, GridSlot rev, GridSlot vel,
                                                            int nb, float4 *__restrict__ grid_bv,
                                                            float4 *__restrict__ grid_bmp,
                                                            float4 *__restrict__ grid_v,
                                                            float *__restrict__ g_wind) {
    __shared__ WindGroup wg[GRID_THREADS / 64];
    pdl_wait();
    pdl_trigger();
    const int sub = threadIdx.x >> 6, lt = threadIdx.x & 63;
    const int stride = (gridDim.x >> 1) * 4;
    int e = (blockIdx.x >> 1) * 4 + sub;
    const bool back = !(blockIdx.x & 1);
    const GridSlot &S = back ? rev : vel;
    if (!S.mp) return;
    const int nblk = nb * nb * nb;
    int b = e < nblk ? S.list[e] : 0;  // read beside the count; used only below it
    float4 mp = e < nblk ? S.mp[(size_t)e * 64 + lt] : make_float4(0.f, 0.f, 0.f, 0.f);
    const int count = *S.count;
    for (; e < count; e += stride) {
        int i, j, k;
        const bool node_in = active_node(P, nb, b, lt, i, j, k);
        const int64_t node = ((int64_t)k * P.N + j) * P.N + i;
        if (back) {
            float3 gw = make_float3(0.f, 0.f, 0.f);
            bool act = false;
            if (node_in) {
                float4 out;
                act = rev_node_value(P, i, j, k, mp, grid_bv[node], out, gw);
                grid_bv[node] = make_float4(0.f, 0.f, 0.f, 0.f);
                grid_bmp[node] = out;
            }
            if (g_wind) wind_scatter_block(P, wind, act, i, j, k, t_rev, gw, g_wind, wg[sub], sub + 1);
        } else if (node_in) {
            grid_v[node] = grid_node_value(P, wind, t_vel, i, j, k, mp);
        }
        if (e + stride < count) {
            b = S.list[e + stride];
            mp = S.mp[(size_t)(e + stride) * 64 + lt];
        }
    }
}

dw_status segment_reverse(MpmHandle *h, const dw_mpm_state *start, const float *tape,
                          const dw_mpm_state *g, const uint8_t *pinned, const WindDev &wd, float t0,
                          int n_substeps, float *g_wind, float *g_E, int *reset_count,
                          cudaStream_t s) {
    const int64_t n = start->n;
    LayerRev R{};
    R.pinned = pinned;
    R.grid_bmp = h->grid_bmp;
    R.grid_v = h->grid_v;
    R.grid_bv = h->grid_bv;
    R.scratch = h->pscratch;
    R.gx = g->x;
    R.gv = g->v;
    R.gC = g->C;
    R.gF = g->F;
    R.gE_part = g_E ? h->gE_part : nullptr;
    R.n = n;
    R.cap = h->desc.max_particles;
    const unsigned ctas = grid_for(n, LAYER_P);
    auto rows = [&](int k) { return tape + (size_t)(k - 1) * 24 * (size_t)n; };  // state k >= 1
    auto slot = [&](int k) {
        return GridSlot{h->gtape + (size_t)k * h->nblk * 64, h->gtape_list + (size_t)k * h->nblk,
                        h->gtape_count + k};
    };
    for (int j = n_substeps; j >= 0; --j) {  // the reverse P2G of j, the reverse G2P of j - 1
        if (j < n_substeps) {
            ProfScope ps(h, DW_K_REV_GRID, s);
            const GridSlot none{nullptr, nullptr, nullptr};
            DW_CUDA(launch_pdl(k_rev_nodes, GRID_CTAS, GRID_THREADS, s, h->P, wd,
                               fmaf((float)j, h->P.dt, t0), fmaf((float)(j - 1), h->P.dt, t0),
                               slot(j), j > 0 ? slot(j - 1) : none, h->nb, h->grid_bv, h->grid_bmp,
                               h->grid_v, g_wind));
            R.xj = j > 0 ? rows(j) : start->x;
            R.vj = j > 0 ? rows(j) + 3 * n : start->v;
            R.Cj = j > 0 ? rows(j) + 6 * n : start->C;
            R.Fj = j > 0 ? rows(j) + 15 * n : start->F;
        }
        if (j > 0) {
            R.xi = j > 1 ? rows(j - 1) : start->x;
            R.Fi = j > 1 ? rows(j - 1) + 15 * n : start->F;
        }
        R.reset_count = j == n_substeps ? reset_count : nullptr;
        ProfScope ps(h, j < n_substeps ? DW_K_REV_P2G : DW_K_REV_G2P, s);
        auto kern = j == n_substeps ? k_layer_rev<true, false>
                                    : (j == 0 ? k_layer_rev<false, true> : k_layer_rev<false, false>);
        DW_CUDA(launch_pdl(kern, ctas, LAYER_THREADS, s, h->P, R));
    }
    if (g_E) {
        ProfScope ps(h, DW_K_REV_P2G, s);
        DW_CUDA(launch_pdl(k_layer_gE, 1, 256, s, (const double *)h->gE_part, (int)ctas, g_E));
    }
    return DW_OK;
}

}  // namespace dw
