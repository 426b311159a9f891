// Reverse mode of one MLS-MPM substep (Eq. simulation_mpm), per particle and
// per node, shared by the single-scene adjoint (mpm.cu) and the batched one
// (mpm_batch.cu).
//
// Reverse G2P: the forward G2P maps the grid velocities v_i to v_p, C_p and
// then x_p, F_p (Eq. G2P, Eq. deformation_update); its adjoint gives
// dL/dv_i (scattered, in the form of a P2G value), the partial dL/dx_p of the
// weights and dL/dF_p. Reverse grid update: dL/dm_i, dL/dp_i and the wind
// gradient. Reverse P2G: gathers (dL/dm_i, dL/dp_i) back to the particle
// (dL/dx_p, dL/dv_p, dL/dC_p, dL/dF_p through the stress, dL/dE).
#pragma once

#include "mpm_grid.cuh"
#include "mpm_p2g.cuh"
#include "wind.cuh"

namespace dw {

// Sums over a particle's 27 stencil nodes i, with val = the node's (x, y, z),
// or its (y, z, w) beside a mass channel x with MASS, and
// u_i = mv + A (x_i - x_p), linear in the node's offset o:
//   B_c  = sum W_i val_c,   S_cb = sum W_i o_b val_c (with MOMENTS),
//   G_a  = sum dW_i/dx_a (val . u_i [+ p_mass x with MASS] - ref),
// where ref, the middle node's bracket, changes nothing (the weights'
// derivatives add up to zero) but keeps the part that all nodes share out of
// the rounding. The weights are products, so lines along x are summed first:
// about 600 operations instead of the 1,200 to 1,600 of the sums written out
// per node. With the kernels' registers bounded (k_batch_rev_g2p) a 16-scene
// segment adjoint takes 10.4 ms instead of 11.9.
template <bool MASS, bool MOMENTS>
__device__ __forceinline__ void rev_gather(const MpmParams &P, const Stencil &s, const float A[9],
                                           const float mv[3], const float4 *__restrict__ grid,
                                           float B[3], float S[9], float G[3]) {
    const int N = P.N;
    const float4 *g0 = grid + ((int64_t)s.base[2] * N + s.base[1]) * N + s.base[0];
    float r[3], sx[3], sy[3], sz[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        sx[c] = A[3 * c] * P.dx;
        sy[c] = A[3 * c + 1] * P.dx;
        sz[c] = A[3 * c + 2] * P.dx;
        r[c] = mv[c] - (sx[c] * s.fx[0] + sy[c] * s.fx[1] + sz[c] * s.fx[2]);
        B[c] = G[c] = 0.0f;
    }
    if (MOMENTS)
#pragma unroll
        for (int k = 0; k < 9; ++k) S[k] = 0.0f;
    auto bracket = [&](const float4 &g, float u0, float u1, float u2) {
        return MASS ? P.p_mass * g.x + g.y * u0 + g.z * u1 + g.w * u2 : g.x * u0 + g.y * u1 + g.z * u2;
    };
    const float ref = bracket(g0[(N + 1) * N + 1], r[0] + sx[0] + sy[0] + sz[0], r[1] + sx[1] + sy[1] + sz[1],
                              r[2] + sx[2] + sy[2] + sz[2]);
#pragma unroll
    for (int ok = 0; ok < 3; ++ok)
#pragma unroll
        for (int oj = 0; oj < 3; ++oj) {
            float u[3], a[3] = {0.f, 0.f, 0.f}, bx[3] = {0.f, 0.f, 0.f}, f = 0.0f, fx = 0.0f;
#pragma unroll
            for (int c = 0; c < 3; ++c) u[c] = r[c] + (float)oj * sy[c] + (float)ok * sz[c];
#pragma unroll
            for (int oi = 0; oi < 3; ++oi) {
                const float4 g = g0[(ok * N + oj) * N + oi];
                const float w = s.w[0][oi];
                const float b = bracket(g, u[0] + (float)oi * sx[0], u[1] + (float)oi * sx[1],
                                        u[2] + (float)oi * sx[2]) - ref;
                f += w * b;
                fx += s.dw[0][oi] * b;
                const float v[3] = {MASS ? g.y : g.x, MASS ? g.z : g.y, MASS ? g.w : g.z};
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    a[c] += w * v[c];
                    if (MOMENTS && oi) bx[c] += (float)oi * w * v[c];
                }
            }
            const float wy = s.w[1][oj], wz = s.w[2][ok], wyz = wy * wz;
            G[0] += wyz * fx;
            G[1] += s.dw[1][oj] * wz * f;
            G[2] += wy * s.dw[2][ok] * f;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float t = wyz * a[c];
                B[c] += t;
                if (MOMENTS) {
                    S[3 * c] += wyz * bx[c];
                    if (oj) S[3 * c + 1] += (float)oj * t;
                    if (ok) S[3 * c + 2] += (float)ok * t;
                }
            }
        }
#pragma unroll
    for (int a = 0; a < 3; ++a) G[a] *= P.inv_dx;
}

// Reverse G2P of one particle at input position xp, input F Fp. bxo, bvo,
// bCo, bFo: dL/d(output x, v, C, F). Writes q (the node value
// W_ip (bv_p + D bC_p (x_i - x_p)), i.e. a P2G value with m v -> bv and
// A -> D bC, to be scattered with the mass channel off), bx = partial dL/dx_p
// and bFin = dL/dF_p through the F update. A particle outside the domain
// gets bx = bFin = 0 and q.valid = false. Cout (or NULL): the C array of the
// substep's output state (row stride `stride`, particle p), when a recompute
// kept it; then C' is read instead of gathered again from the grid.
__device__ __forceinline__ void rev_g2p_particle(const MpmParams &P, const float xp[3],
                                                 const float Fp[9], bool pin,
                                                 const float4 *__restrict__ grid_v,
                                                 const float bxo[3], const float bvo[3],
                                                 const float bCo[9], const float bFo[9],
                                                 P2GParticle &q, float bx[3], float bFin[9],
                                                 const float *__restrict__ Cout = nullptr,
                                                 int64_t stride = 0, int64_t p = 0) {
    q.valid = false;
    Stencil s;
    if (!make_stencil(P, xp[0], xp[1], xp[2], s)) {
#pragma unroll
        for (int a = 0; a < 3; ++a) bx[a] = 0.0f;
#pragma unroll
        for (int k = 0; k < 9; ++k) bFin[k] = 0.0f;
        return;
    }
    // F' = (I + dt C') F  ->  bF_in = (I + dt C')^T bF', bC' += dt bF' F^T
    float bFoFt[9], bv[3];
    mul3_abt(bFo, Fp, bFoFt);
#pragma unroll
    for (int k = 0; k < 9; ++k) q.A[k] = P.D * (bCo[k] + P.dt * bFoFt[k]);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        bv[a] = bvo[a] + P.dt * bxo[a];
        bx[a] = bxo[a];
    }
    if (pin) {  // C' = 0
#pragma unroll
        for (int k = 0; k < 9; ++k) bFin[k] = bFo[k];
        return;
    }
    // C' of the output state (v' is not needed: its adjoint only uses the
    // weights): kept by the recompute, else gathered from the grid again
    float M[9], B[3], G[3];
    if (Cout) {
#pragma unroll
        for (int k = 0; k < 9; ++k) M[k] = P.dt * Cout[k * stride + p];
        rev_gather<false, false>(P, s, q.A, bv, grid_v, B, nullptr, G);
    } else {
        float S[9];
        rev_gather<false, true>(P, s, q.A, bv, grid_v, B, S, G);
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int b = 0; b < 3; ++b)
                M[3 * c + b] = P.dt * (P.D * P.dx * (S[3 * c + b] - B[c] * s.fx[b]));
    }
    M[0] += 1.0f;
    M[4] += 1.0f;
    M[8] += 1.0f;
    mul3_atb(M, bFo, bFin);
#pragma unroll
    for (int a = 0; a < 3; ++a)
        bx[a] += G[a] - (q.A[a] * B[0] + q.A[3 + a] * B[1] + q.A[6 + a] * B[2]);
    q.s = s;
#pragma unroll
    for (int a = 0; a < 3; ++a) q.mv[a] = bv[a];
    q.valid = true;
}

// Reverse grid update of one node with mp = (m, p) and b4 = (0, dL/dv_i): out =
// (dL/dm_i, dL/dp_i). Returns whether the node took part in the grid update
// (m_i > 0, outside the sticky band); then gw is dt dL/dv_i, the cotangent of
// the wind force sampled at the node, for wind_scatter_block.
__device__ __forceinline__ bool rev_node_value(const MpmParams &P, int i, int j, int k,
                                               float4 mp, float4 b4, float4 &out,
                                               float3 &gw) {
    out = make_float4(0.f, 0.f, 0.f, 0.f);
    gw = make_float3(0.f, 0.f, 0.f);
    if (!(mp.x > 0.0f) || sticky_node(P, i, j, k)) return false;
    const float inv_m = 1.0f / mp.x;
    out.y = b4.y * inv_m;
    out.z = b4.z * inv_m;
    out.w = b4.w * inv_m;
    out.x = -(mp.y * b4.y + mp.z * b4.z + mp.w * b4.w) * inv_m * inv_m;
    gw = make_float3(P.dt * b4.y, P.dt * b4.z, P.dt * b4.w);
    return true;
}

// The same on the grid arrays, which also clears grid_mp and grid_bv for the
// next call.
__device__ __forceinline__ bool rev_grid_node(const MpmParams &P, int64_t node, int i, int j,
                                              int k, float4 *__restrict__ grid_mp,
                                              float4 *__restrict__ grid_bv,
                                              float4 *__restrict__ grid_bmp, float3 &gw) {
    float4 out;
    const bool live = rev_node_value(P, i, j, k, grid_mp[node], grid_bv[node], out, gw);
    grid_mp[node] = make_float4(0.f, 0.f, 0.f, 0.f);
    grid_bv[node] = make_float4(0.f, 0.f, 0.f, 0.f);
    grid_bmp[node] = out;
    return live;
}

// Reverse P2G of one particle at input state (xp, vp, Cp, Fp), gathering
// grid_bmp = (dL/dm_i, dL/dp_i). bx and bF enter with the reverse-G2P
// partials and leave as the complete dL/dx_p, dL/dF_p; writes bvp = dL/dv_p,
// bC = dL/dC_p and gE = this particle's dL/dE.
__device__ __forceinline__ void rev_p2g_particle(const MpmParams &P, const float xp[3],
                                                 const float vp[3], const float Cp[9],
                                                 const float Fp[9],
                                                 const float4 *__restrict__ grid_bmp, float bx[3],
                                                 float bF[9], float bvp[3], float bC[9],
                                                 float &gE) {
    Stencil s;
    float bA[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int a = 0; a < 3; ++a) bvp[a] = 0.0f;
    gE = 0.0f;
    if (make_stencil(P, xp[0], xp[1], xp[2], s)) {
        float Pk[9], PFt[9], A[9];
        stress_P(P, Fp, Pk);
        mul3_abt(Pk, Fp, PFt);
#pragma unroll
        for (int k = 0; k < 9; ++k) A[k] = -P.kappa * PFt[k] + P.p_mass * Cp[k];
        float mv[3], B[3], S[9], G[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) mv[c] = P.p_mass * vp[c];
        rev_gather<true, true>(P, s, A, mv, grid_bmp, B, S, G);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            bvp[c] = P.p_mass * B[c];
            bx[c] += G[c] - (A[c] * B[0] + A[3 + c] * B[1] + A[6 + c] * B[2]);
#pragma unroll
            for (int b = 0; b < 3; ++b) bA[3 * c + b] = P.dx * (S[3 * c + b] - B[c] * s.fx[b]);
        }
        // A = -kappa P F^T + m C
        float bAF[9], bAtP[9], bP[9];
        mul3(bA, Fp, bAF);
        mul3_atb(bA, Pk, bAtP);
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            bP[k] = -P.kappa * bAF[k];
            bF[k] += -P.kappa * bAtP[k];
        }
        stress_P_adjoint(P, Fp, bP, bF);
        float pp = 0.0f;
#pragma unroll
        for (int k = 0; k < 9; ++k) pp += bP[k] * Pk[k];
        gE = pp / P.E;
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) bC[k] = P.p_mass * bA[k];
}

// Sum of v over the CTA (blockDim.x a multiple of 32, at most 1024), valid in
// thread 0.
__device__ __forceinline__ float block_sum(float v) {
    __shared__ float red[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) red[wid] = v;
    __syncthreads();
    float s = 0.0f;
    if (wid == 0) {
        s = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.0f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    return s;
}

}  // namespace dw
