// Device-side sampling of the wind force field a_w(x, t): trilinear in space
// over a node-centred nf^3 grid on the unit cube (node j at j / (nf - 1)),
// linear in time between keyframes at k * t_total / (n_frames - 1), clamped
// (the force property of the wind grid field, Sec. 3 and Sec. 3.3).
#pragma once

#include "mpm_math.cuh"

namespace dw {

struct WindDev {
    const float *values;  // [n_frames][nf][nf][nf][3], x fastest
    int nf;
    int n_frames;
    float t_total;
};

// The up-to-16 (frame, corner) taps of one sample: element offsets of the
// first component of each tap and its weight.
struct WindTaps {
    int base;       // node index of corner (i0, j0, k0) in frame k0
    int sx, sy, sz; // node strides to the +1 corner per axis (0 if nf == 1)
    int st;         // node stride to the next frame (0 if n_frames == 1)
    int i0[3];      // corner (i0, j0, k0) of the spatial cell
    int kf;         // first keyframe
    float fr[3];
    float ft;
};

__device__ __forceinline__ WindTaps wind_taps(const WindDev &w, float px, float py, float pz,
                                              float t) {
    WindTaps tp;
    const int nf = w.nf;
    float p[3] = {px, py, pz};
    int i0[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        float q = fminf(fmaxf(p[a], 0.0f), 1.0f);
        if (nf < 2) {
            i0[a] = 0;
            tp.fr[a] = 0.0f;
        } else {
            float s = q * (float)(nf - 1);
            int i = (int)floorf(s);
            i = min(max(i, 0), nf - 2);
            i0[a] = i;
            tp.fr[a] = s - (float)i;
        }
    }
    int k0 = 0;
    tp.ft = 0.0f;
    if (w.n_frames > 1) {
        float tc = fminf(fmaxf(t, 0.0f), w.t_total);
        float s = tc / w.t_total * (float)(w.n_frames - 1);
        k0 = min(max((int)floorf(s), 0), w.n_frames - 2);
        tp.ft = s - (float)k0;
    }
    tp.base = ((k0 * nf + i0[2]) * nf + i0[1]) * nf + i0[0];
#pragma unroll
    for (int a = 0; a < 3; ++a) tp.i0[a] = i0[a];
    tp.kf = k0;
    tp.sx = nf > 1 ? 1 : 0;
    tp.sy = nf > 1 ? nf : 0;
    tp.sz = nf > 1 ? nf * nf : 0;
    tp.st = w.n_frames > 1 ? nf * nf * nf : 0;
    return tp;
}

__device__ __forceinline__ float3 wind_sample_dev(const WindDev &w, float px, float py, float pz,
                                                  float t) {
    WindTaps tp = wind_taps(w, px, py, pz, t);
    float3 acc = make_float3(0.f, 0.f, 0.f);
#pragma unroll
    for (int dk = 0; dk < 2; ++dk) {
        float wt_t = dk ? tp.ft : 1.0f - tp.ft;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            int cx = c & 1, cy = (c >> 1) & 1, cz = c >> 2;
            float wt = wt_t * (cx ? tp.fr[0] : 1.0f - tp.fr[0]) *
                       (cy ? tp.fr[1] : 1.0f - tp.fr[1]) * (cz ? tp.fr[2] : 1.0f - tp.fr[2]);
            // every tap lies inside the field (wind_taps clamps the corner),
            // so all 48 loads are issued without a branch; a zero weight adds
            // a signed zero, which leaves the (never negative-zero) sum as it is
            int node = tp.base + dk * tp.st + cx * tp.sx + cy * tp.sy + cz * tp.sz;
            const float *v = w.values + 3 * (size_t)node;
            acc.x += wt * __ldg(v + 0);
            acc.y += wt * __ldg(v + 1);
            acc.z += wt * __ldg(v + 2);
        }
    }
    return acc;
}

// g_values += taps^T g (atomic scatter into the field gradient).
__device__ __forceinline__ void wind_sample_adjoint_dev(const WindDev &w, float px, float py,
                                                        float pz, float t, float3 g,
                                                        float *g_values) {
    WindTaps tp = wind_taps(w, px, py, pz, t);
#pragma unroll
    for (int dk = 0; dk < 2; ++dk) {
        float wt_t = dk ? tp.ft : 1.0f - tp.ft;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            int cx = c & 1, cy = (c >> 1) & 1, cz = c >> 2;
            float wt = wt_t * (cx ? tp.fr[0] : 1.0f - tp.fr[0]) *
                       (cy ? tp.fr[1] : 1.0f - tp.fr[1]) * (cz ? tp.fr[2] : 1.0f - tp.fr[2]);
            if (wt == 0.0f) continue;
            int node = tp.base + dk * tp.st + cx * tp.sx + cy * tp.sy + cz * tp.sz;
            float *gv = g_values + 3 * (size_t)node;
            atomicAdd(gv + 0, wt * g.x);
            atomicAdd(gv + 1, wt * g.y);
            atomicAdd(gv + 2, wt * g.z);
        }
    }
}

// Shared memory of wind_scatter_block, one per group of 64 threads.
struct WindGroup {
    float g[3][64];     // the nodes' cotangents, then the sums over x
    float t[3][64];     // the sums over x and y
    float w[3][4][4];   // weight of wind node e at grid node i, per axis
};

__device__ __forceinline__ void group_sync(int id) {
    asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory");
}

// group_sync that also tells whether any thread of the group passed true.
__device__ __forceinline__ bool group_any(int id, bool v) {
    unsigned r;
    asm volatile(
        "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.or.pred q, %2, 64, p;\n"
        "selp.u32 %0, 1, 0, q;\n}"
        : "=r"(r)
        : "r"((unsigned)v), "r"(id)
        : "memory");
    return r != 0;
}

// g_values += taps^T g for the 64 nodes of one 4^3 grid block, called by all
// 64 threads of a group (thread lt at node (i, j, k), lt = its place in the
// block, x fastest; active = false adds nothing) with the same field and time
// and the group's barrier id. The sample's weights are a product over the axes,
// so the block's contributions to the wind nodes it touches (at most four per
// axis when three grid cells span less than three wind cells, else every node
// scatters its own taps) are summed one axis at a time in shared memory, and
// each touched wind node gets one atomic per component and keyframe instead of
// 16 taps per grid node. 5,504 particles, 12^3 wind nodes: the reverse grid
// update took 13.0 us with per-warp shared-memory atomics.
__device__ __forceinline__ void wind_scatter_block(const MpmParams &P, const WindDev &w,
                                                   bool active, int i, int j, int k, float t,
                                                   float3 g, float *g_values, WindGroup &G, int id) {
    const int lt = threadIdx.x & 63;
    if (!group_any(id, active)) return;  // (the previous block's sums are read by now)
    // the taps of the block's first and last node on each axis
    const int b[3] = {i - (lt & 3), j - ((lt >> 2) & 3), k - (lt >> 4)};
    const WindTaps lo = wind_taps(w, b[0] * P.dx, b[1] * P.dx, b[2] * P.dx, t);
    const WindTaps hi = wind_taps(w, (b[0] + 3) * P.dx, (b[1] + 3) * P.dx, (b[2] + 3) * P.dx, t);
    if (hi.i0[0] - lo.i0[0] > 2 || hi.i0[1] - lo.i0[1] > 2 || hi.i0[2] - lo.i0[2] > 2) {
        if (active) wind_sample_adjoint_dev(w, i * P.dx, j * P.dx, k * P.dx, t, g, g_values);
        return;
    }
    G.g[0][lt] = active ? g.x : 0.0f;
    G.g[1][lt] = active ? g.y : 0.0f;
    G.g[2][lt] = active ? g.z : 0.0f;
    if (lt < 4) {  // the weights at grid node lt of each axis
        const WindTaps tp = wind_taps(w, (b[0] + lt) * P.dx, (b[1] + lt) * P.dx, (b[2] + lt) * P.dx, t);
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int d = lo.i0[a] + e - tp.i0[a];
                G.w[a][lt][e] = d == 0 ? 1.0f - tp.fr[a] : (d == 1 ? tp.fr[a] : 0.0f);
            }
    }
    // (a cotangent that is not finite must not meet the zero weights of other wind nodes)
    if (group_any(id, active && !isfinite(g.x + g.y + g.z))) {
        if (active) wind_sample_adjoint_dev(w, i * P.dx, j * P.dx, k * P.dx, t, g, g_values);
        return;
    }
    const int ex = lt & 3, q1 = (lt >> 2) & 3, q2 = lt >> 4;
    float s[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {  // wind node ex of x, grid row (q1, q2)
        s[c] = 0.0f;
#pragma unroll
        for (int m = 0; m < 4; ++m) s[c] += G.w[0][m][ex] * G.g[c][(q2 * 4 + q1) * 4 + m];
        G.t[c][lt] = s[c];
    }
    group_sync(id);
#pragma unroll
    for (int c = 0; c < 3; ++c) {  // wind nodes (ex, q1) of x and y, grid plane q2
        s[c] = 0.0f;
#pragma unroll
        for (int m = 0; m < 4; ++m) s[c] += G.w[1][m][q1] * G.t[c][(q2 * 4 + m) * 4 + ex];
        G.g[c][lt] = s[c];
    }
    group_sync(id);
#pragma unroll
    for (int c = 0; c < 3; ++c) {  // wind node (ex, q1, q2)
        s[c] = 0.0f;
#pragma unroll
        for (int m = 0; m < 4; ++m) s[c] += G.w[2][m][q2] * G.g[c][(m * 4 + q1) * 4 + ex];
    }
    const int nx = lo.i0[0] + ex, ny = lo.i0[1] + q1, nz = lo.i0[2] + q2;
    if (nx >= w.nf || ny >= w.nf || nz >= w.nf) return;  // no weight there
    for (int dk = 0; dk < 2; ++dk) {
        const float wt = dk ? lo.ft : 1.0f - lo.ft;
        if (wt == 0.0f) continue;
        float *gv = g_values + 3 * (size_t)((((lo.kf + dk) * w.nf + nz) * w.nf + ny) * w.nf + nx);
#pragma unroll
        for (int c = 0; c < 3; ++c)
            if (s[c] != 0.0f) atomicAdd(gv + c, wt * s[c]);
    }
}

// Host-side validation of a dw_wind_field; fills the device view.
dw_status wind_check(const dw_wind_field *w, WindDev *out);

}  // namespace dw
