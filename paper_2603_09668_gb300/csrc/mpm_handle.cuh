// Internal view of an MPM handle shared by the MPM translation units: the
// workspace layout, launch instrumentation and the kernels and host helpers
// one unit launches from another.
#pragma once

#include <vector>

#include "mpm_g2p.cuh"
#include "mpm_grid.cuh"
#include "mpm_math.cuh"
#include "mpm_p2g.cuh"
#include "wind.cuh"

namespace dw {

struct MpmHandle {
    dw_mpm_desc desc;
    MpmParams P;
    int64_t n_nodes;
    float4 *grid_mp = nullptr;   // (m, p) after P2G; zero between calls
    float4 *grid_v = nullptr;    // (v, m) after the grid update
    float4 *grid_bv = nullptr;   // (0, dL/dv_i) during the adjoint; zero between calls
    float4 *grid_bmp = nullptr;  // (dL/dm_i, dL/dp_i) during the adjoint
    float *pscratch = nullptr;   // [12][max_particles]: partial dL/dx (3), dL/dF (9)
    double *gE_part = nullptr;   // [max_particles / 32 + 1]: dL/dE per CTA of a segment's reverse
    int *err = nullptr;          // device status bits
    // active 4^3 blocks of the grid (built by P2G, consumed by the grid update)
    int64_t nblk = 0;            // nb^3
    int *block_flag = nullptr;   // [nblk]
    int *block_list = nullptr;   // [2][nblk]: two lists so a fused kernel can fill one
    int *block_count = nullptr;  // [2]      while the grid update consumes the other
    // grid tape of a segment adjoint's recompute: per recomputed substep the
    // consumed list and each listed node's (m, p) (nblk entries of 64 nodes)
    float4 *gtape = nullptr;
    int *gtape_list = nullptr, *gtape_count = nullptr;
    int gtape_slots = 0;
    int gtape_refused = 0;       // slots a failed or oversized allocation was refused for
    // rollout workspace: the second state buffer of the sort ping-pong
    float *roll_state = nullptr;     // [24][max_particles]
    uint8_t *roll_pinned = nullptr;  // [max_particles]
    int32_t *roll_ids = nullptr;     // [max_particles]
    // sort workspace
    int nb = 0;                  // 4^3 blocks per axis
    int64_t n_keys = 0;
    int *keys = nullptr;         // [max_particles]
    int *counts = nullptr;       // [n_keys + 1]
    int *scan_tmp = nullptr;     // block sums for the exclusive scan
    int64_t scan_tmp_len = 0;
    // instrumentation: event pairs around kernel launches
    std::vector<cudaEvent_t> ev_start, ev_stop;
    std::vector<int> ev_kernel;
    int prof_used = 0;
};

// Brackets one kernel launch with events when profiling is enabled.
struct ProfScope {
    MpmHandle *h;
    cudaStream_t s;
    int slot = -1;
    ProfScope(MpmHandle *h_, int kid, cudaStream_t s_) : h(h_), s(s_) {
        if (h->prof_used < (int)h->ev_start.size()) {
            slot = h->prof_used++;
            h->ev_kernel[slot] = kid;
            cudaEventRecord(h->ev_start[slot], s);
        }
    }
    ~ProfScope() {
        if (slot >= 0) cudaEventRecord(h->ev_stop[slot], s);
    }
};

inline void profile_free(MpmHandle *h) {
    for (auto e : h->ev_start) cudaEventDestroy(e);
    for (auto e : h->ev_stop) cudaEventDestroy(e);
    h->ev_start.clear();
    h->ev_stop.clear();
    h->ev_kernel.clear();
    h->prof_used = 0;
}

inline MpmParams params_of(const dw_mpm_desc &d) {
    MpmParams P;
    P.N = d.n_grid;
    P.dx = 1.0f / (float)d.n_grid;
    P.inv_dx = (float)d.n_grid;
    P.dt = d.dt;
    P.D = 4.0f * (float)d.n_grid * (float)d.n_grid;
    P.gx = d.gravity[0];
    P.gy = d.gravity[1];
    P.gz = d.gravity[2];
    P.band = d.bc_band;
    P.material = d.material;
    double E = d.E, nu = d.nu;
    P.mu = (float)(E / (2.0 * (1.0 + nu)));                       // Eq. young_poisson
    P.lam = (float)(E * nu / ((1.0 + nu) * (1.0 - 2.0 * nu)));
    P.E = d.E;
    P.p_mass = d.p_mass;
    P.p_vol = d.p_vol;
    P.kappa = d.dt * d.p_vol * P.D;
    return P;
}

inline void fill_params(MpmHandle *h) { h->P = params_of(h->desc); }

constexpr int GRID_THREADS = 256;  // four 4^3 blocks per CTA iteration
constexpr int GRID_CTAS = 4 * 152;

inline ActiveBlocks active_blocks(MpmHandle *h, int which = 0) {
    return ActiveBlocks{h->block_flag, h->block_list + (size_t)which * h->nblk,
                        h->block_count + which, h->nb, 0};
}

// kernels of mpm.cu launched from other units
__global__ void k_grid_update_active(MpmParams P, WindDev wind, float t,
                                     float4 *__restrict__ grid_mp, float4 *__restrict__ grid_v,
                                     int clear, ActiveBlocks ab);
__global__ void k_grid_update_tape(MpmParams P, WindDev wind, float t, float4 *__restrict__ grid_mp,
                                   float4 *__restrict__ grid_v, ActiveBlocks ab,
                                   float4 *__restrict__ gtape, int *__restrict__ gtape_list,
                                   int *__restrict__ gtape_count);

// The recompute of a segment adjoint (mpm_rollout.cu): states 1 .. n_substeps
// - 1 from `start` into the tape slots, as one fused chain (the P2G of the
// start state, then per substep the grid update, kept in grid tape slot k
// when `keep_grid`, and the fused G2P/P2G kernel writing state k + 1 to its
// slot). with_last: also the grid of the last substep, into its grid tape slot
// and grid_v; *last_list is the active list its update consumed, whose count
// the next launch clears. For p2g modes AUTO and PAIR.
dw_status segment_recompute(MpmHandle *h, const dw_mpm_state *start, float *tape,
                            const uint8_t *pinned, const WindDev &wd, float t0, int n_substeps,
                            bool keep_grid, bool with_last, int *last_list, cudaStream_t s);

// The reverse pass of a segment whose recompute kept every substep's grid
// (with_last) and state, fused across substeps (mpm_layer.cu). Two launches per
// substep instead of four, which pays up to REV_CHAIN_MAX particles (us per
// substep of a segment, fused / four launches; a sheet on 64^3, a sheet on 128^3
// and a block on 64^3, in cell order; in random order):
//   100,000: 38.4 / 41.5, 43.1 / 46.2, 47.7 / 50.8; 101.1 / 106.8, 93.3 / 94.5, 91.7 / 92.8
//   140,000: 48.3 / 50.9, 52.0 / 55.2, 56.1 / 58.1; 131.2 / 126.8, 120.6 / 119.3, 122.1 / 120.3
//   200,000: 62.7 / 63.1, 66.3 / 66.4, 72.9 / 72.8; 197.2 / 188.2, 167.8 / 158.7, 167.1 / 156.7
//   400,000: 109.0 / 104.9, 114.3 / 110.8, 119.8 / 116.7; 299.8 / 284.1, 286.0 / 264.8, 279.5 / 256.6
constexpr int64_t REV_CHAIN_MAX = 3 << 16;
dw_status segment_reverse(MpmHandle *h, const dw_mpm_state *start, const float *tape,
                          const dw_mpm_state *g, const uint8_t *pinned, const WindDev &wd, float t0,
                          int n_substeps, float *g_wind, float *g_E, int *reset_count,
                          cudaStream_t s);

// The layer-split kernels (mpm_layer.cu), which DW_P2G_AUTO takes, and the particle
// counts up to which they are the faster ones (measured, us). A fused launch with
// its grid update: 7.9 against 11.9 at 5,504 particles, 9.4 / 11.6 at 32,768, 11.5 /
// 11.7 at 38,912, 12.3 / 11.5 at 40,960, 14.3 / 12.5 at 49,151 of a sheet; 13.7 /
// 15.6 at 38,912, 15.0 / 15.3 at 40,960, 18.9 / 17.3 at 65,535 of a block: the
// line lies where the layer kernel's CTAs (32 particles, eight per SM on 152 SMs)
// no longer run all at once.
// A whole substep, particles in cell order / in random order, of a sheet on 64^3,
// a sheet on 128^3 and a block on 64^3:
//   with both layer kernels      with the layer G2P        with neither
//   5,000:  12.4 12.3 12.3 / 14.4 14.4 14.4;  16.4 18.5 16.5 / 18.0 20.6 18.6;  18.5 20.1 18.5 / 20.4 20.6 20.6
//   38,912: 14.4 14.4 14.5 / 43.4 29.2 28.7;  18.3 16.5 18.5 / 35.4 24.7 26.7;  18.5 18.1 20.6 / 35.5 26.7 27.2
//   65,536: 18.5 18.6 20.7 / 69.2 45.2 41.7;  18.4 18.5 20.6 / 50.2 35.7 34.9;  18.6 18.5 20.2 / 49.4 35.2 35.0
//   131,072: 24.7 25.2 29.1 / 87.8 61.4 56.9 with both,  20.9 22.6 22.7 / 81.9 56.4 53.4 with neither
// P2G: the line of the fused kernel; above it the layer kernel's gain in cell
// order (2 us) is gone by 65,536, and in random order, where every particle adds
// to the grid by itself, it loses a quarter and more. G2P: 65,536, where it has
// stopped gaining in either order.
// The first P2G of a rollout or segment is another matter: the kernels after it
// keep the split of the SMs' memory that it leaves, and after the layer kernel's
// (most of it shared memory) they overlap better. A rollout's substep / 20 of them
// and a segment of 6 (us), block on 64^3 in cell order, layer P2G first against the
// one-particle one: 40,000: 18.3 / 607, 21.8 / 685; 100,000: 20.5 / 716, 20.9 / 746;
// 131,072: 27.5 / 772, 28.2 / 779; in random order 30.2 / 953, 41.9 / 1245; 48.7 /
// 1565, 55.8 / 1765; 57.1 / 1864, 66.2 / 2070 (sheets likewise). Not measured above.
constexpr int64_t LAYER_ROUND = 32 * 8 * 152, LAYER_MAX_P2G = LAYER_ROUND, LAYER_MAX_G2P = 1 << 16;
constexpr int64_t LAYER_MAX_CHAIN = 1 << 17;
inline bool layer_fused(int mode, int64_t n) { return mode == DW_P2G_AUTO && n <= LAYER_ROUND; }
dw_status launch_layer_p2g(const MpmParams &P, const float *x, const float *v, const float *C,
                           const float *F, int64_t n, float4 *grid, int *err,
                           const ActiveBlocks &ab, cudaStream_t st);
dw_status launch_layer_g2p(const MpmParams &P, const float *x, const float *F,
                           const uint8_t *pinned, const float4 *grid_v, const dw_mpm_state &out,
                           int64_t n, int *err, int *reset_count, cudaStream_t st);
// keys, counts: the next sort's (see PairOut), or NULL.
dw_status launch_layer_g2p2g(const MpmParams &P, const float *x, const float *F,
                             const uint8_t *pinned, const float4 *grid_v, const dw_mpm_state &out,
                             float4 *grid_next, int64_t n, int *err, const ActiveBlocks &ab_next,
                             int *reset_count, int *keys, int *counts, cudaStream_t st);

// particle sort (mpm.cu): counting sort by cell key, keys already counted
constexpr int SCAN_BLOCK = 1024;
constexpr int SCAN_ITEMS = 8;                         // consecutive elements per scan thread
constexpr int SCAN_TILE = SCAN_BLOCK * SCAN_ITEMS;    // elements per scan block
__global__ void k_sort_move(const int *__restrict__ keys, int64_t n, int *__restrict__ offsets,
                            const float *__restrict__ x, const float *__restrict__ v,
                            const float *__restrict__ C, const float *__restrict__ F,
                            const uint8_t *__restrict__ pin_in, const int *__restrict__ ids_in,
                            float *__restrict__ xo, float *__restrict__ vo, float *__restrict__ Co,
                            float *__restrict__ Fo, uint8_t *__restrict__ pin_out,
                            int *__restrict__ ids_out);
// In-place exclusive prefix sum of data[0, len); tmp holds at least
// len / SCAN_BLOCK + 1 ints.
dw_status exclusive_scan(int *data, int64_t len, int *tmp, int64_t tmp_len, cudaStream_t st);

// host helpers of mpm.cu
// G2P of n particles (x, F) into `out` (mode DW_P2G_*: AUTO takes the layer-split
// kernel where it is the faster one, the others never do); reset_count, when
// given, is the active-list count to clear.
dw_status launch_g2p(int mode, const MpmParams &P, const float *x, const float *F, const uint8_t *pinned,
                     const float4 *grid_v, const dw_mpm_state &out, int64_t n, int *err,
                     int *reset_count, cudaStream_t s);
dw_status validate_desc(const dw_mpm_desc *desc);
dw_status check_state(const MpmHandle *h, const dw_mpm_state *s, const char *name);
// with_vc = false leaves v and C of `out` unwritten (a rollout between fused
// launches, where v and C are not kept). keys_ready: h->keys and h->counts
// already hold the keys of `in` and their counts (the fused launch before
// the sort wrote them). clear_after: the counts are cleared at the end, for
// a fused launch that counts the next sort's keys.
dw_status sort_particles(MpmHandle *h, const dw_mpm_state *in, const dw_mpm_state *out,
                         const uint8_t *pinned_in, uint8_t *pinned_out, const int32_t *ids_in,
                         int32_t *ids_out, cudaStream_t s, bool with_vc = true,
                         bool keys_ready = false, bool clear_after = false);

}  // namespace dw

struct dw_mpm_s : dw::MpmHandle {};
