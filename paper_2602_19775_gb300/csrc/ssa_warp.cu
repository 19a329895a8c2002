// ssa_warp.cu -- warp-per-trajectory forward and adjoint for networks with many reactions
// (arXiv 2602.19775, Section 2, Section 3.2, Eqs. 3, 5, 6, 7, Section 3.1).
//
// One warp simulates one trajectory. Lane l owns the Philox blocks b = l, l + 32, ... of each step,
// i.e. the words q = 4b..4b+3 and the reactions j = q - 1 they drive, so no Philox word is computed
// twice. Per step:
//   - the propensities are kept in shared memory from step to step; an event forms again those of the reactions
//     that react in a species it changed;
//   - each lane adds its partial sum of a0 (fixed order) and the upper bounds of its race keys, one approximate
//     reciprocal per reaction; a0 is a butterfly sum over the lanes (every lane obtains the same bits);
//   - the Gumbel-max choice is the one reaction whose bound reaches the best lower bound, or, where several do, the
//     exact race (a butterfly argmax of (a_j, E_j, j) with a_i E_b > a_b E_i and ties to the lowest j);
//   - the clock, the sample writes and the state update are warp-uniform (lanes share the stoichiometry
//     and observable loops).
// Per-reaction values lie by the word that drives them: a lane reads and writes its block of four at once.
// The adjoint keeps per-reaction values in per-warp shared memory and accumulates the state adjoint
// through a species -> reactions table in a fixed order (no atomics, deterministic).
// Bound: instruction issue (ncu, 11 species and 301 reactions, 2,500 trajectories: ~63% issue active at four to five
// warps per scheduler, the rest fixed-latency dependences of a step). Instructions per step: forward 1,340 -> 725
// (the logarithms of the race and the propensities of untouched reactions are gone), adjoint 4,430 -> 1,756 (the same,
// one division per species instead of two per reaction, keys without logarithms of E). One gradient step of those
// trajectories to t = 2: 30.1 -> 13.8 ms.
#include <cstdint>

#include "ssa_warp_body.cuh"

namespace ssa {

// Resident blocks the warp adjoint is compiled for: 5 (102 registers) and 6 (80) are within 2% of each other on a
// 301-reaction network, 4 and 7 slower by 2% and 7%.
constexpr int kWarpAdjBlocks = 5;

// STAGED: the tables are copied to shared memory, where every step reads them; a network whose tables do not fit
// beside the warps' arrays reads them from global memory through L1.
template <int READOUT, bool RECORD, bool STAGED>
__global__ void __launch_bounds__(128, READOUT == SSA_READOUT_BIN ? 5 : 6) fwd_warp_kernel(const FwdParams p)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int wib = threadIdx.x >> 5, W = blockDim.x >> 5;
    const int Npad = (p.N + 3) & ~3;
    // staged: rx and stoichiometry | rates | barrier, status | second region; then per warp X [Npad],
    // a [wide_len]
    unsigned char *s_k = smem + p.inc_off, *s_bar = s_k + p.k_bytes, *s_more = s_bar + 16;
    float *wbase = reinterpret_cast<float *>(STAGED ? s_more + p.wtab_bytes : smem) + wib * (Npad + wide_len(p.M));
    if (STAGED && !stage_tables(smem, p.rx, p.inc_off, s_k, p.k_rates, p.k_bytes, reinterpret_cast<uint64_t *>(s_bar),
                                reinterpret_cast<int *>(s_bar + 8), p.err, s_more, p.wtab, p.wtab_bytes))
        return;
    const WarpTab tab = STAGED ? warp_tab(p, reinterpret_cast<const int4 *>(smem), reinterpret_cast<const int4 *>(s_more),
                                          reinterpret_cast<const float *>(s_k))
                               : warp_tab(p, p.rx, p.wtab, p.k_rates);
    const int64_t i = (int64_t)blockIdx.x * W + wib;
    if (i >= p.n_traj) return;  // whole warp
    warp_fwd_body<READOUT, RECORD>(p, tab, reinterpret_cast<int *>(wbase), wbase + Npad, i);
}

// The soft forward (Eq. 4) on the warp layout: the staged tables and rates, then the species-major update
// list; per warp X [Npad], dX [Npad] (floats) and the keys / weights y [Mp].
template <int READOUT, bool RECORD>
__global__ void __launch_bounds__(256) fwd_warp_soft_kernel(const FwdParams p)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int wib = threadIdx.x >> 5, W = blockDim.x >> 5;
    const int Npad = (p.N + 3) & ~3;
    int4 *s_rx = reinterpret_cast<int4 *>(smem);
    float *s_k = reinterpret_cast<float *>(smem + p.tab_bytes);
    uint64_t *s_bar = reinterpret_cast<uint64_t *>(smem + p.tab_bytes + p.k_bytes);
    int *s_ok = reinterpret_cast<int *>(smem + p.tab_bytes + p.k_bytes + 8);
    int *s_upd = reinterpret_cast<int *>(smem + p.tab_bytes + p.k_bytes + 16);
    float *wbase = reinterpret_cast<float *>(s_upd + p.upd_words) + wib * (2 * Npad + p.Mp);

    if (!stage_tables(smem, p.rx, p.tab_bytes, s_k, p.k_rates, p.k_bytes, s_bar, s_ok, p.err)) return;
    for (uint32_t q = threadIdx.x; q < p.upd_words; q += blockDim.x) s_upd[q] = p.upd[q];
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * W + wib;
    if (i >= p.n_traj) return;  // whole warp
    warp_soft_fwd_body<READOUT, RECORD>(p, s_rx, s_k, s_upd, wbase, wbase + Npad, wbase + 2 * Npad, i);
}

// Gradient of the soft forward on the warp layout: tables, rates, the update list, then per warp
// Xs [kSoftK][Npad], lam [Npad], dX [Npad], a, h, y, c1, c2, dA [Mp]; dA reduced over the block in a fixed order.
template <int READOUT>
__global__ void __launch_bounds__(256) adj_warp_soft_kernel(const AdjParams p, const int *upd, uint32_t upd_words)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, W = blockDim.x >> 5;
    const int N = p.N, M = p.M, Mp = p.Mp;
    const int Npad = (N + 3) & ~3;
    int4 *s_rx = reinterpret_cast<int4 *>(smem);
    int *s_st = reinterpret_cast<int *>(smem + 16 * Mp);
    const int *s_inc_ptr = reinterpret_cast<const int *>(smem + p.inc_off);
    const int *s_inc = reinterpret_cast<const int *>(smem + p.inc_list_off);
    float *s_k = reinterpret_cast<float *>(smem + p.tab_bytes);
    uint64_t *s_bar = reinterpret_cast<uint64_t *>(smem + p.tab_bytes + p.k_bytes);
    int *s_ok = reinterpret_cast<int *>(smem + p.tab_bytes + p.k_bytes + 8);
    int *s_upd = reinterpret_cast<int *>(smem + p.tab_bytes + p.k_bytes + 16);
    const size_t per_warp = (size_t)(kSoftK + 2) * Npad + 6 * (size_t)Mp;
    float *base0 = reinterpret_cast<float *>(s_upd + upd_words);
    float *wbase = base0 + wib * per_warp;
    float *Xs = wbase;
    float *lam = Xs + kSoftK * Npad;
    float *dX = lam + Npad;
    float *aj = dX + Npad;
    float *hj = aj + Mp;
    float *y = hj + Mp;
    float *c1 = y + Mp;
    float *c2 = c1 + Mp;
    float *dA = c2 + Mp;

    if (!stage_tables(smem, p.rx, p.tab_bytes, s_k, p.k_rates, p.k_bytes, s_bar, s_ok, p.err)) {
        for (int j = threadIdx.x; j < M; j += blockDim.x) p.partial[(int64_t)blockIdx.x * M + j] = 0.0f;
        return;
    }
    for (uint32_t q = threadIdx.x; q < upd_words; q += blockDim.x) s_upd[q] = upd[q];
    for (int j = lane; j < Mp; j += 32) dA[j] = 0.0f;
    __syncthreads();

    const int64_t n = p.n_traj;
    const int64_t i = (int64_t)blockIdx.x * W + wib;
    int st = -1;
    if (i < n) st = p.status[i];
    const bool active = st == SSA_TRAJ_OK || st == SSA_TRAJ_ABSORBED || st == SSA_TRAJ_STEP_CAP;
    if (active)
        warp_soft_adj_body<READOUT>(p, s_rx, s_st, s_inc_ptr, s_inc, s_k, s_upd, Xs, lam, dX, aj, hj, y, c1, c2, dA, i,
                                    st);
    __syncthreads();
    const int nb = (M + 4) >> 2;
    for (int j = threadIdx.x; j < M; j += blockDim.x) {
        float acc = 0.0f;
        for (int w = 0; w < W; ++w) acc += base0[w * per_warp + (kSoftK + 2) * Npad + 5 * Mp + jpos(j, nb)];
        p.partial[(int64_t)blockIdx.x * M + j] = acc;
    }
}

template <int READOUT, bool STAGED, bool HOT>
__global__ void __launch_bounds__(128, kWarpAdjBlocks) adj_warp_kernel(const AdjParams p)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, W = blockDim.x >> 5;
    const int M = p.M, Mw = wide_len(M), Npad = (p.N + 3) & ~3;
    // staged as in the forward; per warp: X [Npad] int, lambda [Npad], propensities, keys / weights / per-reaction
    // adjoints, w_j, dA [wide_len each]
    const size_t per_warp = (size_t)2 * Npad + 4 * (size_t)Mw;
    unsigned char *s_k = smem + p.inc_off, *s_bar = s_k + p.k_bytes, *s_more = s_bar + 16;
    float *base0 = reinterpret_cast<float *>(STAGED ? s_more + p.wtab_bytes : smem);
    float *wbase = base0 + wib * per_warp;
    int *X = reinterpret_cast<int *>(wbase);
    float *lam = wbase + Npad;
    float *ad = lam + Npad;
    float *rj = ad + Mw;
    float *ct = rj + Mw;
    float *dA = ct + Mw;

    if (STAGED && !stage_tables(smem, p.rx, p.inc_off, s_k, p.k_rates, p.k_bytes, reinterpret_cast<uint64_t *>(s_bar),
                                reinterpret_cast<int *>(s_bar + 8), p.err, s_more, p.wtab, p.wtab_bytes)) {
        for (int j = threadIdx.x; j < M; j += blockDim.x) p.partial[(int64_t)blockIdx.x * M + j] = 0.0f;
        return;
    }
    const WarpTab tab = STAGED ? warp_tab(p, reinterpret_cast<const int4 *>(smem), reinterpret_cast<const int4 *>(s_more),
                                          reinterpret_cast<const float *>(s_k))
                               : warp_tab(p, p.rx, p.wtab, p.k_rates);
    for (int j = lane; j < Mw; j += 32) dA[j] = 0.0f;

    const int64_t n = p.n_traj;
    const int64_t i = (int64_t)blockIdx.x * W + wib;
    int st = -1;
    if (i < n) st = p.status[i];
    const bool active = st == SSA_TRAJ_OK || st == SSA_TRAJ_ABSORBED || st == SSA_TRAJ_STEP_CAP;
    if (active) warp_adj_body<READOUT, HOT>(p, tab, X, lam, ad, rj, ct, dA, i, st);
    __syncthreads();
    // fixed-order reduction over the block's warps
    for (int j = threadIdx.x; j < M; j += blockDim.x) {
        float acc = 0.0f;
        for (int w = 0; w < W; ++w) acc += base0[w * per_warp + 2 * Npad + 3 * Mw + j + 1];
        p.partial[(int64_t)blockIdx.x * M + j] = acc;
    }
}

// ---------------------------------------------------------------------------------------------
// shared memory of a block: the staged tables (0 where they do not fit beside the warps' arrays) and the arrays
static size_t staged_bytes(uint32_t inc_off, uint32_t k_bytes, uint32_t wtab_bytes)
{
    return (size_t)inc_off + k_bytes + 16 + wtab_bytes;
}

template <int R, bool REC>
static cudaError_t launch_fwd_w(const FwdParams &p, int warps, size_t limit, cudaStream_t st)
{
    const size_t own = (size_t)warps * (((p.N + 3) & ~3) + wide_len(p.M)) * 4;
    const size_t full = own + staged_bytes(p.inc_off, p.k_bytes, p.wtab_bytes);
    const bool staged = full <= limit;
    auto kern = staged ? fwd_warp_kernel<R, REC, true> : fwd_warp_kernel<R, REC, false>;
    const size_t smem = staged ? full : own;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t grid = (p.n_traj + warps - 1) / warps;
    kern<<<(unsigned)grid, warps * 32, smem, st>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_forward_warp(const FwdParams &p, int readout, bool record, int warps, size_t limit, cudaStream_t st)
{
    if (p.n_traj == 0) return cudaSuccess;
    if (readout == SSA_READOUT_HOLD)
        return record ? launch_fwd_w<0, true>(p, warps, limit, st) : launch_fwd_w<0, false>(p, warps, limit, st);
    if (readout == SSA_READOUT_BIN)
        return record ? launch_fwd_w<2, true>(p, warps, limit, st) : launch_fwd_w<2, false>(p, warps, limit, st);
    return record ? launch_fwd_w<1, true>(p, warps, limit, st) : launch_fwd_w<1, false>(p, warps, limit, st);
}

template <int R, bool REC>
static cudaError_t launch_fwd_soft_w(const FwdParams &p, int warps, size_t smem, cudaStream_t st)
{
    auto kern = fwd_warp_soft_kernel<R, REC>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t grid = (p.n_traj + warps - 1) / warps;
    kern<<<(unsigned)grid, warps * 32, smem, st>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_forward_warp_soft(const FwdParams &p, int readout, bool record, int warps, size_t smem,
                                     cudaStream_t st)
{
    if (p.n_traj == 0) return cudaSuccess;
    if (readout == SSA_READOUT_HOLD)
        return record ? launch_fwd_soft_w<0, true>(p, warps, smem, st) : launch_fwd_soft_w<0, false>(p, warps, smem, st);
    if (readout == SSA_READOUT_BIN)
        return record ? launch_fwd_soft_w<2, true>(p, warps, smem, st) : launch_fwd_soft_w<2, false>(p, warps, smem, st);
    return record ? launch_fwd_soft_w<1, true>(p, warps, smem, st) : launch_fwd_soft_w<1, false>(p, warps, smem, st);
}

template <int R>
static cudaError_t launch_adj_soft_w(const AdjParams &p, const int *upd, uint32_t upd_words, int warps, size_t smem,
                                     int64_t grid, cudaStream_t st)
{
    auto kern = adj_warp_soft_kernel<R>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)grid, warps * 32, smem, st>>>(p, upd, upd_words);
    return cudaGetLastError();
}

cudaError_t launch_backward_warp_soft(const AdjParams &p, const int *upd, uint32_t upd_words, int readout, int warps,
                                      size_t smem, int64_t grid, cudaStream_t st)
{
    if (grid == 0) return cudaSuccess;
    if (readout == SSA_READOUT_HOLD) return launch_adj_soft_w<0>(p, upd, upd_words, warps, smem, grid, st);
    if (readout == SSA_READOUT_BIN) return launch_adj_soft_w<2>(p, upd, upd_words, warps, smem, grid, st);
    return launch_adj_soft_w<1>(p, upd, upd_words, warps, smem, grid, st);
}

template <int R, bool HOT>
static cudaError_t launch_adj_w(const AdjParams &p, int warps, size_t limit, int64_t grid, cudaStream_t st)
{
    const size_t own = (size_t)warps * (2 * ((p.N + 3) & ~3) + 4 * (size_t)wide_len(p.M)) * 4;
    const size_t full = own + staged_bytes(p.inc_off, p.k_bytes, p.wtab_bytes);
    const bool staged = full <= limit;
    auto kern = staged ? adj_warp_kernel<R, true, HOT> : adj_warp_kernel<R, false, HOT>;
    const size_t smem = staged ? full : own;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)grid, warps * 32, smem, st>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_backward_warp(const AdjParams &p, int readout, int warps, size_t limit, int64_t grid,
                                 cudaStream_t st)
{
    if (grid == 0) return cudaSuccess;
    const bool hot = hot_weights(p.invT);
    switch (readout) {
    case SSA_READOUT_HOLD:
        return hot ? launch_adj_w<0, true>(p, warps, limit, grid, st) : launch_adj_w<0, false>(p, warps, limit, grid, st);
    case SSA_READOUT_LINEAR:
        return hot ? launch_adj_w<1, true>(p, warps, limit, grid, st) : launch_adj_w<1, false>(p, warps, limit, grid, st);
    default:
        return hot ? launch_adj_w<2, true>(p, warps, limit, grid, st) : launch_adj_w<2, false>(p, warps, limit, grid, st);
    }
}

}  // namespace ssa
