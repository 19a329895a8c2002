// ssa_batch.cu -- many networks of uneven size, parameter sets and trajectory counts in one
// persistent launch per direction (forward, then the straight-through adjoint), captured with the
// rate, validation and reduction kernels in one CUDA graph (arXiv 2602.19775, Sections 2-3: every
// network runs the same exact SSA and the same adjoint as the single-network entry points).
//
// Work is cut into units: 32 trajectories of one network for the thread-per-trajectory variant (one
// per lane), or one trajectory run by a whole warp for the warp-per-trajectory
// variant. The host orders the units longest first (estimated draws x reactions x trajectories, from
// the autotuner's pilot runs) and every warp of a persistent grid (one wave: SMs x resident blocks)
// pulls the next unit from an atomic counter. The per-trajectory code is the same as the
// single-network kernels', with the network tables read from global memory through the read-only
// path. Each unit writes its per-reaction adjoints to its own slot, and the slots of a network are
// summed in a fixed order, so gradients do not depend on which warp ran which unit.
#include <algorithm>
#include <cstring>
#include <new>
#include <vector>

#include "ssa_fwd_body.cuh"
#include "ssa_host.h"
#include "ssa_warp_body.cuh"

#define CUDA_TRY_B(expr)                                                                                \
    do {                                                                                                \
        cudaError_t e_ = (expr);                                                                        \
        if (e_ != cudaSuccess) return set_error(SSA_ERR_CUDA, cudaGetErrorString(e_));                 \
    } while (0)

namespace ssa {
cudaError_t launch_unpack_events(const uint4 *ev, const int *draws, int64_t n_traj, int64_t stride, int *out,
                                 cudaStream_t st);
cudaError_t launch_transpose_brackets(const int *brk, int64_t n_traj, int S, const int *first, const int *nslots,
                                      int *out, cudaStream_t st);

struct BatchItem {
    FwdParams f;
    AdjParams a;
    int variant;             // 1: thread per trajectory (compile-time bound mc), 32: warp per trajectory
    int mc;
    int64_t slot_off;        // first float of this network's partial slots
    int n_units;
    const float *log_rates;  // caller's theta
    const int *rate_index;
    int P;
    float *dtheta;           // caller's dL/dlog k
    float *dA;               // per-reaction sums (workspace)
};

struct BatchUnit {
    int item;
    int count;           // trajectories in the unit
    int64_t traj_begin;  // local trajectory index within the network
    int slot;            // canonical index of the unit within its network
};

constexpr int kBatchWarps = 4;
constexpr int kBatchThreadMaxN = 16;  // thread variant inside a batch: N <= 16 and M <= 16
// Resident blocks per SM the warp-unit kernels are compiled for: more hide more latency, fewer let each trajectory run
// faster, which counts where one long trajectory ends a launch, and leave more of the SM's 256 KB to L1, through which the
// batch kernels read their tables. Milliseconds at 3, 4 and 5 blocks: 24 uneven networks (up to 32,768 draws) 177-191,
// 174-184, 200-208; 12 of them x 512 trajectories to t = 1 32.0, 27.6, 32.6; 40 networks of 30 to 100 reactions x 512 33.2,
// 27.4, 25.6 (bin readout 34.7, 29.6, 30.5).
#ifndef SSA_BATCH_WARP_BLOCKS
#define SSA_BATCH_WARP_BLOCKS 4
#endif
constexpr int kBatchWarpBlocks = SSA_BATCH_WARP_BLOCKS;
constexpr int kBatchWarpUnit = 1;     // trajectories per warp-variant unit (one: the finest grain for the tail)

__global__ void batch_prepare_kernel(const BatchItem *items, int n_items, int strict)
{
    // per network: k_j = exp(theta_{r(j)}) rounded once, and the check of its sample grid
    for (int it = blockIdx.x; it < n_items; it += gridDim.x) {
        const BatchItem &b = items[it];
        float *k = const_cast<float *>(b.f.k_rates);
        const int nb = (b.f.M + 4) >> 2;
        for (int e = threadIdx.x; e < b.f.Mp; e += blockDim.x) {
            // warp items keep their rates lane-major (position q nb + b holds reaction 4 b + q - 1)
            const int j = b.variant == 1 ? e : (e < 4 * nb ? 4 * (e % nb) + e / nb - 1 : -1);
            k[e] = (j >= 0 && j < b.f.M) ? (float)exp((double)b.log_rates[b.rate_index[j]]) : 0.0f;
        }
        int *flag = const_cast<int *>(b.f.flag);
        for (int s = threadIdx.x; s < b.f.S; s += blockDim.x) {
            // the bin readout needs strictly increasing edges with the first above 0 (its bins are (t_{s-1}, t_s])
            const bool ok = b.f.ts[s] >= 0.0 && b.f.ts[s] <= b.f.t_end &&
                            (s == 0 ? (!strict || b.f.ts[0] > 0.0)
                                    : (strict ? b.f.ts[s] > b.f.ts[s - 1] : b.f.ts[s] >= b.f.ts[s - 1]));
            if (!ok) atomicOr(flag, kErrBadSamples);
        }
        for (int c = threadIdx.x; c < b.f.n_obs; c += blockDim.x)
            if (b.f.obs_sp[c] < 0 || b.f.obs_sp[c] >= b.f.N) atomicOr(flag, kErrBadObs);
    }
}

// bin readout with a shared upstream gradient: one block per such item forms its binary64 prefix sums over
// bins (the single-network path's scan, so the same bits)
__global__ void __launch_bounds__(kPrefixThreads) batch_prefix_kernel(const BatchItem *items, int n_items)
{
    for (int it = blockIdx.x; it < n_items; it += gridDim.x) {
        const AdjParams &a = items[it].a;
        if (a.bin_prefix) bin_prefix_block(a.dl_dobs, a.S, a.n_obs, const_cast<double *>(a.bin_prefix));
    }
}

// the descriptor of the warp's current network is copied to shared memory, where the per-step
// reads of its sizes and pointers cost a shared load instead of a global one
constexpr int kItemWords = (int)((sizeof(BatchItem) + 15) / 16 * 4);

__device__ __forceinline__ int load_item(const BatchItem *items, int item, BatchItem *dst)
{
    __syncwarp();
    const int *src = reinterpret_cast<const int *>(items + item);
    int *d = reinterpret_cast<int *>(dst);
    for (int w = threadIdx.x & 31; w < (int)(sizeof(BatchItem) / 4); w += 32) d[w] = src[w];
    __syncwarp();
    return item;
}

__device__ __forceinline__ int next_unit(int *counter)
{
    int u = 0;
    if ((threadIdx.x & 31) == 0) u = atomicAdd(counter, 1);
    return __shfl_sync(0xffffffffu, u, 0);
}

template <int READOUT, int MC>
__device__ __forceinline__ void batch_fwd_thread_unit(const BatchItem &b, const BatchUnit &u, int *Xw)
{
    const FwdParams &p = b.f;
    const int lane = threadIdx.x & 31;
    const int4 *rx = p.rx;
    const int *st = reinterpret_cast<const int *>(reinterpret_cast<const unsigned char *>(p.rx) + 16 * p.Mp);
    if (lane < u.count) thread_fwd_body<READOUT, true, false, MC>(p, rx, st, p.k_rates, Xw + lane, 32, u.traj_begin + lane);
}

// VARIANT 1 runs the thread units, VARIANT 32 the warp units (separate kernels, so that the warp
// kernel is not compiled with the register budget of the unrolled thread bodies)
template <int READOUT, int VARIANT, bool SOFT = false>
__global__ void __launch_bounds__(32 * kBatchWarps, VARIANT == 1 ? 1 : kBatchWarpBlocks) batch_fwd_kernel(const BatchItem *items, const BatchUnit *units,
                                                                    int n_units, int *counter, int x_words)
{
    extern __shared__ __align__(16) int bsm[];
    BatchItem *s_items = reinterpret_cast<BatchItem *>(bsm);
    const int wib = threadIdx.x >> 5;
    int *Xw = bsm + kItemWords * (blockDim.x >> 5) + wib * x_words;
    int cached = -1;
    for (;;) {
        const int ui = next_unit(counter);
        if (ui >= n_units) break;
        const BatchUnit u = units[ui];
        if (u.item != cached) cached = load_item(items, u.item, s_items + wib);
        const BatchItem &b = s_items[wib];
        if constexpr (VARIANT == 1) {
            switch (b.mc) {
            case 2: batch_fwd_thread_unit<READOUT, 2>(b, u, Xw); break;
            case 4: batch_fwd_thread_unit<READOUT, 4>(b, u, Xw); break;
            case 8: batch_fwd_thread_unit<READOUT, 8>(b, u, Xw); break;
            default: batch_fwd_thread_unit<READOUT, 16>(b, u, Xw); break;
            }
        } else if constexpr (SOFT) {
            // the soft forward (Eq. 4), recorded: per warp X, dX [Npad] and the keys / weights [Mp] (floats)
            const FwdParams &p = b.f;
            float *Xf = reinterpret_cast<float *>(Xw);
            const int Npad = (p.N + 3) & ~3;
            for (int c = 0; c < u.count; ++c) {
                warp_soft_fwd_body<READOUT, true>(p, p.rx, p.k_rates, p.upd, Xf, Xf + Npad, Xf + 2 * Npad,
                                                  u.traj_begin + c);
                __syncwarp();
            }
        } else {
            const FwdParams &p = b.f;
            const WarpTab tab = warp_tab(p, p.rx, p.wtab, p.k_rates);
            float *a = reinterpret_cast<float *>(Xw) + ((p.N + 3) & ~3);
            for (int c = 0; c < u.count; ++c) {
                warp_fwd_body<READOUT, true>(p, tab, Xw, a, u.traj_begin + c);
                __syncwarp();
            }
        }
        __syncwarp();
    }
}

template <int READOUT, int MC, bool HOT>
__device__ __forceinline__ void batch_adj_thread_unit(const BatchItem &b, const BatchUnit &u, float *wsm)
{
    const AdjParams &p = b.a;
    const int lane = threadIdx.x & 31;
    const int4 *rx = p.rx;
    const int *st = reinterpret_cast<const int *>(reinterpret_cast<const unsigned char *>(p.rx) + 16 * p.Mp);
    int *X = reinterpret_cast<int *>(wsm);
    float *lam = wsm + kBatchThreadMaxN * 32;
    float *dlam = lam + kBatchThreadMaxN * 32;
    float dAr[MC];
#pragma unroll
    for (int j = 0; j < MC; ++j) dAr[j] = 0.0f;
    const int64_t i = u.traj_begin + lane;
    int stt = -1;
    if (lane < u.count) stt = p.status[i];
    const bool active = stt == SSA_TRAJ_OK || stt == SSA_TRAJ_ABSORBED || stt == SSA_TRAJ_STEP_CAP;
    if (active)
        thread_adj_body<READOUT, MC, HOT>(p, rx, st, p.k_rates, X + lane, lam + lane, dlam + lane, nullptr, nullptr, 32, i,
                                          stt, dAr);
    // fixed-order sum over the lanes (butterfly: every lane holds the same bits), lane 0 writes the slot
    float *slot = p.partial + b.slot_off + (int64_t)u.slot * p.M;
#pragma unroll
    for (int j = 0; j < MC; ++j) {
        const float v = warp_sum(dAr[j]);
        if (lane == 0 && j < p.M) slot[j] = v;
    }
}

template <int READOUT, int VARIANT, bool SOFT = false, bool HOT = false>
__global__ void __launch_bounds__(32 * kBatchWarps, VARIANT == 1 ? 1 : kBatchWarpBlocks) batch_adj_kernel(const BatchItem *items, const BatchUnit *units,
                                                                    int n_units, int *counter, int w_words)
{
    extern __shared__ __align__(16) float bsa[];
    BatchItem *s_items = reinterpret_cast<BatchItem *>(bsa);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    float *wsm = bsa + kItemWords * (blockDim.x >> 5) + wib * w_words;
    int cached = -1;
    for (;;) {
        const int ui = next_unit(counter);
        if (ui >= n_units) break;
        const BatchUnit u = units[ui];
        if (u.item != cached) cached = load_item(items, u.item, s_items + wib);
        const BatchItem &b = s_items[wib];
        if constexpr (VARIANT == 1) {
            switch (b.mc) {
            case 2: batch_adj_thread_unit<READOUT, 2, HOT>(b, u, wsm); break;
            case 4: batch_adj_thread_unit<READOUT, 4, HOT>(b, u, wsm); break;
            case 8: batch_adj_thread_unit<READOUT, 8, HOT>(b, u, wsm); break;
            default: batch_adj_thread_unit<READOUT, 16, HOT>(b, u, wsm); break;
            }
        } else {
            const AdjParams &p = b.a;
            const int Npad = (p.N + 3) & ~3;
            const int4 *rx = p.rx;
            float *dA;
            if constexpr (SOFT) {
                const unsigned char *tb = reinterpret_cast<const unsigned char *>(p.rx);
                const int *st = reinterpret_cast<const int *>(tb + 16 * p.Mp);
                const int *inc_ptr = reinterpret_cast<const int *>(tb + p.inc_off);
                const int *inc = reinterpret_cast<const int *>(tb + p.inc_list_off);
                // the soft forward's gradient: Xs [kSoftK][Npad], lam, dX [Npad]; a, h, y, c1, c2, dA [Mp]
                float *Xs = wsm;
                float *lam = Xs + kSoftK * Npad;
                float *dX = lam + Npad;
                float *aj = dX + Npad;
                float *hj = aj + p.Mp;
                float *y = hj + p.Mp;
                float *c1 = y + p.Mp;
                float *c2 = c1 + p.Mp;
                dA = c2 + p.Mp;
                for (int j = lane; j < p.Mp; j += 32) dA[j] = 0.0f;
                __syncwarp();
                for (int c = 0; c < u.count; ++c) {
                    const int64_t i = u.traj_begin + c;
                    const int stt = p.status[i];
                    if (stt == SSA_TRAJ_OK || stt == SSA_TRAJ_ABSORBED || stt == SSA_TRAJ_STEP_CAP)
                        warp_soft_adj_body<READOUT>(p, rx, st, inc_ptr, inc, p.k_rates, b.f.upd, Xs, lam, dX, aj, hj, y,
                                                    c1, c2, dA, i, stt);
                    __syncwarp();
                }
            } else {
                int *X = reinterpret_cast<int *>(wsm);
                float *lam = wsm + Npad;
                float *aj = lam + Npad;
                const int Mw = wide_len(p.M);
                float *lj = aj + Mw;
                float *ct = lj + Mw;
                dA = ct + Mw;
                const WarpTab tab = warp_tab(p, rx, p.wtab, p.k_rates);
                for (int j = lane; j < Mw; j += 32) dA[j] = 0.0f;
                __syncwarp();
                for (int c = 0; c < u.count; ++c) {
                    const int64_t i = u.traj_begin + c;
                    const int stt = p.status[i];
                    if (stt == SSA_TRAJ_OK || stt == SSA_TRAJ_ABSORBED || stt == SSA_TRAJ_STEP_CAP)
                        warp_adj_body<READOUT, HOT>(p, tab, X, lam, aj, lj, ct, dA, i, stt);
                    __syncwarp();
                }
            }
            float *slot = p.partial + b.slot_off + (int64_t)u.slot * p.M;
            const int nb = (p.M + 4) >> 2;
            for (int j = lane; j < p.M; j += 32) slot[j] = dA[SOFT ? jpos(j, nb) : j + 1];
        }
        __syncwarp();
    }
}

// dA of network `it` = fixed-order sum of its unit slots; one block per (network, reaction)
__global__ void batch_reduce_kernel(const BatchItem *items, const int *blk_item, const int *blk_j)
{
    __shared__ float red[256];
    const BatchItem &b = items[blk_item[blockIdx.x]];
    const int j = blk_j[blockIdx.x];
    const float *base = b.a.partial + b.slot_off;
    float acc = 0.0f;
    for (int u = threadIdx.x; u < b.n_units; u += blockDim.x) acc += base[(int64_t)u * b.a.M + j];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) b.dA[j] = red[0];
}

__global__ void batch_params_kernel(const BatchItem *items, int n_items)
{
    for (int it = blockIdx.x; it < n_items; it += gridDim.x) {
        const BatchItem &b = items[it];
        for (int r = threadIdx.x; r < b.P; r += blockDim.x) {
            float acc = 0.0f;
            for (int j = 0; j < b.a.M; ++j)
                if (b.rate_index[j] == r) acc += b.dA[j];
            b.dtheta[r] = acc;
        }
    }
}

}  // namespace ssa

// =============================================================================================
// C ABI
// =============================================================================================
using namespace ssa;

using BatchAdjKernel = void (*)(const BatchItem *, const BatchUnit *, int, int *, int);

struct ssa_batch {
    std::vector<ssa_batch_item> items;
    std::vector<int> variant, mc, K;
    std::vector<double> est_draws;
    double ckpt_scale = 1.0;  // the autotuner's multiple of the default checkpoint interval
    bool soft = false;        // every item runs the soft forward (Eq. 4) and its exact gradient, on warp units
    int readout;
    float temperature;
    // laid out in the caller's workspace by the first run with it
    unsigned char *ws = nullptr;
    int *d_flags = nullptr;  // [n_items][16]
    BatchItem *d_items = nullptr;
    BatchUnit *d_units = nullptr;
    int *d_counters = nullptr;
    int *d_blk_item = nullptr, *d_blk_j = nullptr;
    int n_red_blocks = 0;
    // per kernel variant (0: thread units, 1: warp units): units [unit_begin, unit_begin + n_units)
    int unit_begin[2] = {0, 0}, n_units[2] = {0, 0};
    int x_words[2] = {0, 0}, w_words[2] = {0, 0};
    int fwd_blocks[2] = {0, 0}, adj_blocks[2] = {0, 0};
    size_t fwd_smem[2] = {0, 0}, adj_smem[2] = {0, 0};
    int warps[2] = {0, 0};  // per block
    bool hot() const { return hot_weights(1.0f / temperature); }
    std::vector<BatchItem> h_items;
    cudaGraphExec_t graph = nullptr;
    bool ready = false;
};

namespace {

int batch_mc(int M) { return M <= 2 ? 2 : M <= 4 ? 4 : M <= 8 ? 8 : 16; }

bool thread_eligible(const ssa_network *net) { return net->N <= kBatchThreadMaxN && net->M <= 16; }

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

int64_t units_of(const ssa_batch *bt, size_t it)
{
    const int64_t n = bt->items[it].n_traj;
    const int per = bt->variant[it] == 1 ? 32 : kBatchWarpUnit;
    return (n + per - 1) / per;
}

// Workspace layout, shared by the size query and the build:
//   flags [n_items][16] int | per item: k [Mp] | draws [n] | status [n] | xfinal [N][n] |
//   events [rows][n] uint4 | checkpoints [n_ckpt][N][n] | brackets k, alpha [S][n] | bin readout: slot
//   edges [S][n], slot counts [n], prefix sums of a shared upstream gradient [S + 1][4] double | dA [M] |
//   unit slots [units][M] | item descriptors | units | reduction maps (item, j) | counters
struct BatchLayout {
    size_t flags = 0;
    std::vector<size_t> k, draws, status, xfinal, ev, ckpt, brk_k, brk_a, brk_s, brk_tail, prefix, dA;
    size_t partial = 0, items = 0, units = 0, blk_item = 0, blk_j = 0, counters = 0, total = 0;
    int64_t n_units = 0, n_slots = 0, n_red = 0;
};

BatchLayout batch_layout(const ssa_batch *bt)
{
    BatchLayout L;
    size_t off = 0;
    auto take = [&](size_t b) {
        const size_t at = off;
        off += align256(std::max<size_t>(b, 1));
        return at;
    };
    const size_t n_items = bt->items.size();
    L.flags = take(n_items * 16 * sizeof(int));
    for (size_t it = 0; it < n_items; ++it) {
        const ssa_batch_item &b = bt->items[it];
        const ssa_network *net = b.net;
        const size_t n = (size_t)b.n_traj;
        const size_t rows = (size_t)(b.max_steps + 7) / 8, nck = (size_t)(b.max_steps / bt->K[it] + 1);
        L.k.push_back(take((size_t)net->Mp * 4));
        L.draws.push_back(take(n * 4));
        L.status.push_back(take(n * 4));
        L.xfinal.push_back(take((size_t)net->N * n * 4));
        L.ev.push_back(take(rows * n * 16));
        L.ckpt.push_back(take(nck * net->N * n * 4));
        L.brk_k.push_back(take((size_t)b.n_samples * n * 4));
        L.brk_a.push_back(take((size_t)b.n_samples * n * 4));
        const bool bin = bt->readout == SSA_READOUT_BIN;
        L.brk_s.push_back(bin ? take((size_t)b.n_samples * n * 4) : 0);
        L.brk_tail.push_back(bin ? take(n * 4) : 0);
        L.prefix.push_back(bin && b.dl_traj_stride == 0 ? take((size_t)(b.n_samples + 1) * SSA_BIN_MAX_OBS * 8) : 0);
        L.dA.push_back(take((size_t)net->M * 4));
        L.n_units += units_of(bt, it);
        L.n_slots += units_of(bt, it) * net->M;
        L.n_red += net->M;
    }
    L.partial = take((size_t)L.n_slots * 4);
    L.items = take(n_items * sizeof(BatchItem));
    L.units = take((size_t)L.n_units * sizeof(BatchUnit));
    L.blk_item = take((size_t)L.n_red * 4);
    L.blk_j = take((size_t)L.n_red * 4);
    L.counters = take(64);
    L.total = off;
    return L;
}

void drop_graph(ssa_batch *bt)
{
    if (bt->graph) cudaGraphExecDestroy(bt->graph);
    bt->graph = nullptr;
}

int default_ckpt(const ssa_network *net)
{
    // checkpoints cost 4N/K bytes per draw beside the 2-byte event; K ~ 16 N keeps them near an eighth of
    // the log
    return std::min(1024, std::max(16, (16 * net->N + 7) / 8 * 8));
}

// c x the default interval, a multiple of 8 in [8, 4096]
int scaled_ckpt(const ssa_network *net, double c)
{
    const int k = (int)(c * default_ckpt(net) / 8.0 + 0.5) * 8;
    return std::min(4096, std::max(8, k));
}

}  // namespace

extern "C" ssa_status ssa_batch_create(const ssa_batch_item *items, int32_t n_items, int32_t readout,
                                       float temperature, ssa_batch **out)
{
    if (!out) return set_error(SSA_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (!items || n_items < 1) return set_error(SSA_ERR_INVALID_ARG, "no items");
    if (readout != SSA_READOUT_HOLD && readout != SSA_READOUT_LINEAR && readout != SSA_READOUT_BIN)
        return set_error(SSA_ERR_INVALID_ARG, "bad readout");
    if (!(temperature > 0.0f)) return set_error(SSA_ERR_INVALID_ARG, "temperature must be > 0");
    for (int it = 0; it < n_items; ++it) {
        const ssa_batch_item &b = items[it];
        if (!b.net || !b.log_rates || !b.x0 || b.n_traj < 0 || b.n_traj > 0x7fffffffLL || b.traj_offset < 0 ||
            b.n_samples < 0 || b.n_obs < 0 || b.n_obs > 64 || (b.n_samples > 0 && !b.sample_times) ||
            (b.n_obs > 0 && !b.obs_species) || !(b.t_end >= 0.0) || !b.dl_dlog_rates || b.max_steps < 1 ||
            b.max_steps > 0x7fffffffLL || b.ckpt_interval < 0 || (b.ckpt_interval % 8) ||
            (b.threads_per_traj != 0 && b.threads_per_traj != 1 && b.threads_per_traj != 32) || b.dl_traj_stride < 0)
            return set_error(SSA_ERR_INVALID_ARG, "invalid batch item");
        if (b.n_traj > 0 && b.n_samples > 0 && b.n_obs > 0 && (!b.obs_out || !b.dl_dobs))
            return set_error(SSA_ERR_INVALID_ARG, "batch item without outputs or upstream gradient");
        if (b.threads_per_traj == 1 && !thread_eligible(b.net))
            return set_error(SSA_ERR_UNSUPPORTED, "thread variant in a batch needs N <= 16 and M <= 16");
        if (readout == SSA_READOUT_BIN && b.n_obs > SSA_BIN_MAX_OBS)
            return set_error(SSA_ERR_UNSUPPORTED, "the bin readout takes at most SSA_BIN_MAX_OBS observables per item");
    }
    ssa_batch *bt = new (std::nothrow) ssa_batch();
    if (!bt) return set_error(SSA_ERR_CUDA, "host allocation failed");
    bt->items.assign(items, items + n_items);
    bt->readout = readout;
    bt->temperature = temperature;
    for (int it = 0; it < n_items; ++it) {
        const ssa_batch_item &b = items[it];
        int v = b.threads_per_traj;
        if (v == 0) v = thread_eligible(b.net) ? 1 : 32;
        bt->variant.push_back(v);
        bt->mc.push_back(batch_mc(b.net->M));
        bt->K.push_back(b.ckpt_interval ? b.ckpt_interval : default_ckpt(b.net));
        bt->est_draws.push_back((double)b.max_steps / 4.0);
    }
    *out = bt;
    return SSA_OK;
}

extern "C" void ssa_batch_destroy(ssa_batch *bt)
{
    if (!bt) return;
    drop_graph(bt);
    delete bt;
}

extern "C" ssa_status ssa_batch_set_plan(ssa_batch *bt, int32_t item, int32_t threads_per_traj, int32_t ckpt_interval,
                                         double est_draws)
{
    if (!bt || item < 0 || item >= (int)bt->items.size()) return set_error(SSA_ERR_INVALID_ARG, "bad item");
    if (threads_per_traj != 1 && threads_per_traj != 32) return set_error(SSA_ERR_INVALID_ARG, "threads_per_traj 1 or 32");
    if (threads_per_traj == 1 && !thread_eligible(bt->items[item].net))
        return set_error(SSA_ERR_UNSUPPORTED, "thread variant in a batch needs N <= 16 and M <= 16");
    if (threads_per_traj == 1 && bt->soft)
        return set_error(SSA_ERR_UNSUPPORTED, "a soft batch runs warp units only");
    if (ckpt_interval < 8 || ckpt_interval % 8) return set_error(SSA_ERR_INVALID_ARG, "ckpt_interval: multiple of 8");
    bt->variant[item] = threads_per_traj;
    bt->K[item] = bt->soft ? kSoftK : ckpt_interval;
    if (est_draws > 0) bt->est_draws[item] = est_draws;
    bt->ready = false;
    bt->ws = nullptr;
    drop_graph(bt);
    return SSA_OK;
}

extern "C" ssa_status ssa_batch_set_soft(ssa_batch *bt, int32_t soft)
{
    if (!bt) return set_error(SSA_ERR_INVALID_ARG, "batch is NULL");
    if (soft != 0 && soft != 1) return set_error(SSA_ERR_INVALID_ARG, "soft must be 0 or 1");
    for (size_t it = 0; soft && it < bt->items.size(); ++it)
        if (bt->items[it].threads_per_traj == 1)
            return set_error(SSA_ERR_UNSUPPORTED, "a soft batch runs warp units only (an item asks for threads_per_traj = 1)");
    bt->soft = soft != 0;
    for (size_t it = 0; it < bt->items.size(); ++it) {
        const ssa_batch_item &b = bt->items[it];
        if (bt->soft) {
            bt->variant[it] = 32;
            bt->K[it] = kSoftK;  // float checkpoints every 8 steps, re-run by the adjoint
        } else {
            bt->variant[it] = b.threads_per_traj ? b.threads_per_traj : (thread_eligible(b.net) ? 1 : 32);
            bt->K[it] = b.ckpt_interval ? b.ckpt_interval : default_ckpt(b.net);
        }
    }
    bt->ready = false;
    bt->ws = nullptr;
    drop_graph(bt);
    return SSA_OK;
}

extern "C" size_t ssa_batch_workspace_bytes(const ssa_batch *bt) { return bt ? batch_layout(bt).total : 0; }

// the adjoint kernel of a variant (soft: of the relaxed model, whose keys keep their range at every temperature)
template <int R>
static BatchAdjKernel batch_adj_of_r(int variant, bool soft, bool hot)
{
    if (variant == 1) return hot ? batch_adj_kernel<R, 1, false, true> : batch_adj_kernel<R, 1, false, false>;
    if (soft) return batch_adj_kernel<R, 32, true>;
    return hot ? batch_adj_kernel<R, 32, false, true> : batch_adj_kernel<R, 32, false, false>;
}

static const void *batch_adj_of(int readout, int variant, bool soft, bool hot)
{
    return (const void *)(readout == 0   ? batch_adj_of_r<0>(variant, soft, hot)
                          : readout == 1 ? batch_adj_of_r<1>(variant, soft, hot)
                                         : batch_adj_of_r<2>(variant, soft, hot));
}

static ssa_status batch_build(ssa_batch *bt, void *workspace, size_t bytes, cudaStream_t st)
{
    const BatchLayout L = batch_layout(bt);
    if (!workspace || bytes < L.total) return set_error(SSA_ERR_WORKSPACE, "batch workspace too small");
    if (reinterpret_cast<uintptr_t>(workspace) % 256) return set_error(SSA_ERR_WORKSPACE, "workspace not 256-byte aligned");
    unsigned char *ws = static_cast<unsigned char *>(workspace);
    const int n_items = (int)bt->items.size();
    bt->h_items.assign(n_items, BatchItem{});
    bt->d_flags = reinterpret_cast<int *>(ws + L.flags);
    float *partial = reinterpret_cast<float *>(ws + L.partial);
    int maxN = 1, maxMp = 4;
    int64_t slot_off = 0;
    for (int it = 0; it < n_items; ++it) {
        const ssa_batch_item &b = bt->items[it];
        const ssa_network *net = b.net;
        int *flag = bt->d_flags + 16 * it;
        float *k = reinterpret_cast<float *>(ws + L.k[it]);
        int *draws = reinterpret_cast<int *>(ws + L.draws[it]);
        int *status = reinterpret_cast<int *>(ws + L.status[it]);
        int *xfinal = reinterpret_cast<int *>(ws + L.xfinal[it]);
        uint4 *ev = reinterpret_cast<uint4 *>(ws + L.ev[it]);
        int *ckpt = reinterpret_cast<int *>(ws + L.ckpt[it]);
        int *brk_k = reinterpret_cast<int *>(ws + L.brk_k[it]);
        float *brk_a = reinterpret_cast<float *>(ws + L.brk_a[it]);
        const bool bin = bt->readout == SSA_READOUT_BIN;
        int *brk_s = bin ? reinterpret_cast<int *>(ws + L.brk_s[it]) : nullptr;
        int *brk_tail = bin ? reinterpret_cast<int *>(ws + L.brk_tail[it]) : nullptr;
        double *prefix = (bin && b.dl_traj_stride == 0 && b.n_samples > 0 && b.n_obs > 0)
                             ? reinterpret_cast<double *>(ws + L.prefix[it]) : nullptr;
        BatchItem &bi = bt->h_items[it];
        FwdParams &p = bi.f;
        AdjParams &a = bi.a;
        p.rx = a.rx = bt->variant[it] == 32 ? net->d_rx_warp : net->d_rx;  // warp items: lane-major tables
        p.k_rates = a.k_rates = k;
        p.tab_bytes = a.tab_bytes = net->tab_bytes;
        p.k_bytes = a.k_bytes = (uint32_t)(net->Mp * 4);
        p.N = a.N = net->N;
        p.M = a.M = net->M;
        p.Mp = a.Mp = net->Mp;
        p.inc_off = a.inc_off = net->inc_off;
        p.inc_list_off = a.inc_list_off = net->inc_list_off;
        p.nnz = a.nnz = net->nnz;
        p.n_traj = a.n_traj = b.n_traj;
        p.traj_offset = a.traj_offset = (uint64_t)b.traj_offset;
        p.seed = a.seed = b.seed;
        p.ts = a.ts = b.sample_times;
        p.S = a.S = b.n_samples;
        p.obs_sp = a.obs_sp = b.obs_species;
        p.n_obs = a.n_obs = b.n_obs;
        p.K = a.K = bt->K[it];
        p.x0 = b.x0;
        p.x0_per_traj = 0;
        p.t_end = b.t_end;
        p.max_steps = b.max_steps;
        p.obs_out = b.obs_out;
        p.draws = draws;
        p.status = status;
        p.flag = flag;
        p.err = flag + 1;
        p.ev = ev;
        p.ckpt = ckpt;
        p.brk_k = brk_k;
        p.brk_a = brk_a;
        p.brk_s = brk_s;
        p.brk_tail = brk_tail;
        p.xfinal = xfinal;
        a.draws = draws;
        a.status = status;
        a.ev = ev;
        a.ckpt = ckpt;
        a.brk_k = brk_k;
        a.brk_a = brk_a;
        a.brk_s = brk_s;
        a.brk_tail = brk_tail;
        a.bin_prefix = prefix;
        a.xfinal = xfinal;
        a.dl_dobs = b.dl_dobs;
        a.dl_stride = b.dl_traj_stride;
        a.invT = 1.0f / bt->temperature;
        p.invT = bt->soft ? a.invT : 0.0f;  // the soft forward's T is the gradient's
        p.upd = net->d_upd;
        p.upd_words = net->upd_words;
        p.wtab = a.wtab = net->d_wtab;
        p.wtab_bytes = a.wtab_bytes = net->wtab_bytes;
        a.partial = partial;
        a.mismatch = flag + 2;
        a.err = flag + 1;
        bi.variant = bt->variant[it];
        bi.mc = bt->mc[it];
        bi.slot_off = slot_off;
        bi.n_units = (int)units_of(bt, it);
        bi.log_rates = b.log_rates;
        bi.rate_index = net->d_rate_index;
        bi.P = net->P;
        bi.dtheta = b.dl_dlog_rates;
        bi.dA = reinterpret_cast<float *>(ws + L.dA[it]);
        slot_off += (int64_t)bi.n_units * net->M;
        maxN = std::max(maxN, net->N);
        maxMp = std::max(maxMp, net->Mp);
    }
    // work units, longest first by the planned cost (draws x per-draw work x trajectories per unit)
    std::vector<BatchUnit> units;
    std::vector<double> cost;
    for (int it = 0; it < n_items; ++it) {
        const int per = bt->variant[it] == 1 ? 32 : kBatchWarpUnit;
        const int M = bt->items[it].net->M;
        for (int u = 0; u < bt->h_items[it].n_units; ++u) {
            BatchUnit bu;
            bu.item = it;
            bu.traj_begin = (int64_t)u * per;
            bu.count = (int)std::min<int64_t>(per, bt->items[it].n_traj - bu.traj_begin);
            bu.slot = u;
            units.push_back(bu);
            // a thread unit runs its lanes side by side; a warp unit runs its trajectories in turn
            const double per_draw = bt->variant[it] == 1 ? (double)bt->mc[it] : (double)(M + 32) / 8.0;
            cost.push_back(bt->est_draws[it] * per_draw * (bt->variant[it] == 1 ? 1.0 : bu.count));
        }
    }
    std::vector<size_t> order(units.size());
    for (size_t q = 0; q < order.size(); ++q) order[q] = q;
    std::stable_sort(order.begin(), order.end(), [&](size_t x, size_t y) {
        const bool tx = bt->variant[units[x].item] == 1, ty = bt->variant[units[y].item] == 1;
        if (tx != ty) return tx;  // thread units first: they run in their own kernel
        return cost[x] > cost[y];
    });
    std::vector<BatchUnit> sorted(units.size());
    for (size_t q = 0; q < order.size(); ++q) sorted[q] = units[order[q]];
    std::vector<int> blk_item, blk_j;
    for (int it = 0; it < n_items; ++it)
        for (int j = 0; j < bt->items[it].net->M; ++j) {
            blk_item.push_back(it);
            blk_j.push_back(j);
        }
    bt->d_items = reinterpret_cast<BatchItem *>(ws + L.items);
    bt->d_units = reinterpret_cast<BatchUnit *>(ws + L.units);
    bt->d_blk_item = reinterpret_cast<int *>(ws + L.blk_item);
    bt->d_blk_j = reinterpret_cast<int *>(ws + L.blk_j);
    bt->d_counters = reinterpret_cast<int *>(ws + L.counters);
    CUDA_TRY_B(cudaMemcpyAsync(bt->d_items, bt->h_items.data(), n_items * sizeof(BatchItem), cudaMemcpyHostToDevice, st));
    if (!sorted.empty())
        CUDA_TRY_B(cudaMemcpyAsync(bt->d_units, sorted.data(), sorted.size() * sizeof(BatchUnit), cudaMemcpyHostToDevice, st));
    CUDA_TRY_B(cudaMemcpyAsync(bt->d_blk_item, blk_item.data(), blk_item.size() * 4, cudaMemcpyHostToDevice, st));
    CUDA_TRY_B(cudaMemcpyAsync(bt->d_blk_j, blk_j.data(), blk_j.size() * 4, cudaMemcpyHostToDevice, st));
    CUDA_TRY_B(cudaStreamSynchronize(st));  // the host vectors above go out of scope
    int n_thread_units = 0;
    for (const BatchUnit &u : sorted) n_thread_units += bt->variant[u.item] == 1;
    bt->unit_begin[0] = 0;
    bt->n_units[0] = n_thread_units;
    bt->unit_begin[1] = n_thread_units;
    bt->n_units[1] = (int)sorted.size() - n_thread_units;
    bt->n_red_blocks = (int)blk_item.size();
    int maxNw = 1, maxMpw = 4, maxMpq = 4;  // largest warp-variant network
    for (int it = 0; it < n_items; ++it)
        if (bt->variant[it] != 1) {
            maxNw = std::max(maxNw, bt->items[it].net->N);
            maxMpq = std::max(maxMpq, bt->items[it].net->Mp);
            maxMpw = std::max(maxMpw, bt->soft ? bt->items[it].net->Mp : wide_len(bt->items[it].net->M));
        }
    const int maxNpad = (maxNw + 3) & ~3;
    bt->x_words[0] = kBatchThreadMaxN * 32;
    bt->w_words[0] = 3 * kBatchThreadMaxN * 32;
    bt->x_words[1] = bt->soft ? 2 * maxNpad + maxMpw : maxNpad + maxMpw;
    bt->w_words[1] = bt->soft ? (kSoftK + 2) * maxNpad + 6 * maxMpw : 2 * maxNpad + 4 * maxMpw;
    int dev = 0, sms = 0, limit = 0;
    CUDA_TRY_B(cudaGetDevice(&dev));
    CUDA_TRY_B(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    CUDA_TRY_B(cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    const int ro = bt->readout;
    const bool sf = bt->soft;
    const void *fk[2] = {ro == 0 ? (const void *)batch_fwd_kernel<0, 1>
                                 : ro == 1 ? (const void *)batch_fwd_kernel<1, 1> : (const void *)batch_fwd_kernel<2, 1>,
                         sf ? (ro == 0 ? (const void *)batch_fwd_kernel<0, 32, true>
                                       : ro == 1 ? (const void *)batch_fwd_kernel<1, 32, true>
                                                 : (const void *)batch_fwd_kernel<2, 32, true>)
                            : (ro == 0 ? (const void *)batch_fwd_kernel<0, 32>
                                       : ro == 1 ? (const void *)batch_fwd_kernel<1, 32> : (const void *)batch_fwd_kernel<2, 32>)};
    const void *ak[2] = {batch_adj_of(ro, 1, false, bt->hot()), batch_adj_of(ro, 32, sf, bt->hot())};
    for (int v = 0; v < 2; ++v) {
        // A block of four warps, of three where the padding of the arrays by word leaves no room for four. What a batch
        // takes is set by four warps' arrays without that padding: about 7,200 species, well inside the sizes that have
        // a second table region.
        const size_t words = kItemWords + (size_t)std::max(bt->x_words[v], bt->w_words[v]);
        bt->warps[v] = kBatchWarps;
        if (v == 1 && !bt->soft)
            while (bt->warps[v] > 1 && bt->warps[v] * words * 4 > (size_t)limit) --bt->warps[v];
        bt->fwd_smem[v] = (size_t)bt->warps[v] * (kItemWords + bt->x_words[v]) * 4;
        bt->adj_smem[v] = (size_t)bt->warps[v] * (kItemWords + bt->w_words[v]) * 4;
        if (bt->n_units[v] == 0) continue;
        const size_t unpadded = kItemWords + 2 * (size_t)maxNpad + 4 * (size_t)maxMpq;
        if (bt->fwd_smem[v] > (size_t)limit || bt->adj_smem[v] > (size_t)limit ||
            (v == 1 && !bt->soft && 4 * kBatchWarps * unpadded > (size_t)limit))
            return set_error(SSA_ERR_UNSUPPORTED, "a network in the batch is too large for the batch kernels");
        int per_sm_f = 0, per_sm_a = 0;
        CUDA_TRY_B(cudaFuncSetAttribute(fk[v], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bt->fwd_smem[v]));
        CUDA_TRY_B(cudaFuncSetAttribute(ak[v], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bt->adj_smem[v]));
        CUDA_TRY_B(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_f, fk[v], 32 * bt->warps[v], bt->fwd_smem[v]));
        CUDA_TRY_B(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_a, ak[v], 32 * bt->warps[v], bt->adj_smem[v]));
        if (per_sm_f < 1 || per_sm_a < 1) return set_error(SSA_ERR_UNSUPPORTED, "batch kernels do not fit on an SM");
        // one persistent wave, never more warps than units
        const int64_t need_blocks = (bt->n_units[v] + bt->warps[v] - 1) / bt->warps[v];
        bt->fwd_blocks[v] = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * per_sm_f, need_blocks));
        bt->adj_blocks[v] = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * per_sm_a, need_blocks));
    }
    bt->ws = ws;
    bt->ready = true;
    return SSA_OK;
}

template <int R>
static void batch_launch_kernels(const ssa_batch *bt, cudaStream_t st)
{
    const BatchUnit *u0 = bt->d_units + bt->unit_begin[0], *u1 = bt->d_units + bt->unit_begin[1];
    const dim3 blk(32 * bt->warps[0]), blkw(32 * bt->warps[1]);
    if (bt->n_units[0] > 0) {  // thread units: forward then adjoint
        batch_fwd_kernel<R, 1><<<bt->fwd_blocks[0], blk, bt->fwd_smem[0], st>>>(bt->d_items, u0, bt->n_units[0],
                                                                              bt->d_counters, bt->x_words[0]);
        batch_adj_of_r<R>(1, false, bt->hot())<<<bt->adj_blocks[0], blk, bt->adj_smem[0], st>>>(bt->d_items, u0, bt->n_units[0],
                                                                              bt->d_counters + 1, bt->w_words[0]);
    }
    if (bt->n_units[1] > 0 && bt->soft) {  // warp units of a soft batch
        batch_fwd_kernel<R, 32, true><<<bt->fwd_blocks[1], blkw, bt->fwd_smem[1], st>>>(
            bt->d_items, u1, bt->n_units[1], bt->d_counters + 2, bt->x_words[1]);
        batch_adj_kernel<R, 32, true><<<bt->adj_blocks[1], blkw, bt->adj_smem[1], st>>>(
            bt->d_items, u1, bt->n_units[1], bt->d_counters + 3, bt->w_words[1]);
    } else if (bt->n_units[1] > 0) {  // warp units
        batch_fwd_kernel<R, 32><<<bt->fwd_blocks[1], blkw, bt->fwd_smem[1], st>>>(bt->d_items, u1, bt->n_units[1],
                                                                               bt->d_counters + 2, bt->x_words[1]);
        batch_adj_of_r<R>(32, false, bt->hot())<<<bt->adj_blocks[1], blkw, bt->adj_smem[1], st>>>(bt->d_items, u1, bt->n_units[1],
                                                                               bt->d_counters + 3, bt->w_words[1]);
    }
}

static ssa_status batch_enqueue(ssa_batch *bt, cudaStream_t st)
{
    const int n_items = (int)bt->items.size();
    const bool bin = bt->readout == SSA_READOUT_BIN;
    CUDA_TRY_B(cudaMemsetAsync(bt->d_flags, 0, (size_t)n_items * 16 * sizeof(int), st));
    CUDA_TRY_B(cudaMemsetAsync(bt->d_counters, 0, 64, st));
    batch_prepare_kernel<<<std::min(n_items, 1024), 128, 0, st>>>(bt->d_items, n_items, bin ? 1 : 0);
    if (bin) batch_prefix_kernel<<<std::min(n_items, 1024), kPrefixThreads, 0, st>>>(bt->d_items, n_items);
    switch (bt->readout) {
    case SSA_READOUT_HOLD: batch_launch_kernels<0>(bt, st); break;
    case SSA_READOUT_LINEAR: batch_launch_kernels<1>(bt, st); break;
    default: batch_launch_kernels<2>(bt, st); break;
    }
    if (bt->n_red_blocks > 0) batch_reduce_kernel<<<bt->n_red_blocks, 256, 0, st>>>(bt->d_items, bt->d_blk_item, bt->d_blk_j);
    batch_params_kernel<<<std::min(n_items, 1024), 128, 0, st>>>(bt->d_items, n_items);
    CUDA_TRY_B(cudaGetLastError());
    return SSA_OK;
}

extern "C" ssa_status ssa_batch_run(ssa_batch *bt, void *workspace, size_t workspace_bytes, int32_t use_graph,
                                    void *stream)
{
    if (!bt) return set_error(SSA_ERR_INVALID_ARG, "batch is NULL");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (!bt->ready || bt->ws != workspace) {
        drop_graph(bt);
        const ssa_status s = batch_build(bt, workspace, workspace_bytes, st);
        if (s != SSA_OK) return s;
    }
    if (!use_graph) return batch_enqueue(bt, st);
    if (!bt->graph) {
        if (!st) return set_error(SSA_ERR_INVALID_ARG, "graph capture needs a non-default stream");
        CUDA_TRY_B(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
        const ssa_status s = batch_enqueue(bt, st);
        cudaGraph_t g = nullptr;
        const cudaError_t e = cudaStreamEndCapture(st, &g);
        if (s != SSA_OK) {
            if (g) cudaGraphDestroy(g);
            return s;
        }
        if (e != cudaSuccess) return set_error(SSA_ERR_CUDA, cudaGetErrorString(e));
        const cudaError_t ei = cudaGraphInstantiate(&bt->graph, g, 0);
        cudaGraphDestroy(g);
        if (ei != cudaSuccess) {
            bt->graph = nullptr;
            return set_error(SSA_ERR_CUDA, cudaGetErrorString(ei));
        }
    }
    CUDA_TRY_B(cudaGraphLaunch(bt->graph, st));
    return SSA_OK;
}

extern "C" ssa_status ssa_batch_item_outputs(const ssa_batch *bt, int32_t item, int32_t *draws_out, int32_t *status_out,
                                             int64_t *host_mismatch, void *stream)
{
    if (!bt || !bt->ready || item < 0 || item >= (int)bt->items.size()) return set_error(SSA_ERR_INVALID_ARG, "bad item");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const BatchItem &b = bt->h_items[item];
    const int64_t n = b.f.n_traj;
    if (n > 0 && draws_out) CUDA_TRY_B(cudaMemcpyAsync(draws_out, b.f.draws, n * 4, cudaMemcpyDeviceToDevice, st));
    if (n > 0 && status_out) CUDA_TRY_B(cudaMemcpyAsync(status_out, b.f.status, n * 4, cudaMemcpyDeviceToDevice, st));
    if (host_mismatch) {
        int f[4];
        CUDA_TRY_B(cudaMemcpyAsync(f, b.f.flag, sizeof(f), cudaMemcpyDeviceToHost, st));
        CUDA_TRY_B(cudaStreamSynchronize(st));
        *host_mismatch = f[2];
        if (f[1] & kErrStageTimeout) return set_error(SSA_ERR_CUDA, "a kernel timed out staging its tables");
    }
    return SSA_OK;
}

extern "C" ssa_status ssa_batch_item_events(const ssa_batch *bt, int32_t item, int32_t *events_out, int64_t stride,
                                            void *stream)
{
    if (!bt || !bt->ready || item < 0 || item >= (int)bt->items.size() || !events_out || stride < 1)
        return set_error(SSA_ERR_INVALID_ARG, "bad arguments");
    if (bt->soft) return set_error(SSA_ERR_STATE, "a soft batch keeps no event log");
    const FwdParams &p = bt->h_items[item].f;
    CUDA_TRY_B(launch_unpack_events(p.ev, p.draws, p.n_traj, stride, events_out, static_cast<cudaStream_t>(stream)));
    return SSA_OK;
}

extern "C" ssa_status ssa_batch_item_brackets(const ssa_batch *bt, int32_t item, int32_t *brackets_out, void *stream)
{
    if (!bt || !bt->ready || item < 0 || item >= (int)bt->items.size()) return set_error(SSA_ERR_INVALID_ARG, "bad item");
    const FwdParams &p = bt->h_items[item].f;
    if (!brackets_out && p.n_traj > 0 && p.S > 0) return set_error(SSA_ERR_INVALID_ARG, "brackets_out is NULL");
    CUDA_TRY_B(launch_transpose_brackets(p.brk_k, p.n_traj, p.S, nullptr, nullptr, brackets_out,
                                         static_cast<cudaStream_t>(stream)));
    return SSA_OK;
}

// Pilot-based plan. Items that may run either variant (N, M <= 16 and no variant requested) time a
// pilot of `pilot_traj` trajectories through the single-network entry points (forward with record,
// then the adjoint) under both variants and keep the faster. Every item's cost estimate is the mean
// draw count of its pilot trajectories, all of which run together as one pilot batch (one persistent
// launch per direction), so the plan costs about one launch of the pilot sizes. Buffers are
// allocated once.
extern "C" ssa_status ssa_batch_autotune(ssa_batch *bt, int64_t pilot_traj, void *stream, double *host_draws_out)
{
    if (!bt || pilot_traj < 1) return set_error(SSA_ERR_INVALID_ARG, "bad batch or pilot size");
    if (bt->soft) {  // warp units and a checkpoint every 8 steps: nothing to choose
        if (host_draws_out)
            for (size_t it = 0; it < bt->items.size(); ++it) host_draws_out[it] = bt->est_draws[it];
        return SSA_OK;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t n_items = bt->items.size();
    std::vector<int64_t> np(n_items);
    size_t obs_total = 0, ws_max = 0, p_max = 1, n_max = 1;
    for (size_t it = 0; it < n_items; ++it) {
        const ssa_batch_item &b = bt->items[it];
        np[it] = std::min<int64_t>(pilot_traj, b.n_traj);
        obs_total += (size_t)np[it] * b.n_samples * b.n_obs;
        p_max = std::max(p_max, (size_t)b.net->P);
        n_max = std::max(n_max, (size_t)std::max<int64_t>(np[it], 1));
        if (!b.threads_per_traj && thread_eligible(b.net) && np[it] > 0) {
            for (int v : {1, 32}) {
                ssa_fwd_opts o{};
                o.readout = bt->readout;
                o.record = 1;
                o.ckpt_interval = bt->K[it];
                o.threads_per_traj = v;
                o.max_steps = b.max_steps;
                o.no_specialize = 1;  // the batch runs the generic kernels
                const size_t w = ssa_forward_workspace_bytes(b.net, np[it], b.n_samples, &o);
                if (w == 0) return set_error(SSA_ERR_INVALID_ARG, "pilot workspace size");
                ws_max = std::max(ws_max, w);
            }
        }
    }
    void *obs = nullptr, *dl = nullptr, *dth = nullptr, *dr = nullptr, *ws = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    ssa_status rc = SSA_OK;
    if (cudaMalloc(&obs, std::max<size_t>(obs_total, 1) * 4) != cudaSuccess ||
        cudaMalloc(&dl, std::max<size_t>(obs_total, 1) * 4) != cudaSuccess ||
        cudaMalloc(&dth, p_max * 4 * n_items) != cudaSuccess || cudaMalloc(&dr, n_max * 4) != cudaSuccess ||
        (ws_max > 0 && cudaMalloc(&ws, ws_max) != cudaSuccess) || cudaEventCreate(&e0) != cudaSuccess ||
        cudaEventCreate(&e1) != cudaSuccess)
        rc = set_error(SSA_ERR_CUDA, "pilot allocation failed");
    if (rc == SSA_OK && cudaMemsetAsync(dl, 0, std::max<size_t>(obs_total, 1) * 4, st) != cudaSuccess)
        rc = set_error(SSA_ERR_CUDA, "pilot memset failed");
    // 1. variant choice for the items that have one
    for (size_t it = 0; it < n_items && rc == SSA_OK; ++it) {
        const ssa_batch_item &b = bt->items[it];
        if (b.threads_per_traj || !thread_eligible(b.net) || np[it] == 0) continue;
        float best = -1.0f;
        for (int v : {1, 32}) {
            ssa_fwd_opts o{};
            o.readout = bt->readout;
            o.record = 1;
            o.ckpt_interval = bt->K[it];
            o.threads_per_traj = v;
            o.max_steps = b.max_steps;
            o.no_specialize = 1;
            float ms = -1.0f;
            ssa_status s = SSA_OK;
            for (int rep = 0; rep < 2 && s == SSA_OK; ++rep) {  // the first repetition warms the kernels up
                ssa_run *run = nullptr;
                cudaEventRecord(e0, st);
                s = ssa_forward(b.net, b.log_rates, np[it], b.traj_offset, b.x0, 0, b.t_end, b.sample_times,
                                b.n_samples, b.obs_species, b.n_obs, b.seed, &o, ws, ws_max, obs,
                                static_cast<int32_t *>(dr), nullptr, stream, &run);
                if (s == SSA_OK) s = ssa_backward(run, static_cast<float *>(dl), (int64_t)b.n_samples * b.n_obs,
                                                  bt->temperature, static_cast<float *>(dth), stream);
                cudaEventRecord(e1, st);
                if (run) ssa_destroy_run(run);
                if (s == SSA_OK && cudaEventSynchronize(e1) == cudaSuccess) cudaEventElapsedTime(&ms, e0, e1);
            }
            if (s != SSA_OK) {
                rc = s;
                break;
            }
            if (best < 0.0f || ms < best) {
                best = ms;
                bt->variant[it] = v;
            }
        }
    }
    // 2. cost estimates from one pilot batch under the chosen variants
    if (rc == SSA_OK) {
        std::vector<ssa_batch_item> pil(bt->items);
        size_t off = 0;
        for (size_t it = 0; it < n_items; ++it) {
            ssa_batch_item &q = pil[it];
            q.n_traj = np[it];
            q.threads_per_traj = bt->variant[it];
            q.ckpt_interval = bt->K[it];
            q.obs_out = static_cast<float *>(obs) + off;
            q.dl_dobs = static_cast<float *>(dl) + off;
            q.dl_traj_stride = (int64_t)q.n_samples * q.n_obs;
            q.dl_dlog_rates = static_cast<float *>(dth) + p_max * it;
            off += (size_t)np[it] * q.n_samples * q.n_obs;
        }
        ssa_batch *pb = nullptr;
        rc = ssa_batch_create(pil.data(), (int32_t)n_items, bt->readout, bt->temperature, &pb);
        void *pws = nullptr;
        if (rc == SSA_OK) {
            const size_t need = ssa_batch_workspace_bytes(pb);
            if (cudaMalloc(&pws, need) != cudaSuccess) rc = set_error(SSA_ERR_CUDA, "pilot batch allocation failed");
            if (rc == SSA_OK) rc = ssa_batch_run(pb, pws, need, 0, stream);
            std::vector<int> hd(n_max);
            for (size_t it = 0; it < n_items && rc == SSA_OK; ++it) {
                if (np[it] == 0) continue;
                rc = ssa_batch_item_outputs(pb, (int32_t)it, static_cast<int32_t *>(dr), nullptr, nullptr, stream);
                if (rc == SSA_OK && cudaMemcpyAsync(hd.data(), dr, (size_t)np[it] * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess)
                    rc = set_error(SSA_ERR_CUDA, "pilot copy failed");
                if (rc == SSA_OK && cudaStreamSynchronize(st) != cudaSuccess) rc = set_error(SSA_ERR_CUDA, "pilot failed");
                if (rc != SSA_OK) break;
                double sum = 0.0;
                for (int64_t k = 0; k < np[it]; ++k) sum += hd[k];
                bt->est_draws[it] = std::max(1.0, sum / (double)np[it]);
            }
        }
        if (pws) cudaFree(pws);
        ssa_batch_destroy(pb);
    }
    // 3. checkpoint interval: the reverse walk rebuilds every state exactly from the event log, so K only sets
    // how often the forward stores the state (4 N / K bytes per draw beside the 2-byte event) and the adjoint
    // checks it. Time the pilot batch with K = c x the default of each network for c in {1/4, 1, 4} (one
    // untimed and one timed launch each) and keep the fastest c.
    if (rc == SSA_OK) {
        const double scales[3] = {0.25, 1.0, 4.0};
        float best_ms = -1.0f;
        double best_c = 1.0;
        for (double c : scales) {
            std::vector<ssa_batch_item> pil(bt->items);
            size_t off = 0;
            for (size_t it = 0; it < n_items; ++it) {
                ssa_batch_item &q = pil[it];
                q.n_traj = np[it];
                q.threads_per_traj = bt->variant[it];
                q.ckpt_interval = scaled_ckpt(bt->items[it].net, c);
                q.obs_out = static_cast<float *>(obs) + off;
                q.dl_dobs = static_cast<float *>(dl) + off;
                q.dl_traj_stride = (int64_t)q.n_samples * q.n_obs;
                q.dl_dlog_rates = static_cast<float *>(dth) + p_max * it;
                off += (size_t)np[it] * q.n_samples * q.n_obs;
            }
            ssa_batch *pb = nullptr;
            rc = ssa_batch_create(pil.data(), (int32_t)n_items, bt->readout, bt->temperature, &pb);
            for (size_t it = 0; it < n_items && rc == SSA_OK; ++it)
                rc = ssa_batch_set_plan(pb, (int32_t)it, bt->variant[it], pil[it].ckpt_interval, bt->est_draws[it]);
            void *pws = nullptr;
            float ms = -1.0f;
            if (rc == SSA_OK) {
                const size_t need = ssa_batch_workspace_bytes(pb);
                if (cudaMalloc(&pws, need) != cudaSuccess) rc = set_error(SSA_ERR_CUDA, "pilot batch allocation failed");
                if (rc == SSA_OK) rc = ssa_batch_run(pb, pws, need, 0, stream);
                if (rc == SSA_OK) {
                    cudaEventRecord(e0, st);
                    rc = ssa_batch_run(pb, pws, need, 0, stream);
                    cudaEventRecord(e1, st);
                    if (rc == SSA_OK && cudaEventSynchronize(e1) == cudaSuccess) cudaEventElapsedTime(&ms, e0, e1);
                }
            }
            if (pws) cudaFree(pws);
            ssa_batch_destroy(pb);
            if (rc != SSA_OK) break;
            if (ms >= 0.0f && (best_ms < 0.0f || ms < best_ms)) {
                best_ms = ms;
                best_c = c;
            }
        }
        if (rc == SSA_OK)
            for (size_t it = 0; it < n_items; ++it)
                if (!bt->items[it].ckpt_interval) bt->K[it] = scaled_ckpt(bt->items[it].net, best_c);
        bt->ckpt_scale = best_c;
    }
    if (host_draws_out)
        for (size_t it = 0; it < n_items; ++it) host_draws_out[it] = bt->est_draws[it];
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(ws);
    cudaFree(obs);
    cudaFree(dl);
    cudaFree(dth);
    cudaFree(dr);
    bt->ready = false;
    bt->ws = nullptr;
    drop_graph(bt);
    return rc;
}

extern "C" int32_t ssa_batch_item_variant(const ssa_batch *bt, int32_t item)
{
    if (!bt || item < 0 || item >= (int)bt->items.size()) return 0;
    return bt->variant[item];
}

extern "C" int32_t ssa_batch_item_ckpt_interval(const ssa_batch *bt, int32_t item)
{
    if (!bt || item < 0 || item >= (int)bt->items.size()) return 0;
    return bt->K[item];
}
