// ssa_grn.cu -- the gene-regulatory-network classifier of arXiv 2602.19775, Section 4.3 (Figure 4A):
// n_in clamped input transcription factors x (counts round(255 p)), n_hid hidden gene products h and
// n_out output gene products y. Reactions (j < n_dyn: production of dynamic species j; j >= n_dyn:
// degradation of species j - n_dyn, with n_dyn = n_hid + n_out):
//     production of h_i:  k_max sigma(E1_i),  E1 = W1 x + b1
//     production of y_o:  k_max sigma(E2_o),  E2 = W2 h + b2
//     degradation of s:   d_s X_s,            d = exp(log_d)
// Parameters W1, b1, W2, b2, log_d (203,796 for 784 -> 256 -> 10).
//
// The dense contraction E1 = W1 x runs on the tcgen05 tensor cores, once per image. W1 (bf16) is
// split into 6-bit limbs on a common power-of-two grid; with integer counts x <= 255 every partial
// sum of one limb is an integer multiple of the limb's quantum below 2^24 quanta, so the binary32
// accumulation in TMEM is exact; the epilogue turns each accumulator into that integer and adds the limbs
// in int64 (two 42-bit halves), which is W1 x exactly, rounded once to binary64 before b1 is added. E2 = W2 h is kept exactly as an int64 fixed-point sum (bf16 W2 on its own
// grid times integer counts), updated by +-W2[:, i] when h_i changes.
//
// The SSA and the straight-through adjoint run one warp per trajectory (lanes own Philox blocks as
// in the mass-action warp kernels). With the HOLD readout the loss does not depend on event times,
// so the waiting-time path contributes nothing and the adjoint is the choice path of Eqs. 3, 5, 7.
// The backward accumulates dL/dE1 per trajectory (dW1 = G^T x follows on the tensor cores with bf16
// hi/lo limbs of G), and dW2 = sum_k G2_k h_k^T by summation by parts: with R = sum_{m >= k} G2_m
// accumulated backwards, undoing an event that changed h_i by delta adds delta R to dW2[:, i]
// (h starts at zero), so each step costs O(n_out) instead of O(n_out n_hid).
#include <algorithm>
#include <cstring>
#include <new>

#include <cuda.h>

#include "ssa_host.h"
#include "ssa_tc.cuh"
#include "ssa_warp_body.cuh"

namespace ssa {

cudaError_t launch_reduce_partials(const float *partial, int64_t nblk, int M, const int *rate_index, int P,
                                   float *dA_tmp, float *dtheta, cudaStream_t st);
cudaError_t launch_validate_inputs(const double *ts, int S, double t_end, const int *obs_sp, int n_obs, int N,
                                  int strict, int *flag, cudaStream_t st);
cudaError_t launch_column_sums(const float *x, int64_t n_rows, int64_t row_len, float *partial, int64_t chunk, float *out,
                               cudaStream_t st);

constexpr int kGrnLimbs = 8;       // 6-bit limbs of W1 on one grid: 48 bits of dynamic range
constexpr int kGrnLimbBits = 6;
constexpr int kGrnWarps = 4;       // warps per block, fewer for networks whose arrays leave no room (grn_warps)
constexpr int kGrnRegSpecies = 288;  // dynamic species up to this: the adjoint's per-species sums stay in registers

struct GrnParams {
    int n_in, n_hid, n_out, n_dyn, M, Mp, nb;
    float k_max;
    int64_t n_traj, tpi;
    uint64_t traj_offset, seed;
    const float *E1;      // [n_img][n_hid]
    const int *W2fix;     // [n_out][n_hid]: W2 = W2fix * 2^g2
    const float *W2f;     // [n_out][n_hid]
    const float4 *W2t;    // [n_dyn][ceil(n_out / 4)]: the columns of W2, padded with zeros; rows of zeros for the outputs
    const float *b2;      // [n_out]
    const float *dvec;    // [n_dyn]: d = exp(log_d)
    const int *grid;      // [0] = g2
    double t_end;
    const double *ts;
    int S;
    int64_t max_steps;
    int *obs_out;         // [n_traj][S][n_out]
    int *draws, *status;
    const int *flag;
    int *err;
    int K;
    uint4 *ev;
    int *ckpt;            // hard path: [n_ckpt][n_dyn][n_traj]
    int *brk_k;           // [S][n_traj]
    int *xfinal;          // [n_dyn][n_traj]
    // backward
    const float *dl_dobs;
    int64_t dl_stride;
    float invT;
    float *G1;            // [n_traj][n_hid]
    float *dW2t;          // [n_traj][n_out n_hid]: per-trajectory dL/dW2
    float *partial;       // [blocks][n_out + n_dyn]
    int *mismatch;
    // soft path: float checkpoints [n_traj][n_ckpt][n_dyn] (trajectory-major, one warp writes a row) and the
    // adjoint's scratch [n_traj][8][grn_soft_row]: per step of the segment being walked, its state, output
    // propensities, unnormalised soft weights and 1/Z
    int64_t n_ckpt;
    float *seg;
};

namespace {

// logistic sigma(e) in binary32 from expf and correctly rounded divisions (a few ulp)
__device__ __forceinline__ float sigmoid_f(float e)
{
    if (e >= 0.0f) return __fdiv_rn(1.0f, __fadd_rn(1.0f, expf(-e)));
    const float z = expf(e);
    return __fdiv_rn(z, __fadd_rn(1.0f, z));
}

__device__ __forceinline__ float e2_value(long long acc, float scale, float b2)
{
    return __fadd_rn(b2, __fmul_rn(__ll2float_rn(acc), scale));
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// preparation: exponent range of the weights, W1 limbs, fixed-point W2, inputs in bf16
// ---------------------------------------------------------------------------------------------
__global__ void grn_exponents_kernel(const uint16_t *W1, int64_t n1, const uint16_t *W2, int64_t n2, int *grid)
{
    // grid[0]: max exponent field of W1, grid[1]: min exponent field of nonzero W2 (bf16 fields)
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n1 + n2; q += (int64_t)gridDim.x * blockDim.x) {
        const uint16_t v = q < n1 ? W1[q] : W2[q - n1];
        const int e = (v >> 7) & 0xff;
        if (e == 0) continue;  // zero (or subnormal, treated on the slow path below)
        if (q < n1) atomicMax(&grid[0], e);
        else atomicMin(&grid[1], e);
    }
}

__device__ __forceinline__ float bf16_to_float(uint16_t v) { return __uint_as_float((uint32_t)v << 16); }

__device__ __forceinline__ uint16_t float_to_bf16_exact(float f) { return (uint16_t)(__float_as_uint(f) >> 16); }

// bf16 -> bf16 with round to nearest even (the hi/lo split of the backward)
__device__ __forceinline__ uint16_t float_to_bf16_rn(float f)
{
    const uint32_t u = __float_as_uint(f);
    return (uint16_t)((u + 0x7fffu + ((u >> 16) & 1u)) >> 16);
}

__global__ void grn_prepare_kernel(const uint16_t *W1, const uint16_t *W2, const int32_t *x_img, const float *log_d,
                                   int n_in, int n_hid, int n_out, int64_t n_img, int n_in_pad, uint16_t *W1L,
                                   int *W2fix, float *W2f, float *W2t, uint16_t *xb, float *dvec, int *grid)
{
    // W1 on the grid 2^g1, g1 = (max exponent + 1) - 48: |W1| = n 2^g1, n < 2^48, limbs of 6 bits
    const int g1 = (grid[0] - 127 + 1) - kGrnLimbBits * kGrnLimbs;
    // W2 on the grid 2^g2, g2 = (min exponent) - 7: every nonzero bf16 value is an integer multiple
    const int g2 = grid[1] - 127 - 7;
    const int64_t nW1 = (int64_t)n_hid * n_in_pad;
    const int64_t total = kGrnLimbs * nW1 + (int64_t)n_out * n_hid + n_img * n_in_pad + n_hid + n_out;
    for (int64_t qq = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; qq < total; qq += (int64_t)gridDim.x * blockDim.x) {
        int64_t q = qq;
        if (q < kGrnLimbs * nW1) {
            const int t = (int)(q / nW1);
            const int64_t r = q % nW1;
            const int h = (int)(r / n_in_pad), p = (int)(r % n_in_pad);
            float limb = 0.0f;
            if (p < n_in) {
                const float w = bf16_to_float(W1[(int64_t)h * n_in + p]);
                if (w != 0.0f) {
                    const double nd = fabs((double)w) * exp2(-(double)g1);
                    const unsigned long long nn = (unsigned long long)nd;
                    if ((double)nn != nd && t == 0) atomicOr(&grid[2], 1);  // below the grid: inexact
                    const unsigned digit = (unsigned)((nn >> (kGrnLimbBits * t)) & ((1u << kGrnLimbBits) - 1));
                    limb = (float)ldexp((double)digit, g1 + kGrnLimbBits * t) * (w < 0.0f ? -1.0f : 1.0f);
                }
            }
            W1L[q] = float_to_bf16_exact(limb);  // at most 6 significant bits: exact in bf16
            continue;
        }
        q -= kGrnLimbs * nW1;
        if (q < (int64_t)n_out * n_hid) {
            const float w = bf16_to_float(W2[q]);
            W2f[q] = w;
            W2t[(q % n_hid) * ((n_out + 3) & ~3) + q / n_hid] = w;  // the padding was cleared before
            const double nd = (double)w * exp2(-(double)g2);
            if (fabs(nd) >= 1073741824.0 || (double)(long long)nd != nd) atomicOr(&grid[2], 2);
            W2fix[q] = (int)fmax(-1073741823.0, fmin(1073741823.0, nd));
            continue;
        }
        q -= (int64_t)n_out * n_hid;
        if (q < n_img * n_in_pad) {
            const int64_t img = q / n_in_pad;
            const int p = (int)(q % n_in_pad);
            const int xv = p < n_in ? x_img[img * n_in + p] : 0;
            if (xv < 0 || xv > 256) atomicOr(&grid[2], 4);  // counts above 256 are not exact in bf16
            xb[q] = float_to_bf16_exact((float)xv);
            continue;
        }
        q -= n_img * n_in_pad;
        dvec[q] = (float)exp((double)log_d[q]);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        grid[3] = g2;
        grid[4] = g1;  // the limb grid of the tensor-core contraction's exact sum
    }
}

// ---------------------------------------------------------------------------------------------
// forward: one warp per trajectory
// ---------------------------------------------------------------------------------------------
// The warp-per-trajectory forward's step (ssa_warp_body.cuh) over propensities kept by word: those of the hidden
// productions are constant, an event changes one degradation and, for a hidden gene, the output productions. Bound
// by instruction issue: 1,620 -> 796 warp instructions per step at 784-256-10.
// W2S: W2 in shared memory; else its columns are read through L1 (networks where it leaves room for fewer warps).
template <bool W2S>
__global__ void __launch_bounds__(128, 6) grn_fwd_kernel(const GrnParams p, int record)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, W = blockDim.x >> 5;
    const int nh = p.n_hid, no = p.n_out, nd = p.n_dyn;
    int *s_W2fix = reinterpret_cast<int *>(smem);
    const int w2_words = W2S ? no * nh : 0;
    float *s_d = reinterpret_cast<float *>(s_W2fix + w2_words);
    float *s_b2 = s_d + nd;
    const int ndp = (nd + 3) & ~3, wide = wide_len(p.M), rounds = wide >> 7;
    const int nop = (no + 3) & ~3;
    const size_t per_warp = (size_t)ndp + wide + 2 * (size_t)nop;  // X, a, E2acc (2 words each)
    // offsets from the shared array itself (not through an integer round trip), so that every access below
    // compiles to a shared-memory load or store with 32-bit addressing
    unsigned char *wb = smem + ((4 * ((size_t)w2_words + nd + ((no + 3) & ~3)) + 15) & ~(size_t)15);
    int *X = reinterpret_cast<int *>(wb) + wib * per_warp;
    float *a = reinterpret_cast<float *>(X + ndp);
    long long *E2acc = reinterpret_cast<long long *>(a + wide);

    for (int q = threadIdx.x; q < w2_words; q += blockDim.x) s_W2fix[q] = p.W2fix[q];
    for (int q = threadIdx.x; q < nd; q += blockDim.x) s_d[q] = p.dvec[q];
    for (int q = threadIdx.x; q < no; q += blockDim.x) s_b2[q] = p.b2[q];
    __syncthreads();

    const int64_t i = (int64_t)blockIdx.x * W + wib;
    if (i >= p.n_traj) return;
    const int64_t n = p.n_traj;
    const float scale = exp2f((float)p.grid[0]);
    const float *E1 = p.E1 + (i / p.tpi) * nh;
    for (int s = lane; s < nd; s += 32) X[s] = 0;
    for (int q = lane; q < wide; q += 32) a[q] = 0.0f;  // every gene starts at zero: no degradation
    __syncwarp();
    for (int h = lane; h < nh; h += 32) a[h + 1] = p.k_max * sigmoid_f(E1[h]);
    for (int o = lane; o < no; o += 32) {
        E2acc[o] = 0;
        a[nh + o + 1] = p.k_max * sigmoid_f(s_b2[o]);
    }
    __syncwarp();
    const bool bad_input = (*p.flag & kErrBadSamples) != 0;
    const uint64_t gid = p.traj_offset + (uint64_t)i;
    const WarpNoise noise{(uint32_t)gid, (uint32_t)(gid >> 32), (uint32_t)p.seed, (uint32_t)(p.seed >> 32)};

    double t = 0.0;
    int s = 0;
    double thr = p.S > 0 ? p.ts[0] : p.t_end;
    int status = bad_input ? SSA_TRAJ_BAD_INPUT : SSA_TRAJ_OK;
    int k = 0, draws = 0, ck_left = p.K, ck_row = 0;
    uint32_t e0 = 0, e1 = 0, e2 = 0, e3 = 0;
    while (!bad_input) {
        if (k >= p.max_steps) { status = SSA_TRAJ_STEP_CAP; break; }
        float a0, E0;
        int jb;
        warp_step_eval(rounds, k, noise, a, a0, E0, jb);
        if (!(a0 < CUDART_INF_F)) { status = SSA_TRAJ_BAD_RATE; break; }
        if (a0 == 0.0f) { status = SSA_TRAJ_ABSORBED; break; }
        if (jb < 0) { status = SSA_TRAJ_BAD_RATE; break; }
        const float tau = waiting_time(E0, a0);
        const double t_next = t + f2d_pos(tau);
        const bool slow = gt_nonneg(t_next, thr);
        const bool cross = slow && gt_nonneg(t_next, p.t_end);
        const int sp = jb < nd ? jb : jb - nd;
        const int delta = jb < nd ? 1 : -1;
        if (!cross && delta > 0 && X[sp] == 2147483647) status = SSA_TRAJ_OVERFLOW;
        if (record) {
            e0 = __funnelshift_r(e0, e1, 16);
            e1 = __funnelshift_r(e1, e2, 16);
            e2 = __funnelshift_r(e2, e3, 16);
            e3 = (e3 >> 16) | ((uint32_t)jb << 16);
            if (lane == 0 && (k & 7) == 7) p.ev[(int64_t)(k >> 3) * n + i] = make_uint4(e0, e1, e2, e3);
        }
        draws = k + 1;
        if (status != SSA_TRAJ_OK) break;
        if (slow) {
            while (s < p.S && gt_nonneg(t_next, p.ts[s])) {
                int *o = p.obs_out + ((int64_t)i * p.S + s) * no;
                for (int c = lane; c < no; c += 32) o[c] = X[nh + c];
                if (record && lane == 0) p.brk_k[(int64_t)s * n + i] = k;
                ++s;
            }
            thr = s < p.S ? p.ts[s] : p.t_end;
            if (cross) break;
        }
        __syncwarp();
        if (lane == 0) {
            const int x = X[sp] + delta;
            X[sp] = x;
            a[nd + sp + 1] = __fmul_rn(s_d[sp], int2f(x));
        }
        if (sp < nh) {
            for (int o = lane; o < no; o += 32) {
                E2acc[o] += (long long)delta * (W2S ? s_W2fix[o * nh + sp] : __ldg(p.W2fix + o * nh + sp));
                a[nh + o + 1] = p.k_max * sigmoid_f(e2_value(E2acc[o], scale, s_b2[o]));
            }
        }
        __syncwarp();
        t = t_next;
        ++k;
        if (record && --ck_left == 0) {
            ck_left = p.K;
            ++ck_row;
            int *ck = p.ckpt + (int64_t)ck_row * nd * n + i;
            for (int q = lane; q < nd; q += 32) ck[(int64_t)q * n] = X[q];
        }
    }
    __syncwarp();
    for (; s < p.S; ++s) {
        int *o = p.obs_out + ((int64_t)i * p.S + s) * no;
        for (int c = lane; c < no; c += 32) o[c] = X[nh + c];
        if (record && lane == 0) p.brk_k[(int64_t)s * n + i] = k;
    }
    if (lane == 0) {
        p.draws[i] = draws;
        p.status[i] = status;
    }
    if (record) {
        if ((draws & 7) && lane == 0) {
            for (int pad = draws & 7; pad < 8; ++pad) {
                e0 = __funnelshift_r(e0, e1, 16);
                e1 = __funnelshift_r(e1, e2, 16);
                e2 = __funnelshift_r(e2, e3, 16);
                e3 = e3 >> 16;
            }
            p.ev[(int64_t)((draws - 1) >> 3) * n + i] = make_uint4(e0, e1, e2, e3);
        }
        for (int q = lane; q < nd; q += 32) {
            p.xfinal[(int64_t)q * n + i] = X[q];
            p.ckpt[(int64_t)q * n + i] = 0;  // checkpoint 0: every gene starts at zero
        }
    }
}

// ---------------------------------------------------------------------------------------------
// soft forward (Section 3.3, Eq. 4; the first training phase of Section 3.5): one warp per trajectory and
// real-valued counts. Every step all reactions enter the soft sample y~ = softmax((log a + G)/T) of the same
// Gumbel noise, and every count moves by its expected change y~_prod - y~_deg; a negative count degrades at
// rate 0. E2 = W2 h + b2 is recomputed from the relaxed hidden counts (binary32 W2). The step is one shared
// routine, so the adjoint's re-runs from the float checkpoints reproduce the forward's states bit for bit.
// ---------------------------------------------------------------------------------------------
namespace {

constexpr int kGrnSoftK = 8;  // float checkpoints of the soft forward every 8 steps

// Propensities and keys lie by word (index j + 1), as in the exact path. Per step at 784-256-10: ~1,200 warp
// instructions; with an accurate logarithm of every variate and two accurate log2 of every key, and the outputs'
// sigmoids evaluated one lane at a time, ~3,300.

// output propensities k_max sigma(W2 h + b2) of the relaxed state X (the warp's lanes cooperate); aO: a + nh + 1
__device__ __forceinline__ void grn_soft_outputs(const GrnParams &p, const float *s_W2, const float *s_b2,
                                                 const float *X, float *aO, int lane)
{
    const int nh = p.n_hid, no = p.n_out;
    for (int o0 = 0; o0 < no; o0 += 32) {  // up to 32 outputs, then one sigmoid per lane
        float mine = 0.0f;
        for (int o = o0; o < min(no, o0 + 32); ++o) {
            float part = 0.0f;
#pragma unroll 8
            for (int h = lane; h < nh; h += 32) part = __fmaf_rn(s_W2[(size_t)o * nh + h], X[h], part);
            const float sum = warp_sum(part);
            if (lane == o - o0) mine = sum;
        }
        if (o0 + lane < no) aO[o0 + lane] = p.k_max * sigmoid_f(__fadd_rn(mine, s_b2[o0 + lane]));
    }
    __syncwarp();
}

// one soft step at step k from the propensities a: the race's keys a_j / E_j, then the unnormalised weights
// q_j = (key_j / largest)^(1/T) in their place; returns a0 and sets E0 and invZ = 1/sum q
template <bool HOT>
__device__ __forceinline__ float grn_soft_weights(const GrnParams &p, const float *a, float *key, int k,
                                                  const WarpNoise &z, int lane, float &E0, float &invZ)
{
    const int rounds = wide_len(p.M) >> 7;
    const float4 *a4 = reinterpret_cast<const float4 *>(a);
    float4 *key4 = reinterpret_cast<float4 *>(key);
    float a0p = 0.0f, rmax = 0.0f;
    uint32_t x0 = 0;
    for (int c = 0; c < rounds; ++c) {
        const int b = 32 * c + lane;
        const uint4 r = philox4x32_10(make_uint4((uint32_t)b, (uint32_t)k, z.c2, z.c3), z.key0, z.key1);
        if (c == 0) x0 = r.x;
        const float4 av = a4[b];  // the waiting-time word's and the padded ones are 0
        a0p = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(a0p, av.x), av.y), av.z), av.w);
        const float4 kv = make_float4(av.x * inv_exp_of_word(r.x), av.y * inv_exp_of_word(r.y),
                                      av.z * inv_exp_of_word(r.z), av.w * inv_exp_of_word(r.w));
        rmax = fmaxf(rmax, fmaxf(fmaxf(kv.x, kv.y), fmaxf(kv.z, kv.w)));
        key4[b] = kv;
    }
    const float a0 = warp_sum(a0p);
    rmax = warp_max_nonneg(rmax);
    E0 = neg_log_unit(u01(__shfl_sync(0xffffffffu, x0, 0)));
    if (HOT || !(a0 >= 0x1p-60f && a0 <= 0x1p100f)) rmax = warp_keys_scaled(rounds, a, k, z, a0, HOT, key);
    const float invT_q = HOT ? 8.0f * p.invT : p.invT;
    const KeyTop top = key_top(rmax);
    float Zp = 0.0f;
    for (int c = 0; c < rounds; ++c) {
        const float4 kv = key4[32 * c + lane];
        auto weight = [&](float v) { return ex2_approx(top.lg2(v) * invT_q); };
        const float4 q = make_float4(weight(kv.x), weight(kv.y), weight(kv.z), weight(kv.w));
        key4[32 * c + lane] = q;
        Zp += (q.x + q.y) + (q.z + q.w);
    }
    invZ = __fdividef(1.0f, warp_sum(Zp));
    __syncwarp();
    return a0;
}

// the relaxed update X += y~_prod - y~_deg for every dynamic species, and its degradation's propensity
__device__ __forceinline__ void grn_soft_update(const GrnParams &p, const float *s_d, float *X, float *a, const float *q,
                                                float invZ, int lane)
{
    const int nd = p.n_dyn;
    for (int u = lane; u < nd; u += 32) {
        const float x = __fadd_rn(X[u], (q[u + 1] - q[nd + u + 1]) * invZ);
        X[u] = x;
        a[nd + u + 1] = __fmul_rn(s_d[u], fmaxf(x, 0.0f));
    }
    __syncwarp();
}

}  // namespace

template <bool HOT>
__global__ void __launch_bounds__(128) grn_soft_fwd_kernel(const GrnParams p, float *obs, int record)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, W = blockDim.x >> 5;
    const int nh = p.n_hid, no = p.n_out, nd = p.n_dyn;
    const int ndp = (nd + 3) & ~3, nop = (no + 3) & ~3, wide = wide_len(p.M);
    float *s_W2 = reinterpret_cast<float *>(smem);  // [no][nh]
    float *s_d = s_W2 + (size_t)no * nh;            // [nd]
    float *s_b2 = s_d + nd;                         // [no]
    float *X = reinterpret_cast<float *>(smem + ((4 * ((size_t)no * nh + nd + nop) + 15) & ~(size_t)15)) +
               (size_t)wib * (ndp + 2 * wide);
    float *a = X + ndp;    // propensities by word
    float *q = a + wide;   // keys, then unnormalised soft weights
    float *aO = a + nh + 1;
    for (int u = threadIdx.x; u < no * nh; u += blockDim.x) s_W2[u] = p.W2f[u];
    for (int u = threadIdx.x; u < nd; u += blockDim.x) s_d[u] = p.dvec[u];
    for (int u = threadIdx.x; u < no; u += blockDim.x) s_b2[u] = p.b2[u];
    __syncthreads();

    const int64_t i = (int64_t)blockIdx.x * W + wib;
    if (i >= p.n_traj) return;
    const int64_t n = p.n_traj;
    float *ckf = reinterpret_cast<float *>(p.ckpt);
    const float *E1 = p.E1 + (i / p.tpi) * nh;
    for (int u = lane; u < nd; u += 32) X[u] = 0.0f;
    for (int u = lane; u < wide; u += 32) a[u] = 0.0f;
    __syncwarp();
    for (int h = lane; h < nh; h += 32) a[h + 1] = p.k_max * sigmoid_f(E1[h]);  // constant per image
    __syncwarp();
    grn_soft_outputs(p, s_W2, s_b2, X, aO, lane);
    const bool bad_input = (*p.flag & kErrBadSamples) != 0;
    const uint64_t gid = p.traj_offset + (uint64_t)i;
    const WarpNoise noise{(uint32_t)gid, (uint32_t)(gid >> 32), (uint32_t)p.seed, (uint32_t)(p.seed >> 32)};

    double t = 0.0;
    int s = 0;
    double thr = p.S > 0 ? p.ts[0] : p.t_end;
    int status = bad_input ? SSA_TRAJ_BAD_INPUT : SSA_TRAJ_OK;
    int k = 0, draws = 0, ck_left = kGrnSoftK, ck_row = 0;
    while (!bad_input) {
        if (k >= p.max_steps) { status = SSA_TRAJ_STEP_CAP; break; }
        float E0, invZ;
        const float a0 = grn_soft_weights<HOT>(p, a, q, k, noise, lane, E0, invZ);
        if (!(a0 < CUDART_INF_F)) { status = SSA_TRAJ_BAD_RATE; break; }
        if (a0 == 0.0f) { status = SSA_TRAJ_ABSORBED; break; }
        const float tau = waiting_time(E0, a0);
        const double t_next = t + f2d_pos(tau);
        const bool slow = gt_nonneg(t_next, thr);
        const bool cross = slow && gt_nonneg(t_next, p.t_end);
        draws = k + 1;
        if (slow) {
            while (s < p.S && gt_nonneg(t_next, p.ts[s])) {
                float *o = obs + ((int64_t)i * p.S + s) * no;
                for (int c = lane; c < no; c += 32) o[c] = X[nh + c];
                if (record && lane == 0) p.brk_k[(int64_t)s * n + i] = k;
                ++s;
            }
            thr = s < p.S ? p.ts[s] : p.t_end;
            if (cross) break;
        }
        grn_soft_update(p, s_d, X, a, q, invZ, lane);
        grn_soft_outputs(p, s_W2, s_b2, X, aO, lane);
        t = t_next;
        ++k;
        if (record && --ck_left == 0) {
            ck_left = kGrnSoftK;
            ++ck_row;
            for (int u = lane; u < nd; u += 32) ckf[((int64_t)i * p.n_ckpt + ck_row) * nd + u] = X[u];
        }
    }
    __syncwarp();
    for (; s < p.S; ++s) {
        float *o = obs + ((int64_t)i * p.S + s) * no;
        for (int c = lane; c < no; c += 32) o[c] = X[nh + c];
        if (record && lane == 0) p.brk_k[(int64_t)s * n + i] = k;
    }
    if (lane == 0) {
        p.draws[i] = draws;
        p.status[i] = status;
    }
    if (record)
        for (int u = lane; u < nd; u += 32) ckf[(int64_t)i * p.n_ckpt * nd + u] = 0.0f;  // checkpoint 0: all at zero
}

// ---------------------------------------------------------------------------------------------
// soft adjoint: the exact gradient of the relaxed model (the straight-through adjoint's arithmetic along
// the soft path). Per 8-step segment the forward's own step routines re-run the states from their float
// checkpoint (the end must equal the next checkpoint bit for bit) and leave, per step, the state, the output
// propensities, the unnormalised soft weights and 1/Z in the trajectory's row of a global scratch; the walk
// back reads them instead of drawing the step again. In the relaxed model every hidden count changes every
// step, so dL/dW2 = sum_k G2_k h_k^T takes a rank-8 update of the trajectory's dW2 row once per segment.
// Shared memory holds W2 per block and ~8 KB per warp.
// ---------------------------------------------------------------------------------------------
namespace {

// one step's row of the soft adjoint's segment scratch: X [ndp] | aO [nop] | q [Mq] | 1/Z and padding [4]
__host__ __device__ inline int grn_soft_row(int nd, int no, int M)
{
    return ((nd + 3) & ~3) + ((no + 3) & ~3) + ((M + 3) & ~3) + 4;
}

// words of one warp's arrays in the soft adjoint: X, a, key, lam, dlogd, 1 - sigma(E1), G1, db2, G2 of a segment
__host__ __device__ inline size_t grn_soft_adj_words(int nh, int no)
{
    const int nd = nh + no, ndp = (nd + 3) & ~3, nhp = (nh + 3) & ~3, nop = (no + 3) & ~3;
    return 3 * (size_t)ndp + 2 * (size_t)wide_len(2 * nd) + 2 * (size_t)nhp + (1 + kGrnSoftK) * (size_t)nop;
}

}  // namespace

// NS rounds of species (n_dyn <= 32 NS) read a step's weights and state into registers together, one wait for memory a
// step; NS = 0: any number, read where they are used.
template <int NS, bool HOT>
__global__ void __launch_bounds__(128, 4) grn_soft_adj_kernel(const GrnParams p)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, W = blockDim.x >> 5;
    const int nh = p.n_hid, no = p.n_out, nd = p.n_dyn, M = p.M;
    const int ndp = (nd + 3) & ~3, nhp = (nh + 3) & ~3, nop = (no + 3) & ~3, Mq = (M + 3) & ~3, wide = wide_len(M);
    const int RS = grn_soft_row(nd, no, M);
    float *s_W2 = reinterpret_cast<float *>(smem);
    float *s_d = s_W2 + (size_t)no * nh;
    float *s_b2 = s_d + nd;
    const size_t per_warp = grn_soft_adj_words(nh, no);
    float *base0 = reinterpret_cast<float *>(smem + ((4 * ((size_t)no * nh + nd + nop) + 15) & ~(size_t)15));
    float *X = base0 + (size_t)wib * per_warp;       // the state being stepped or differentiated
    float *a = X + ndp;                               // propensities by word
    float *q = a + wide;                              // keys, then unnormalised weights, by word
    float *lam = q + wide;                            // dL/dX of the state after the step
    float *dlogd = lam + ndp;
    float *cH = dlogd + ndp;                          // 1 - sigma(E1)
    float *G1 = cH + nhp;
    float *db2 = G1 + nhp;
    float *G2h = db2 + nop;                           // [kGrnSoftK][nop]: dL/dE2 of the segment's steps
    float *aO = a + nh + 1;
    for (int u = threadIdx.x; u < no * nh; u += blockDim.x) s_W2[u] = p.W2f[u];
    for (int u = threadIdx.x; u < nd; u += blockDim.x) s_d[u] = p.dvec[u];
    for (int u = threadIdx.x; u < no; u += blockDim.x) s_b2[u] = p.b2[u];
    for (int u = lane; u < nd; u += 32) dlogd[u] = 0.0f;
    for (int u = lane; u < no; u += 32) db2[u] = 0.0f;
    __syncthreads();

    const int64_t n = p.n_traj;
    const int64_t i = (int64_t)blockIdx.x * W + wib;
    int st = -1;
    if (i < n) st = p.status[i];
    const bool active = st == SSA_TRAJ_OK || st == SSA_TRAJ_ABSORBED || st == SSA_TRAJ_STEP_CAP;
    if (i < n) {  // zeroed with the lane mapping of the per-segment updates
        float *dW2 = p.dW2t + i * (int64_t)no * nh;
        for (int h = lane; h < nh; h += 32)
            for (int o = 0; o < no; ++o) dW2[(size_t)o * nh + h] = 0.0f;
        if (!active)
            for (int h = lane; h < nh; h += 32) p.G1[i * nh + h] = 0.0f;
    }
    if (active) {
        const float *ckf = reinterpret_cast<const float *>(p.ckpt) + i * p.n_ckpt * nd;
        float *seg = p.seg + i * (int64_t)kGrnSoftK * RS;
        float *dW2 = p.dW2t + i * (int64_t)no * nh;
        const float *E1 = p.E1 + (i / p.tpi) * nh;
        const int d = p.draws[i];
        // a finished run's last draw is the crossing one, which moves no observed state
        const int L = (st == SSA_TRAJ_OK) ? d - 1 : d;
        for (int u = lane; u < nd; u += 32) lam[u] = 0.0f;
        for (int u = lane; u < wide; u += 32) a[u] = 0.0f;
        for (int u = lane; u < kGrnSoftK * nop; u += 32) G2h[u] = 0.0f;
        __syncwarp();
        const float inv_kmax = 1.0f / p.k_max;
        for (int h = lane; h < nh; h += 32) {
            a[h + 1] = p.k_max * sigmoid_f(E1[h]);
            cH[h] = 1.0f - a[h + 1] * inv_kmax;
            G1[h] = 0.0f;
        }
        __syncwarp();
        const uint64_t gid = p.traj_offset + (uint64_t)i;
        const WarpNoise noise{(uint32_t)gid, (uint32_t)(gid >> 32), (uint32_t)p.seed, (uint32_t)(p.seed >> 32)};
        const float invT = p.invT;
        const float *gl = p.dl_dobs + i * p.dl_stride;
        int s_hi = p.S - 1;
        int brk_next = s_hi >= 0 ? p.brk_k[(int64_t)s_hi * n + i] : -1;
        int mism = 0;
        for (int c = L / kGrnSoftK; c >= 0; --c) {
            const int k0 = c * kGrnSoftK, k1 = min(k0 + kGrnSoftK - 1, L);
            for (int u = lane; u < nd; u += 32) {
                const float x = ckf[(int64_t)c * nd + u];
                X[u] = x;
                a[nd + u + 1] = __fmul_rn(s_d[u], fmaxf(x, 0.0f));
            }
            __syncwarp();
            for (int kk = k0; kk <= k1; ++kk) {  // re-run the segment with the forward's routines
                float *row = seg + (kk - k0) * RS;
                for (int u = lane; u < nd; u += 32) row[u] = X[u];
                if (kk < L) {
                    grn_soft_outputs(p, s_W2, s_b2, X, aO, lane);
                    float E0, invZ;
                    grn_soft_weights<HOT>(p, a, q, kk, noise, lane, E0, invZ);
                    for (int o = lane; o < no; o += 32) row[ndp + o] = aO[o];
                    for (int j = lane; j < M; j += 32) row[ndp + nop + j] = q[j + 1];
                    if (lane == 0) row[ndp + nop + Mq] = invZ;
                    grn_soft_update(p, s_d, X, a, q, invZ, lane);
                }
            }
            if (k1 < L) {
                int bad = 0;
                for (int u = lane; u < nd; u += 32) bad += X[u] != ckf[(int64_t)(c + 1) * nd + u];
                mism += __reduce_add_sync(0xffffffffu, bad);
            }
            __syncwarp();  // the scratch rows were written lane-strided; the walk reads them across lanes
            for (int k = k1; k >= k0; --k) {
                const float *row = seg + (k - k0) * RS;
                float *G2 = G2h + (k - k0) * nop;
                for (int o = lane; o < no; o += 32) G2[o] = 0.0f;
                const int s_top = s_hi;
                while (s_hi >= 0 && brk_next == k) {
                    --s_hi;
                    brk_next = s_hi >= 0 ? p.brk_k[(int64_t)s_hi * n + i] : -1;
                }
                if (k < L) {
                    const float invZ = row[ndp + nop + Mq];
                    const float *qrow = row + ndp + nop;
                    // W = sum_j q_j w_j / Z with w_j = +lam_s (production) or -lam_s (degradation); a lane takes both
                    // reactions of its species
                    float Wp = 0.0f;
                    constexpr int NR = NS > 0 ? NS : 1;
                    float qpr[NR], qdr[NR], xr[NR];
                    if constexpr (NS > 0) {
#pragma unroll
                        for (int c2 = 0; c2 < NS; ++c2) {
                            const int u = min(32 * c2 + lane, nd - 1);
                            qpr[c2] = qrow[u];
                            qdr[c2] = qrow[nd + u];
                            xr[c2] = row[u];
                        }
#pragma unroll
                        for (int c2 = 0; c2 < NS; ++c2)
                            if (32 * c2 + lane < nd) Wp = fmaf(qpr[c2] - qdr[c2], lam[32 * c2 + lane], Wp);
                    } else {
                        for (int u = lane; u < nd; u += 32) Wp = fmaf(qrow[u] - qrow[nd + u], lam[u], Wp);
                    }
                    const float Wbar = warp_sum(Wp) * invZ, scale = invZ * invT;
                    // choice-path adjoints psi_j = dL/dlog a_j (HOLD readout: no waiting-time path), the outputs first
                    for (int o = lane; o < no; o += 32) {
                        const float qp = qrow[nh + o], psi = qp * scale * (lam[nh + o] - Wbar);
                        G2[o] = (qp > 0.0f ? psi : 0.0f) * (1.0f - row[ndp + o] * inv_kmax);
                    }
                    __syncwarp();
                    // the degradations: psi of d_u max(X_u, 0); a weight q > 0 implies a > 0, so X_u > 0 there
                    auto species = [&](int u, float qp, float qd, float x) {
                        const float l = lam[u];
                        float psi = qd * scale * (-l - Wbar);
                        psi = qd > 0.0f ? psi : 0.0f;
                        dlogd[u] += psi;
                        float acc = __fdividef(psi, x);
                        acc = qd > 0.0f ? acc : 0.0f;
                        if (u < nh) {
                            const float psi_p = qp * scale * (l - Wbar);
                            G1[u] += (qp > 0.0f ? psi_p : 0.0f) * cH[u];
                            const float4 *w = p.W2t + (int64_t)u * (nop >> 2), *g = reinterpret_cast<const float4 *>(G2);
                            for (int v = 0; v < nop >> 2; ++v) {  // in output order; the padding adds 0
                                const float4 wv = __ldg(w + v), gv = g[v];
                                acc = fmaf(wv.w, gv.w, fmaf(wv.z, gv.z, fmaf(wv.y, gv.y, fmaf(wv.x, gv.x, acc))));
                            }
                        }
                        lam[u] = l + acc;
                    };
                    if constexpr (NS > 0) {
#pragma unroll
                        for (int c2 = 0; c2 < NS; ++c2)
                            if (32 * c2 + lane < nd) species(32 * c2 + lane, qpr[c2], qdr[c2], xr[c2]);
                    } else {
                        for (int u = lane; u < nd; u += 32) species(u, qrow[u], qrow[nd + u], row[u]);
                    }
                }
                __syncwarp();
                // HOLD samples of the outputs at state k
                for (int s = s_hi + 1; s <= s_top; ++s)
                    for (int o = lane; o < no; o += 32) lam[nh + o] += gl[(int64_t)s * no + o];
                __syncwarp();
            }
            // the segment's rank-(k1 - k0 + 1) update of dL/dW2 and dL/db2
            const int len = k1 - k0 + 1;
            for (int h = lane; h < nh; h += 32) {
                float xs[kGrnSoftK];
#pragma unroll
                for (int r = 0; r < kGrnSoftK; ++r) xs[r] = r < len ? seg[r * RS + h] : 0.0f;
                for (int o = 0; o < no; ++o) {
                    // rows past the segment's end carry 0; added without waiting for memory (one lane's adds to a place
                    // keep their order)
                    float acc = 0.0f;
#pragma unroll
                    for (int r = 0; r < kGrnSoftK; ++r) acc = __fmaf_rn(G2h[r * nop + o], xs[r], acc);
                    atomicAdd(dW2 + (size_t)o * nh + h, acc);
                }
            }
            for (int o = lane; o < no; o += 32)
                for (int r = 0; r < len; ++r) db2[o] += G2h[r * nop + o];
            __syncwarp();
        }
        for (int h = lane; h < nh; h += 32) p.G1[i * nh + h] = G1[h];
        if (lane == 0 && mism) atomicAdd(p.mismatch, mism);
    }
    __syncthreads();
    // fixed-order sum over the block's warps: [db2 | dlogd]
    const int red = no + nd;
    for (int u = threadIdx.x; u < red; u += blockDim.x) {
        float acc = 0.0f;
        for (int w = 0; w < W; ++w) {
            const float *wp = base0 + w * per_warp;
            acc += u < no ? wp[3 * ndp + 2 * wide + 2 * nhp + u] : wp[2 * ndp + 2 * wide + (u - no)];
        }
        p.partial[(int64_t)blockIdx.x * red + u] = acc;
    }
}

// ---------------------------------------------------------------------------------------------
// backward: one warp per trajectory, reverse walk
// ---------------------------------------------------------------------------------------------
// words of one warp's arrays in the adjoint (grn_adj_kernel)
__host__ __device__ inline size_t grn_adj_words(int nh, int no, bool shared_sums)
{
    const int nd = nh + no, ndp = (nd + 3) & ~3, nop = (no + 3) & ~3;
    return 2 * (size_t)wide_len(2 * nd) + 2 * ndp + 6 * (size_t)nop + (shared_sums ? 3 * (size_t)ndp : 0);
}

// Per step: pass 1, by Philox block, forms the race's keys a_j / E_j from the kept propensities; pass 2, by species
// (a lane's species s = lane, lane + 32, ... with their productions and degradations), the soft weights and their
// moment with lambda; pass 3, by species again, psi of both reactions and the state adjoint. With NS rounds of
// species (n_dyn <= 32 NS) lambda, dL/dE1 and dL/dlog d live in registers; NS = 0 keeps them in shared memory.
// Bound by instruction issue; 784-256-10: 4,280 -> 1,610 warp instructions per step, a training step of 48 x 64
// trajectories 127 -> 63 ms with the forward. Four resident blocks (128 registers): 63 ms; five 75, six 70 (spills),
// six with the sums in shared memory 77.
constexpr int kGrnAdjBlocks = 4;
// NF: the first rounds of species that are full (n_dyn >= 32 NF).
template <int NS, int NF, bool HOT>
__global__ void __launch_bounds__(128, kGrnAdjBlocks) grn_adj_kernel(const GrnParams p)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, W = blockDim.x >> 5;
    const int nh = p.n_hid, no = p.n_out, nd = p.n_dyn;
    float *s_d = reinterpret_cast<float *>(smem);
    float *s_b2 = s_d + nd;
    const int ndp = (nd + 3) & ~3, nop = (no + 3) & ~3, wide = wide_len(p.M), rounds = wide >> 7;
    const int ns = NS > 0 ? NS : (nd + 31) >> 5;  // rounds of species
    // per warp (words): a, key [wide each], X [ndp], 1 - sigma(E1), 0 for the outputs
    // [ndp], E2acc [2 nop], 1 - sigma(E2), G2, R, db2
    // [nop each]; NS = 0 also lam, G1, dlogd [ndp]. dL/dW2 goes to the trajectory's own row of p.dW2t
    // (global, L2-resident while the warp works on it).
    const size_t per_warp = grn_adj_words(nh, no, NS == 0);
    unsigned char *wb = smem + ((4 * ((size_t)nd + nop) + 15) & ~(size_t)15);  // shared-space offsets (see the forward)
    float *wbase = reinterpret_cast<float *>(wb) + wib * per_warp;
    float *a = wbase;
    float *key = a + wide;
    int *X = reinterpret_cast<int *>(key + wide);
    float *cH = reinterpret_cast<float *>(X + ndp);
    long long *E2acc = reinterpret_cast<long long *>(cH + ndp);
    float *cO = reinterpret_cast<float *>(E2acc + nop);
    float *G2 = cO + nop;
    float *R = G2 + nop;
    float *db2 = R + nop;
    float *lam_s = db2 + nop, *G1_s = lam_s + ndp, *dlogd_s = G1_s + ndp;
    const int *__restrict__ W2fix = p.W2fix;
    const float4 *__restrict__ W2t = p.W2t;

    for (int q = threadIdx.x; q < nd; q += blockDim.x) s_d[q] = p.dvec[q];
    for (int q = threadIdx.x; q < no; q += blockDim.x) s_b2[q] = p.b2[q];
    for (int q = lane; q < wide; q += 32) key[q] = 0.0f;
    for (int q = lane; q < nop; q += 32) db2[q] = G2[q] = 0.0f;
    __syncthreads();

    const int64_t n = p.n_traj;
    const int64_t i = (int64_t)blockIdx.x * W + wib;
    int st = -1;
    if (i < n) st = p.status[i];
    const bool active = st == SSA_TRAJ_OK || st == SSA_TRAJ_ABSORBED || st == SSA_TRAJ_STEP_CAP;
    float *dW2 = p.dW2t + (i < n ? i : 0) * (int64_t)no * nh;
    if (i < n)
        for (int q = lane; q < no * nh; q += 32) dW2[q] = 0.0f;
    float lam_r[NS > 0 ? NS : 1], G1_r[NS > 0 ? NS : 1], dlogd_r[NS > 0 ? NS : 1];
    auto lam = [&](int c) -> float & { return NS > 0 ? lam_r[NS > 0 ? c : 0] : lam_s[32 * c + lane]; };
    auto G1 = [&](int c) -> float & { return NS > 0 ? G1_r[NS > 0 ? c : 0] : G1_s[32 * c + lane]; };
    auto dlogd = [&](int c) -> float & { return NS > 0 ? dlogd_r[NS > 0 ? c : 0] : dlogd_s[32 * c + lane]; };
    auto each_species = [&](auto body) {  // body(c, s) for this lane's species s = 32 c + lane below n_dyn
#pragma unroll (NS > 0 ? NS : 1)
        for (int c = 0; c < ns; ++c) {
            const int s = 32 * c + lane;
            if (c < NF) body(c, s);
            else if (s < nd) body(c, s);
        }
    };
    if (active) {
        const float scale = exp2f((float)p.grid[0]);
        const float inv_kmax = 1.0f / p.k_max;
        const float *E1 = p.E1 + (i / p.tpi) * nh;
        const int d = p.draws[i];
        const int L = (st == SSA_TRAJ_OK) ? d - 1 : d;
        for (int q = lane; q < wide; q += 32) a[q] = 0.0f;
        __syncwarp();
        each_species([&](int c, int s) {
            const int x = p.xfinal[(int64_t)s * n + i];
            X[s] = x;
            a[nd + s + 1] = __fmul_rn(s_d[s], int2f(x));
            lam(c) = 0.0f;
            dlogd(c) = 0.0f;
            G1(c) = 0.0f;
            cH[s] = 0.0f;  // the outputs take no part in dL/dE1
            if (s < nh) {
                const float ah = p.k_max * sigmoid_f(E1[s]);
                a[s + 1] = ah;
                cH[s] = 1.0f - ah * inv_kmax;  // d log(k_max sigma(E)) / dE = 1 - sigma(E)
            }
        });
        __syncwarp();
        // E2 at the final state, exactly (integer fixed point)
        auto set_output = [&](int o) {
            const float ao = p.k_max * sigmoid_f(e2_value(E2acc[o], scale, s_b2[o]));
            a[nh + o + 1] = ao;
            cO[o] = 1.0f - ao * inv_kmax;
        };
        for (int o = lane; o < no; o += 32) {
            long long acc = 0;
            for (int h = 0; h < nh; ++h) acc += (long long)__ldg(W2fix + o * nh + h) * X[h];
            E2acc[o] = acc;
            set_output(o);
            R[o] = 0.0f;
        }
        __syncwarp();
        const uint64_t gid = p.traj_offset + (uint64_t)i;
        const WarpNoise noise{(uint32_t)gid, (uint32_t)(gid >> 32), (uint32_t)p.seed, (uint32_t)(p.seed >> 32)};
        const float invT = p.invT, invT_q = HOT ? weight_factor(8.0f * invT) : invT;
        const float *gl = p.dl_dobs + i * p.dl_stride;
        int row_cached = -1;
        uint4 row = make_uint4(0, 0, 0, 0), row_below = row;  // the log row below is loaded ahead of its use
        auto event_at = [&](int kk) -> int {
            const int r = kk >> 3;
            if (r != row_cached) {
                row = (r == row_cached - 1) ? row_below : p.ev[(int64_t)r * n + i];
                row_cached = r;
                if (r > 0) row_below = p.ev[(int64_t)(r - 1) * n + i];
            }
            const int slot = kk & 7;
            const uint32_t w = word_of(row, slot >> 1);
            return (slot & 1) ? (int)(w >> 16) : (int)(w & 0xffff);
        };
        int s_hi = p.S - 1;
        int brk_next = s_hi >= 0 ? p.brk_k[(int64_t)s_hi * n + i] : -1;
        int mism = 0;
        int ck_row = L / p.K, ck_off = L - ck_row * p.K;
        const float4 *a4 = reinterpret_cast<const float4 *>(a);
        float4 *key4 = reinterpret_cast<float4 *>(key);
        const float4 *G24 = reinterpret_cast<const float4 *>(G2);
        const int nq = nop >> 2;
        for (int k = L; k >= 0; --k) {
            const bool draw = (k < L) || (st == SSA_TRAJ_OK);
            const int s_top = s_hi;
            while (s_hi >= 0 && brk_next == k) {
                --s_hi;
                brk_next = s_hi >= 0 ? p.brk_k[(int64_t)s_hi * n + i] : -1;
            }
            if (draw) {
                const int jk = event_at(k);
                // pass 1: the keys; the waiting-time word and the padded ones have rate 0 and key 0
                float rmax = 0.0f;
                for (int c = 0; c < rounds; ++c) {
                    const int b = 32 * c + lane;
                    const uint4 r = philox4x32_10(make_uint4((uint32_t)b, (uint32_t)k, noise.c2, noise.c3), noise.key0,
                                                  noise.key1);
                    const float4 av = a4[b];
                    const float4 kv = make_float4(av.x * inv_exp_of_word(r.x), av.y * inv_exp_of_word(r.y),
                                                  av.z * inv_exp_of_word(r.z), av.w * inv_exp_of_word(r.w));
                    rmax = fmaxf(rmax, fmaxf(fmaxf(kv.x, kv.y), fmaxf(kv.z, kv.w)));
                    key4[b] = kv;
                }
                rmax = warp_max_nonneg(rmax);
                if (HOT || !(rmax >= 0x1p-60f && rmax <= 0x1p120f))
                    rmax = warp_keys_scaled(rounds, a, k, noise, rmax > 1.0f ? 0x1p110f : 0.0f, HOT, key);
                __syncwarp();
                const KeyTop top = key_top(rmax);
                const float top_edge = rmax * (1.0f - kTieMargin);  // keys from here on may be the largest
                const bool k_tops = key[jk + 1] >= top_edge;
                if (NS == 0) __syncwarp();  // every lane has read that key before its owner puts a weight in its place
                // pass 2: soft-sample weights q_j = (key_j / largest)^(1/T), Z = sum q, W = sum q w with
                // w_j = +lam_s (production of s) or -lam_s (degradation of s)
                float Zp = 0.0f, Wp = 0.0f;
                int near = 0;  // keys within the tie margin of the largest
                float qp[NS > 0 ? NS : 1], qd[NS > 0 ? NS : 1];
                each_species([&](int c, int s) {
                    const float rp = key[s + 1], rd = key[nd + s + 1];
                    near += (rp >= top_edge) + (rd >= top_edge);
                    const float q1 = ex2_approx(top.lg2(rp) * invT_q), q2 = ex2_approx(top.lg2(rd) * invT_q);
                    Zp += q1 + q2;
                    Wp = fmaf(q1 - q2, lam(c), Wp);
                    if (NS > 0) {
                        qp[NS > 0 ? c : 0] = q1;
                        qd[NS > 0 ? c : 0] = q2;
                    } else {
                        key[s + 1] = q1;
                        key[nd + s + 1] = q2;
                    }
                });
                // the recorded reaction won the race if its key is the only one at the top; near ties are raced again
                if (__reduce_add_sync(0xffffffffu, near) == 1) mism += !k_tops;
                else mism += warp_race_exact(rounds, a, k, noise) != jk;
                const float Z = warp_sum(Zp), Wq = warp_sum(Wp);
                const float invZ = __fdividef(1.0f, Z), Wbar = Wq * invZ, cz = invZ * invT;
                // pass 3: psi_j = q_j / Z (w_j - W/Z) / T (HOLD readout: no waiting-time path); the outputs first,
                // since lambda_h receives (W2^T G2)_h
                auto weight_p = [&](int c, int s) { return NS > 0 ? qp[NS > 0 ? c : 0] : key[s + 1]; };
                auto weight_d = [&](int c, int s) { return NS > 0 ? qd[NS > 0 ? c : 0] : key[nd + s + 1]; };
                each_species([&](int c, int s) {
                    if (32 * c + 31 >= nh && s >= nh) {
                        const int o = s - nh;
                        const float g = weight_p(c, s) * cz * (lam(c) - Wbar) * cO[o];
                        G2[o] = g;
                        db2[o] += g;
                        R[o] += g;
                    }
                });
                __syncwarp();
                each_species([&](int c, int s) {
                    const float l = lam(c), psi = weight_d(c, s) * cz * (-l - Wbar);
                    const int x = X[s];
                    dlogd(c) += psi;
                    float acc = __fdividef(psi, __int2float_rn(x));
                    acc = x > 0 ? acc : 0.0f;  // a = d X > 0 where X > 0
                    G1(c) = fmaf(weight_p(c, s) * cz * (l - Wbar), cH[s], G1(c));
                    const float4 *w = W2t + (int64_t)s * nq;
                    auto column = [&](int q) {  // in output order; the padding and the outputs' rows add 0
                        const float4 wv = __ldg(w + q), g = G24[q];
                        acc = fmaf(wv.w, g.w, fmaf(wv.z, g.z, fmaf(wv.y, g.y, fmaf(wv.x, g.x, acc))));
                    };
#pragma unroll
                    for (int q = 0; q < 3; ++q)
                        if (q < nq) column(q);
                    for (int q = 3; q < nq; ++q) column(q);
                    lam(c) = l + acc;
                });
            }
            // HOLD samples of the outputs at state k
            for (int s2 = s_hi + 1; s2 <= s_top; ++s2)
                each_species([&](int c, int s) {
                    if (32 * c + 31 >= nh && s >= nh) lam(c) += gl[(int64_t)s2 * no + s - nh];
                });
            if (ck_off == 0) {
                const int *ck = p.ckpt + (int64_t)ck_row * nd * n + i;
                int bad = 0;
                for (int q = lane; q < nd; q += 32) bad += (ck[(int64_t)q * n] != X[q]);
                mism += __reduce_add_sync(0xffffffffu, bad);
                --ck_row;
                ck_off = p.K;
            }
            --ck_off;
            __syncwarp();
            if (k > 0) {
                // undo event k-1 (state k -> k-1); a hidden change adds delta R to dW2[:, i] (a reduction without a
                // returned value: the warp does not wait for memory, and one lane's adds to a place keep their order)
                const int jp = event_at(k - 1);
                const int sp = jp < nd ? jp : jp - nd;
                const int delta = jp < nd ? 1 : -1;
                if (lane == 0) {
                    const int x = X[sp] - delta;
                    X[sp] = x;
                    a[nd + sp + 1] = __fmul_rn(s_d[sp], int2f(x));
                }
                if (sp < nh) {
                    for (int o = lane; o < no; o += 32) {
                        atomicAdd(dW2 + o * nh + sp, (float)delta * R[o]);
                        E2acc[o] -= (long long)delta * __ldg(W2fix + o * nh + sp);
                        set_output(o);
                    }
                }
            }
            __syncwarp();
        }
        each_species([&](int c, int s) {
            if (s < nh) p.G1[i * nh + s] = G1(c);
            key[s] = dlogd(c);  // for the block's sum
        });
        if (lane == 0 && mism) atomicAdd(p.mismatch, mism);
    } else if (i < n) {
        for (int h = lane; h < nh; h += 32) p.G1[i * nh + h] = 0.0f;
    }
    __syncthreads();
    // fixed-order sum over the block's warps: [db2 | dlogd]
    const int red = no + nd;
    const float *base0 = reinterpret_cast<const float *>(wb);
    const size_t at_db2 = (db2 - wbase), at_dlogd = wide;
    for (int q = threadIdx.x; q < red; q += blockDim.x) {
        float acc = 0.0f;
        for (int w = 0; w < W; ++w) {
            const float *wp = base0 + w * per_warp;
            acc += q < no ? wp[at_db2 + q] : wp[at_dlogd + (q - no)];
        }
        p.partial[(int64_t)blockIdx.x * red + q] = acc;
    }
}

// per-image sums of dL/dE1 (fixed order over the image's trajectories), db1, and the transposed
// hi/lo bf16 limbs G^T for the tensor-core dW1 = G^T x
__global__ void grn_image_grad_kernel(const float *G1, int64_t n_img, int64_t tpi, int nh, int n_img_pad, float *Gimg,
                                      uint16_t *Gt_hi, uint16_t *Gt_lo)
{
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < (int64_t)nh * n_img_pad;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int h = (int)(q / n_img_pad);
        const int64_t img = q % n_img_pad;
        float acc = 0.0f;
        if (img < n_img)
            for (int64_t t = 0; t < tpi; ++t) acc += G1[(img * tpi + t) * nh + h];
        if (img < n_img) Gimg[img * nh + h] = acc;
        const uint16_t hi = float_to_bf16_rn(acc);
        Gt_hi[q] = hi;
        Gt_lo[q] = float_to_bf16_rn(acc - bf16_to_float(hi));
    }
}

__global__ void grn_db1_kernel(const float *Gimg, int64_t n_img, int nh, float *db1)
{
    for (int h = blockIdx.x * blockDim.x + threadIdx.x; h < nh; h += gridDim.x * blockDim.x) {
        float acc = 0.0f;
        for (int64_t img = 0; img < n_img; ++img) acc += Gimg[img * nh + h];
        db1[h] = acc;
    }
}

__global__ void grn_transpose_x_kernel(const int32_t *x_img, int64_t n_img, int n_in, int n_img_pad, uint16_t *xT)
{
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < (int64_t)n_in * n_img_pad;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int p = (int)(q / n_img_pad);
        const int64_t img = q % n_img_pad;
        xT[q] = float_to_bf16_exact(img < n_img ? (float)x_img[img * n_in + p] : 0.0f);
    }
}

__global__ void grn_split_partials_kernel(const float *red, int no, int nd, float *db2, float *dlogd)
{
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < no + nd; q += gridDim.x * blockDim.x) {
        if (q < no) db2[q] = red[q];
        else dlogd[q - no] = red[q];
    }
}

}  // namespace ssa

// =============================================================================================
// C ABI
// =============================================================================================
using namespace ssa;

namespace {

// N-tile of the tensor-core dW1 = G^T x (n_in columns)
int grn_dw1_nt(const ssa_grn *g) { return (g->n_in % 112 == 0) ? 112 : 64; }

// shared memory one CTA may hold on sm_103a
constexpr size_t kGrnMaxSmem = 227 * 1024;

size_t grn_fwd_smem(const ssa_grn *g, int warps)  // without W2
{
    const int ndp = (g->n_dyn + 3) & ~3, nop = (g->n_out + 3) & ~3;
    return 4 * ((size_t)g->n_dyn + nop) + 16 + 4 * (size_t)warps * (ndp + wide_len(g->M) + 2 * (size_t)nop);
}
size_t grn_fwd_smem_w2(const ssa_grn *g, int warps) { return grn_fwd_smem(g, warps) + 4 * (size_t)g->n_out * g->n_hid; }

bool grn_sums_in_registers(const ssa_grn *g) { return g->n_dyn <= kGrnRegSpecies; }  // 288 = 9 rounds

size_t grn_adj_smem(const ssa_grn *g, int warps)
{
    const int nop = (g->n_out + 3) & ~3;
    return 4 * ((size_t)g->n_dyn + nop) + 16 +
           4 * (size_t)warps * grn_adj_words(g->n_hid, g->n_out, !grn_sums_in_registers(g));
}

// Warps per block: four, or as many as the kernel's own per-warp arrays leave room for. The exact forward gives up W2's place
// in shared memory before it gives up a warp: 1,024 trajectories of 3,000-10, a forward to t = 0.3 in 29.3 ms with two
// warps beside W2, 15.9 with four and W2 through L1 (28.0 with four and W2 before the propensities were kept); 3,800-4 76.5
// with the adjoint's one warp, 23.9 with four.
int grn_warps(size_t (*smem)(const ssa_grn *, int), const ssa_grn *g)
{
    int w = kGrnWarps;
    while (w > 1 && smem(g, w) > kGrnMaxSmem) --w;
    return w;
}

// The relaxed path takes networks whose W2 leaves this much room (four warps with four arrays of the species and one of
// the reactions each, and the segment's dL/dE2); a block has fewer warps where four of the kernels' own arrays do not
// fit.
bool grn_soft_fits(const ssa_grn *g, bool record)
{
    const size_t ndp = (g->n_dyn + 3) & ~3, nhp = (g->n_hid + 3) & ~3, nop = (g->n_out + 3) & ~3, Mq = (g->M + 3) & ~3;
    const size_t shared = (size_t)g->n_out * g->n_hid + g->n_dyn + nop;
    const size_t fwd = 4 * (shared + 4 * (ndp + nhp + nop + Mq));
    const size_t adj = 4 * (shared + 4 * (3 * ndp + 2 * nhp + (2 + kGrnSoftK) * nop + Mq));
    return fwd <= kGrnMaxSmem && (!record || adj <= kGrnMaxSmem);
}

size_t grn_soft_fwd_smem(const ssa_grn *g, int warps)
{
    const size_t ndp = (g->n_dyn + 3) & ~3, nop = (g->n_out + 3) & ~3;
    return 4 * ((size_t)g->n_out * g->n_hid + g->n_dyn + nop + warps * (ndp + 2 * (size_t)wide_len(g->M))) + 16;
}

size_t grn_soft_adj_smem(const ssa_grn *g, int warps)
{
    const size_t nop = (g->n_out + 3) & ~3;
    return 4 * ((size_t)g->n_out * g->n_hid + g->n_dyn + nop + warps * grn_soft_adj_words(g->n_hid, g->n_out)) + 16;
}

WsLayout grn_layout(const ssa_grn *g, int64_t n_img, int64_t tpi, int32_t S, const ssa_fwd_opts *o)
{
    WsLayout L{};
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t at = off;
        off = (off + bytes + 255) / 256 * 256;
        return at;
    };
    const int64_t n = n_img * tpi;
    L.n_in_pad = (g->n_in + 7) / 8 * 8;
    L.n_img_pad = (int)((n_img + 7) / 8 * 8);
    L.limbs = kGrnLimbs;
    L.red_len = g->n_out + g->n_dyn;
    L.M_pad = g->Mp;
    L.flag = take(16 * sizeof(int));
    L.counts = take(SSA_TRAJ_N_CODES * sizeof(unsigned long long));
    L.k_rates = take(16);
    L.ts = take((size_t)(S > 0 ? S : 1) * sizeof(double));
    L.obs_sp = take(16);
    L.draws = take((size_t)(n > 0 ? n : 1) * sizeof(int));
    L.status = take((size_t)(n > 0 ? n : 1) * sizeof(int));
    L.E1 = take((size_t)(n_img > 0 ? n_img : 1) * g->n_hid * sizeof(float));
    L.W1L = take((size_t)kGrnLimbs * g->n_hid * L.n_in_pad * 2);
    L.xb = take((size_t)(n_img > 0 ? n_img : 1) * L.n_in_pad * 2);
    L.W2fix = take((size_t)g->n_out * g->n_hid * 4);
    L.W2f = take((size_t)g->n_out * g->n_hid * 4);
    L.W2t = take((size_t)((g->n_out + 3) & ~3) * g->n_dyn * 4);
    L.dvec = take((size_t)g->n_dyn * 4);
    L.grid = take(16 * sizeof(int));
    // split-K partial sums of E1 (forward) and of dW1 (backward), when the product fills too few SMs
    size_t tc_words = n_img > 0 ? 2 * tc_split_words((int)n_img, g->n_hid, g->n_in, 64) : 0;  // (lo, hi) pairs
    if (o->record && n_img > 0)
        tc_words = std::max(tc_words, tc_split_words(g->n_hid, g->n_in, (int)n_img, grn_dw1_nt(g)));
    L.tcpart = take(std::max<size_t>(tc_words, 1) * sizeof(double));
    if (o->record) {
        // the soft forward keeps float checkpoints every 8 steps; the hard one int counts every K
        const int K = o->selector == SSA_SELECT_SOFT ? kGrnSoftK : o->ckpt_interval > 0 ? o->ckpt_interval : 64;
        L.ev_rows = (o->max_steps + 7) / 8;
        L.n_ckpt = o->max_steps / K + 1;
        const int wpb = grn_warps(o->selector == SSA_SELECT_SOFT ? grn_soft_adj_smem : grn_adj_smem, g);
        L.max_blocks = (n + wpb - 1) / wpb;
        L.xfinal = take((size_t)g->n_dyn * n * 4);
        L.ev = take((size_t)L.ev_rows * n * sizeof(uint4));
        L.ckpt = take((size_t)L.n_ckpt * g->n_dyn * n * 4);
        L.brk_k = take((size_t)S * n * 4);
        L.brk_a = take(16);
        L.partial = take((size_t)(L.max_blocks > 0 ? L.max_blocks : 1) * L.red_len * 4);
        L.dA = take(16);
        L.G1 = take((size_t)(n > 0 ? n : 1) * g->n_hid * 4);
        L.Gimg = take((size_t)(n_img > 0 ? n_img : 1) * g->n_hid * 4);
        L.Gt = take((size_t)2 * g->n_hid * L.n_img_pad * 2);
        L.xT = take((size_t)g->n_in * L.n_img_pad * 2);
        L.red = take((size_t)L.red_len * 4);
        L.dW2t = take((size_t)(n > 0 ? n : 1) * g->n_out * g->n_hid * 4);
        L.dW2_chunk = std::max<int64_t>(256, (n + 65534) / 65535);
        L.dW2p = take((size_t)((n + L.dW2_chunk - 1) / L.dW2_chunk + 1) * g->n_out * g->n_hid * 4);
        if (o->selector == SSA_SELECT_SOFT)
            L.soft_seg = take((size_t)(n > 0 ? n : 1) * kGrnSoftK * grn_soft_row(g->n_dyn, g->n_out, g->M) * 4);
    }
    L.total = off;
    return L;
}


#define GRN_CUDA_TRY(expr)                                                                              \
    do {                                                                                                \
        cudaError_t e_ = (expr);                                                                        \
        if (e_ != cudaSuccess) return set_error(SSA_ERR_CUDA, cudaGetErrorString(e_));                   \
    } while (0)

}  // namespace

extern "C" ssa_status ssa_grn_create(int32_t n_in, int32_t n_hid, int32_t n_out, float k_max, ssa_grn **out)
{
    if (!out) return set_error(SSA_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    if (n_in < 1 || n_hid < 1 || n_out < 1 || n_in > (1 << 16) || n_hid > 4096 || n_out > 1024)
        return set_error(SSA_ERR_INVALID_ARG, "GRN sizes out of range");
    if (2 * (n_hid + n_out) > 65535) return set_error(SSA_ERR_UNSUPPORTED, "too many reactions for the uint16 log");
    // exactness of the tensor-core contraction: one 6-bit limb times 8-bit counts, summed over n_in,
    // stays below 2^24 quanta
    if ((int64_t)n_in * 63 * 256 >= (int64_t)1 << 24) return set_error(SSA_ERR_UNSUPPORTED, "n_in above 1040");
    if (!(k_max > 0.0f)) return set_error(SSA_ERR_INVALID_ARG, "k_max must be positive");
    ssa_grn *g = new (std::nothrow) ssa_grn();
    if (!g) return set_error(SSA_ERR_CUDA, "host allocation failed");
    g->n_in = n_in;
    g->n_hid = n_hid;
    g->n_out = n_out;
    g->n_dyn = n_hid + n_out;
    g->M = 2 * g->n_dyn;
    g->Mp = (g->M + 4) / 4 * 4;
    g->k_max = k_max;
    *out = g;
    return SSA_OK;
}

extern "C" void ssa_grn_destroy(ssa_grn *g) { delete g; }

extern "C" size_t ssa_grn_workspace_bytes(const ssa_grn *g, int64_t n_img, int64_t traj_per_img, int32_t n_samples,
                                          const ssa_fwd_opts *opts)
{
    if (!g || n_img < 0 || traj_per_img < 1 || n_samples < 0 || !opts || opts->max_steps < 1) return 0;
    return grn_layout(g, n_img, traj_per_img, n_samples, opts).total;
}

extern "C" ssa_status ssa_grn_forward(const ssa_grn *g, const uint16_t *W1, const float *b1, const uint16_t *W2,
                                      const float *b2, const float *log_d, int64_t n_img, int64_t traj_per_img,
                                      int64_t traj_offset, const int32_t *x_img, double t_end,
                                      const double *sample_times, int32_t S, uint64_t seed, const ssa_fwd_opts *opts,
                                      void *workspace, size_t workspace_bytes, int32_t *obs_out, int32_t *draws_out,
                                      int32_t *status_out, void *stream, ssa_run **run_out)
{
    if (run_out) *run_out = nullptr;
    if (!g || !opts) return set_error(SSA_ERR_INVALID_ARG, "NULL network or options");
    if (opts->readout != SSA_READOUT_HOLD) return set_error(SSA_ERR_UNSUPPORTED, "the GRN reads out with HOLD only");
    const bool soft = opts->selector == SSA_SELECT_SOFT;
    if (!soft && (opts->selector != SSA_SELECT_GUMBEL || opts->temperature != 0.0f))
        return set_error(SSA_ERR_UNSUPPORTED, "the GRN runs the Gumbel-max selector or the soft forward");
    if (soft && (!(opts->temperature > 0.0f) || !(opts->temperature < 3.0e38f)))
        return set_error(SSA_ERR_UNSUPPORTED, "the GRN's soft forward needs T > 0");
    if (soft && !grn_soft_fits(g, opts->record != 0))
        return set_error(SSA_ERR_UNSUPPORTED, "the GRN's soft path keeps W2 (and a recorded run dL/dW2) in shared memory: "
                                              "n_out * n_hid too large");
    if (opts->max_steps < 1 || opts->max_steps > 0x7fffffffLL || (opts->ckpt_interval % 8) || opts->ckpt_interval < 0)
        return set_error(SSA_ERR_INVALID_ARG, "invalid options");
    if (n_img < 0 || traj_per_img < 1 || traj_offset < 0 || S < 0 || !(t_end >= 0.0) || !(t_end < 1e300))
        return set_error(SSA_ERR_INVALID_ARG, "bad sizes or horizon");
    if (!W1 || !b1 || !W2 || !b2 || !log_d || (n_img > 0 && !x_img) || (S > 0 && !sample_times))
        return set_error(SSA_ERR_INVALID_ARG, "NULL input pointer");
    const int64_t n = n_img * traj_per_img;
    if (n > 0 && S > 0 && !obs_out) return set_error(SSA_ERR_INVALID_ARG, "obs_out is NULL");
    const WsLayout L = grn_layout(g, n_img, traj_per_img, S, opts);
    if (!workspace || workspace_bytes < L.total) return set_error(SSA_ERR_WORKSPACE, "workspace too small");
    if (reinterpret_cast<uintptr_t>(workspace) % 256) return set_error(SSA_ERR_WORKSPACE, "workspace not 256-byte aligned");
    if ((reinterpret_cast<uintptr_t>(W1) | reinterpret_cast<uintptr_t>(W2)) & 1)
        return set_error(SSA_ERR_INVALID_ARG, "weights must be 2-byte aligned");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned char *ws = static_cast<unsigned char *>(workspace);
    int *flag = reinterpret_cast<int *>(ws + L.flag);
    int *grid = reinterpret_cast<int *>(ws + L.grid);
    GRN_CUDA_TRY(cudaMemsetAsync(flag, 0, 16 * sizeof(int), st));
    const int init_grid[4] = {0, 255, 0, 0};
    GRN_CUDA_TRY(cudaMemcpyAsync(grid, init_grid, sizeof(init_grid), cudaMemcpyHostToDevice, st));
    if (S > 0) GRN_CUDA_TRY(cudaMemcpyAsync(ws + L.ts, sample_times, (size_t)S * 8, cudaMemcpyDeviceToDevice, st));
    GRN_CUDA_TRY(launch_validate_inputs(reinterpret_cast<const double *>(ws + L.ts), S, t_end, nullptr, 0, g->n_dyn,
                                        0, flag, st));
    GRN_CUDA_TRY(cudaMemsetAsync(ws + L.W2t, 0, (size_t)((g->n_out + 3) & ~3) * g->n_dyn * 4, st));
    grn_exponents_kernel<<<64, 256, 0, st>>>(W1, (int64_t)g->n_hid * g->n_in, W2, (int64_t)g->n_out * g->n_hid, grid);
    grn_prepare_kernel<<<256, 256, 0, st>>>(W1, W2, x_img, log_d, g->n_in, g->n_hid, g->n_out, n_img, L.n_in_pad,
                                            reinterpret_cast<uint16_t *>(ws + L.W1L), reinterpret_cast<int *>(ws + L.W2fix),
                                            reinterpret_cast<float *>(ws + L.W2f), reinterpret_cast<float *>(ws + L.W2t),
                                            reinterpret_cast<uint16_t *>(ws + L.xb),
                                            reinterpret_cast<float *>(ws + L.dvec), grid);
    GRN_CUDA_TRY(cudaGetLastError());
    // E1 = W1 x + b1 on the tensor cores: one accumulator per limb, summed in binary64
    if (n_img > 0) {
        TcMaps maps;
        memset(&maps, 0, sizeof(maps));
        if (!tc_make_map(&maps.a[0], ws + L.xb, (int)n_img, g->n_in, L.n_in_pad, 128))
            return set_error(SSA_ERR_CUDA, "tensor map encoding failed");
        for (int t = 0; t < kGrnLimbs; ++t)
            if (!tc_make_map(&maps.b[t], ws + L.W1L + (size_t)t * g->n_hid * L.n_in_pad * 2, g->n_hid, g->n_in,
                             L.n_in_pad, 64))
                return set_error(SSA_ERR_CUDA, "tensor map encoding failed");
        TcArgs args{(int)n_img, g->n_hid, g->n_in, 1, kGrnLimbs, kGrnLimbs, 1, b1,
                    reinterpret_cast<float *>(ws + L.E1), g->n_hid, flag + 4};
        args.Dpart = reinterpret_cast<double *>(ws + L.tcpart);  // split K when the tiles underfill the SMs
        args.limb_grid = grid + 4;  // limb t is an integer multiple of 2^(g1 + 6 t): summed exactly in int64
        args.limb_bits = kGrnLimbBits;
        GRN_CUDA_TRY(tc_gemm_launch(maps, args, 64, st));
    }
    GrnParams p{};
    p.n_in = g->n_in;
    p.n_hid = g->n_hid;
    p.n_out = g->n_out;
    p.n_dyn = g->n_dyn;
    p.M = g->M;
    p.Mp = g->Mp;
    p.nb = (g->M + 4) >> 2;
    p.k_max = g->k_max;
    p.n_traj = n;
    p.tpi = traj_per_img;
    p.traj_offset = (uint64_t)traj_offset;
    p.seed = seed;
    p.E1 = reinterpret_cast<const float *>(ws + L.E1);
    p.W2fix = reinterpret_cast<const int *>(ws + L.W2fix);
    p.W2f = reinterpret_cast<const float *>(ws + L.W2f);
    p.W2t = reinterpret_cast<const float4 *>(ws + L.W2t);
    p.b2 = b2;
    p.dvec = reinterpret_cast<const float *>(ws + L.dvec);
    p.grid = grid + 3;
    p.t_end = t_end;
    p.ts = reinterpret_cast<const double *>(ws + L.ts);
    p.S = S;
    p.max_steps = opts->max_steps;
    p.obs_out = obs_out;
    p.draws = reinterpret_cast<int *>(ws + L.draws);
    p.status = reinterpret_cast<int *>(ws + L.status);
    p.flag = flag;
    p.err = flag + 1;
    p.K = opts->ckpt_interval > 0 ? opts->ckpt_interval : 64;
    if (opts->record) {
        p.ev = reinterpret_cast<uint4 *>(ws + L.ev);
        p.ckpt = reinterpret_cast<int *>(ws + L.ckpt);
        p.brk_k = reinterpret_cast<int *>(ws + L.brk_k);
        p.xfinal = reinterpret_cast<int *>(ws + L.xfinal);
        p.n_ckpt = L.n_ckpt;
    }
    if (n > 0 && soft) {
        p.invT = 1.0f / opts->temperature;
        const int wpb = grn_warps(grn_soft_fwd_smem, g);
        const size_t smem = grn_soft_fwd_smem(g, wpb);
        auto kern = hot_weights(p.invT) ? grn_soft_fwd_kernel<true> : grn_soft_fwd_kernel<false>;
        GRN_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        kern<<<(unsigned)((n + wpb - 1) / wpb), 32 * wpb, smem, st>>>(
            p, reinterpret_cast<float *>(obs_out), opts->record);
        GRN_CUDA_TRY(cudaGetLastError());
    } else if (n > 0) {
        const int wpb = grn_warps(grn_fwd_smem, g);
        // (a network whose W2 leaves no room for one warp is refused by the launch, as it always was)
        const bool w2s = grn_fwd_smem_w2(g, wpb) <= kGrnMaxSmem || grn_fwd_smem_w2(g, 1) > kGrnMaxSmem;
        const size_t smem = w2s ? grn_fwd_smem_w2(g, wpb) : grn_fwd_smem(g, wpb);
        auto kern = w2s ? grn_fwd_kernel<true> : grn_fwd_kernel<false>;
        GRN_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        kern<<<(unsigned)((n + wpb - 1) / wpb), 32 * wpb, smem, st>>>(p, opts->record);
        GRN_CUDA_TRY(cudaGetLastError());
    }
    if (n > 0 && draws_out) GRN_CUDA_TRY(cudaMemcpyAsync(draws_out, p.draws, (size_t)n * 4, cudaMemcpyDeviceToDevice, st));
    if (n > 0 && status_out) GRN_CUDA_TRY(cudaMemcpyAsync(status_out, p.status, (size_t)n * 4, cudaMemcpyDeviceToDevice, st));
    if (run_out) {
        ssa_run *run = new (std::nothrow) ssa_run();
        if (!run) return set_error(SSA_ERR_CUDA, "host allocation failed");
        run->net = nullptr;
        run->variant = 32;
        run->grn = g;
        run->n_img = n_img;
        run->traj_per_img = traj_per_img;
        run->n_traj = n;
        run->traj_offset = (uint64_t)traj_offset;
        run->seed = seed;
        run->S = S;
        run->n_obs = g->n_out;
        run->opts = *opts;
        run->t_end = t_end;
        run->ws = ws;
        run->L = L;
        run->x_img = x_img;
        run->b2 = b2;
        *run_out = run;
    }
    return SSA_OK;
}

extern "C" ssa_status ssa_grn_backward(ssa_run *run, const float *dl_dobs, int64_t dl_traj_stride, float temperature,
                                       float *dW1, float *db1, float *dW2, float *db2, float *dlog_d, void *stream)
{
    if (!run || !run->grn) return set_error(SSA_ERR_INVALID_ARG, "not a GRN run");
    if (!run->opts.record) return set_error(SSA_ERR_STATE, "the forward was not recorded");
    if (!(temperature > 0.0f)) return set_error(SSA_ERR_INVALID_ARG, "temperature must be > 0");
    const bool soft = run->opts.selector == SSA_SELECT_SOFT;
    if (soft && temperature != run->opts.temperature)
        return set_error(SSA_ERR_INVALID_ARG, "the gradient of the soft forward is taken at the forward's temperature");
    if (!dW1 || !db1 || !dW2 || !db2 || !dlog_d) return set_error(SSA_ERR_INVALID_ARG, "NULL gradient output");
    if (dl_traj_stride != 0 && dl_traj_stride < (int64_t)run->S * run->n_obs)
        return set_error(SSA_ERR_INVALID_ARG, "dl_traj_stride must be 0 or >= n_samples * n_out");
    if (!dl_dobs && run->n_traj > 0 && run->S > 0) return set_error(SSA_ERR_INVALID_ARG, "dl_dobs is NULL");
    const ssa_grn *g = run->grn;
    const WsLayout &L = run->L;
    unsigned char *ws = run->ws;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int *flag = reinterpret_cast<int *>(ws + L.flag);
    GRN_CUDA_TRY(cudaMemsetAsync(flag + 2, 0, sizeof(int), st));
    const int64_t n = run->n_traj;
    GrnParams p{};
    p.n_in = g->n_in;
    p.n_hid = g->n_hid;
    p.n_out = g->n_out;
    p.n_dyn = g->n_dyn;
    p.M = g->M;
    p.Mp = g->Mp;
    p.nb = (g->M + 4) >> 2;
    p.k_max = g->k_max;
    p.n_traj = n;
    p.tpi = run->traj_per_img;
    p.traj_offset = run->traj_offset;
    p.seed = run->seed;
    p.E1 = reinterpret_cast<const float *>(ws + L.E1);
    p.W2fix = reinterpret_cast<const int *>(ws + L.W2fix);
    p.W2f = reinterpret_cast<const float *>(ws + L.W2f);
    p.W2t = reinterpret_cast<const float4 *>(ws + L.W2t);
    p.b2 = run->b2;
    p.dvec = reinterpret_cast<const float *>(ws + L.dvec);
    p.grid = reinterpret_cast<const int *>(ws + L.grid) + 3;
    p.S = run->S;
    p.K = run->opts.ckpt_interval > 0 ? run->opts.ckpt_interval : 64;
    p.draws = reinterpret_cast<int *>(ws + L.draws);
    p.status = reinterpret_cast<int *>(ws + L.status);
    p.ev = reinterpret_cast<uint4 *>(ws + L.ev);
    p.ckpt = reinterpret_cast<int *>(ws + L.ckpt);
    p.brk_k = reinterpret_cast<int *>(ws + L.brk_k);
    p.xfinal = reinterpret_cast<int *>(ws + L.xfinal);
    p.dl_dobs = dl_dobs;
    p.dl_stride = dl_traj_stride;
    p.invT = 1.0f / temperature;
    p.G1 = reinterpret_cast<float *>(ws + L.G1);
    p.dW2t = reinterpret_cast<float *>(ws + L.dW2t);
    p.partial = reinterpret_cast<float *>(ws + L.partial);
    p.mismatch = flag + 2;
    p.err = flag + 1;
    p.n_ckpt = L.n_ckpt;
    p.seg = soft ? reinterpret_cast<float *>(ws + L.soft_seg) : nullptr;
    const int wpb = grn_warps(soft ? grn_soft_adj_smem : grn_adj_smem, g);
    const bool hot = hot_weights(p.invT);
    const int64_t nblk = (n + wpb - 1) / wpb;
    float *red = reinterpret_cast<float *>(ws + L.red);
    if (n > 0 && soft) {
        const size_t smem = grn_soft_adj_smem(g, wpb);
        auto kern = grn_sums_in_registers(g) ? (hot ? grn_soft_adj_kernel<9, true> : grn_soft_adj_kernel<9, false>)
                                             : (hot ? grn_soft_adj_kernel<0, true> : grn_soft_adj_kernel<0, false>);
        GRN_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        kern<<<(unsigned)nblk, 32 * wpb, smem, st>>>(p);
        GRN_CUDA_TRY(cudaGetLastError());
    } else if (n > 0) {
        const size_t smem = grn_adj_smem(g, wpb);
        const int nd = g->n_dyn;
        auto kern = !grn_sums_in_registers(g) ? (hot ? grn_adj_kernel<0, 0, true> : grn_adj_kernel<0, 0, false>)
                    : nd > 192                ? (hot ? grn_adj_kernel<9, 6, true> : grn_adj_kernel<9, 6, false>)
                    : nd > 96                 ? (hot ? grn_adj_kernel<6, 3, true> : grn_adj_kernel<6, 3, false>)
                                              : (hot ? grn_adj_kernel<3, 0, true> : grn_adj_kernel<3, 0, false>);
        GRN_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        kern<<<(unsigned)nblk, 32 * wpb, smem, st>>>(p);
        GRN_CUDA_TRY(cudaGetLastError());
    }
    GRN_CUDA_TRY(launch_reduce_partials(p.partial, nblk, L.red_len, nullptr, 0, red, nullptr, st));
    grn_split_partials_kernel<<<(L.red_len + 255) / 256, 256, 0, st>>>(red, g->n_out, g->n_dyn, db2, dlog_d);
    GRN_CUDA_TRY(launch_column_sums(p.dW2t, n, (int64_t)g->n_out * g->n_hid, reinterpret_cast<float *>(ws + L.dW2p),
                                    L.dW2_chunk, dW2, st));
    uint16_t *Gt = reinterpret_cast<uint16_t *>(ws + L.Gt);
    uint16_t *xT = reinterpret_cast<uint16_t *>(ws + L.xT);
    const size_t gt_len = (size_t)g->n_hid * L.n_img_pad;
    grn_image_grad_kernel<<<256, 256, 0, st>>>(p.G1, run->n_img, run->traj_per_img, g->n_hid, L.n_img_pad,
                                               reinterpret_cast<float *>(ws + L.Gimg), Gt, Gt + gt_len);
    grn_db1_kernel<<<(g->n_hid + 127) / 128, 128, 0, st>>>(reinterpret_cast<const float *>(ws + L.Gimg), run->n_img,
                                                           g->n_hid, db1);
    grn_transpose_x_kernel<<<256, 256, 0, st>>>(run->x_img, run->n_img, g->n_in, L.n_img_pad, xT);
    GRN_CUDA_TRY(cudaGetLastError());
    if (run->n_img == 0) {  // no images: dL/dW1 is an empty sum (and a zero-length K has no tensor map)
        GRN_CUDA_TRY(cudaMemsetAsync(dW1, 0, (size_t)g->n_hid * g->n_in * sizeof(float), st));
        return SSA_OK;
    }
    // dW1[h][p] = sum_img G[img][h] x[img][p] on the tensor cores (hi + lo bf16 limbs of G)
    TcMaps maps;
    memset(&maps, 0, sizeof(maps));
    const int nt = grn_dw1_nt(g);
    if (!tc_make_map(&maps.a[0], Gt, g->n_hid, (int)run->n_img, L.n_img_pad, 128) ||
        !tc_make_map(&maps.a[1], Gt + gt_len, g->n_hid, (int)run->n_img, L.n_img_pad, 128) ||
        !tc_make_map(&maps.b[0], xT, g->n_in, (int)run->n_img, L.n_img_pad, nt))
        return set_error(SSA_ERR_CUDA, "tensor map encoding failed");
    TcArgs args{g->n_hid, g->n_in, (int)run->n_img, 2, 1, 2, 0, nullptr, dW1, g->n_in, flag + 4};
    args.Dpart = reinterpret_cast<double *>(ws + L.tcpart);
    GRN_CUDA_TRY(tc_gemm_launch(maps, args, nt, st));
    return SSA_OK;
}

extern "C" ssa_status ssa_grn_activations(const ssa_run *run, float *E1_out, int32_t *host_flags, void *stream)
{
    if (!run || !run->grn || !E1_out) return set_error(SSA_ERR_INVALID_ARG, "not a GRN run");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    GRN_CUDA_TRY(cudaMemcpyAsync(E1_out, run->ws + run->L.E1, (size_t)run->n_img * run->grn->n_hid * 4,
                                 cudaMemcpyDeviceToDevice, st));
    if (host_flags) {
        int f[4];
        GRN_CUDA_TRY(cudaMemcpyAsync(f, run->ws + run->L.grid, sizeof(f), cudaMemcpyDeviceToHost, st));
        int e[8];
        GRN_CUDA_TRY(cudaMemcpyAsync(e, run->ws + run->L.flag, sizeof(e), cudaMemcpyDeviceToHost, st));
        GRN_CUDA_TRY(cudaStreamSynchronize(st));
        host_flags[0] = f[2];  // inexact limbs / fixed point / counts
        host_flags[1] = e[4];  // tensor-core wait timeout
    }
    return SSA_OK;
}
