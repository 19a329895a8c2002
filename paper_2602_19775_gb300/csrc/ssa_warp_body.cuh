// ssa_warp_body.cuh -- per-trajectory bodies of the warp-per-trajectory forward and adjoint, shared by
// the single-network kernels and the batch kernel.
#pragma once

#include <type_traits>

#include "ssa_adj_body.cuh"

namespace ssa {

// The network's tables for one launch: rx (then st) and the second region, both in shared or both in global
// memory.
template <class P>
__device__ __forceinline__ WarpTab warp_tab(const P &p, const int4 *rx, const int4 *wtab, const float *k)
{
    const int4 *inc = wtab + wide_len(p.M);
    const int nb = (p.M + 4) >> 2;
    return WarpTab{rx, reinterpret_cast<const int *>(rx + p.Mp), wtab, inc, reinterpret_cast<const int *>(inc + p.N + 1),
                   k, p.M, nb, (nb + 31) >> 5, inc[p.N].w != 0};
}

// ------------------------------------------------------------------------------------------
// Propensities kept between steps. An event changes a few species and so a few propensities; a warp keeps all
// of them in shared memory by lane-major position and forms again, from the new counts, those of the reactions
// its event touches (the same expression, so the same bits as forming every one each step). On a 301-reaction
// network with 11 species an event touches ~50 reactions.
// SIGNED (the adjoint): where a_j = 0 the array holds -D_j instead, D_j = k_j dh_j/dX for the reactant at zero
// (the waiting-time path's derivative there, with k_j times the other count; homodimers, whose derivative
// needs no other count, hold 0), so that a_j = max(value, 0).
// ------------------------------------------------------------------------------------------
template <bool SIGNED>
__device__ __forceinline__ float warp_propensity(const WarpTab &t, int pos, const int *X)
{
    const int4 rx = t.rx[pos];
    const float k = t.k[pos];
    if (!SIGNED) return __fmul_rn(k, mass_action_h_sel(rx, X));
    const bool homo = rx.y >= 0 && rx.y == rx.x;
    const int x1 = rx.x >= 0 ? X[rx.x >= 0 ? rx.x : 0] : 1;
    const int xr2 = X[rx.y >= 0 ? rx.y : 0];
    const int x2 = homo ? max(x1 - 1, 0) : (rx.y >= 0 ? xr2 : 1);
    float d = small2f(max(x1, x2));
    float h = __fmul_rn(small2f(x1), small2f(x2));
    if ((unsigned)(x1 | x2) >= (1u << 23)) {
        h = mass_action_h(rx, X, 1);
        d = __int2float_rn(max(x1, x2));
    } else if (homo) {
        h *= 0.5f;
    }
    const float a = __fmul_rn(k, h);
    return a > 0.0f ? a : (homo ? 0.0f : -(k * d));
}

template <bool SIGNED>
__device__ __forceinline__ void warp_propensities_all(const WarpTab &t, const int *X, float *a)
{
    const int lane = threadIdx.x & 31;
    for (int c = 0; c < t.rounds; ++c)
        for (int q = 0; q < 4; ++q) {
            const int b = 32 * c + lane;
            a[4 * b + q] = b < t.nb ? warp_propensity<SIGNED>(t, q * t.nb + b, X) : 0.0f;
        }
    __syncwarp();
}

// after a change of the species named by four entries: the reactions on their lists, one lane each
template <bool SIGNED>
__device__ __forceinline__ void warp_propensities_touched(const WarpTab &t, const int4 en, const int *X, float *a)
{
    const int4 c0 = t.inc[ent_species(en.x)], c1 = t.inc[ent_species(en.y)], c2 = t.inc[ent_species(en.z)],
               c3 = t.inc[ent_species(en.w)];
    const int o1 = c0.z - c0.x, o2 = o1 + c1.z - c1.x, o3 = o2 + c2.z - c2.x, tot = o3 + c3.z - c3.x;
    for (int q = threadIdx.x & 31; q < tot; q += 32) {
        const int e = q < o1 ? c0.x + q : q < o2 ? c1.x + (q - o1) : q < o3 ? c2.x + (q - o2) : c3.x + (q - o3);
        const int le = t.list[e];
        a[le & 0xffff] = warp_propensity<SIGNED>(t, le >> 16, X);
    }
}

// X += sign v_j, then the touched propensities; all lanes
template <bool SIGNED>
__device__ __forceinline__ void warp_apply(const WarpTab &t, int j, int sign, int *X, float *a)
{
    const int lane = threadIdx.x & 31;
    const int4 en = t.ent[wpos(j)];
    if (!t.many || en.x != kEntMany) {
        const int e = lane == 0 ? en.x : lane == 1 ? en.y : lane == 2 ? en.z : en.w;
        const int d = (int)ent_change(e);
        if (lane < 4 && d != 0) X[ent_species(e)] += sign * d;  // the entries of one reaction name distinct species
        __syncwarp();
        warp_propensities_touched<SIGNED>(t, en, X, a);
    } else {
        const int4 rj = t.rx[jpos(j, t.nb)];
        for (int e = rj.z + lane; e < rj.w; e += 32) X[stoich_species(t.st[e])] += sign * stoich_delta(t.st[e]);
        __syncwarp();
        for (int e = rj.z; e < rj.w; ++e) {
            const int4 c = t.inc[stoich_species(t.st[e])];
            for (int q = c.x + lane; q < c.z; q += 32)
                a[t.list[q] & 0xffff] = warp_propensity<SIGNED>(t, t.list[q] >> 16, X);
        }
    }
    __syncwarp();
}

// ------------------------------------------------------------------------------------------
// The Gumbel-max choice without its logarithms. The race argmax_j a_j / E_j, E_j = -ln(1 - v_j) with
// v_j = 1 - u_j, has a key K_j = a_j / E_j with
//     a_j (1/v_j - 1/2 - v_j/2)  <=  K_j  <=  a_j (1/v_j - 1/2) =: B_j
// (1/v + 1/ln(1 - v) = 1/2 + v/12 + v^2/24 + ... has positive coefficients: convex, from 1/2 at v = 0 to 1 at
// v = 1). Each lane keeps its two largest B_j (one approximate reciprocal each, the slot's number in the six low
// bits); the largest lower bound over the warp is the threshold. If a single B_j reaches it, less a margin far
// above every rounding here and in the exact comparison (2^-13 against 2^-16), that reaction wins the race as the
// binary32 comparisons of E decide it; else the race is run on the variates themselves (warp_race_exact). One
// logarithm per step remains, E_0's. A logarithm costs 32 issue slots and B_j with its bookkeeping 8.
// The bounds assume a0 in [2^-40, 2^100] (no B_j of interest is subnormal or overflows) and the slot number
// six bits, i.e. up to 16 rounds of blocks (M <= 2047); other steps take the exact race.
// ------------------------------------------------------------------------------------------
struct WarpTop {
    float m1, m2;  // the two largest B_j of this lane, low bits replaced
};

__device__ __forceinline__ void warp_top_add(WarpTop &top, float a, uint32_t x, int slot)
{
    const float v = u01(~x);  // 1 - u, exact
    const float B = a * (rcp_approx(v) - 0.5f);
    const float key = __uint_as_float((__float_as_uint(B) & ~63u) | (uint32_t)slot);
    top.m2 = fmaxf(top.m2, fminf(top.m1, key));
    top.m1 = fmaxf(top.m1, key);
}

// the winner's lane and slot if it is certain; a_of(slot): this lane's propensity in that slot
template <class AF>
__device__ __forceinline__ bool warp_top_decide(const WarpTop &top, float a0, const AF &a_of, int &src, int &slot)
{
    const int mine = (int)(__float_as_uint(top.m1) & 63u);
    const float a1 = a_of(mine);
    const float half = 0.5f * a1;
    // a v / 2 with v from B = a (1/v - 1/2)
    const float width = half * a1 * rcp_approx(top.m1 + half + 1e-30f);
    const float thr = warp_max_nonneg(fmaxf(top.m1 - width - 0x1p-13f * top.m1, 0.0f));
    const unsigned c1 = __ballot_sync(0xffffffffu, top.m1 >= thr), c2 = __ballot_sync(0xffffffffu, top.m2 >= thr);
    src = __ffs(c1) - 1;
    slot = __shfl_sync(0xffffffffu, mine, src);
    return c2 == 0 && (c1 & (c1 - 1)) == 0 && a0 >= 0x1p-40f && a0 <= 0x1p100f;
}

// the race itself over this lane's blocks, with the accurate variates; returns the winner (-1: no positive key)
static __device__ __noinline__ int warp_race_exact(int rounds, const float *a, int k, WarpNoise z)
{
    const int lane = threadIdx.x & 31;
    float ab = 0.0f, Eb = 1.0f;
    int jb = -1;
    for (int c = 0; c < rounds; ++c) {
        const int b = 32 * c + lane;
        const uint4 r = philox4x32_10(make_uint4((uint32_t)b, (uint32_t)k, z.c2, z.c3), z.key0, z.key1);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            race(fmaxf(a[4 * b + q], 0.0f), neg_log_unit(u01(word_of(r, q))), 4 * b + q - 1, ab, Eb, jb);
    }
    warp_race_combine(ab, Eb, jb);
    return jb;
}

// One step of the forward: a0 over this lane's blocks b = lane, lane + 32, ... in increasing j and a butterfly over
// the lanes, E_0, and the choice. The lane's blocks are drawn four at a time (independent chains for the
// scheduler).
__device__ __forceinline__ void warp_step_eval(int n_rounds, int k, const WarpNoise &z, const float *a, float &a0, float &E0,
                                               int &jb)
{
    const int lane = threadIdx.x & 31;
    float a0p = 0.0f;
    uint32_t x0 = 0;
    WarpTop top{0.0f, 0.0f};
    // C rounds from t0 on; a lane past its last block draws one all the same and finds propensities of 0
    auto rounds = [&](auto count, int t0) {
        constexpr int C = decltype(count)::value;
        uint4 r[C];
#pragma unroll
        for (int t = 0; t < C; ++t)
            r[t] = philox4x32_10(make_uint4((uint32_t)(lane + 32 * (t0 + t)), (uint32_t)k, z.c2, z.c3), z.key0, z.key1);
        if (t0 == 0) x0 = r[0].x;
#pragma unroll
        for (int t = 0; t < C; ++t) {
            // the waiting-time word's slot (j = -1) and the padded ones have rate 0: they add 0 to a0 and never win
            const float4 av = reinterpret_cast<const float4 *>(a)[lane + 32 * (t0 + t)];
            const float aq[4] = {av.x, av.y, av.z, av.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                a0p = __fadd_rn(a0p, aq[q]);
                warp_top_add(top, aq[q], word_of(r[t], q), 4 * (t0 + t) + q);
            }
        }
    };
    int t0 = 0;
    for (; t0 + 4 <= n_rounds; t0 += 4) rounds(std::integral_constant<int, 4>{}, t0);
    if (n_rounds & 2) {
        rounds(std::integral_constant<int, 2>{}, t0);
        t0 += 2;
    }
    if (n_rounds & 1) rounds(std::integral_constant<int, 1>{}, t0);
    a0 = warp_sum(a0p);
    E0 = neg_log_unit(u01(__shfl_sync(0xffffffffu, x0, 0)));
    int src, slot;
    const bool sure = warp_top_decide(top, a0, [&](int s) { return a[4 * (lane + 32 * min(s >> 2, n_rounds - 1)) + (s & 3)]; }, src, slot);
    if (sure && n_rounds <= 16) jb = 4 * (src + 32 * (slot >> 2)) + (slot & 3) - 1;
    else jb = warp_race_exact(n_rounds, a, k, z);
}

// Bin readout (Section 4.4) on a warp-per-trajectory forward. Every lane runs the same bookkeeping on the
// same values (the running integrals, the edges found by bisection, the slot count); lane 0 stores the bin an
// interval's first edge closes and the slot record, and whole bins held at one state are written by the
// warp along the trajectory's own row (consecutive lanes on consecutive floats). The values are those of
// the thread kernels' bin readout.
template <class XF>
__device__ __forceinline__ void warp_bin_held(const FwdParams &p, int64_t i, int lo, int hi, const XF &xobs, bool zero)
{
    if (lo > hi) return;
    const int lane = threadIdx.x & 31, no = p.n_obs;
    float xv[kBinMaxObs];
#pragma unroll
    for (int c = 0; c < kBinMaxObs; ++c) xv[c] = (c < no && !zero) ? obs_f(xobs(c)) : 0.0f;
    float *row = static_cast<float *>(p.obs_out) + i * (int64_t)p.S * no;
    for (int64_t e = (int64_t)lo * no + lane; e < (int64_t)(hi + 1) * no; e += 32) {
        const int c = no == 1 ? 0 : (int)(e % no);
        float v = xv[0];
#pragma unroll
        for (int c2 = 1; c2 < kBinMaxObs; ++c2) v = c == c2 ? xv[c2] : v;
        row[e] = v;
    }
}

template <bool RECORD, class XF>
__device__ __forceinline__ void warp_bin_first_edge(const FwdParams &p, int64_t i, int s, double t_k, int k,
                                                    float (&acc)[kBinMaxObs], const XF &xobs, int &slots, bool zero)
{
    float o[kBinMaxObs];
    const float d = bin_close(acc, xobs, p.n_obs, p.ts, s, t_k, true, o);
    if ((threadIdx.x & 31) == 0) {
        float *dst = static_cast<float *>(p.obs_out) + ((int64_t)i * p.S + s) * p.n_obs;
        for (int c = 0; c < p.n_obs; ++c) dst[c] = zero ? 0.0f : o[c];
        if (RECORD) {
            const int64_t at = (int64_t)slots * p.n_traj + i;
            p.brk_k[at] = k;
            p.brk_s[at] = s;
            p.brk_a[at] = d;
        }
    }
    if (RECORD) ++slots;
}

// the edges in the state interval [t_k, t_next) from s on; returns the first edge at or after t_next
template <bool RECORD, class XF>
__device__ __forceinline__ int warp_bin_edges(const FwdParams &p, int64_t i, int s, double t_k, double t_next, int k,
                                              float (&acc)[kBinMaxObs], const XF &xobs, int &slots)
{
    int lo = s, hi = p.S;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (gt_nonneg(t_next, p.ts[mid])) lo = mid + 1;
        else hi = mid;
    }
    if (lo > s) {
        warp_bin_first_edge<RECORD>(p, i, s, t_k, k, acc, xobs, slots, false);
        warp_bin_held(p, i, s + 1, lo - 1, xobs, false);
    }
    return lo;
}

// after the last state (held from t_k on): close the first remaining bin, hold the rest, record the slot count
template <bool RECORD, class XF>
__device__ __forceinline__ void warp_bin_tail(const FwdParams &p, int64_t i, int s, double t_k, int k,
                                              float (&acc)[kBinMaxObs], const XF &xobs, bool bad_obs, int &slots)
{
    if (s < p.S) {
        warp_bin_first_edge<RECORD>(p, i, s, t_k, k, acc, xobs, slots, bad_obs);
        warp_bin_held(p, i, s + 1, p.S - 1, xobs, bad_obs);
    }
    if (RECORD && (threadIdx.x & 31) == 0) p.brk_tail[i] = slots;
}

// Per-trajectory body of the warp forward (all 32 lanes of one warp); X, a = this warp's counts and propensities.
template <int READOUT, bool RECORD>
__device__ __forceinline__ void warp_fwd_body(const FwdParams &p, const WarpTab &tab, int *X, float *a, const int64_t i)
{
    const int lane = threadIdx.x & 31;
    const int N = p.N;
    const int64_t n = p.n_traj;

    const int *x0 = p.x0 + (p.x0_per_traj ? i * N : 0);
    const bool bad_obs = (*p.flag & kErrBadObs) != 0;
    bool neg = false;
    for (int s = lane; s < N; s += 32) {
        X[s] = x0[s];
        neg |= x0[s] < 0;
    }
    const bool bad_input = __any_sync(0xffffffffu, neg) || (*p.flag & (kErrBadSamples | kErrBadObs)) != 0;
    __syncwarp();
    const uint64_t gid = p.traj_offset + (uint64_t)i;
    const WarpNoise noise{(uint32_t)gid, (uint32_t)(gid >> 32), (uint32_t)p.seed, (uint32_t)(p.seed >> 32)};
    if (!bad_input) warp_propensities_all<false>(tab, X, a);

    double t = 0.0;
    int s = 0;
    double thr = p.S > 0 ? p.ts[0] : p.t_end;
    int status = bad_input ? SSA_TRAJ_BAD_INPUT : SSA_TRAJ_OK;
    int k = 0, draws = 0, ck_left = p.K, ck_row = 0;
    uint32_t e0 = 0, e1 = 0, e2 = 0, e3 = 0;
    constexpr bool kBin = READOUT == SSA_READOUT_BIN;
    float bacc[kBinMaxObs];
    int osp[kBinMaxObs];
#pragma unroll
    for (int c = 0; c < kBinMaxObs; ++c) {
        bacc[c] = 0.0f;
        osp[c] = (kBin && c < p.n_obs && !bad_obs) ? p.obs_sp[c] : 0;
    }
    auto xobs = [&](int c) { return X[osp[c]]; };
    int slots = 0;

    while (!bad_input) {
        if (k >= p.max_steps) { status = SSA_TRAJ_STEP_CAP; break; }
        float a0, E0;
        int jb;
        warp_step_eval(tab.rounds, k, noise, a, a0, E0, jb);
        if (!(a0 < CUDART_INF_F)) { status = SSA_TRAJ_BAD_RATE; break; }
        if (a0 == 0.0f) { status = SSA_TRAJ_ABSORBED; break; }
        if (jb < 0) { status = SSA_TRAJ_BAD_RATE; break; }
        const float tau = waiting_time(E0, a0);
        const double t_next = t + f2d_pos(tau);
        const int jpb = jpos(jb, tab.nb);
        const int4 rj = tab.rx[jpb];
        const bool slow = gt_nonneg(t_next, thr);
        const bool cross = slow && gt_nonneg(t_next, p.t_end);
        if (!cross) {
            bool bad_neg = false, bad_ovf = false;
            if (rj.w - rj.z <= 4) {
                const int e = reinterpret_cast<const int *>(tab.ent + wpos(jb))[lane & 3];
                const int x = X[min(ent_species(e), N - 1)], d = (int)ent_change(e);
                bad_neg = x + d < 0 && d < 0;
                bad_ovf = d > 0 && x > 2147483647 - d;
            } else for (int e = rj.z + lane; e < rj.w; e += 32) {
                const int st = tab.st[e];
                const int x = X[stoich_species(st)], d = stoich_delta(st);
                bad_neg |= d < 0 && x + d < 0;
                bad_ovf |= d > 0 && x > 2147483647 - d;
            }
            if (__any_sync(0xffffffffu, bad_neg || bad_ovf))
                status = __any_sync(0xffffffffu, bad_neg) ? SSA_TRAJ_NEG_COUNT : SSA_TRAJ_OVERFLOW;
        }
        if (RECORD) {
            e0 = __funnelshift_r(e0, e1, 16);
            e1 = __funnelshift_r(e1, e2, 16);
            e2 = __funnelshift_r(e2, e3, 16);
            e3 = (e3 >> 16) | ((uint32_t)jb << 16);
            if (lane == 0 && (k & 7) == 7) p.ev[(int64_t)(k >> 3) * n + i] = make_uint4(e0, e1, e2, e3);
        }
        draws = k + 1;
        if (status != SSA_TRAJ_OK) break;
        if (slow && kBin) {
            const int s_first = s;
            s = warp_bin_edges<RECORD>(p, i, s, t, t_next, k, bacc, xobs, slots);
            if (!cross && s > s_first) bin_accumulate(bacc, xobs, p.n_obs, d2f_nonneg(t_next - p.ts[s - 1]));
            thr = s < p.S ? p.ts[s] : p.t_end;
            if (cross) break;
        } else if (kBin) {
            bin_accumulate(bacc, xobs, p.n_obs, tau);
        }
        if (slow && !kBin) {
            while (s < p.S && gt_nonneg(t_next, p.ts[s])) {
                if (READOUT == SSA_READOUT_HOLD) {
                    int *o = static_cast<int *>(p.obs_out) + ((int64_t)i * p.S + s) * p.n_obs;
                    for (int c = lane; c < p.n_obs; c += 32) o[c] = X[p.obs_sp[c]];
                } else {
                    const float alpha = __fdiv_rn(d2f_nonneg(p.ts[s] - t), tau);
                    float *o = static_cast<float *>(p.obs_out) + ((int64_t)i * p.S + s) * p.n_obs;
                    for (int c = lane; c < p.n_obs; c += 32) {
                        const int sp = p.obs_sp[c];
                        int dv = 0;
                        for (int e = rj.z; e < rj.w; ++e)
                            if (stoich_species(tab.st[e]) == sp) dv += stoich_delta(tab.st[e]);
                        o[c] = __fmaf_rn(alpha, (float)dv, (float)X[sp]);
                    }
                    if (RECORD && lane == 0) p.brk_a[(int64_t)s * n + i] = alpha;
                }
                if (RECORD && lane == 0) p.brk_k[(int64_t)s * n + i] = k;
                ++s;
            }
            thr = s < p.S ? p.ts[s] : p.t_end;
            if (cross) break;
        }
        __syncwarp();
        warp_apply<false>(tab, jb, 1, X, a);
        t = t_next;
        ++k;
        if (RECORD && --ck_left == 0) {
            ck_left = p.K;
            ++ck_row;
            int *ck = p.ckpt + (int64_t)ck_row * N * n + i;
            for (int sp = lane; sp < N; sp += 32) ck[(int64_t)sp * n] = X[sp];
        }
    }
    __syncwarp();
    if constexpr (kBin) warp_bin_tail<RECORD>(p, i, s, t, k, bacc, xobs, bad_obs, slots);
    for (; !kBin && s < p.S; ++s) {
        if (READOUT == SSA_READOUT_HOLD) {
            int *o = static_cast<int *>(p.obs_out) + ((int64_t)i * p.S + s) * p.n_obs;
            for (int c = lane; c < p.n_obs; c += 32) o[c] = bad_obs ? 0 : X[p.obs_sp[c]];
        } else {
            float *o = static_cast<float *>(p.obs_out) + ((int64_t)i * p.S + s) * p.n_obs;
            for (int c = lane; c < p.n_obs; c += 32) o[c] = bad_obs ? 0.0f : (float)X[p.obs_sp[c]];
            if (RECORD && lane == 0) p.brk_a[(int64_t)s * n + i] = -1.0f;
        }
        if (RECORD && lane == 0) p.brk_k[(int64_t)s * n + i] = k;
    }
    if (lane == 0) {
        p.draws[i] = draws;
        p.status[i] = status;
    }
    if (RECORD) {
        if ((draws & 7) && lane == 0) {
            for (int pad = draws & 7; pad < 8; ++pad) {
                e0 = __funnelshift_r(e0, e1, 16);
                e1 = __funnelshift_r(e1, e2, 16);
                e2 = __funnelshift_r(e2, e3, 16);
                e3 = e3 >> 16;
            }
            p.ev[(int64_t)((draws - 1) >> 3) * n + i] = make_uint4(e0, e1, e2, e3);
        }
        for (int sp = lane; sp < N; sp += 32) {
            p.xfinal[(int64_t)sp * n + i] = X[sp];
            p.ckpt[(int64_t)sp * n + i] = x0[sp];
        }
    }
}

// One step of the soft forward (Section 3.3, Eq. 4) at the real state X, all 32 lanes: lane l evaluates the
// reactions of its Philox blocks (relaxed propensities with negative factors clipped at 0, keys
// l_j = log2 a_j - log2 E_j), the warp reduces a0 and the largest key, the lanes turn their keys into
// unnormalised weights w_j = exp2((l_j - l_max)/T) (kept in y by lane-major position), and each species sums
// its own change dX_s = sum_j (w_j / Z) v_js through the species-major update list in increasing j (no atomics:
// the specialised thread kernels' order of the update). With AH, a_j and h_j are kept too (the adjoint's
// re-evaluation). Returns a0; sets E0, invZ = 1/Z and whether X + dX is finite. The forward and the adjoint's
// segment re-runs call this one function, so the regenerated states are the forward's bit for bit.
template <bool AH>
__device__ __forceinline__ float warp_soft_step(const int4 *s_rx, const float *s_k, const int *s_upd, int N, int M,
                                                float invT, int k, uint32_t c2, uint32_t c3, uint32_t key0,
                                                uint32_t key1, const float *X, float *a_out, float *h_out, float *y,
                                                float *dX, float &E0, float &invZ, bool &finite)
{
    const int lane = threadIdx.x & 31, nb = (M + 4) >> 2;
    const int upd_base = (N + 1 + 3) & ~3;  // the list follows the padded pointer array
    float a0p = 0.0f, lmaxp = -CUDART_INF_F;
    E0 = 0.0f;
    for (int b = lane; b < nb; b += 32) {
        const uint4 r = philox4x32_10(make_uint4((uint32_t)b, (uint32_t)k, c2, c3), key0, key1);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            // predicated: the waiting-time word's slot (j = -1) and the padded ones have rate 0 (they add 0 to
            // a0 and have key -inf), and the factor is chosen by selects rather than by branches on the order
            const int j = 4 * b + q - 1;
            const float E = neg_log_unit(u01(word_of(r, q)));
            if (q == 0 && j < 0) E0 = E;
            const int pos = q * nb + b;
            const int4 rx = s_rx[pos];
            const float x1 = X[rx.x >= 0 ? rx.x : 0], x2 = X[rx.y >= 0 ? rx.y : 0];
            const float h = rx.x < 0 ? 1.0f : rx.y < 0 ? hs_first(x1) : rx.y == rx.x ? hs_homodimer(x1) : hs_hetero(x1, x2);
            const float a = __fmul_rn(s_k[pos], h);
            a0p = __fadd_rn(a0p, a);
            const float l = a > 0.0f ? log2f(a) - log2f(E) : -CUDART_INF_F;
            if (j >= 0 && j < M) {
                y[pos] = l;
                if (AH) {
                    a_out[pos] = a;
                    h_out[pos] = h;
                }
            }
            lmaxp = fmaxf(lmaxp, l);
        }
    }
    const float a0 = warp_sum(a0p), lmax = warp_max(lmaxp);
    E0 = __shfl_sync(0xffffffffu, E0, 0);
    float Zp = 0.0f;
    for (int b = lane; b < nb; b += 32) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int j = 4 * b + q - 1;
            const bool live = j >= 0 && j < M;
            const int pos = q * nb + b;
            const float l = live ? y[pos] : -CUDART_INF_F;
            const float w = l == -CUDART_INF_F ? 0.0f : exp2f((l - lmax) * invT);
            if (live) y[pos] = w;
            Zp += w;  // + 0 outside the live slots: the same bits
        }
    }
    invZ = __fdividef(1.0f, warp_sum(Zp));
    __syncwarp();
    bool fin = true;
    for (int sp = lane; sp < N; sp += 32) {
        float d = 0.0f;
        for (int e = s_upd[sp]; e < s_upd[sp + 1]; ++e) {
            const int ent = s_upd[upd_base + e];
            d = __fmaf_rn(y[ent >> 8] * invZ, (float)(int)(signed char)(ent & 0xff), d);
        }
        dX[sp] = d;
        fin &= fabsf(__fadd_rn(X[sp], d)) < CUDART_INF_F;
    }
    finite = __all_sync(0xffffffffu, fin);
    __syncwarp();
    return a0;
}

// Per-trajectory body of the warp soft forward (Eq. 4). Clock, samples and readouts are the forward's;
// recorded, the float state is checkpointed every kSoftK steps ([n_ckpt][N][n_traj], checkpoint 0 = X_0) with
// the sample brackets, for the adjoint's segment re-runs.
template <int READOUT, bool RECORD>
__device__ __forceinline__ void warp_soft_fwd_body(const FwdParams &p, const int4 *s_rx, const float *s_k,
                                                   const int *s_upd, float *X, float *dX, float *y, const int64_t i)
{
    const int lane = threadIdx.x & 31;
    const int N = p.N, M = p.M;
    const int64_t n = p.n_traj;
    const int *x0 = p.x0 + (p.x0_per_traj ? i * N : 0);
    const bool bad_obs = (*p.flag & kErrBadObs) != 0;
    bool neg = false;
    for (int sp = lane; sp < N; sp += 32) {
        X[sp] = int2f(x0[sp]);
        neg |= x0[sp] < 0;
    }
    const bool bad_input = __any_sync(0xffffffffu, neg) || (*p.flag & (kErrBadSamples | kErrBadObs)) != 0;
    __syncwarp();
    const uint64_t gid = p.traj_offset + (uint64_t)i;
    const uint32_t c2 = (uint32_t)gid, c3 = (uint32_t)(gid >> 32), key0 = (uint32_t)p.seed,
                   key1 = (uint32_t)(p.seed >> 32);
    double t = 0.0;
    int s = 0;
    double thr = p.S > 0 ? p.ts[0] : p.t_end;
    int status = bad_input ? SSA_TRAJ_BAD_INPUT : SSA_TRAJ_OK;
    int k = 0, draws = 0, ck_left = p.K, ck_row = 0;
    constexpr bool kBin = READOUT == SSA_READOUT_BIN;
    float bacc[kBinMaxObs];
    int osp[kBinMaxObs];
#pragma unroll
    for (int c = 0; c < kBinMaxObs; ++c) {
        bacc[c] = 0.0f;
        osp[c] = (kBin && c < p.n_obs && !bad_obs) ? p.obs_sp[c] : 0;
    }
    auto xobs = [&](int c) { return X[osp[c]]; };
    int slots = 0;
    float *obs = static_cast<float *>(p.obs_out);
    float *ckf = reinterpret_cast<float *>(p.ckpt);

    while (!bad_input) {
        if (k >= p.max_steps) { status = SSA_TRAJ_STEP_CAP; break; }
        float E0, invZ;
        bool finite;
        const float a0 = warp_soft_step<false>(s_rx, s_k, s_upd, N, M, p.invT, k, c2, c3, key0, key1, X, nullptr,
                                               nullptr, y, dX, E0, invZ, finite);
        if (!(a0 < CUDART_INF_F)) { status = SSA_TRAJ_BAD_RATE; break; }
        if (a0 == 0.0f) { status = SSA_TRAJ_ABSORBED; break; }
        const float tau = waiting_time(E0, a0);
        const double t_next = t + f2d_pos(tau);
        const bool slow = gt_nonneg(t_next, thr);
        const bool cross = slow && gt_nonneg(t_next, p.t_end);
        draws = k + 1;
        if (!cross && !finite) { status = SSA_TRAJ_BAD_RATE; break; }
        if (slow && kBin) {
            const int s_first = s;
            s = warp_bin_edges<RECORD>(p, i, s, t, t_next, k, bacc, xobs, slots);
            if (!cross && s > s_first) bin_accumulate(bacc, xobs, p.n_obs, d2f_nonneg(t_next - p.ts[s - 1]));
            thr = s < p.S ? p.ts[s] : p.t_end;
            if (cross) break;
        } else if (kBin) {
            bin_accumulate(bacc, xobs, p.n_obs, tau);
        }
        if (slow && !kBin) {
            while (s < p.S && gt_nonneg(t_next, p.ts[s])) {
                float *o = obs + ((int64_t)i * p.S + s) * p.n_obs;
                if (READOUT == SSA_READOUT_HOLD) {
                    for (int c = lane; c < p.n_obs; c += 32) o[c] = X[p.obs_sp[c]];
                } else {
                    const float alpha = __fdiv_rn(d2f_nonneg(p.ts[s] - t), tau);
                    for (int c = lane; c < p.n_obs; c += 32) {
                        const int sp = p.obs_sp[c];
                        o[c] = __fmaf_rn(alpha, dX[sp], X[sp]);
                    }
                    if (RECORD && lane == 0) p.brk_a[(int64_t)s * n + i] = alpha;
                }
                if (RECORD && lane == 0) p.brk_k[(int64_t)s * n + i] = k;
                ++s;
            }
            thr = s < p.S ? p.ts[s] : p.t_end;
            if (cross) break;
        }
        __syncwarp();
        for (int sp = lane; sp < N; sp += 32) X[sp] = __fadd_rn(X[sp], dX[sp]);
        __syncwarp();
        t = t_next;
        ++k;
        if (RECORD && --ck_left == 0) {
            ck_left = p.K;
            ++ck_row;
            for (int sp = lane; sp < N; sp += 32) ckf[((int64_t)ck_row * N + sp) * n + i] = X[sp];
        }
    }
    __syncwarp();
    if constexpr (kBin) warp_bin_tail<RECORD>(p, i, s, t, k, bacc, xobs, bad_obs, slots);
    for (; !kBin && s < p.S; ++s) {
        float *o = obs + ((int64_t)i * p.S + s) * p.n_obs;
        for (int c = lane; c < p.n_obs; c += 32) o[c] = bad_obs ? 0.0f : X[p.obs_sp[c]];
        if (RECORD && lane == 0) {
            if (READOUT == SSA_READOUT_LINEAR) p.brk_a[(int64_t)s * n + i] = -1.0f;
            p.brk_k[(int64_t)s * n + i] = k;
        }
    }
    if (lane == 0) {
        p.draws[i] = draws;
        p.status[i] = status;
    }
    if (RECORD)
        for (int sp = lane; sp < N; sp += 32) ckf[(int64_t)sp * n + i] = int2f(x0[sp]);  // checkpoint 0 = X_0
}

// Exact gradient of the soft forward on the warp layout, one trajectory (all 32 lanes): the specialised thread
// kernels' soft adjoint in the warp's arrays. Segment by segment from the end, the kSoftK states are
// regenerated from the float checkpoint with the forward's own step (the state after a segment must equal the
// next checkpoint bit for bit), then walked back: the step is evaluated again at X_k, the readout terms give
// the waiting-time adjoint, w_j = v_j . lambda, psi_j = y~_j (w_j - sum y~ w) / T, dA_j += psi_j + dL/da0 a_j,
// and every reactant slot's contribution (choice path and waiting-time path, clipped where a factor is) is
// gathered per species through the reactant-slot incidence list in increasing j, added to lambda in that
// order. Per-warp arrays: Xs [kSoftK][Npad], lam, dX [Npad]; a, h, y, c1, c2 [Mp]; dA [Mp] accumulates.
template <int READOUT>
__device__ __forceinline__ void warp_soft_adj_body(const AdjParams &p, const int4 *s_rx, const int *s_st,
                                                   const int *s_inc_ptr, const int *s_inc, const float *s_k,
                                                   const int *s_upd, float *Xs, float *lam, float *dX, float *aj,
                                                   float *hj, float *y, float *c1, float *c2, float *dA,
                                                   const int64_t i, const int st)
{
    const int lane = threadIdx.x & 31;
    const int N = p.N, M = p.M, nb = (M + 4) >> 2, Npad = (N + 3) & ~3;
    const int64_t n = p.n_traj;
    const int d = p.draws[i];
    const int L = (st == SSA_TRAJ_OK) ? d - 1 : d;  // index of the last visited state
    const bool draw_last = st == SSA_TRAJ_OK;
    const int K = p.K;  // kSoftK
    const uint64_t gid = p.traj_offset + (uint64_t)i;
    const uint32_t c2w = (uint32_t)gid, c3w = (uint32_t)(gid >> 32), key0 = (uint32_t)p.seed,
                   key1 = (uint32_t)(p.seed >> 32);
    const float invT = p.invT;
    const float *gl = p.dl_dobs + i * p.dl_stride;
    const float *ckf = reinterpret_cast<const float *>(p.ckpt);
    for (int sp = lane; sp < N; sp += 32) lam[sp] = 0.0f;
    int s_hi = p.S - 1;
    int brk_next = (READOUT != SSA_READOUT_BIN && s_hi >= 0) ? p.brk_k[(int64_t)s_hi * n + i] : -1;
    constexpr bool kBin = READOUT == SSA_READOUT_BIN;
    BinSlots bslots{-1, -1};
    float d_first = 0.0f, d_last = 0.0f;
    if (kBin) bin_slots_init(bslots, p.brk_k, p.brk_tail, n, i);
    float mu = 0.0f;
    int mism = 0;
    float gq[kBinMaxObs], gk[kBinMaxObs];
    int osp[kBinMaxObs];
#pragma unroll
    for (int c = 0; c < kBinMaxObs; ++c) osp[c] = (kBin && c < p.n_obs) ? p.obs_sp[c] : 0;
    auto addx = [&](int c, float v) { lam[osp[c]] += v; };
    if (kBin) bin_grad(gq, gl, p.n_obs, p.ts, p.S, p.S);
    __syncwarp();

    for (int c = L / K; c >= 0; --c) {
        const int k0 = c * K, k1 = min(k0 + K - 1, L);
        // regenerate the segment's states: Xs[kk - k0] = X_kk
        for (int sp = lane; sp < N; sp += 32) Xs[sp] = ckf[((int64_t)c * N + sp) * n + i];
        __syncwarp();
        for (int kk = k0; kk < k1 || (kk == k1 && k1 < L); ++kk) {
            const float *Xc = Xs + (size_t)(kk - k0) * Npad;
            float E0, invZ;
            bool finite;
            warp_soft_step<false>(s_rx, s_k, s_upd, N, M, invT, kk, c2w, c3w, key0, key1, Xc, nullptr, nullptr, y, dX,
                                  E0, invZ, finite);
            if (kk < k1) {
                float *Xn = Xs + (size_t)(kk + 1 - k0) * Npad;
                for (int sp = lane; sp < N; sp += 32) Xn[sp] = __fadd_rn(Xc[sp], dX[sp]);
            } else {  // the state after the segment: the next checkpoint
                int bad = 0;
                for (int sp = lane; sp < N; sp += 32)
                    bad += __fadd_rn(Xc[sp], dX[sp]) != ckf[((int64_t)(c + 1) * N + sp) * n + i];
                mism += __reduce_add_sync(0xffffffffu, bad);
            }
            __syncwarp();
        }
        for (int k = k1; k >= k0; --k) {
            const float *Xk = Xs + (size_t)(k - k0) * Npad;
            const bool draw = (k < L) || draw_last;
            const int s_top = s_hi;
            if (kBin) {
                bin_slots_step(bslots, p.brk_k, p.brk_s, p.brk_a, p.ts, n, i, k, s_hi, d_first, d_last);
                if (s_hi < s_top) bin_grad(gk, gl, p.n_obs, p.ts, p.S, s_hi + 1);
                else {
#pragma unroll
                    for (int q = 0; q < kBinMaxObs; ++q) gk[q] = gq[q];
                }
            } else {
                while (s_hi >= 0 && brk_next == k) {
                    --s_hi;
                    brk_next = s_hi >= 0 ? p.brk_k[(int64_t)s_hi * n + i] : -1;
                }
            }
            float tau_k = 0.0f;
            if (draw) {
                float E0, invZ;
                bool finite;
                const float a0 = warp_soft_step<true>(s_rx, s_k, s_upd, N, M, invT, k, c2w, c3w, key0, key1, Xk, aj,
                                                      hj, y, dX, E0, invZ, finite);
                const float tau = waiting_time(E0, a0);
                tau_k = tau;
                float dt_dir = 0.0f, dtau_dir = 0.0f;
                if (kBin) {  // t_{k+1} ends this interval and starts the next, in the bin of gq
                    float cb = 0.0f;
#pragma unroll
                    for (int q = 0; q < kBinMaxObs; ++q)
                        if (q < p.n_obs) cb = __fmaf_rn(gq[q], dX[osp[q]], cb);
                    mu -= cb;
                }
                if (READOUT == SSA_READOUT_LINEAR) {
                    // serial on lane 0 (observed species may repeat), broadcast afterwards
                    if (lane == 0) {
                        for (int s = s_hi + 1; s <= s_top; ++s) {
                            const float alpha = p.brk_a[(int64_t)s * n + i];
                            if (alpha < 0.0f) continue;
                            float cl = 0.0f;
                            for (int o = 0; o < p.n_obs; ++o) {
                                const float g = gl[(int64_t)s * p.n_obs + o];
                                const int sp = p.obs_sp[o];
                                lam[sp] += alpha * g;
                                cl += g * dX[sp];
                            }
                            const float c_tau = __fdividef(cl, tau);
                            dt_dir -= c_tau;
                            dtau_dir -= alpha * c_tau;
                        }
                    }
                    dt_dir = __shfl_sync(0xffffffffu, dt_dir, 0);
                    dtau_dir = __shfl_sync(0xffffffffu, dtau_dir, 0);
                }
                __syncwarp();
                const float dtau = mu + dtau_dir;
                const float dLda0 = -dtau * tau / a0;
                // w_j = v_j . lambda (kept in c1 until the slots take it) and sum_j y~_j w_j
                float Wp = 0.0f;
                for (int b = lane; b < nb; b += 32) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int j = 4 * b + q - 1;
                        if (j < 0 || j >= M) continue;
                        const int pos = q * nb + b;
                        const int4 rx = s_rx[pos];
                        float w = 0.0f;
                        for (int e = rx.z; e < rx.w; ++e) w += (float)stoich_delta(s_st[e]) * lam[stoich_species(s_st[e])];
                        c1[pos] = w;
                        Wp += (y[pos] * invZ) * w;
                    }
                }
                const float Wbar = warp_sum(Wp);
                __syncwarp();
                // psi, dA and the reactant-slot contributions (choice path where a > 0, waiting-time path where
                // the factor is not clipped)
                for (int b = lane; b < nb; b += 32) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int j = 4 * b + q - 1;
                        if (j < 0 || j >= M) continue;
                        const int pos = q * nb + b;
                        const float yj = y[pos] * invZ, a = aj[pos];
                        const float psi = yj > 0.0f ? yj * (c1[pos] - Wbar) * invT : 0.0f;
                        dA[pos] += psi + dLda0 * a;
                        const float ctau = dLda0 * s_k[pos];
                        const int4 rx = s_rx[pos];
                        float v1 = 0.0f, v2 = 0.0f;
                        if (rx.x >= 0) {
                            const float x1 = Xk[rx.x];
                            if (rx.y < 0) {
                                v1 = sadj_first(x1, a, psi, x1 < 0.0f ? 0.0f : ctau);
                            } else if (rx.y == rx.x) {
                                v1 = sadj_homodimer(x1, a, hj[pos], psi, __fmul_rn(x1, x1 - 1.0f) < 0.0f ? 0.0f : ctau);
                            } else {
                                const float x2 = Xk[rx.y];
                                const float cc = __fmul_rn(x1, x2) < 0.0f ? 0.0f : ctau;
                                v1 = sadj_hetero(x1, x2, a, psi, cc);
                                v2 = sadj_hetero(x2, x1, a, psi, cc);
                            }
                        }
                        c1[pos] = v1;
                        c2[pos] = v2;
                    }
                }
                __syncwarp();
                // lambda_s += the contributions of its reactant slots, one at a time in increasing j
                for (int sp = lane; sp < N; sp += 32) {
                    float acc = lam[sp];
                    for (int e = s_inc_ptr[sp]; e < s_inc_ptr[sp + 1]; ++e) {
                        const int slot = s_inc[e];  // 2 j + reactant slot
                        acc += ((slot & 1) ? c2 : c1)[jpos(slot >> 1, nb)];
                    }
                    lam[sp] = acc;
                }
                mu += dt_dir;
            }
            __syncwarp();
            if (kBin) {
                if (lane == 0)
                    bin_state_terms(addx, d_first, d_last, gl, p.bin_prefix, p.n_obs, s_hi + 1, s_top, draw, tau_k, gq,
                                    gk);
#pragma unroll
                for (int q = 0; q < kBinMaxObs; ++q) gq[q] = gk[q];
            } else if (lane == 0) {
                for (int s = s_hi + 1; s <= s_top; ++s) {
                    float coef = 1.0f;
                    if (READOUT == SSA_READOUT_LINEAR && draw) {
                        const float alpha = p.brk_a[(int64_t)s * n + i];
                        if (alpha >= 0.0f) coef = 1.0f - alpha;
                    }
                    for (int o = 0; o < p.n_obs; ++o) lam[p.obs_sp[o]] += coef * gl[(int64_t)s * p.n_obs + o];
                }
            }
            __syncwarp();
        }
    }
    if (lane == 0 && mism) atomicAdd(p.mismatch, mism);
}

// The keys of a step whose a0 lies where a_j / E_j could leave the binary32 range, scaled by a power of two (all
// that follows uses ratios of keys); returns the largest. hot (hot_weights): the eighth root of each key's ratio to the
// largest instead, from its log2, so that no positive key flushes; the weights' exponent is then 8/T.
static __device__ __noinline__ float warp_keys_scaled(int rounds, const float *ad, int k, WarpNoise z, float a0, bool hot,
                                                      float *rj)
{
    if (hot) {
        const int lane = threadIdx.x & 31;
        float top = -CUDART_INF_F;
        for (int c = 0; c < rounds; ++c) {
            const uint4 r = philox4x32_10(make_uint4((uint32_t)(32 * c + lane), (uint32_t)k, z.c2, z.c3), z.key0, z.key1);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int w = 4 * (32 * c + lane) + q;
                rj[w] = key_log2(fmaxf(ad[w], 0.0f), inv_exp_of_word(word_of(r, q)));
                top = fmaxf(top, rj[w]);
            }
        }
        top = warp_max(top);
        for (int c = 0; c < rounds; ++c)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int w = 4 * (32 * c + lane) + q;
                rj[w] = ex2_approx((rj[w] - top) * 0.125f);
            }
        return 1.0f;
    }
    const float sc = key_scale(a0);
    const int lane = threadIdx.x & 31;
    float rmax = 0.0f;
    for (int c = 0; c < rounds; ++c) {
        const uint4 r = philox4x32_10(make_uint4((uint32_t)(32 * c + lane), (uint32_t)k, z.c2, z.c3), z.key0, z.key1);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int w = 4 * (32 * c + lane) + q;
            const float key = (fmaxf(ad[w], 0.0f) * sc) * inv_exp_of_word(word_of(r, q));
            rmax = fmaxf(rmax, key);
            rj[w] = key;
        }
    }
    return warp_max_nonneg(rmax);
}

// Per-trajectory body of the warp adjoint (all 32 lanes). X, lam [Npad], ad, rj, ct, dA [wide_len] are this warp's
// buffers, contiguous in that order (lam[N] is read as 0: a padding word, or ad[0], the waiting-time word's slot);
// dA accumulates over every trajectory the warp processes.
// Per step: the keys (pass 1), soft weights and w_j = v_j . lambda (pass 2), the per-reaction
// adjoints g_j = psi_j + dL/da0 a_j (pass 3), which are also all that the state adjoint needs: a_j is
// proportional to the count of each plain reactant, so lambda_s += (1/X_s) sum g_j over the reactions of s, a
// homodimer's share carries (2 X - 1) / (X (X - 1)), and where a reactant is absent (a_j = 0) only the
// waiting-time path remains, dL/da0 D_j. One division per species replaces two per reaction.
template <int READOUT, bool HOT>
__device__ __forceinline__ void warp_adj_body(const AdjParams &p, const WarpTab &tab, int *X, float *lam, float *ad,
                                              float *rj, float *ct, float *dA, const int64_t i, const int st)
{
    const int lane = threadIdx.x & 31;
    const int N = p.N, nb = tab.nb, n_rounds = tab.rounds;
    const int64_t n = p.n_traj;
    const int d = p.draws[i];
    const int L = (st == SSA_TRAJ_OK) ? d - 1 : d;
    for (int s = lane; s < N; s += 32) {
        X[s] = p.xfinal[(int64_t)s * n + i];
        lam[s] = 0.0f;
    }
    for (int s = N + lane; s < ((N + 3) & ~3); s += 32) lam[s] = 0.0f;
    __syncwarp();
    warp_propensities_all<true>(tab, X, ad);
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
    constexpr bool kBin = READOUT == SSA_READOUT_BIN;
    int s_hi = p.S - 1;
    int brk_next = (!kBin && s_hi >= 0) ? p.brk_k[(int64_t)s_hi * n + i] : -1;
    // BIN readout: the recorded slots (one per state interval with edges), gq = g of the bin that contains
    // t_{k+1}, xo = X_{k+1} at the observables; every lane keeps the same copies
    BinSlots bslots{-1, -1};
    float d_first = 0.0f, d_last = 0.0f;
    float gq[kBinMaxObs], gk[kBinMaxObs];
    int osp[kBinMaxObs], xo[kBinMaxObs];
#pragma unroll
    for (int c = 0; c < kBinMaxObs; ++c) osp[c] = (kBin && c < p.n_obs) ? p.obs_sp[c] : 0;
    auto xobs = [&](int c) { return X[osp[c]]; };
    auto addx = [&](int c, float v) { lam[osp[c]] += v; };
    if (kBin) {
        bin_slots_init(bslots, p.brk_k, p.brk_tail, n, i);
        bin_grad(gq, gl, p.n_obs, p.ts, p.S, p.S);
#pragma unroll
        for (int c = 0; c < kBinMaxObs; ++c) xo[c] = c < p.n_obs ? xobs(c) : 0;
    }
    float mu = 0.0f;
    int mism = 0;
    int ck_row = L / p.K, ck_off = L - ck_row * p.K;
    // species groups of the state adjoint: with N <= 32 each species gets 32 / 2^ceil(log2 N) lanes that stride over
    // its list and combine by a butterfly inside the group; with more species each lane takes whole species
    int pow2 = 1;
    while (pow2 < N && pow2 < 32) pow2 <<= 1;
    const int gsz = N <= 32 ? 32 / pow2 : 1;
    const int g_first = lane / gsz, g_lane = lane % gsz, g_step = 32 / gsz;

    for (int k = L; k >= 0; --k) {
        const bool draw = (k < L) || (st == SSA_TRAJ_OK);
        const int s_top = s_hi;
        if (kBin) {
            bin_slots_step(bslots, p.brk_k, p.brk_s, p.brk_a, p.ts, n, i, k, s_hi, d_first, d_last);
            if (s_hi < s_top) bin_grad(gk, gl, p.n_obs, p.ts, p.S, s_hi + 1);
            else {
#pragma unroll
                for (int c = 0; c < kBinMaxObs; ++c) gk[c] = gq[c];
            }
        } else {
            while (s_hi >= 0 && brk_next == k) {
                --s_hi;
                brk_next = s_hi >= 0 ? p.brk_k[(int64_t)s_hi * n + i] : -1;
            }
        }
        float tau_k = 0.0f;
        if (draw) {
            const int jk = event_at(k);
            // pass 1: a0, E_0 and the race's keys r_j = a_j / E_j over this lane's blocks; the waiting-time word's
            // slot and the padded ones have rate 0: they add 0 and have key 0
            float a0p = 0.0f, rmax = 0.0f;
            uint32_t x0 = 0;
            float4 *ad4 = reinterpret_cast<float4 *>(ad), *rj4 = reinterpret_cast<float4 *>(rj),
                   *ct4 = reinterpret_cast<float4 *>(ct), *dA4 = reinterpret_cast<float4 *>(dA);
            for (int c = 0; c < n_rounds; ++c) {
                const uint4 r = philox4x32_10(make_uint4((uint32_t)(lane + 32 * c), (uint32_t)k, noise.c2, noise.c3),
                                              noise.key0, noise.key1);
                if (c == 0) x0 = r.x;
                const float4 av = ad4[32 * c + lane];
                const float aq[4] = {av.x, av.y, av.z, av.w};
                float key[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float a = fmaxf(aq[q], 0.0f);
                    a0p = __fadd_rn(a0p, a);
                    key[q] = a * inv_exp_of_word(word_of(r, q));
                    rmax = fmaxf(rmax, key[q]);
                }
                rj4[32 * c + lane] = make_float4(key[0], key[1], key[2], key[3]);
            }
            const float a0 = warp_sum(a0p);
            const float E0 = neg_log_unit(u01(__shfl_sync(0xffffffffu, x0, 0)));
            rmax = warp_max_nonneg(rmax);
            if (HOT || !(a0 >= 0x1p-60f && a0 <= 0x1p100f)) rmax = warp_keys_scaled(n_rounds, ad, k, noise, a0, HOT, rj);
            __syncwarp();
            const KeyTop top = key_top(rmax);
            const float top_edge = rmax * (1.0f - kTieMargin);  // keys from here on may be the largest
            const bool k_tops = rj[jk + 1] >= top_edge;
            const float tau = waiting_time(E0, a0);
            tau_k = tau;
            const int4 rk = tab.rx[jpos(jk, nb)];
            // BIN: t_{k+1} ends this interval and starts the next, in the bin of gq
            if (kBin) mu -= bin_transition(xobs, xo, gq, p.n_obs);
            float dt_dir = 0.0f, dtau_dir = 0.0f;
            if (READOUT == SSA_READOUT_LINEAR) {
                // serial on lane 0 (observed species may repeat), broadcast afterwards
                if (lane == 0) {
                    for (int s = s_hi + 1; s <= s_top; ++s) {
                        const float alpha = p.brk_a[(int64_t)s * n + i];
                        if (alpha < 0.0f) continue;
                        float c = 0.0f;
                        for (int o = 0; o < p.n_obs; ++o) {
                            const float g = gl[(int64_t)s * p.n_obs + o];
                            const int sp = p.obs_sp[o];
                            lam[sp] += alpha * g;
                            int dv = 0;
                            for (int e = rk.z; e < rk.w; ++e)
                                if (stoich_species(tab.st[e]) == sp) dv += stoich_delta(tab.st[e]);
                            c += g * (float)dv;
                        }
                        const float c_tau = __fdividef(c, tau);
                        dt_dir -= c_tau;
                        dtau_dir -= alpha * c_tau;
                    }
                }
                dt_dir = __shfl_sync(0xffffffffu, dt_dir, 0);
                dtau_dir = __shfl_sync(0xffffffffu, dtau_dir, 0);
            }
            __syncwarp();
            const float dtau = mu + dtau_dir;
            const float dLda0 = -dtau * tau / a0;
            // pass 2: soft-sample weights q_j = (r_j / r_max)^(1/T) and w_j
            float Zp = 0.0f, Wp = 0.0f;
            int near = 0;  // keys within the tie margin of the largest
            auto at = [&](int e) { return *reinterpret_cast<const float *>(reinterpret_cast<const char *>(lam) + ent_offset(e)); };
            auto weights = [&](auto many) {
                for (int c = 0; c < n_rounds; ++c) {
                    const float4 rv = rj4[32 * c + lane];
                    float qv[4] = {rv.x, rv.y, rv.z, rv.w}, wv[4];
                    const int4 *el = tab.ent + 128 * c + lane;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        near += qv[q] >= top_edge;
                        qv[q] = ex2_approx(top.lg2(qv[q]) * invT_q);
                        const int4 en = el[32 * q];
                        float w = ent_change(en.x) * at(en.x);
                        w = __fmaf_rn(ent_change(en.y), at(en.y), w);
                        w = __fmaf_rn(ent_change(en.z), at(en.z), w);
                        w = __fmaf_rn(ent_change(en.w), at(en.w), w);
                        if (decltype(many)::value && en.x == kEntMany) {
                            const int4 rx = tab.rx[q * nb + 32 * c + lane];
                            w = 0.0f;
                            for (int e = rx.z; e < rx.w; ++e)
                                w = __fmaf_rn((float)stoich_delta(tab.st[e]), lam[stoich_species(tab.st[e])], w);
                        }
                        wv[q] = w;
                        Zp += qv[q];
                        const float qw = qv[q] * w;
                        Wp += qv[q] > 0.0f ? qw : 0.0f;
                    }
                    rj4[32 * c + lane] = make_float4(qv[0], qv[1], qv[2], qv[3]);
                    ct4[32 * c + lane] = make_float4(wv[0], wv[1], wv[2], wv[3]);
                }
            };
            if (tab.many) weights(std::true_type{});
            else weights(std::false_type{});
            // the recorded reaction won the race if its key is the only one at the top; near ties are raced again
            if (__reduce_add_sync(0xffffffffu, near) == 1) mism += !k_tops;
            else mism += warp_race_exact(n_rounds, ad, k, noise) != jk;
            const float Z = warp_sum(Zp), Wq = warp_sum(Wp);
            const float invZ = __fdividef(1.0f, Z), Wbar = Wq * invZ, scale = invZ * invT;
            // pass 3: g_j = psi_j + dL/da0 a_j
            for (int c = 0; c < n_rounds; ++c) {
                const int b = 32 * c + lane;
                const float4 qf = rj4[b], wf = ct4[b], af = ad4[b];
                float4 df = dA4[b];
                auto adjoint = [&](float qv, float w, float a, float &sum) {
                    float psi = qv * scale * (w - Wbar);
                    psi = qv > 0.0f ? psi : 0.0f;
                    const float g = __fmaf_rn(dLda0, fmaxf(a, 0.0f), psi);
                    sum += g;
                    return g;
                };
                const float4 gf = make_float4(adjoint(qf.x, wf.x, af.x, df.x), adjoint(qf.y, wf.y, af.y, df.y),
                                              adjoint(qf.z, wf.z, af.z, df.z), adjoint(qf.w, wf.w, af.w, df.w));
                dA4[b] = df;
                rj4[b] = gf;
            }
            __syncwarp();
            // the state adjoint, in a fixed order
            for (int sp0 = 0; sp0 < N; sp0 += g_step) {
                const int sp = sp0 + g_first;
                float acc = 0.0f;
                if (sp < N) {
                    const int4 c = tab.inc[sp];
                    const int x = X[sp];
                    const float xf = int2f(x);
                    // plain reactants: g_j / X, or D_j dL/da0 where the species is absent (a_j = 0 on its whole list)
                    const float *src = x > 0 ? rj : ad;
                    float c0 = 0.0f, c1 = 0.0f, c2 = 0.0f, c3 = 0.0f;
                    int e = c.x + g_lane;
                    for (; e + 3 * gsz < c.y; e += 4 * gsz) {
                        c0 += src[tab.list[e] & 0xffff];
                        c1 += src[tab.list[e + gsz] & 0xffff];
                        c2 += src[tab.list[e + 2 * gsz] & 0xffff];
                        c3 += src[tab.list[e + 3 * gsz] & 0xffff];
                    }
                    for (; e < c.y; e += gsz) c0 += src[tab.list[e] & 0xffff];
                    acc = (c0 + c1) + (c2 + c3);
                    acc = x > 0 ? __fdividef(acc, xf) : -dLda0 * acc;
                    if (c.y < c.z) {  // homodimers: d log h/dX = (2 X - 1)/(X (X - 1)), dh/dX = X - 1/2 below X = 2
                        float ch = 0.0f;
                        for (int eh = c.y + g_lane; eh < c.z; eh += gsz) {
                            const int le = tab.list[eh];
                            ch += x >= 2 ? rj[le & 0xffff] : tab.k[le >> 16];
                        }
                        acc += x >= 2 ? __fdividef(ch * (xf - 0.5f), __fmul_rn(xf, xf - 1.0f) * 0.5f)
                                      : dLda0 * (xf - 0.5f) * ch;
                    }
                }
                for (int off = gsz >> 1; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
                if (g_lane == 0 && sp < N) lam[sp] += acc;
            }
            mu += dt_dir;
        }
        __syncwarp();
        if (kBin) {
            if (lane == 0)
                bin_state_terms(addx, d_first, d_last, gl, p.bin_prefix, p.n_obs, s_hi + 1, s_top, draw, tau_k, gq, gk);
#pragma unroll
            for (int c = 0; c < kBinMaxObs; ++c) {
                gq[c] = gk[c];
                if (c < p.n_obs) xo[c] = xobs(c);
            }
        } else if (lane == 0) {
            for (int s = s_hi + 1; s <= s_top; ++s) {
                float coef = 1.0f;
                if (READOUT == SSA_READOUT_LINEAR && draw) {
                    const float alpha = p.brk_a[(int64_t)s * n + i];
                    if (alpha >= 0.0f) coef = 1.0f - alpha;
                }
                for (int o = 0; o < p.n_obs; ++o) lam[p.obs_sp[o]] += coef * gl[(int64_t)s * p.n_obs + o];
            }
        }
        if (ck_off == 0) {
            const int *ck = p.ckpt + (int64_t)ck_row * N * n + i;
            int bad = 0;
            for (int s = lane; s < N; s += 32) bad += (ck[(int64_t)s * n] != X[s]);
            mism += __reduce_add_sync(0xffffffffu, bad);
            --ck_row;
            ck_off = p.K;
        }
        --ck_off;
        __syncwarp();
        if (k > 0) warp_apply<true>(tab, event_at(k - 1), -1, X, ad);
    }
    if (lane == 0 && mism) atomicAdd(p.mismatch, mism);
}

}  // namespace ssa
