// ssa_jit.cu -- network-specialised kernels compiled at run time with NVRTC.
//
// For a network with few species and reactions, the thread-per-trajectory forward and adjoint are
// generated with the network written into the code: the reactant indices, orders and stoichiometric
// changes become constants, so the counts X and the state adjoint lambda live in registers, every
// propensity is a fixed expression, and the update X += v_j is a switch over j with immediate
// increments. The per-step arithmetic is the generic kernels' (the shared helpers of ssa_device.cuh
// in the same order), so both give the same trajectories bit for bit; only the table lookups and
// the shared-memory traffic go away. The generated source is compiled once per distinct network and
// process (cached for its lifetime) for sm_103a and loaded as a context-independent CUDA library.
#include <algorithm>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include <nvrtc.h>

#include "ssa_host.h"
#include "ssa_jit_text.h"  // generated by build.py: the texts of ssa_device.cuh, ssa_jit_body.cuh, ssa.h

namespace ssa {

constexpr int kJitMaxSpecies = 24;
constexpr int kJitMaxReactions = 24;
constexpr int kJitMaxNnz = 96;

struct JitKernels {
    cudaKernel_t fwd[3][2];     // [readout][record], Gumbel-max choice (soft set: the soft forward)
    cudaKernel_t fwd_direct[3]; // [readout], direct method, forward only (not in the soft set)
    cudaKernel_t adj[3];        // [readout]
    cudaKernel_t adj_wide[2];   // [HOLD, LINEAR], wide-range adjoint (not in the soft set)
    cudaKernel_t adj_multi[2][2];  // [HOLD, LINEAR][2 or 3 temperatures] in one walk (not in the soft set)
};

namespace {

std::mutex g_jit_mu;
// source text -> kernels; libraries stay loaded until the process exits
std::map<std::string, JitKernels> g_jit_cache;
std::map<std::string, std::string> g_jit_failed;  // source text -> reason

void emit(std::string &out, const char *fmt, ...) __attribute__((format(printf, 2, 3)));
void emit(std::string &out, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    out += buf;
}

int st_species(int e) { return e >> 8; }
int st_delta(int e) { return (int)(signed char)(e & 0xff); }

// The network hooks that ssa_jit_body.cuh calls, written out for one network.
std::string jit_source(const ssa_network *net)
{
    const int N = net->N, M = net->M;
    std::string s;
    s += "#include \"ssa_device.cuh\"\n";
    emit(s, "#define JN %d\n#define JM %d\nnamespace ssa {\n", N, M);
    // propensities, in reaction order. Counts below 2^23 are exact in binary32 and need no further cases; one test over
    // the reactant species sends a step with a larger one to the general expressions (returned: whether it did).
    auto props = [&](bool general) {
        for (int j = 0; j < M; ++j) {
            const int4 r = net->h_rx[j];
            const char *in = "        ";
            if (r.x < 0) emit(s, "%sh[%d] = 1.0f;\n", in, j);
            else if (r.y < 0) emit(s, general ? "%sh[%d] = h_first(X[%d]);\n" : "%sh[%d] = f[%d];\n", in, j, r.x);
            else if (r.y == r.x && general) emit(s, "%sh[%d] = h_homodimer(X[%d]);\n", in, j, r.x);
            else if (r.y == r.x) emit(s, "%sh[%d] = __fmul_rn(f[%d], fmaxf(f[%d] - 1.0f, 0.0f)) * 0.5f;\n", in, j, r.x, r.x);
            else emit(s, general ? "%sh[%d] = h_hetero(X[%d], X[%d]);\n" : "%sh[%d] = __fmul_rn(f[%d], f[%d]);\n", in, j, r.x, r.y);
        }
    };
    s += "__device__ __forceinline__ bool jit_props(const int (&X)[JN], const float (&k)[JM], float (&a)[JM], "
         "float (&h)[JM])\n{\n    unsigned m = 0;\n";
    std::vector<bool> reacts(N, false);
    for (int j = 0; j < M; ++j) {
        if (net->h_rx[j].x >= 0) reacts[net->h_rx[j].x] = true;
        if (net->h_rx[j].y >= 0) reacts[net->h_rx[j].y] = true;
    }
    for (int sp = 0; sp < N; ++sp) emit(s, "    m |= (unsigned)X[%d];\n", sp);
    s += "    const bool big = m >= (1u << 23);\n    if (!big) {\n        float f[JN];\n";
    for (int sp = 0; sp < N; ++sp)
        if (reacts[sp]) emit(s, "        f[%d] = __int2float_rn(X[%d]);\n", sp, sp);
    props(false);
    s += "    } else {\n";
    props(true);
    s += "    }\n#pragma unroll\n    for (int j = 0; j < JM; ++j) a[j] = __fmul_rn(k[j], h[j]);\n    return big;\n}\n";
    // The changes of every reaction, int8 by species, four to a word: the kernels keep the table in shared memory and
    // apply an event with one 4-way byte dot product per species, whatever events the other lanes drew. (As a switch
    // on the event, the cases of a warp's lanes ran one after another.)
    const int W = (N + 3) / 4;
    emit(s, "#define JW %d\n__device__ const int jit_changes[JM * JW] = {", W);
    for (int j = 0; j < M; ++j)
        for (int w = 0; w < W; ++w) {
            uint32_t v = 0;
            for (int e = net->h_rx[j].z; e < net->h_rx[j].w; ++e)
                if (st_species(net->h_st[e]) / 4 == w)
                    v |= (uint32_t)(uint8_t)st_delta(net->h_st[e]) << (8 * (st_species(net->h_st[e]) % 4));
            emit(s, "(int)0x%08xu, ", v);
        }
    s += "};\n";
    // A reaction that only consumes its own reactants cannot take a count below zero (its propensity was positive), and
    // no count below 2^23 can overflow: such networks check a step only where a count is large.
    bool safe = true;
    for (int j = 0; j < M; ++j)
        for (int e = net->h_rx[j].z; e < net->h_rx[j].w; ++e) {
            const int4 r = net->h_rx[j];
            const int sp = st_species(net->h_st[e]), d = st_delta(net->h_st[e]);
            const int held = (r.x == sp) + (r.y == sp);  // a > 0: at least this many of the species
            safe &= d >= -held;
        }
    emit(s, "constexpr bool kJitSafe = %s;\n", safe ? "true" : "false");
    // range check of X + v_jb (entries in table order; the last failing entry decides)
    s += "__device__ __forceinline__ int jit_check(const int (&X)[JN], int jb)\n{\n    int st = SSA_TRAJ_OK;\n";
    {
        s += "    switch (jb) {\n";
        for (int j = 0; j < M; ++j) {
            emit(s, "    case %d:\n", j);
            for (int e = net->h_rx[j].z; e < net->h_rx[j].w; ++e) {
                const int sp = st_species(net->h_st[e]), d = st_delta(net->h_st[e]);
                if (d < 0) emit(s, "        if (X[%d] + (%d) < 0) st = SSA_TRAJ_NEG_COUNT;\n", sp, d);
                else if (d > 0) emit(s, "        if (X[%d] > 2147483647 - %d) st = SSA_TRAJ_OVERFLOW;\n", sp, d);
            }
            s += "        break;\n";
        }
        s += "    default: break;\n    }\n";
    }
    s += "    return st;\n}\n";
    // w_j = v_j . lambda, summed over the entries in table order from zero
    s += "__device__ __forceinline__ void jit_w(const float (&lam)[JN], float (&w)[JM])\n{\n";
    for (int j = 0; j < M; ++j) {
        s += "    {\n        float v = 0.0f;\n";
        for (int e = net->h_rx[j].z; e < net->h_rx[j].w; ++e)
            emit(s, "        v += (float)(%d) * lam[%d];\n", st_delta(net->h_st[e]), st_species(net->h_st[e]));
        emit(s, "        w[%d] = v;\n    }\n", j);
    }
    s += "}\n";
    // State adjoint from the per-reaction adjoints g_j = psi_j + dL/da0 a_j: a_j is proportional to the count of each
    // plain reactant, so its species receive g_j / X; a homodimer's receives g_j (X - 1/2) / h; where a reactant is
    // absent (a_j = 0) only the waiting-time path remains, dL/da0 k_j dh_j/dX. The coefficients of a state serve every
    // temperature: rx[s] = 1/X_s or 0, dz[s] = the sum of k_j dh_j/dX over the reactions of an absent species,
    // ch[j], cz[j] = the same two for homodimers.
    s += "struct JitCoef {\n    float rx[JN], dz[JN], ch[JM], cz[JM];\n};\n"
         "__device__ __forceinline__ void jit_coef(const int (&X)[JN], const float (&k)[JM], const float (&a)[JM], "
         "const float (&h)[JM], JitCoef &c)\n{\n";
    for (int sp = 0; sp < N; ++sp) {
        std::string absent;
        for (int j = 0; j < M; ++j) {
            const int4 r = net->h_rx[j];
            if (r.x == r.y || (r.x != sp && r.y != sp)) continue;
            const int other = r.x == sp ? r.y : r.x;
            absent += absent.empty() ? "" : " + ";
            absent += "k[" + std::to_string(j) + "]";
            if (other >= 0) absent += " * __int2float_rn(X[" + std::to_string(other) + "])";
        }
        if (absent.empty()) continue;
        emit(s, "    c.rx[%d] = X[%d] > 0 ? __fdividef(1.0f, __int2float_rn(X[%d])) : 0.0f;\n", sp, sp, sp);
        s += "    c.dz[" + std::to_string(sp) + "] = X[" + std::to_string(sp) + "] > 0 ? 0.0f : " + absent + ";\n";
    }
    for (int j = 0; j < M; ++j) {
        const int4 r = net->h_rx[j];
        if (r.x < 0 || r.x != r.y) continue;
        emit(s, "    {\n        const float d = __int2float_rn(X[%d]) - 0.5f;\n", r.x);
        emit(s, "        c.ch[%d] = a[%d] > 0.0f ? __fdividef(d, h[%d]) : 0.0f;\n", j, j, j);
        emit(s, "        c.cz[%d] = a[%d] > 0.0f ? 0.0f : k[%d] * d;\n    }\n", j, j, j);
    }
    s += "}\n__device__ __forceinline__ void jit_state_adj(const JitCoef &c, const float (&g)[JM], float dLda0, "
         "float (&lam)[JN])\n{\n";
    for (int sp = 0; sp < N; ++sp) {
        std::string sum;
        for (int j = 0; j < M; ++j) {
            const int4 r = net->h_rx[j];
            if (r.x == r.y || (r.x != sp && r.y != sp)) continue;
            sum += (sum.empty() ? "g[" : " + g[") + std::to_string(j) + "]";
        }
        if (!sum.empty()) {
            const std::string at = std::to_string(sp);
            s += "    lam[" + at + "] += fmaf(c.rx[" + at + "], " + sum + ", dLda0 * c.dz[" + at + "]);\n";
        }
    }
    for (int j = 0; j < M; ++j) {
        const int4 r = net->h_rx[j];
        if (r.x < 0 || r.x != r.y) continue;
        emit(s, "    lam[%d] += fmaf(c.ch[%d], g[%d], dLda0 * c.cz[%d]);\n", r.x, j, j, j);
    }
    s += "}\n";
    // soft forward (Eq. 4): propensities of the real-valued state (negative factors clipped to 0), the
    // relaxed update dX = sum_j y_j v_j (entries in table order), and the state adjoint with the
    // waiting-time derivative of a clipped factor removed
    s += "__device__ __forceinline__ void jit_props_soft(const float (&X)[JN], const float (&k)[JM], float (&a)[JM], "
         "float (&h)[JM])\n{\n";
    for (int j = 0; j < M; ++j) {
        const int4 r = net->h_rx[j];
        if (r.x < 0) emit(s, "    h[%d] = 1.0f;\n", j);
        else if (r.y < 0) emit(s, "    h[%d] = hs_first(X[%d]);\n", j, r.x);
        else if (r.y == r.x) emit(s, "    h[%d] = hs_homodimer(X[%d]);\n", j, r.x);
        else emit(s, "    h[%d] = hs_hetero(X[%d], X[%d]);\n", j, r.x, r.y);
        emit(s, "    a[%d] = __fmul_rn(k[%d], h[%d]);\n", j, j, j);
    }
    s += "}\n";
    s += "__device__ __forceinline__ void jit_dx_soft(const float (&y)[JM], float (&dX)[JN])\n{\n";
    s += "#pragma unroll\n    for (int q = 0; q < JN; ++q) dX[q] = 0.0f;\n";
    for (int j = 0; j < M; ++j)
        for (int e = net->h_rx[j].z; e < net->h_rx[j].w; ++e)
            emit(s, "    dX[%d] = __fmaf_rn(y[%d], %d.0f, dX[%d]);\n", st_species(net->h_st[e]), j, st_delta(net->h_st[e]),
                 st_species(net->h_st[e]));
    s += "}\n";
    s += "__device__ __forceinline__ void jit_state_adj_soft(const float (&X)[JN], const float (&a)[JM], "
         "const float (&h)[JM], const float (&psi)[JM], const float (&ctau)[JM], float (&lam)[JN])\n{\n";
    for (int j = 0; j < M; ++j) {
        const int4 r = net->h_rx[j];
        if (r.x < 0) continue;
        if (r.y < 0) {
            emit(s, "    lam[%d] += sadj_first(X[%d], a[%d], psi[%d], X[%d] < 0.0f ? 0.0f : ctau[%d]);\n", r.x, r.x, j, j,
                 r.x, j);
        } else if (r.y == r.x) {
            emit(s, "    lam[%d] += sadj_homodimer(X[%d], a[%d], h[%d], psi[%d], __fmul_rn(X[%d], X[%d] - 1.0f) < 0.0f ? "
                    "0.0f : ctau[%d]);\n", r.x, r.x, j, j, j, r.x, r.x, j);
        } else {
            emit(s, "    {\n        const float x1 = X[%d], x2 = X[%d];\n", r.x, r.y);
            emit(s, "        const float c = __fmul_rn(x1, x2) < 0.0f ? 0.0f : ctau[%d];\n", j);
            emit(s, "        lam[%d] += sadj_hetero(x1, x2, a[%d], psi[%d], c);\n", r.x, j, j);
            emit(s, "        lam[%d] += sadj_hetero(x2, x1, a[%d], psi[%d], c);\n    }\n", r.y, j, j);
        }
    }
    s += "}\n}  // namespace ssa\n#include \"ssa_jit_body.cuh\"\n";
    return s;
}

const char *kStddef = "#pragma once\ntypedef unsigned long size_t;\n";
const char *kStdint =
    "#pragma once\ntypedef signed char int8_t;\ntypedef short int16_t;\ntypedef int int32_t;\ntypedef long int64_t;\n"
    "typedef unsigned char uint8_t;\ntypedef unsigned short uint16_t;\ntypedef unsigned int uint32_t;\n"
    "typedef unsigned long uint64_t;\ntypedef unsigned long uintptr_t;\n";

bool compile(const std::string &src, std::vector<char> &cubin, std::string &why)
{
    const char *hdr_text[] = {kJitTextDevice, kJitTextBody, kJitTextApi, kStddef, kStdint};
    const char *hdr_name[] = {"ssa_device.cuh", "ssa_jit_body.cuh", "../../include/ssa.h", "stddef.h", "stdint.h"};
    nvrtcProgram prog;
    nvrtcResult r = nvrtcCreateProgram(&prog, src.c_str(), "ssa_network.cu", 5, hdr_text, hdr_name);
    if (r != NVRTC_SUCCESS) {
        why = nvrtcGetErrorString(r);
        return false;
    }
    // -default-device: the C declarations of ssa.h (for its constants) are read as device declarations
    const char *opts[] = {"--gpu-architecture=sm_103a", "--std=c++17", "--fmad=true", "-default-device"};
    r = nvrtcCompileProgram(prog, 4, opts);
    if (r != NVRTC_SUCCESS) {
        size_t n = 0;
        nvrtcGetProgramLogSize(prog, &n);
        std::string log(n, '\0');
        if (n) nvrtcGetProgramLog(prog, &log[0]);
        why = std::string(nvrtcGetErrorString(r)) + ": " + log.substr(0, 400);
        nvrtcDestroyProgram(&prog);
        return false;
    }
    size_t n = 0;
    nvrtcGetCUBINSize(prog, &n);
    cubin.resize(n);
    nvrtcGetCUBIN(prog, cubin.data());
    nvrtcDestroyProgram(&prog);
    return n > 0;
}

}  // namespace

bool jit_eligible(const ssa_network *net)
{
    return net->N <= kJitMaxSpecies && net->M <= kJitMaxReactions && net->nnz <= kJitMaxNnz;
}

namespace {
// Kernels of `net` (soft: the soft-forward program of the same text; hot: the adjoints at temperatures at which
// hot_weights holds, their forwards' and wide walks' entries empty), compiling and loading them on
// first use. Returns nullptr (with the reason in `why`) if the network is not eligible or compilation
// failed.
const JitKernels *jit_load(const ssa_network *net, bool soft, bool hot, std::string &why)
{
    if (!jit_eligible(net)) {
        why = "network above the specialisation limits (24 species, 24 reactions, 96 stoichiometric entries)";
        return nullptr;
    }
    const std::string src = (soft ? "#define SSA_JIT_SOFT 1\n" : hot ? "#define SSA_JIT_HOT 1\n" : "") + jit_source(net);
    std::lock_guard<std::mutex> lock(g_jit_mu);
    auto f = g_jit_failed.find(src);
    if (f != g_jit_failed.end()) {
        why = f->second;
        return nullptr;
    }
    auto it = g_jit_cache.find(src);
    if (it != g_jit_cache.end()) return &it->second;
    std::vector<char> cubin;
    if (!compile(src, cubin, why)) {
        g_jit_failed[src] = why;
        return nullptr;
    }
    cudaLibrary_t lib = nullptr;
    cudaError_t e = cudaLibraryLoadData(&lib, cubin.data(), nullptr, nullptr, 0, nullptr, nullptr, 0);
    if (e != cudaSuccess) {
        why = std::string("cudaLibraryLoadData: ") + cudaGetErrorString(e);
        g_jit_failed[src] = why;
        return nullptr;
    }
    JitKernels k{};
    const char *rname[3] = {"hold", "linear", "bin"};
    bool ok = true;
    for (int r = 0; r < 3; ++r) {
        const std::string base = std::string(rname[r]) + (soft ? "_soft" : "");
        for (int rec = 0; rec < 2 && !hot; ++rec) {
            const std::string nm = "ssa_jit_fwd_" + base + (rec ? "_rec" : "");
            ok &= cudaLibraryGetKernel(&k.fwd[r][rec], lib, nm.c_str()) == cudaSuccess;
        }
        ok &= cudaLibraryGetKernel(&k.adj[r], lib, ("ssa_jit_adj_" + base).c_str()) == cudaSuccess;
        if (!soft && !hot)
            ok &= cudaLibraryGetKernel(&k.fwd_direct[r], lib, ("ssa_jit_fwd_" + base + "_direct").c_str()) == cudaSuccess;
        if (!soft && r < 2) {
            ok &= hot || cudaLibraryGetKernel(&k.adj_wide[r], lib, ("ssa_jit_adj_" + base + "_wide").c_str()) == cudaSuccess;
            for (int nt = 2; nt <= 3; ++nt)
                ok &= cudaLibraryGetKernel(&k.adj_multi[r][nt - 2], lib,
                                           ("ssa_jit_adj_" + base + "_t" + std::to_string(nt)).c_str()) == cudaSuccess;
        }
    }
    if (!ok) {
        why = "a specialised kernel is missing from the library";
        g_jit_failed[src] = why;
        cudaLibraryUnload(lib);
        return nullptr;
    }
    return &(g_jit_cache[src] = k);
}
}  // namespace

const JitKernels *jit_kernels(const ssa_network *net, std::string &why) { return jit_load(net, false, false, why); }
const JitKernels *jit_soft_kernels(const ssa_network *net, std::string &why) { return jit_load(net, true, false, why); }
const JitKernels *jit_hot_kernels(const ssa_network *net, std::string &why) { return jit_load(net, false, true, why); }

// Bits of the chunk size for the bin readout's chunk sums, 0: none. One observable, a gradient per trajectory, at most
// kChunkRows chunks a row (28 KB a block), a chunk no wider than a warp's loads.
constexpr int kChunkRows = 56;
static int jit_chunk_shift(const AdjParams &p, int readout)
{
    if (readout != SSA_READOUT_BIN || p.bin_prefix || p.n_obs != 1 || p.S < 32) return 0;
    int shift = 4;
    while (((p.S - 1) >> shift) >= kChunkRows) ++shift;
    const bool pieces = (p.S & 3) == 0 && (p.dl_stride & 3) == 0 && (reinterpret_cast<uintptr_t>(p.dl_dobs) & 15) == 0;
    return shift <= (pieces ? 7 : 5) ? shift : 0;
}

cudaError_t jit_launch_forward(const JitKernels *k, const FwdParams &p, int readout, bool record, int selector,
                               int block, cudaStream_t st)
{
    if (p.n_traj == 0) return cudaSuccess;
    const unsigned grid = (unsigned)((p.n_traj + block - 1) / block);
    void *args[] = {const_cast<FwdParams *>(&p)};
    const int r = readout;  // SSA_READOUT_HOLD, _LINEAR, _BIN index the tables
    const cudaKernel_t f = selector == SSA_SELECT_DIRECT ? k->fwd_direct[r] : k->fwd[r][record ? 1 : 0];
    const size_t smem = readout == SSA_READOUT_BIN ? (size_t)4 * (kBinRuns + 1) * (2 + p.n_obs) * block : 0;
    return cudaLaunchKernel(reinterpret_cast<const void *>(f), dim3(grid), dim3((unsigned)block), args, smem, st);
}

cudaError_t jit_launch_backward(const JitKernels *k, const AdjParams &p, int readout, int block, int64_t grid,
                                cudaStream_t st)
{
    if (grid == 0) return cudaSuccess;
    AdjParams q = p;
    q.chunk_shift = jit_chunk_shift(p, readout);
    void *args[] = {&q};
    const size_t rows = q.chunk_shift ? ((p.S - 1) >> q.chunk_shift) + 1 : 0;
    const size_t smem = (size_t)4 * std::max<size_t>(p.M, rows) * block;
    return cudaLaunchKernel(reinterpret_cast<const void *>(k->adj[readout]),
                            dim3((unsigned)grid), dim3((unsigned)block), args, smem, st);
}

cudaError_t jit_launch_backward_wide(const JitKernels *k, const AdjParams &p, int readout, int block, int64_t grid,
                                     cudaStream_t st)
{
    if (grid == 0) return cudaSuccess;
    if (readout != SSA_READOUT_HOLD && readout != SSA_READOUT_LINEAR) return cudaErrorInvalidValue;
    void *args[] = {const_cast<AdjParams *>(&p)};
    const size_t smem = (size_t)8 * p.M * block;  // binary64 block reduction
    return cudaLaunchKernel(reinterpret_cast<const void *>(k->adj_wide[readout]),
                            dim3((unsigned)grid), dim3((unsigned)block), args, smem, st);
}

cudaError_t jit_launch_backward_multi(const JitKernels *k, const AdjParams &p, int readout, int n_temps, int block,
                                      int64_t grid, cudaStream_t st)
{
    if (grid == 0) return cudaSuccess;
    if ((readout != SSA_READOUT_HOLD && readout != SSA_READOUT_LINEAR) || n_temps < 2 || n_temps > 3)
        return cudaErrorInvalidValue;
    void *args[] = {const_cast<AdjParams *>(&p)};
    const size_t smem = (size_t)4 * n_temps * p.M * block;
    return cudaLaunchKernel(reinterpret_cast<const void *>(k->adj_multi[readout][n_temps - 2]),
                            dim3((unsigned)grid), dim3((unsigned)block), args, smem, st);
}

}  // namespace ssa

using namespace ssa;

extern "C" ssa_status ssa_network_specialize(ssa_network *net, int32_t *host_ok)
{
    if (!net || !host_ok) return set_error(SSA_ERR_INVALID_ARG, "NULL argument");
    std::string why;
    *host_ok = jit_kernels(net, why) ? 1 : 0;
    if (!*host_ok) set_error(SSA_OK, why.c_str());
    return SSA_OK;
}
