// C ABI of the GB300 column multigrid solver: handle, set-up, V-cycle driver (Algorithm 1),
// GCR outer solves and the mixed-system Schur-complement preconditioner.
// See include/mgsolve.h for the contract of every entry point.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <type_traits>
#include <utility>
#include <vector>

#include "../../include/mgsolve.h"
#include "kernels.cuh"
#include "krylov.cuh"
#include "mesh.h"
#include "sweep64.cuh"
#include "sweep_tma.cuh"

using mg::Lvl;
using mg::Lvl32;
using mg::Lvl64;
typedef __nv_bfloat16 bf16;

namespace {

struct DevLevel {
    int n = 0, ncol = 0;
    int32_t* nbr = nullptr;
    int32_t* fof = nullptr;
    double* rA64 = nullptr;
    double* Th64 = nullptr;
    double* Tv64 = nullptr;
    int32_t* hd = nullptr;       // [4][ncol] rim cells of the padded FP32 fields (sweep32.cuh)
    int32_t* par = nullptr;      // [5][ncol] coarse parents of the neighbours and of the column
    // FP64 level data (sweep64.cuh; also mg_smooth and mg_residual_restrict)
    double *te64 = nullptr, *tn64 = nullptr, *tbw64 = nullptr, *tbs64 = nullptr, *tv64 = nullptr;
    double *e64 = nullptr, *ip64 = nullptr, *pr64 = nullptr;
    double* wA64 = nullptr;      // area x scale
    bool wants64 = false, packed64 = false;   // somebody uses them; they are those of the face form (ready64)
    // FP32 level data (sweep32.cuh): couplings in FP32 or BF16, reciprocal pivots, 1 / area; the
    // FP64 elimination of MG_FP32_P64's finest level; restriction weights onto the next level
    // [4][ncol_next] (the 9-cell stencil's as well); tensor maps, iterate in x32[0] / x32[1]
    float *te32 = nullptr, *tn32 = nullptr, *tv32 = nullptr;
    bf16 *te16 = nullptr, *tn16 = nullptr, *tv16 = nullptr;
    float* ip32 = nullptr;
    double *ipd = nullptr, *md = nullptr, *ed = nullptr;
    float* rA32 = nullptr;
    double* w64 = nullptr;
    float* w32 = nullptr;
    std::vector<mg::SweepMaps> maps;
    // 9-cell stencil in FP32: the face form
    float* Th32 = nullptr;
    float* Tv32 = nullptr;
    // workspace: two iterates, the level's rhs and the result handed to the finer level
    double* x64[2] = {nullptr, nullptr};
    double* b64 = nullptr;
    double* r64 = nullptr;
    float* x32[2] = {nullptr, nullptr};
    float* b32 = nullptr;
    float* r32 = nullptr;
    // launch shapes chosen by mg_autotune (0 / -1: the built-in choice)
    int sweep_bd = 0;          // FP32 sweep: 64: register chunks, 128: tensor-copy tiles
    int restrict_kc = 0;       // levels per thread of the residual + restriction
    // 9-cell stencil: fluxes two levels apart [nlev][ncol] and three scratch fields (the
    // residual and the two Thomas factors of a sweep)
    double* T2_64 = nullptr;
    float* T2_32 = nullptr;
    double* s64[3] = {nullptr, nullptr, nullptr};
    float* s32[3] = {nullptr, nullptr, nullptr};
};

}  // namespace

struct mg_handle {
    int device = 0;
    int L = 0, nlev = 0, n = 0;
    int nsm = 0;
    mg_params prm{};
    std::vector<DevLevel> lv;
    double* rdz64 = nullptr;
    float* rdz32 = nullptr;
    double om0 = 1.0;           // relaxation factor folded into the FP64 factors (prm.omega)
    double scale = 1.0;         // power of two in the FP64 volume weights, 1 / (largest finest area x depth)
    double* a6 = nullptr;       // finest level: six premultiplied FP64 couplings and 1 + their sum, per cell
    bool nine = false;          // 9-cell stencil (mg_setup_9pt)
    double* area0 = nullptr;    // finest level: column areas and layer depths (cell volumes, adjoint solve)
    double* dz = nullptr;
    double* adj = nullptr;      // [N] the scaled right-hand side of the adjoint solve
    // finest-level face tables for caller-supplied couplings (mg_setup_coeffs, mg_set_coefficients)
    int32_t* faceL0 = nullptr;
    int32_t* faceR0 = nullptr;
    int32_t* faceSide0 = nullptr;
    int32_t* nbrSide0 = nullptr;
    unsigned int* flag = nullptr;
    unsigned int* timeout = nullptr;   // device: a bounded wait of a sweep ran into its limit
    int polls = mg::WAIT_POLLS;        // that limit (mg_inject_wait_limit)
    // pressure solver K_H(A_H, P_H, eps_H) of the Schur-complement step (Sec. 4.1, Table 1)
    mg_pressure_solver ps{MG_PS_MG, 1e-2, 0.8, 10, 200};
    double* bv[8] = {};             // BiCGStab vectors r^, r, p, v, s, t, p^, s^ (allocated on demand)
    mg::BicgScal* bs = nullptr;     // its device scalars
    mg::BicgScal* host_bs = nullptr;   // pinned copy read once per iteration
    long long ps_solves = 0;        // pressure solves since the last mg_inner_stats
    double ps_iters = 0.0;          // their BiCGStab iterations (a half step counts 0.5)
    // GCR
    size_t glen = 0;            // length of a GCR vector (N, or nu + N with mixed data)
    double* Z = nullptr;        // [restart][glen]
    double* W = nullptr;        // [restart][glen]
    double* r = nullptr;        // [glen]
    mg::GcrScal* gs = nullptr;  // device scalars of the GCR iteration
    double* partials = nullptr;
    size_t npartials = 0;
    unsigned int* tickets = nullptr;
    double* host_sc = nullptr;  // pinned: <r, r>, <b, b>
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    // one CUDA graph per GCR slot j and system (0 pressure, 1 mixed, 2 the mixed adjoint's
    // A-hat): the V-cycle, the
    // operator with its sums, the orthogonalisation and the read-back of <r, r>, captured on
    // `cap` the first time and replayed on the caller's stream afterwards
    cudaStream_t cap = nullptr;
    cudaStream_t run = nullptr;   // the handle's stream inside an ensemble solve, and for ready64 under capture
    std::mutex pack_mutex;        // ready64
    cudaEvent_t evx = nullptr;    // ordering event (no timing)
    cudaGraphExec_t gexec[3][mg::MAXR] = {};
    bool graphs_off = false;
    int red_grid = 0;
    // mixed
    bool mixed = false;
    int64_t nu = 0;
    mg::MixedDev md{};
    double* schurB = nullptr;
    double* mb = nullptr;       // concatenated mixed rhs [nu + N]
    double* mx = nullptr;       // concatenated mixed solution [nu + N]
    std::vector<void*> allocs;
    // per-launch event profiling (mg_profile_start / mg_profile_stop)
    struct Rec {
        int kind, level, variant;
        double bytes;
    };
    bool prof = false;
    int prof_kind = -1, prof_level = -1;   // record only this kind / level (-1: all)
    std::vector<cudaEvent_t> evpool;
    std::vector<Rec> recs;
};

namespace {

enum { TK_DOT = 0, TK_SUMS, TK_ORTH, TK_BICG, TK_COUNT };

// k-chunk of the column kernels that have no vertical recurrence (apply): short chunks give
// many independent threads, so the loads of different threads overlap
constexpr int APPLY_KCHUNK = 8;

// the CUDA error behind the last MG_ERR_CUDA of this thread (mg_last_cuda_error)
thread_local cudaError_t g_last_cuda = cudaSuccess;

// A failed runtime call returns MG_ERR_CUDA; a non-sticky error is cleared so that it does not
// surface again in a later, unrelated call.
#define CK(call)                       \
    do {                               \
        cudaError_t e_ = (call);       \
        if (e_ != cudaSuccess) {       \
            g_last_cuda = e_;          \
            cudaGetLastError();        \
            return MG_ERR_CUDA;        \
        }                              \
    } while (0)

#define TRY(call)                         \
    do {                                  \
        mg_status s_ = (call);            \
        if (s_ != MG_OK) return s_;       \
    } while (0)

// Every device and pinned-host allocation of the library goes through mem_alloc / mem_free.
// They count the live allocations (mg_live_allocations) and carry the failure injection of
// mg_inject_alloc_failure: with g_fail_at = n > 0, the n-th allocation attempted after the call
// fails as if the memory were exhausted.
std::atomic<long long> g_fail_at{0}, g_alloc_seen{0}, g_live{0};

enum MemKind { MEM_DEVICE, MEM_PINNED };

bool mem_alloc(void** p, size_t bytes, MemKind kind) {
    *p = nullptr;
    const long long seen = g_alloc_seen.fetch_add(1) + 1;
    const long long at = g_fail_at.load();
    if (at > 0 && seen == at) return false;
    const cudaError_t e = kind == MEM_DEVICE ? cudaMalloc(p, bytes) : cudaMallocHost(p, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return false;
    }
    g_live.fetch_add(1);
    return true;
}

void mem_free(void* p, MemKind kind) {
    if (!p) return;
    if (kind == MEM_DEVICE) cudaFree(p);
    else cudaFreeHost(p);
    g_live.fetch_sub(1);
}

template <typename P>
mg_status dalloc(mg_handle* h, P** p, size_t count) {
    *p = nullptr;
    if (count == 0) return MG_OK;
    void* q = nullptr;
    if (!mem_alloc(&q, count * sizeof(P), MEM_DEVICE)) return MG_ERR_NOMEM;
    h->allocs.push_back(q);
    *p = static_cast<P*>(q);
    return MG_OK;
}

// Several arrays in one allocation, each from a 256-byte boundary on.
struct Pieces {
    struct Piece {
        void** to;
        size_t at;
    };
    std::vector<Piece> pieces;
    size_t bytes = 0;
    template <typename P>
    void add(P** to, size_t count) {
        *to = nullptr;
        pieces.push_back({reinterpret_cast<void**>(to), bytes});
        bytes += (count * sizeof(P) + 255) / 256 * 256;
    }
    mg_status alloc(mg_handle* h) {
        char* base = nullptr;
        TRY(dalloc(h, &base, bytes));
        for (const Piece& p : pieces) *p.to = base + p.at;
        return MG_OK;
    }
};

template <typename P, typename S>
mg_status upload(mg_handle* h, P** p, const std::vector<S>& src) {
    mg_status st = dalloc(h, p, src.size());
    if (st != MG_OK) return st;
    if (src.empty()) return MG_OK;
    std::vector<P> tmp(src.size());
    for (size_t i = 0; i < src.size(); ++i) tmp[i] = (P)src[i];
    CK(cudaMemcpy(*p, tmp.data(), tmp.size() * sizeof(P), cudaMemcpyHostToDevice));
    return MG_OK;
}

// An NVTX range over the scope (shows the library's calls and GCR iterations on a profiler's
// timeline; costs nothing without a tool attached)
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
};

inline cudaStream_t S(void* s) { return static_cast<cudaStream_t>(s); }

inline size_t cells(const mg_handle* h, int l) { return (size_t)h->nlev * h->lv[l].ncol; }

// Brackets one kernel launch with a pair of events when profiling is on.  `bytes` is the
// algorithmic traffic of the launch: every array element the kernel must read or write,
// counted once (neighbour re-reads within a launch are cache traffic, not counted).
struct Prof {
    mg_handle* h;
    cudaStream_t s;
    int idx = -1;
    Prof(mg_handle* h_, int kind, int level, double bytes, cudaStream_t s_, int variant = 0) : h(h_), s(s_) {
        if (h && h->prof && 2 * (h->recs.size() + 1) <= h->evpool.size() &&
            (h->prof_kind < 0 || h->prof_kind == kind) && (h->prof_level < 0 || h->prof_level == level)) {
            idx = (int)h->recs.size();
            h->recs.push_back({kind, level, variant, bytes});
            cudaEventRecord(h->evpool[2 * idx], s);
        }
    }
    ~Prof() {
        if (idx >= 0) cudaEventRecord(h->evpool[2 * idx + 1], s);
    }
};

// ---- per-precision views of a level ----
template <typename T, typename C>
struct View;

template <>
struct View<double, double> {
    static Lvl<double, double> lvl(const mg_handle* h, int l) {
        const DevLevel& d = h->lv[l];
        return {d.n, d.ncol, h->nlev, d.nbr, d.fof, d.Th64, d.Tv64, d.rA64, h->rdz64};
    }
    static double* x(DevLevel& d, int i) { return d.x64[i]; }
    static double* b(DevLevel& d) { return d.b64; }
    static double* r(DevLevel& d) { return d.r64; }
    static const double* w(const DevLevel& d) { return d.w64; }
    static const double* t2(const DevLevel& d) { return d.T2_64; }
    static double* scratch(DevLevel& d, int i) { return d.s64[i]; }
};
template <>
struct View<float, float> {
    static Lvl<float, float> lvl(const mg_handle* h, int l) {
        const DevLevel& d = h->lv[l];
        return {d.n, d.ncol, h->nlev, d.nbr, d.fof, d.Th32, d.Tv32, d.rA32, h->rdz32};
    }
    static float* x(DevLevel& d, int i) { return d.x32[i]; }
    static float* b(DevLevel& d) { return d.b32; }
    static float* r(DevLevel& d) { return d.r32; }
    static const float* w(const DevLevel& d) { return d.w32; }
    static const float* t2(const DevLevel& d) { return d.T2_32; }
    static float* scratch(DevLevel& d, int i) { return d.s32[i]; }
};

Lvl64 lvl64(const mg_handle* h, int l) {
    const DevLevel& d = h->lv[l];
    return {d.n, d.ncol, h->nlev, d.nbr, d.par, d.te64, d.tn64, d.tbw64, d.tbs64, d.tv64, d.e64, d.ip64, d.pr64,
            d.wA64, h->dz, h->om0};
}

template <typename C, typename P>
Lvl32<C, P> lvl32(const mg_handle* h, int l) {
    const DevLevel& d = h->lv[l];
    Lvl32<C, P> L{d.n, d.ncol, h->nlev, mg::pad_row(d.n), mg::padded(d.n), d.hd};
    if constexpr (sizeof(C) == 4) {
        L.te = d.te32;
        L.tn = d.tn32;
        L.tv = d.tv32;
    } else {
        L.te = d.te16;
        L.tn = d.tn16;
        L.tv = d.tv16;
    }
    if constexpr (sizeof(P) == 4) {
        L.ip = d.ip32;
        L.m = L.e = nullptr;
    } else {
        L.ip = d.ipd;
        L.m = d.md;
        L.e = d.ed;
    }
    L.rA = d.rA32;
    L.rdz = h->rdz32;
    return L;
}

// ---- launchers ----
template <typename T, typename C, typename X, typename Y>
mg_status launch_apply(mg_handle* h, int lev, const Lvl<T, C>& L, const X* x, Y* y, cudaStream_t s) {
    const double nc = (double)L.nlev * L.ncol;
    Prof pr(h, MG_K_APPLY, lev, nc * (sizeof(X) + 3 * sizeof(C) + sizeof(Y)), s);
    const int bd = 128;
    const int kc = APPLY_KCHUNK;
    dim3 grid((L.ncol + bd - 1) / bd, (L.nlev + kc - 1) / kc);
    mg::k_apply<T, C, X, Y><<<grid, bd, 0, s>>>(L, x, y, kc);
    CK(cudaGetLastError());
    return MG_OK;
}

// FP32 levels that run their sweeps on tensor-copy tiles rather than register chunks.  A V-cycle on its own /
// eight side by side [us each] with the chunks and with the tiles on levels of these cells:
//   columns of more than 40 levels, whose chunks fill an SM with one block, 250k: C32L50 74.0/28.2 and 72.7/25.5,
//   C32L70 94/35 and 88/32, C48L41 89/52 and 86/41 (C48L50 92.9/55 and 94.9/50; C24L70, 242k: 92.9 and 93.7);
//   up to 40 levels, 700k: C64L30 81/47 and 80/42 (C56L30, 564k: 71 and 78; C48L37 77/34 and 81/36).
// C48L50 alone is 2 us slower for it; what decides there is the throughput beside other solves.
//   more than 80 levels, one block of tiles per SM, 2M: C128L100 778 and 537 (alone; before the chunks 725),
//   C192L100 1467 and 1050 (1333), C64L128 324 and 274, C80L100 365 and 335; C48L100, 1.4M: 190 and 195,
//   C48L81 166 and 178.
// Short columns stay on chunks where these hold a half without waste and the tiles' chunks of 7 would be about
// half empty: 8 levels (a chunk of 4) and 15 to 20 (two of 4 or 5).  Finest sweep from zero / plain / with
// prolongation, tiles and chunks: C256L8 49/47/54 and 19/33/37, C224L16 59/61/68 and 41/52/57, C192L20 45/49/51 and
// 35/43/47; C256L9 49/47/55 and 45/55/59, C224L14 33/39/42 and 39/51/55, C192L24 45/51/53 and 37/76/82.
inline bool tma_level(int nlev, int ncol) {
    if (nlev <= 8 || (nlev >= 15 && nlev <= 20)) return false;
    return (double)nlev * ncol >= (nlev > 80 ? 2e6 : nlev > 40 ? 2.5e5 : 7e5);
}

// Grid of a vector pass with or without a reduction: two elements per thread until the GPU is full (C12L30's
// <b, b>: 8.8 us; one per thread 10.6; C192L70's orthogonalisations 121 us on average, with 6, 16 or 32 blocks
// per SM instead of 8: 131, 124, 129).
inline int vec_grid(const mg_handle* h, size_t n) {
    constexpr size_t per_block = 2 * mg::RED_THREADS;
    return (int)std::max<size_t>(1, std::min<size_t>(h->red_grid, (n + per_block - 1) / per_block));
}

inline bool aligned(const void* p, size_t bytes) { return (reinterpret_cast<uintptr_t>(p) & (bytes - 1)) == 0; }

inline int sweep_mode(const void* x, const void* xc) {
    return xc ? (x ? mg::XM_PROLONG : mg::XM_PROLONG0) : (x ? mg::XM_PLAIN : mg::XM_ZERO);
}

// levels per thread of the residual + restriction: a few (fewer prologues) where the level fills the GPU
// several times over, one on small levels, which need every thread (C48L30: 6.5 us a launch against 13 with
// eight).  V-cycle on two levels with 1 / 2 / 4 / 8 / 35 a thread: C192L70 482/478/477/480/480 us (FP64
// 2218/2191/2179/2178/2221), C144L36 FP64 763/756/754/756/783, C160L20 162/162/161/162/176, C130L128
// 674/669/670/672/672; C96L70's restriction 21 us with 2 or 6, 22 with 12.
inline int restrict_chunk(const mg_handle* h, int lev) {
    const DevLevel& d = h->lv[lev];
    if (d.restrict_kc > 0) return d.restrict_kc;
    return d.ncol >= 100000 ? 4 : (double)h->nlev * d.ncol >= 2e6 ? 2 : 1;
}

// One FP64 block-Jacobi sweep on level `lev`.  The iterate it starts from is x (NULL: zero) plus,
// with xc, the prolongation of xc.  b: weighted, or with `raw` the caller's, whose weighted form is
// stored in bcopy when that is given.  (h is NULL where no launch may be recorded.)
template <bool RAW, bool COPY, int K>
cudaError_t sweep64_go(const Lvl64& L, int mode, const double* x, const double* xc, int ncol_c, const double* b,
                       double* bcopy, double* xo, double om, cudaStream_t s) {
    const dim3 g((L.ncol + 31) / 32), t(32 * ((L.nlev + K - 1) / K));
    switch (mode) {
        case mg::XM_ZERO: mg::k_sweep64<mg::XM_ZERO, RAW, COPY, K><<<g, t, 0, s>>>(L, x, xc, ncol_c, b, bcopy, xo, om); break;
        case mg::XM_PLAIN: mg::k_sweep64<mg::XM_PLAIN, RAW, COPY, K><<<g, t, 0, s>>>(L, x, xc, ncol_c, b, bcopy, xo, om); break;
        case mg::XM_PROLONG: mg::k_sweep64<mg::XM_PROLONG, RAW, COPY, K><<<g, t, 0, s>>>(L, x, xc, ncol_c, b, bcopy, xo, om); break;
        default: mg::k_sweep64<mg::XM_PROLONG0, RAW, COPY, K><<<g, t, 0, s>>>(L, x, xc, ncol_c, b, bcopy, xo, om); break;
    }
    return cudaGetLastError();
}

mg_status launch_sweep64(mg_handle* h, int lev, const Lvl64& L, const double* x, const double* xc, int ncol_c,
                         const double* b, bool raw, double* bcopy, double* xo, double om, cudaStream_t s) {
    const int mode = sweep_mode(x, xc);
    Prof pr(h, MG_K_SWEEP, lev, 8.0 * L.nlev * L.ncol * (4 + (mode != mg::XM_ZERO ? 2 : 0) + (x ? 1 : 0) +
                                                         (xc ? 0.25 : 0.0) + (bcopy ? 1 : 0)), s, mode);
    auto shape = [&](auto r, auto c) -> cudaError_t {
        constexpr bool R = decltype(r)::value, B = decltype(c)::value;
        switch (mg::sweep64_levels(L.nlev, L.ncol)) {
            case 16: return sweep64_go<R, B, 16>(L, mode, x, xc, ncol_c, b, bcopy, xo, om, s);
            case 5: return sweep64_go<R, B, 5>(L, mode, x, xc, ncol_c, b, bcopy, xo, om, s);
            default: return sweep64_go<R, B, 10>(L, mode, x, xc, ncol_c, b, bcopy, xo, om, s);
        }
    };
    if (raw && bcopy) CK(shape(std::true_type(), std::true_type()));
    else if (raw) CK(shape(std::true_type(), std::false_type()));
    else CK(shape(std::false_type(), std::false_type()));
    return MG_OK;
}

// FP64 residual and restriction of level lev onto lev + 1 (weighted right-hand sides; RAW: the caller's
// unweighted arrays, mg_residual_restrict).
template <bool RAW>
mg_status launch_restrict64(mg_handle* h, int lev, const double* x, const double* b, double* bc, cudaStream_t s) {
    const Lvl64 L = lvl64(h, lev);
    const int ncol_c = h->lv[lev + 1].ncol, kc = restrict_chunk(h, lev);
    const double* wAc = h->lv[lev + 1].wA64;
    Prof pr(h, MG_K_RESTRICT, lev, 8.0 * L.nlev * L.ncol * (1.25 + (x ? 3.5 : 0.0)), s);
    const bool vec = aligned(b, 16) && aligned(x, 16);
    const dim3 grid((ncol_c + 127) / 128, (L.nlev + kc - 1) / kc);
    if (!x) mg::k_restrict64<true, RAW, false><<<grid, 128, 0, s>>>(L, x, b, wAc, bc, ncol_c, kc);
    else if (vec) mg::k_restrict64<false, RAW, true><<<grid, 128, 0, s>>>(L, x, b, wAc, bc, ncol_c, kc);
    else mg::k_restrict64<false, RAW, false><<<grid, 128, 0, s>>>(L, x, b, wAc, bc, ncol_c, kc);
    CK(cudaGetLastError());
    return MG_OK;
}

// The same of the FP32 V-cycle (fields padded).  raw: b is the caller's FP64 array, its FP32 copy goes
// to bcopy unless that is NULL.  xo: padded FP32, or FP64 with out64.
template <typename C, typename P>
mg_status launch_sweep32(mg_handle* h, int lev, const float* x, const float* xc, const void* b, bool raw, float* bcopy,
                         void* xo, bool out64, double om, cudaStream_t s) {
    const Lvl32<C, P> L = lvl32<C, P>(h, lev);
    const DevLevel& d = h->lv[lev];
    const int mode = sweep_mode(x, xc);
    double per = (raw ? (bcopy ? 12.0 : 8.0) : 4.0) + sizeof(C) + (sizeof(P) == 8 ? 24.0 : 4.0) + (out64 ? 8.0 : 4.0);
    if (mode != mg::XM_ZERO) per += 2.0 * sizeof(C);
    if (x) per += 4.0;
    if (xc) per += 1.0;
    Prof pr(h, MG_K_SWEEP, lev, (double)L.nlev * L.ncol * per, s, mode);
    const mg::SweepMaps* maps = nullptr;
    const bool tiles = d.sweep_bd > 0 ? d.sweep_bd == 128 : tma_level(L.nlev, L.ncol);
    // (an FP64 elimination's chunks of taller columns have no room beside the boxes)
    const bool has = sizeof(P) == 4 || L.nlev <= mg::tma_max_levels(8);
    if (tiles && has && d.maps.size() == 2) maps = &d.maps[x == d.x32[1]];
    const mg::SweepCall32<C, P> q{L, mode, x, xc, b, raw, bcopy, xo, out64, om, maps, h->nsm, h->polls, h->timeout};
    CK((mg::sweep32_run<C, P>(q, s)));
    if (L.n == 1 && !out64) {   // (a C1 column has several edges on one axis)
        mg::k_fill_rims<float><<<dim3(1, L.nlev), 32, 0, s>>>(L.n, L.ncol, L.hd, static_cast<float*>(xo));
        CK(cudaGetLastError());
    }
    return MG_OK;
}

template <typename C>
mg_status launch_restrict32(mg_handle* h, int lev, const float* x, const float* b, float* bc, cudaStream_t s) {
    const Lvl32<C, float> L = lvl32<C, float>(h, lev);
    const DevLevel& d = h->lv[lev];
    const int ncol_c = h->lv[lev + 1].ncol, kc = restrict_chunk(h, lev);
    Prof pr(h, MG_K_RESTRICT, lev, (double)L.nlev * L.ncol * (5.0 + (x ? 4.0 + 3.0 * sizeof(C) : 0.0)), s);
    const dim3 grid((ncol_c + 127) / 128, (L.nlev + kc - 1) / kc);
    const bool tree = L.n % 16 == 0;
    if (!x && tree) mg::k_restrict32<C, true, true><<<grid, 128, 0, s>>>(L, x, b, d.w32, bc, ncol_c, kc);
    else if (!x) mg::k_restrict32<C, true, false><<<grid, 128, 0, s>>>(L, x, b, d.w32, bc, ncol_c, kc);
    else if (tree) mg::k_restrict32<C, false, true><<<grid, 128, 0, s>>>(L, x, b, d.w32, bc, ncol_c, kc);
    else mg::k_restrict32<C, false, false><<<grid, 128, 0, s>>>(L, x, b, d.w32, bc, ncol_c, kc);
    CK(cudaGetLastError());
    return MG_OK;
}

template <typename T, bool ZB, typename X, typename O>
mg_status launch_prolong(mg_handle* h, int lev, int n, int ncol, int ncol_c, int nlev, const X* x, const T* xc,
                         O* xo, cudaStream_t s) {
    Prof pr(h, MG_K_PROLONG, lev, (double)nlev * ncol * (0.25 * sizeof(T) + (ZB ? 0 : sizeof(X)) + sizeof(O)), s);
    const int bd = 128;
    mg::k_prolong<T, ZB, X, O><<<(ncol + bd - 1) / bd, bd, 0, s>>>(n, ncol, ncol_c, nlev, x, xc, xo);
    CK(cudaGetLastError());
    return MG_OK;
}

template <typename A, typename B>
mg_status launch_convert(mg_handle* h, int lev, size_t n, const A* a, B* b, cudaStream_t s) {
    Prof pr(h, MG_K_CONVERT, lev, (double)n * (sizeof(A) + sizeof(B)), s);
    mg::k_convert<A, B><<<4 * 152, 256, 0, s>>>(n, a, b);
    CK(cudaGetLastError());
    return MG_OK;
}

// Settings of one cycle: levels used, over-relaxation and sweep counts.  A single-level
// cycle with n_coarse sweeps is the block-Jacobi iteration P_H^(Jac)(omega, n_coarse) of
// Sec. 4.1 (line relaxation).
struct Cycle {
    int L;
    double omega;
    int n_pre, n_post, n_coarse;
};

inline Cycle vcycle_of(const mg_handle* h) {
    return {h->L, h->prm.omega, h->prm.n_pre, h->prm.n_post, h->prm.n_coarse};
}

// out = (x or 0) + Prolongate(xc), or without xc the conversion of x, into a level's result
template <typename T, typename O>
mg_status launch_emit(mg_handle* h, int lev, const T* x, const T* xc, O* out, cudaStream_t s) {
    const DevLevel& d = h->lv[lev];
    Prof pr(h, xc ? MG_K_PROLONG : MG_K_CONVERT, lev,
            (double)cells(h, lev) * ((xc ? 0.25 * sizeof(T) : 0.0) + (x ? sizeof(T) : 0) + sizeof(O)), s);
    const int kc = (double)h->nlev * d.ncol >= 1e6 ? 8 : 1;   // (C192L70 finest: 62 and 109 us for the
    // FP32 copy of b, 35 and 72 for the prolongation)
    mg::k_emit<T, O><<<dim3((d.ncol + 127) / 128, (h->nlev + kc - 1) / kc), 128, 0, s>>>(d.n, d.ncol, h->nlev, kc, d.hd, x,
                                                                                         xc, out);
    CK(cudaGetLastError());
    return MG_OK;
}

// The precisions of the V-cycle: workspace and launches of one level.
struct Cyc64 {
    typedef double T;
    static T* x(DevLevel& d, int i) { return d.x64[i]; }
    static T* b(DevLevel& d) { return d.b64; }
    static T* r(DevLevel& d) { return d.r64; }
    static mg_status sweep(mg_handle* h, int l, const T* x, const T* xc, const void* b, bool raw, T* bcopy, void* xo,
                           bool, double om, cudaStream_t s) {
        return launch_sweep64(h, l, lvl64(h, l), x, xc, xc ? h->lv[l + 1].ncol : 0, static_cast<const double*>(b), raw,
                              bcopy, static_cast<double*>(xo), om, s);
    }
    static mg_status restrict_(mg_handle* h, int l, const T* x, const T* b, T* bc, cudaStream_t s) {
        return launch_restrict64<false>(h, l, x, b, bc, s);
    }
    static mg_status copy_b(mg_handle* h, const double* b, cudaStream_t s) {
        const DevLevel& d = h->lv[0];
        Prof pr(h, MG_K_CONVERT, 0, 16.0 * cells(h, 0), s);
        mg::k_weight64<<<dim3((d.ncol + 127) / 128, h->nlev), 128, 0, s>>>(d.ncol, b, d.wA64, h->dz, d.b64);
        CK(cudaGetLastError());
        return MG_OK;
    }
};

template <typename C>
struct Cyc32 {
    typedef float T;
    static T* x(DevLevel& d, int i) { return d.x32[i]; }
    static T* b(DevLevel& d) { return d.b32; }
    static T* r(DevLevel& d) { return d.r32; }
    static mg_status sweep(mg_handle* h, int l, const T* x, const T* xc, const void* b, bool raw, T* bcopy, void* xo,
                           bool out64, double om, cudaStream_t s) {
        if constexpr (sizeof(C) == 4) {
            // MG_FP32_P64: the finest level eliminates with FP64 pivots
            if (l == 0 && h->lv[0].ipd) return launch_sweep32<C, double>(h, l, x, xc, b, raw, bcopy, xo, out64, om, s);
        }
        return launch_sweep32<C, float>(h, l, x, xc, b, raw, bcopy, xo, out64, om, s);
    }
    static mg_status restrict_(mg_handle* h, int l, const T* x, const T* b, T* bc, cudaStream_t s) {
        return launch_restrict32<C>(h, l, x, b, bc, s);
    }
    static mg_status copy_b(mg_handle* h, const double* b, cudaStream_t s) {
        return launch_emit<double, float>(h, 0, b, nullptr, h->lv[0].b32, s);
    }
};

// Algorithm 1 on level l; the result goes to `out` (FP64 on the finest level, the cycle's type
// below).  On every level the iterate starts at zero (x^(l+1) <- 0 of Algorithm 1; the V-cycle is
// used as a preconditioner, so x^(1) = 0 as well).  The finest level's right-hand side is the
// caller's FP64 array; its first sweep stores it in the cycle's form for the level's later kernels.
template <typename Cyc>
mg_status mgv(mg_handle* h, const Cycle& cy, int l, const void* b, void* out, cudaStream_t s) {
    static const char* const level_range[MG_MAX_LEVELS] = {"V-cycle level 0", "V-cycle level 1", "V-cycle level 2",
                                                           "V-cycle level 3", "V-cycle level 4", "V-cycle level 5",
                                                           "V-cycle level 6", "V-cycle level 7"};
    NvtxRange nvtx_(level_range[l]);   // the level and the levels below it (nested ranges)
    typedef typename Cyc::T T;
    DevLevel& d = h->lv[l];
    const bool coarsest = (l == cy.L - 1), finest = l == 0;
    const double om = cy.omega;
    const bool wide = finest && sizeof(T) == 4;   // the level's result leaves in FP64
    T* ws[2] = {Cyc::x(d, 0), Cyc::x(d, 1)};
    const T* bT = finest ? Cyc::b(d) : static_cast<const T*>(b);
    const int npre = coarsest ? cy.n_coarse : cy.n_pre;
    if (finest && npre == 0) TRY(Cyc::copy_b(h, static_cast<const double*>(b), s));
    T* cur = nullptr;
    for (int i = 0; i < npre; ++i) {
        const bool final = coarsest && i == npre - 1;
        T* dst = (cur == ws[0]) ? ws[1] : ws[0];
        const bool raw = finest && i == 0;
        // (a cycle of one sweep has no use for b in the cycle's form)
        TRY(Cyc::sweep(h, l, cur, nullptr, raw ? b : bT, raw, raw && !final ? Cyc::b(d) : nullptr, final ? out : dst,
                       final && wide, om, s));
        if (final) return MG_OK;
        cur = dst;
    }
    // residual and restriction onto level l+1
    DevLevel& dc = h->lv[l + 1];
    T* bc = Cyc::b(dc);
    TRY(Cyc::restrict_(h, l, cur, bT, bc, s));
    T* xc = Cyc::r(dc);
    TRY(mgv<Cyc>(h, cy, l + 1, bc, xc, s));
    // coarse-grid correction fused into the first post-smoothing sweep
    const int npost = cy.n_post;
    if (npost == 0) {
        if (wide) return launch_emit<T, double>(h, l, cur, xc, static_cast<double*>(out), s);
        return launch_emit<T, T>(h, l, cur, xc, static_cast<T*>(out), s);
    }
    for (int i = 0; i < npost; ++i) {
        const bool last = i == npost - 1;
        T* dst = (cur == ws[0]) ? ws[1] : ws[0];
        TRY(Cyc::sweep(h, l, cur, i == 0 ? xc : nullptr, bT, false, nullptr, last ? out : dst, last && wide, om, s));
        cur = dst;
    }
    return MG_OK;
}

// ---- the 9-cell stencil (Sec. 3.5): V-cycle with the tridiagonal smoother H_z-hat ----
// x_out = x + omega Hz^-1 (b - H x), x == NULL meaning a zero iterate: the residual with the
// full 9-cell stencil, then the column solves without the next-to-nearest fluxes
template <typename T, typename B, typename O>
mg_status sweep9(mg_handle* h, int lev, const T* x, const B* b, O* xo, double omega, cudaStream_t s) {
    typedef View<T, T> V;
    DevLevel& d = h->lv[lev];
    const Lvl<T, T> L = V::lvl(h, lev);
    Prof pr(h, MG_K_SWEEP, lev, (double)L.nlev * L.ncol * (sizeof(B) + 4.0 * sizeof(T) + sizeof(O) +
                                                           (x ? 2.0 * sizeof(T) : 0.0)), s);
    const dim3 g2((L.ncol + 127) / 128, L.nlev);
    mg::k_resid9<T, B><<<g2, 128, 0, s>>>(L, V::t2(d), x, b, V::scratch(d, 0));
    mg::k_thomas9<T, O><<<(L.ncol + 127) / 128, 128, 0, s>>>(L, V::scratch(d, 0), x, V::scratch(d, 1),
                                                              V::scratch(d, 2), xo, (T)omega);
    CK(cudaGetLastError());
    return MG_OK;
}

// y = H x on level `lev` in FP64 for the 9-cell stencil
mg_status launch_apply9(mg_handle* h, int lev, const double* x, double* y, cudaStream_t s) {
    const Lvl<double, double> L = View<double, double>::lvl(h, lev);
    Prof pr(h, MG_K_APPLY, lev, (double)L.nlev * L.ncol * 8.0 * 6, s);
    mg::k_apply9<double, double, double><<<dim3((L.ncol + 127) / 128, L.nlev), 128, 0, s>>>(L, h->lv[lev].T2_64, x, y);
    CK(cudaGetLastError());
    return MG_OK;
}

// bc = Restrict(b - H x) onto level lev + 1 (9-cell stencil; x == NULL: zero iterate)
template <typename T, typename B, typename O>
mg_status restrict9(mg_handle* h, int lev, const T* x, const B* b, O* bc, cudaStream_t s) {
    typedef View<T, T> V;
    DevLevel& d = h->lv[lev];
    const DevLevel& dc = h->lv[lev + 1];
    const Lvl<T, T> L = V::lvl(h, lev);
    Prof pr(h, MG_K_RESTRICT, lev, (double)L.nlev * L.ncol * (sizeof(B) + 2.0 * sizeof(T) + 0.25 * sizeof(O)), s);
    const dim3 g2((L.ncol + 127) / 128, L.nlev);
    mg::k_resid9<T, B><<<g2, 128, 0, s>>>(L, V::t2(d), x, b, V::scratch(d, 0));
    mg::k_restrict_sum<T, O><<<dim3((dc.ncol + 127) / 128, L.nlev), 128, 0, s>>>(d.n, d.ncol, L.nlev, V::scratch(d, 0),
                                                                               V::w(d), bc, dc.ncol);
    CK(cudaGetLastError());
    return MG_OK;
}

// Algorithm 1 for the 9-cell stencil: the same steps as mgv, each a plain kernel (the
// right-hand side converted on entry and the result on exit in the FP32 variant)
template <typename T, typename B, typename O>
mg_status mgv9(mg_handle* h, const Cycle& cy, int l, const B* b, O* out, cudaStream_t s) {
    typedef View<T, T> V;
    DevLevel& d = h->lv[l];
    const size_t n = cells(h, l);
    const bool coarsest = (l == cy.L - 1);
    const double om = cy.omega;
    const T* bT = (const T*)(const void*)b;
    if (!std::is_same<B, T>::value) {
        TRY(launch_convert(h, l, n, b, V::b(d), s));
        bT = V::b(d);
    }
    T* ws[2] = {V::x(d, 0), V::x(d, 1)};
    T* cur = nullptr;
    auto other = [&]() { return cur == ws[0] ? ws[1] : ws[0]; };
    const int npre = coarsest ? cy.n_coarse : cy.n_pre;
    for (int i = 0; i < npre; ++i) {
        T* dst = other();
        TRY((sweep9<T, T, T>(h, l, cur, bT, dst, om, s)));
        cur = dst;
    }
    if (!coarsest) {
        DevLevel& dc = h->lv[l + 1];
        TRY((restrict9<T, T, T>(h, l, cur, bT, V::b(dc), s)));
        T* xc = V::r(dc);
        TRY((mgv9<T, T, T>(h, cy, l + 1, V::b(dc), xc, s)));
        T* dst = other();
        if (cur) TRY((launch_prolong<T, false, T, T>(h, l, d.n, d.ncol, dc.ncol, h->nlev, cur, xc, dst, s)));
        else TRY((launch_prolong<T, true, T, T>(h, l, d.n, d.ncol, dc.ncol, h->nlev, cur, xc, dst, s)));
        cur = dst;
        for (int i = 0; i < cy.n_post; ++i) {
            T* dst2 = other();
            TRY((sweep9<T, T, T>(h, l, cur, bT, dst2, om, s)));
            cur = dst2;
        }
    }
    if (!cur) {
        CK(cudaMemsetAsync(out, 0, n * sizeof(O), s));
        return MG_OK;
    }
    return launch_convert(h, l, n, (const T*)cur, out, s);
}

mg_status run_cycle(mg_handle* h, const Cycle& cy, const double* b, double* x, cudaStream_t s) {
    if (h->nine) {
        switch (h->prm.vcycle_precision) {
            case MG_FP64: return mgv9<double, double, double>(h, cy, 0, b, x, s);
            case MG_FP32: return mgv9<float, double, double>(h, cy, 0, b, x, s);   // (MG_FP32_P64: not built)
            default: return MG_ERR_UNSUPPORTED;
        }
    }
    switch (h->prm.vcycle_precision) {
        case MG_FP64: return mgv<Cyc64>(h, cy, 0, b, x, s);
        case MG_FP32:
        case MG_FP32_P64: return mgv<Cyc32<float>>(h, cy, 0, b, x, s);
        case MG_FP32_BF16COEF: return mgv<Cyc32<bf16>>(h, cy, 0, b, x, s);
        default: return MG_ERR_ARG;
    }
}

mg_status run_vcycle(mg_handle* h, const double* b, double* x, cudaStream_t s) {
    return run_cycle(h, vcycle_of(h), b, x, s);
}

// P_H^(Jac)(omega, n) of Sec. 4.1: n block-Jacobi sweeps from zero on the finest level, in the
// handle's V-cycle precision (a one-level cycle)
mg_status run_jacobi(mg_handle* h, double omega, int sweeps, const double* b, double* x, cudaStream_t s) {
    return run_cycle(h, Cycle{1, omega, 0, 0, sweeps}, b, x, s);
}

// The status of a solve whose residual is no longer finite: a sweep's copy that did not arrive leaves NaN
// and a flag, which every solve clears at its start.
mg_status broken(mg_handle* h, cudaStream_t s) {
    unsigned int late = 0;
    CK(cudaMemcpyAsync(&late, h->timeout, sizeof late, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    return late ? MG_ERR_TIMEOUT : MG_ERR_BREAKDOWN;
}

// BiCGStab(H, P, tol) on the finest level (Sec. 4.1 solver list; Table 1 "Krylov" rows) from
// x = 0: the vector updates and inner products run in the kernels above with device scalars;
// the host reads them once per iteration to test convergence.  *iters counts a half step as 0.5.
template <typename Pre>
mg_status bicgstab(mg_handle* h, const double* b, double* x, double tol, int maxit, Pre& P, cudaStream_t s,
                   double* iters) {
    const size_t n = cells(h, 0);
    double *rh = h->bv[0], *r = h->bv[1], *p = h->bv[2], *v = h->bv[3], *sv = h->bv[4], *t = h->bv[5],
           *ph = h->bv[6], *sh = h->bv[7];
    if (!rh) return MG_ERR_UNSUPPORTED;
    const Lvl<double, double> L = View<double, double>::lvl(h, 0);
    const dim3 ag((L.ncol + 127) / 128, L.nlev);
    const int G = vec_grid(h, cells(h, 0)), B = mg::RED_THREADS;
    unsigned int* tk = h->tickets + TK_BICG;
    auto apply = [&](const double* in, double* out) -> mg_status {
        if (h->nine) return launch_apply9(h, 0, in, out, s);
        Prof pr(h, MG_K_APPLY, 0, 8.0 * n * 9, s);
        mg::k_apply_a6<<<ag, 128, 0, s>>>(L, h->a6, in, out);
        CK(cudaGetLastError());
        return MG_OK;
    };
    *iters = 0.0;
    mg::k_bicg_start<<<G, B, 0, s>>>(n, b, r, rh, x, tol, h->partials, tk, h->bs, h->timeout);
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(h->host_bs, h->bs, sizeof(mg::BicgScal), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (!std::isfinite(h->host_bs->bb)) return MG_ERR_BREAKDOWN;
    if (h->host_bs->bb == 0.0) return MG_OK;
    for (int i = 0; i < maxit; ++i) {
        mg::k_bicg_dir<<<G, B, 0, s>>>(n, r, v, p, i == 0, h->bs);
        CK(cudaGetLastError());
        TRY(P(p, ph));
        TRY(apply(ph, v));
        mg::k_bicg_alpha<<<G, B, 0, s>>>(n, rh, v, h->partials, tk, h->bs);
        mg::k_bicg_s<<<G, B, 0, s>>>(n, r, v, sv, h->partials, tk, h->bs);
        CK(cudaGetLastError());
        TRY(P(sv, sh));
        TRY(apply(sh, t));
        mg::k_bicg_omega<<<G, B, 0, s>>>(n, t, sv, h->partials, tk, h->bs);
        mg::k_bicg_xr<<<G, B, 0, s>>>(n, x, r, ph, sh, sv, t, rh, h->partials, tk, h->bs);
        CK(cudaGetLastError());
        CK(cudaMemcpyAsync(h->host_bs, h->bs, sizeof(mg::BicgScal), cudaMemcpyDeviceToHost, s));
        CK(cudaStreamSynchronize(s));
        const mg::BicgScal& S = *h->host_bs;
        if (!std::isfinite(S.alpha) || !std::isfinite(S.ss)) return broken(h, s);
        if (S.half) {
            *iters = i + 0.5;
            return MG_OK;
        }
        if (!std::isfinite(S.omega) || !std::isfinite(S.rr) || !std::isfinite(S.rho)) return broken(h, s);
        *iters = i + 1.0;
        if (S.rr <= S.tol2bb) return MG_OK;
        if (S.omega == 0.0 || S.rho == 0.0) return MG_ERR_BREAKDOWN;
    }
    return MG_ERR_NOT_CONVERGED;
}

// x ~ H^-1 b by the handle's pressure solver: one V-cycle (MG(L)), line relaxation, or
// BiCGStab to eps_H preconditioned by one of the two (Table 1); *iters as for bicgstab
mg_status run_pressure_solver(mg_handle* h, const double* b, double* x, cudaStream_t s, double* iters) {
    const mg_pressure_solver& ps = h->ps;
    *iters = 0.0;
    mg_status st = MG_OK;
    switch (ps.kind) {
        case MG_PS_MG: st = run_vcycle(h, b, x, s); break;
        case MG_PS_JACOBI: st = run_jacobi(h, ps.omega, ps.sweeps, b, x, s); break;
        case MG_PS_BICGSTAB_JACOBI: {
            auto P = [&](const double* in, double* out) { return run_jacobi(h, ps.omega, ps.sweeps, in, out, s); };
            st = bicgstab(h, b, x, ps.eps, ps.max_iter, P, s, iters);
            break;
        }
        case MG_PS_BICGSTAB_MG: {
            auto P = [&](const double* in, double* out) { return run_vcycle(h, in, out, s); };
            st = bicgstab(h, b, x, ps.eps, ps.max_iter, P, s, iters);
            break;
        }
        default: return MG_ERR_ARG;
    }
    if (ps.kind == MG_PS_BICGSTAB_JACOBI || ps.kind == MG_PS_BICGSTAB_MG) {
        h->ps_solves += 1;
        h->ps_iters += *iters;
    }
    return st;
}

// the pressure solver synchronises with the host (BiCGStab): the mixed GCR then launches its
// iterations directly instead of capturing them into graphs
inline bool ps_syncs(const mg_handle* h) {
    return h->ps.kind == MG_PS_BICGSTAB_JACOBI || h->ps.kind == MG_PS_BICGSTAB_MG;
}

// ---- GCR (Sec. 4.1; textbook generalised conjugate residual, right preconditioned) ----
// Per iteration j of a restart cycle: z_j = P r (raw), w_j = A z_j with the inner products
// <w_j, w_i>, <r, w_i>, <w_j, w_j>, <r, w_j> fused into the same pass (coefficients by
// classical Gram-Schmidt), then one pass orthogonalises w_j in place and updates r with
// <r, r>.  x is formed from the raw z_i once per cycle (or at the end).
// Run-time direction count j -> kernel instantiated for exactly j directions.
template <template <int> class K, typename... A>
mg_status dispatch_j(int j, A&&... a) {
    switch (j) {
#define MG_J(n) \
    case n: return K<n>::run(std::forward<A>(a)...);
        MG_J(0) MG_J(1) MG_J(2) MG_J(3) MG_J(4) MG_J(5) MG_J(6) MG_J(7)
        MG_J(8) MG_J(9) MG_J(10) MG_J(11) MG_J(12) MG_J(13) MG_J(14) MG_J(15)
#undef MG_J
        default: return MG_ERR_ARG;
    }
}

template <int J>
struct RunSums {
    static mg_status run(mg_handle* h, size_t n, const double* w, cudaStream_t s) {
        Prof pr(h, MG_K_GCR_DOTS, 0, 8.0 * n * (J + 2), s);   // w, r, w_i
        mg::k_gcr_sums<J><<<vec_grid(h, n), mg::RED_THREADS, 0, s>>>(n, w, h->W, h->glen, h->r, h->partials,
                                                                   h->tickets + TK_SUMS, h->gs);
        CK(cudaGetLastError());
        return MG_OK;
    }
};

template <int J>
struct RunApplyGcr {
    static mg_status run(mg_handle* h, const double* z, double* w, cudaStream_t s) {
        const Lvl<double, double> L = View<double, double>::lvl(h, 0);
        const double nc = (double)L.nlev * L.ncol;
        // z, the couplings (6 and the diagonal), w, r, w_i
        Prof pr(h, MG_K_APPLY, 0, nc * 8.0 * (1 + 7 + 1 + 1 + J), s, J);
        const int groups = (L.ncol + 31) / 32, per_block = mg::RED_THREADS / 32;
        const int kc = mg::apply_chunk(groups, L.nlev, mg::APPLY_BLOCKS * h->nsm * per_block), nk = (L.nlev + kc - 1) / kc;
        const int grid = std::min(mg::APPLY_BLOCKS * h->nsm, (int)(((long long)groups * nk + per_block - 1) / per_block));
        mg::k_apply_gcr<J><<<grid, mg::RED_THREADS, 0, s>>>(L, h->a6, z, w, h->W, h->glen, h->r, kc, nk,
                                                            h->partials,
                                                            h->tickets + TK_SUMS, h->gs);
        CK(cudaGetLastError());
        return MG_OK;
    }
};

template <int J>
struct RunOrth {
    static mg_status run(mg_handle* h, size_t n, cudaStream_t s) {
        Prof pr(h, MG_K_GCR_ORTH, 0, 8.0 * n * (J > 0 ? J + 4 : 3), s);
        mg::k_gcr_orth_update<J><<<vec_grid(h, n), mg::RED_THREADS, 0, s>>>(n, h->W, h->glen, h->r, h->partials,
                                                                         h->tickets + TK_ORTH, h->gs);
        CK(cudaGetLastError());
        return MG_OK;
    }
};

template <int J>
struct RunXupd {
    static mg_status run(mg_handle* h, size_t n, double* x, cudaStream_t s) {
        Prof pr(h, MG_K_GCR_UPDATE, 0, 8.0 * n * (J + 3), s);
        mg::k_gcr_xupdate<J><<<vec_grid(h, n), mg::RED_THREADS, 0, s>>>(n, x, h->Z, h->glen, h->gs);
        CK(cudaGetLastError());
        return MG_OK;
    }
};

mg_status gcr_sums(mg_handle* h, size_t n, const double* w, int j, cudaStream_t s) {
    return dispatch_j<RunSums>(j, h, n, w, s);
}

mg_status apply_gcr(mg_handle* h, const double* z, double* w, int j, cudaStream_t s) {
    if (h->nine) {
        TRY(launch_apply9(h, 0, z, w, s));
        return gcr_sums(h, cells(h, 0), w, j, s);
    }
    return dispatch_j<RunApplyGcr>(j, h, z, w, s);
}

// Capture the launches of `body` into *out (left null, and graphs switched off for the
// handle, if the capture or the instantiation fails; the caller then launches directly).
template <typename Body>
void capture_graph(mg_handle* h, Body& body, cudaGraphExec_t* out) {
    *out = nullptr;
    cudaGraph_t g = nullptr;
    if (cudaStreamBeginCapture(h->cap, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
        const mg_status st = body(h->cap);
        const cudaError_t e = cudaStreamEndCapture(h->cap, &g);
        if (st == MG_OK && e == cudaSuccess && g && cudaGraphInstantiate(out, g, 0) != cudaSuccess) *out = nullptr;
        if (g) cudaGraphDestroy(g);
    }
    if (!*out) {
        h->graphs_off = true;
        cudaGetLastError();
    }
}

// Drop the cached graphs of the systems from `first` on; the next solve captures them again.
void drop_graphs(mg_handle* h, int first) {
    for (int sys = first; sys < 3; ++sys)
        for (cudaGraphExec_t& g : h->gexec[sys])
            if (g) {
                cudaGraphExecDestroy(g);
                g = nullptr;
            }
}

// One GCR solve as resumable steps, so that several solves (an ensemble of handles) can
// interleave their iterations on their own streams: start (enqueue r = b, x = 0, <b, b>),
// started (after a synchronisation: read <b, b>), launch (enqueue one iteration, ending with
// the read-back of <r, r>), landed (after a synchronisation: read <r, r>, decide, enqueue the
// solution update when the cycle ends or the solve stops), end (enqueue the closing event).
struct GcrRun {
    int sys = 0;          // 0 pressure, 1 mixed, 2 mixed adjoint: selects the handle's cached graphs
    size_t n = 0;
    double* x = nullptr;
    double tol = 0.0;
    double bb = 0.0, rel = 0.0;
    int it = 0;
    mg_status st = MG_OK;
    bool active = false;  // iterations left to launch
};

mg_status gcr_start(mg_handle* h, GcrRun& g, const double* b, cudaStream_t s) {
    CK(cudaEventRecord(h->ev0, s));
    {
        Prof pr(h, MG_K_DOT, 0, 24.0 * g.n, s);
        mg::k_gcr_start<<<vec_grid(h, g.n), mg::RED_THREADS, 0, s>>>(g.n, b, h->r, g.x, h->partials, h->tickets + TK_DOT,
                                                                    &h->gs->bb, h->host_sc + 1, h->timeout);
        CK(cudaGetLastError());
    }
    return MG_OK;
}

void gcr_started(mg_handle* h, GcrRun& g) {
    g.bb = h->host_sc[1];
    g.it = 0;
    g.rel = 0.0;
    g.active = false;
    g.st = MG_OK;
    if (!std::isfinite(g.bb)) {
        g.st = MG_ERR_BREAKDOWN;
    } else if (g.bb > 0.0) {
        g.rel = 1.0;
        g.st = MG_ERR_NOT_CONVERGED;
        g.active = h->prm.max_iter > 0;
    }
}

template <typename ApplyAS, typename ApplyP>
mg_status gcr_launch(mg_handle* h, GcrRun& g, cudaStream_t s, ApplyAS& applyAS, ApplyP& applyP) {
    const int j = g.it % h->prm.gcr_restart;
    double* z = h->Z + (size_t)j * h->glen;
    double* w = h->W + (size_t)j * h->glen;
    const size_t n = g.n;
    // every buffer of the iteration belongs to the handle, so its launches form a fixed
    // sequence per slot j
    auto body = [&](cudaStream_t q) -> mg_status {
        TRY(applyP(h->r, z, q));
        TRY(applyAS(z, w, j, q));
        TRY(dispatch_j<RunOrth>(j, h, n, q));
        CK(cudaMemcpyAsync(h->host_sc, &h->gs->rr, sizeof(double), cudaMemcpyDeviceToHost, q));
        return MG_OK;
    };
    cudaGraphExec_t& ge = h->gexec[g.sys][j];
    const bool direct = h->prof || (g.sys != 0 && ps_syncs(h));
    if (!ge && !direct && !h->graphs_off) capture_graph(h, body, &ge);
    if (ge && !direct) CK(cudaGraphLaunch(ge, s));
    else TRY(body(s));
    return MG_OK;
}

mg_status gcr_landed(mg_handle* h, GcrRun& g, cudaStream_t s) {
    const int j = g.it % h->prm.gcr_restart;
    ++g.it;
    const double rr = h->host_sc[0];
    if (!std::isfinite(rr)) {
        g.st = broken(h, s);
        g.active = false;
        return MG_OK;
    }
    g.rel = std::sqrt(rr / g.bb);
    const bool done = g.rel <= g.tol;
    if (j == h->prm.gcr_restart - 1 || done || g.it == h->prm.max_iter)
        TRY(dispatch_j<RunXupd>(j, h, g.n, g.x, s));
    if (done) g.st = MG_OK;
    g.active = !done && g.it < h->prm.max_iter;
    return MG_OK;
}

void gcr_info(mg_handle* h, const GcrRun& g, mg_solve_info* info) {
    if (!info) return;
    float ms = 0.f;
    cudaEventElapsedTime(&ms, h->ev0, h->ev1);
    info->iters = g.it;
    info->rel_res = g.rel;
    info->ms = ms;
}

template <typename ApplyAS, typename ApplyP>
mg_status gcr(mg_handle* h, int sys, size_t n, const double* b, double* x, double tol, mg_solve_info* info,
              cudaStream_t s, ApplyAS applyAS, ApplyP applyP) {
    GcrRun g;
    g.sys = sys;
    g.n = n;
    g.x = x;
    g.tol = tol;
    TRY(gcr_start(h, g, b, s));
    CK(cudaStreamSynchronize(s));
    gcr_started(h, g);
    while (g.active) {
        NvtxRange it_("gcr iteration");
        TRY(gcr_launch(h, g, s, applyAS, applyP));
        CK(cudaStreamSynchronize(s));
        TRY(gcr_landed(h, g, s));
    }
    CK(cudaEventRecord(h->ev1, s));
    CK(cudaEventSynchronize(h->ev1));
    gcr_info(h, g, info);
    return g.st;
}

// ---- mixed operator and Schur-complement preconditioner ----
// One form of k_mixed (krylov.cuh), with the GCR sums of direction J unless J < 0; wu: see there.
template <int MODE, int J>
mg_status launch_mixed(mg_handle* h, const double* u, const double* p, double* yu, double* yp, double* wu,
                       cudaStream_t s) {
    const mg::MixedDev& M = h->md;
    const int gh = (M.nfh + 31) / 32, gc = (M.ncol + 31) / 32, per_block = mg::RED_THREADS / 32;
    const int G = MODE == mg::MX_RHS ? gc : MODE >= mg::MX_UPDATE ? gh + gc : gh + 2 * gc;
    const int slots = mg::mixed_blocks(MODE) * h->nsm, kc = mg::apply_chunk(G, M.nlev, slots * per_block);
    const int nk = (M.nlev + kc - 1) / kc;
    const int grid = (int)std::min((long long)slots, ((long long)G * nk + per_block - 1) / per_block);
    mg::k_mixed<MODE, J><<<grid, mg::RED_THREADS, 0, s>>>(M, u, p, yu, yp, wu, h->W, h->glen, h->r, kc, nk,
                                                          h->partials, h->tickets + TK_SUMS, h->gs);
    CK(cudaGetLastError());
    return MG_OK;
}

// y = A v (MX_A) or A-hat v (MX_HAT, wu = W v_u) of a concatenated v = [u; p], with the GCR sums of direction j
template <int MODE>
struct RunMixed {
    template <int J>
    struct K {
        static mg_status run(mg_handle* h, const double* v, double* y, double* wu, cudaStream_t s) {
            const size_t nu = (size_t)h->nu;
            const double n = nu + cells(h, 0);
            // u, kd (W u) per velocity row and the row, p; of the sums r and the stored directions
            Prof pr(h, MG_K_MIXED, 0, 8.0 * ((MODE == mg::MX_HAT ? 3.0 : 2.0) * nu + 3.0 * cells(h, 0) + (J + 1) * n), s,
                    MODE == mg::MX_HAT ? 2 : 0);
            return launch_mixed<MODE, J>(h, v, v + nu, y, y + nu, wu, s);
        }
    };
};

template <bool MULT>
mg_status mixed_adj_scale(mg_handle* h, const double* in_u, const double* in_p, double* out_u, double* out_p,
                          cudaStream_t s) {
    Prof pr(h, MG_K_DOT, 0, 16.0 * ((double)h->nu + (double)cells(h, 0)), s, MULT ? 1 : 0);
    mg::k_mx_adj_scale<MULT><<<4 * h->nsm, 256, 0, s>>>(h->md, (size_t)h->nu, h->area0, h->dz, in_u, in_p, out_u,
                                                          out_p);
    CK(cudaGetLastError());
    return MG_OK;
}

// wu: takes W u' as well (null: not wanted)
mg_status schur_impl(mg_handle* h, const double* ru, const double* rp, double* u, double* p, double* wu,
                     cudaStream_t s) {
    // Step 1: B = r_p - D M-ring^{-1} r_u
    TRY((launch_mixed<mg::MX_RHS, -1>(h, ru, rp, nullptr, h->schurB, nullptr, s)));
    // Step 2: H Pi' = B by the pressure solver K_H(A_H, P_H, eps_H) (one V-cycle by default);
    // an inexact inner solve (BiCGStab at its iteration limit) is still a usable preconditioner
    double it = 0.0;
    const mg_status st = run_pressure_solver(h, h->schurB, p, s, &it);
    if (st != MG_OK && st != MG_ERR_NOT_CONVERGED) return st;
    // Step 3: u' = M-ring^{-1} (r_u - G Pi')
    if (wu) return launch_mixed<mg::MX_UPDATE_W, -1>(h, ru, p, u, nullptr, wu, s);
    return launch_mixed<mg::MX_UPDATE, -1>(h, ru, p, u, nullptr, nullptr, s);
}

// the rim cell of the padded fields that repeats each edge column (Lvl32::hd), [4][ncol]
__global__ void k_rims(int n, int ncol, const int32_t* __restrict__ nbr, int32_t* __restrict__ hd) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, s = blockIdx.y;
    if (c >= ncol) return;
    const int np = mg::pad_row(n), step[4] = {1, -1, np, -np};
    const mg::Pos at(c, n, np);
    const bool edge = s == 0 ? at.i + 1 == (unsigned)n : s == 1 ? at.i == 0 : s == 2 ? at.j + 1 == (unsigned)n : at.j == 0;
    int d = -1;
    if (edge) {
        const int nb = nbr[(size_t)s * ncol + c];
        for (int t = 0; t < 4; ++t)   // the neighbour's side that faces this column
            if (nbr[(size_t)t * ncol + nb] == c) d = (int)mg::Pos(nb, n, np).cp + step[t];
    }
    hd[(size_t)s * ncol + c] = d;
}

__global__ void k_reciprocal(size_t n, const double* __restrict__ a, double* __restrict__ r) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        r[i] = 1.0 / a[i];
}

// parents of the neighbours E, W, N, S and of the column itself (Lvl64::par), [5][ncol]
__global__ void k_parents(int n, int ncol, const int32_t* __restrict__ nbr, int32_t* __restrict__ par) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, s = blockIdx.y;
    if (c < ncol) par[(size_t)s * ncol + c] = mg::parent_col(s < 4 ? nbr[(size_t)s * ncol + c] : c, n);
}

// Tensor maps of the TMA sweep (sweep_tma.cuh) for an FP32 level of 8 levels or more.
mg_status build_maps(mg_handle* h, int l) {
    DevLevel& d = h->lv[l];
    d.maps.clear();
    if (h->nine || !d.ip32 || h->nlev < 8) return MG_OK;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult found;
    CK(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found));
    if (!fn || found != cudaDriverEntryPointSuccess) return MG_ERR_CUDA;
    const auto encode = reinterpret_cast<decltype(&cuTensorMapEncodeTiled)>(fn);
    bool ok = true;
    const int H = (h->nlev + 1) / 2;
    // a padded field of C_n, boxes of `cols` columns x `rows` levels
    auto map = [&](CUtensorMap* out, const auto* base, int n, int levels, int cols, int rows) {
        const cuuint64_t size = sizeof(*base), dims[2] = {(cuuint64_t)mg::padded(n), (cuuint64_t)levels};
        const cuuint64_t stride[1] = {size * dims[0]};
        const cuuint32_t boxes[2] = {(cuuint32_t)cols, (cuuint32_t)rows}, one[2] = {1, 1};
        ok &= encode(out, size == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                     const_cast<void*>(static_cast<const void*>(base)), dims, stride, boxes, one,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    d.maps.resize(2);
    for (int i = 0; i < 2; ++i) {
        mg::SweepMaps& m = d.maps[i];
        const int n = d.n, N = h->nlev;
        auto coefs = [&](const auto* te, const auto* tn, const auto* tv) {
            map(&m.te, te, n, N, 32 + 16 / (int)sizeof(*te), H);
            map(&m.tn, tn, n, N, 32, H);
            map(&m.tv, tv, n, N + 1, 32, H + 1);
        };
        if (d.te32) coefs(d.te32, d.tn32, d.tv32);
        else coefs(d.te16, d.tn16, d.tv16);
        map(&m.b, d.b32, n, N, 32, H);
        map(&m.ip, d.ip32, n, N, 32, H);
        map(&m.x, d.x32[i], n, N, 40, H + 1);
        map(&m.xr, d.x32[i], n, N, 32, H);
        if (l + 1 < h->L) {
            map(&m.xc, h->lv[l + 1].r32, h->lv[l + 1].n, N, 24, H + 1);
            map(&m.xca, h->lv[l + 1].r32, h->lv[l + 1].n, N, 24, H);
        }
    }
    return ok ? MG_OK : MG_ERR_CUDA;
}

// Memory of level l's FP64 level data, in one piece: a failed call leaves nothing behind.
mg_status alloc64(mg_handle* h, int l) {
    DevLevel& d = h->lv[l];
    const size_t N = cells(h, l), rim = (size_t)h->nlev * 6 * d.n;
    Pieces p;
    for (double** q : {&d.te64, &d.tn64, &d.e64, &d.ip64}) p.add(q, N);
    for (double** q : {&d.tbw64, &d.tbs64}) p.add(q, rim);
    if (mg::sweep64_levels(h->nlev, d.ncol) == 10) p.add(&d.pr64, (size_t)mg::sweep64_chunks(h->nlev, d.ncol) * d.ncol);
    p.add(&d.tv64, N + d.ncol);
    return p.alloc(h);
}

mg_status pack64(mg_handle* h, int l, cudaStream_t s) {
    DevLevel& d = h->lv[l];
    const dim3 grid((d.ncol + 127) / 128, h->nlev + 1);
    mg::k_pack64<<<grid, 128, 0, s>>>(d.n, d.ncol, h->nlev, d.fof, d.Th64, d.Tv64, d.wA64, h->dz, h->scale, d.te64, d.tn64,
                                      d.tbw64, d.tbs64, d.tv64, d.ip64);
    mg::k_factor64<<<(d.ncol + 63) / 64, 64, 0, s>>>(d.ncol, h->nlev, d.tv64, d.e64, d.ip64, d.pr64,
                                                     mg::sweep64_chunks(h->nlev, d.ncol), h->om0);
    CK(cudaGetLastError());
    return MG_OK;
}

// A handle whose V-cycle is not in FP64 has FP64 level data for mg_smooth, mg_smooth_noalloc and
// mg_residual_restrict alone (40 of about 300 bytes per cell, C96L70: 0.12 ms for the finest level).  They are
// packed when one of these first asks, and from then on by mg_set_coefficients; levels that mg_smooth_noalloc
// takes have their memory from set-up, others from that first call.  The first call waits for the packing, so
// that calls on other streams and from other threads find the data complete.  Under stream capture it runs
// on the handle's own stream (the couplings are in place: set-up and mg_set_coefficients synchronise), so that a
// graph does not pack again each time it is replayed; only then, because a process that has run work on
// several streams launches slower from then on (C64L40 solve 1.57 -> 1.67 ms after seven handles' streams).
mg_status ready64(mg_handle* h, int l, cudaStream_t s) {
    DevLevel& d = h->lv[l];
    std::lock_guard<std::mutex> lock(h->pack_mutex);
    if (d.packed64) return MG_OK;
    cudaStreamCaptureStatus cst;
    CK(cudaStreamIsCapturing(s, &cst));
    if (cst != cudaStreamCaptureStatusNone) s = h->run;
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;   // (none of this is work of a stream under capture)
    CK(cudaThreadExchangeStreamCaptureMode(&mode));
    const mg_status st = [&]() -> mg_status {
        if (!d.tv64) TRY(alloc64(h, l));
        TRY(pack64(h, l, s));
        CK(cudaStreamSynchronize(s));
        return MG_OK;
    }();
    CK(cudaThreadExchangeStreamCaptureMode(&mode));
    TRY(st);
    d.wants64 = d.packed64 = true;
    return MG_OK;
}

// The level data of the sweeps and restrictions from level l's FP64 face form, in every precision that
// is in use.
mg_status pack_level(mg_handle* h, int l, cudaStream_t s) {
    DevLevel& d = h->lv[l];
    d.packed64 = d.wants64;
    if (d.wants64) TRY(pack64(h, l, s));
    const dim3 grid((d.ncol + 127) / 128, h->nlev + 1);
    const dim3 halves((d.ncol + 63) / 64, 2);
    if (d.te32) {
        mg::k_pack32<float><<<grid, 128, 0, s>>>(d.n, d.ncol, h->nlev, d.fof, d.Th64, d.Tv64, d.te32, d.tn32, d.tv32);
        mg::k_factor32<float, float><<<halves, 64, 0, s>>>(lvl32<float, float>(h, l), d.ip32, nullptr, nullptr);
        if (d.ipd)
            mg::k_factor32<float, double><<<halves, 64, 0, s>>>(lvl32<float, double>(h, l), d.ipd, d.md, d.ed);
    }
    if (d.te16) {
        mg::k_pack32<bf16><<<grid, 128, 0, s>>>(d.n, d.ncol, h->nlev, d.fof, d.Th64, d.Tv64, d.te16, d.tn16, d.tv16);
        mg::k_factor32<bf16, float><<<halves, 64, 0, s>>>(lvl32<bf16, float>(h, l), d.ip32, nullptr, nullptr);
    }
    CK(cudaGetLastError());
    return MG_OK;
}

// Replaces the finest-level operator by the caller's couplings a[s][k][c] (DEVICE, 6 N): the
// FP64 operator of the GCR apply takes them as they are, the V-cycle's finest level their face
// form in its precision.  A first pass only checks them (flux symmetry, sign, no flux through
// surface and lid); the operator is changed only if every check passes.
mg_status set_coefficients_impl(mg_handle* h, const double* a, cudaStream_t s) {
    const int ncol = h->lv[0].ncol, nlev = h->nlev, blocks = (2 * ncol + 127) / 128;
    const DevLevel& d = h->lv[0];
    mg::k_coef<false><<<dim3(blocks, 2 * nlev + 1), 128, 0, s>>>(ncol, nlev, h->faceL0, h->faceR0, h->faceSide0, h->nbrSide0,
                                                                 h->area0, h->dz, a, d.Th64, d.Tv64, h->a6, h->flag);
    CK(cudaGetLastError());
    unsigned int* const bad = reinterpret_cast<unsigned int*>(h->host_sc + 2);
    CK(cudaMemcpyAsync(bad, h->flag, sizeof *bad, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (*bad) {
        CK(cudaMemsetAsync(h->flag, 0, sizeof *h->flag, s));   // (clear at the start of every call)
        CK(cudaStreamSynchronize(s));
        return MG_ERR_ARG;
    }
    mg::k_coef<true><<<dim3(blocks, 3 * nlev + 1), 128, 0, s>>>(ncol, nlev, h->faceL0, h->faceR0, h->faceSide0, h->nbrSide0,
                                                                h->area0, h->dz, a, d.Th64, d.Tv64, h->a6, h->flag);
    CK(cudaGetLastError());
    TRY(pack_level(h, 0, s));
    CK(cudaStreamSynchronize(s));
    return MG_OK;
}

// x_out = x_in (NULL: zero) after `sweeps` block-Jacobi sweeps in FP64 with one scratch array: they alternate
// between it and x_out, ordered so that the last one writes x_out.  A sweep never writes the array it
// reads: where x_in is x_out and that would be the first target, the first sweep goes to the scratch array and
// the result is copied at the end.  (rec is NULL where no launch may be recorded.)
mg_status smooth_into(mg_handle* h, mg_handle* rec, int level, const double* b, const double* x_in, double* x_out,
                      int sweeps, double* scratch, cudaStream_t s) {
    const size_t n = cells(h, level);
    if (sweeps == 0) {
        if (!x_in) CK(cudaMemsetAsync(x_out, 0, n * sizeof(double), s));
        else if (x_in != x_out) CK(cudaMemcpyAsync(x_out, x_in, n * sizeof(double), cudaMemcpyDeviceToDevice, s));
        return MG_OK;
    }
    if (!h->nine) TRY(ready64(h, level, s));
    const Lvl64 L = lvl64(h, level);
    bool to_out = sweeps % 2 == 1 && x_in != x_out;
    const double* cur = x_in;
    for (int i = 0; i < sweeps; ++i) {
        double* dst = to_out ? x_out : scratch;
        if (h->nine) TRY((sweep9<double, double, double>(h, level, cur, b, dst, h->prm.omega, s)));
        else TRY(launch_sweep64(rec, level, L, cur, nullptr, 0, b, true, nullptr, dst, h->prm.omega, s));
        cur = dst;
        to_out = !to_out;
    }
    if (cur != x_out) CK(cudaMemcpyAsync(x_out, cur, n * sizeof(double), cudaMemcpyDeviceToDevice, s));
    return MG_OK;
}

mg_status check_level(const mg_handle* h, int level) {
    if (!h || level < 0 || level >= h->L) return MG_ERR_ARG;
    return MG_OK;
}

struct DeviceGuard {
    int prev = -1;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) cudaSetDevice(dev);
        else prev = -1;
    }
    ~DeviceGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

// Horizontal-face velocity mass M_h = M2 + tau_u dt M_C of the mixed system (level-
// independent): the self weight, up to 6 couplings per face (the opposite face in each of
// its two cells, then the two perpendicular faces in each) and the lumped diagonal.
struct HMass {
    int ncf = 0;                  // couplings per face (0 or 6)
    double ms = 1.0;              // self weight (2/3 consistent, 1 lumped)
    std::vector<int32_t> cf;      // [6][nfh] coupled face
    std::vector<double> wf;       // [6][nfh] its weight
    std::vector<double> mlump;    // [nfh] row sums in the cells' own axes
};

void horizontal_mass(const mg::HGeom& G, bool consistent, double f0, HMass& hm) {
    const int ncol = G.ncol, nfh = 2 * ncol;
    const double outward[4] = {1.0, -1.0, 1.0, -1.0};   // E, W, N, S along +xi, -xi, +eta, -eta
    hm.ms = consistent ? 2.0 / 3.0 : 1.0;
    hm.ncf = (consistent || f0 != 0.0) ? 6 : 0;
    hm.mlump.assign(nfh, 0.0);
    hm.cf.assign((size_t)hm.ncf * nfh, 0);
    hm.wf.assign((size_t)hm.ncf * nfh, 0.0);
    // sign of the normal of face (side s of column c) along the cell's axis
    auto tau = [&](int c, int s) {
        const int f = G.face_of[s * ncol + c];
        return outward[s] * (G.faceL[f] == c ? 1.0 : -1.0);
    };
    for (int f = 0; f < nfh; ++f) {
        const int cells[2] = {G.faceL[f], G.faceR[f]};
        const int sides[2] = {G.faceSide[f], G.nbr_side[G.faceSide[f] * ncol + G.faceL[f]]};
        double lump = 0.0;
        for (int e = 0; e < 2; ++e) {
            const int c = cells[e], a = sides[e];
            const bool xi = a < 2;
            const double Fc = f0 * G.sinlat[c], ta = tau(c, a);
            // element row sum: 1/3 + 1/6 (or the lumped 1/2) and -+ 2 F_c / 4
            lump += 0.5 + (xi ? -0.5 : 0.5) * Fc;
            if (hm.ncf == 0) continue;
            const int b = a ^ 1;   // opposite side
            hm.cf[(size_t)e * nfh + f] = G.face_of[b * ncol + c];
            hm.wf[(size_t)e * nfh + f] = consistent ? ta * tau(c, b) / 6.0 : 0.0;
            const int p0 = xi ? 2 : 0;   // perpendicular sides
            for (int t = 0; t < 2; ++t) {
                const int bp = p0 + t;
                const size_t slot = (size_t)(2 + 2 * e + t) * nfh + f;
                hm.cf[slot] = G.face_of[bp * ncol + c];
                hm.wf[slot] = ta * tau(c, bp) * Fc * (xi ? -0.25 : 0.25);
            }
        }
        hm.mlump[f] = lump;
    }
}

mg_status setup_impl(mg_handle* h, const mg_mesh* mesh, const mg_params* prm, const double* g,
                     const mg_mixed* mixed, double gamma2 = 0.0) {
    const int L = prm->levels, n = mesh->n, nlev = mesh->nlev;
    h->L = L;
    h->n = n;
    h->nlev = nlev;
    h->prm = *prm;
    // (a factor near the ends of FP64's range stays outside: a pressure solver with another omega divides it out)
    if (std::fabs(prm->omega) >= 0x1p-100 && std::fabs(prm->omega) <= 0x1p100) h->om0 = prm->omega;
    CK(cudaGetDevice(&h->device));
    CK(cudaDeviceGetAttribute(&h->nsm, cudaDevAttrMultiProcessorCount, h->device));
    h->red_grid = 8 * h->nsm;
    // host hierarchy
    std::vector<mg::HGeom> hg(L);
    for (int l = 0; l < L; ++l) {
        const std::string err = mg::build_hgeom(n >> l, mesh->radius, hg[l]);
        if (!err.empty()) return MG_ERR_ARG;
    }
    mg::VGeom vg;
    if (!mg::build_vgeom(mesh->z_interfaces, nlev, vg).empty()) return MG_ERR_ARG;
    const int ncol0 = hg[0].ncol;
    const size_t N0 = (size_t)nlev * ncol0, NV0 = (size_t)(nlev + 1) * ncol0;
    std::vector<mg::LevelCoef> co(L);
    co[0].g.assign(g, g + N0);
    for (size_t i = 0; i < N0; ++i)
        if (!(g[i] > 0.0) || !std::isfinite(g[i])) return MG_ERR_ARG;
    co[0].mu.assign(NV0, 1.0);
    std::vector<double> w_up, w_dn;
    HMass hm;
    double mv = 1.0;
    if (mixed) {
        // vertical faces: consistent mass 2/3 on the face and 1/6 to the interior faces
        // above and below, plus eps B_w; lumped to the row sums
        const double off = mixed->consistent ? 1.0 / 6.0 : 0.0;
        mv = mixed->consistent ? 2.0 / 3.0 : 1.0;
        w_up.assign(NV0, 0.0);
        w_dn.assign(NV0, 0.0);
        for (int kf = 1; kf < nlev; ++kf) {
            for (int c = 0; c < ncol0; ++c) {
                const size_t o = (size_t)kf * ncol0 + c;
                if (kf + 1 <= nlev - 1) w_up[o] = mixed->eps * mixed->beta_up[o] + off;
                if (kf - 1 >= 1) w_dn[o] = mixed->eps * mixed->beta_dn[o] + off;
                co[0].mu[o] = 1.0 / (mv + w_up[o] + w_dn[o]);   // 1 / row sum
            }
        }
        horizontal_mass(hg[0], mixed->consistent != 0, mixed->coriolis_f0, hm);
        co[0].muh.resize(hm.mlump.size());
        for (size_t f = 0; f < hm.mlump.size(); ++f) co[0].muh[f] = 1.0 / hm.mlump[f];
    }
    for (int l = 1; l < L; ++l) {
        co[l].g.resize((size_t)nlev * hg[l].ncol);
        co[l].mu.resize((size_t)(nlev + 1) * hg[l].ncol);
        mg::restrict_mean(hg[l - 1], hg[l], nlev, co[l - 1].g.data(), co[l].g.data());
        mg::restrict_mean(hg[l - 1], hg[l], nlev + 1, co[l - 1].mu.data(), co[l].mu.data());
        if (!co[l - 1].muh.empty()) {
            co[l].muh.resize(2 * (size_t)hg[l].ncol);
            mg::restrict_face_mean(hg[l - 1], hg[l], co[l - 1].muh.data(), co[l].muh.data());
        }
    }
    for (int l = 0; l < L; ++l) mg::level_coefficients(hg[l], vg, mesh->cs_dt, co[l]);
    // upload
    std::vector<double> rdz(nlev);
    for (int k = 0; k < nlev; ++k) rdz[k] = 1.0 / vg.dz[k];
    TRY(upload(h, &h->rdz64, rdz));
    TRY(upload(h, &h->dz, vg.dz));
    TRY(upload(h, &h->area0, hg[0].area));
    TRY(upload(h, &h->rdz32, rdz));
    // V = area x depth x scale is at most about 1 on the finest level (a power of two: exact)
    h->scale = std::exp2(-std::ceil(std::log2(*std::max_element(hg[0].area.begin(), hg[0].area.end()) *
                                              *std::max_element(vg.dz.begin(), vg.dz.end()))));
    TRY(upload(h, &h->faceL0, hg[0].faceL));
    TRY(upload(h, &h->faceR0, hg[0].faceR));
    TRY(upload(h, &h->faceSide0, hg[0].faceSide));
    TRY(upload(h, &h->nbrSide0, hg[0].nbr_side));
    TRY(dalloc(h, &h->flag, 1));
    TRY(dalloc(h, &h->timeout, 1));
    CK(cudaMemset(h->flag, 0, sizeof(unsigned int)));
    CK(cudaMemset(h->timeout, 0, sizeof(unsigned int)));
    // MG_FP32_P64 stores and computes as MG_FP32; only the finest level's elimination differs
    const int prec = prm->vcycle_precision == MG_FP32_P64 ? MG_FP32 : prm->vcycle_precision;
    h->lv.resize(L);
    for (int l = 0; l < L; ++l) {
        DevLevel& d = h->lv[l];
        const mg::HGeom& G = hg[l];
        d.n = G.n;
        d.ncol = G.ncol;
        std::vector<double> rA(G.ncol), columns(2 * (size_t)G.ncol);   // 1 / area; that and area x scale
        for (int c = 0; c < G.ncol; ++c) {
            columns[c] = rA[c] = 1.0 / G.area[c];
            columns[G.ncol + c] = G.area[c] * h->scale;
        }
        std::vector<int32_t> sides(G.nbr);   // neighbours, then faces
        sides.insert(sides.end(), G.face_of.begin(), G.face_of.end());
        TRY(upload(h, &d.nbr, sides));
        d.fof = d.nbr + G.nbr.size();
        TRY(upload(h, &d.rA64, columns));
        d.wA64 = d.rA64 + G.ncol;
        TRY(upload(h, &d.Th64, co[l].Th));
        TRY(upload(h, &d.Tv64, co[l].Tv));
        const size_t Nl = (size_t)nlev * G.ncol;
        const size_t Np = gamma2 > 0.0 ? Nl : (size_t)nlev * mg::padded(G.n);   // an FP32 field
        Pieces own;   // (arrays that set-up does not upload: small handles' set-up is mostly allocations)
        if (prec != MG_FP64) TRY(upload(h, &d.rA32, rA));
        if (gamma2 > 0.0) {
            if (prec != MG_FP64) {
                TRY(upload(h, &d.Th32, co[l].Th));
                TRY(upload(h, &d.Tv32, co[l].Tv));
            }
        } else {
            d.wants64 = prec == MG_FP64;
            if (d.wants64 || Nl <= (size_t)MG_NOALLOC_MAX_CELLS) TRY(alloc64(h, l));
            if (prec == MG_FP32) {
                for (float** p : {&d.te32, &d.tn32}) own.add(p, Np);
                own.add(&d.tv32, Np + mg::padded(G.n));
            } else if (prec == MG_FP32_BF16COEF) {
                for (bf16** p : {&d.te16, &d.tn16}) own.add(p, Np);
                own.add(&d.tv16, Np + mg::padded(G.n));
            }
            if (prec != MG_FP64) {
                own.add(&d.ip32, Np);
                if (l == 0 && prm->vcycle_precision == MG_FP32_P64)
                    for (double** p : {&d.ipd, &d.md, &d.ed}) own.add(p, Np);
                own.add(&d.hd, 4 * (size_t)G.ncol);
            }
            if (l + 1 < L && prec == MG_FP64) own.add(&d.par, 5 * (size_t)G.ncol);
        }
        // (mg_smooth's scratch array; the second iterate of an FP64 V-cycle)
        for (int i = 0; i < (prec == MG_FP64 ? 2 : 1); ++i) own.add(&d.x64[i], Nl);
        // right-hand sides and, below the finest level, the iterate that goes up
        if (prec == MG_FP64) {
            own.add(&d.b64, Nl);
            if (l > 0) own.add(&d.r64, Nl);
        } else {
            for (float*& p : d.x32) own.add(&p, Np);
            own.add(&d.b32, Np);
            if (l > 0) own.add(&d.r32, Np);
        }
        if (gamma2 > 0.0) {
            // 9-cell stencil: flux between cells k and k + 2 of every column,
            // gamma2 (c_s dt)^2 (g_k + g_k+2) / 2 / (z_c[k+2] - z_c[k])
            h->nine = true;
            std::vector<double> t2(Nl, 0.0);
            const double c2 = mesh->cs_dt * mesh->cs_dt;
            const double* z = mesh->z_interfaces;
            for (int k = 0; k + 2 < nlev; ++k) {
                const double dzc2 = 0.5 * (z[k + 3] + z[k + 2]) - 0.5 * (z[k + 1] + z[k]);
                for (int c = 0; c < G.ncol; ++c)
                    t2[(size_t)k * G.ncol + c] =
                        gamma2 * c2 * 0.5 * (co[l].g[(size_t)k * G.ncol + c] + co[l].g[(size_t)(k + 2) * G.ncol + c]) /
                        dzc2;
            }
            TRY(upload(h, &d.T2_64, t2));
            for (double*& p : d.s64) own.add(&p, Nl);
            if (prec == MG_FP32) {
                TRY(upload(h, &d.T2_32, t2));
                for (float*& p : d.s32) own.add(&p, Nl);
            }
        }
        TRY(own.alloc(h));
        if (l + 1 < L) {
            const mg::HGeom& Gc = hg[l + 1];
            std::vector<double> w(4 * (size_t)Gc.ncol);
            for (int C = 0; C < Gc.ncol; ++C)
                for (int q = 0; q < 4; ++q) w[(size_t)q * Gc.ncol + C] = G.area[mg::child_col(G.n, C, q)] / Gc.area[C];
            if (gamma2 > 0.0) TRY(upload(h, &d.w64, w));
            if (prec != MG_FP64) TRY(upload(h, &d.w32, w));
        }
    }
    for (int l = 0; l < L; ++l) TRY(build_maps(h, l));
    {
        // finest level: a_side = Th[k][face] / area, a_up = Tv[k+1] / dz, a_dn = Tv[k] / dz,
        // and the diagonal 1 + sum of the six
        const mg::HGeom& G = hg[0];
        const size_t N = (size_t)nlev * ncol0;
        std::vector<double> a6(7 * N);
        for (int k = 0; k < nlev; ++k)
            for (int c = 0; c < ncol0; ++c) {
                const size_t e = (size_t)k * ncol0 + c;
                const double rA = 1.0 / G.area[c];
                for (int sd = 0; sd < 4; ++sd)
                    a6[sd * N + e] = co[0].Th[(size_t)k * 2 * ncol0 + G.face_of[sd * ncol0 + c]] * rA;
                a6[4 * N + e] = co[0].Tv[(size_t)(k + 1) * ncol0 + c] * rdz[k];
                a6[5 * N + e] = co[0].Tv[(size_t)k * ncol0 + c] * rdz[k];
                double d = 1.0;
                for (int f = 0; f < 6; ++f) d += a6[f * N + e];
                a6[6 * N + e] = d;
            }
        TRY(upload(h, &h->a6, a6));
    }
    // mixed system arrays (finest level)
    h->mixed = mixed != nullptr;
    if (h->mixed) {
        const mg::HGeom& G = hg[0];
        const int nfh = 2 * ncol0;
        // gradient and divergence each carry one factor c_s dt; their product is the
        // Helmholtz coupling (c_s dt)^2 g_f A_f / (V_i d_f)
        const double c = mesh->cs_dt;
        std::vector<double> kd_h((size_t)nlev * nfh), kd_v(NV0, 0.0), sdiv(4 * (size_t)ncol0), divv(nlev);
        for (int k = 0; k < nlev; ++k) divv[k] = c / vg.dz[k];
        for (int f = 0; f < nfh; ++f) {
            const int Lc = G.faceL[f], Rc = G.faceR[f], sd = G.faceSide[f];
            const double dist = G.cdist[sd * ncol0 + Lc];
            for (int k = 0; k < nlev; ++k)
                kd_h[(size_t)k * nfh + f] = c * 0.5 * (g[(size_t)k * ncol0 + Lc] + g[(size_t)k * ncol0 + Rc]) / dist;
        }
        for (int kf = 1; kf < nlev; ++kf)
            for (int col = 0; col < ncol0; ++col)
                kd_v[(size_t)kf * ncol0 + col] =
                    c * 0.5 * (g[(size_t)(kf - 1) * ncol0 + col] + g[(size_t)kf * ncol0 + col]) / vg.dzc[kf];
        for (int col = 0; col < ncol0; ++col)
            for (int sd = 0; sd < 4; ++sd) {
                const int f = G.face_of[sd * ncol0 + col];
                const double sgn = (G.faceL[f] == col) ? 1.0 : -1.0;
                sdiv[(size_t)sd * ncol0 + col] = sgn * c * G.edge_len[sd * ncol0 + col] / G.area[col];
            }
        // adjoint: face weights W_f = A_f d_f / g_f and the rows of M_h^T.  The surface and lid
        // faces are decoupled identity rows, so any weight keeps A^T = S J A-hat J S^-1; they
        // take area dz / g of their cell, the size of the interior weights (a weight far from
        // those would let their entries dominate the residual norm of the scaled system)
        std::vector<double> Wf((size_t)nlev * nfh + NV0, 1.0);
        for (int col = 0; col < ncol0; ++col) {
            Wf[(size_t)nlev * nfh + col] = G.area[col] * vg.dz[0] / g[col];
            Wf[(size_t)nlev * nfh + (size_t)nlev * ncol0 + col] =
                G.area[col] * vg.dz[nlev - 1] / g[(size_t)(nlev - 1) * ncol0 + col];
        }
        for (int f = 0; f < nfh; ++f) {
            const int Lc = G.faceL[f], Rc = G.faceR[f], sd = G.faceSide[f];
            const double el = G.edge_len[sd * ncol0 + Lc], dist = G.cdist[sd * ncol0 + Lc];
            for (int k = 0; k < nlev; ++k)
                Wf[(size_t)k * nfh + f] =
                    el * vg.dz[k] * dist / (0.5 * (g[(size_t)k * ncol0 + Lc] + g[(size_t)k * ncol0 + Rc]));
        }
        for (int kf = 1; kf < nlev; ++kf)
            for (int col = 0; col < ncol0; ++col)
                Wf[(size_t)nlev * nfh + (size_t)kf * ncol0 + col] =
                    G.area[col] * vg.dzc[kf] /
                    (0.5 * (g[(size_t)(kf - 1) * ncol0 + col] + g[(size_t)kf * ncol0 + col]));
        std::vector<double> wfT(hm.wf.size(), 0.0);
        for (int f = 0; f < nfh; ++f)
            for (int t = 0; t < hm.ncf; ++t) {
                const int gf = hm.cf[(size_t)t * nfh + f];
                int found = -1;
                for (int u = 0; u < hm.ncf; ++u)
                    if (hm.cf[(size_t)u * nfh + gf] == f) found = u;
                if (found < 0) return MG_ERR_ARG;   // the coupling pattern is symmetric by construction
                wfT[(size_t)t * nfh + f] = hm.wf[(size_t)found * nfh + gf];
            }
        std::vector<double> cdh(nfh), cdv(nlev + 1, 0.0);
        for (int f = 0; f < nfh; ++f) cdh[f] = c / (2.0 * G.cdist[G.faceSide[f] * ncol0 + G.faceL[f]]);
        for (int kf = 1; kf < nlev; ++kf) cdv[kf] = c / (2.0 * vg.dzc[kf]);
        int32_t *fL, *fR, *dcf = nullptr;
        double *dkd_h, *dkd_v, *dsdiv, *dwu, *dwd, *dml, *ddivv, *dwf = nullptr, *dmlh, *dwfT = nullptr, *dWf, *dcdh,
            *dcdv, *drW;
        TRY(upload(h, &fL, G.faceL));
        TRY(upload(h, &fR, G.faceR));
        TRY(upload(h, &dkd_h, kd_h));
        TRY(upload(h, &dkd_v, kd_v));
        TRY(upload(h, &dsdiv, sdiv));
        TRY(upload(h, &dwu, w_up));
        TRY(upload(h, &dwd, w_dn));
        TRY(upload(h, &dml, co[0].mu));     // 1 / lumped mass (1 on the boundary faces)
        TRY(upload(h, &ddivv, divv));
        TRY(upload(h, &dmlh, co[0].muh));
        if (hm.ncf > 0) {
            TRY(upload(h, &dcf, hm.cf));
            TRY(upload(h, &dwf, hm.wf));
            TRY(upload(h, &dwfT, wfT));
        }
        TRY(upload(h, &dWf, Wf));
        TRY(upload(h, &dcdh, cdh));
        TRY(upload(h, &dcdv, cdv));
        TRY(dalloc(h, &drW, Wf.size()));
        k_reciprocal<<<4 * h->nsm, 256>>>(Wf.size(), dWf, drW);
        CK(cudaGetLastError());
        h->md = mg::MixedDev{ncol0, nlev, nfh, fL, fR, h->lv[0].fof, dsdiv, dkd_h, dkd_v, dwu, dwd, dml, ddivv,
                             hm.ncf, dcf, dwf, hm.ms, mv, dmlh, dwfT, dWf, dcdh, dcdv, drW, mixed->eps};
        h->nu = (int64_t)nlev * nfh + (int64_t)NV0;
        TRY(dalloc(h, &h->schurB, N0));
        TRY(dalloc(h, &h->mb, (size_t)h->nu + N0));
        TRY(dalloc(h, &h->mx, (size_t)h->nu + N0));
    }
    // the levels' packed fields and factors: after the uploads, which would wait for them
    for (int l = 0; l < L && gamma2 <= 0.0; ++l) {
        DevLevel& d = h->lv[l];
        if (d.hd) k_rims<<<dim3((d.ncol + 127) / 128, 4), 128>>>(d.n, d.ncol, d.nbr, d.hd);
        if (d.par) k_parents<<<dim3((d.ncol + 127) / 128, 5), 128>>>(d.n, d.ncol, d.nbr, d.par);
        TRY(pack_level(h, l, nullptr));
    }
    // GCR workspace; the slot stride is padded off a multiple of large powers of two so
    // the directions streamed side by side do not share their low address bits
    h->glen = (N0 + (size_t)h->nu + 63) / 64 * 64 + 96;
    TRY(dalloc(h, &h->Z, (size_t)prm->gcr_restart * h->glen));
    TRY(dalloc(h, &h->W, (size_t)prm->gcr_restart * h->glen));
    TRY(dalloc(h, &h->r, h->glen));
    TRY(dalloc(h, &h->adj, N0));
    TRY(dalloc(h, &h->gs, 1));
    {
        // (every reduction's grid is at most red_grid blocks)
        h->npartials = (size_t)h->red_grid * (2 * mg::MAXR + 2);
        TRY(dalloc(h, &h->partials, h->npartials));
    }
    TRY(dalloc(h, &h->tickets, TK_COUNT));
    CK(cudaMemset(h->tickets, 0, TK_COUNT * sizeof(unsigned int)));
    CK(cudaMemset(h->gs, 0, sizeof(mg::GcrScal)));
    if (!mem_alloc((void**)&h->host_sc, 4 * sizeof(double), MEM_PINNED)) return MG_ERR_NOMEM;
    if (!mem_alloc((void**)&h->host_bs, sizeof(mg::BicgScal), MEM_PINNED)) return MG_ERR_NOMEM;
    TRY(dalloc(h, &h->bs, 1));
    CK(cudaStreamCreateWithFlags(&h->cap, cudaStreamNonBlocking));
    CK(cudaStreamCreateWithFlags(&h->run, cudaStreamNonBlocking));
    CK(cudaEventCreateWithFlags(&h->evx, cudaEventDisableTiming));
    CK(cudaEventCreate(&h->ev0));
    CK(cudaEventCreate(&h->ev1));
    CK(cudaDeviceSynchronize());
    return MG_OK;
}

void free_handle(mg_handle* h) {
    if (!h) return;
    for (void* p : h->allocs) mem_free(p, MEM_DEVICE);
    mem_free(h->host_sc, MEM_PINNED);
    mem_free(h->host_bs, MEM_PINNED);
    for (auto& row : h->gexec)
        for (cudaGraphExec_t g : row)
            if (g) cudaGraphExecDestroy(g);
    if (h->cap) cudaStreamDestroy(h->cap);
    if (h->run) cudaStreamDestroy(h->run);
    if (h->evx) cudaEventDestroy(h->evx);
    if (h->ev0) cudaEventDestroy(h->ev0);
    if (h->ev1) cudaEventDestroy(h->ev1);
    for (cudaEvent_t e : h->evpool) cudaEventDestroy(e);
    delete h;
}

}  // namespace

// ---- an ensemble of pressure solves as one CUDA graph ----
struct mg_ensemble {
    int device = 0;
    int count = 0;
    std::vector<mg_handle*> hs;
    cudaStream_t cs = nullptr;            // capture stream
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    mg::EnsState* st = nullptr;           // device, one per member
    mg::EnsState* host_st = nullptr;      // pinned copy, written by the graph's last node
    unsigned long long* stamps = nullptr; // device: launch time, then every member's end [ns]
    unsigned long long* host_stamps = nullptr;
};

namespace {

void free_ensemble(mg_ensemble* e) {
    if (!e) return;
    if (e->exec) cudaGraphExecDestroy(e->exec);
    if (e->graph) cudaGraphDestroy(e->graph);
    mem_free(e->st, MEM_DEVICE);
    mem_free(e->host_st, MEM_PINNED);
    mem_free(e->stamps, MEM_DEVICE);
    mem_free(e->host_stamps, MEM_PINNED);
    if (e->cs) cudaStreamDestroy(e->cs);
    delete e;
}

// Ends the capture on e->cs and returns the nodes the next work depends on.
mg_status end_segment(mg_ensemble* e, std::vector<cudaGraphNode_t>& deps) {
    cudaStreamCaptureStatus cst;
    const cudaGraphNode_t* d = nullptr;
    size_t nd = 0;
    CK(cudaStreamGetCaptureInfo(e->cs, &cst, nullptr, nullptr, &d, nullptr, &nd));
    deps.assign(d, d + nd);
    cudaGraph_t g = nullptr;
    CK(cudaStreamEndCapture(e->cs, &g));
    return MG_OK;
}

mg_status add_conditional(cudaGraph_t g, const std::vector<cudaGraphNode_t>& deps, cudaGraphConditionalHandle hnd,
                          cudaGraphConditionalNodeType type, cudaGraphNode_t* node, cudaGraph_t* body) {
    cudaGraphNodeParams p{};
    p.type = cudaGraphNodeTypeConditional;
    p.conditional.handle = hnd;
    p.conditional.type = type;
    p.conditional.size = 1;
    CK(cudaGraphAddNode(node, g, deps.empty() ? nullptr : deps.data(), nullptr, deps.size(), &p));
    *body = p.conditional.phGraph_out[0];
    return MG_OK;
}

// The launches of one member: start, then WHILE { IF slot 0 {iteration}, IF {update}, ..., IF slot R-1
// {iteration}, IF {update} }, then the member's end event.
mg_status build_member(mg_ensemble* e, int i, mg_handle* h, const double* b, double* x, double tol,
                       const std::vector<cudaGraphNode_t>& root, std::vector<cudaGraphNode_t>& ends) {
    const int R = h->prm.gcr_restart;
    const size_t n = cells(h, 0);
    const cudaStreamCaptureMode mode = cudaStreamCaptureModeThreadLocal;
    mg::EnsHandles hs{};
    CK(cudaGraphConditionalHandleCreate(&hs.w, e->graph, 0, cudaGraphCondAssignDefault));
    for (int j = 0; j < R; ++j) {
        CK(cudaGraphConditionalHandleCreate(&hs.c[j], e->graph, 0, cudaGraphCondAssignDefault));
        CK(cudaGraphConditionalHandleCreate(&hs.x[j], e->graph, 0, cudaGraphCondAssignDefault));
    }
    mg::EnsState* st = e->st + i;
    // start: r = b, x = 0, <b, b>, first decision
    std::vector<cudaGraphNode_t> deps;
    CK(cudaStreamBeginCaptureToGraph(e->cs, e->graph, root.data(), nullptr, root.size(), mode));
    mg::k_gcr_start<<<vec_grid(h, n), mg::RED_THREADS, 0, e->cs>>>(n, b, h->r, x, h->partials, h->tickets + TK_DOT,
                                                                   &h->gs->bb, nullptr, h->timeout);
    mg::k_ens_init<<<1, 1, 0, e->cs>>>(h->gs, st, R, h->prm.max_iter, hs);
    CK(cudaGetLastError());
    TRY(end_segment(e, deps));
    cudaGraphNode_t wnode;
    cudaGraph_t wbody;
    TRY(add_conditional(e->graph, deps, hs.w, cudaGraphCondTypeWhile, &wnode, &wbody));
    std::vector<cudaGraphNode_t> prev;
    for (int j = 0; j < R; ++j) {
        cudaGraphNode_t inode, xnode;
        cudaGraph_t ibody, xbody;
        TRY(add_conditional(wbody, prev, hs.c[j], cudaGraphCondTypeIf, &inode, &ibody));
        CK(cudaStreamBeginCaptureToGraph(e->cs, ibody, nullptr, nullptr, 0, mode));
        double* z = h->Z + (size_t)j * h->glen;
        double* w = h->W + (size_t)j * h->glen;
        TRY(run_vcycle(h, h->r, z, e->cs));
        TRY(apply_gcr(h, z, w, j, e->cs));
        TRY(dispatch_j<RunOrth>(j, h, n, e->cs));
        mg::k_ens_decide<<<1, 1, 0, e->cs>>>(h->gs, st, j, R, h->prm.max_iter, tol, hs, h->timeout);
        CK(cudaGetLastError());
        TRY(end_segment(e, deps));
        TRY(add_conditional(wbody, {inode}, hs.x[j], cudaGraphCondTypeIf, &xnode, &xbody));
        CK(cudaStreamBeginCaptureToGraph(e->cs, xbody, nullptr, nullptr, 0, mode));
        TRY(dispatch_j<RunXupd>(j, h, n, x, e->cs));
        TRY(end_segment(e, deps));
        prev.assign(1, xnode);
    }
    // the member's end
    CK(cudaStreamBeginCaptureToGraph(e->cs, e->graph, &wnode, nullptr, 1, mode));
    mg::k_stamp<<<1, 1, 0, e->cs>>>(e->stamps + 1 + i);
    CK(cudaGetLastError());
    TRY(end_segment(e, deps));
    ends.insert(ends.end(), deps.begin(), deps.end());
    return MG_OK;
}

mg_status build_ensemble(mg_ensemble* e, const double* const* b, double* const* x, double tol) {
    CK(cudaStreamCreateWithFlags(&e->cs, cudaStreamNonBlocking));
    if (!mem_alloc((void**)&e->st, e->count * sizeof(mg::EnsState), MEM_DEVICE) ||
        !mem_alloc((void**)&e->host_st, e->count * sizeof(mg::EnsState), MEM_PINNED) ||
        !mem_alloc((void**)&e->stamps, (e->count + 1) * sizeof(unsigned long long), MEM_DEVICE) ||
        !mem_alloc((void**)&e->host_stamps, (e->count + 1) * sizeof(unsigned long long), MEM_PINNED))
        return MG_ERR_NOMEM;
    CK(cudaGraphCreate(&e->graph, 0));
    // root: the launch time; every member starts after it
    std::vector<cudaGraphNode_t> root, deps;
    CK(cudaStreamBeginCaptureToGraph(e->cs, e->graph, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    mg::k_stamp<<<1, 1, 0, e->cs>>>(e->stamps);
    CK(cudaGetLastError());
    TRY(end_segment(e, root));
    std::vector<cudaGraphNode_t> ends;
    for (int i = 0; i < e->count; ++i) TRY(build_member(e, i, e->hs[i], b[i], x[i], tol, root, ends));
    // last nodes: every member's state and time stamp to the host
    CK(cudaStreamBeginCaptureToGraph(e->cs, e->graph, ends.data(), nullptr, ends.size(), cudaStreamCaptureModeThreadLocal));
    CK(cudaMemcpyAsync(e->host_st, e->st, e->count * sizeof(mg::EnsState), cudaMemcpyDeviceToHost, e->cs));
    CK(cudaMemcpyAsync(e->host_stamps, e->stamps, (e->count + 1) * sizeof(unsigned long long),
                       cudaMemcpyDeviceToHost, e->cs));
    TRY(end_segment(e, deps));
    CK(cudaGraphInstantiate(&e->exec, e->graph, 0));
    return MG_OK;
}

}  // namespace

// =====================================================================================
static mg_status mg_setup_check(const mg_mesh* mesh, const mg_params* prm, const double* g, const mg_mixed* mixed);

extern "C" {

const char* mg_last_cuda_error(void) {
    return g_last_cuda == cudaSuccess ? "no CUDA error" : cudaGetErrorName(g_last_cuda);
}

int64_t mg_inject_alloc_failure(int64_t nth) {
    const long long seen = g_alloc_seen.exchange(0);
    g_fail_at.store(nth > 0 ? nth : 0);
    return seen;
}

int64_t mg_live_allocations(void) { return g_live.load(); }

mg_status mg_inject_wait_limit(mg_handle* h, int32_t polls) {
    if (!h) return MG_ERR_ARG;
    DeviceGuard dg(h->device);
    CK(cudaDeviceSynchronize());
    h->polls = polls < 0 ? mg::WAIT_POLLS : polls;
    drop_graphs(h, 0);
    return MG_OK;
}

const char* mg_status_string(mg_status s) {
    switch (s) {
        case MG_OK: return "ok";
        case MG_ERR_ARG: return "invalid argument";
        case MG_ERR_CUDA: return "CUDA runtime error";
        case MG_ERR_NOMEM: return "out of memory";
        case MG_ERR_NOT_CONVERGED: return "not converged within max_iter";
        case MG_ERR_BREAKDOWN: return "Krylov breakdown (zero or non-finite scalar)";
        case MG_ERR_TIMEOUT: return "device wait timed out";
        case MG_ERR_UNSUPPORTED: return "unsupported request for this handle";
    }
    return "unknown status";
}

mg_status mg_setup(const mg_mesh* mesh, const mg_params* prm, const double* g, const mg_mixed* mixed,
                   mg_handle** out) {
    if (!out) return MG_ERR_ARG;
    *out = nullptr;
    TRY(mg_setup_check(mesh, prm, g, mixed));
    mg_handle* h = new (std::nothrow) mg_handle();
    if (!h) return MG_ERR_NOMEM;
    mg_status st = setup_impl(h, mesh, prm, g, mixed);
    if (st != MG_OK) {
        free_handle(h);
        return st;
    }
    *out = h;
    return MG_OK;
}

}  // extern "C"

static mg_status mg_setup_check(const mg_mesh* mesh, const mg_params* prm, const double* g, const mg_mixed* mixed) {
    if (!mesh || !prm || !g || !mesh->z_interfaces) return MG_ERR_ARG;
    if (mesh->n < 1 || mesh->nlev < 1 || mesh->nlev > MG_MAX_NLEV) return MG_ERR_ARG;
    if (!(mesh->radius > 0.0) || !(mesh->cs_dt > 0.0) || !std::isfinite(mesh->cs_dt)) return MG_ERR_ARG;
    if (prm->levels < 1 || prm->levels > MG_MAX_LEVELS) return MG_ERR_ARG;
    if (mesh->n % (1 << (prm->levels - 1)) != 0) return MG_ERR_ARG;
    if (!std::isfinite(prm->omega) || prm->n_pre < 0 || prm->n_post < 0 || prm->n_coarse < 1) return MG_ERR_ARG;
    if (prm->vcycle_precision < MG_FP64 || prm->vcycle_precision > MG_FP32_P64) return MG_ERR_ARG;
    if (prm->gcr_restart < 1 || prm->gcr_restart > MG_MAX_RESTART || prm->max_iter < 1) return MG_ERR_ARG;
    if (mixed && (!mixed->beta_up || !mixed->beta_dn || !std::isfinite(mixed->eps) || mixed->eps < 0.0 ||
                  (mixed->consistent != 0 && mixed->consistent != 1) || !std::isfinite(mixed->coriolis_f0) ||
                  std::fabs(mixed->coriolis_f0) >= 0.5))
        return MG_ERR_ARG;
    // the column kernels address a level with 32-bit offsets (horizontal faces: 2 kc)
    if (2.0 * (mesh->nlev + 1) * 6.0 * (double)mesh->n * mesh->n >= 4294967296.0) return MG_ERR_UNSUPPORTED;
    return MG_OK;
}

extern "C" {

mg_status mg_setup_9pt(const mg_mesh* mesh, const mg_params* prm, const double* g, double gamma2, mg_handle** out) {
    if (!out) return MG_ERR_ARG;
    *out = nullptr;
    if (!(gamma2 > 0.0) || !std::isfinite(gamma2) || !prm) return MG_ERR_ARG;
    if (prm->vcycle_precision == MG_FP32_BF16COEF || prm->vcycle_precision == MG_FP32_P64)
        return MG_ERR_UNSUPPORTED;
    if (!mesh || !g || !mesh->z_interfaces) return MG_ERR_ARG;
    mg_handle* h = nullptr;
    // validate exactly as mg_setup does, then build with the next-to-nearest fluxes
    TRY(mg_setup_check(mesh, prm, g, nullptr));
    h = new (std::nothrow) mg_handle();
    if (!h) return MG_ERR_NOMEM;
    const mg_status st = setup_impl(h, mesh, prm, g, nullptr, gamma2);
    if (st != MG_OK) {
        free_handle(h);
        return st;
    }
    *out = h;
    return MG_OK;
}

mg_status mg_setup_coeffs(const mg_mesh* mesh, const mg_params* prm, const double* coeffs, const double* cell_factors,
                          mg_handle** out) {
    if (!out) return MG_ERR_ARG;
    *out = nullptr;
    if (!coeffs) return MG_ERR_ARG;
    mg_handle* h = nullptr;
    TRY(mg_setup(mesh, prm, cell_factors, nullptr, &h));
    const size_t n6 = 6 * cells(h, 0);
    double* tmp = nullptr;
    mg_status st = MG_OK;
    if (!mem_alloc((void**)&tmp, n6 * sizeof(double), MEM_DEVICE)) {
        st = MG_ERR_NOMEM;
    } else if (cudaMemcpy(tmp, coeffs, n6 * sizeof(double), cudaMemcpyHostToDevice) != cudaSuccess) {
        st = MG_ERR_CUDA;
    } else {
        st = set_coefficients_impl(h, tmp, nullptr);
        if (st == MG_OK && cudaDeviceSynchronize() != cudaSuccess) st = MG_ERR_CUDA;
    }
    mem_free(tmp, MEM_DEVICE);
    if (st != MG_OK) {
        mg_destroy(h);
        return st;
    }
    *out = h;
    return MG_OK;
}

mg_status mg_set_pressure_solver(mg_handle* h, const mg_pressure_solver* ps) {
    if (!h || !ps) return MG_ERR_ARG;
    if (ps->kind < MG_PS_MG || ps->kind > MG_PS_BICGSTAB_MG) return MG_ERR_ARG;
    const bool jac = ps->kind == MG_PS_JACOBI || ps->kind == MG_PS_BICGSTAB_JACOBI;
    const bool bicg = ps->kind == MG_PS_BICGSTAB_JACOBI || ps->kind == MG_PS_BICGSTAB_MG;
    if (jac && (ps->sweeps < 1 || !std::isfinite(ps->omega))) return MG_ERR_ARG;
    if (bicg && (!(ps->eps >= 0.0) || ps->max_iter < 1)) return MG_ERR_ARG;
    DeviceGuard dg(h->device);
    if (bicg && !h->bv[0]) {
        const size_t n = cells(h, 0);
        for (double*& v : h->bv) TRY(dalloc(h, &v, n));
    }
    CK(cudaDeviceSynchronize());
    h->ps = *ps;
    drop_graphs(h, 1);   // (those of the mixed solves hold the previous pressure solver)
    return MG_OK;
}

mg_status helmholtz_solve(mg_handle* h, const double* b, double* x, double* iterations, void* stream) {
    NvtxRange nvtx_("helmholtz_solve");
    if (!h || !b || !x || b == x) return MG_ERR_ARG;
    DeviceGuard dg(h->device);
    double it = 0.0;
    const mg_status st = run_pressure_solver(h, b, x, S(stream), &it);
    if (iterations) *iterations = it;
    return st;
}

mg_status mg_inner_stats(mg_handle* h, int64_t* solves, double* iterations) {
    if (!h) return MG_ERR_ARG;
    if (solves) *solves = h->ps_solves;
    if (iterations) *iterations = h->ps_iters;
    h->ps_solves = 0;
    h->ps_iters = 0.0;
    return MG_OK;
}

mg_status mg_set_coefficients(mg_handle* h, const double* coeffs, void* stream) {
    if (!h || !coeffs) return MG_ERR_ARG;
    if (h->mixed || h->nine) return MG_ERR_UNSUPPORTED;
    DeviceGuard dg(h->device);
    return set_coefficients_impl(h, coeffs, S(stream));
}

void mg_destroy(mg_handle* h) {
    if (!h) return;
    DeviceGuard dg(h->device);
    cudaDeviceSynchronize();
    free_handle(h);
}

mg_status mg_sizes(const mg_handle* h, int64_t* ncol, int64_t* ncell, int64_t* nu) {
    if (!h) return MG_ERR_ARG;
    if (ncol) *ncol = h->lv[0].ncol;
    if (ncell) *ncell = (int64_t)cells(h, 0);
    if (nu) *nu = h->nu;
    return MG_OK;
}

mg_status helmholtz_apply(mg_handle* h, const double* x, double* y, void* stream) {
    if (!h || !x || !y || x == y) return MG_ERR_ARG;
    DeviceGuard dg(h->device);
    if (h->nine) return launch_apply9(h, 0, x, y, S(stream));
    return launch_apply(h, 0, View<double, double>::lvl(h, 0), x, y, S(stream));
}

mg_status vcycle(mg_handle* h, const double* b, double* x, void* stream) {
    NvtxRange nvtx_("vcycle");
    if (!h || !b || !x || b == x) return MG_ERR_ARG;
    DeviceGuard dg(h->device);
    return run_vcycle(h, b, x, S(stream));
}

mg_status pressure_solve(mg_handle* h, const double* b, double* x, double tol, mg_solve_info* info,
                         void* stream) {
    NvtxRange nvtx_("pressure_solve");
    if (!h || !b || !x || b == x || !(tol >= 0.0)) return MG_ERR_ARG;
    DeviceGuard dg(h->device);
    cudaStream_t s = S(stream);
    auto A = [&](const double* z, double* w, int j, cudaStream_t q) { return apply_gcr(h, z, w, j, q); };
    auto P = [&](const double* r, double* z, cudaStream_t q) { return run_vcycle(h, r, z, q); };
    return gcr(h, 0, cells(h, 0), b, x, tol, info, s, A, P);
}

mg_status pressure_solve_adjoint(mg_handle* h, const double* g, double* lambda, double tol, mg_solve_info* info,
                                 void* stream) {
    NvtxRange nvtx_("pressure_solve_adjoint");
    if (!h || !g || !lambda || g == lambda || !(tol >= 0.0)) return MG_ERR_ARG;
    DeviceGuard dg(h->device);
    cudaStream_t s = S(stream);
    const int ncol = h->lv[0].ncol, nlev = h->nlev;
    const size_t n = cells(h, 0);
    const dim3 grid((ncol + 127) / 128, nlev);
    // H^T = V H V^-1 (V H is symmetric): lambda = V H^-1 (V^-1 g)
    {
        Prof pr(h, MG_K_DOT, 0, 16.0 * n, s);
        mg::k_scale_volume<<<grid, 128, 0, s>>>(ncol, nlev, h->area0, h->dz, g, h->adj, false);
        CK(cudaGetLastError());
    }
    auto A = [&](const double* z, double* w, int j, cudaStream_t q) { return apply_gcr(h, z, w, j, q); };
    auto P = [&](const double* r, double* z, cudaStream_t q) { return run_vcycle(h, r, z, q); };
    const mg_status st = gcr(h, 0, n, h->adj, lambda, tol, info, s, A, P);
    if (st == MG_OK || st == MG_ERR_NOT_CONVERGED) {
        Prof pr(h, MG_K_DOT, 0, 16.0 * n, s);
        mg::k_scale_volume<<<grid, 128, 0, s>>>(ncol, nlev, h->area0, h->dz, lambda, lambda, true);
        CK(cudaGetLastError());
        CK(cudaStreamSynchronize(s));
    }
    return st;
}

mg_status helmholtz_coefficient_gradient(mg_handle* h, const double* lambda, const double* x, double* grad,
                                         void* stream) {
    if (!h || !lambda || !x || !grad) return MG_ERR_ARG;
    if (h->nine) return MG_ERR_UNSUPPORTED;
    DeviceGuard dg(h->device);
    cudaStream_t s = S(stream);
    const Lvl<double, double> L = View<double, double>::lvl(h, 0);
    Prof pr(h, MG_K_DOT, 0, 64.0 * cells(h, 0), s);   // lambda, x (read), 6 gradients (written)
    mg::k_coef_grad<<<dim3((L.ncol + 127) / 128, L.nlev), 128, 0, s>>>(L, lambda, x, grad);
    CK(cudaGetLastError());
    return MG_OK;
}

mg_status ensemble_pressure_solve(mg_handle* const* handles, int32_t count, const double* const* b,
                                  double* const* x, double tol, mg_solve_info* infos, int32_t* statuses,
                                  void* stream) {
    NvtxRange nvtx_("ensemble_pressure_solve");
    if (count < 0 || (count > 0 && (!handles || !b || !x)) || !(tol >= 0.0)) return MG_ERR_ARG;
    if (count == 0) return MG_OK;
    for (int i = 0; i < count; ++i) {
        if (!handles[i] || !b[i] || !x[i] || b[i] == x[i] || handles[i]->device != handles[0]->device)
            return MG_ERR_ARG;
        for (int k = 0; k < i; ++k)
            if (handles[k] == handles[i]) return MG_ERR_ARG;   // a handle holds one solve's workspace
    }
    DeviceGuard dg(handles[0]->device);
    // every member starts after the work already queued on the caller's stream
    CK(cudaEventRecord(handles[0]->evx, S(stream)));
    std::vector<GcrRun> g(count);
    for (int i = 0; i < count; ++i) {
        mg_handle* h = handles[i];
        g[i].sys = 0;
        g[i].n = cells(h, 0);
        g[i].x = x[i];
        g[i].tol = tol;
        CK(cudaStreamWaitEvent(h->run, handles[0]->evx, 0));
        TRY(gcr_start(h, g[i], b[i], h->run));
    }
    for (int i = 0; i < count; ++i) {
        CK(cudaStreamSynchronize(handles[i]->run));
        gcr_started(handles[i], g[i]);
    }
    // rounds: every unfinished member launches one iteration on its stream (the members run
    // side by side on the GPU), then the host collects the residual norms
    for (bool any = true; any;) {
        any = false;
        for (int i = 0; i < count; ++i) {
            if (!g[i].active) continue;
            mg_handle* h = handles[i];
            auto A = [h](const double* z, double* w, int j, cudaStream_t q) { return apply_gcr(h, z, w, j, q); };
            auto P = [h](const double* r, double* z, cudaStream_t q) { return run_vcycle(h, r, z, q); };
            TRY(gcr_launch(h, g[i], h->run, A, P));
        }
        for (int i = 0; i < count; ++i) {
            if (!g[i].active) continue;
            CK(cudaStreamSynchronize(handles[i]->run));
            TRY(gcr_landed(handles[i], g[i], handles[i]->run));
            any = any || g[i].active;
        }
    }
    mg_status st = MG_OK;
    for (int i = 0; i < count; ++i) CK(cudaEventRecord(handles[i]->ev1, handles[i]->run));
    for (int i = 0; i < count; ++i) {
        CK(cudaEventSynchronize(handles[i]->ev1));
        gcr_info(handles[i], g[i], infos ? infos + i : nullptr);
        if (statuses) statuses[i] = g[i].st;
        if (st == MG_OK) st = g[i].st;
    }
    return st;
}

mg_status mg_ensemble_create(mg_handle* const* handles, int32_t count, const double* const* b, double* const* x,
                             double tol, mg_ensemble** out) {
    if (!out) return MG_ERR_ARG;
    *out = nullptr;
    if (count < 1 || !handles || !b || !x || !(tol >= 0.0)) return MG_ERR_ARG;
    for (int i = 0; i < count; ++i) {
        if (!handles[i] || !b[i] || !x[i] || b[i] == x[i] || handles[i]->device != handles[0]->device)
            return MG_ERR_ARG;
        for (int k = 0; k < i; ++k)
            if (handles[k] == handles[i]) return MG_ERR_ARG;
        if (handles[i]->prof || handles[i]->mixed) return MG_ERR_UNSUPPORTED;
    }
    DeviceGuard dg(handles[0]->device);
    mg_ensemble* e = new (std::nothrow) mg_ensemble();
    if (!e) return MG_ERR_NOMEM;
    e->device = handles[0]->device;
    e->count = count;
    e->hs.assign(handles, handles + count);
    const mg_status st = build_ensemble(e, b, x, tol);
    if (st != MG_OK) {
        cudaStreamCaptureStatus cst;
        if (e->cs && cudaStreamIsCapturing(e->cs, &cst) == cudaSuccess && cst != cudaStreamCaptureStatusNone) {
            cudaGraph_t g = nullptr;
            cudaStreamEndCapture(e->cs, &g);
        }
        cudaGetLastError();
        free_ensemble(e);
        return st;
    }
    *out = e;
    return MG_OK;
}

mg_status mg_ensemble_solve(mg_ensemble* e, mg_solve_info* infos, int32_t* statuses, void* stream) {
    NvtxRange nvtx_("mg_ensemble_solve");
    if (!e) return MG_ERR_ARG;
    DeviceGuard dg(e->device);
    cudaStream_t s = S(stream);
    CK(cudaGraphLaunch(e->exec, s));
    CK(cudaStreamSynchronize(s));
    mg_status st = MG_OK;
    for (int i = 0; i < e->count; ++i) {
        const mg::EnsState& m = e->host_st[i];
        if (infos) {
            infos[i].iters = m.it;
            infos[i].rel_res = m.rel;
            infos[i].ms = 1e-6 * (double)(e->host_stamps[1 + i] - e->host_stamps[0]);
        }
        if (statuses) statuses[i] = m.status;
        if (st == MG_OK) st = (mg_status)m.status;
    }
    return st;
}

void mg_ensemble_destroy(mg_ensemble* e) {
    if (!e) return;
    DeviceGuard dg(e->device);
    cudaDeviceSynchronize();
    free_ensemble(e);
}

mg_status mixed_solve(mg_handle* h, const double* rhs_u, const double* rhs_p, double* u, double* p, double tol,
                      mg_solve_info* info, void* stream) {
    NvtxRange nvtx_("mixed_solve");
    if (!h || !rhs_u || !rhs_p || !u || !p || !(tol >= 0.0)) return MG_ERR_ARG;
    if (!h->mixed) return MG_ERR_UNSUPPORTED;
    DeviceGuard dg(h->device);
    cudaStream_t s = S(stream);
    const size_t nu = (size_t)h->nu, np = cells(h, 0), n = nu + np;
    // GCR runs on concatenated [u; p] vectors held by the handle
    CK(cudaMemcpyAsync(h->mb, rhs_u, nu * sizeof(double), cudaMemcpyDeviceToDevice, s));
    CK(cudaMemcpyAsync(h->mb + nu, rhs_p, np * sizeof(double), cudaMemcpyDeviceToDevice, s));
    auto A = [&](const double* v, double* y, int j, cudaStream_t q) {
        return dispatch_j<RunMixed<mg::MX_A>::K>(j, h, v, y, nullptr, q);
    };
    auto P = [&](const double* r, double* z, cudaStream_t q) { return schur_impl(h, r, r + nu, z, z + nu, nullptr, q); };
    const mg_status st = gcr(h, 1, n, h->mb, h->mx, tol, info, s, A, P);
    if (st == MG_OK || st == MG_ERR_NOT_CONVERGED || st == MG_ERR_BREAKDOWN) {
        CK(cudaMemcpyAsync(u, h->mx, nu * sizeof(double), cudaMemcpyDeviceToDevice, s));
        CK(cudaMemcpyAsync(p, h->mx + nu, np * sizeof(double), cudaMemcpyDeviceToDevice, s));
    }
    return st;
}

mg_status mixed_solve_adjoint(mg_handle* h, const double* g_u, const double* g_p, double* lam_u, double* lam_p,
                              double tol, mg_solve_info* info, void* stream) {
    NvtxRange nvtx_("mixed_solve_adjoint");
    if (!h || !g_u || !g_p || !lam_u || !lam_p || !(tol >= 0.0)) return MG_ERR_ARG;
    if (!h->mixed) return MG_ERR_UNSUPPORTED;
    DeviceGuard dg(h->device);
    cudaStream_t s = S(stream);
    const size_t nu = (size_t)h->nu, np = cells(h, 0), n = nu + np;
    // A^T = S J A-hat J S^-1: lambda = S J A-hat^-1 (J S^-1 g), A-hat preconditioned by the
    // Schur-complement step of A itself (its transpose is S J P J S^-1 as well)
    TRY(mixed_adj_scale<false>(h, g_u, g_p, h->mb, h->mb + nu, s));
    auto A = [&](const double* v, double* y, int j, cudaStream_t q) {
        return dispatch_j<RunMixed<mg::MX_HAT>::K>(j, h, v, y, h->mb, q);
    };
    // (mb is free once the iteration has taken its right-hand side: W z_u of the direction under way)
    auto P = [&](const double* r, double* z, cudaStream_t q) { return schur_impl(h, r, r + nu, z, z + nu, h->mb, q); };
    const mg_status st = gcr(h, 2, n, h->mb, h->mx, tol, info, s, A, P);
    if (st == MG_OK || st == MG_ERR_NOT_CONVERGED || st == MG_ERR_BREAKDOWN) {
        TRY(mixed_adj_scale<true>(h, h->mx, h->mx + nu, lam_u, lam_p, s));
        CK(cudaStreamSynchronize(s));
    }
    return st;
}

mg_status mixed_coefficient_gradient(mg_handle* h, const double* lam_u, const double* u, const double* p,
                                     double* grad_g, double* grad_beta_up, double* grad_beta_dn, void* stream) {
    if (!h || !lam_u || !u || !p || !grad_g || !grad_beta_up || !grad_beta_dn) return MG_ERR_ARG;
    if (!h->mixed) return MG_ERR_UNSUPPORTED;
    DeviceGuard dg(h->device);
    cudaStream_t s = S(stream);
    const mg::MixedDev& M = h->md;
    const size_t nh = (size_t)M.nlev * M.nfh;
    const int bd = 128;
    Prof pr(h, MG_K_DOT, 0, 8.0 * (3.0 * h->nu + 2.0 * cells(h, 0)), s, 3);
    mg::k_mx_grad_g<<<dim3((M.ncol + bd - 1) / bd, M.nlev), bd, 0, s>>>(M, lam_u, p, grad_g);
    mg::k_mx_grad_beta<<<dim3((M.ncol + bd - 1) / bd, M.nlev + 1), bd, 0, s>>>(M, lam_u + nh, u + nh, grad_beta_up,
                                                                              grad_beta_dn);
    CK(cudaGetLastError());
    return MG_OK;
}

mg_status mixed_apply_transpose(mg_handle* h, const double* u, const double* p, double* yu, double* yp,
                                void* stream) {
    if (!h || !u || !p || !yu || !yp || u == yu || p == yp) return MG_ERR_ARG;
    if (!h->mixed) return MG_ERR_UNSUPPORTED;
    DeviceGuard dg(h->device);
    cudaStream_t s = S(stream);
    const size_t nu = (size_t)h->nu;
    TRY(mixed_adj_scale<false>(h, u, p, h->mb, h->mb + nu, s));
    {
        Prof pr(h, MG_K_MIXED, 0, 8.0 * (3.0 * h->nu + 3.0 * cells(h, 0)), s, 2);
        // (W times the scaled velocity is u itself)
        TRY((launch_mixed<mg::MX_HAT, -1>(h, h->mb, h->mb + nu, h->mx, h->mx + nu, const_cast<double*>(u), s)));
    }
    return mixed_adj_scale<true>(h, h->mx, h->mx + nu, yu, yp, s);
}

mg_status mg_level_apply(mg_handle* h, int32_t level, const double* x, double* y, void* stream) {
    TRY(check_level(h, level));
    if (!x || !y || x == y) return MG_ERR_ARG;
    DeviceGuard dg(h->device);
    if (h->nine) return launch_apply9(h, level, x, y, S(stream));
    return launch_apply(h, level, View<double, double>::lvl(h, level), x, y, S(stream));
}

mg_status mg_smooth(mg_handle* h, int32_t level, const double* b, const double* x_in, double* x_out,
                    int32_t sweeps, void* stream) {
    TRY(check_level(h, level));
    if (!b || !x_out || sweeps < 0 || b == x_out) return MG_ERR_ARG;
    DeviceGuard dg(h->device);
    cudaStream_t s = S(stream);
    DevLevel& d = h->lv[level];
    return smooth_into(h, h, level, b, x_in, x_out, sweeps, d.x64[0], s);
}

mg_status mg_residual_restrict(mg_handle* h, int32_t level, const double* b, const double* x, double* bc,
                               void* stream) {
    TRY(check_level(h, level));
    if (level + 1 >= h->L || !b || !x || !bc) return MG_ERR_ARG;
    DeviceGuard dg(h->device);
    if (h->nine) return restrict9<double, double, double>(h, level, x, b, bc, S(stream));
    TRY(ready64(h, level, S(stream)));
    return launch_restrict64<true>(h, level, x, b, bc, S(stream));
}

mg_status mg_prolong_add(mg_handle* h, int32_t level, const double* xc, double* x, void* stream) {
    TRY(check_level(h, level));
    if (level + 1 >= h->L || !xc || !x) return MG_ERR_ARG;
    DeviceGuard dg(h->device);
    const DevLevel& d = h->lv[level];
    return launch_prolong<double, false, double, double>(h, level, d.n, d.ncol, h->lv[level + 1].ncol, h->nlev, x, xc, x,
                                                         S(stream));
}

mg_status mixed_apply(mg_handle* h, const double* u, const double* p, double* yu, double* yp, void* stream) {
    if (!h || !u || !p || !yu || !yp) return MG_ERR_ARG;
    if (!h->mixed) return MG_ERR_UNSUPPORTED;
    DeviceGuard dg(h->device);
    cudaStream_t s = S(stream);
    const bool in_place = yp == p;   // (velocity rows read p of both cells: the pressure rows wait in mx then)
    double* const to = in_place ? h->mx + h->nu : yp;
    {
        Prof pr(h, MG_K_MIXED, 0, 8.0 * (2.0 * h->nu + 3.0 * cells(h, 0)), s);
        TRY((launch_mixed<mg::MX_A, -1>(h, u, p, yu, to, nullptr, s)));
    }
    if (in_place) CK(cudaMemcpyAsync(yp, to, cells(h, 0) * sizeof(double), cudaMemcpyDeviceToDevice, s));
    return MG_OK;
}

mg_status schur_precond(mg_handle* h, const double* ru, const double* rp, double* u, double* p, void* stream) {
    if (!h || !ru || !rp || !u || !p) return MG_ERR_ARG;
    if (!h->mixed) return MG_ERR_UNSUPPORTED;
    DeviceGuard dg(h->device);
    return schur_impl(h, ru, rp, u, p, nullptr, S(stream));
}

mg_status mg_autotune(mg_handle* h, int32_t* choices, void* stream) {
    NvtxRange nvtx_("mg_autotune");
    if (!h) return MG_ERR_ARG;
    if (h->prof || h->nine) return MG_ERR_UNSUPPORTED;   // the tuner uses the per-launch profiler itself
    DeviceGuard dg(h->device);
    cudaStream_t s = S(stream);
    const int L = h->L;
    const size_t N = cells(h, 0);
    constexpr int REPS = 3;
    // every launch of REPS V-cycles is recorded: 2 kinds x L levels x (sweeps + 1) at most
    const int cap = 2 * REPS * L * (h->prm.n_pre + h->prm.n_post + h->prm.n_coarse + 4);
    while ((int)h->evpool.size() < 2 * cap) {
        cudaEvent_t e;
        CK(cudaEventCreate(&e));
        h->evpool.push_back(e);
    }
    // a V-cycle on the handle's own buffers: b = 0 (the launches, and so their times, do not
    // depend on the values)
    CK(cudaMemsetAsync(h->r, 0, N * sizeof(double), s));
    std::vector<double> sweep_ms(L), restr_ms(L);
    auto measure = [&]() -> mg_status {
        TRY(run_vcycle(h, h->r, h->adj, s));   // warm-up with this shape
        h->prof_kind = -1;
        h->prof_level = -1;
        h->recs.clear();
        h->prof = true;
        mg_status st = MG_OK;
        for (int i = 0; i < REPS && st == MG_OK; ++i) st = run_vcycle(h, h->r, h->adj, s);
        h->prof = false;
        TRY(st);
        CK(cudaStreamSynchronize(s));
        std::fill(sweep_ms.begin(), sweep_ms.end(), 0.0);
        std::fill(restr_ms.begin(), restr_ms.end(), 0.0);
        for (size_t i = 0; i < h->recs.size(); ++i) {
            float ms = 0.f;
            CK(cudaEventElapsedTime(&ms, h->evpool[2 * i], h->evpool[2 * i + 1]));
            const auto& r = h->recs[i];
            if (r.level < 0 || r.level >= L) continue;
            if (r.kind == MG_K_SWEEP) sweep_ms[r.level] += ms;
            if (r.kind == MG_K_RESTRICT) restr_ms[r.level] += ms;
        }
        h->recs.clear();
        return MG_OK;
    };
    // FP32 sweeps: 64: register chunks, 128: tensor-copy tiles where the level has them
    std::vector<int> best_bd(L, 0);
    std::vector<double> best_t(L, 1e300);
    for (int bd : {64, 128}) {
        for (int l = 0; l < L; ++l) h->lv[l].sweep_bd = bd;
        TRY(measure());
        for (int l = 0; l < L; ++l)
            if (sweep_ms[l] < best_t[l]) best_t[l] = sweep_ms[l], best_bd[l] = bd;
    }
    for (int l = 0; l < L; ++l) h->lv[l].sweep_bd = best_bd[l];
    // residual + restriction: the built-in levels per thread (kc = 0) unless another is faster (1 or 2 on most
    // levels: none of the others, C48L30 6.5 us against 13 with eight)
    std::vector<int> best_kc(L, 0), built_in(L, -1);
    std::vector<double> own_t(L);
    std::fill(best_t.begin(), best_t.end(), 1e300);
    for (int kc : {0, 4, 8, 16, 24, 35, 70}) {
        for (int l = 0; l < L; ++l) h->lv[l].restrict_kc = kc;
        TRY(measure());
        if (kc == 0) own_t = restr_ms;
        for (int l = 0; l + 1 < L && kc > 0; ++l)
            if (restr_ms[l] < best_t[l]) best_t[l] = restr_ms[l], best_kc[l] = kc;
    }
    for (int l = 0; l < L; ++l) {
        if (l + 1 < L) built_in[l] = own_t[l] <= best_t[l];
        h->lv[l].restrict_kc = built_in[l] == 1 ? 0 : best_kc[l];
    }
    drop_graphs(h, 0);   // (they hold the old launch shapes)
    if (choices)
        for (int l = 0; l < L; ++l) {
            choices[3 * l] = best_bd[l];
            choices[3 * l + 1] = best_kc[l];
            choices[3 * l + 2] = built_in[l];
        }
    return MG_OK;
}

mg_status mg_apply_choices(mg_handle* h, const int32_t* choices) {
    if (!h || !choices) return MG_ERR_ARG;
    for (int l = 0; l < h->L; ++l) {
        const int form = choices[3 * l], kc = choices[3 * l + 1];
        if ((form != 0 && form != 64 && form != 128) || kc < 0 || kc > MG_MAX_NLEV) return MG_ERR_ARG;
    }
    DeviceGuard dg(h->device);
    CK(cudaDeviceSynchronize());
    for (int l = 0; l < h->L; ++l) {
        h->lv[l].sweep_bd = choices[3 * l];
        h->lv[l].restrict_kc = choices[3 * l + 2] == 1 ? 0 : choices[3 * l + 1];
    }
    drop_graphs(h, 0);
    return MG_OK;
}

mg_status mg_profile_start(mg_handle* h, int32_t capacity, int32_t kind, int32_t level) {
    if (!h || capacity < 1 || capacity > (1 << 20)) return MG_ERR_ARG;
    h->prof_kind = kind < 0 ? -1 : kind;
    h->prof_level = level < 0 ? -1 : level;
    DeviceGuard dg(h->device);
    while ((int)h->evpool.size() < 2 * capacity) {
        cudaEvent_t e;
        CK(cudaEventCreate(&e));
        h->evpool.push_back(e);
    }
    h->recs.clear();
    h->recs.reserve(capacity);
    h->prof = true;
    return MG_OK;
}

mg_status mg_profile_stop(mg_handle* h, mg_kernel_record* out, int32_t cap, int32_t* count) {
    if (!h || !count || (cap > 0 && !out)) return MG_ERR_ARG;
    DeviceGuard dg(h->device);
    h->prof = false;
    CK(cudaDeviceSynchronize());
    const int n = (int)h->recs.size();
    for (int i = 0; i < n && i < cap; ++i) {
        float ms = 0.f;
        CK(cudaEventElapsedTime(&ms, h->evpool[2 * i], h->evpool[2 * i + 1]));
        out[i].kind = h->recs[i].kind;
        out[i].level = h->recs[i].level;
        out[i].variant = h->recs[i].variant;
        out[i].bytes = h->recs[i].bytes;
        out[i].ms = ms;
    }
    *count = n;
    h->recs.clear();
    return MG_OK;
}

}  // extern "C"

// =====================================================================================
// Block-Jacobi smoothing without allocation (see mg_smooth_noalloc in mgsolve.h).
//
// The intermediate iterates that mg_smooth keeps in the handle's workspace live here in
// one fixed device array instead.  Every GPU that loads this library holds the array until
// the process exits, and every call shares it.
static __device__ __align__(256) double g_smooth_scratch[MG_NOALLOC_MAX_CELLS];

namespace {
// Host code cannot use g_smooth_scratch as a device address: on the host it names a
// stand-in object.  Its device address is looked up once per device (with that device
// current) and kept here.
constexpr int kMaxDevices = 64;
std::mutex g_scratch_mutex;
double* g_scratch_addr[kMaxDevices] = {};

mg_status scratch_address(int device, double** out) {
    if (device < 0 || device >= kMaxDevices) return MG_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    if (!g_scratch_addr[device]) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_smooth_scratch);
        if (e != cudaSuccess || !p) {
            cudaGetLastError();
            return MG_ERR_CUDA;
        }
        g_scratch_addr[device] = static_cast<double*>(p);
    }
    *out = g_scratch_addr[device];
    return MG_OK;
}
}  // namespace

extern "C" mg_status mg_smooth_noalloc(mg_handle* h, int32_t level, const double* b, const double* x_in,
                                       double* x_out, int32_t sweeps, void* stream) {
    TRY(check_level(h, level));
    if (!b || !x_out || sweeps < 0 || b == x_out) return MG_ERR_ARG;
    if (h->nine) return MG_ERR_UNSUPPORTED;
    const size_t n = cells(h, level);
    if (n > (size_t)MG_NOALLOC_MAX_CELLS) return MG_ERR_ARG;
    DeviceGuard dg(h->device);
    double* scratch = nullptr;
    TRY(scratch_address(h->device, &scratch));
    cudaStream_t s = S(stream);
    return smooth_into(h, nullptr, level, b, x_in, x_out, sweeps, scratch, s);
}
