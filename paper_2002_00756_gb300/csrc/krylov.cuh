// FP64 vector kernels of the outer GCR iteration (Sec. 4.1 solver framework: axpy and
// inner products of the abstract vector type) and of the mixed system (Sec. 3.3-3.4).
//
// Inner products use a fixed grid, a fixed in-block shuffle tree and a last-block final
// sum in block order, so every run of the same launch gives bitwise the same scalars.
// The last block is found with a ticket counter (no block ever waits on another).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "kernels.cuh"

namespace mg {

constexpr int RED_THREADS = 256;
constexpr int MAXR = 16;   // maximum GCR restart length (MG_MAX_RESTART)

// device scalar block of the GCR iteration
struct GcrScal {
    double beta[MAXR * MAXR];   // beta[j * MAXR + i]: w_j orthogonalised against w_i, i < j
    double alpha[MAXR];         // step length of direction j
    double ww[MAXR];            // <w_i, w_i> of the orthogonalised directions
    double rr, bb;              // <r, r>, <b, b>
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// Sums v[0..ND) over the whole grid (any 1-D or 2-D grid of RED_THREADS-thread blocks).
// Each block writes its ND partial sums; the last block to finish (ticket counter, no
// waiting) adds all partials with every thread taking a fixed stride of blocks, then a
// fixed tree; thread 0 of that block gets the totals in `tot` and the function returns
// true there.  The order of every addition is fixed, so results are bitwise repeatable.
//
// An FP64 instruction of a warp takes the SM's pipe 16 cycles whatever its lanes do, so a block's
// threads meet in shared memory and one warp per sum adds 8 values a lane before its tree: 12
// instructions per block and sum, where a shuffle tree in each warp takes 40 and more.  With event
// overhead (about 4 us), C48L30: orthogonalisation 14.4 -> 12.3 us, fused apply 20.5 .. 30.8 -> 18.4 .. 24.6;
// C12L30: 12.3 -> 8.2 and 10.2 .. 14.4 -> 10.2 .. 12.3.
template <int ND>
__device__ __forceinline__ void block_sums(const double (&v)[ND], double (*sm)[RED_THREADS], double* to, size_t stride) {
    constexpr int W = RED_THREADS / 32;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < ND; ++i) sm[i][threadIdx.x] = v[i];
    __syncthreads();
    for (int i = wid; i < ND; i += W) {
        double s = sm[i][lane];
#pragma unroll
        for (int w = 1; w < W; ++w) s += sm[i][w * 32 + lane];
        s = warp_sum(s);
        if (lane == 0) {
            to[i * stride] = s;
            __threadfence();
        }
    }
    __syncthreads();
}

template <int ND>
__device__ bool grid_reduce(const double (&v)[ND], double* partials, unsigned int* ticket, double (&tot)[ND]) {
    __shared__ double sm[ND][RED_THREADS], total[ND];
    __shared__ bool last;
    const unsigned nblk = gridDim.x * gridDim.y, bid = blockIdx.y * gridDim.x + blockIdx.x;
    block_sums<ND>(v, sm, partials + bid, nblk);
    if (threadIdx.x == 0) last = (atomicAdd(ticket, 1u) == nblk - 1);
    __syncthreads();
    if (!last) return false;
    __threadfence();
    double a[ND];
#pragma unroll
    for (int i = 0; i < ND; ++i) a[i] = 0.0;
    for (unsigned b = threadIdx.x; b < nblk; b += RED_THREADS) {
#pragma unroll
        for (int i = 0; i < ND; ++i) a[i] += __ldcg(partials + (size_t)i * nblk + b);
    }
    block_sums<ND>(a, sm, total, 1);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int i = 0; i < ND; ++i) tot[i] = total[i];
        *ticket = 0u;
    }
    return threadIdx.x == 0;
}

// out = V x (multiply) or V^-1 x, V = area[col] * dz[k] the finest level's cell volumes
__global__ void k_scale_volume(int ncol, int nlev, const double* __restrict__ area, const double* __restrict__ dz,
                               const double* x, double* out, bool multiply) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (c >= ncol || k >= nlev) return;
    const size_t e = (size_t)k * ncol + c;
    const double v = __ldg(area + c) * __ldg(dz + k);
    out[e] = multiply ? x[e] * v : x[e] / v;
}

// ---- caller-supplied couplings a[s][k][c] (s = E, W, N, S, up, down) of the finest level ----
// Their face form: Th[k][f] = a_(owner, side)(k) area(owner) (horizontal), Tv[kf][c] =
// a_up(kf-1, c) dz[kf-1] (vertical).  Valid only for a flux-symmetric operator, V_i a_if = V_j a_jf:
// the other cell's product must agree to 1e-10 relative, every coupling must be finite and
// >= 0, and none may cross the surface or the lid.  A first pass (WRITE false) sets *bad where a check
// fails; the second stores the face form, checked by then.  The FP64 pipe bounds the first: signs,
// finiteness and closeness are tested on the words, and only doubtful pairs are compared in FP64 (C96L70: 40 and
// 33 us, second pass 34 and 18; four passes that all compared in FP64: 338 us).
// u and v finite, not negative and equal to 1e-10 of the larger
__device__ __forceinline__ bool coef_agree(double u, double v) {
    const long long tiny = 0x0010000000000000ll, inf = 0x7ff0000000000000ll;
    const long long iu = __double_as_longlong(u), iv = __double_as_longlong(v), dist = iu > iv ? iu - iv : iv - iu;
    // positive normal numbers at most 2^18 units in the last place apart: within 2^-34 = 5.8e-11
    if (iu >= tiny && iv >= tiny && iu < inf && iv < inf && dist <= (1 << 18)) return true;
    return u >= 0.0 && v >= 0.0 && isfinite(u) && isfinite(v) && fabs(u - v) <= 1e-10 * fmax(fabs(u), fabs(v));
}

// horizontal face f of level k
template <bool WRITE>
__device__ __forceinline__ void coef_face(int f, int k, int ncol, int nlev, const int32_t* __restrict__ faceL,
                                          const int32_t* __restrict__ faceR, const int32_t* __restrict__ faceSide,
                                          const int32_t* __restrict__ nbrSide, const double* __restrict__ area,
                                          const double* __restrict__ a, double* __restrict__ Th, unsigned int* bad) {
    const size_t N = (size_t)nlev * ncol, o = (size_t)k * ncol;
    const int L = faceL[f], s = faceSide[f];
    const double tl = a[s * N + o + L] * area[L];
    if (WRITE) {
        Th[(size_t)k * 2 * ncol + f] = tl;
    } else {
        const int R = faceR[f], sr = nbrSide[s * ncol + L];
        if (!coef_agree(tl, a[sr * N + o + R] * area[R])) atomicOr(bad, 1u);
    }
}

// vertical face kf of column c
template <bool WRITE>
__device__ __forceinline__ void coef_vertical(int c, int kf, int ncol, int nlev, const double* __restrict__ dz,
                                              const double* __restrict__ a, double* __restrict__ Tv, unsigned int* bad) {
    const size_t N = (size_t)nlev * ncol;
    if (WRITE) {
        Tv[(size_t)kf * ncol + c] = kf == 0 || kf == nlev ? 0.0 : a[4 * N + (size_t)(kf - 1) * ncol + c] * dz[kf - 1];
    } else if (kf == 0) {
        if (a[5 * N + c] != 0.0) atomicOr(bad, 1u);                             // a_dn of the bottom cell
    } else if (kf == nlev) {
        if (a[4 * N + (size_t)(nlev - 1) * ncol + c] != 0.0) atomicOr(bad, 1u);  // a_up of the top cell
    } else {
        const double up = a[4 * N + (size_t)(kf - 1) * ncol + c], dn = a[5 * N + (size_t)kf * ncol + c];
        const bool signs = (__double_as_longlong(up) | __double_as_longlong(dn)) >= 0 || (up >= 0.0 && dn >= 0.0);
        if (!signs || !coef_agree(up * dz[kf - 1], dn * dz[kf])) atomicOr(bad, 1u);
    }
}

// a6[s][e] = a[s][e] (s < 6) and a6[6][e] = 1 + their sum: the FP64 operator of the GCR apply
__device__ __forceinline__ void coef_cell(size_t e, size_t N, const double* __restrict__ a, double* __restrict__ a6) {
    double d = 1.0;
#pragma unroll
    for (int s = 0; s < 6; ++s) {
        const double v = a[s * N + e];
        a6[s * N + e] = v;
        d += v;
    }
    a6[6 * N + e] = d;
}

// One launch for the checks and one for the stores: rows of the grid are the horizontal faces' levels,
// then the vertical faces', then (WRITE) the cells'.  Small handles' calls are mostly launches and two host
// round trips: C12L30 FP64 60 us, with a launch per
// kind, a cleared flag and pageable read-back 78; C30L1 47 and 64.
template <bool WRITE>
__global__ void __launch_bounds__(128) k_coef(int ncol, int nlev, const int32_t* __restrict__ faceL, const int32_t* __restrict__ faceR,
                       const int32_t* __restrict__ faceSide, const int32_t* __restrict__ nbrSide,
                       const double* __restrict__ area, const double* __restrict__ dz, const double* __restrict__ a,
                       double* __restrict__ Th, double* __restrict__ Tv, double* __restrict__ a6, unsigned int* bad) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (k < nlev) {
        if (i < 2 * ncol) coef_face<WRITE>(i, k, ncol, nlev, faceL, faceR, faceSide, nbrSide, area, a, Th, bad);
    } else if (i < ncol) {
        if (k <= 2 * nlev) coef_vertical<WRITE>(i, k - nlev, ncol, nlev, dz, a, Tv, bad);
        else if (WRITE) coef_cell((size_t)(k - 2 * nlev - 1) * ncol + i, (size_t)nlev * ncol, a, a6);
    }
}

// grad[s][e] = -lam_e (x_e - x_(neighbour s of e)), s = E, W, N, S, up, down (0 without a
// neighbour): the gradient of L(x) with respect to the six couplings of the finest level
__global__ void k_coef_grad(Lvl<double, double> L, const double* __restrict__ lam, const double* __restrict__ x,
                            double* __restrict__ grad) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (c >= L.ncol || k >= L.nlev) return;
    const size_t ncol = L.ncol, N = (size_t)L.nlev * ncol, e = (size_t)k * ncol + c;
    const double l = lam[e], x0 = x[e];
#pragma unroll
    for (int s = 0; s < 4; ++s) grad[s * N + e] = -l * (x0 - x[(size_t)k * ncol + __ldg(L.nbr + s * ncol + c)]);
    grad[4 * N + e] = k + 1 < L.nlev ? -l * (x0 - x[e + ncol]) : 0.0;
    grad[5 * N + e] = k > 0 ? -l * (x0 - x[e - ncol]) : 0.0;
}

// Start of a GCR solve: r = b, x = 0, <b, b> and no wait run out yet, in one pass over memory (a copy, a fill and
// a product before).  <b, b> goes straight to the host, which waits for it before the first iteration: a zero
// right-hand side costs no more than this (C192L70 98 us).  Launching the first iteration ahead of <b, b>
// instead: a zero right-hand side 985 us, other solves 342 -> 343 us (C12L30), 711 -> 718 (C48L30), 9.33 -> 9.27 ms
// (C192L70).
__global__ void __launch_bounds__(RED_THREADS) k_gcr_start(size_t n, const double* __restrict__ b, double* __restrict__ r,
                                                           double* __restrict__ x, double* partials,
                                                           unsigned int* ticket, double* bb, double* host_bb,
                                                           unsigned int* timeout) {
    double v[1] = {0.0}, t[1];
    if (blockIdx.x == 0 && threadIdx.x == 0) *timeout = 0u;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const double e = __ldg(b + i);
        r[i] = e;
        x[i] = 0.0;
        v[0] = fma(e, e, v[0]);
    }
    if (grid_reduce<1>(v, partials, ticket, t)) {
        *bb = t[0];
        if (host_bb) *host_bb = t[0];   // (pinned; a copy of its own would be one more step before the host knows)
    }
}

// ---- BiCGStab for the pressure system (van der Vorst 1992, right-preconditioned) ----
// Device scalars of one solve: every vector kernel reads them, the last block of each
// reduction writes the ones it completes, and the host reads the block once per iteration.
struct BicgScal {
    double bb;              // <b, b>
    double rho, rho_old;    // <r^, r> of this step and of the one before
    double alpha, omega;
    double ss, rr;          // <s, s>, <r, r>
    double tol2bb;          // tol^2 <b, b>
    int half;               // ||s|| <= tol ||b||: the step ends after its first half
};

// y = H z on the finest level from the premultiplied couplings a6 (diagonal form, FP64)
__global__ void k_apply_a6(Lvl<double, double> L, const double* __restrict__ a6, const double* __restrict__ z,
                           double* __restrict__ w) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (c >= L.ncol || k >= L.nlev) return;
    const size_t ncol = L.ncol, N = (size_t)L.nlev * ncol, o = (size_t)k * ncol, e = o + c;
    double we = __ldg(a6 + 6 * N + e) * __ldg(z + e);
#pragma unroll
    for (int s = 0; s < 4; ++s) we = fma(-__ldg(a6 + s * N + e), __ldg(z + o + __ldg(L.nbr + s * ncol + c)), we);
    if (k + 1 < L.nlev) we = fma(-__ldg(a6 + 4 * N + e), __ldg(z + e + ncol), we);
    if (k > 0) we = fma(-__ldg(a6 + 5 * N + e), __ldg(z + e - ncol), we);
    w[e] = we;
}

#define MG_GRID_STRIDE(i, n) \
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < (n); i += (size_t)gridDim.x * blockDim.x)

// r = r^ = b, x = 0; rho = <b, b>
__global__ void __launch_bounds__(RED_THREADS) k_bicg_start(size_t n, const double* __restrict__ b, double* r,
                                                            double* rh, double* x, double tol, double* partials,
                                                            unsigned int* ticket, BicgScal* S, unsigned int* timeout) {
    double v[1] = {0.0}, t[1];
    if (blockIdx.x == 0 && threadIdx.x == 0) *timeout = 0u;
    MG_GRID_STRIDE(i, n) {
        const double bi = b[i];
        r[i] = bi;
        rh[i] = bi;
        x[i] = 0.0;
        v[0] += bi * bi;
    }
    if (grid_reduce<1>(v, partials, ticket, t)) {
        S->bb = t[0];
        S->rho = t[0];
        S->rho_old = 1.0;
        S->alpha = 1.0;
        S->omega = 1.0;
        S->tol2bb = tol * tol * t[0];
        S->half = 0;
    }
}

// p = r (first step) or p = r + (rho / rho_old)(alpha / omega)(p - omega v)
__global__ void k_bicg_dir(size_t n, const double* __restrict__ r, const double* __restrict__ v, double* p, bool first,
                           const BicgScal* S) {
    const double om = S->omega, beta = (S->rho / S->rho_old) * (S->alpha / om);
    MG_GRID_STRIDE(i, n) p[i] = first ? r[i] : r[i] + beta * (p[i] - om * v[i]);
}

// alpha = rho / <r^, v>
__global__ void __launch_bounds__(RED_THREADS) k_bicg_alpha(size_t n, const double* __restrict__ rh,
                                                            const double* __restrict__ v, double* partials,
                                                            unsigned int* ticket, BicgScal* S) {
    double a[1] = {0.0}, t[1];
    MG_GRID_STRIDE(i, n) a[0] += rh[i] * v[i];
    if (grid_reduce<1>(a, partials, ticket, t)) S->alpha = S->rho / t[0];
}

// s = r - alpha v, <s, s>, and whether the step ends here
__global__ void __launch_bounds__(RED_THREADS) k_bicg_s(size_t n, const double* __restrict__ r,
                                                        const double* __restrict__ v, double* sv, double* partials,
                                                        unsigned int* ticket, BicgScal* S) {
    const double al = S->alpha;
    double a[1] = {0.0}, t[1];
    MG_GRID_STRIDE(i, n) {
        const double si = r[i] - al * v[i];
        sv[i] = si;
        a[0] += si * si;
    }
    if (grid_reduce<1>(a, partials, ticket, t)) {
        S->ss = t[0];
        S->half = t[0] <= S->tol2bb;
    }
}

// omega = <t, s> / <t, t>
__global__ void __launch_bounds__(RED_THREADS) k_bicg_omega(size_t n, const double* __restrict__ tv,
                                                            const double* __restrict__ sv, double* partials,
                                                            unsigned int* ticket, BicgScal* S) {
    double a[2] = {0.0, 0.0}, t[2];
    MG_GRID_STRIDE(i, n) {
        a[0] += tv[i] * sv[i];
        a[1] += tv[i] * tv[i];
    }
    if (grid_reduce<2>(a, partials, ticket, t)) S->omega = t[0] / t[1];
}

// x += alpha p^ + omega s^, r = s - omega t (after a half step: x += alpha p^, r = s);
// then rho_old = rho, rho = <r^, r>, rr = <r, r>
__global__ void __launch_bounds__(RED_THREADS) k_bicg_xr(size_t n, double* x, double* r, const double* __restrict__ ph,
                                                         const double* __restrict__ sh, const double* __restrict__ sv,
                                                         const double* __restrict__ tv, const double* __restrict__ rh,
                                                         double* partials, unsigned int* ticket, BicgScal* S) {
    const double al = S->alpha, om = S->omega;
    const bool half = S->half != 0;
    double a[2] = {0.0, 0.0}, t[2];
    MG_GRID_STRIDE(i, n) {
        double ri;
        if (half) {
            x[i] += al * ph[i];
            ri = sv[i];
        } else {
            x[i] += al * ph[i] + om * sh[i];
            ri = sv[i] - om * tv[i];
        }
        r[i] = ri;
        a[0] += rh[i] * ri;
        a[1] += ri * ri;
    }
    if (grid_reduce<2>(a, partials, ticket, t)) {
        S->rho_old = S->rho;
        S->rho = t[0];
        S->rr = t[1];
    }
}

// ---- one graph launch for an ensemble of pressure solves ----
// Every member's GCR iterations run inside a conditional WHILE node of one CUDA graph; within
// it, an IF node per restart slot j holds the V-cycle, the fused apply and the orthogonalisation
// of slot j, and a second IF node the solution update that closes a restart cycle.  The
// decisions the host takes after each iteration of a single solve (converged, breakdown,
// iteration limit, end of a restart cycle) are taken here by one thread, in the same order
// and FP64 arithmetic, by setting the conditions of those nodes.
struct EnsState {
    double bb;     // <b, b>
    double rel;    // ||r|| / ||b|| after the last iteration
    int it;        // iterations done
    int status;    // MG_OK, MG_ERR_NOT_CONVERGED, MG_ERR_BREAKDOWN or MG_ERR_TIMEOUT
};

struct EnsHandles {
    cudaGraphConditionalHandle w;          // WHILE: another iteration
    cudaGraphConditionalHandle c[MAXR];    // IF: iteration of slot j
    cudaGraphConditionalHandle x[MAXR];    // IF: solution update after slot j
};

// the device's global nanosecond clock
__global__ void k_stamp(unsigned long long* out) {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    *out = t;
}

__device__ void ens_set_slots(const EnsHandles& hs, int R, int next, bool go) {
    for (int k = 0; k < R; ++k) {
        cudaGraphSetConditional(hs.c[k], (go && k == next) ? 1u : 0u);
        cudaGraphSetConditional(hs.x[k], 0u);
    }
}

// after <b, b>: start iterating unless b = 0, <b, b> is not finite or no iteration is allowed
__global__ void k_ens_init(const GcrScal* S, EnsState* st, int R, int max_iter, EnsHandles hs) {
    const double bb = S->bb;
    const bool bad = !isfinite(bb);
    const bool go = !bad && bb > 0.0 && max_iter > 0;
    st->bb = bb;
    st->it = 0;
    st->rel = (!bad && bb > 0.0) ? 1.0 : 0.0;
    st->status = bad ? MG_ERR_BREAKDOWN : (go ? MG_ERR_NOT_CONVERGED : MG_OK);
    ens_set_slots(hs, R, 0, go);
    cudaGraphSetConditional(hs.w, go ? 1u : 0u);
}

// after the iteration of slot j: the convergence test and the solution update of a single solve
__global__ void k_ens_decide(const GcrScal* S, EnsState* st, int j, int R, int max_iter, double tol, EnsHandles hs,
                             const unsigned int* timeout) {
    const int it = st->it + 1;
    st->it = it;
    const double rr = S->rr;
    if (!isfinite(rr)) {   // breakdown: stop without the update (x keeps the last cycle's value)
        st->status = *timeout ? MG_ERR_TIMEOUT : MG_ERR_BREAKDOWN;
        ens_set_slots(hs, R, 0, false);
        cudaGraphSetConditional(hs.w, 0u);
        return;
    }
    const double rel = sqrt(rr / st->bb);
    st->rel = rel;
    const bool done = rel <= tol;
    if (done) st->status = MG_OK;
    const bool go = !done && it < max_iter;
    ens_set_slots(hs, R, j + 1 < R ? j + 1 : 0, go);
    cudaGraphSetConditional(hs.x[j], (j == R - 1 || done || it == max_iter) ? 1u : 0u);
    cudaGraphSetConditional(hs.w, go ? 1u : 0u);
}

// GCR step coefficients for direction J (classical Gram-Schmidt, one pass):
//   beta_i = <w, w_i> / <w_i, w_i>,  <w', w'> = <w, w> - sum_i beta_i <w, w_i>,
//   alpha = <r, w'> / <w', w'> with <r, w'> = <r, w> (the GCR residual is orthogonal to
//   all earlier directions w_i), from sums = [<w, w_i> (J), <w, w>, <r, w>].
// Every kernel below is instantiated for the exact number J of stored directions, so no
// FP64 instruction is spent on absent directions (FP64 issue rate bounds these kernels).
// <w', w'> is kept for the later directions' beta: the orthogonalisation pass does not
// recompute it (the FP64 pipe bounds that pass on GB300).
template <int J>
__device__ void gcr_coeffs(const double (&t)[J + 2], GcrScal* S) {
    double ww = t[J];
#pragma unroll
    for (int i = 0; i < J; ++i) {
        const double beta = t[i] / S->ww[i];
        S->beta[J * MAXR + i] = beta;
        ww -= beta * t[i];
    }
    S->ww[J] = ww;
    S->alpha[J] = t[J + 1] / ww;
}


template <int J>
__device__ __forceinline__ void gcr_accumulate(double (&v)[J + 2], double we, double re,
                                               const double* __restrict__ Wb, size_t ld, size_t e) {
#pragma unroll
    for (int i = 0; i < J; ++i) v[i] += we * __ldg(Wb + (size_t)i * ld + e);
    v[J] += we * we;
    v[J + 1] += re * we;
}

// GCR sums for a new direction w of the 9-cell stencil, whose operator is a kernel of its own.
template <int J>
__global__ void __launch_bounds__(RED_THREADS) k_gcr_sums(size_t n, const double* __restrict__ w,
                                                          const double* __restrict__ Wb, size_t ld,
                                                          const double* __restrict__ r, double* partials,
                                                          unsigned int* ticket, GcrScal* S) {
    double v[J + 2], t[J + 2];
#pragma unroll
    for (int i = 0; i < J + 2; ++i) v[i] = 0.0;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
        gcr_accumulate<J>(v, __ldg(w + e), __ldg(r + e), Wb, ld, e);
    if (grid_reduce<J + 2>(v, partials, ticket, t)) gcr_coeffs<J>(t, S);
}

// w_J <- w_J - sum_i beta_i w_i (stored in place), r <- r - alpha_J w_J, then <r, r> -> rr
// (FP64: the residual spans the right-hand side's whole range, whose squares FP32 would
// flush to zero below about 1e-19).
template <int J>
__global__ void __launch_bounds__(RED_THREADS) k_gcr_orth_update(size_t n, double* __restrict__ Wb, size_t ld,
                                                                 double* __restrict__ r, double* partials,
                                                                 unsigned int* ticket, GcrScal* S) {
    double beta[J > 0 ? J : 1];
#pragma unroll
    for (int i = 0; i < J; ++i) beta[i] = S->beta[J * MAXR + i];
    const double a = S->alpha[J];
    double* w = Wb + (size_t)J * ld;
    double v[1] = {0.0}, t[1];
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        double we = w[e];
#pragma unroll
        for (int i = 0; i < J; ++i) we = fma(-beta[i], __ldg(Wb + (size_t)i * ld + e), we);
        if (J > 0) w[e] = we;
        const double re = fma(-a, we, r[e]);
        r[e] = re;
        v[0] = fma(re, re, v[0]);
    }
    if (grid_reduce<1>(v, partials, ticket, t)) S->rr = t[0];
}

// x += sum_{i <= JL} gamma_i z_i with the raw (not orthogonalised) directions z_i:
// x = sum_i alpha_i zhat_i, zhat_i = z_i - sum_{m<i} beta_im zhat_m, unrolled from the top.
template <int JL>
__global__ void k_gcr_xupdate(size_t n, double* __restrict__ x, const double* __restrict__ Zb, size_t ld,
                              const GcrScal* __restrict__ S) {
    __shared__ double g[JL + 1];
    if (threadIdx.x == 0) {
        double a[JL + 1];
        for (int i = 0; i <= JL; ++i) a[i] = S->alpha[i];
        for (int i = JL; i >= 0; --i) {
            g[i] = a[i];
            for (int m = 0; m < i; ++m) a[m] -= a[i] * S->beta[i * MAXR + m];
        }
    }
    __syncthreads();
    double gr[JL + 1];
#pragma unroll
    for (int i = 0; i <= JL; ++i) gr[i] = g[i];
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
        double xe = x[e];
#pragma unroll
        for (int i = 0; i <= JL; ++i) xe += gr[i] * __ldg(Zb + (size_t)i * ld + e);
        x[e] = xe;
    }
}

// ---------------------------------------------------------------------------------------
// Mixed system (u, p) kernels; see mgsolve.h for the velocity layout.
struct MixedDev {
    int ncol, nlev, nfh;            // nfh = 2 ncol horizontal faces per level
    const int32_t* faceL;           // [nfh]
    const int32_t* faceR;           // [nfh]
    const int32_t* fof;             // [4][ncol]
    const double* sdiv;             // [4][ncol] +-c_s dt (edge length / area), + if the column owns the face
    const double* kd_h;             // [nlev][nfh]   kappa_f / d_f, kappa_f = c_s dt g_f
    const double* kd_v;             // [nlev+1][ncol]
    const double* w_up;             // [nlev+1][ncol] eps beta_up (interior couplings only)
    const double* w_dn;             // [nlev+1][ncol]
    const double* rmlump;           // [nlev+1][ncol] 1 / row sums of M-bar
    const double* divv;             // [nlev] c_s dt / dz
    // horizontal faces: M_h u_f = ms u_f + sum_t wf[t][f] u_cf[t][f] (t < ncf), the same on
    // every level; lumped to 1 / rmlump_h
    int ncf;
    const int32_t* cf;              // [ncf][nfh]
    const double* wf;               // [ncf][nfh]
    double ms;                      // horizontal self weight
    double mv;                      // vertical self weight (interior faces)
    const double* rmlump_h;         // [nfh] 1 / lumped mass
    // adjoint: wfT[t][f] = weight of the entry of row cf[t][f] of M_h that points to f (the
    // rows of M_h^T), and the face weights W_f = A_f d_f / g_f on [u_h, u_v] (area dz / g of
    // the cell on the surface and lid faces), under which A^T = S J A-hat J S^-1 with S = diag(W, V)
    const double* wfT;              // [ncf][nfh]
    const double* Wf;               // [nlev][nfh] then [nlev+1][ncol]
    // coefficient gradient: d(kappa_f / d_f) / d g_i = c_s dt / (2 d_f) for both cells of f
    const double* cdh;              // [nfh]      c_s dt / (2 centre distance)
    const double* cdv;              // [nlev+1]   c_s dt / (2 dzc), 0 on surface and lid
    const double* rW;               // 1 / Wf, of the same rounded weights (their own errors cancel in W^-1 M^T W)
    double eps;                     // strength of B_w
};

// [out_u; out_p] = J S^-1 [in_u; in_p] (MULT false) or S J [in_u; in_p] (MULT true), with
// S = diag(W, V) (V = area dz, the cell volumes) and J = diag(I, -I)
template <bool MULT>
__global__ void k_mx_adj_scale(MixedDev M, size_t nu, const double* __restrict__ area, const double* __restrict__ dz,
                               const double* in_u, const double* in_p, double* out_u, double* out_p) {
    const size_t np = (size_t)M.nlev * M.ncol;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nu + np; i += (size_t)gridDim.x * blockDim.x) {
        if (i < nu) {
            const double w = __ldg(M.Wf + i);
            out_u[i] = MULT ? in_u[i] * w : in_u[i] / w;
        } else {
            const size_t e = i - nu;
            const int k = (int)(e / M.ncol), c = (int)(e - (size_t)k * M.ncol);
            const double v = __ldg(area + c) * __ldg(dz + k);
            out_p[e] = MULT ? -(in_p[e] * v) : -(in_p[e] / v);
        }
    }
}

// dL/dg_i = -sum over the faces f of cell i of lam_f (p_R(f) - p_L(f)) c_s dt / (2 d_f): the
// background factors enter the mixed operator only through the gradient weights
// kappa_f / d_f = c_s dt (g_i + g_j) / (2 d_f).  One thread per cell.
__global__ void k_mx_grad_g(MixedDev M, const double* __restrict__ lam_u, const double* __restrict__ p,
                            double* __restrict__ grad_g) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (c >= M.ncol) return;
    const size_t ncol = M.ncol, op = (size_t)k * ncol;
    const double* lh = lam_u + (size_t)k * M.nfh;
    const double* lv = lam_u + (size_t)M.nlev * M.nfh;
    double s = 0.0;
#pragma unroll
    for (int d = 0; d < 4; ++d) {
        const int f = __ldg(M.fof + d * ncol + c);
        s -= lh[f] * (__ldg(p + op + __ldg(M.faceR + f)) - __ldg(p + op + __ldg(M.faceL + f))) * __ldg(M.cdh + f);
    }
    if (k >= 1)   // face k below the cell
        s -= lv[op + c] * (__ldg(p + op + c) - __ldg(p + op - ncol + c)) * __ldg(M.cdv + k);
    if (k + 1 <= M.nlev - 1)   // face k + 1 above it
        s -= lv[op + ncol + c] * (__ldg(p + op + ncol + c) - __ldg(p + op + c)) * __ldg(M.cdv + k + 1);
    grad_g[op + c] = s;
}

// dL/dbeta_up[kf] = -eps lam_kf u_kf+1 and dL/dbeta_dn[kf] = -eps lam_kf u_kf-1 on the
// vertical faces whose coupling exists (both faces interior), 0 elsewhere.
__global__ void k_mx_grad_beta(MixedDev M, const double* __restrict__ lam_v, const double* __restrict__ uv,
                               double* __restrict__ gup, double* __restrict__ gdn) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, kf = blockIdx.y;
    if (c >= M.ncol) return;
    const size_t ncol = M.ncol, o = (size_t)kf * ncol + c;
    const int nlev = M.nlev;
    gup[o] = (kf >= 1 && kf + 1 <= nlev - 1) ? -M.eps * lam_v[o] * uv[o + ncol] : 0.0;
    gdn[o] = (kf >= 2 && kf <= nlev - 1) ? -M.eps * lam_v[o] * uv[o - ncol] : 0.0;
}

// Pressure-system GCR pass 1: w = H z (FP64, Eq. helmholtz_operator) fused with the GCR sums of the
// new direction J.  The finest level keeps its six couplings and the diagonal 1 + sum_f a_f per cell
// premultiplied in FP64 (a6[side][k][c], sides E, W, N, S, up, down, then the diagonal), so H z costs 7
// and the sums J + 2 FP64 operations per cell: the FP64 pipe (two lanes per clock and SM), not memory,
// bounds this kernel.
//
// The units of work, 32 columns x kchunk levels, are dealt out over a grid that is resident at once,
// and a warp keeps its sums over all its units: one reduction per warp (it runs on the FP64 pipe as
// well) instead of one per 24 levels, and no last wave of blocks on a part of the chip.  At C192L70
// 252 / 276 / 305 / 330 / 356 us for J = 0..4 (one unit per thread, blocks in waves: 280 / 314 / 343 / 381
// / 417; the FP64 pipe's bound: 223 / 248 / 273 / 298 / 322); C48L30 18-25 us instead of 35-49.  Two, four
// and five blocks per SM: 256-369, 256-385, 258-391.
constexpr int APPLY_BLOCKS = 3;   // resident blocks per SM

// Levels per unit: the fewest rounds x (levels + about one level's worth of prologue); more than 18
// levels in a row cost more in cache reuse than they save.
inline int apply_chunk(int groups, int nlev, int warps) {
    int best = 1;
    double t = 1e300;
    for (int kc = 1; kc <= 18 && kc <= nlev; ++kc) {
        const long long units = (long long)groups * ((nlev + kc - 1) / kc);
        const double tk = (double)((units + warps - 1) / warps) * (kc + 1);
        if (tk <= t) t = tk, best = kc;
    }
    return best;
}

template <int J>
__global__ void __launch_bounds__(RED_THREADS, APPLY_BLOCKS) k_apply_gcr(
    Lvl<double, double> L, const double* __restrict__ a6, const double* __restrict__ z, double* __restrict__ w,
    const double* __restrict__ Wb, size_t ld, const double* __restrict__ r, int kchunk, int nchunk, double* partials,
    unsigned int* ticket, GcrScal* S) {
    double v[J + 2], t[J + 2];
#pragma unroll
    for (int i = 0; i < J + 2; ++i) v[i] = 0.0;
    const unsigned ncol = L.ncol, ngroup = (ncol + 31) >> 5, nunit = ngroup * nchunk;
    const unsigned lane = threadIdx.x & 31, nwarp = gridDim.x * (RED_THREADS / 32);
    const size_t N = (size_t)L.nlev * ncol;
    for (unsigned u = blockIdx.x * (RED_THREADS / 32) + (threadIdx.x >> 5); u < nunit; u += nwarp) {
        const unsigned ch = u / ngroup, c = (u - ch * ngroup) * 32 + lane;
        if (c >= ncol) continue;
        const int k0 = ch * kchunk, k1 = min(L.nlev, k0 + kchunk);
        unsigned nb[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) nb[s] = __ldg(L.nbr + s * ncol + c);
        double xm = k0 > 0 ? __ldg(z + (size_t)(k0 - 1) * ncol + c) : 0.0;
        double x0 = __ldg(z + (size_t)k0 * ncol + c);
#pragma unroll 2
        for (int k = k0; k < k1; ++k) {
            const size_t o = (size_t)k * ncol, e = o + c;
            const double xp = (k + 1 < L.nlev) ? __ldg(z + e + ncol) : 0.0;
            double we = __ldg(a6 + 6 * N + e) * x0;
            we = fma(-__ldg(a6 + e), __ldg(z + o + nb[0]), we);
            we = fma(-__ldg(a6 + N + e), __ldg(z + o + nb[1]), we);
            we = fma(-__ldg(a6 + 2 * N + e), __ldg(z + o + nb[2]), we);
            we = fma(-__ldg(a6 + 3 * N + e), __ldg(z + o + nb[3]), we);
            we = fma(-__ldg(a6 + 4 * N + e), xp, we);
            we = fma(-__ldg(a6 + 5 * N + e), xm, we);
            w[e] = we;
            gcr_accumulate<J>(v, we, __ldg(r + e), Wb, ld, e);
            xm = x0;
            x0 = xp;
        }
    }
    if (grid_reduce<J + 2>(v, partials, ticket, t)) gcr_coeffs<J>(t, S);
}

// Mixed system, the forms of k_mixed:
//   MX_A         y = A [u; p]: velocity rows M u + kd (p_R - p_L), pressure rows p + D u
//   MX_HAT       the same with W^-1 M^T W for M (rows of A-hat), from u and wu = W u
//   MX_RHS       Step 1: B = r_p - D M-ring^{-1} r_u (pressure rows only; p = r_p)
//   MX_UPDATE    Step 3: u' = M-ring^{-1} (r_u - kd (p_R - p_L)) (velocity rows only)
//   MX_UPDATE_W  the same, and W u' to wu
enum { MX_A = 0, MX_HAT = 1, MX_RHS = 2, MX_UPDATE = 3, MX_UPDATE_W = 4 };

// Units of work: 32 horizontal faces, vertical faces or cells by a run of levels, dealt out over a grid
// that is resident at once (as k_apply_gcr's).  Face numbers, couplings and weights of the columns are
// read once per unit, not once per level; with J >= 0 the GCR sums of the new direction J are taken in
// the same pass, while its rows are in registers (a pass over J + 2 vectors and three launches less).
// The FP64 pipe bounds MX_A and MX_HAT: 29 and 32 operations per cell (18 / 20 of them on its two
// horizontal faces) and 4 (J + 2) of the sums.  A-hat's weights therefore come from Step 3, which
// stores W u' beside u' (one product per face instead of six), and its quotient by W is a product with
// the stored reciprocal.  (1 / W put together from kd and the geometry would save the load, but its error is
// not the one of W u': RMS error of A^T v against long double 7.9e-17 at C24L30, 7.2e-17 with the stored
// reciprocal, 6.7e-17 with the quotient.)
// C48L30, sums of 0..4 directions included, on average: MX_A 38 us (four launches of a thread per row and
// level: 56), MX_HAT 54 us (91); the FP64 pipe's bound with J = 2: 32 and 36.  Steps 1 and 3 have few
// registers and run on five blocks per SM.
constexpr int mixed_blocks(int mode) { return mode >= MX_RHS ? 5 : APPLY_BLOCKS; }   // resident per SM

template <int MODE, int J>
__global__ void __launch_bounds__(RED_THREADS, mixed_blocks(MODE)) k_mixed(
    MixedDev M, const double* __restrict__ u, const double* __restrict__ p, double* __restrict__ yu,
    double* __restrict__ yp, double* __restrict__ wu, const double* __restrict__ Wb, size_t ld, const double* __restrict__ r, int kchunk,
    int nchunk, double* partials, unsigned int* ticket, GcrScal* S) {
    constexpr int NV = J >= 0 ? J + 2 : 1, JJ = J >= 0 ? J : 0;
    double v[NV], t[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = 0.0;
    const unsigned ncol = M.ncol, nfh = M.nfh, lane = threadIdx.x & 31, nwarp = gridDim.x * (RED_THREADS / 32);
    constexpr bool UPD = MODE == MX_UPDATE || MODE == MX_UPDATE_W;
    const unsigned gh = MODE == MX_RHS ? 0 : (nfh + 31) >> 5, gc = (ncol + 31) >> 5;
    const unsigned G = MODE == MX_RHS ? gc : UPD ? gh + gc : gh + 2 * gc;
    const size_t nh = (size_t)M.nlev * nfh, nu = nh + (size_t)(M.nlev + 1) * ncol;
    const double *uv = u + nh, *wv = MODE == MX_HAT ? wu + nh : uv;
    // m / W_e: the plain quotient in mixed_apply_transpose, the reciprocal in a solve's operator
    auto over_w = [&](double m, size_t e) { return J < 0 ? m / __ldg(M.Wf + e) : m * __ldg(M.rW + e); };
    // row e of [u; p] comes out as y
    auto put = [&](double* to, size_t e, double y) {
        *to = y;
        if (MODE == MX_UPDATE_W) wu[e] = __ldg(M.Wf + e) * y;
        if constexpr (J >= 0) gcr_accumulate<JJ>(v, y, __ldg(r + e), Wb, ld, e);
    };
    for (unsigned q = blockIdx.x * (RED_THREADS / 32) + (threadIdx.x >> 5); q < G * nchunk; q += nwarp) {
        const unsigned ch = q / G, g = q - ch * G;
        const int k0 = ch * kchunk, k1 = min(M.nlev, k0 + kchunk);
        if (MODE != MX_RHS && g < gh) {   // horizontal faces
            const unsigned f = g * 32 + lane;
            if (f >= nfh) continue;
            const unsigned fl = __ldg(M.faceL + f), fr = __ldg(M.faceR + f);
            const bool coupled = !UPD && M.ncf > 0;
            unsigned cf[6] = {};
            double wt[6] = {};
            if (coupled) {
#pragma unroll
                for (int i = 0; i < 6; ++i) {
                    cf[i] = __ldg(M.cf + (size_t)i * nfh + f);
                    wt[i] = __ldg((MODE == MX_HAT ? M.wfT : M.wf) + (size_t)i * nfh + f);
                }
            }
            const double rm = UPD ? __ldg(M.rmlump_h + f) : 0.0;
#pragma unroll 2
            for (int k = k0; k < k1; ++k) {
                const double *ul = (MODE == MX_HAT ? wu : u) + (size_t)k * nfh, *pl = p + (size_t)k * ncol;
                const size_t o = (size_t)k * nfh + f;
                const double kd = __ldg(M.kd_h + o), dp = __ldg(pl + fr) - __ldg(pl + fl), uf = __ldg(u + o);
                double y;
                if (UPD) {
                    y = fma(-kd, dp, uf) * rm;
                } else {
                    y = M.ms * uf;
                    double m = 0.0;
                    if (coupled) {
                        if (MODE == MX_A) m = y;
#pragma unroll
                        for (int i = 0; i < 6; ++i) m = fma(wt[i], __ldg(ul + cf[i]), m);
                        if (MODE == MX_A) y = m;
                        if (MODE == MX_HAT) y = fma(M.ms, uf, over_w(m, o));
                    }
                    y = fma(kd, dp, y);
                }
                put(yu + o, o, y);
            }
        } else if (MODE != MX_RHS && g < gh + gc) {   // vertical faces; the last run has the lid's as well
            const unsigned c = (g - gh) * 32 + lane;
            if (c >= ncol) continue;
            const int k2 = k1 == M.nlev ? k1 + 1 : k1;
            double ub = k0 > 0 ? __ldg(uv + (size_t)(k0 - 1) * ncol + c) : 0.0, u0 = __ldg(uv + (size_t)k0 * ncol + c);
            double pb = k0 > 0 ? __ldg(p + (size_t)(k0 - 1) * ncol + c) : 0.0;
#pragma unroll 2
            for (int k = k0; k < k2; ++k) {
                const size_t o = (size_t)k * ncol + c;
                double y = u0, ua = 0.0, pa = 0.0;
                if (k < M.nlev) {
                    ua = __ldg(uv + o + ncol);
                    pa = __ldg(p + o);
                    if (k > 0) {
                        const double kd = __ldg(M.kd_v + o), dp = pa - pb;
                        if (MODE == MX_A)
                            y = fma(kd, dp, fma(__ldg(M.w_dn + o), ub, fma(__ldg(M.w_up + o), ua, M.mv * u0)));
                        if (MODE == MX_HAT) {   // the couplings of the faces above and below to this one
                            const double m = fma(__ldg(M.w_up + o - ncol), __ldg(wv + o - ncol),
                                                 __ldg(M.w_dn + o + ncol) * __ldg(wv + o + ncol));
                            y = fma(kd, dp, fma(M.mv, u0, over_w(m, nh + o)));
                        }
                        if (UPD) y = fma(-kd, dp, u0) * __ldg(M.rmlump + o);
                    }
                }
                put(yu + nh + o, nh + o, y);
                ub = u0;
                u0 = ua;
                pb = pa;
            }
        } else if (!UPD) {   // cells
            const unsigned c = (MODE == MX_RHS ? g : g - gh - gc) * 32 + lane;
            if (c >= ncol) continue;
            unsigned ff[4];
            double sd[4];
#pragma unroll
            for (int d = 0; d < 4; ++d) {
                ff[d] = __ldg(M.fof + d * ncol + c);
                sd[d] = __ldg(M.sdiv + d * ncol + c);
                if (MODE == MX_RHS) sd[d] *= __ldg(M.rmlump_h + ff[d]);
            }
            // flux through the faces below and above (none through surface and lid)
            auto flux = [&](int k) {
                if (k <= 0 || k >= M.nlev) return 0.0;
                const size_t o = (size_t)k * ncol + c;
                return MODE == MX_RHS ? __ldg(uv + o) * __ldg(M.rmlump + o) : __ldg(uv + o);
            };
            double below = flux(k0);
#pragma unroll 2
            for (int k = k0; k < k1; ++k) {
                const double* ul = u + (size_t)k * nfh;
                const size_t o = (size_t)k * ncol + c;
                const double above = flux(k + 1);
                double y = __ldg(p + o);
#pragma unroll
                for (int d = 0; d < 4; ++d) y = fma(MODE == MX_RHS ? -sd[d] : sd[d], __ldg(ul + ff[d]), y);
                y = fma(MODE == MX_RHS ? -__ldg(M.divv + k) : __ldg(M.divv + k), above - below, y);
                put(yp + o, nu + o, y);
                below = above;
            }
        }
    }
    if constexpr (J >= 0) {
        if (grid_reduce<NV>(v, partials, ticket, t)) gcr_coeffs<JJ>(t, S);
    }
}

}  // namespace mg
