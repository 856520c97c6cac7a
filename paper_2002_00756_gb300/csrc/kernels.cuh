// Device kernels of the column multigrid solver (sm_103a).
//
// Layout: cell fields are level-major f[k * ncol + col], so the threads of a warp, one
// column each, read consecutive words at every level k.  Coefficients are stored in
// face form (see mesh.h): Th[k][face] for horizontal faces, Tv[kf][col] for vertical
// faces, with 1/area per column and 1/dz per level supplying the volume normalisation.
// The V-cycle's sweeps and restrictions have level data of their own: sweep32.cuh and
// sweep64.cuh.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace mg {

template <typename T, typename C>
struct Lvl {
    int n, ncol, nlev;
    const int32_t* nbr;   // [4][ncol]
    const int32_t* fof;   // [4][ncol]
    const C* Th;          // [nlev][2 ncol]
    const C* Tv;          // [nlev+1][ncol], rows 0 and nlev are zero
    const T* rA;          // [ncol] 1 / area
    const T* rdz;         // [nlev] 1 / dz
};

template <typename T, typename C>
__device__ __forceinline__ T ldc(const C* p) {
    return (T)__ldg(p);
}
template <>
__device__ __forceinline__ float ldc<float, __nv_bfloat16>(const __nv_bfloat16* p) {
    return __bfloat162float(__ldg(p));
}

template <typename T, typename X>
__device__ __forceinline__ T ldx(const X* p) {
    return (T)__ldg(p);
}

// 1 / p: FP32 reciprocal and one cubic step (r = 1 - p y: y + y r + y r^2, relative error r^3 < 2^-66
// before rounding), 4 FP64 operations instead of a division's dozen; values outside FP32's range are
// divided.
__device__ __forceinline__ double recip64(double p) {
    if (!(p > 1e-30 && p < 1e30)) return 1.0 / p;
    const double y = (double)(1.0f / (float)p), r = fma(-p, y, 1.0);
    return fma(fma(r, r, r), y, y);
}

__device__ __forceinline__ int parent_col(int col, int n) {
    const int nn = n * n, p = col / nn, r = col - p * nn, j = r / n, i = r - j * n, nc = n >> 1;
    return p * nc * nc + (j >> 1) * nc + (i >> 1);
}

__device__ __forceinline__ int child_col_dev(int n_fine, int C, int q) {
    const int nc = n_fine >> 1, ncc = nc * nc;
    const int p = C / ncc, r = C - p * ncc, J = r / nc, I = r - J * nc;
    return p * n_fine * n_fine + (2 * J + (q >> 1)) * n_fine + 2 * I + (q & 1);
}

// Source of the current iterate x on the fine level of a kernel:
//   XM_PLAIN    x[k][col]
//   XM_ZERO     0 (the first sweep of a level)
//   XM_PROLONG  x[k][col] + xc[k][parent(col)]   (prolongation fused into the sweep)
//   XM_PROLONG0 xc[k][parent(col)]               (prolongation onto a zero iterate)
enum { XM_PLAIN = 0, XM_ZERO = 1, XM_PROLONG = 2, XM_PROLONG0 = 3 };

// ---------------------------------------------------------------------------------------
// y = H x (Eq. helmholtz_operator): one thread per column, levels [k0, k0 + kchunk).
template <typename T, typename C, typename X, typename Y>
__global__ void __launch_bounds__(256) k_apply(Lvl<T, C> L, const X* __restrict__ x,
                                               Y* __restrict__ y, int kchunk) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= L.ncol) return;
    const size_t ncol = L.ncol, nf = 2 * ncol;
    const int k0 = blockIdx.y * kchunk;
    const int k1 = min(L.nlev, k0 + kchunk);
    int nb[4], fo[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        nb[s] = __ldg(L.nbr + s * ncol + c);
        fo[s] = __ldg(L.fof + s * ncol + c);
    }
    const T rA = __ldg(L.rA + c);
    T xm = k0 > 0 ? ldx<T>(x + (size_t)(k0 - 1) * ncol + c) : T(0);
    T x0 = ldx<T>(x + (size_t)k0 * ncol + c);
    T tdn = ldc<T>(L.Tv + (size_t)k0 * ncol + c);
    for (int k = k0; k < k1; ++k) {
        const size_t o = (size_t)k * ncol;
        const T xp = (k + 1 < L.nlev) ? ldx<T>(x + o + ncol + c) : T(0);
        const T tup = ldc<T>(L.Tv + o + ncol + c);
        const C* th = L.Th + (size_t)k * nf;
        T h = ldc<T>(th + fo[0]) * (x0 - ldx<T>(x + o + nb[0]));
        h += ldc<T>(th + fo[1]) * (x0 - ldx<T>(x + o + nb[1]));
        h += ldc<T>(th + fo[2]) * (x0 - ldx<T>(x + o + nb[2]));
        h += ldc<T>(th + fo[3]) * (x0 - ldx<T>(x + o + nb[3]));
        const T v = __ldg(L.rdz + k) * (tup * (x0 - xp) + tdn * (x0 - xm));
        y[o + c] = (Y)(x0 + (rA * h + v));
        xm = x0;
        x0 = xp;
        tdn = tup;
    }
}

// x_out[k][c] = (ZB ? 0 : x[k][c]) + xc[k][parent(c)]  (Eq. prolongation, natural injection)
template <typename T, bool ZB, typename X, typename O>
__global__ void k_prolong(int n, int ncol, int ncol_c, int nlev, const X* __restrict__ x,
                          const T* __restrict__ xc, O* __restrict__ xo) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncol) return;
    const int pc = parent_col(c, n);
    for (int k = 0; k < nlev; ++k) {
        const size_t o = (size_t)k * ncol;
        T v = __ldg(xc + (size_t)k * ncol_c + pc);
        if (!ZB) v += ldx<T>(x + o + c);
        xo[o + c] = (O)v;
    }
}

// ---------------------------------------------------------------------------------------
// The 9-cell stencil (Sec. 3.5, Fig. 2): H also couples every cell to the cells two levels
// above and below, through the fluxes T2[k][c] (k <-> k+2; rows nlev-2 and nlev-1 are zero):
// b_up(k) = T2[k] / dz_k, b_dn(k) = T2[k-2] / dz_k.  These kernels run one thread per cell or
// per column without staging: the 9-cell stencil is the paper's comparison configuration,
// not the headline path.
template <typename T, typename X>
__device__ __forceinline__ T h9_cell(const Lvl<T, T>& L, const T* __restrict__ T2, const X* __restrict__ x, int k,
                                     int c) {
    const size_t ncol = L.ncol, o = (size_t)k * ncol;
    const T x0 = ldx<T>(x + o + c);
    const T* th = L.Th + (size_t)k * 2 * ncol;
    T h = T(0);
#pragma unroll
    for (int s = 0; s < 4; ++s) h += __ldg(th + __ldg(L.fof + s * ncol + c)) * (x0 - ldx<T>(x + o + __ldg(L.nbr + s * ncol + c)));
    T v = T(0);
    if (k + 1 < L.nlev) v += __ldg(L.Tv + o + ncol + c) * (x0 - ldx<T>(x + o + ncol + c));
    if (k > 0) v += __ldg(L.Tv + o + c) * (x0 - ldx<T>(x + o - ncol + c));
    if (k + 2 < L.nlev) v += __ldg(T2 + o + c) * (x0 - ldx<T>(x + o + 2 * ncol + c));
    if (k > 1) v += __ldg(T2 + o - 2 * ncol + c) * (x0 - ldx<T>(x + o - 2 * ncol + c));
    return x0 + (__ldg(L.rA + c) * h + __ldg(L.rdz + k) * v);
}

// y = H x (9-cell stencil), one thread per cell
template <typename T, typename X, typename Y>
__global__ void k_apply9(Lvl<T, T> L, const T* __restrict__ T2, const X* __restrict__ x, Y* __restrict__ y) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (c >= L.ncol || k >= L.nlev) return;
    y[(size_t)k * L.ncol + c] = (Y)h9_cell<T, X>(L, T2, x, k, c);
}

// r = b - H x (9-cell stencil; x == NULL: r = b), one thread per cell
template <typename T, typename B>
__global__ void k_resid9(Lvl<T, T> L, const T* __restrict__ T2, const T* __restrict__ x, const B* __restrict__ b,
                         T* __restrict__ r) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (c >= L.ncol || k >= L.nlev) return;
    const size_t e = (size_t)k * L.ncol + c;
    r[e] = x ? (T)b[e] - h9_cell<T, T>(L, T2, x, k, c) : (T)b[e];
}

// x_out = x + omega Hz^-1 r per column (x == NULL: zero iterate), Hz the tridiagonal column
// matrix of the nearest couplings (the next-to-nearest fluxes dropped, Sec. 3.6), solved by
// the pivot-excess Thomas recurrence; sw, se hold its y / p and a_up / p per cell
template <typename T, typename O>
__global__ void k_thomas9(Lvl<T, T> L, const T* __restrict__ r, const T* __restrict__ x, T* __restrict__ sw,
                          T* __restrict__ se, O* __restrict__ xo, T omega) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= L.ncol) return;
    const size_t ncol = L.ncol;
    const T rA = __ldg(L.rA + c);
    T q = T(0), p = T(1), y = T(0);
    for (int k = 0; k < L.nlev; ++k) {
        const size_t o = (size_t)k * ncol, e = o + c;
        const T* thk = L.Th + (size_t)k * 2 * ncol;
        T sh = T(0);
#pragma unroll
        for (int s = 0; s < 4; ++s) sh += __ldg(thk + __ldg(L.fof + s * ncol + c));
        const T rdz = __ldg(L.rdz + k);
        const T adn = k > 0 ? rdz * __ldg(L.Tv + e) : T(0);
        const T aup = k + 1 < L.nlev ? rdz * __ldg(L.Tv + e + ncol) : T(0);
        const T m = k > 0 ? adn / p : T(0);
        q = (T(1) + rA * sh) + m * q;
        p = q + aup;
        y = r[e] + m * y;
        sw[e] = y / p;
        se[e] = aup / p;
    }
    T d = T(0);
    for (int k = L.nlev - 1; k >= 0; --k) {
        const size_t e = (size_t)k * ncol + c;
        d = sw[e] + se[e] * d;
        xo[e] = (O)((x ? x[e] : T(0)) + omega * d);
    }
}

// bc[k][C] = sum_q w[q][C] r[k][child_q] (restriction of a residual already formed)
template <typename T, typename O>
__global__ void k_restrict_sum(int n, int ncol, int nlev, const T* __restrict__ r, const T* __restrict__ w,
                               O* __restrict__ bc, int ncol_c) {
    const int C = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (C >= ncol_c || k >= nlev) return;
    T acc = T(0);
#pragma unroll
    for (int q = 0; q < 4; ++q) acc += __ldg(w + (size_t)q * ncol_c + C) * r[(size_t)k * ncol + child_col_dev(n, C, q)];
    bc[(size_t)k * ncol_c + C] = (O)acc;
}

template <typename A, typename B>
__global__ void k_convert(size_t n, const A* __restrict__ a, B* __restrict__ b) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        b[i] = (B)a[i];
}

}  // namespace mg
