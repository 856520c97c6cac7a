// Block-Jacobi column sweep and residual + restriction in FP64 (the FP64 V-cycle, mg_smooth,
// mg_residual_restrict), bound by the FP64 pipe (two lanes per clock and SM on GB300).
//
// Packed level data, plain [levels][ncol]: every horizontal coupling sits under the cell on whose
// east / north side it lies, the west / south faces of a panel's first column / row, which no cell
// of the panel has on its east / north side, are two short extra rows.  Everything is weighted by the
// cell volume V = area dz (times one power of two for the whole hierarchy, so that V is about 1): the
// weighted operator is symmetric, one number serves both cells of a face, restriction is a plain sum,
// and the column matrix V Hz factors as L D L^T with the SAME multipliers e forwards and backwards:
//     Q_k = V_k + sum of the horizontal couplings + e_{k-1} Q_{k-1},  P_k = Q_k + tv_{k+1},
//     ip_k = 1 / P_k,  e_k = tv_{k+1} / P_k       (every term positive: no cancellation)
//     y_k = f_k + e_{k-1} y_{k-1},   d_k = ip_k y_k + e_k d_{k+1}.
// The factors depend on the couplings alone, so they are computed once, when the couplings are set,
// not in every sweep: about 14 FP64 operations per cell and sweep instead of about 35 (division).
#pragma once

#include "kernels.cuh"

namespace mg {

struct Lvl64 {
    int n, ncol, nlev;
    const int32_t* nbr;   // [4][ncol] neighbour columns E, W, N, S
    const int32_t* par;   // [5][ncol] coarse parent of the neighbours E, W, N, S and of the column
    const double* te;     // [nlev][ncol] east face
    const double* tn;     // [nlev][ncol] north face
    const double* tbw;    // [nlev][6 n] west face of each panel's first column, by (panel, j)
    const double* tbs;    // [nlev][6 n] south face of each panel's first row, by (panel, i)
    const double* tv;     // [nlev + 1][ncol] vertical faces, rows 0 and nlev zero
    const double* e;      // [nlev][ncol] factors; ip times om0
    const double* ip;
    const double* pr;     // [chunks][ncol] product of e over each chunk of 10 levels, where sweeps use those
    const double* wA;     // [ncol] area x scale
    const double* dz;     // [nlev] layer depth
    double om0;           // relaxation factor that ip holds
};

// v = *p where `on`, else v unchanged: a predicated load, not a branch.  A branch around the few
// lanes that load a neighbour (ends of a warp's columns, panel edges) would keep the compiler from
// issuing the loads that follow before this one has returned (finest restriction at C192L70 in
// this form: 97 us instead of 122).
__device__ __forceinline__ void ldp(double& v, const double* p, bool on) {
    asm("{\n .reg .pred q;\n setp.ne.s32 q, %2, 0;\n @q ld.global.nc.f64 %0, [%1];\n}" : "+d"(v) : "l"(p), "r"((int)on));
}

// Levels per chunk: 10, where two blocks fit on an SM, 5 below 2M cells (twice the threads), 16 for
// columns of more than 80 levels; and the chunks of a column, W.
inline int sweep64_levels(int nlev, int ncol) { return nlev > 80 ? 16 : (double)nlev * ncol < 2e6 ? 5 : 10; }
inline int sweep64_chunks(int nlev, int ncol) {
    const int K = sweep64_levels(nlev, ncol);
    return (nlev + K - 1) / K;
}

__host__ __device__ constexpr int sweep64_warps(int K) { return ((K < 16 ? 80 : 128) + K - 1) / K; }

// One sweep x_out = x + omega Hz^{-1} (b - H x) in direct form: with H = Hz - (horizontal
// off-diagonals),
//     x_out = (1 - omega) x + omega Hz^{-1} (b + sum_faces a_f x_neighbour),
// so a sweep needs neither the vertical couplings nor the vertical neighbours of x, and a sweep
// from zero (MODE XM_ZERO) reads b and the two factors only.
//
// W warps share 32 consecutive columns; warp w owns the levels [w nlev / W, (w + 1) nlev / W), at
// most K, and holds them in registers.  The two recurrences run per chunk from a zero inflow, the
// chunks' (outflow, product of e) pairs are folded in order by every warp, outflows exchanged through
// shared memory, and a second pass applies the true inflow.  The FP64 pipe bounds it: chunks of 10 read
// their products, and ip holds omega already (10.9 operations per cell of a plain sweep, 7.9 of a first one
// instead of 12.9 and 9.9): plain 121 -> 104 us at C96L70, first 84 -> 74, with the prolongation 160 -> 156.
// Chunks of 5 (small levels) multiply their products up: reading 16 of them costs more latency than the
// operations saved (C12L30 solve 364 us against 347).
//
// BRAW: b is unweighted and weighted here (and, with BCOPY, stored for the later sweeps of the level).
template <int MODE, bool BRAW, bool BCOPY, int K>
__global__ void __launch_bounds__(32 * sweep64_warps(K), K == 10 ? 2 : 1)
    k_sweep64(Lvl64 L, const double* __restrict__ x, const double* __restrict__ xc, int ncol_c,
              const double* __restrict__ b, double* __restrict__ bcopy, double* __restrict__ xo, double omega) {
    constexpr bool PRO = (MODE == XM_PROLONG || MODE == XM_PROLONG0);
    constexpr bool RAW = (MODE == XM_PLAIN || MODE == XM_PROLONG);   // reads the fine iterate
    constexpr bool ZERO = MODE == XM_ZERO;
    constexpr int WMAX = sweep64_warps(K);
    constexpr bool STORED = K == 10;   // the chunks' products of e are read, not multiplied up
    __shared__ double s_[STORED ? 2 : 3][WMAX][32];   // outflow upwards, downwards, product of e
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, W = blockDim.x >> 5;
    const unsigned ncol = L.ncol, n = L.n;
    const unsigned c_raw = blockIdx.x * 32 + lane;
    const bool active = c_raw < ncol;
    const unsigned c = active ? c_raw : ncol - 1;
    const int k0 = w * L.nlev / W, k1 = (w + 1) * L.nlev / W;

    // neighbour columns; E / W come from the adjacent lanes where those hold them
    unsigned nE = 0, nW = 0, nN = 0, nS = 0, sW = 0, sS = 0, gE = 0, gW = 0, gN = 0, gS = 0, gC = 0;
    bool shE = false, shW = false;
    const double *ptw = nullptr, *pts = nullptr;
    if constexpr (!ZERO) {
        const unsigned row = c / n, i = c - row * n, p = row / n, j = row - p * n;
        shE = i + 1 < n && lane != 31;
        shW = i > 0 && lane != 0;
        nE = __ldg(L.nbr + c);
        nW = __ldg(L.nbr + ncol + c);
        nN = __ldg(L.nbr + 2 * ncol + c);
        nS = __ldg(L.nbr + 3 * ncol + c);
        ptw = i > 0 ? L.te + c - 1 : L.tbw + row;
        sW = i > 0 ? ncol : 6 * n;
        pts = j > 0 ? L.tn + c - n : L.tbs + p * n + i;
        sS = j > 0 ? ncol : 6 * n;
        if (PRO) {
            gE = __ldg(L.par + c);
            gW = __ldg(L.par + ncol + c);
            gN = __ldg(L.par + 2 * ncol + c);
            gS = __ldg(L.par + 3 * ncol + c);
            gC = __ldg(L.par + 4 * ncol + c);
        }
    }
    const double wA = BRAW ? __ldg(L.wA + c) : 0.0;

    double f[K], e[K], ip[K], x0[K];
#pragma unroll
    for (int q = 0; q < K; ++q) {
        const bool in = k0 + q < k1;
        const unsigned k = in ? k0 + q : k1 - 1, o = k * ncol, oc = k * (unsigned)ncol_c;
        double fb = __ldg(b + (o + c));
        e[q] = __ldg(L.e + (o + c));
        ip[q] = __ldg(L.ip + (o + c));
        if (BRAW) {
            fb *= wA * __ldg(L.dz + k);
            if (BCOPY && in && active) bcopy[o + c] = fb;
        }
        if constexpr (!ZERO) {
            const double te = __ldg(L.te + (o + c)), tn = __ldg(L.tn + (o + c)), ts = __ldg(pts + (size_t)(k * sS));
            double tw = 0.0, xm = 0.0, xE = 0.0, xW = 0.0, xN = 0.0, xS = 0.0;
            ldp(tw, ptw + (size_t)(k * sW), !shW);
            if (RAW) {
                xm = __ldg(x + (o + c));
                xN = __ldg(x + (o + nN));
                xS = __ldg(x + (o + nS));
                ldp(xE, x + (o + nE), !shE);
                ldp(xW, x + (o + nW), !shW);
            }
            if (PRO) {
                double cE = 0.0, cW = 0.0;
                ldp(cE, xc + (oc + gE), !shE);
                ldp(cW, xc + (oc + gW), !shW);
                xm += __ldg(xc + (oc + gC));
                xN += __ldg(xc + (oc + gN));
                xS += __ldg(xc + (oc + gS));
                xE += cE;
                xW += cW;
            }
            const double xEl = __shfl_down_sync(0xffffffffu, xm, 1), xWl = __shfl_up_sync(0xffffffffu, xm, 1);
            const double twl = __shfl_up_sync(0xffffffffu, te, 1);
            if (shE) xE = xEl;
            if (shW) {
                xW = xWl;
                tw = twl;
            }
            fb = fma(tw, xW, fb);
            fb = fma(te, xE, fb);
            fb = fma(tn, xN, fb);
            fb = fma(ts, xS, fb);
            x0[q] = xm;
        }
        f[q] = in ? fb : 0.0;   // levels past the chunk's end pass their inflow through
        if (!in) {
            e[q] = 1.0;
            ip[q] = 0.0;
        }
    }
    // forwards: outflow e y of the chunk from zero inflow, fold, then y with the true inflow
    double pr[WMAX];   // every chunk's product of e, for both directions
    if (W > 1) {
        if constexpr (STORED) {
#pragma unroll
            for (int u = 0; u < WMAX; ++u)
                if (u < W) pr[u] = __ldg(L.pr + ((unsigned)u * ncol + c));
        }
        double y = f[0], g = e[0];
#pragma unroll
        for (int q = 1; q < K; ++q) {
            y = fma(e[q - 1], y, f[q]);
            if (!STORED) g *= e[q];
        }
        s_[0][w][lane] = e[K - 1] * y;
        if constexpr (!STORED) s_[2][w][lane] = g;
        __syncthreads();
        double in = 0.0;
#pragma unroll
        for (int u = 0; u < WMAX; ++u)
            if (u < W) {
                if constexpr (!STORED) pr[u] = s_[2][u][lane];
                if (u < w) in = fma(pr[u], in, s_[0][u][lane]);
            }
        f[0] += in;
    }
#pragma unroll
    for (int q = 1; q < K; ++q) f[q] = fma(e[q - 1], f[q - 1], f[q]);
#pragma unroll
    for (int q = 0; q < K; ++q) f[q] *= ip[q];
    if (omega != L.om0) {   // (a pressure solver with a relaxation factor of its own)
        const double scale = omega / L.om0;
#pragma unroll
        for (int q = 0; q < K; ++q) f[q] *= scale;
    }
    // backwards: the chunk's lowest value from zero inflow, fold, then d (times omega) and the update
    double d = 0.0;
    if (W > 1) {
        double g = f[K - 1];
#pragma unroll
        for (int q = K - 2; q >= 0; --q) g = fma(e[q], g, f[q]);
        s_[1][w][lane] = g;
        __syncthreads();
#pragma unroll
        for (int u = WMAX - 1; u >= 0; --u)
            if (u > w && u < W) d = fma(pr[u], d, s_[1][u][lane]);
    }
    const double om1 = 1.0 - omega;
#pragma unroll
    for (int q = K - 1; q >= 0; --q) {
        d = fma(e[q], d, f[q]);
        if (active && k0 + q < k1)
            xo[(unsigned)(k0 + q) * ncol + c] = ZERO ? d : fma(om1, x0[q], d);
    }
}

// ---------------------------------------------------------------------------------------
// Residual and restriction (Algorithm 1) in weighted form: the weighted residual of a coarse cell
// is the plain sum over its four children, in which the fluxes through the four faces inside
// the coarse cell cancel, so only its eight outer horizontal faces are read (37 FP64 operations per
// coarse cell instead of 60).  One thread per coarse column (2 x 2 fine columns, read 2 wide with
// VEC) and kchunk levels; the vertical flux through a level's upper face is carried to the next
// level.  E / W neighbours and the W faces come from the adjacent lanes.
//   RAW: b unweighted and the result divided by the coarse volume (wAc dz).
template <bool XZERO, bool RAW, bool VEC>
__global__ void __launch_bounds__(128) k_restrict64(Lvl64 L, const double* __restrict__ x, const double* __restrict__ b,
                                                    const double* __restrict__ wAc, double* __restrict__ bc, int ncol_c,
                                                    int kchunk) {
    const unsigned ncol = L.ncol, n = L.n, nc = n >> 1;
    const unsigned C_raw = blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const bool active = C_raw < (unsigned)ncol_c;
    const unsigned Cc = active ? C_raw : ncol_c - 1;
    const unsigned p = Cc / (nc * nc), rem = Cc - p * nc * nc, J = rem / nc, I = rem - J * nc;
    const unsigned c[2] = {p * n * n + 2 * J * n + 2 * I, p * n * n + (2 * J + 1) * n + 2 * I};
    const int k0 = blockIdx.y * kchunk, k1 = min(L.nlev, k0 + kchunk);
    auto own2 = [](const double* q, double(&v)[2]) {   // (the handle's arrays)
        const double2 t = __ldg(reinterpret_cast<const double2*>(q));
        v[0] = t.x;
        v[1] = t.y;
    };
    auto ld2 = [&](const double* q, double(&v)[2]) {   // (the caller's, or the handle's)
        if constexpr (VEC) {
            own2(q, v);
        } else {
            v[0] = __ldg(q);
            v[1] = __ldg(q + 1);
        }
    };
    double wA[2][2];
    own2(L.wA + c[0], wA[0]);
    own2(L.wA + c[1], wA[1]);
    const bool shE = I + 1 < nc && lane != 31, shW = I > 0 && lane != 0;
    unsigned nE[2], nW[2], nN[2], nS[2];
    const double* ptw[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        nE[r] = __ldg(L.nbr + c[r] + 1);
        nW[r] = __ldg(L.nbr + ncol + c[r]);
        nN[r] = __ldg(L.nbr + 2 * ncol + c[1] + r);
        nS[r] = __ldg(L.nbr + 3 * ncol + c[0] + r);
        ptw[r] = I > 0 ? L.te + c[r] - 1 : L.tbw + p * n + 2 * J + r;
    }
    const double* pts = J > 0 ? L.tn + c[0] - n : L.tbs + p * n + 2 * I;
    const unsigned sW = I > 0 ? ncol : 6 * n, sS = J > 0 ? ncol : 6 * n;
    const double cw = (active && RAW) ? __ldg(wAc + Cc) : 1.0;
    // weighted flux sum through the faces between levels k and k + 1 (upwards)
    auto vflux = [&](unsigned ov, const double(&lo)[2][2], const double(&hi)[2][2]) -> double {
        double s = 0.0;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            double tv[2];
            own2(L.tv + (ov + c[r]), tv);
#pragma unroll
            for (int v = 0; v < 2; ++v) s = fma(tv[v], lo[r][v] - hi[r][v], s);
        }
        return s;
    };
    double x0[2][2] = {{0.0, 0.0}, {0.0, 0.0}}, xp[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
    double below = 0.0;
    if (!XZERO) {
#pragma unroll
        for (int r = 0; r < 2; ++r) ld2(x + ((unsigned)k0 * ncol + c[r]), x0[r]);
        if (k0 > 0) {
            double xm[2][2];
#pragma unroll
            for (int r = 0; r < 2; ++r) ld2(x + ((unsigned)(k0 - 1) * ncol + c[r]), xm[r]);
            below = vflux((unsigned)k0 * ncol, xm, x0);
        }
    }
#pragma unroll 2
    for (int k = k0; k < k1; ++k) {
        const unsigned o = (unsigned)k * ncol;
        const double dz = __ldg(L.dz + k);
        double bb[2][2], s = 0.0;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            ld2(b + (o + c[r]), bb[r]);
#pragma unroll
            for (int v = 0; v < 2; ++v) s = RAW ? fma(wA[r][v], bb[r][v], s) : s + bb[r][v];
        }
        if (RAW) s *= dz;
        if (!XZERO) {
            double te[2], tn[2], ts[2], xE[2] = {0.0, 0.0}, xW[2] = {0.0, 0.0}, tw[2] = {0.0, 0.0}, xN[2], xS[2];
            if (k + 1 < L.nlev) {
#pragma unroll
                for (int r = 0; r < 2; ++r) ld2(x + (o + ncol + c[r]), xp[r]);
            }
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                te[r] = __ldg(L.te + (o + c[r] + 1));
                ldp(xE[r], x + (o + nE[r]), !shE);
                ldp(xW[r], x + (o + nW[r]), !shW);
                ldp(tw[r], ptw[r] + (size_t)(k * sW), !shW);
                xN[r] = __ldg(x + (o + nN[r]));
                xS[r] = __ldg(x + (o + nS[r]));
            }
            own2(L.tn + (o + c[1]), tn);
            own2(pts + (size_t)(k * sS), ts);
            double h = 0.0, m = 0.0;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const double e1 = __shfl_down_sync(0xffffffffu, x0[r][0], 1);
                const double w1 = __shfl_up_sync(0xffffffffu, x0[r][1], 1);
                const double t1 = __shfl_up_sync(0xffffffffu, te[r], 1);
                if (shE) xE[r] = e1;
                if (shW) {
                    xW[r] = w1;
                    tw[r] = t1;
                }
                h = fma(te[r], x0[r][1] - xE[r], h);
                h = fma(tw[r], x0[r][0] - xW[r], h);
                h = fma(tn[r], x0[1][r] - xN[r], h);   // (r runs over the two columns here)
                h = fma(ts[r], x0[0][r] - xS[r], h);
                m = fma(wA[r][0], x0[r][0], m);
                m = fma(wA[r][1], x0[r][1], m);
            }
            const double above = vflux(o + ncol, x0, xp);
            s -= fma(dz, m, h + (above - below));
            below = above;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                x0[r][0] = xp[r][0];
                x0[r][1] = xp[r][1];
            }
        }
        if (active) bc[(size_t)k * ncol_c + Cc] = RAW ? s / (cw * dz) : s;
    }
}

// ---------------------------------------------------------------------------------------
// Packed level data from the face form (Th [nlev][2 ncol], Tv [nlev + 1][ncol]).  One thread per
// column and level (tv: rows 0 .. nlev).
__global__ void k_pack64(int n, int ncol, int nlev, const int32_t* __restrict__ fof, const double* __restrict__ Th,
                         const double* __restrict__ Tv, const double* __restrict__ wA, const double* __restrict__ dz,
                         double scale, double* __restrict__ te, double* __restrict__ tn, double* __restrict__ tbw,
                         double* __restrict__ tbs, double* __restrict__ tv, double* __restrict__ diag) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (c >= ncol) return;
    const size_t e = (size_t)k * ncol + c;
    tv[e] = Tv[e] * wA[c];
    if (k >= nlev) return;
    const double wt = dz[k] * scale;
    const double* t = Th + (size_t)k * 2 * ncol;
    const double E = t[__ldg(fof + c)] * wt, W = t[__ldg(fof + ncol + c)] * wt;
    const double Nn = t[__ldg(fof + 2 * ncol + c)] * wt, S = t[__ldg(fof + 3 * ncol + c)] * wt;
    te[e] = E;
    tn[e] = Nn;
    diag[e] = fma(wA[c], dz[k], (E + W) + (Nn + S));
    const int row = c / n, i = c - row * n, p = row / n, j = row - p * n;
    if (i == 0) tbw[(size_t)k * 6 * n + row] = W;
    if (j == 0) tbs[(size_t)k * 6 * n + p * n + i] = S;
}

// The factors e, ip of every column from its diagonals (in ip_, k_pack64); one thread per column.  The
// pivots are one dependent chain; the next BATCH levels' operands are under way while a batch is
// eliminated (level of C12L70 95 -> 32 us, C96L70 132 -> 97; the FP64 pipe's bound there: 74).
__global__ void k_factor64(int ncol, int nlev, const double* __restrict__ tv, double* __restrict__ e_, double* ip_,
                           double* __restrict__ pr, int chunks, double om0) {
    constexpr int BATCH = 8;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncol) return;
    double Q = 0.0, e = 0.0, g = 1.0, D[BATCH], T[BATCH], Dn[BATCH], Tn[BATCH];
    auto load = [&](int k0, double (&dd)[BATCH], double (&tt)[BATCH]) {
#pragma unroll
        for (int q = 0; q < BATCH; ++q) {
            const size_t o = (size_t)min(k0 + q, nlev - 1) * ncol + c;
            dd[q] = ip_[o];
            tt[q] = __ldg(tv + o + ncol);
        }
    };
    load(0, Dn, Tn);
    int w = 0, end = nlev / chunks;
    for (int k0 = 0; k0 < nlev; k0 += BATCH) {
#pragma unroll
        for (int q = 0; q < BATCH; ++q) D[q] = Dn[q], T[q] = Tn[q];
        if (k0 + BATCH < nlev) load(k0 + BATCH, Dn, Tn);
#pragma unroll
        for (int q = 0; q < BATCH; ++q) {
            const int k = k0 + q;
            if (k < nlev) {
                const size_t o = (size_t)k * ncol + c;
                Q = fma(e, Q, D[q]);
                const double ip = recip64(Q + T[q]);
                e = T[q] * ip;
                e_[o] = e;
                ip_[o] = om0 * ip;
                if (pr) {
                    g *= e;
                    if (k + 1 == end) {
                        pr[(size_t)w++ * ncol + c] = g;
                        g = 1.0;
                        end = (w + 1) * nlev / chunks;
                    }
                }
            }
        }
    }
}

// V b of an unweighted right-hand side (a level that starts without a sweep)
__global__ void k_weight64(int ncol, const double* __restrict__ b, const double* __restrict__ wA,
                           const double* __restrict__ dz, double* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (c >= ncol) return;
    const size_t o = (size_t)k * ncol + c;
    out[o] = b[o] * (__ldg(wA + c) * __ldg(dz + k));
}

}  // namespace mg
