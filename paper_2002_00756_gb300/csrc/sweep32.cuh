// Block-Jacobi column sweep and residual + restriction of the FP32 V-cycle.
//
// Layout ("padded"): FP32 fields -- iterates, right-hand sides, couplings, reciprocal pivots -- are
// stored with a rim of one cell around every panel that holds the neighbours' values across its
// edges: [levels][6 panels][n + 2 rows][np], cell (p, j, i) at padded column
// ((n + 2) p + j + 1) np + off + i (pad_row, pad_off).  The four neighbours of every cell are then
// at +-1 and +-np, with no connectivity to read and no special case at a panel's edge; whoever
// writes an iterate also writes its edge columns into the rims they belong to (table hd).  Every
// horizontal coupling sits under the cell on whose east / north side it lies (te, tn; the rims hold
// the west and south faces of a panel's first column and row).
//
// Arithmetic: two walks per column eliminate its tridiagonal system from both ends (a twisted
// factorisation), the lower half of its levels upwards, the upper half downwards.  With the coupling
// to the eliminated neighbour a_prev and to the next one a_next, step by step
//     m = a_prev / p_prev,  q = s + m q_prev,  p = q + a_next,  y = r + m y_prev
// (s = 1 + horizontal coefficients: pivots are sums of positive terms).  The halves meet in
//     [p_A  -a_A] [d_A]   [y_A]
//     [-a_B  p_B] [d_B] = [y_B],   det = q_A p_B + a_A q_B  (no cancellation)
// and the back substitution runs directly on the output,
//     out_i = w_i + e_i out_{i+1},  w_i = x_i + omega y_i / p_i - e_i x_{i+1},  e_i = a_next / p_i.
// The pivots depend on the couplings alone: their reciprocals are computed once, by the same
// recurrence in the same precision, when the couplings are set (k_factor32), so a sweep has neither
// the division nor the pivot chain of every step -- what bounded the walks before: 121 us per
// finest sweep at C192L70 with two threads per column, 16 warps per SM and 121 instructions per cell.
// What is left of the chain is one FMA per level, which is handed from chunk to chunk.
//
// The order of every rounding is fixed (explicit FMAs below).  The outer Krylov solve sees the FP32
// V-cycle's rounding noise multiplied by the vertical couplings (up to 1e-2 of H z at 70 levels), so
// another order would move every iterate of a solve by a few per cent of its error.
#pragma once

#include "kernels.cuh"

namespace mg {

// Columns before a field's first cell, and the length of a padded row: rows start on 128-byte lines, on
// 32-byte sectors on small meshes.  A row's east rim and the next row's west rim share the gap between
// them; tensor boxes reach beyond a row's end into the next row, for lanes that store nothing.
__host__ __device__ inline int pad_off(int n) { return n >= 48 ? 32 : 8; }
__host__ __device__ inline int pad_row(int n) { return n >= 48 ? (n + 2 + 31) / 32 * 32 : (n + 2 + 7) / 8 * 8; }
__host__ __device__ inline int padded(int n) { return 6 * (n + 2) * pad_row(n) + pad_off(n); }

// a column's position: panel, row and column in it, and its padded column
struct Pos {
    unsigned p, j, i, cp;
    __device__ __forceinline__ Pos(unsigned c, unsigned n, unsigned np) {
        const unsigned row = c / n;
        i = c - row * n;
        p = row / n;
        j = row - p * n;
        cp = (row + 2 * p + 1) * np + pad_off(n) + i;
    }
    // padded column, on the next coarser level, of the cell (dj, di) away's parent
    __device__ __forceinline__ unsigned parent(int dj, int di, unsigned n, unsigned npc) const {
        return ((n >> 1) + 2) * p * npc + (unsigned)((((int)j + dj) >> 1) + 1) * npc + pad_off(n >> 1) +
               (unsigned)(((int)i + di) >> 1);
    }
};

// FP32 level data.  C: couplings (FP32 or BF16); P: the column elimination (FP32, or FP64 on the
// finest level of MG_FP32_P64).  All padded but rA, rdz.
template <typename C, typename P>
struct Lvl32 {
    int n, ncol, nlev;
    int np, ncolp;        // padded row length, padded columns per level
    const int32_t* hd;    // [4][ncol] padded column of the rim cell that repeats this column across
                          // the panel edge on its side E, W, N, S; -1 where that side is no edge
    const C* te;          // east faces (rims: west faces of first columns)
    const C* tn;          // north faces (rims: south faces of first rows)
    const C* tv;          // [nlev + 1] vertical faces, rows 0 and nlev zero
    const P* ip;          // reciprocal pivots 1 / p; q at the last step of either half
    const P* m;           // P = double: the multipliers a_prev / p_prev and e = a_next / p
    const P* e;
    const float* rA;      // [ncol] 1 / area
    const float* rdz;     // [nlev] 1 / dz
};

__device__ __forceinline__ float mulr(float a, float b) { return __fmul_rn(a, b); }   // never fused
__device__ __forceinline__ double mulr(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fmad(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmad(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float addr(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float subr(float a, float b) { return __fsub_rn(a, b); }

// r = b - H x of one cell: couplings and iterates E, W, N, S; "ahead" and "behind" in the walk.  ALT:
// the rounding order of the restriction onto levels whose children are not summed in pairs.
template <bool ALT = false>
__device__ __forceinline__ float residual32(float b, float x0, float xE, float xW, float xN, float xS, float te,
                                            float tw, float tn, float ts, float rA, float rdz, float ta, float xa,
                                            float tb, float xb) {
    float h = fmad(te, subr(x0, xE), mulr(tw, subr(x0, xW)));
    h = fmad(tn, subr(x0, xN), h);
    h = fmad(ts, subr(x0, xS), h);
    if (ALT) {
        const float v = fmad(ta, subr(x0, xa), mulr(tb, subr(x0, xb)));
        return subr(b, addr(x0, fmad(rA, h, mulr(rdz, v))));
    }
    const float v = fmad(tb, subr(x0, xb), mulr(ta, subr(x0, xa)));
    return subr(b, addr(x0, fmad(rdz, v, mulr(rA, h))));
}

template <typename C>
__device__ __forceinline__ float ldf(const C* p) {
    return ldc<float, C>(p);
}

// d at the last steps of the halves, from this half's q, y, a_next there and the other's
template <typename P>
__device__ __forceinline__ P interface32(P q, P y, P a, P qo, P yo, P ao) {
    const P po = qo + ao;
    return fmad(a, yo, mulr(y, po)) / fmad(a, qo, mulr(q, po));
}

// The elimination of a chunk of up to K steps held in registers: multipliers, reciprocal pivots and
// e = a_next / p, then y, w and out in their place.  Only forward() and backward() are handed from
// chunk to chunk.
template <typename P, int K>
struct Chunk {
    float r[K], x[K + 1];   // right-hand side of the elimination; iterates of the steps and of the next one
    P m[K], ip[K], e[K];

    // y of every step (in place of m) from y before the chunk: the serial part, nothing else
    __device__ __forceinline__ P forward(P y, int len) {
#pragma unroll
        for (int q = 0; q < K; ++q)
            if (q < len) m[q] = y = fmad(m[q], y, P(r[q]));
        return y;
    }
    // w of every step in place of r
    __device__ __forceinline__ void stash(float omega) {
#pragma unroll
        for (int q = 0; q < K; ++q)
            r[q] = float(fmad(-e[q], P(x[q + 1]), fmad(P(omega), mulr(m[q], ip[q]), P(x[q]))));
    }
    // out of every step in place of w, from out behind it (`last`: the walk's last step holds it)
    __device__ __forceinline__ float backward(float out, bool last, int len) {
#pragma unroll
        for (int q = K - 1; q >= 0; --q)
            if (q < len) {
                if (!(last && q == len - 1)) out = fmad(float(e[q]), out, r[q]);
                r[q] = out;
            }
        return out;
    }
};

// ---------------------------------------------------------------------------------------
// Register sweep: small levels and short columns.  A block has 32 columns; its 2 G warps take the chunks of
// the two halves' walks, up to K steps each, and load them independently; the recurrence is then handed
// from warp to warp through shared memory and named barriers (one per pair of neighbouring chunks and half).
//   BRAW: b is the caller's FP64 array, its FP32 copy is stored in bcopy unless that is NULL.
//   xo: padded FP32 iterate, or the caller's FP64 array.
// (chunks of 8 for columns of more than 80 levels: at most 8 chunks a half, whose barriers are the
// block's 16)
__host__ __device__ constexpr int sweep32_warps(int K) { return K < 5 ? 2 : K == 8 ? 16 : 2 * ((40 + K - 1) / K); }

// Groups of 32 columns per block: short columns, whose halves are a warp each, take four (blocks of two warps
// start too slowly: FP32 V-cycle of C256L6 on three levels 250 -> 153 us, of C192L4 140 -> 112).
__host__ __device__ constexpr int sweep32_groups(int K) { return K < 5 ? 4 : 1; }

// Two warps meet: both wait, so that the two uses of a barrier (forwards, backwards) cannot mix; the
// receiving warp is there first as a rule.
__device__ __forceinline__ void pair_sync(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }

template <typename C, typename P, int MODE, typename B, typename O, bool BRAW, int K>
__global__ void __launch_bounds__(32 * sweep32_warps(K) * sweep32_groups(K), sizeof(P) == 4 && K == 8 && MODE == XM_ZERO ? 2 : 1)
    k_sweep32(Lvl32<C, P> L, const float* __restrict__ x, const float* __restrict__ xc, const B* __restrict__ b,
              float* __restrict__ bcopy, O* __restrict__ xo, float omega) {
    constexpr bool PRO = (MODE == XM_PROLONG || MODE == XM_PROLONG0);
    constexpr bool RAW = (MODE == XM_PLAIN || MODE == XM_PROLONG);   // reads the fine iterate
    constexpr bool ZERO = MODE == XM_ZERO, PADO = sizeof(O) == 4;
    __shared__ P sy[sweep32_warps(K)][32];   // handed-on y, then (halves' ends) the interface's values
    constexpr int M = sweep32_groups(K);
    __shared__ P si_[M][2][3][32];
    __shared__ float so[sweep32_warps(K)][32];   // handed-back out
    const int lane = threadIdx.x & 31, group = M > 1 ? threadIdx.x >> 6 : 0;
    const int w = (threadIdx.x >> 5) - 2 * group, G = M > 1 ? 1 : blockDim.x >> 6;
    P(&si)[2][3][32] = si_[group];
    const bool up = w >= G;   // the upper half, walked downwards
    const int u = up ? w - G : w;
    const int nlev = L.nlev, hs = (nlev + 1) >> 1, ns = up ? nlev - hs : hs;
    const unsigned ncol = L.ncol, n = L.n, np = L.np, ncolp = L.ncolp;
    const unsigned c_raw = (blockIdx.x * M + group) * 32 + lane;
    const bool active = c_raw < ncol;
    const unsigned c = active ? c_raw : ncol - 1;
    const int s0 = u * ns / G, len = (u + 1) * ns / G - s0;
    const Pos at(c, n, np);
    const float rA = __ldg(L.rA + c);
    // edge columns: the rim cells that repeat them across the E or W (rw) and the N or S edge (rn),
    // looked up here, long before the stores.  (C1, where a column has all four edges, is filled by
    // k_fill_rims instead.)
    int rw = -1, rn = -1;
    if (PADO && active) {
        if (at.i == 0) rw = __ldg(L.hd + ncol + c);
        else if (at.i + 1 == n) rw = __ldg(L.hd + c);
        if (at.j == 0) rn = __ldg(L.hd + 3 * ncol + c);
        else if (at.j + 1 == n) rn = __ldg(L.hd + 2 * ncol + c);
    }
    // the column's coarse parent, and those of its E / W and of its N / S neighbours, one of which is
    // the column's own
    unsigned gC = 0, gE = 0, gN = 0, lc = 0;
    if (PRO) {
        const unsigned npc = pad_row(n >> 1);
        gC = at.parent(0, 0, n, npc);
        gE = at.parent(0, (at.i & 1) ? 1 : -1, n, npc);
        gN = at.parent((at.j & 1) ? 1 : -1, 0, n, npc);
        lc = padded(n >> 1);
    }
    const bool oi = at.i & 1, oj = at.j & 1;
    auto level = [&](int s) { return (unsigned)(up ? nlev - 1 - s : s); };   // of step s of the walk
    // own iterate at step s, 0 beyond the column's ends
    auto own = [&](int s) -> float {
        if (ZERO) return 0.f;
        const int k = up ? nlev - 1 - s : s;
        const bool in = k >= 0 && k < nlev;
        const unsigned kk = in ? k : 0;
        float v = 0.f;
        if (RAW) v = __ldg(x + (kk * ncolp + at.cp));
        if (PRO) v += __ldg(xc + (kk * lc + gC));
        return in ? v : 0.f;
    };
    Chunk<P, K> q;
    {
        const int last = ns > 0 ? ns - 1 : 0;
        float xb = ZERO || s0 == 0 ? 0.f : own(s0 - 1), x0 = own(min(s0, last));
        const unsigned kf = level(min(s0, last));
        float tb = ldf(L.tv + ((up ? kf + 1 : kf) * ncolp + at.cp));
        P ipb = P(0);
        if (sizeof(P) == 4) ipb = s0 > 0 ? __ldg(L.ip + (level(s0 - 1) * ncolp + at.cp)) : P(0);
#pragma unroll
        for (int j = 0; j < K; ++j) {
            const int s = min(s0 + j, last);   // (steps past the chunk's end repeat the walk's last one, unused)
            const unsigned k = level(s), o = k * ncolp + at.cp;
            const float bk = BRAW ? (float)__ldg(b + (k * ncol + c)) : (float)__ldg(b + o);
            if (BRAW && bcopy && active && j < len) bcopy[o] = bk;
            const float ta = ldf(L.tv + ((up ? k : k + 1) * ncolp + at.cp)), rdz = __ldg(L.rdz + k);
            q.ip[j] = __ldg(L.ip + o);
            if constexpr (K == 1) {   // (a half's only step: nothing behind it, and out does not need e)
                q.m[j] = q.e[j] = P(0);
            } else if constexpr (sizeof(P) == 8) {
                q.m[j] = __ldg(L.m + o);
                q.e[j] = __ldg(L.e + o);
            } else {
                q.m[j] = mulr(mulr(rdz, tb), ipb);
                q.e[j] = mulr(mulr(rdz, ta), q.ip[j]);
                ipb = q.ip[j];
            }
            q.x[j] = x0;
            const float xa = own(s + 1);
            q.r[j] = bk;
            if constexpr (!ZERO) {
                const float te = ldf(L.te + o), tw = ldf(L.te + (o - 1)), tn = ldf(L.tn + o), ts = ldf(L.tn + (o - np));
                float xE = 0.f, xW = 0.f, xN = 0.f, xS = 0.f;
                if (RAW) {
                    xE = __ldg(x + (o + 1));
                    xW = __ldg(x + (o - 1));
                    xN = __ldg(x + (o + np));
                    xS = __ldg(x + (o - np));
                }
                if (PRO) {
                    const float* pc = xc + k * lc;
                    const float cm = __ldg(pc + gC), co = __ldg(pc + gE), ca = __ldg(pc + gN);
                    xE += oi ? co : cm;
                    xW += oi ? cm : co;
                    xN += oj ? ca : cm;
                    xS += oj ? cm : ca;
                }
                q.r[j] = residual32(bk, x0, xE, xW, xN, xS, te, tw, tn, ts, rA, rdz, ta, xa, tb, xb);
                xb = x0;
                x0 = xa;
            }
            tb = ta;
        }
        q.x[K] = ZERO ? 0.f : x0;
    }
    // forwards: y from the chunk before, w of every step
    const int bar = 1 + (up ? G - 1 : 0);   // barriers bar .. bar + G - 2 between the half's chunks
    P y = P(0);
    if (u > 0) {
        pair_sync(bar + u - 1);
        y = sy[w - 1][lane];
    }
    y = q.forward(y, len);
    if (u < G - 1) {
        sy[w][lane] = y;
        pair_sync(bar + u);
    }
    q.stash(omega);
    // the two halves meet: q and a_next of either half's last step
    float out = 0.f;
    if (u == G - 1) {
        P ql = P(0), an = P(0);
        float xl = 0.f;
        if (ns > 0) {
#pragma unroll
            for (int j = 0; j < K; ++j) {   // (the last of the chunk's steps)
                ql = j < len ? q.ip[j] : ql;
                xl = j < len ? q.x[j] : xl;
            }
            const unsigned k = level(ns - 1);
            an = mulr(P(__ldg(L.rdz + k)), P(ldf(L.tv + ((up ? k : k + 1) * ncolp + at.cp))));
        }
        si[up][0][lane] = ql;
        si[up][1][lane] = y;
        si[up][2][lane] = an;
        pair_sync(2 * G - 1 + group);
        // (a single level: nothing above, and p = q + a_next)
        const P dlt = nlev == 1 ? mulr(y, P(1) / (ql + an))
                                : interface32(ql, y, an, si[!up][0][lane], si[!up][1][lane], si[!up][2][lane]);
        out = float(fmad(P(omega), dlt, P(xl)));
    } else {
        pair_sync(bar + u);
        out = so[w + 1][lane];
    }
    out = q.backward(out, u == G - 1, len);
    if (u > 0) {
        so[w][lane] = out;
        pair_sync(bar + u - 1);
    }
    if (!active) return;
#pragma unroll
    for (int j = 0; j < K; ++j)
        if (j < len) {
            O* const pk = xo + level(s0 + j) * (PADO ? ncolp : ncol);
            pk[PADO ? at.cp : c] = (O)q.r[j];
            if (PADO) {
                if (rw >= 0) pk[rw] = (O)q.r[j];
                if (rn >= 0) pk[rn] = (O)q.r[j];
            }
        }
}

// Rims of a C1 level's iterate (a column there has several edges on one axis)
template <typename T>
__global__ void k_fill_rims(int n, int ncol, const int32_t* __restrict__ hd, T* __restrict__ x) {
    const unsigned c = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (c >= (unsigned)ncol) return;
    const unsigned np = pad_row(n), o = k * padded(n);
    for (int s = 0; s < 4; ++s) {
        const int d = hd[(unsigned)s * ncol + c];
        if (d >= 0) x[o + d] = x[o + Pos(c, n, np).cp];
    }
}

// ---------------------------------------------------------------------------------------
// Residual and restriction (Algorithm 1): bc[k][C] = sum_q w_q (b - H x)[k][child_q],
// w = area_child / area_C.  One thread per coarse column (2 x 2 fine columns, whose rows are read 2
// wide) and kchunk levels.  TREE: the children are summed in pairs (levels of n % 16 == 0), else
// one after the other: either order is as accurate, both stay because another would move every solve's
// result within its tolerance (above).  The loads in flight bound it: the loop stays rolled (two levels at a
// time need more registers, fewer blocks fit: C192L70 72 us instead of 56, C96L70 21 instead of 17; three
// couplings, x, b and the result at copy speed: 46 and 12).
template <typename C, bool XZERO, bool TREE>
__global__ void __launch_bounds__(128) k_restrict32(Lvl32<C, float> L, const float* __restrict__ x,
                                                    const float* __restrict__ b, const float* __restrict__ wq,
                                                    float* __restrict__ bc, int ncol_c, int kchunk) {
    const unsigned n = L.n, nc = n >> 1, np = L.np, lx = L.ncolp;
    const unsigned Cc = blockIdx.x * blockDim.x + threadIdx.x;
    if (Cc >= (unsigned)ncol_c) return;
    const Pos at(Cc, nc, pad_row(nc));
    const unsigned lc = padded(nc);
    const unsigned c0 = at.p * n * n + 2 * at.j * n + 2 * at.i;
    const unsigned cx[2] = {((n + 2) * at.p + 2 * at.j + 1) * np + pad_off(n) + 2 * at.i,
                            ((n + 2) * at.p + 2 * at.j + 2) * np + pad_off(n) + 2 * at.i};
    const int k0 = blockIdx.y * kchunk, k1 = min(L.nlev, k0 + kchunk);
    auto ld2 = [](const auto* q, float(&v)[2]) {
        using S = typename std::remove_cv<typename std::remove_reference<decltype(*q)>::type>::type;
        if constexpr (sizeof(S) == 4) {
            const float2 t = __ldg(reinterpret_cast<const float2*>(q));
            v[0] = t.x;
            v[1] = t.y;
        } else {
            const uint32_t t = __ldg(reinterpret_cast<const uint32_t*>(q));
            v[0] = __uint_as_float(t << 16);
            v[1] = __uint_as_float(t & 0xffff0000u);
        }
    };
    float rA[2][2], ww[2][2];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            rA[r][v] = __ldg(L.rA + c0 + r * n + v);
            ww[r][v] = __ldg(wq + (unsigned)(2 * r + v) * ncol_c + Cc);
        }
    float x0[2][2], xb[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, tb[2][2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        if (!XZERO) {
            ld2(x + (k0 * lx + cx[r]), x0[r]);
            if (k0 > 0) ld2(x + ((k0 - 1) * lx + cx[r]), xb[r]);
            ld2(L.tv + (k0 * lx + cx[r]), tb[r]);
        }
    }
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
        const unsigned o = (unsigned)k * lx;
        float r_[2][2];
#pragma unroll
        for (int r = 0; r < 2; ++r) ld2(b + (o + cx[r]), r_[r]);
        if (!XZERO) {
            const float rdz = __ldg(L.rdz + k);
            float xa[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, ta[2][2], te[2][2], tw[2], xE[2], xW[2], tn[2][2], ts[2], xN[2], xS[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                if (k + 1 < L.nlev) ld2(x + (o + lx + cx[r]), xa[r]);
                ld2(L.tv + (o + lx + cx[r]), ta[r]);
                ld2(L.te + (o + cx[r]), te[r]);
                ld2(L.tn + (o + cx[r]), tn[r]);
                tw[r] = ldf(L.te + (o + cx[r] - 1));
                xE[r] = __ldg(x + (o + cx[r] + 2));
                xW[r] = __ldg(x + (o + cx[r] - 1));
            }
            ld2(L.tn + (o + cx[0] - np), ts);
            ld2(x + (o + cx[1] + np), xN);
            ld2(x + (o + cx[0] - np), xS);
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int v = 0; v < 2; ++v)
                    r_[r][v] = residual32<!TREE>(r_[r][v], x0[r][v], v ? xE[r] : x0[r][1], v ? x0[r][0] : xW[r],
                                          r ? xN[v] : x0[1][v], r ? x0[0][v] : xS[v], te[r][v], v ? te[r][0] : tw[r],
                                          tn[r][v], r ? tn[0][v] : ts[v], rA[r][v], rdz, ta[r][v], xa[r][v], tb[r][v],
                                          xb[r][v]);
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    xb[r][v] = x0[r][v];
                    x0[r][v] = xa[r][v];
                    tb[r][v] = ta[r][v];
                }
        }
        float s;
        if (TREE) {
            s = addr(addr(mulr(ww[0][0], r_[0][0]), mulr(ww[0][1], r_[0][1])),
                     addr(mulr(ww[1][0], r_[1][0]), mulr(ww[1][1], r_[1][1])));
        } else {
            s = mulr(ww[0][0], r_[0][0]);
            s = fmad(ww[0][1], r_[0][1], s);
            s = fmad(ww[1][0], r_[1][0], s);
            s = fmad(ww[1][1], r_[1][1], s);
        }
        bc[(unsigned)k * lc + at.cp] = s;
    }
}

// ---------------------------------------------------------------------------------------
// Padded couplings from the FP64 face form (Th [nlev][2 ncol], Tv [nlev + 1][ncol]); one thread per
// column and level (tv: rows 0 .. nlev).
template <typename C>
__device__ __forceinline__ C pack_value(double v) {
    return (C)v;
}
template <>
__device__ __forceinline__ __nv_bfloat16 pack_value<__nv_bfloat16>(double v) {
    return __float2bfloat16_rn((float)v);
}

template <typename C>
__global__ void k_pack32(int n, int ncol, int nlev, const int32_t* __restrict__ fof, const double* __restrict__ Th,
                         const double* __restrict__ Tv, C* __restrict__ te, C* __restrict__ tn, C* __restrict__ tv) {
    const unsigned c = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
    if (c >= (unsigned)ncol) return;
    const int np = pad_row(n);
    const Pos at(c, n, np);
    const size_t o = (size_t)k * padded(n) + at.cp;
    tv[o] = pack_value<C>(Tv[(size_t)k * ncol + c]);
    if (k >= (unsigned)nlev) return;
    const double* t = Th + (size_t)k * 2 * ncol;
    te[o] = pack_value<C>(t[__ldg(fof + c)]);
    tn[o] = pack_value<C>(t[__ldg(fof + 2 * ncol + c)]);
    if (at.i == 0) te[o - 1] = pack_value<C>(t[__ldg(fof + ncol + c)]);
    if (at.j == 0) tn[o - np] = pack_value<C>(t[__ldg(fof + 3 * ncol + c)]);
}

// The pivots of both halves of every column: ip (1 / p; q at a half's last step) and, for an FP64
// elimination, the multipliers m and e.  One thread per column and half (blockIdx.y); the next BATCH
// steps' operands are under way while a batch is eliminated (as in k_factor64; with k_pack32 at C24L128 46 -> 25 us).
template <typename C, typename P>
__global__ void k_factor32(Lvl32<C, P> L, P* __restrict__ ip_, P* __restrict__ m_, P* __restrict__ e_) {
    constexpr int BATCH = 8;
    const unsigned c = blockIdx.x * blockDim.x + threadIdx.x;
    const bool up = blockIdx.y;
    const int nlev = L.nlev, hs = (nlev + 1) >> 1, ns = up ? nlev - hs : hs;
    if (c >= (unsigned)L.ncol || ns == 0) return;
    const unsigned np = L.np, ncolp = L.ncolp;
    const Pos at(c, L.n, np);
    const float rA = __ldg(L.rA + c);
    auto level = [&](int s) { return (unsigned)(up ? nlev - 1 - s : s); };
    float H[BATCH], T[BATCH], Z[BATCH], Hn[BATCH], Tn[BATCH], Zn[BATCH];   // horizontal sum, face ahead, 1 / dz
    auto load = [&](int s0) {
#pragma unroll
        for (int q = 0; q < BATCH; ++q) {
            const unsigned k = level(min(s0 + q, ns - 1)), o = k * ncolp + at.cp;
            Hn[q] = addr(addr(ldf(L.te + o), ldf(L.te + (o - 1))), addr(ldf(L.tn + o), ldf(L.tn + (o - np))));
            Tn[q] = ldf(L.tv + ((up ? k : k + 1) * ncolp + at.cp));
            Zn[q] = __ldg(L.rdz + k);
        }
    };
    load(0);
    P q = P(0), ip = P(0);
    float tb = 0.f;
    for (int s0 = 0; s0 < ns; s0 += BATCH) {
#pragma unroll
        for (int i = 0; i < BATCH; ++i) H[i] = Hn[i], T[i] = Tn[i], Z[i] = Zn[i];
        if (s0 + BATCH < ns) load(s0 + BATCH);
#pragma unroll
        for (int i = 0; i < BATCH; ++i) {
            const int s = s0 + i;
            if (s < ns) {
                const unsigned o = level(s) * ncolp + at.cp;
                const P an = mulr(P(Z[i]), P(T[i])), m = mulr(mulr(P(Z[i]), P(tb)), ip);
                q = fmad(m, q, fmad(P(rA), P(H[i]), P(1)));
                ip = P(1) / (q + an);
                ip_[o] = s == ns - 1 ? q : ip;
                if (sizeof(P) == 8) {
                    m_[o] = m;
                    e_[o] = mulr(an, ip);
                }
                tb = T[i];
            }
        }
    }
}

// x_out = (x or 0) + xc[parent] (Eq. prolongation, natural injection) or, without xc, the
// conversion of x; T or O FP32: padded, FP64: plain; one thread per column and kchunk levels, which share the
// column's position and edges.
template <typename T, typename O>
__global__ void k_emit(int n, int ncol, int nlev, int kchunk, const int32_t* __restrict__ hd, const T* __restrict__ x,
                       const T* __restrict__ xc, O* __restrict__ xo) {
    constexpr bool PAD = sizeof(T) == 4, PADO = sizeof(O) == 4;
    const unsigned c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= (unsigned)ncol) return;
    const unsigned np = pad_row(n), ncolp = padded(n);
    const Pos at(c, n, np);
    const unsigned from = PAD ? at.cp : c, to = PADO ? at.cp : c, parent = !xc ? 0 : PAD ? at.parent(0, 0, n, pad_row(n >> 1)) : parent_col(c, n);
    const unsigned lf = PAD ? ncolp : ncol, lt = PADO ? ncolp : ncol, lc = PAD ? padded(n >> 1) : ncol >> 2;
    int rim[4] = {-1, -1, -1, -1};
    if (PADO && (at.i == 0 || at.j == 0 || at.i + 1 == (unsigned)n || at.j + 1 == (unsigned)n)) {
#pragma unroll
        for (int s = 0; s < 4; ++s) rim[s] = __ldg(hd + (unsigned)s * ncol + c);
    }
    const unsigned k0 = blockIdx.y * kchunk, k1 = min(nlev, (int)k0 + kchunk);
#pragma unroll 4
    for (unsigned k = k0; k < k1; ++k) {
        T v = T(0);
        if (x) v = __ldg(x + (k * lf + from));
        if (xc) v += __ldg(xc + (k * lc + parent));
        xo[k * lt + to] = (O)v;
        if constexpr (PADO) {
#pragma unroll
            for (int s = 0; s < 4; ++s)
                if (rim[s] >= 0) xo[k * lt + rim[s]] = (O)v;
        }
    }
}

// ---- launch interface (instantiated per precision in sweep_*.cu) ----
struct SweepMaps;

template <typename C, typename P>
struct SweepCall32 {
    Lvl32<C, P> L;
    int mode;            // XM_*
    const float* x;
    const float* xc;
    const void* b;       // FP64 when raw, padded FP32 otherwise
    bool raw;
    float* bcopy;        // raw: where to store the FP32 copy, or NULL
    void* xo;            // plain FP64 with out64, padded FP32 otherwise
    bool out64;
    double omega;
    const SweepMaps* maps;   // tensor maps of x, xc, b and the level's data (sweep_tma.cuh), or NULL
    int nsm;
    int polls;               // limit of a TMA wait
    unsigned int* timeout;   // set by a TMA wait that runs into its limit
};

template <typename C, typename P>
cudaError_t sweep32_run(const SweepCall32<C, P>& q, cudaStream_t s);

}  // namespace mg
