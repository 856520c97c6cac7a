// The column sweep of large FP32 levels with every operand brought by TMA (the same arithmetic as
// k_sweep32 in sweep32.cuh).
//
// A tile is up to 32 consecutive columns of one row of a panel, all levels.  One thread issues one
// tensor copy per stream and half tile (box: columns x nlev / 2 of the level-major array), so no
// thread computes global addresses or holds loads in registers: the walk reads shared memory at
// fixed offsets.  The fields are padded (sweep32.cuh): the iterate's box has 4 columns more on each
// side and the east faces' box 4 on the west, so E / W neighbours are the adjacent columns of the
// box, and the N / S neighbours and south faces are boxes one padded row up / down, at a panel's
// edges as anywhere else.
//
// Blocks are persistent (tma_blocks per SM): as soon as a tile's values are in
// registers the copies of the block's next tile are issued into the same buffers, and run during
// the recurrences and the stores.
//
// Measured (finest level of C192L70, 15.5M cells, us per sweep; two threads per column with the pivot
// chain in the walk before): plain 86 (121), with prolongation 90 (134), from zero 72 (108); BF16
// couplings at C90L41 18 (27); FP64 elimination at C96L70 102 (194).  A plain sweep moves 433 MB (28 B
// per cell: x, b, three couplings, the reciprocal pivot, the result), 64 us at the measured copy rate; its
// boxes alone, nothing computed or stored, stream in 61 us.  Of the rest, 10 us are the stores, the others
// the time a group's buffers wait for its warps.  Columns of more than 80 levels, one block per SM: C128L100,
// 9.8M cells, 78 us in every mode (the register chunks 103 to 142).
// With the panel edges fetched by threads instead of kept in rims the plain sweep took 96 us.
#pragma once

#include <cuda.h>

#include "sweep32.cuh"

namespace mg {

// boxes (columns x levels, H = ceil(nlev / 2)): b, ip, tn (also ts, one row down) and xr (N, S)
// 32 x H; te 32 + 16 bytes' worth of columns to the west x H; tv 32 x (H + 1); x 40 x (H + 1) from four
// columns to the west; xc 24 x (H + 1), xca 24 x H
struct SweepMaps {
    CUtensorMap b, ip, te, tn, tv, x, xr, xc, xca;
};

constexpr int TMA_COLS = 32;
// Resident blocks per SM that the registers are capped for: two where shared memory allows no more, and
// for a caller's right-hand side read ahead in registers (three: 91 us instead of 72 at C192L70, spills);
// three for the other sweeps from zero (17 us instead of 19 on C96L70).
// One for columns of more than 80 levels (chunks of 10), whose boxes take up to 190 KB.
__host__ __device__ constexpr int tma_blocks(int mode, bool braw, int psize, int K) {
    return K == 10 ? 1 : mode == XM_ZERO && !braw && psize == 4 ? 3 : 2;
}

template <typename C>
__device__ __forceinline__ float lds(const C* p) {
    if constexpr (sizeof(C) == 2) return __bfloat162float(*p);
    else return *p;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
constexpr int WAIT_POLLS = 1 << 20;   // default limit of a wait, and that of a late copy's second wait
// waits for the phase of the given parity; false after `polls` polls
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int polls) {
    for (int i = 0; i < polls; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}
__device__ __forceinline__ void tma_load(void* dst, const CUtensorMap* m, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_addr(dst)),
        "l"(m), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// The lower half of the levels is walked upwards, the upper half downwards, each by a group of G
// warps with a chunk of up to K steps per warp.  Each group has its own boxes, its own mbarrier and
// issues its own copies, so its buffers are refilled as soon as its own warps have read them.
//
// A copy that does not arrive within the limit: the group's threads agree on it where they meet anyway
// (a reduction over the barrier: 0.2-0.5 % of a solve; a mark in shared memory costs more), and from then
// on issue no copy and touch the mbarrier no more, whose phase is still open.  They go through their
// remaining tiles all the same, because the other group's interface waits for them, and give NaN, which
// the interface hands to the other half of the column.  Before they leave they wait once more, with the
// default limit, for the copies in flight, and report.
__host__ __device__ constexpr int tma_max_levels(int K) { return K == 7 ? 70 : K == 8 ? 80 : 128; }
__host__ __device__ constexpr int tma_chunks(int nlev, int K) { return ((nlev + 1) / 2 + K - 1) / K; }
__host__ __device__ constexpr int tma_threads(int K) { return 64 * tma_chunks(tma_max_levels(K), K); }

// Shared memory of a group: the streams' boxes ([rows][columns], each start a multiple of 128 bytes).
// Reads of a short chunk may run up to K rows past its box's end (or, in the upper half, before its
// start): into the neighbouring stream, the lower group's boxes or `slack`.  After the two groups
// 1 / dz, the exchanged values and the mbarriers.
template <typename C, typename P, int MODE, bool BRAW, int K>
struct TmaLayout {
    int b, ip, te, tn, ts, tv, x, xn, xs, c0, c1, group, rdz, sy, so, si, bar, total;
    uint32_t tx;   // bytes of one group's copies
    __host__ __device__ explicit TmaLayout(int nlev) {
        constexpr int CS = sizeof(C);
        const int H = (nlev + 1) / 2, G = tma_chunks(nlev, K);
        int o = 0;
        uint32_t bytes = 0;
        auto add = [&](bool used, int rows, int row_bytes) {
            const int at = o;
            if (used) {
                o += (rows * row_bytes + 127) / 128 * 128;
                bytes += rows * row_bytes;
            }
            return at;
        };
        const bool it = MODE != XM_ZERO;
        b = add(!BRAW, H, 128);
        ip = add(sizeof(P) == 4, H, 128);
        tv = add(sizeof(P) == 4 || it, H + 1, 32 * CS);
        te = add(it, H, 32 * CS + 16);
        tn = add(it, H, 32 * CS);
        ts = add(it, H, 32 * CS);
        x = add(it && MODE != XM_PROLONG0, H + 1, 160);
        xn = add(it && MODE != XM_PROLONG0, H, 128);
        xs = add(it && MODE != XM_PROLONG0, H, 128);
        c0 = add(MODE == XM_PROLONG || MODE == XM_PROLONG0, H + 1, 96);
        c1 = add(MODE == XM_PROLONG || MODE == XM_PROLONG0, H, 96);
        tx = bytes;
        group = o;
        rdz = 2 * o + K * 160;
        sy = rdz + (nlev + K) / 4 * 16 + 16;
        so = sy + 2 * G * 32 * (int)sizeof(P);
        si = so + 2 * G * 128;
        bar = si + 2 * 2 * 3 * 32 * (int)sizeof(P);
        total = bar + 16;
    }
};

// FULL: every chunk has K steps.  BRAW: b is the caller's plain FP64 array, read directly one tile
// ahead; its FP32 copy is stored in bcopy unless that is NULL.  P = double: the FP64 pivots and multipliers are read
// directly as well (their boxes would leave room for one block per SM only).
template <typename C, typename P, int MODE, typename O, bool BRAW, int K, bool FULL>
__global__ void __launch_bounds__(tma_threads(K), tma_blocks(MODE, BRAW, sizeof(P), K))
    k_sweep_tma(const __grid_constant__ SweepMaps M, Lvl32<C, P> L, const double* __restrict__ braw,
                float* __restrict__ bcopy, O* __restrict__ xo, float omega, int tiles_row, int tile_w,
                int polls, unsigned int* __restrict__ timeout) {
    constexpr bool PRO = MODE == XM_PROLONG || MODE == XM_PROLONG0;
    constexpr bool RAW = MODE == XM_PLAIN || MODE == XM_PROLONG;   // reads the fine iterate
    constexpr bool ZERO = MODE == XM_ZERO, PADO = sizeof(O) == 4, D64 = sizeof(P) == 8;
    constexpr int TW = 16 / (int)sizeof(C), TP = 32 + TW;   // te: columns to the west, row pitch
    extern __shared__ __align__(128) unsigned char sm_all[];
    const TmaLayout<C, P, MODE, BRAW, K> Y(L.nlev);
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, G = blockDim.x >> 6;
    const bool up = w >= G;
    const int u = up ? w - G : w, gtid = tid - (up ? blockDim.x >> 1 : 0), gthreads = blockDim.x >> 1;
    const int n = L.n, nlev = L.nlev, nc = n >> 1, hs = (nlev + 1) >> 1, ns = up ? nlev - hs : hs;
    const int np = L.np, npc = pad_row(nc), of = pad_off(n), ofc = pad_off(nc);
    const int kb = up ? hs : 0, kx = up ? hs - 1 : 0;   // first level of the group's boxes, and of x's
    unsigned char* const sm = sm_all + (up ? Y.group : 0);
    const uint32_t bar = smem_addr(sm_all + Y.bar + 8 * up);
    const int ntiles = 6 * n * tiles_row;
    auto fp = [&](int at) { return reinterpret_cast<const float*>(sm + at); };
    auto cp_ = [&](int at) { return reinterpret_cast<const C*>(sm + at); };
    float* const srdz = reinterpret_cast<float*>(sm_all + Y.rdz);
    P* const sy = reinterpret_cast<P*>(sm_all + Y.sy) + w * 32 + lane;
    float* const so = reinterpret_cast<float*>(sm_all + Y.so) + w * 32 + lane;
    P* const si = reinterpret_cast<P*>(sm_all + Y.si) + lane;   // [2 tiles][2 halves][3][32]
    // the group meets; whether any of its threads says v
    auto group_any = [&](bool v) {
        uint32_t any;
        if (up)
            asm volatile("{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, 2, %2, p;\n selp.u32 %0, 1, 0, q;\n}"
                         : "=r"(any)
                         : "r"((uint32_t)v), "r"(gthreads)
                         : "memory");
        else
            asm volatile("{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, 1, %2, p;\n selp.u32 %0, 1, 0, q;\n}"
                         : "=r"(any)
                         : "r"((uint32_t)v), "r"(gthreads)
                         : "memory");
        return any != 0;
    };
    const int pair = 3 + (up ? G - 1 : 0);   // barriers pair .. pair + G - 2 between the group's chunks
    // padded column of a tile's first parent, and of the row of parents its N (odd rows) or S (even
    // rows) neighbours have instead
    auto coarse = [&](int p, int j, int i0, bool adj) {
        return ((nc + 2) * p + (j >> 1) + 1 + (adj ? ((j & 1) ? 1 : -1) : 0)) * npc + ofc + (i0 >> 1);
    };

    auto issue = [&](int t) {
        const int row = t / tiles_row, i0 = (t - row * tiles_row) * tile_w, p = row / n;
        const int c = (row + 2 * p + 1) * np + of + i0;
        mbar_expect(bar, Y.tx);
        if (!BRAW) tma_load(sm + Y.b, &M.b, c, kb, bar);
        if (!D64) tma_load(sm + Y.ip, &M.ip, c, kb, bar);
        if (!D64 || !ZERO) tma_load(sm + Y.tv, &M.tv, c, kb, bar);
        if (!ZERO) {
            if (RAW) {
                tma_load(sm + Y.x, &M.x, c - 4, kx, bar);
                tma_load(sm + Y.xn, &M.xr, c + np, kb, bar);
                tma_load(sm + Y.xs, &M.xr, c - np, kb, bar);
            }
            tma_load(sm + Y.te, &M.te, c - TW, kb, bar);
            tma_load(sm + Y.tn, &M.tn, c, kb, bar);
            tma_load(sm + Y.ts, &M.tn, c - np, kb, bar);
        }
        if (PRO) {
            const int j = row - p * n;
            tma_load(sm + Y.c0, &M.xc, (coarse(p, j, i0, false) - 1) & ~3, kx, bar);
            tma_load(sm + Y.c1, &M.xca, coarse(p, j, i0, true) & ~3, kb, bar);
        }
    };
    if (gtid == 0) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if ((int)blockIdx.x < ntiles) issue(blockIdx.x);
    }
    for (int k = tid; k < nlev; k += blockDim.x) srdz[k] = __ldg(L.rdz + k);
    __syncthreads();
    const int s0 = u * ns / G, len = FULL ? K : (u + 1) * ns / G - s0;
    // (steps past a short chunk's end repeat its half's last one, unused)
    auto level = [&](int i) { return (unsigned)(up ? nlev - 1 - min(s0 + i, ns - 1) : min(s0 + i, ns - 1)); };
    double bn[BRAW ? K : 1];   // b of the coming tile
    auto fetch_b = [&](int t) {
        const int row = t / tiles_row, i0 = (t - row * tiles_row) * tile_w;
        const unsigned c = row * n + i0 + min(lane, min(tile_w, n - i0) - 1);
#pragma unroll
        for (int i = 0; i < (BRAW ? K : 0); ++i) bn[i] = __ldg(braw + (level(i) * L.ncol + c));
    };
    if (BRAW && (int)blockIdx.x < ntiles) fetch_b(blockIdx.x);
    uint32_t phase = 0, open = 0;   // open: parity of the phase that a late copy has left open
    bool late = false;              // the same for all of the group's threads
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, phase ^= 1) {
        const int row = t / tiles_row, i0 = (t - row * tiles_row) * tile_w;
        const int p = row / n, j = row - p * n, cols = min(tile_w, n - i0);
        // (lanes beyond the tile repeat its last column: rows are too short on small meshes to read on)
        const unsigned c = row * n + i0 + min(lane, cols - 1), cp = (row + 2 * p + 1) * np + of + i0 + min(lane, cols - 1);
        const float rA = __ldg(L.rA + c);
        // (an edge column is repeated in one rim, a corner column in two)
        int rim0 = -1, rim1 = -1;
        if (PADO && lane < cols) {
            const int i = i0 + lane;
            if (i == 0) rim0 = __ldg(L.hd + L.ncol + c);
            if (i == n - 1) rim0 = __ldg(L.hd + c);
            if (j == n - 1) rim1 = __ldg(L.hd + 2 * L.ncol + c);
            if (j == 0) rim1 = __ldg(L.hd + 3 * L.ncol + c);
        }
        const int ca0 = coarse(p, j, i0, false), ca1 = coarse(p, j, i0, true);
        const int off0 = ca0 - ((ca0 - 1) & ~3) + (lane >> 1), off1 = ca1 - (ca1 & ~3) + (lane >> 1);
        Chunk<P, K> q;
        if constexpr (D64) {
#pragma unroll
            for (int i = 0; i < K; ++i) {
                const unsigned o = level(i) * L.ncolp + cp;
                q.m[i] = __ldg(L.m + o);
                q.ip[i] = __ldg(L.ip + o);
                q.e[i] = __ldg(L.e + o);
            }
        }
        const bool miss = !late && !mbar_wait(bar, phase, polls);
        P an = P(0);   // a_next of the chunk's last step
        // reads the chunk, walking the rows of the boxes in direction D
        auto read = [&](auto dir) {
            constexpr int D = decltype(dir)::value;
            // row of step s0: of the x boxes, of the others, of the vertical face ahead
            const int rx = D > 0 ? s0 : ns - s0, r0 = D > 0 ? s0 : ns - 1 - s0, rt = D > 0 ? s0 + 1 : ns - 1 - s0;
            const float* qx = fp(Y.x) + rx * 40 + 4 + lane;
            const float* qc = fp(Y.c0) + rx * 24 + off0;
            [[maybe_unused]] const float* qo = qc + ((lane & 1) ? 1 : -1);
            const float* qa = fp(Y.c1) + r0 * 24 + off1;
            const float *qn = fp(Y.xn) + r0 * 32 + lane, *qs = fp(Y.xs) + r0 * 32 + lane;
            const C *qte = cp_(Y.te) + r0 * TP + TW + lane, *qtn = cp_(Y.tn) + r0 * 32 + lane;
            const C *qts = cp_(Y.ts) + r0 * 32 + lane, *qtv = cp_(Y.tv) + rt * 32 + lane;
            const float *qb = fp(Y.b) + r0 * 32 + lane, *qi = fp(Y.ip) + r0 * 32 + lane;
            const float* qz = srdz + (D > 0 ? s0 : nlev - 1 - s0);
            // (before the walk's first step the face behind and its m are zero)
            float xb = 0.f, x0 = 0.f, tb = 0.f, ipb = 0.f;
            if (!D64 || !ZERO) tb = lds<C>(qtv - D * 32);
            if (RAW) x0 = qx[0];
            if (PRO) x0 += qc[0];
            if (s0 > 0) {
                if (RAW) xb = qx[-D * 40];
                if (PRO) xb += qc[-D * 24];
                if (!D64) ipb = qi[-D * 32];
            }
#pragma unroll
            for (int i = 0; i < K; ++i) {
                float ta = 0.f;
                [[maybe_unused]] const float rdz = qz[D * i];
                if (!D64 || !ZERO) ta = lds<C>(qtv + D * i * 32);
                if constexpr (!D64) {
                    q.ip[i] = qi[D * i * 32];
                    q.m[i] = mulr(mulr(rdz, tb), ipb);
                    const float a = mulr(rdz, ta);
                    q.e[i] = mulr(a, q.ip[i]);
                    if (FULL ? i == K - 1 : i == len - 1) an = a;
                    ipb = q.ip[i];
                }
                const float bk = BRAW ? (float)bn[BRAW ? i : 0] : qb[D * i * 32];
                q.x[i] = x0;
                q.r[i] = bk;
                if constexpr (!ZERO) {
                    float xa = 0.f, xE = 0.f, xW = 0.f, xN = 0.f, xS = 0.f;
                    if (RAW) {
                        xa = qx[D * (i + 1) * 40];
                        xE = qx[D * i * 40 + 1];
                        xW = qx[D * i * 40 - 1];
                        xN = qn[D * i * 32];
                        xS = qs[D * i * 32];
                    }
                    if (PRO) {
                        const float cm = qc[D * i * 24], co = qo[D * i * 24], ca = qa[D * i * 24];
                        xa += qc[D * (i + 1) * 24];
                        xE += (lane & 1) ? co : cm;
                        xW += (lane & 1) ? cm : co;
                        xN += (j & 1) ? ca : cm;
                        xS += (j & 1) ? cm : ca;
                    }
                    q.r[i] = residual32(bk, x0, xE, xW, xN, xS, lds<C>(qte + D * i * TP), lds<C>(qte + (D * i * TP - 1)),
                                        lds<C>(qtn + D * i * 32), lds<C>(qts + D * i * 32), rA, rdz, ta, xa, tb, xb);
                    xb = x0;
                    x0 = xa;
                }
                tb = ta;
            }
            q.x[K] = x0;
        };
        if (up) read(std::integral_constant<int, -1>());
        else read(std::integral_constant<int, 1>());
        // the group's values are in registers: the next tile's copies may overwrite its boxes
        if (group_any(miss)) {
            late = true;
            open = phase;
        }
        if (t + (int)gridDim.x < ntiles) {
            if (gtid == 0 && !late) issue(t + gridDim.x);
            if (BRAW) fetch_b(t + gridDim.x);
        }
        if (BRAW && bcopy && lane < cols) {
#pragma unroll
            for (int i = 0; i < K; ++i)
                if (FULL || i < len) bcopy[level(i) * L.ncolp + cp] = q.r[i];
        }
        if (D64 && u == G - 1) {
            const unsigned k = level(len - 1);
            an = mulr(P(srdz[k]), P(ldf(L.tv + ((up ? k : k + 1) * L.ncolp + cp))));
        }
        // forwards, chunk by chunk
        P y = P(0);
        float out;
        if (u > 0) {
            pair_sync(pair + u - 1);
            y = sy[-32];
        }
        y = q.forward(y, len);
        if (u < G - 1) {
            *sy = y;
            pair_sync(pair + u);
            q.stash(omega);
            // backwards: out of the chunk ahead
            pair_sync(pair + u);
            out = so[32];
        } else {   // the two halves meet
            P ql = P(0);
            float xl = 0.f;
#pragma unroll
            for (int i = 0; i < K; ++i) {   // (the last of the chunk's steps)
                ql = FULL || i < len ? q.ip[i] : ql;
                xl = FULL || i < len ? q.x[i] : xl;
            }
            if (late) y = P(__int_as_float(0x7fc00000));
            P* const mine = si + (2 * phase + up) * 96;
            const P* const other = si + (2 * phase + !up) * 96;
            mine[0] = ql;
            mine[32] = y;
            mine[64] = an;
            pair_sync(2 * G + 1);
            q.stash(omega);
            out = float(fmad(P(omega), interface32(ql, y, an, other[0], other[32], other[64]), P(xl)));
        }
        if (late) out = __int_as_float(0x7fc00000);
        out = q.backward(out, u == G - 1, len);
        if (u > 0) {
            *so = out;
            pair_sync(pair + u - 1);
        }
        const unsigned lo = PADO ? L.ncolp : L.ncol;
        const int d = up ? -(int)lo : (int)lo;
        O* const po = xo + (up ? nlev - 1 - s0 : s0) * lo;
        if (lane < cols) {
            O* pc = po + (PADO ? cp : c);
#pragma unroll
            for (int i = 0; i < K; ++i)
                if (FULL || i < len) pc[(ptrdiff_t)i * d] = (O)q.r[i];
        }
        if (PADO) {
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int rim = r ? rim1 : rim0;
                if (rim < 0) continue;
#pragma unroll
                for (int i = 0; i < K; ++i)
                    if (FULL || i < len) po[(ptrdiff_t)i * d + rim] = (O)q.r[i];
            }
        }
    }
    if (late) {
        atomicExch(timeout, 1u);
        mbar_wait(bar, open, WAIT_POLLS);
    }
}

}  // namespace mg
