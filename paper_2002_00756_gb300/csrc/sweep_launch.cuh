// Launcher of the FP32 column sweep (sweep32.cuh, sweep_tma.cuh).
#pragma once

#include <algorithm>
#include <type_traits>

#include "sweep_tma.cuh"

namespace mg {
namespace {

// Levels per chunk of the register sweep: 5; columns of more than 80 levels take 8, so that a block has at
// most 16 warps (a sweep from zero on the registers of two blocks per SM: C50L110 21 -> 17 us, C40L128 16 -> 13).
constexpr int CHUNK_K = 5, TALL_K = 8;

template <typename C, typename P, int MODE, typename B, typename O, bool BRAW, int K>
cudaError_t go(const SweepCall32<C, P>& q, cudaStream_t s) {
    constexpr int M = sweep32_groups(K);   // (G is 1 where M is not)
    const int G = ((q.L.nlev + 1) / 2 + K - 1) / K;
    k_sweep32<C, P, MODE, B, O, BRAW, K><<<(q.L.ncol + 32 * M - 1) / (32 * M), 64 * G * M, 0, s>>>(
        q.L, q.x, q.xc, static_cast<const B*>(q.b), q.bcopy, static_cast<O*>(q.xo), (float)q.omega);
    return cudaGetLastError();
}

// The short columns' chunk is a whole half: with 5 or 10 steps for one or three, the steps past its end cost
// more than the chunk (V-cycle, FP32 / FP64 elimination, 64 threads a block: C192L1 160 / 310 us with 5, 127 / 179
// with 1; C192L4 165 / 340 and 142 / 245 with 2; C256L6 463 / 899 with 10, 299 / 606 with 5, 268 / 484 with 3).
template <typename C, typename P, int MODE, typename B, typename O, bool BRAW>
cudaError_t shape(const SweepCall32<C, P>& q, cudaStream_t s) {
    switch ((q.L.nlev + 1) / 2) {
        case 1: return go<C, P, MODE, B, O, BRAW, 1>(q, s);
        case 2: return go<C, P, MODE, B, O, BRAW, 2>(q, s);
        case 3: return go<C, P, MODE, B, O, BRAW, 3>(q, s);
        case 4: return go<C, P, MODE, B, O, BRAW, 4>(q, s);
        default: break;
    }
    if (q.L.nlev > 80) return go<C, P, MODE, B, O, BRAW, TALL_K>(q, s);
    return go<C, P, MODE, B, O, BRAW, CHUNK_K>(q, s);
}

constexpr int TMA_SMEM = 227 * 1024;   // shared memory of an SM, and the most a block can have

template <typename C, typename P, int MODE, typename O, bool BRAW, int K, bool FULL>
cudaError_t go_tma(const SweepCall32<C, P>& q, cudaStream_t s) {
    const TmaLayout<C, P, MODE, BRAW, K> Y(q.L.nlev);
    auto kern = k_sweep_tma<C, P, MODE, O, BRAW, K, FULL>;
    // (the limit is the function's, for every thread and handle: the device's maximum, whatever this launch
    // takes.  Two threads with handles of different heights could lower one of Y.total under each other.)
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, TMA_SMEM);
    if (e != cudaSuccess) return e;
    const int threads = 64 * tma_chunks(q.L.nlev, K);
    // tiles: up to 32 columns of a row, a multiple of 16 bytes of the couplings wide (tensor coordinates)
    constexpr int Q = 16 / (int)sizeof(C);
    const int tr = (q.L.n + TMA_COLS - 1) / TMA_COLS, tw = ((q.L.n + tr - 1) / tr + Q - 1) / Q * Q;
    const int per_sm = std::max(1, std::min({TMA_SMEM / (Y.total + 1024), tma_blocks(MODE, BRAW, sizeof(P), K) * tma_threads(K) / threads, 8}));
    const int grid = std::min(6 * q.L.n * tr, per_sm * q.nsm);
    kern<<<grid, threads, Y.total, s>>>(*q.maps, q.L, static_cast<const double*>(BRAW ? q.b : nullptr), q.bcopy,
                                        static_cast<O*>(q.xo), (float)q.omega, tr, tw, q.polls, q.timeout);
    return cudaGetLastError();
}

// tiles where the level has them, else register chunks
template <typename C, typename P, int MODE, typename O, bool BRAW>
cudaError_t form(const SweepCall32<C, P>& q, cudaStream_t s) {
    if (q.maps) {
        if constexpr (sizeof(P) == 4) {
            if (q.L.nlev > tma_max_levels(8)) return go_tma<C, P, MODE, O, BRAW, 10, false>(q, s);
        }
        if (q.L.nlev > tma_max_levels(7)) return go_tma<C, P, MODE, O, BRAW, 8, false>(q, s);
        if (q.L.nlev == tma_chunks(q.L.nlev, 7) * 14) return go_tma<C, P, MODE, O, BRAW, 7, true>(q, s);
        return go_tma<C, P, MODE, O, BRAW, 7, false>(q, s);
    }
    return shape<C, P, MODE, typename std::conditional<BRAW, double, float>::type, O, BRAW>(q, s);
}

template <typename C, typename P, int MODE>
cudaError_t outs(const SweepCall32<C, P>& q, cudaStream_t s) {
    if (q.out64) return form<C, P, MODE, double, false>(q, s);
    return form<C, P, MODE, float, false>(q, s);
}

}  // namespace

template <typename C, typename P>
cudaError_t sweep32_run(const SweepCall32<C, P>& q, cudaStream_t s) {
    if (q.raw) {
        if (q.mode != XM_ZERO) return cudaErrorInvalidValue;
        if (q.out64) return form<C, P, XM_ZERO, double, true>(q, s);
        return form<C, P, XM_ZERO, float, true>(q, s);
    }
    switch (q.mode) {
        case XM_ZERO: return outs<C, P, XM_ZERO>(q, s);
        case XM_PLAIN: return outs<C, P, XM_PLAIN>(q, s);
        case XM_PROLONG: return outs<C, P, XM_PROLONG>(q, s);
        case XM_PROLONG0: return outs<C, P, XM_PROLONG0>(q, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace mg
