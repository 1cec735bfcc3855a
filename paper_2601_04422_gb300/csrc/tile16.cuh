// A small tile of a complex product by 64 threads, shared by the FP64 products (k_fp64.cu)
// and the read-out (k_readout.cu): 8 x 8, one output per thread.
//
// The read-out's products are chains of small matrices, so a tile's time is its latency and
// what counts is how many SMs and schedulers share a product.  FP64 issues once in 64 cycles
// per scheduler: one output per thread is 4 FP64 instructions per k and warp.  (2 x 2 outputs
// per thread: 13 us for a complex128 24 x 12 x 12 product, the zeros of the K step included,
// against 3; a transfer of the read-out at chi 128, complex64, 24.5 us with 16 x 16 tiles in
// K steps of 16, 17 with 8 x 8 in steps of 64: fewer waits for a step's operands.)
// The next K step's operands are loaded while this one's are used.
#pragma once
#include <cuda_runtime.h>

#include "tnsim_internal.h"

namespace tnsim {

constexpr int TILE_THREADS = 64;
// edge, outputs per thread and side, K step
template <typename C> struct TileOf { static constexpr int E = 8, R = 1, K = sizeof(C) == 8 ? 64 : 16; };

// acc += a b; acc += conj(a) b; acc += a conj(b) -- one fixed order of the roundings
struct MulAdd {
    template <typename C> static __device__ __forceinline__ void op(C& acc, const C& a, const C& b) {
        acc.x = fma(a.x, b.x, acc.x);
        acc.x = fma(-a.y, b.y, acc.x);
        acc.y = fma(a.x, b.y, acc.y);
        acc.y = fma(a.y, b.x, acc.y);
    }
};
struct ConjMulAdd {
    template <typename C> static __device__ __forceinline__ void op(C& acc, const C& a, const C& b) {
        acc.x = fma(a.x, b.x, acc.x);
        acc.x = fma(a.y, b.y, acc.x);
        acc.y = fma(a.x, b.y, acc.y);
        acc.y = fma(-a.y, b.x, acc.y);
    }
};
// acc += a b, the products of the imaginary parts first
struct MulAddIm {
    template <typename C> static __device__ __forceinline__ void op(C& acc, const C& a, const C& b) {
        acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
        acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
    }
};
struct MulAddConj {
    template <typename C> static __device__ __forceinline__ void op(C& acc, const C& a, const C& b) {
        ConjMulAdd::op(acc, b, a);
    }
};

// acc += sum over k < K of OP(la(i, k), lb(k, j)): thread (rx, cy) = (tid % 8, tid / 8)
// holds rows rx + 8 i (PAIRED: 2 rx + i) and columns cy + 8 j, i, j < R.  la and lb give the
// operands' elements for tile row i / tile column j (zero outside them); AK / BK: memory
// runs along k (consecutive threads then load consecutive k).  k ascends; SPLIT sums every
// K step by itself first (rounding grows with sqrt(16 + K / 16) instead of sqrt(K), for
// 3 - 6 % more instructions); products of up to kPlain64 terms are one run of sums.
template <typename C, bool AK, bool BK, bool PAIRED, bool SPLIT, typename OP, typename LA, typename LB>
__device__ __forceinline__ void tile_product(int K, LA la, LB lb, C (&acc)[TileOf<C>::R][TileOf<C>::R]) {
    constexpr int E = TileOf<C>::E, R = TileOf<C>::R, TILE_K = TileOf<C>::K, PER = E * TILE_K / TILE_THREADS;
    __shared__ C As[TILE_K][E + 1], Bs[TILE_K][E + 1];
    const int tid = threadIdx.x, rx = tid & 7, cy = tid >> 3;
    C na[PER], nb[PER];
    const bool split = SPLIT && K > kPlain64;
    // element e of a K step: (edge index, k) with k running fastest (KF) or slowest
    auto at = [](int e, bool kf, int& i, int& k) {
        if (kf) { k = e % TILE_K; i = e / TILE_K; }
        else { i = e % E; k = e / E; }
    };
    auto fetch = [&](int k0) {
#pragma unroll
        for (int t = 0; t < PER; ++t) {
            int i, k;
            na[t] = C{};
            nb[t] = C{};
            at(tid + TILE_THREADS * t, AK, i, k);
            if (k0 + k < K) na[t] = la(i, k0 + k);
            at(tid + TILE_THREADS * t, BK, i, k);
            if (k0 + k < K) nb[t] = lb(k0 + k, i);
        }
    };
    fetch(0);
    for (int k0 = 0; k0 < K; k0 += TILE_K) {
#pragma unroll
        for (int t = 0; t < PER; ++t) {
            int i, k;
            at(tid + TILE_THREADS * t, AK, i, k);
            As[k][i] = na[t];
            at(tid + TILE_THREADS * t, BK, i, k);
            Bs[k][i] = nb[t];
        }
        __syncthreads();
        if (k0 + TILE_K < K) fetch(k0 + TILE_K);
        C part[R][R] = {};
        if (!split)
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int j = 0; j < R; ++j) part[i][j] = acc[i][j];
        const int kn = min(TILE_K, K - k0);
#pragma unroll 4
        for (int kk = 0; kk < kn; ++kk) {
            C a[R], b[R];
#pragma unroll
            for (int i = 0; i < R; ++i) {
                a[i] = As[kk][PAIRED ? R * rx + i : rx + 8 * i];
                b[i] = Bs[kk][cy + 8 * i];
            }
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int j = 0; j < R; ++j) OP::op(part[i][j], a[i], b[j]);
        }
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < R; ++j) {
                if (split) {
                    acc[i][j].x += part[i][j].x;
                    acc[i][j].y += part[i][j].y;
                } else {
                    acc[i][j] = part[i][j];
                }
            }
        __syncthreads();
    }
}

// The tile in shared memory, for outputs that mix entries of several threads.
template <typename C, bool PAIRED>
__device__ __forceinline__ void tile_share(C (*S)[TileOf<C>::E + 1], const C (&acc)[TileOf<C>::R][TileOf<C>::R]) {
    constexpr int R = TileOf<C>::R;
    const int rx = threadIdx.x & 7, cy = threadIdx.x >> 3;
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) S[PAIRED ? R * rx + i : rx + 8 * i][cy + 8 * j] = acc[i][j];
    __syncthreads();
}

}  // namespace tnsim
