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

constexpr int TILE_THREADS = 64, TILE_E = 8;   // threads, edge
template <typename C> constexpr int TILE_K = sizeof(C) == 8 ? 64 : 16;   // K step

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

// acc += sum over k < K of OP(la(i, k), lb(k, j)): thread tid holds row tid % 8 and column
// tid / 8.  la and lb give the operands' elements for tile row i / tile column j (zero
// outside them); AK / BK: memory runs along k (consecutive threads then load consecutive k).
// k ascends; SPLIT sums every K step by itself first (rounding of 16-byte elements grows with
// sqrt(16 + K / 16) instead of sqrt(K), for 3 - 6 % more instructions); products of up to
// kPlain64 terms are one run of sums.
template <typename C, bool AK, bool BK, bool SPLIT, typename OP, typename LA, typename LB>
__device__ __forceinline__ void tile_product(int K, LA la, LB lb, C& acc) {
    constexpr int E = TILE_E, KS = TILE_K<C>, PER = E * KS / TILE_THREADS;
    __shared__ C As[KS][E + 1], Bs[KS][E + 1];
    const int tid = threadIdx.x, rx = tid & 7, cy = tid >> 3;
    C na[PER], nb[PER];
    const bool split = SPLIT && K > kPlain64;
    // element e of a K step: (edge index, k) with k running fastest (KF) or slowest
    auto at = [](int e, bool kf, int& i, int& k) {
        if (kf) { k = e % KS; i = e / KS; }
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
    for (int k0 = 0; k0 < K; k0 += KS) {
#pragma unroll
        for (int t = 0; t < PER; ++t) {
            int i, k;
            at(tid + TILE_THREADS * t, AK, i, k);
            As[k][i] = na[t];
            at(tid + TILE_THREADS * t, BK, i, k);
            Bs[k][i] = nb[t];
        }
        __syncthreads();
        if (k0 + KS < K) fetch(k0 + KS);
        C part = {};
        if (!split) part = acc;
        const int kn = min(KS, K - k0);
#pragma unroll 4
        for (int kk = 0; kk < kn; ++kk) OP::op(part, As[kk][rx], Bs[kk][cy]);
        if (split) {
            acc.x += part.x;
            acc.y += part.y;
        } else {
            acc = part;
        }
        __syncthreads();
    }
}

// The tile in shared memory, for outputs that mix entries of several threads.
template <typename C>
__device__ __forceinline__ void tile_share(C (*S)[TILE_E + 1], const C& acc) {
    S[threadIdx.x & 7][threadIdx.x >> 3] = acc;
    __syncthreads();
}

}  // namespace tnsim
