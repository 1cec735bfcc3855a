// A 16 x 16 tile of a complex product by 64 threads, shared by the FP64 products
// (k_fp64.cu) and the read-out (k_readout.cu).
//
// Small tiles: FP64 issues at 1/64 of the FP32 rate, and the read-out's products are
// chains of small matrices, so a tile's time is its latency and what counts is how many
// SMs share a product.  The next K step's operands are loaded while this one's are used.
#pragma once
#include <cuda_runtime.h>

namespace tnsim {

constexpr int TILE = 16;           // tile edge and K step
constexpr int TILE_THREADS = 64;   // 2 x 2 outputs per thread

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
struct MulAddConj {
    template <typename C> static __device__ __forceinline__ void op(C& acc, const C& a, const C& b) {
        ConjMulAdd::op(acc, b, a);
    }
};

// acc += sum over k < K of OP(la(i, k), lb(k, j)): thread (rx, cy) = (tid % 8, tid / 8)
// holds rows rx + 8 i (PAIRED: 2 rx + i) and columns cy + 8 j.  la and lb give the
// operands' elements for tile row i / tile column j (zero outside them); AK / BK: memory
// runs along k (consecutive threads then load consecutive k).  k ascends; SPLIT sums every
// K step by itself first (rounding grows with sqrt(16 + K / 16) instead of sqrt(K), for
// 3 % more instructions).
template <typename C, bool AK, bool BK, bool PAIRED, bool SPLIT, typename OP, typename LA, typename LB>
__device__ __forceinline__ void tile_product(int K, LA la, LB lb, C (&acc)[2][2]) {
    constexpr int PER = TILE * TILE / TILE_THREADS;
    __shared__ C As[TILE][TILE + 1], Bs[TILE][TILE + 1];
    const int tid = threadIdx.x, rx = tid & 7, cy = tid >> 3;
    C na[PER], nb[PER];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int t = 0; t < PER; ++t) {
            const int e = tid + TILE_THREADS * t, lo = e & (TILE - 1), hi = e / TILE;
            na[t].x = na[t].y = nb[t].x = nb[t].y = 0;
            if (k0 + (AK ? lo : hi) < K) na[t] = la(AK ? hi : lo, k0 + (AK ? lo : hi));
            if (k0 + (BK ? lo : hi) < K) nb[t] = lb(k0 + (BK ? lo : hi), BK ? hi : lo);
        }
    };
    fetch(0);
    for (int k0 = 0; k0 < K; k0 += TILE) {
#pragma unroll
        for (int t = 0; t < PER; ++t) {
            const int e = tid + TILE_THREADS * t, lo = e & (TILE - 1), hi = e / TILE;
            As[AK ? lo : hi][AK ? hi : lo] = na[t];
            Bs[BK ? lo : hi][BK ? hi : lo] = nb[t];
        }
        __syncthreads();
        if (k0 + TILE < K) fetch(k0 + TILE);
        C part[2][2] = {};
#pragma unroll 4
        for (int kk = 0; kk < TILE; ++kk) {
            C a[2], b[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                a[i] = As[kk][PAIRED ? 2 * rx + i : rx + 8 * i];
                b[i] = Bs[kk][cy + 8 * i];
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) OP::op(SPLIT ? part[i][j] : acc[i][j], a[i], b[j]);
        }
        if (SPLIT) {
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) { acc[i][j].x += part[i][j].x; acc[i][j].y += part[i][j].y; }
        }
        __syncthreads();
    }
}

}  // namespace tnsim
