// Read-out of an MPS: amplitudes <x|psi> and transfer-matrix steps for <psi|P|psi>.
//
//  k_amplitudes : <x|psi> = A_0[x_0] A_1[x_1] ... A_{n-1}[x_{n-1}] (Eq. 2 with every
//                 physical leg fixed): one CTA per bitstring carries the row vector
//                 v (<= chi entries, shared memory) across the chain; each step is a
//                 vector-matrix product whose matrix rows are read coalesced.
//  k_amp_group  : the same sums in the same order for a group of bitstrings per cluster.
//  k_transfer1/2: transfer of an environment through site q with a one-qubit operator O,
//                 left:  E'[a,b] = sum_{x,y,p,p'} conj(A[x,p,a]) O[p,p'] E[x,y] A[y,p',b];
//                 right: R'[x,y] = sum conj(A[x,p,a]) O[p,p'] A[y,p',b] R[a,b], stored
//                 transposed (Rt[b][a]).
//  k_close*     : sum_{x,y} E[x,y] Rt[y,x] of many (E, R) pairs.
#include <cooperative_groups.h>

#include "tile8.cuh"
#include "tnsim_internal.h"

namespace cg = cooperative_groups;
namespace tnsim {

template <typename C> __device__ __forceinline__ void cfma_(C& acc, C a, C b) {
    acc.x = fma(a.x, b.x, acc.x); acc.x = fma(-a.y, b.y, acc.x);
    acc.y = fma(a.x, b.y, acc.y); acc.y = fma(a.y, b.x, acc.y);
}
template <typename T>
__global__ void __launch_bounds__(256) k_amplitudes(void* const* __restrict__ sites,
                                                    const int* __restrict__ chi, int n,
                                                    const uint8_t* __restrict__ bits,
                                                    double* __restrict__ amps, int chi_cap) {
    using C = typename CT<T>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* v0 = reinterpret_cast<C*>(smem_raw);
    C* v1 = v0 + chi_cap;
    const int64_t s = blockIdx.x;
    if (threadIdx.x == 0) { v0[0].x = 1; v0[0].y = 0; }
    __syncthreads();
    for (int q = 0; q < n; ++q) {
        const int x = bits[s * n + q] ? 1 : 0;
        const int cl = chi[q], cr = chi[q + 1];
        const C* A = (const C*)sites[q];
        for (int r = threadIdx.x; r < cr; r += blockDim.x) {
            C acc; acc.x = 0; acc.y = 0;
            for (int l = 0; l < cl; ++l) cfma_(acc, v0[l], A[(size_t)(2 * l + x) * cr + r]);
            v1[r] = acc;
        }
        __syncthreads();
        C* t = v0; v0 = v1; v1 = t;
    }
    if (threadIdx.x == 0) {
        amps[2 * s] = (double)v0[0].x;
        amps[2 * s + 1] = (double)v0[0].y;
    }
}

// complex64, many bitstrings, large bonds: one CTA per bitstring read every site from L2
// for each string (46 GB for 1024 strings of 100 sites at chi 256: 7.9 ms, bound by L2).
// Here a cluster carries S bitstrings, CTA r of it the columns [64 r, 64 r + 64): the site's
// tile is read once per cluster (2.8 GB), and the new entries of the S row vectors go to
// every CTA of the cluster through distributed shared memory.  A warp holds four strings by
// 64 columns (two per lane), so a tile element feeds four FMA groups: FP32-bound.  The
// strings are ordered by their bit at this site, so a warp's four strings share a matrix
// (A[2l] or A[2l + 1]) except in at most one warp.  Tiles of 16 rows of l arrive by
// asynchronous copies, three chunks ahead; a site's first chunks are requested before the
// cluster's barrier of the site before.
constexpr int AG_K = 16, AG_ST = 4;

template <int MODE>   // strings' bits: 0, 1: all equal; 2: mixed
__device__ __forceinline__ void amp_step(float4 (&acc)[4], const float4* __restrict__ tile, const float2 (&v)[4],
                                         const bool (&one)[4]) {
    float4 a0, a1;
    if (MODE != 1) a0 = tile[0];
    if (MODE != 0) a1 = tile[32];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 a = MODE == 0 ? a0 : MODE == 1 ? a1 : (one[i] ? a1 : a0);
        acc[i].x = fmaf(v[i].x, a.x, acc[i].x);
        acc[i].x = fmaf(-v[i].y, a.y, acc[i].x);
        acc[i].y = fmaf(v[i].x, a.y, acc[i].y);
        acc[i].y = fmaf(v[i].y, a.x, acc[i].y);
        acc[i].z = fmaf(v[i].x, a.z, acc[i].z);
        acc[i].z = fmaf(-v[i].y, a.w, acc[i].z);
        acc[i].w = fmaf(v[i].x, a.w, acc[i].w);
        acc[i].w = fmaf(v[i].y, a.z, acc[i].w);
    }
}
template <int MODE>
__device__ __forceinline__ void amp_chunk(float4 (&acc)[4], const float4* __restrict__ tile,
                                          const float2* const (&v)[4], int k0, int kn, const bool (&one)[4]) {
    int k = 0;
    for (; k + 2 <= kn; k += 2) {
        float2 va[4], vb[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 t = *reinterpret_cast<const float4*>(v[i] + k0 + k);
            va[i] = make_float2(t.x, t.y);
            vb[i] = make_float2(t.z, t.w);
        }
        amp_step<MODE>(acc, tile + k * 64, va, one);
        amp_step<MODE>(acc, tile + k * 64 + 64, vb, one);
    }
    if (k < kn) {
        float2 va[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) va[i] = v[i][k0 + k];
        amp_step<MODE>(acc, tile + k * 64, va, one);
    }
}

template <int S>
__global__ void __launch_bounds__(S * 8) k_amp_group(void* const* __restrict__ sites, const int* __restrict__ chi,
                                                     int n, const uint8_t* __restrict__ bits, int64_t n_str,
                                                     double* __restrict__ amps, int pitch) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cg::cluster_group cl = cg::this_cluster();
    const int ranks = (int)cl.num_blocks(), rank = (int)cl.block_rank(), c0 = 64 * rank;
    const int64_t s0 = (int64_t)(blockIdx.x / ranks) * S;
    float2* const vbuf = reinterpret_cast<float2*>(smem_raw);                    // [2][S][pitch]
    float4* const tiles = reinterpret_cast<float4*>(vbuf + (size_t)2 * S * pitch); // [AG_ST][AG_K][2][32]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int s = tid; s < S; s += S * 8) vbuf[(size_t)s * pitch] = make_float2(1.f, 0.f);
    cl.sync();
    auto bit_at = [&](int q) { return lane < S && s0 + lane < n_str && q < n ? (int)bits[(s0 + lane) * n + q] : 0; };
    int bit = bit_at(0);
    for (int q = 0; q < n; ++q) {
        const int rl = chi[q], cr = chi[q + 1];
        const int nk = c0 < cr ? (rl + AG_K - 1) / AG_K : 0, nc = min(64, cr - c0);
        const float2* A = (const float2*)sites[q] + c0;
        const bool wide = (cr & 1) == 0;   // 16-byte rows
        auto request = [&](int k) {
            if (k < nk) {
                float4* dst = tiles + (k % AG_ST) * (AG_K * 64);
                const int rows = 2 * min(AG_K, rl - k * AG_K);
                const float2* src = A + (size_t)(2 * k * AG_K) * cr;
                if (wide) {
                    for (int u = tid; u < rows * 32; u += S * 8) {
                        const int r = u >> 5, c = u & 31;
                        if (2 * c < nc) {
                            const unsigned a = (unsigned)__cvta_generic_to_shared(dst + u);
                            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(a), "l"(src + (size_t)r * cr + 2 * c) : "memory");
                        }
                    }
                } else {
                    for (int u = tid; u < rows * 64; u += S * 8) {
                        const int r = u >> 6, c = u & 63;
                        if (c < nc) {
                            const unsigned a = (unsigned)__cvta_generic_to_shared(reinterpret_cast<float2*>(dst) + u);
                            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(a), "l"(src + (size_t)r * cr + c) : "memory");
                        }
                    }
                }
            }
            asm volatile("cp.async.commit_group;\n" ::: "memory");
        };
        for (int k = 0; k < AG_ST - 1; ++k) request(k);
        // this warp's strings: positions 4 warp .. 4 warp + 3 of the order (bit 0 first)
        const unsigned ones = __ballot_sync(0xffffffffu, bit != 0) & (S == 32 ? 0xffffffffu : (1u << S) - 1u);
        const int n0 = S - __popc(ones);
        const unsigned below = (1u << lane) - 1u;
        const int pos = lane >= S ? S : (bit ? n0 + __popc(ones & below) : lane - __popc(ones & below));
        int str[4];
        bool one[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            str[i] = __ffs(__ballot_sync(0xffffffffu, pos == 4 * warp + i)) - 1;
            one[i] = 4 * warp + i >= n0;
        }
        bit = bit_at(q + 1);
        if (q > 0) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");   // the entries of site q - 1
        const float2* v[4];
        float4 acc[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[i] = vbuf + ((size_t)(q & 1) * S + str[i]) * pitch;
            acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        for (int k = 0; k < nk; ++k) {
            asm volatile("cp.async.wait_group %0;\n" ::"n"(AG_ST - 2) : "memory");
            __syncthreads();
            request(k + AG_ST - 1);
            const float4* tile = tiles + (k % AG_ST) * (AG_K * 64) + lane;
            const int kn = min(AG_K, rl - k * AG_K);
            if (!one[3]) amp_chunk<0>(acc, tile, v, k * AG_K, kn, one);
            else if (one[0]) amp_chunk<1>(acc, tile, v, k * AG_K, kn, one);
            else amp_chunk<2>(acc, tile, v, k * AG_K, kn, one);
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        __syncthreads();   // before the next site's requests reuse the stages
        if (c0 + 2 * lane < cr) {
            for (int r = 0; r < ranks; ++r) {
                float2* dst = cl.map_shared_rank(vbuf, r) + (size_t)((q + 1) & 1) * S * pitch + c0 + 2 * lane;
#pragma unroll
                for (int i = 0; i < 4; ++i) *reinterpret_cast<float4*>(dst + (size_t)str[i] * pitch) = acc[i];
            }
        }
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    }
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    if (rank == 0 && tid < S && s0 + tid < n_str) {
        const float2 z = vbuf[((size_t)(n & 1) * S + tid) * pitch];
        amps[2 * (s0 + tid)] = (double)z.x;
        amps[2 * (s0 + tid) + 1] = (double)z.y;
    }
}

template <int S>
static cudaError_t launch_amp_group(void* const* sites, const int* chi, int n, int ranks, int pitch,
                                    const uint8_t* bits, int64_t n_str, double* amps, cudaStream_t s) {
    const size_t smem = (size_t)2 * S * pitch * sizeof(float2) + (size_t)AG_ST * AG_K * 64 * sizeof(float4);
    static SmemLimit limit;
    cudaError_t e = allow_dynamic_smem((const void*)k_amp_group<S>, limit);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = ranks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)((n_str + S - 1) / S * ranks));
    cfg.blockDim = dim3(S * 8);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_amp_group<S>, sites, chi, n, bits, n_str, amps, pitch);
}

template <typename T>
cudaError_t launch_amplitudes(void* const* sites, const int* chi, int n_qubits, int chi_cap,
                              const uint8_t* bits, int64_t n_str, double* amps, cudaStream_t s) {
    using C = typename CT<T>::type;
    if (n_str <= 0) return cudaSuccess;
    if constexpr (sizeof(T) == 4) {
        // groups of strings pay where a site's tile is large and several strings share it;
        // the group is as large as the row vectors leave room for (two of S x chi) and as
        // still gives work to most SMs
        int ranks = 1;
        while (64 * ranks < chi_cap) ranks *= 2;
        const int pitch = (chi_cap + 1) & ~1;
        if (chi_cap >= 48 && ranks <= 8 && n_str >= 8 && (n_str + 7) / 8 * ranks <= 0x7fffffff) {
            int S = chi_cap <= 256 ? 32 : 16;
            while (S > 8 && (n_str + S - 1) / S * ranks < 100) S /= 2;
            if (S == 32) return launch_amp_group<32>(sites, chi, n_qubits, ranks, pitch, bits, n_str, amps, s);
            if (S == 16) return launch_amp_group<16>(sites, chi, n_qubits, ranks, pitch, bits, n_str, amps, s);
            return launch_amp_group<8>(sites, chi, n_qubits, ranks, pitch, bits, n_str, amps, s);
        }
    }
    const size_t smem = 2 * (size_t)chi_cap * sizeof(C);
    static SmemLimit limit;
    cudaError_t e = allow_dynamic_smem((const void*)k_amplitudes<T>, limit);
    if (e != cudaSuccess) return e;
    k_amplitudes<T><<<(unsigned)n_str, 256, smem, s>>>(sites, chi, n_qubits, bits, amps, chi_cap);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Transfer steps, two products each (d.left: from the left):
//   left   w[(x, p), b] = sum_{p'} O[p,p'] sum_y E[x, y] A[y, p', b]
//          E'[a, b] = sum_{x,p} conj(A[x,p,a]) w[(x, p), b]
//   right  (Rt[b][a] = R[a][b], a: bra, b: ket on bond q + 1)
//          w[y, (a, p)] = sum_{p'} O[p,p'] sum_b A[y, p', b] Rt[b, a]
//          Rt'[y, x] = sum_{a,p} w[y, (a, p)] conj(A[x,p,a])
// Small tiles over a grid of (tiles, steps): a step's time is its latency, so small tiles
// over many SMs, and every step that does not depend on another in the same launch.  (One
// thread per element, with its operands from L2 on every k: 21 + 38 us per step at chi 64,
// complex64, against 7 + 9.)  The sums keep the order of that form, k ascending in
// one accumulator, then p'.
template <typename T>
__global__ void __launch_bounds__(TILE_THREADS) k_transfer1(const TransferDesc* __restrict__ list, TransferDesc one) {
    using C = typename CT<T>::type;
    constexpr int E = TILE_E, H = E / 2;
    const TransferDesc& d = list ? list[blockIdx.y] : one;
    if (!d.site) return;
    const int cl = d.chi[d.q], cr = d.chi[d.q + 1];
    // left: tile of E rows x and H columns b for both p'; right: H rows y for both p', E columns a
    const int nx = d.left ? cl : cr, nh = d.left ? cr : cl, K = d.left ? cl : cr;
    const int th = (nh + H - 1) / H, x0 = (int)(blockIdx.x / th) * E, h0 = (int)(blockIdx.x % th) * H;
    if (x0 >= nx) return;
    const C* site = (const C*)d.site;
    const C* env = (const C*)d.e_in;
    C acc = {};
    if (d.left)
        tile_product<C, true, false, false, MulAdd>(
            K, [&](int i, int k) { return x0 + i < cl ? env[(size_t)(x0 + i) * cl + k] : C{}; },
            [&](int k, int j) {
                const int b = h0 + j % H;
                return b < cr ? site[((size_t)k * 2 + j / H) * cr + b] : C{};
            },
            acc);
    else
        tile_product<C, true, false, false, MulAdd>(
            K,
            [&](int i, int k) {
                const int y = h0 + i % H;
                return y < cl ? site[((size_t)y * 2 + i / H) * cr + k] : C{};
            },
            [&](int k, int j) { return x0 + j < cr ? env[(size_t)k * cr + x0 + j] : C{}; }, acc);
    __shared__ C S[E][E + 1];
    tile_share(S, acc);
    C o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) { o[i].x = (T)d.op[2 * i]; o[i].y = (T)d.op[2 * i + 1]; }
    C* tmp = (C*)d.tmp;
    for (int e = threadIdx.x; e < E * E; e += TILE_THREADS) {
        // p, index h of the halved side, index x of the full side; consecutive threads write
        // consecutive elements
        const int p = d.left ? e / H % 2 : e % 2;
        const int h = d.left ? e % H : e / (2 * E), x = d.left ? e / E : e / 2 % E;
        if (h0 + h >= nh || x0 + x >= nx) continue;
        const C t0 = d.left ? S[x][h] : S[h][x], t1 = d.left ? S[x][H + h] : S[H + h][x];
        C w = {};
        MulAdd::op(w, p ? o[2] : o[0], t0);
        MulAdd::op(w, p ? o[3] : o[1], t1);
        const size_t g = d.left ? ((size_t)(x0 + x) * 2 + p) * cr + h0 + h : (size_t)(h0 + h) * 2 * cr + 2 * (x0 + x) + p;
        tmp[g] = w;
    }
}

template <typename T>
__global__ void __launch_bounds__(TILE_THREADS) k_transfer2(const TransferDesc* __restrict__ list, TransferDesc one) {
    using C = typename CT<T>::type;
    constexpr int TE = TILE_E;
    const TransferDesc& d = list ? list[blockIdx.y] : one;
    if (!d.site) return;
    const int cl = d.chi[d.q], cr = d.chi[d.q + 1];
    const int M = d.left ? cr : cl, K = d.left ? 2 * cl : 2 * cr;   // M x M output
    const int tn = (M + TE - 1) / TE, i0 = (int)(blockIdx.x / tn) * TE, j0 = (int)(blockIdx.x % tn) * TE;
    if (i0 >= M) return;
    const C* A = (const C*)d.site;
    const C* w = (const C*)d.tmp;
    C acc = {};
    if (d.left)
        tile_product<C, false, false, false, ConjMulAdd>(
            K, [&](int i, int k) { return i0 + i < M ? A[(size_t)k * cr + i0 + i] : C{}; },
            [&](int k, int j) { return j0 + j < M ? w[(size_t)k * cr + j0 + j] : C{}; }, acc);
    else
        tile_product<C, true, true, false, MulAddConj>(
            K, [&](int i, int k) { return i0 + i < M ? w[(size_t)(i0 + i) * K + k] : C{}; },
            [&](int k, int j) { return j0 + j < M ? A[(size_t)(2 * (j0 + j) + (k & 1)) * cr + (k >> 1)] : C{}; }, acc);
    C* out = (C*)d.e_out;
    const int r = i0 + (threadIdx.x & 7), c = j0 + (threadIdx.x >> 3);
    if (r < M && c < M) out[(size_t)r * M + c] = acc;
}

// out[l, p, r] += coef sum_{l'} E[l, l'] w[l', (r, p)]  (E: left environment, bra x ket)
template <typename T>
__global__ void __launch_bounds__(TILE_THREADS) k_site_adj(const SiteAdjDesc* __restrict__ list) {
    using C = typename CT<T>::type;
    constexpr int TE = TILE_E;
    const SiteAdjDesc& d = list[blockIdx.y];
    const int cl = d.chi[d.q], cr = d.chi[d.q + 1], N = 2 * cr;
    const int tn = (N + TE - 1) / TE, i0 = (int)(blockIdx.x / tn) * TE, j0 = (int)(blockIdx.x % tn) * TE;
    if (i0 >= cl) return;
    const C* E = (const C*)d.E;
    const C* w = (const C*)d.w;
    C acc = {};
    tile_product<C, true, false, false, MulAddIm>(
        cl, [&](int i, int k) { return i0 + i < cl ? E[(size_t)(i0 + i) * cl + k] : C{}; },
        [&](int k, int j) { return j0 + j < N ? w[(size_t)k * N + j0 + j] : C{}; }, acc);
    C* out = (C*)d.out;
    const T f = (T)d.coef;
    const int l = i0 + (threadIdx.x & 7), c = j0 + (threadIdx.x >> 3);
    if (l >= cl || c >= N) return;
    C* o = out + ((size_t)l * 2 + (c & 1)) * cr + (c >> 1);
    o->x += f * acc.x;
    o->y += f * acc.y;
}

// Steps of a list go to grid.y, which ends at 65535: f(first, count) for parts of a list.
template <typename F>
static cudaError_t in_parts(int count, F f) {
    for (int first = 0; first < count; first += kMaxGridY) {
        f(first, min(kMaxGridY, count - first));
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename T>
cudaError_t launch_transfers(const TransferDesc* list, const TransferDesc& one, int count, int chi_cap,
                             cudaStream_t s) {
    constexpr int E = TILE_E;
    const int te = (chi_cap + E - 1) / E, th = (chi_cap + E / 2 - 1) / (E / 2);
    return in_parts(count, [&](int first, int part) {
        const TransferDesc* l = list ? list + first : nullptr;
        k_transfer1<T><<<dim3(te * th, part), TILE_THREADS, 0, s>>>(l, one);
        k_transfer2<T><<<dim3(te * te, part), TILE_THREADS, 0, s>>>(l, one);
    });
}
template <typename T>
cudaError_t launch_transfer(const void* site, const int* chi, int q, const double* op,
                            const void* e_in, void* tmp, void* e_out, int chi_cap,
                            int from_left, cudaStream_t s) {
    return launch_transfers<T>(nullptr, TransferDesc{site, chi, op, e_in, tmp, e_out, q, from_left}, 1, chi_cap, s);
}

template <typename T>
cudaError_t launch_site_adjs(const TransferDesc* t, const SiteAdjDesc* a, int count, int chi_cap, cudaStream_t s) {
    constexpr int E = TILE_E;
    const int te = (chi_cap + E - 1) / E, th = (chi_cap + E / 2 - 1) / (E / 2), t2 = (2 * chi_cap + E - 1) / E;
    return in_parts(count, [&](int first, int part) {
        k_transfer1<T><<<dim3(te * th, part), TILE_THREADS, 0, s>>>(t + first, TransferDesc{});
        k_site_adj<T><<<dim3(te * t2, part), TILE_THREADS, 0, s>>>(a + first);
    });
}
template cudaError_t launch_site_adjs<float>(const TransferDesc*, const SiteAdjDesc*, int, int, cudaStream_t);
template cudaError_t launch_site_adjs<double>(const TransferDesc*, const SiteAdjDesc*, int, int, cudaStream_t);
template cudaError_t launch_transfers<float>(const TransferDesc*, const TransferDesc&, int, int, cudaStream_t);
template cudaError_t launch_transfers<double>(const TransferDesc*, const TransferDesc&, int, int, cudaStream_t);

// Closure: out = sum_{x,y} E[x,y] Rt[y,x] over one bond, E and Rt both chi x chi.  CLOSE_PARTS
// CTAs per pair, then one thread per pair adds their sums in order.  Products and sums are
// FP64 for complex64 too: each environment of an unnormalised state may fill FP32's range by
// itself.  (FP32 pairs are no faster -- 99 terms at chi 64 take 1.06 ms with both -- and give 0
// or infinity below a squared norm of 1e-31 or above 1e38.)
template <typename T>
__global__ void __launch_bounds__(256) k_close(const CloseDesc* __restrict__ list, double* __restrict__ parts) {
    using C = typename CT<T>::type;
    const CloseDesc d = list[blockIdx.y];
    const int c = d.chi[d.bond];
    const C* E = (const C*)d.e;
    const C* Rt = (const C*)d.rt;
    double a = 0.0, b = 0.0;
    for (int t = blockIdx.x * 256 + threadIdx.x; t < c * c; t += CLOSE_PARTS * 256) {
        const int x = t / c, y = t - x * c;
        const C e = E[t], r = Rt[(size_t)y * c + x];
        const double ex = e.x, ey = e.y, rx = r.x, ry = r.y;
        a = fma(ex, rx, a);
        a = fma(-ey, ry, a);
        b = fma(ex, ry, b);
        b = fma(ey, rx, b);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    __shared__ double2 red[8];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_double2(a, b);
    __syncthreads();
    if (threadIdx.x < 2) {
        double v = 0.0;
        for (int w = 0; w < 8; ++w) v += threadIdx.x ? red[w].y : red[w].x;
        parts[((size_t)blockIdx.y * CLOSE_PARTS + blockIdx.x) * 2 + threadIdx.x] = v;
    }
}
__global__ void k_close_sum(const double* __restrict__ parts, int count, double* __restrict__ out) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 2 * count) return;
    double v = 0.0;
    for (int p = 0; p < CLOSE_PARTS; ++p) v += parts[((size_t)(t >> 1) * CLOSE_PARTS + p) * 2 + (t & 1)];
    out[t] = v;
}

template <typename T>
cudaError_t launch_close(const CloseDesc* list, int count, double* parts, double* out, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    const cudaError_t e = in_parts(count, [&](int first, int part) {
        k_close<T><<<dim3(CLOSE_PARTS, part), 256, 0, s>>>(list + first, parts + (size_t)2 * CLOSE_PARTS * first);
    });
    if (e != cudaSuccess) return e;
    k_close_sum<<<(2 * count + 127) / 128, 128, 0, s>>>(parts, count, out);
    return cudaGetLastError();
}

template cudaError_t launch_amplitudes<float>(void* const*, const int*, int, int, const uint8_t*, int64_t, double*, cudaStream_t);
template cudaError_t launch_amplitudes<double>(void* const*, const int*, int, int, const uint8_t*, int64_t, double*, cudaStream_t);
template cudaError_t launch_transfer<float>(const void*, const int*, int, const double*, const void*, void*, void*, int, int, cudaStream_t);
template cudaError_t launch_transfer<double>(const void*, const int*, int, const double*, const void*, void*, void*, int, int, cudaStream_t);
template cudaError_t launch_close<float>(const CloseDesc*, int, double*, double*, cudaStream_t);
template cudaError_t launch_close<double>(const CloseDesc*, int, double*, double*, cudaStream_t);

}  // namespace tnsim
