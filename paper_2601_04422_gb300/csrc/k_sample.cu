// Perfect sampling of an MPS with memoised prefixes (Sec. III.A "Sampling",
// Sec. IV.A measurement).
//
// Shot s draws qubit q from the weights of its two outcomes given its bits so far:
// with v the (normalised) row vector of its prefix and R_{q+1} the right environment
// of bond q+1,
//     w_b = v A_q[:, b, :],   p_b = w_b R_{q+1} w_b^H,
//     b_q = 1  exactly when  u[s, q] (p0 + p1) >= p0,
// and the prefix becomes w_b / sqrt(p_b) (projection on the outcome, renormalised).
// Using R_{q+1} gives the same weights as first bringing the MPS to right-canonical
// form (where every right environment is the identity).
//
// Memoisation: shots with the same prefix share v, so each site works on the
// distinct prefixes ("nodes") only -- at most min(shots, 2^q) of them -- and a shot
// just carries the index of its node.  Per site:
//   k_nodes      v = w_b / sqrt(p_b) of the parents, W = v A_q (nodes x 2 chi_R),
//                Y = W' Rt_{q+1} (2 nodes x chi_R; W' = W as rows (node, b)) and
//                p[(node, b)] = Re <w, y> (FP64 sums), a few nodes per CTA
//   k_draw       every shot: its bit from its uniform, and mark child (node, bit); number
//                the marked children, which are the next site's nodes; every shot moves
//                to its child (more than 8192 shots: k_decide, k_scan and k_advance)
// The node count lives in device memory; grids are sized by the host bound
// min(shots, 2^q) and the kernels read the actual count.
// A site is a chain of small steps, so its launches and passes over memory were what it
// cost: as two 64 x 64-tiled products (64 CTAs), a row product, a projection and the draw in
// four more launches, 1024 shots over 64 sites at chi 128 took 5.8 ms, 3.5 now.
#include <algorithm>

#include "tnsim_internal.h"

namespace tnsim {

namespace {

template <typename C>
__device__ __forceinline__ void cmac(C& acc, const C& a, const C& b) {
    acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
    acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
}

// NR = 2 RT nodes per CTA, every column of their rows: W and the weights need no other CTA.
// Every CTA reads all of A_q and Rt, in tiles of 64 KB that asynchronous copies bring while
// the one before is used: that much in flight hides L2 (loads into registers, 16 rows ahead,
// left the FMAs at a quarter of their rate; tiles shared by clusters of four through
// distributed shared memory were no faster).  A thread owns two adjacent columns of RT rows:
// 8 RT FMAs for a 16-byte load of the tile and RT halves of broadcast ones of the nodes'
// rows.  v comes scaled from the parents' rows.
//   phase 1: 128 pairs of the 2 cr columns by 2 groups of rows
//   phase 2: 64 pairs of the cr columns by 2 outcomes by 2 groups of rows
constexpr int NODE_THREADS = 256, NODE_P = NODE_THREADS / 2;
constexpr int NODE_TILE = 64 << 10;   // bytes
template <typename C> struct NodeK { static constexpr int K = 1024 / sizeof(C); };   // nodes' elements in shared memory
// 16 (8) bytes, the first have of them from memory and zeros after
__device__ __forceinline__ void copy16(void* dst, const void* src, int have) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(have) : "memory");
}
__device__ __forceinline__ void copy8(void* dst, const void* src, int have) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(have) : "memory");
}
// acc[i][0, 1] += sum_k S[r0 + i][h][k] B[k][c0 + cp, c0 + cp + 1] for the NC columns from c0
// (nc in all); la(k, kn) brings the next elements of the nodes' rows into S, zeros beyond.
template <typename C, int RT, int NC, typename LA>
__device__ __forceinline__ void node_rows(C (&acc)[RT][2], const C* __restrict__ B, int ldb, int c0, int cp, int nc, int K,
                                          int r0, int h, C (*S)[2][NodeK<C>::K], C* tiles, LA la) {
    constexpr int SK = NodeK<C>::K, V = 16 / sizeof(C), TE = NODE_TILE / sizeof(C), KC = TE / NC;
    static_assert(SK % KC == 0, "whole tiles");
    auto fetch = [&](C* tile, int k) {
        if (ldb % V == 0 && c0 % V == 0 && (reinterpret_cast<size_t>(B) & 15) == 0) {
#pragma unroll 4
            for (int e = threadIdx.x; e < TE / V; e += NODE_THREADS) {
                const int row = e / (NC / V), col = e % (NC / V) * V;
                const int have = k + row < K ? min(max(nc - c0 - col, 0), V) * (int)sizeof(C) : 0;
                copy16(tile + row * NC + col, have ? B + (size_t)(k + row) * ldb + c0 + col : B, have);
            }
        } else {   // complex64, rows that start on 8 bytes
            for (int e = threadIdx.x; e < TE; e += NODE_THREADS) {
                const int row = e / NC, col = e % NC;
                const int have = k + row < K && c0 + col < nc ? 8 : 0;
                copy8(tile + row * NC + col, have ? B + (size_t)(k + row) * ldb + c0 + col : B, have);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    __syncthreads();   // the last phase's tiles and S are free
    fetch(tiles, 0);
    for (int k = 0, turn = 0; k < K; k += KC, ++turn) {
        if (k % SK == 0) {
            if (k > 0) __syncthreads();
            la(k, min(SK, K - k));
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        if (k + KC < K) fetch(tiles + (size_t)((turn + 1) & 1) * TE, k + KC);
        const C* tile = tiles + (size_t)(turn & 1) * TE;
        const int kn = min(KC, (K - k + V - 1) / V * V);
#pragma unroll 4
        for (int kk = 0; kk < kn; kk += V) {
            union { float4 f[2]; C c[V][2]; } b;   // V rows, two columns
            b.f[0] = *reinterpret_cast<const float4*>(tile + kk * NC + cp);
            b.f[1] = *reinterpret_cast<const float4*>(V == 2 ? tile + (kk + 1) * NC + cp : tile + kk * NC + cp + 1);
#pragma unroll
            for (int i = 0; i < RT; ++i) {
                union { float4 f; C c[V]; } a;
                a.f = *reinterpret_cast<const float4*>(&S[r0 + i][h][k % SK + kk]);
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    cmac(acc[i][0], a.c[v], b.c[v][0]);
                    cmac(acc[i][1], a.c[v], b.c[v][1]);
                }
            }
        }
    }
}
// 1 / sqrt(p) rounded to T; FP32: FP64's 150 dependent instructions take 10 k cycles, two
// Newton steps on the FP32 estimate 1 k
__device__ __forceinline__ void inv_sqrt(double p, double& r) { r = p > 0.0 ? 1.0 / sqrt(p) : 0.0; }
__device__ __forceinline__ void inv_sqrt(double p, float& r) {
    if (p > 1e-30 && p < 1e30) {
        double y = (double)rsqrtf((float)p);
        y = fma(y, fma(-0.5 * p * y, y, 0.5), y);
        y = fma(y, fma(-0.5 * p * y, y, 0.5), y);
        r = (float)y;
    } else {
        r = (float)(p > 0.0 ? 1.0 / sqrt(p) : 0.0);
    }
}
template <typename T, int RT>
__global__ void __launch_bounds__(NODE_THREADS)
k_nodes(const typename CT<T>::type* __restrict__ Wp, const double* __restrict__ pp, const int* __restrict__ parent,
        const int* __restrict__ nodes, int cl, int cr, const typename CT<T>::type* __restrict__ A,
        const typename CT<T>::type* __restrict__ Rt, typename CT<T>::type* Wn, double* __restrict__ p) {
    using C = typename CT<T>::type;
    constexpr int NR = 2 * RT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* tiles = reinterpret_cast<C*>(smem_raw);
    const int M = *nodes, i0 = blockIdx.x * NR, tid = threadIdx.x;
    if (i0 >= M) return;
    __shared__ __align__(16) C S[NR][2][NodeK<C>::K];
    __shared__ double prod[2 * NR][NODE_P + 1];
    __shared__ const C* s_row[NR];
    __shared__ T s_sc[NR];
    if (tid < NR && i0 + tid < M) {
        const int k = parent[i0 + tid];
        const double pk = pp[k];
        s_row[tid] = Wp + (size_t)k * cl;
        inv_sqrt(pk, s_sc[tid]);
    }
    for (int c0 = 0; c0 < 2 * cr; c0 += 2 * NODE_P) {
        const int cp = 2 * (tid % NODE_P), c = c0 + cp, r0 = tid / NODE_P * RT;
        C acc[RT][2] = {};
        node_rows<C, RT, 2 * NODE_P>(acc, A, 2 * cr, c0, cp, 2 * cr, cl, r0, 0, S, tiles, [&](int k0, int kn) {
            for (int e = tid; e < NR * NodeK<C>::K; e += NODE_THREADS) {
                const int i = e / NodeK<C>::K, k = e % NodeK<C>::K;
                C v;
                v.x = v.y = 0;
                if (k < kn && i0 + i < M) {
                    v = s_row[i][k0 + k];
                    v.x *= s_sc[i];
                    v.y *= s_sc[i];
                }
                S[i][0][k] = v;
            }
        });
        if (c < 2 * cr)
#pragma unroll
            for (int i = 0; i < RT; ++i)
                if (i0 + r0 + i < M) {
                    Wn[(size_t)(i0 + r0 + i) * 2 * cr + c] = acc[i][0];
                    Wn[(size_t)(i0 + r0 + i) * 2 * cr + c + 1] = acc[i][1];
                }
    }
    constexpr int PER = NODE_THREADS / (2 * NR) < 32 ? NODE_THREADS / (2 * NR) : 32;   // threads per row of prod
    const int h = tid / NODE_P, r0 = tid / (NODE_P / 2) % 2 * RT, cp = 2 * (tid % (NODE_P / 2));
    double sum = 0.0;   // of this thread's share of row tid / PER
    for (int c0 = 0; c0 < cr; c0 += NODE_P) {
        const int c = c0 + cp;
        C acc[RT][2] = {};
        node_rows<C, RT, NODE_P>(acc, Rt, cr, c0, cp, cr, cr, r0, h, S, tiles, [&](int k0, int kn) {
            for (int e = tid; e < 2 * NR * NodeK<C>::K; e += NODE_THREADS) {
                const int r = e / NodeK<C>::K, k = e % NodeK<C>::K;
                C v;
                v.x = v.y = 0;
                if (k < kn && i0 + (r >> 1) < M) v = Wn[((size_t)i0 * 2 + r) * cr + k0 + k];
                S[r >> 1][r & 1][k] = v;
            }
        });
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                double t = 0.0;
                if (c + j < cr && i0 + r0 + i < M) {
                    const C w = Wn[((size_t)(i0 + r0 + i) * 2 + h) * cr + c + j];
                    t = (double)w.x * (double)acc[i][j].x + (double)w.y * (double)acc[i][j].y;
                }
                prod[2 * (r0 + i) + h][cp + j] = t;
            }
        __syncthreads();
        if (tid < 2 * NR * PER)
            for (int k = tid % PER; k < NODE_P; k += PER) sum += prod[tid / PER][k];
        __syncthreads();
    }
#pragma unroll
    for (int o = PER / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (tid < 2 * NR * PER && tid % PER == 0 && i0 + (tid / PER >> 1) < M) p[2 * i0 + tid / PER] = sum;
}

// every shot: its bit from its uniform and its node's weights; mark the child
__global__ void k_decide(const double* __restrict__ u, int n, int q, int64_t shots, const int* __restrict__ node_of,
                         const double* __restrict__ p, uint8_t* __restrict__ bits, int* __restrict__ flag) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= shots) return;
    const int i = node_of[s];
    const double p0 = fmax(p[2 * i], 0.0), p1 = fmax(p[2 * i + 1], 0.0);
    const int b = (u[s * n + q] * (p0 + p1) >= p0) ? 1 : 0;
    bits[s * n + q] = (uint8_t)b;
    flag[2 * i + b] = 1;
}

// exclusive scan of the 2 * nodes child flags in one CTA of 1024 threads: child k
// (= 2 node + bit) gets the next site's node index id[k]; parent[id] = k; the new
// node count replaces *nodes and is added to *total
__device__ __forceinline__ void scan_children(const int* flag, int* id, int* parent, int* nodes,
                                              unsigned long long* total) {
    __shared__ int warp_sum[32];
    __shared__ int s_base;
    const int L = 2 * *nodes;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = (L + 1023) / 1024;
    const int lo = min(L, tid * per), hi = min(L, lo + per);
    int local = 0;
    for (int k = lo; k < hi; ++k) local += flag[k];
    // block-wide exclusive scan of the per-thread sums
    int incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int w = warp_sum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += v;
        }
        warp_sum[lane] = w;   // inclusive over warps
        if (lane == 31) s_base = w;
    }
    __syncthreads();
    int run = incl - local + (warp > 0 ? warp_sum[warp - 1] : 0);
    for (int k = lo; k < hi; ++k) {
        if (flag[k]) {
            id[k] = run;
            parent[run] = k;
            ++run;
        } else {
            id[k] = -1;
        }
    }
    __syncthreads();
    if (tid == 0) {
        *nodes = s_base;
        *total += (unsigned long long)s_base;
    }
}

__global__ void __launch_bounds__(1024) k_scan(const int* __restrict__ flag, int* __restrict__ id,
                                               int* __restrict__ parent, int* __restrict__ nodes,
                                               unsigned long long* __restrict__ total) {
    scan_children(flag, id, parent, nodes, total);
}

__global__ void k_advance(int64_t shots, int n, int q, const uint8_t* __restrict__ bits, const int* __restrict__ id,
                          int* __restrict__ node_of) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= shots) return;
    node_of[s] = id[2 * node_of[s] + bits[s * n + q]];
}

// decide, scan and advance in one CTA
constexpr int64_t DRAW_SHOTS = 8192;
__global__ void __launch_bounds__(1024) k_draw(const double* __restrict__ u, int n, int q, int shots, int* node_of,
                                               const double* __restrict__ p, uint8_t* bits, int* flag, int* id,
                                               int* parent, int* nodes, unsigned long long* total) {
    const int L = 2 * *nodes;
    for (int k = threadIdx.x; k < L; k += 1024) flag[k] = 0;
    __syncthreads();
    int child[DRAW_SHOTS / 1024];
#pragma unroll
    for (int j = 0; j < (int)(DRAW_SHOTS / 1024); ++j) {
        const int s = threadIdx.x + 1024 * j;
        if (s >= shots) break;
        const int i = node_of[s];
        const double p0 = fmax(p[2 * i], 0.0), p1 = fmax(p[2 * i + 1], 0.0);
        const int b = (u[(size_t)s * n + q] * (p0 + p1) >= p0) ? 1 : 0;
        bits[(size_t)s * n + q] = (uint8_t)b;
        child[j] = 2 * i + b;
        flag[child[j]] = 1;
    }
    __syncthreads();
    scan_children(flag, id, parent, nodes, total);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < (int)(DRAW_SHOTS / 1024); ++j) {
        const int s = threadIdx.x + 1024 * j;
        if (s < shots) node_of[s] = id[child[j]];
    }
}

}  // namespace

template <typename T>
cudaError_t launch_sample_site(const void* site, int cl, int cr, const void* rt_next, int q, int n,
                               int64_t shots, int node_bound, const double* u, uint8_t* bits,
                               SampleWork& w, cudaStream_t s) {
    using C = typename CT<T>::type;
    if (node_bound < 1) node_bound = 1;
    const C *Wp = (const C*)w.w, *A = (const C*)site, *Rt = (const C*)rt_next;
    C* Wn = (C*)w.w_next;
    // nodes per CTA: 8 use a tile's elements well; where they would leave SMs idle, 2 take
    // half of the time (256 nodes at chi 128: 16 against 28 us; with 1024 nodes the loads of
    // four times the CTAs make it 46 against 29)
    auto launch = [&](auto* kernel, int nr) {
        const unsigned ctas = (unsigned)((node_bound + nr - 1) / nr);
        const cudaError_t er = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * NODE_TILE);
        if (er != cudaSuccess) return er;
        kernel<<<ctas, NODE_THREADS, 2 * NODE_TILE, s>>>(
            Wp, w.p_cur, w.parent, w.nodes, cl, cr, A, Rt, Wn, w.p_next);
        return cudaGetLastError();
    };
    cudaError_t e = node_bound <= 304 ? launch(k_nodes<T, 1>, 2) : launch(k_nodes<T, 4>, 8);
    if (e != cudaSuccess) return e;
    if (shots <= DRAW_SHOTS) {
        k_draw<<<1, 1024, 0, s>>>(u, n, q, (int)shots, w.node_of, w.p_next, bits, w.flag, w.id, w.parent, w.nodes, w.total);
    } else {
        if ((e = cudaMemsetAsync(w.flag, 0, sizeof(int) * 2 * (size_t)node_bound, s)) != cudaSuccess) return e;
        const unsigned gs = (unsigned)((shots + 255) / 256);
        k_decide<<<gs, 256, 0, s>>>(u, n, q, shots, w.node_of, w.p_next, bits, w.flag);
        k_scan<<<1, 1024, 0, s>>>(w.flag, w.id, w.parent, w.nodes, w.total);
        k_advance<<<gs, 256, 0, s>>>(shots, n, q, bits, w.id, w.node_of);
    }
    std::swap(w.w, w.w_next);
    std::swap(w.p_cur, w.p_next);
    return cudaGetLastError();
}

template cudaError_t launch_sample_site<float>(const void*, int, int, const void*, int, int, int64_t, int,
                                               const double*, uint8_t*, SampleWork&, cudaStream_t);
template cudaError_t launch_sample_site<double>(const void*, int, int, const void*, int, int, int64_t, int,
                                                const double*, uint8_t*, SampleWork&, cudaStream_t);

}  // namespace tnsim
