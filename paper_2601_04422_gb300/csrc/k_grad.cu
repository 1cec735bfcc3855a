// Reverse-mode gradient of an energy through the layered MPS simulation (tnsim_grad).
//
// Conventions: for a complex intermediate X the kernels carry Xb = dE/d(conj X), so
// that dE = 2 Re <Xb, dX>.  The forward is the library's own layer path; the
// backward of one two-qubit update (k_gate_bwd, one cluster per gate) follows the
// chain rule of its steps:
//   right site c Y (Y = U^H T, c = |T|_F / |Y|_F):  Yb = c Bb - (dc c / 2K2) Y,
//     dc = 2 Re <Bb, Y>, plus (dc c / 2F2) T into Tb;
//   kept subspace of T (the left site U; the loss depends on U only through
//   span(U) because a gauge change U R, R^H Y leaves the state unchanged):
//     Tb += U Yb + (I - P) Ut S_k^-2 Y + (Z + Z^H) T,   Ut = Ub + T Yb^H,
//     Z = U_D (G o (U_D^H Ut)) U^H,  G_lj = 1 / (s_j^2 - s_l^2) across the cut,
//     P the projector on the nonzero singular directions (columns of the Jacobi
//     matrix W divided by their norms), U_D the discarded nonzero ones; (I - P) Ut is
//     formed as (I - P) Ub (equal, since (I - P) T = 0), and kept directions with
//     s_j <= sqrt(eps) s_max get no inverse factors (a pseudo-inverse cutoff);
//   gate contraction theta = G (uL x uR) M and merge M = A B: the adjoints of the
//     linear maps, and the 4 x 4 adjoint of G (uL x uR) for the one-qubit gates.
// The final-state adjoint uses transfer-matrix environments (k_env_sum,
// k_site_adj in k_readout.cu, k_adj_combine); k_rot_grad turns the 2 x 2 adjoints of every layer's
// one-qubit gates into angle derivatives.
#include <float.h>

#include <algorithm>

#include <cooperative_groups.h>

#include "tnsim_internal.h"

namespace cg = cooperative_groups;
namespace tnsim {

namespace {

template <typename T> struct EpsG;
template <> struct EpsG<float> { static constexpr double v = FLT_EPSILON; };
template <> struct EpsG<double> { static constexpr double v = DBL_EPSILON; };

template <typename C>
__device__ __forceinline__ C cz() { C r; r.x = 0; r.y = 0; return r; }
template <typename C>
__device__ __forceinline__ C cconj(C a) { a.y = -a.y; return a; }
template <typename C>
__device__ __forceinline__ void cmac(C& acc, const C& a, const C& b) {
    acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
    acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
}

// Operand of cl_gemm: element (i, j) = p[i * rs + j * cs], conjugated if conj.  Read from
// L2: other CTAs of the cluster write most operands between the cluster's barriers.
template <typename C>
struct Op {
    const C* p;
    int64_t rs, cs;
    bool conj;
    __device__ __forceinline__ C at(int i, int j) const {
        C v = __ldcg(p + (int64_t)i * rs + (int64_t)j * cs);
        if (conj) v.y = -v.y;
        return v;
    }
};

// Tile edge and K step.  One CTA of 256 threads per gate in 64 x 64 tiles of 4 x 4 outputs
// issued the whole tile's FP64 instructions, mostly zeros, for a 24 x 24 block: 65 us per K
// step (0.97 ms per gate).  A gate is a cluster of kBwdRanks CTAs now, in 16 x 16 tiles of
// one output per thread.
constexpr int GT = 16, GK = 16, kBwdRanks = 8;

__device__ __forceinline__ void cluster_sync() {
    __threadfence();
    cg::this_cluster().sync();
}

// out(i, j) = alpha * sum_k a(i, k) b(k, j) (+ out(i, j) when acc), for i < M, j < N;
// out element (i, j) at o[i * ors + j * ocs].  Whole cluster, tiles in turn; ends with the
// cluster's barrier.
template <typename T, typename C>
__device__ void cl_gemm(int M, int N, int K, Op<C> a, Op<C> b, C* o, int64_t ors, int64_t ocs, T alpha, bool acc,
                        C (*As)[GT + 1], C (*Bs)[GT + 1], int rank) {
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int tm = (M + GT - 1) / GT, tn = (N + GT - 1) / GT;
    for (int tile = rank; tile < tm * tn; tile += kBwdRanks) {
        const int m0 = (tile / tn) * GT, n0 = (tile % tn) * GT;
        C r = cz<C>(), na, nb;
        auto fetch = [&](int k0) {
            na = (m0 + ty < M && k0 + tx < K) ? a.at(m0 + ty, k0 + tx) : cz<C>();   // row ty, k tx
            nb = (k0 + ty < K && n0 + tx < N) ? b.at(k0 + ty, n0 + tx) : cz<C>();   // k ty, column tx
        };
        fetch(0);
        for (int k0 = 0; k0 < K; k0 += GK) {
            As[tx][ty] = na;
            Bs[ty][tx] = nb;
            __syncthreads();
            if (k0 + GK < K) fetch(k0 + GK);
            const int kn = min(GK, K - k0);
#pragma unroll 4
            for (int kk = 0; kk < kn; ++kk) cmac(r, As[kk][ty], Bs[kk][tx]);
            __syncthreads();
        }
        if (m0 + ty < M && n0 + tx < N) {
            C* dst = o + (int64_t)(m0 + ty) * ors + (int64_t)(n0 + tx) * ocs;
            C v;
            v.x = alpha * r.x;
            v.y = alpha * r.y;
            if (acc) {
                const C w = __ldcg(dst);
                v.x += w.x;
                v.y += w.y;
            }
            *dst = v;
        }
    }
    cluster_sync();
}

// block-wide sum of n doubles per thread (n <= 32); result in out[] of every thread
template <int NV>
__device__ void block_sum(double (&v)[NV], double* red /* NV * 32 */) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int i = 0; i < NV; ++i)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    __syncthreads();
    if (lane == 0)
        for (int i = 0; i < NV; ++i) red[i * 32 + warp] = v[i];
    __syncthreads();
    for (int i = 0; i < NV; ++i) {
        double t = 0.0;
        for (int w = 0; w < nw; ++w) t += red[i * 32 + w];
        v[i] = t;
    }
    __syncthreads();
}

// The backward of one two-qubit update (a cluster of kBwdRanks CTAs of 256 threads per gate).
template <typename T>
__global__ void __launch_bounds__(256) k_gate_bwd(const GradGateDesc* __restrict__ gd) {
    using C = typename CT<T>::type;
    const GradGateDesc& d = gd[blockIdx.x / kBwdRanks];
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    __shared__ C As[GK][GT + 1];
    __shared__ C Bs[GK][GT + 1];
    __shared__ double s_part[kBwdRanks][32];
    __shared__ double red[8 * 32];
    __shared__ C Gt[16];
    __shared__ double s_sc[4];
    const int chiL = d.chiL, chiM = d.chiM, chiR = d.chiR, k = d.k;
    const int m = 2 * chiL, n = 2 * chiR;
    const int tid = threadIdx.x, nt = blockDim.x;
    // of the cluster, for the elementwise passes; the mixing pass spreads its few elements
    // over the ranks' schedulers (mid)
    const int gid = rank * nt + tid, gn = kBwdRanks * nt, mid = tid * kBwdRanks + rank;
    const C* Tm = (const C*)d.theta0;        // column-major m x n
    const C* W = (const C*)d.W;              // column-major m x n
    const C* U = (const C*)d.u_post;         // m x k row-major
    const C* cY = (const C*)d.y_post;        // k x n row-major
    const C* Ub = (const C*)d.ub_post;       // m x k
    const C* Bb = (const C*)d.bb_post;       // k x n
    const C* Apre = (const C*)d.a_pre;       // (chiL, 2, chiM) = m x chiM row-major
    const C* Bpre = (const C*)d.b_pre;       // (chiM, 2, chiR) = chiM x n row-major
    // scratch: nine regions of cm^2 elements (cm = 2 chi_cap >= m, n, k), whatever shapes
    // they hold (X1 is m x k in the null-space term, dd x k in the discarded one)
    C* S = (C*)d.scratch;
    const size_t R = (size_t)d.cm * d.cm;
    C* Tb = S;                               // m x n row-major
    C* Yb = S + R;                           // k x n
    C* Ut = S + 2 * R;                       // m x k
    C* Ua = S + 3 * R;                       // m x nz column-major (nonzero left singular vectors)
    C* Q1 = S + 4 * R;                       // nz x k
    C* X1 = S + 5 * R;                       // m x k or dd x k
    C* X2 = S + 6 * R;                       // k x n or dd x n
    C* Mm = S + 7 * R;                       // m x n (merge)
    C* Mb = S + 8 * R;                       // m x n, or k x n

    // scalars: k, norms, nonzero count, renormalisation (one warp: a thread's sum of n
    // FP64 terms takes 64 n cycles)
    if (tid < 32) {
        double f2 = 0.0, k2 = 0.0;
        const double thr = EpsG<T>::v * (double)max(m, n);
        const double smax2 = d.s2[0], cut = thr * thr * smax2;
        int nz = 0;
        for (int j = tid; j < n; j += 32) {
            const double v = d.s2[j];
            f2 += v;
            if (j < k) k2 += v;
            if (j < min(m, n) && v > cut) nz = j + 1;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            f2 += __shfl_xor_sync(0xffffffffu, f2, o);
            k2 += __shfl_xor_sync(0xffffffffu, k2, o);
            nz = max(nz, __shfl_xor_sync(0xffffffffu, nz, o));
        }
        if (sizeof(T) == 8 && plain64(m, n)) {
            // in their order (see kPlain64): lane 0 all, lane 1 the kept ones
            double t = 0.0;
            const int top = tid == 0 ? n : tid == 1 ? k : 0;
            for (int j = 0; j < n; ++j) {
                const double v = d.s2[j];
                if (j < top) t += v;
            }
            f2 = __shfl_sync(0xffffffffu, t, 0);
            k2 = __shfl_sync(0xffffffffu, t, 1);
        }
        if (tid == 0) {
            s_sc[0] = f2;
            s_sc[1] = k2;
            s_sc[2] = (double)max(nz, k);
            s_sc[3] = (d.renorm && k2 > 0.0) ? sqrt(f2 / k2) : 1.0;
        }
    }
    __syncthreads();
    const double F2 = s_sc[0], K2 = s_sc[1], c = s_sc[3];
    const int nz = (int)s_sc[2];
    // dc = 2 Re <Bb, Y>, Y = cY / c
    double dl[1] = {0.0};
    for (int i = tid; i < k * n; i += nt) {
        const C b = Bb[i], y = cY[i];
        dl[0] += (double)b.x * y.x + (double)b.y * y.y;
    }
    block_sum<1>(dl, red);
    const double dldc = 2.0 * dl[0] / c;
    const bool ren = d.renorm && K2 > 0.0;
    // Yb = c Bb - (dc c / 2K2) Y
    {
        const T a1 = (T)c, a2 = ren ? (T)(-dldc * c / (2.0 * K2) / c) : (T)0;
        for (int i = gid; i < k * n; i += gn) {
            const C b = Bb[i], y = cY[i];
            C v;
            v.x = a1 * b.x + a2 * y.x;
            v.y = a1 * b.y + a2 * y.y;
            Yb[i] = v;
        }
    }
    cluster_sync();
    // Tb = U Yb + (dc c / 2F2) T
    cl_gemm<T, C>(m, n, k, Op<C>{U, k, 1, false}, Op<C>{Yb, n, 1, false}, Tb, n, 1, (T)1, false, As, Bs, rank);
    if (ren) {
        const T a3 = (T)(dldc * c / (2.0 * F2));
        for (int i = gid; i < m * n; i += gn) {
            const int row = i / n, col = i % n;
            const C t = Tm[(size_t)col * m + row];
            C v = __ldcg(Tb + i);
            v.x += a3 * t.x;
            v.y += a3 * t.y;
            Tb[i] = v;
        }
        cluster_sync();
    }
    // Ut = Ub + T Yb^H
    for (int i = gid; i < m * k; i += gn) Ut[i] = Ub[i];
    cluster_sync();
    cl_gemm<T, C>(m, k, n, Op<C>{Tm, 1, m, false}, Op<C>{Yb, 1, n, true}, Ut, k, 1, (T)1, true, As, Bs, rank);
    const bool need_null = nz < m, need_disc = nz > k;
    if (need_null || need_disc) {
        // Ua[:, j] = W[:, perm[j]] / s_j for j < nz (column-major m x nz)
        for (int i = gid; i < m * nz; i += gn) {
            const int j = i / m, row = i % m;
            const double s2j = d.s2[j];
            const T f = s2j > 0.0 ? (T)(1.0 / sqrt(s2j)) : (T)0;
            C w = W[(size_t)d.perm[j] * m + row];
            w.x *= f;
            w.y *= f;
            Ua[i] = w;
        }
        cluster_sync();
        // Q1 = Ua^H Ut (nz x k)
        cl_gemm<T, C>(nz, k, m, Op<C>{Ua, m, 1, true}, Op<C>{Ut, k, 1, false}, Q1, k, 1, (T)1, false, As, Bs, rank);
    }
    // directions below tau s_max get no inverse factors (pseudo-inverse cutoff, tau = sqrt(eps))
    const double tau2s = EpsG<T>::v * d.s2[0];
    if (need_null) {
        // (I - P) Ut = (I - P) Ub exactly ((I - P) T = 0); X1 = Ub - Ua (Ua^H Ub), then
        // Tb += X1 S_k^-2 Y.  Mb holds Ua^H Ub (nz x k) meanwhile.
        cl_gemm<T, C>(nz, k, m, Op<C>{Ua, m, 1, true}, Op<C>{Ub, k, 1, false}, Mb, k, 1, (T)1, false, As, Bs, rank);
        for (int i = gid; i < m * k; i += gn) X1[i] = Ub[i];
        cluster_sync();
        cl_gemm<T, C>(m, k, nz, Op<C>{Ua, 1, m, false}, Op<C>{Mb, k, 1, false}, X1, k, 1, (T)-1, true, As, Bs, rank);
        // X2 = S_k^-2 Y (k x n), Y = cY / c
        for (int i = gid; i < k * n; i += gn) {
            const int j = i / n;
            const T f = d.s2[j] > tau2s ? (T)(1.0 / (c * d.s2[j])) : (T)0;
            C y = cY[i];
            y.x *= f;
            y.y *= f;
            X2[i] = y;
        }
        cluster_sync();
        cl_gemm<T, C>(m, n, k, Op<C>{X1, k, 1, false}, Op<C>{X2, n, 1, false}, Tb, n, 1, (T)1, true, As, Bs, rank);
    }
    if (need_disc) {
        const int dd = nz - k;
        // Lorentzian broadening of the cut's denominators on the scale of their rounding
        // error: s_j^2 - s_l^2 carries an absolute error ~ eps s_max (s_j + s_l), so the
        // broadening is (eps s_max (s_j + s_l))^2 -- it regularises unresolved (degenerate)
        // pairs, where the truncated map is not differentiable, and leaves small but
        // separated singular values alone
        const double e2s = EpsG<T>::v * EpsG<T>::v * d.s2[0];
        // X1 = G o B_D (dd x k), B_D = rows k.. of Q1
        for (int i = gid; i < dd * k; i += gn) {
            const int l = i / k, j = i % k;
            const double dj = d.s2[j] - d.s2[k + l];
            const double sum = sqrt(d.s2[j]) + sqrt(fmax(d.s2[k + l], 0.0));
            const double eps_b = e2s * sum * sum;
            const T g = d.s2[j] > tau2s ? (T)(dj / (dj * dj + eps_b)) : (T)0;
            C b = __ldcg(Q1 + (size_t)(k + l) * k + j);
            b.x *= g;
            b.y *= g;
            X1[i] = b;
        }
        cluster_sync();
        // Z T = U_D (Gb Y): X2 = Gb Y (dd x n), Tb += Ua_D X2
        cl_gemm<T, C>(dd, n, k, Op<C>{X1, k, 1, false}, Op<C>{cY, n, 1, false}, X2, n, 1, (T)(1.0 / c), false, As, Bs, rank);
        cl_gemm<T, C>(m, n, dd, Op<C>{Ua + (size_t)k * m, 1, m, false}, Op<C>{X2, n, 1, false}, Tb, n, 1, (T)1, true,
                       As, Bs, rank);
        // Z^H T = U Gb^H (U_D^H T): X2 = U_D^H T (dd x n), Mb (scratch) = Gb^H X2 (k x n), Tb += U Mb
        cl_gemm<T, C>(dd, n, m, Op<C>{Ua + (size_t)k * m, m, 1, true}, Op<C>{Tm, 1, m, false}, X2, n, 1, (T)1, false,
                       As, Bs, rank);
        cl_gemm<T, C>(k, n, dd, Op<C>{X1, 1, k, true}, Op<C>{X2, n, 1, false}, Mb, n, 1, (T)1, false, As, Bs, rank);
        cl_gemm<T, C>(m, n, k, Op<C>{U, k, 1, false}, Op<C>{Mb, n, 1, false}, Tb, n, 1, (T)1, true, As, Bs, rank);
    }
    // effective gate G (uL x uR) in shared memory
    if (tid < 16) {
        const int o = tid >> 2, i = tid & 3;
        double re = 0.0, im = 0.0;
        for (int j = 0; j < 4; ++j) {
            const double gr = d.g4[2 * (o * 4 + j)], gi = d.g4[2 * (o * 4 + j) + 1];
            double ar = ((j >> 1) == (i >> 1)) ? 1.0 : 0.0, ai = 0.0;
            double br = ((j & 1) == (i & 1)) ? 1.0 : 0.0, bi = 0.0;
            if (d.uL) { ar = d.uL[2 * ((j >> 1) * 2 + (i >> 1))]; ai = d.uL[2 * ((j >> 1) * 2 + (i >> 1)) + 1]; }
            if (d.uR) { br = d.uR[2 * ((j & 1) * 2 + (i & 1))]; bi = d.uR[2 * ((j & 1) * 2 + (i & 1)) + 1]; }
            const double kr = ar * br - ai * bi, ki = ar * bi + ai * br;
            re += gr * kr - gi * ki;
            im += gr * ki + gi * kr;
        }
        Gt[tid].x = (T)re;
        Gt[tid].y = (T)im;
    }
    // merge M = A B (m x n row-major)
    cl_gemm<T, C>(m, n, chiM, Op<C>{Apre, chiM, 1, false}, Op<C>{Bpre, n, 1, false}, Mm, n, 1, (T)1, false, As, Bs, rank);
    // Mb[(l,c),(d,r)] = sum_ab conj(Gt[2a+b][2c+d]) Tb[(l,a),(b,r)]; Gtb = sum_{l,r} Tb conj(M)
    double gacc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) gacc[i] = 0.0;
    // a plain gate's at most 225 elements: one per lane, 32 a rank in order, so the sums below are
    // those of one block of 256 threads (at a degenerate cut they cancel, and their order
    // shows; see kPlain64)
    const int lane = tid & 31, warp = tid >> 5;
    const int at = sizeof(T) == 8 && plain64(m, n) ? (warp == 0 ? 32 * rank + lane : chiL * chiR) : mid;
    for (int i = at; i < chiL * chiR; i += gn) {
        const int l = i / chiR, r = i % chiR;
        C tb[4], mm[4];
#pragma unroll
        for (int ab = 0; ab < 4; ++ab) {
            tb[ab] = __ldcg(Tb + (size_t)(2 * l + (ab >> 1)) * n + (ab & 1) * chiR + r);
            mm[ab] = __ldcg(Mm + (size_t)(2 * l + (ab >> 1)) * n + (ab & 1) * chiR + r);
        }
#pragma unroll
        for (int cd = 0; cd < 4; ++cd) {
            C acc = cz<C>();
#pragma unroll
            for (int ab = 0; ab < 4; ++ab) cmac(acc, cconj(Gt[ab * 4 + cd]), tb[ab]);
            Mb[(size_t)(2 * l + (cd >> 1)) * n + (cd & 1) * chiR + r] = acc;
        }
#pragma unroll
        for (int ab = 0; ab < 4; ++ab)
#pragma unroll
            for (int cd = 0; cd < 4; ++cd) {
                const C a = tb[ab], b = mm[cd];   // a conj(b)
                gacc[2 * (ab * 4 + cd)] += (double)a.x * b.x + (double)a.y * b.y;
                gacc[2 * (ab * 4 + cd) + 1] += (double)a.y * b.x - (double)a.x * b.y;
            }
    }
    // sums of the 32 values over the warp: lane i ends up with value i (31 additions instead
    // of the 160 of 32 separate reductions), then over the warps and the ranks
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const bool up = (lane & o) != 0;
            const double send = up ? gacc[i] : gacc[i + o], keep = up ? gacc[i + o] : gacc[i];
            gacc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    red[warp * 32 + lane] = gacc[0];
    __syncthreads();
    if (tid < 32) {
        double v = red[lane];
        for (int w = 1; w < nt / 32; ++w) v += red[w * 32 + lane];
        cl.map_shared_rank(&s_part[rank][0], 0)[lane] = v;
    }
    cluster_sync();   // the partial sums and Mb
    // site adjoints: Ab = Mb B^H (m x chiM), Bb = A^H Mb (chiM x n)
    cl_gemm<T, C>(m, chiM, n, Op<C>{Mb, n, 1, false}, Op<C>{Bpre, 1, n, true}, (C*)d.ab_pre, chiM, 1, (T)1, false,
                   As, Bs, rank);
    cl_gemm<T, C>(chiM, n, m, Op<C>{Apre, 1, chiM, true}, Op<C>{Mb, n, 1, false}, (C*)d.bb_pre, n, 1, (T)1, false,
                   As, Bs, rank);
    // Kb = G^H Gtb; uLb[a,c] = sum_bd Kb[(ab),(cd)] conj(uR[b,d]); uRb[b,d] = sum_ac Kb[...] conj(uL[a,c])
    if (rank == 0 && tid < 32) {
        __shared__ double s_g[32], s_kb[32];
        double v = s_part[0][lane];
        for (int w = 1; w < kBwdRanks; ++w) v += s_part[w][lane];
        s_g[lane] = v;
        __syncwarp();
        if (lane < 16) {
            const int rI = lane >> 2, cI = lane & 3;
            double re = 0.0, im = 0.0;
            for (int j = 0; j < 4; ++j) {
                const double gr = d.g4[2 * (j * 4 + rI)], gi = -d.g4[2 * (j * 4 + rI) + 1];   // conj(G[j][rI])
                const double xr = s_g[2 * (j * 4 + cI)], xi = s_g[2 * (j * 4 + cI) + 1];
                re += gr * xr - gi * xi;
                im += gr * xi + gi * xr;
            }
            s_kb[2 * lane] = re;
            s_kb[2 * lane + 1] = im;
        }
        __syncwarp();
        if (lane < 8) {
            // lanes 0-3: uLb[a][cc] += Kb[(a b),(cc dd)] conj(uR[b][dd]);
            // lanes 4-7: uRb[a][cc] (as [b][d] = [a][cc]) += Kb[(b' a),(d' cc)] conj(uL[b'][d'])
            const bool left = lane < 4;
            const int a = (lane >> 1) & 1, cc = lane & 1;
            const double* u = left ? d.uR : d.uL;
            double re = 0.0, im = 0.0;
            for (int b = 0; b < 2; ++b)
                for (int dd = 0; dd < 2; ++dd) {
                    const double ur = u ? u[2 * (b * 2 + dd)] : (b == dd ? 1.0 : 0.0), ui = u ? u[2 * (b * 2 + dd) + 1] : 0.0;
                    const int e = left ? (2 * a + b) * 4 + 2 * cc + dd : (2 * b + a) * 4 + 2 * dd + cc;
                    const double kr = s_kb[2 * e], ki = s_kb[2 * e + 1];
                    re += kr * ur + ki * ui;
                    im += ki * ur - kr * ui;
                }
            double* out = (left ? d.ubar_l : d.ubar_r) + 2 * (a * 2 + cc);
            out[0] += re;
            out[1] += im;
        }
    }
}

// ---------------------------------------------------------------------------
// final-state adjoint helpers (environments are compact chi x chi, chi read on the device)

// dst += sum of a list's environments, in its order (one CTA row per dst)
template <typename T>
__global__ void k_env_sum(const EnvSumDesc* __restrict__ list, const EnvTerm* __restrict__ terms) {
    using C = typename CT<T>::type;
    const EnvSumDesc d = list[blockIdx.y];
    const int c = d.chi[d.bond];
    C* dst = (C*)d.dst;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < c * c; i += gridDim.x * blockDim.x) {
        C v = dst[i];
        for (int t = d.first; t < d.first + d.n; ++t) {
            const C s = ((const C*)terms[t].src)[i];
            v.x += (T)terms[t].coef * s.x;
            v.y += (T)terms[t].coef * s.y;
        }
        dst[i] = v;
    }
}

// Ab = (AH - (Hsum / N) AN) / N with Hsum, N the 1 x 1 closing environments (device)
template <typename T>
__global__ void k_adj_combine(typename CT<T>::type* __restrict__ ah, const typename CT<T>::type* __restrict__ an,
                              const typename CT<T>::type* __restrict__ hsum, const typename CT<T>::type* __restrict__ nrm,
                              int64_t count) {
    const double N = nrm->x, E = hsum->x / N;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        auto v = ah[i];
        const auto w = an[i];
        v.x = (T)((v.x - E * w.x) / N);
        v.y = (T)((v.y - E * w.y) / N);
        ah[i] = v;
    }
}

// one-qubit gates u = R_{a_last}(t_last) ... R_{a_0}(t_0) of every (layer, qubit) from angles
__device__ void rot_mat(char ax, double t, double* r /* 8 */) {
    const double c = cos(0.5 * t), s = sin(0.5 * t);
    // cos I - i sin P
    for (int i = 0; i < 8; ++i) r[i] = 0.0;
    r[0] = c; r[6] = c;
    if (ax == 'X') { r[3] = -s; r[5] = -s; }
    else if (ax == 'Y') { r[2] = -s; r[4] = s; }
    else { r[1] = -s; r[7] = s; }
}
__device__ void mul22(const double* a, const double* b, double* o) {
    for (int i = 0; i < 2; ++i)
        for (int j = 0; j < 2; ++j) {
            double re = 0.0, im = 0.0;
            for (int k = 0; k < 2; ++k) {
                const double ar = a[2 * (2 * i + k)], ai = a[2 * (2 * i + k) + 1];
                const double br = b[2 * (2 * k + j)], bi = b[2 * (2 * k + j) + 1];
                re += ar * br - ai * bi;
                im += ar * bi + ai * br;
            }
            o[2 * (2 * i + j)] = re;
            o[2 * (2 * i + j) + 1] = im;
        }
}

__global__ void k_rot_build(const RotLayer* __restrict__ rl, int n_layers, int n, double* __restrict__ u1) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_layers * n) return;
    const int L = i / n, q = i % n;
    const RotLayer& R = rl[L];
    if (R.n_rot == 0) return;
    double u[8] = {1, 0, 0, 0, 0, 0, 1, 0}, r[8], t[8];
    for (int j = 0; j < R.n_rot; ++j) {
        rot_mat(R.axes[j], R.theta[(size_t)q * R.n_rot + j], r);
        mul22(r, u, t);
        for (int e = 0; e < 8; ++e) u[e] = t[e];
    }
    for (int e = 0; e < 8; ++e) u1[R.u1_off + (size_t)q * 8 + e] = u[e];
}

// dE/dt_j = 2 Re <ub, du/dt_j>, dR_a/dt = (-i/2) P_a R_a
__global__ void k_rot_grad(const RotLayer* __restrict__ rl, int n_layers, int n, const double* __restrict__ ub,
                           double* __restrict__ grad) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_layers * n) return;
    const int L = i / n, q = i % n;
    const RotLayer& R = rl[L];
    const double* b = ub + R.u1_off + (size_t)q * 8;
    for (int j = 0; j < R.n_rot; ++j) {
        double u[8] = {1, 0, 0, 0, 0, 0, 1, 0}, r[8], t[8];
        for (int jj = 0; jj < R.n_rot; ++jj) {
            rot_mat(R.axes[jj], R.theta[(size_t)q * R.n_rot + jj], r);
            if (jj == j) {
                // (-i/2) P r
                double p[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                const char ax = R.axes[jj];
                if (ax == 'X') { p[0 + 2] = 1; p[4] = 1; }
                else if (ax == 'Y') { p[3] = -1; p[5] = 1; }
                else { p[0] = 1; p[6] = -1; }
                double pr[8];
                mul22(p, r, pr);
                for (int e = 0; e < 4; ++e) {
                    const double re = pr[2 * e], im = pr[2 * e + 1];
                    r[2 * e] = 0.5 * im;       // (-i/2)(re + i im) = im/2 - i re/2
                    r[2 * e + 1] = -0.5 * re;
                }
            }
            mul22(r, u, t);
            for (int e = 0; e < 8; ++e) u[e] = t[e];
        }
        double acc = 0.0;
        for (int e = 0; e < 4; ++e) acc += b[2 * e] * u[2 * e] + b[2 * e + 1] * u[2 * e + 1];
        grad[R.grad_off + (size_t)q * R.n_rot + j] = 2.0 * acc;
    }
}

// unpaired site of a layer with one-qubit gate u: Ab_pre[l,s,r] = sum_p conj(u[p,s]) Ab[l,p,r],
// ub[p,s] += sum_{l,r} Ab[l,p,r] conj(A_pre[l,s,r]); one CTA per site
template <typename T>
__global__ void __launch_bounds__(256) k_site1_bwd(const Site1Bwd* __restrict__ sd) {
    using C = typename CT<T>::type;
    const Site1Bwd& d = sd[blockIdx.x];
    const C* ab = (const C*)d.ab_post;
    const C* a = (const C*)d.a_pre;
    C* out = (C*)d.ab_pre;
    const int cl = d.cl, cr = d.cr;
    double u[8];
    for (int e = 0; e < 8; ++e) u[e] = d.u[e];
    double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int i = threadIdx.x; i < cl * cr; i += blockDim.x) {
        const int l = i / cr, r = i % cr;
        const C b0 = ab[((size_t)l * 2 + 0) * cr + r], b1 = ab[((size_t)l * 2 + 1) * cr + r];
        const C a0 = a[((size_t)l * 2 + 0) * cr + r], a1 = a[((size_t)l * 2 + 1) * cr + r];
        const C bb[2] = {b0, b1}, aa[2] = {a0, a1};
        for (int s = 0; s < 2; ++s) {
            // sum_p conj(u[p][s]) bb[p]
            double re = 0.0, im = 0.0;
            for (int p = 0; p < 2; ++p) {
                const double ur = u[2 * (p * 2 + s)], ui = -u[2 * (p * 2 + s) + 1];
                re += ur * bb[p].x - ui * bb[p].y;
                im += ur * bb[p].y + ui * bb[p].x;
            }
            C v;
            v.x = (T)re;
            v.y = (T)im;
            out[((size_t)l * 2 + s) * cr + r] = v;
        }
        for (int p = 0; p < 2; ++p)
            for (int s = 0; s < 2; ++s) {
                acc[2 * (p * 2 + s)] += (double)bb[p].x * aa[s].x + (double)bb[p].y * aa[s].y;
                acc[2 * (p * 2 + s) + 1] += (double)bb[p].y * aa[s].x - (double)bb[p].x * aa[s].y;
            }
    }
    __shared__ double red[8 * 32];
    block_sum<8>(acc, red);
    if (threadIdx.x == 0)
        for (int e = 0; e < 8; ++e) d.ubar[e] += acc[e];
}

}  // namespace

template <typename T>
cudaError_t launch_gate_bwd(const GradGateDesc* d, int n_gates, cudaStream_t s) {
    if (n_gates <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kBwdRanks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(n_gates * kBwdRanks));
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_gate_bwd<T>, d);
}
template <typename T>
cudaError_t launch_site1_bwd(const Site1Bwd* d, int n_sites, cudaStream_t s) {
    if (n_sites <= 0) return cudaSuccess;
    k_site1_bwd<T><<<n_sites, 256, 0, s>>>(d);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_env_sums(const EnvSumDesc* d, const EnvTerm* terms, int count, int chi_cap, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    k_env_sum<T><<<dim3((chi_cap * chi_cap + 127) / 128, count), 128, 0, s>>>(d, terms);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_adj_combine(void* ah, const void* an, const void* hsum, const void* nrm, int64_t count,
                               cudaStream_t s) {
    using C = typename CT<T>::type;
    k_adj_combine<T><<<(unsigned)std::min<int64_t>((count + 255) / 256, 4096), 256, 0, s>>>(
        (C*)ah, (const C*)an, (const C*)hsum, (const C*)nrm, count);
    return cudaGetLastError();
}
cudaError_t launch_rot_build(const RotLayer* rl, int n_layers, int n, double* u1, cudaStream_t s) {
    const int tot = n_layers * n;
    k_rot_build<<<(tot + 127) / 128, 128, 0, s>>>(rl, n_layers, n, u1);
    return cudaGetLastError();
}
cudaError_t launch_rot_grad(const RotLayer* rl, int n_layers, int n, const double* ub, double* grad, cudaStream_t s) {
    const int tot = n_layers * n;
    k_rot_grad<<<(tot + 127) / 128, 128, 0, s>>>(rl, n_layers, n, ub, grad);
    return cudaGetLastError();
}

#define TNSIM_GRAD_INST(T)                                                                                      \
    template cudaError_t launch_gate_bwd<T>(const GradGateDesc*, int, cudaStream_t);                              \
    template cudaError_t launch_site1_bwd<T>(const Site1Bwd*, int, cudaStream_t);                                 \
    template cudaError_t launch_env_sums<T>(const EnvSumDesc*, const EnvTerm*, int, int, cudaStream_t);           \
    template cudaError_t launch_adj_combine<T>(void*, const void*, const void*, const void*, int64_t, cudaStream_t);
TNSIM_GRAD_INST(float)
TNSIM_GRAD_INST(double)
#undef TNSIM_GRAD_INST

}  // namespace tnsim
