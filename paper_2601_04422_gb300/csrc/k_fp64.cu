// FP64 products of the two-qubit update, and the mixed-precision preconditioner of the
// complex128 SVD.
//
// GB300 issues FP64 at 1/64 of the FP32 rate, so an FP64 kernel's time is its FP64
// instruction count over the SMs that it keeps busy, and everything else hides behind
// it.  The products therefore use 8 x 8 tiles (tile16.cuh): with 64 x 64 tiles one SM per
// gate did the work (theta and right site of 5 gates at m = n = 64: 88 + 136 -> 9 + 13 us;
// of 20 gates at m = 180: 480 + 790 -> 330 + 350 us).
//
// Preconditioner (mixed-precision Jacobi SVD: Gao, Ma and Shao 2022).  One-sided Jacobi
// converges quadratically, so 9 of its ~12 FP64 sweeps only bring the columns from O(1)
// to ~1e-6 of orthogonal, which FP32 can do at 64 times the rate:
//   k_mix_build  [W; I] in FP32 (W, at first theta, scaled by a power of two to |W|_F in
//                [2^28, 2^29): the squares and their products stay in FP32's range for
//                columns down to 2^-52 |W|_F);
//   k_jacobi     FP32 Jacobi rotations of these columns until W V is orthogonal to
//                kMixTol; the lower n rows become V (k_jacobi.cu, EXT);
//   k_mix_gram   E = I - V^H V in FP64 (V is unitary to ~1e-6 only);
//   k_mix_corr   F = E/2 + 3/8 E^2, so that V (I + F) = V (V^H V)^{-1/2} + O(E^3) is
//                unitary to FP64 rounding (E^2 ~ 1e-12 needs four digits: FP32);
//   k_mix_mul    X = W V, then W <- X + X F, both in FP64.
// This is done twice.  In the first pass the columns of theta, all of about the same
// norm, hide singular values s in FP32 roundings: the small columns of W come out
// orthogonal to ~1e-7 s_max / s only (and below 1e-7 s_max not at all).  W's columns now
// have the singular values as norms, each rounded to FP32 relative to its own norm, so
// the second pass resolves all of them down to FP64's zero, in two or three FP32 sweeps.
// The FP64 Jacobi iteration then starts from W V' with V' unitary: the same SVD to the
// same tolerance, with fewer sweeps and mostly tiny rotations.  A preconditioner that did
// not converge only costs sweeps.
// Measured with the FP64 visit of k_jacobi.cu on 20 gates at m = n = 180: SVD 139 ms
// without, 29 with one pass (12.2 -> 4.7 FP64 sweeps per gate), 23 with two (3.6); 4 gates
// at m = n = 64: 3.2 ms with one pass (6.7 sweeps), 2.1 with two (4.2).  Singular values
// 6e-16 (relative) from LAPACK's in all three.
#include <float.h>

#include "tile16.cuh"
#include "tnsim_internal.h"

namespace tnsim {

namespace {

// ---------------------------------------------------------------------------
// theta (see k_gemm.cu): 4 l x 4 r per CTA; tile rows (l, c), tile columns (d, r).
constexpr int T64 = TileOf<double2>::E;   // 8
__global__ void __launch_bounds__(TILE_THREADS) k_theta64(const GateDesc* __restrict__ gd) {
    const GateDesc& d = gd[blockIdx.z];
    const int q = d.q;
    const int chiL = d.chi[q], chiM = d.chi[q + 1], chiR = d.chi[q + 2];
    constexpr int H = T64 / 2;
    const int l0 = blockIdx.x * H, r0 = blockIdx.y * H;
    if (l0 >= chiL || r0 >= chiR) return;
    __shared__ double2 Gs[16], S[T64][T64 + 1];
    const int tid = threadIdx.x;
    if (tid < 16) {
        const int o = tid >> 2, i = tid & 3;
        double re = 0.0, im = 0.0;
        for (int j = 0; j < 4; ++j) {
            const double gr = d.g4[2 * (o * 4 + j)], gi = d.g4[2 * (o * 4 + j) + 1];
            // K[j][i] = uL[j>>1][i>>1] * uR[j&1][i&1]
            double ar = ((j >> 1) == (i >> 1)) ? 1.0 : 0.0, ai = 0.0;
            double br = ((j & 1) == (i & 1)) ? 1.0 : 0.0, bi = 0.0;
            if (d.uL) { ar = d.uL[2 * ((j >> 1) * 2 + (i >> 1))]; ai = d.uL[2 * ((j >> 1) * 2 + (i >> 1)) + 1]; }
            if (d.uR) { br = d.uR[2 * ((j & 1) * 2 + (i & 1))]; bi = d.uR[2 * ((j & 1) * 2 + (i & 1)) + 1]; }
            const double kr = ar * br - ai * bi, ki = ar * bi + ai * br;
            re += gr * kr - gi * ki;
            im += gr * ki + gi * kr;
        }
        Gs[tid] = make_double2(re, im);
    }
    const double2* A = (const double2*)d.siteA;
    const double2* B = (const double2*)d.siteB;
    const int m = 2 * chiL;
    double2 acc[1][1] = {};
    tile_product<double2, true, false, false, true, MulAdd>(
        chiM,
        [&](int i, int k) {
            const int row = 2 * l0 + i;
            return row < m ? A[(size_t)row * chiM + k] : make_double2(0.0, 0.0);
        },
        [&](int k, int j) {
            const int r = r0 + j % H;
            return r < chiR ? B[((size_t)k * 2 + j / H) * chiR + r] : make_double2(0.0, 0.0);
        },
        acc);
    tile_share<double2, false>(S, acc);
    double2* Wm = (double2*)d.W;
    double2* T0 = (double2*)d.theta0;
    double fro = 0.0;
    // output (l, aa), (bb, r): the four merged entries of (l, r) mixed by the gate
    const int i = tid & 7, j = tid >> 3, li = i >> 1, ri = j % H, aa = i & 1, bb = j / H;
    const int l = l0 + li, r = r0 + ri;
    if (l < chiL && r < chiR) {
        double2 t = make_double2(0.0, 0.0);
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int e = 0; e < 2; ++e) MulAdd::op(t, Gs[(2 * aa + bb) * 4 + 2 * c + e], S[2 * li + c][e * H + ri]);
        const size_t idx = (size_t)(bb * chiR + r) * m + 2 * l + aa;
        Wm[idx] = t;
        T0[idx] = t;
        fro = fma(t.x, t.x, t.y * t.y);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) fro += __shfl_xor_sync(0xffffffffu, fro, o);
    if ((tid & 31) == 0 && fro != 0.0) atomicAdd(&d.out->frob2, fro);
}

// right site (see k_right in k_gemm.cu): R[j, col] = f_j sum_row conj(W[row, perm_j]) theta0[row, col]
__global__ void __launch_bounds__(TILE_THREADS) k_right64(const GateDesc* __restrict__ gd) {
    const GateDesc& d = gd[blockIdx.z];
    const int q = d.q;
    const int m = 2 * d.chi[q], n = 2 * d.chi[q + 2], k = d.out->k;
    if (qr_active(d, m, n)) return;   // QR-preconditioned: k_right_pre (k_qr.cu)
    const int c0 = blockIdx.x * T64, j0 = blockIdx.y * T64;
    if (c0 >= n || j0 >= k) return;
    __shared__ int pj[T64];
    __shared__ double fj[T64];
    const int tid = threadIdx.x;
    if (tid < T64) {
        const int j = j0 + tid;
        const double s2j = j < k ? d.s2[j] : 0.0;
        pj[tid] = j < k ? d.perm[j] : -1;
        if (d.canon) fj[tid] = s2j > 0.0 ? 1.0 / s2j : 0.0;
        else fj[tid] = s2j > 0.0 ? d.out->scale / sqrt(s2j) : 0.0;
    }
    __syncthreads();
    const double2* Wm = (const double2*)d.W;
    const double2* T0 = (const double2*)d.theta0;
    const int lk = d.canon ? *d.lam_k : 0;
    double2 acc[1][1] = {};
    // tile rows: columns of R (they run along its rows in memory); tile columns: rows j
    tile_product<double2, true, true, false, true, MulAdd>(
        m,
        [&](int i, int row) {
            if (c0 + i >= n) return make_double2(0.0, 0.0);
            double2 w = T0[(size_t)(c0 + i) * m + row];
            if ((row >> 1) < lk) {
                const double f = d.lam[row >> 1];
                w.x *= f;
                w.y *= f;
            }
            return w;
        },
        [&](int row, int j) {
            if (pj[j] < 0) return make_double2(0.0, 0.0);
            const double2 v = Wm[(size_t)pj[j] * m + row];
            return make_double2(v.x, -v.y);
        },
        acc);
    double2* R = (double2*)d.siteB;
    const int jj = tid >> 3, col = c0 + (tid & 7);
    if (j0 + jj < k && col < n) R[(size_t)(j0 + jj) * n + col] = make_double2(acc[0][0].x * fj[jj], acc[0][0].y * fj[jj]);
}

// ---------------------------------------------------------------------------
// the preconditioner

__device__ __forceinline__ bool mix_active(const GateDesc& d, int m, int n) {
    return d.pre && n >= kMixMinCols && m + n <= kMixMaxRows;
}

// [W; I] in FP32; a gate outside the preconditioner counts as finished in its launch
__global__ void __launch_bounds__(256) k_mix_build(const GateDesc* __restrict__ gd, JacobiCtl* __restrict__ ctl) {
    const GateDesc& d = gd[blockIdx.y];
    const int m = 2 * d.chi[d.q], n = 2 * d.chi[d.q + 2];
    if (!mix_active(d, m, n)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            d.out->finished = 1;
            atomicAdd(&ctl->n_finished, 1);
        }
        return;
    }
    const int mt = m + n;
    const double f = mix_scale(d.out->frob2);
    const double2* Wm = (const double2*)d.W;
    float2* Y = (float2*)d.pre;
    const int total = mt * n;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const int c = t / mt, r = t - c * mt;
        float2 y;
        if (r < m) {
            const double2 w = Wm[(size_t)c * m + r];
            y = make_float2((float)(w.x * f), (float)(w.y * f));
        } else {
            y = make_float2(r - m == c ? 1.f : 0.f, 0.f);
        }
        Y[t] = y;
    }
}

// E = I - V^H V (Hermitian: tiles on and above the diagonal, mirrored).  The first CTA of
// a gate also readies its record for the FP64 launch: a sweep cap reached in FP32 is no
// error, a timeout is.
__global__ void __launch_bounds__(TILE_THREADS) k_mix_gram(const GateDesc* __restrict__ gd) {
    const GateDesc& d = gd[blockIdx.z];
    const int m = 2 * d.chi[d.q], n = 2 * d.chi[d.q + 2];
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        GateOut* o = d.out;
        if (!o->finished) o->status = 5;
        else if (o->status == 4) o->status = 0;
        o->finished = 0;
        o->done = 0;
        o->rot_sweep = 0;
        o->claim = 0;
    }
    if (!mix_active(d, m, n)) return;
    const int i0 = blockIdx.x * T64, j0 = blockIdx.y * T64;
    if (i0 >= n || j0 >= n || i0 > j0) return;
    const int mt = m + n;
    const float2* V = (const float2*)d.pre + m;
    double2* E = (double2*)d.pre_x;
    // the diagonal sums start from -1: they end near 0, and the last roundings are small
    double2 acc[1][1] = {};
    if (i0 == j0 && (threadIdx.x & 7) == (threadIdx.x >> 3)) acc[0][0].x = -1.0;
    tile_product<double2, true, true, false, true, MulAdd>(
        n,
        [&](int i, int k) {
            if (i0 + i >= n) return make_double2(0.0, 0.0);
            const float2 v = V[(size_t)(i0 + i) * mt + k];
            return make_double2((double)v.x, -(double)v.y);
        },
        [&](int k, int j) {
            if (j0 + j >= n) return make_double2(0.0, 0.0);
            const float2 v = V[(size_t)(j0 + j) * mt + k];
            return make_double2((double)v.x, (double)v.y);
        },
        acc);
    const int i = i0 + (threadIdx.x & 7), j = j0 + (threadIdx.x >> 3);
    if (i >= n || j >= n) return;
    const double re = -acc[0][0].x, im = -acc[0][0].y;
    E[(size_t)j * n + i] = make_double2(re, im);
    if (i0 != j0) E[(size_t)i * n + j] = make_double2(re, -im);
}

constexpr int T32 = TileOf<float2>::E;    // 16
// F = E/2 + 3/8 E^2 (Hermitian)
__global__ void __launch_bounds__(TILE_THREADS) k_mix_corr(const GateDesc* __restrict__ gd) {
    const GateDesc& d = gd[blockIdx.z];
    const int m = 2 * d.chi[d.q], n = 2 * d.chi[d.q + 2];
    if (!mix_active(d, m, n)) return;
    const int i0 = blockIdx.x * T32, j0 = blockIdx.y * T32;
    if (i0 >= n || j0 >= n || i0 > j0) return;
    const double2* E = (const double2*)d.pre_x;
    double2* F = (double2*)d.pre_f;
    float2 acc[2][2] = {};
    tile_product<float2, true, true, false, true, MulAdd>(
        n,
        [&](int i, int k) {   // E[i, k] = conj(E[k, i])
            if (i0 + i >= n) return make_float2(0.f, 0.f);
            const double2 e = E[(size_t)(i0 + i) * n + k];
            return make_float2((float)e.x, -(float)e.y);
        },
        [&](int k, int j) {
            if (j0 + j >= n) return make_float2(0.f, 0.f);
            const double2 e = E[(size_t)(j0 + j) * n + k];
            return make_float2((float)e.x, (float)e.y);
        },
        acc);
    const int rx = threadIdx.x & 7, cy = threadIdx.x >> 3;
#pragma unroll
    for (int jj = 0; jj < 2; ++jj)
#pragma unroll
        for (int ii = 0; ii < 2; ++ii) {
            const int i = i0 + rx + 8 * ii, j = j0 + cy + 8 * jj;
            if (i >= n || j >= n) continue;
            const double2 e = E[(size_t)j * n + i];
            const double re = fma(0.375, (double)acc[ii][jj].x, 0.5 * e.x);
            const double im = fma(0.375, (double)acc[ii][jj].y, 0.5 * e.y);
            F[(size_t)j * n + i] = make_double2(re, im);
            if (i0 != j0) F[(size_t)i * n + j] = make_double2(re, -im);
        }
}

// FIRST: X = W V; else W = X + X F
template <bool FIRST>
__global__ void __launch_bounds__(TILE_THREADS) k_mix_mul(const GateDesc* __restrict__ gd) {
    const GateDesc& d = gd[blockIdx.z];
    const int m = 2 * d.chi[d.q], n = 2 * d.chi[d.q + 2];
    if (!mix_active(d, m, n)) return;
    const int i0 = blockIdx.x * T64, j0 = blockIdx.y * T64;
    if (i0 >= m || j0 >= n) return;
    const int mt = m + n;
    double2* X = (double2*)d.pre_x;
    double2* Wm = (double2*)d.W;
    const double2* A = FIRST ? Wm : X;
    double2 acc[1][1] = {};
    tile_product<double2, false, true, false, true, MulAdd>(
        n,
        [&](int i, int k) { return i0 + i < m ? A[(size_t)k * m + i0 + i] : make_double2(0.0, 0.0); },
        [&](int k, int j) {
            if (j0 + j >= n) return make_double2(0.0, 0.0);
            if (!FIRST) return ((const double2*)d.pre_f)[(size_t)(j0 + j) * n + k];
            const float2 v = ((const float2*)d.pre)[(size_t)(j0 + j) * mt + m + k];
            return make_double2((double)v.x, (double)v.y);
        },
        acc);
    const int i = i0 + (threadIdx.x & 7), j = j0 + (threadIdx.x >> 3);
    if (i >= m || j >= n) return;
    const size_t idx = (size_t)j * m + i;
    if (FIRST) {
        X[idx] = acc[0][0];
    } else {
        const double2 x = X[idx];
        Wm[idx] = make_double2(x.x + acc[0][0].x, x.y + acc[0][0].y);
    }
}

}  // namespace

cudaError_t launch_theta64(const GateDesc* d, int n_gates, int chiL_max, int chiR_max, cudaStream_t s) {
    if (n_gates <= 0) return cudaSuccess;
    dim3 grid((chiL_max + T64 / 2 - 1) / (T64 / 2), (chiR_max + T64 / 2 - 1) / (T64 / 2), n_gates);
    k_theta64<<<grid, TILE_THREADS, 0, s>>>(d);
    return cudaGetLastError();
}

cudaError_t launch_right64(const GateDesc* d, int n_gates, int k_max, int n_max, cudaStream_t s) {
    if (n_gates <= 0) return cudaSuccess;
    dim3 grid((n_max + T64 - 1) / T64, (k_max + T64 - 1) / T64, n_gates);
    k_right64<<<grid, TILE_THREADS, 0, s>>>(d);
    return cudaGetLastError();
}

cudaError_t launch_mix(const GateDesc* d, int n_gates, int m_max, int n_max, JacobiCtl* ctl, cudaStream_t s,
                       int n_lead, unsigned spin_limit) {
    if (n_gates <= 0 || n_max < kMixMinCols) return cudaSuccess;
    const int mt = m_max + n_max < kMixMaxRows ? m_max + n_max : kMixMaxRows;   // of an active gate
    const int mm = m_max < kMixMaxRows ? m_max : kMixMaxRows, nm = n_max < kMixMaxRows ? n_max : kMixMaxRows;
    int bx = (int)(((long long)mt * nm + 1023) / 1024);
    if (bx > 128) bx = 128;
    const int tn = (nm + T64 - 1) / T64, tm = (mm + T64 - 1) / T64, tf = (nm + T32 - 1) / T32;
    for (int pass = 0; pass < 2; ++pass) {
        cudaError_t e = cudaMemsetAsync(ctl, 0, sizeof(JacobiCtl), s);
        if (e != cudaSuccess) return e;
        k_mix_build<<<dim3(bx, n_gates), 256, 0, s>>>(d, ctl);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        e = launch_jacobi_mix(d, n_gates, mt, nm, pass ? DBL_EPSILON : FLT_EPSILON, ctl, s, n_lead, spin_limit);
        if (e != cudaSuccess) return e;
        k_mix_gram<<<dim3(tn, tn, n_gates), TILE_THREADS, 0, s>>>(d);
        k_mix_corr<<<dim3(tf, tf, n_gates), TILE_THREADS, 0, s>>>(d);
        k_mix_mul<true><<<dim3(tm, tn, n_gates), TILE_THREADS, 0, s>>>(d);
        k_mix_mul<false><<<dim3(tm, tn, n_gates), TILE_THREADS, 0, s>>>(d);
    }
    return cudaGetLastError();
}

}  // namespace tnsim
