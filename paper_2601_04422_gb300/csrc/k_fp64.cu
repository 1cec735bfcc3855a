// FP64 products of the two-qubit update, and the mixed-precision preconditioner of the
// complex128 SVD.
//
// GB300 issues FP64 at 1/64 of the FP32 rate, so an FP64 kernel's time is its FP64
// instruction count over the SMs that it keeps busy, and everything else hides behind
// it.  The products therefore use 8 x 8 tiles (tile8.cuh): with 64 x 64 tiles one SM per
// gate did the work (theta and right site of 5 gates at m = n = 64: 88 + 136 -> 9 + 13 us;
// of 20 gates at m = 180: 480 + 790 -> 330 + 350 us).
//
// Preconditioner (mixed-precision Jacobi SVD: Gao, Ma and Shao 2022; refinement of nearly
// orthogonal columns after Ogita and Aishima 2018).  One-sided Jacobi converges
// quadratically, so 9 of its ~12 FP64 sweeps only bring the columns from O(1) to ~1e-6 of
// orthogonal, which FP32 can do at 64 times the rate; and from there all pairs can be
// turned at once, W <- W (I + F), two matrix products instead of a sweep:
//   k_mix_build  [theta; I] in FP32 (theta scaled by a power of two to |theta|_F in [1, 2));
//   k_jacobi     FP32 Jacobi rotations of these columns until theta V is orthogonal to
//                kMixTol; the lower n rows become V (k_jacobi.cu, EXT);
//   k_mix_first  X = W V and E = I - V^H V in FP64 (V is unitary to ~1e-6 only);
//   k_mix_angle  K, anti-Hermitian: the angles of the pairs of X's columns;
//   k_mix_sq     K^2
//   k_mix_r, k_mix_corr
//                I + F = V's correction to a unitary matrix times K + (I + K^2)^{1/2},
//                unitary to FP64 rounding;
//   k_mix_mul    X + X F;
//   k_mix_angle, k_mix_sq, k_mix_mul: a second refinement, whose angles are so small that
//                F = K + K^2 / 2.
// The FP64 Jacobi iteration then starts from W V' with V' unitary: the same SVD to the
// same tolerance.  It usually only finds that the columns are orthogonal, and rotates the
// pairs that the steps left out: those of singular values too close for a small angle.  A
// preconditioner that did not converge only costs sweeps; one whose V is not unitary enough
// to be corrected (mix_off) is left out.
// FP64 enters where rounding would reach the result: in X, E and the second K.  The other
// products are sums of FP32 pairs (48 bits) at a fifth of FP64's time: of small corrections
// (K, F < 2^-10 of X), or where a few digits do.
// Measured: the SVD of 20 gates at m = n = 180, 139 ms without it, 29 without refinement
// (12.2 and 4.7 FP64 sweeps per gate), 9.2 with the products in FP64, 6.6 so (1.5 sweeps,
// 0.1 % of their pairs rotated; FP32 rotations 2.9, products 2.1, FP64 sweeps 1.1; the layer's
// small gates at its ends go with the last); 4 gates at m = n = 64, 3.2 ms without refinement,
// 0.8 with.  Singular values 6e-16 (relative)
// from LAPACK's throughout.  A second FP32 pass on the columns of X in place of the
// refinement left 3.6 sweeps: 20 ms.
#include <float.h>

#include "jacobi_sched.cuh"
#include "tile8.cuh"
#include "tnsim_internal.h"

namespace tnsim {

namespace {

// ---------------------------------------------------------------------------
// theta (see k_gemm.cu): 4 l x 4 r per CTA; tile rows (l, c), tile columns (d, r).
constexpr int T64 = TILE_E;
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
    double2 acc = {};
    tile_product<double2, true, false, true, MulAdd>(
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
    tile_share(S, acc);
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
    double2 acc = {};
    // tile rows: columns of R (they run along its rows in memory); tile columns: rows j
    tile_product<double2, true, true, true, MulAddConj>(
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
        [&](int row, int j) { return pj[j] < 0 ? make_double2(0.0, 0.0) : Wm[(size_t)pj[j] * m + row]; }, acc);
    double2* R = (double2*)d.siteB;
    const int jj = tid >> 3, col = c0 + (tid & 7);
    if (j0 + jj < k && col < n) R[(size_t)(j0 + jj) * n + col] = make_double2(acc.x * fj[jj], acc.y * fj[jj]);
}

// ---------------------------------------------------------------------------
// the preconditioner

__device__ __forceinline__ bool mix_active(const GateDesc& d, int m, int n) {
    return d.pre && n >= kMixMinCols && m + n <= kMixMaxRows && !plain64(m, n);
}

// FP32 pairs: h + l with |l| <= ulp(h), 48 bits; a complex number of two of them.
struct Df {
    float x, y, xl, yl;
};
// h + l += a b (twelve FP32 instructions; one FP64 instruction takes as long as 64)
template <bool LO>
__device__ __forceinline__ void df_mac(float& h, float& l, float a, float al, float b, float bl) {
    const float p = __fmul_rn(a, b);
    float t = fmaf(a, b, -p);
    if (LO) t = fmaf(al, b, fmaf(a, bl, t));
    const float s = __fadd_rn(h, p), z = __fsub_rn(s, h);
    l = __fadd_rn(l, __fadd_rn(t, __fadd_rn(__fsub_rn(h, __fsub_rn(s, z)), __fsub_rn(p, z))));
    h = s;
}
template <bool LO>
struct DfMulAdd {
    static __device__ __forceinline__ void op(Df& acc, const Df& a, const Df& b) {
        df_mac<LO>(acc.x, acc.xl, a.x, a.xl, b.x, b.xl);
        df_mac<LO>(acc.x, acc.xl, -a.y, -a.yl, b.y, b.yl);
        df_mac<LO>(acc.y, acc.yl, a.x, a.xl, b.y, b.yl);
        df_mac<LO>(acc.y, acc.yl, a.y, a.yl, b.x, b.xl);
    }
};
__device__ __forceinline__ double2 from_df(const Df& a) {
    return make_double2((double)a.x + (double)a.xl, (double)a.y + (double)a.yl);
}
__device__ __forceinline__ Df df_of(double x, double y) {
    const float hx = (float)x, hy = (float)y;
    return {hx, hy, (float)(x - (double)hx), (float)(y - (double)hy)};
}
// x 2^-e as a pair by integer operations (a conversion pair takes an FP64 subtraction)
__device__ __forceinline__ void df_scaled(double x, int e, float& h, float& l) {
    h = f32_scaled(x, e);   // truncated: 24 bits, the other 29 follow
    const unsigned hb = __float_as_uint(h), ex = (hb >> 23) & 0xff;
    const float u = __uint2float_rn((unsigned)__double2loint(x) & 0x1fffffffu);
    l = ex > 52 ? u * __uint_as_float((hb & 0x80000000u) | ((ex - 52) << 23)) : 0.f;
}
__device__ __forceinline__ Df to_df(const double2& v, int e, bool conj) {
    Df r;
    df_scaled(v.x, e, r.x, r.xl);
    df_scaled(v.y, e, r.y, r.yl);
    if (conj) { r.y = -r.y; r.yl = -r.yl; }
    return r;
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
    if (blockIdx.x == 0)
        for (int t = threadIdx.x; t < kMixRows * n; t += blockDim.x) d.pre_rows[t] = 0;
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

// The buffers of a gate by the step's number: 0, the polar factor of V and a first
// refinement (X -> B); 1, a second refinement (B -> W).
//   E, X          E = I - V^H V in B; X = W V
//   K             a step's angles in the place of V
//   D             step 0: K^2; step 1: F
struct MixBufs {
    const double2* src;
    double2* dst;
    Df* F;
};
__device__ __forceinline__ MixBufs mix_bufs(const GateDesc& d, int step) {
    if (step == 0) return {(const double2*)d.pre_x, (double2*)d.pre_b, (Df*)d.W};
    return {(const double2*)d.pre_b, (double2*)d.W, (Df*)d.pre_d};
}
// R of the correction (k_mix_r), behind K in the place of V
__device__ __forceinline__ float2* mix_R(const GateDesc& d, int n) { return (float2*)d.pre + (size_t)n * n; }
// Row sums of a matrix, in fixed point (the order of the additions does not matter): they
// bound its norm.  0: K^2 of step 0; 1, 2: K of step 1, all angles and those up to kRefCap2; 3: E.
constexpr float kRowUnit0 = 0x1p-38f, kRowUnit1 = 0x1p-36f;
__device__ __forceinline__ unsigned* mix_rows(const GateDesc& d, int n, int which) { return d.pre_rows + which * n; }
// the tile's elements of size v at (i, j), mirrored at (j, i) off the diagonal tiles
__device__ __forceinline__ void mix_rows_add(unsigned* rows, float v, float unit, int i, int j, int n, bool mirror) {
    const float top = unit * 0x1p24f;
    float r = v, c = v;
#pragma unroll
    for (int o = 8; o < 32; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    const int lane = threadIdx.x & 31;
    if (lane < 8 && i < n) atomicAdd(rows + i, (unsigned)(fminf(r, top) / unit));
    if (mirror && (lane & 7) == 0 && j < n) atomicAdd(rows + j, (unsigned)(fminf(c, top) / unit));
}
__device__ __forceinline__ bool mix_rows_above(const unsigned* rows, int n, float unit, float limit) {
    const unsigned top = (unsigned)(limit / unit);
    bool over = false;
    for (int i = threadIdx.x; i < n; i += TILE_THREADS) over |= rows[i] > top;
    return __syncthreads_or(over);
}
// V too far from unitary for the series of its correction: the gate keeps W as it is
__device__ __forceinline__ bool mix_off(const GateDesc& d, int n) {
    return mix_rows_above(mix_rows(d, n, 3), n, kRowUnit1, kRefRowE);
}
// exponent that scales |W|_F into [2^40, 2^42): FP32 pairs then hold W's elements to 2^-48
// of their size down to 2^-115 |W|_F
__device__ __forceinline__ int mix_exp(double frob2) {
    return frob2 > 0.0 && !isinf(frob2) ? (ilogb(frob2) >> 1) - 40 : -40;
}

// One launch, two products of V: X = W V (the first x_tiles of grid.x) and E = I - V^H V (the
// rest; Hermitian: tiles on and above the diagonal, mirrored).  The first CTA of a gate's E also readies its
// record for the FP64 launch: a sweep cap reached in FP32 is no error, a timeout is.
__global__ void __launch_bounds__(TILE_THREADS) k_mix_first(const GateDesc* __restrict__ gd, int x_tiles) {
    const bool gram = blockIdx.x >= x_tiles;
    const int bx = gram ? blockIdx.x - x_tiles : blockIdx.x;
    const GateDesc& d = gd[blockIdx.z];
    const int m = 2 * d.chi[d.q], n = 2 * d.chi[d.q + 2];
    if (gram && bx == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
        GateOut* o = d.out;
        if (!o->finished) o->status = 5;
        else if (o->status == 4) o->status = 0;
        o->finished = 0;
        o->done = 0;
        o->rot_sweep = 0;
        o->claim = 0;
    }
    if (!mix_active(d, m, n)) return;
    const int i0 = bx * T64, j0 = blockIdx.y * T64;
    if (i0 >= (gram ? n : m) || j0 >= n || (gram && i0 > j0)) return;
    const int mt = m + n;
    const float2* V = (const float2*)d.pre + m;
    const double2* Wm = (const double2*)d.W;
    const int ti = threadIdx.x & 7, tj = threadIdx.x >> 3, i = i0 + ti, j = j0 + tj;
    auto lb = [&](int k, int c) {
        if (j0 + c >= n) return make_double2(0.0, 0.0);
        const float2 v = V[(size_t)(j0 + c) * mt + k];
        return make_double2((double)v.x, (double)v.y);
    };
    double2 acc = {};
    if (!gram) {
        tile_product<double2, false, true, true, MulAdd>(
            n, [&](int r, int k) { return i0 + r < m ? Wm[(size_t)k * m + i0 + r] : make_double2(0.0, 0.0); }, lb, acc);
        if (i < m && j < n) ((double2*)d.pre_x)[(size_t)j * m + i] = acc;
        return;
    }
    // the diagonal sums start from -1: they end near 0, and the last roundings are small
    if (i0 == j0 && ti == tj) acc.x = -1.0;
    tile_product<double2, true, true, true, MulAdd>(
        n,
        [&](int c, int k) {
            if (i0 + c >= n) return make_double2(0.0, 0.0);
            const float2 v = V[(size_t)(i0 + c) * mt + k];
            return make_double2((double)v.x, -(double)v.y);
        },
        lb, acc);
    const double re = -acc.x, im = -acc.y;
    const bool in = i < n && j < n;
    mix_rows_add(mix_rows(d, n, 3), in ? fabsf((float)re) + fabsf((float)im) : 0.f, kRowUnit1, i, j, n, i0 != j0);
    if (!in) return;
    double2* E = (double2*)d.pre_b;
    E[(size_t)j * n + i] = make_double2(re, im);
    if (i0 != j0) E[(size_t)i * n + j] = make_double2(re, -im);
}

// K of a step from S = src^H src: above the diagonal K = tau S, the angle that would
// orthogonalise that pair alone (zero beyond the step's cap, and for columns that are
// zero), -K^H below.  Step 0: S of the corrected columns, X (I + E/2), to first order.
// Step 0 sums FP32 pairs: S of relative size 1e-6 is wanted to a few digits; step 1 FP64.
template <int STEP>
__global__ void __launch_bounds__(TILE_THREADS) k_mix_angle(const GateDesc* __restrict__ gd) {
    const GateDesc& d = gd[blockIdx.z];
    const int m = 2 * d.chi[d.q], n = 2 * d.chi[d.q + 2];
    if (!mix_active(d, m, n)) return;
    const int i0 = blockIdx.x * T64, j0 = blockIdx.y * T64;
    if (i0 >= n || j0 >= n || i0 > j0 || mix_off(d, n)) return;
    const double2* X = mix_bufs(d, STEP).src;
    const double frob2 = d.out->frob2;
    const int e = mix_exp(frob2);
    double2 g;
    if constexpr (STEP == 0) {
        Df acc = {};
        tile_product<Df, true, true, false, DfMulAdd<true>>(
            m,
            [&](int c, int k) { return i0 + c < n ? to_df(X[(size_t)(i0 + c) * m + k], e, true) : Df{}; },
            [&](int k, int c) { return j0 + c < n ? to_df(X[(size_t)(j0 + c) * m + k], e, false) : Df{}; }, acc);
        g = from_df(acc);
    } else {
        double2 acc = {};
        tile_product<double2, true, true, true, MulAdd>(
            m,
            [&](int c, int k) {
                if (i0 + c >= n) return make_double2(0.0, 0.0);
                const double2 v = X[(size_t)(i0 + c) * m + k];
                return make_double2(v.x, -v.y);
            },
            [&](int k, int c) { return j0 + c < n ? X[(size_t)(j0 + c) * m + k] : make_double2(0.0, 0.0); }, acc);
        g = acc;
    }
    // squared norms of the tile's 8 + 8 columns, four threads each
    __shared__ double nrm[2 * T64];
    {
        const int c = threadIdx.x >> 2, col = c < T64 ? i0 + c : j0 + c - T64;
        float h = 0.f, l = 0.f;
        if (col < n)
            for (int r = threadIdx.x & 3; r < m; r += 4) {
                const Df x = to_df(X[(size_t)col * m + r], e, false);
                df_mac<true>(h, l, x.x, x.xl, x.x, x.xl);
                df_mac<true>(h, l, x.y, x.yl, x.y, x.yl);
            }
        double a = (double)h + (double)l;
        a += __shfl_xor_sync(0xffffffffu, a, 1);
        a += __shfl_xor_sync(0xffffffffu, a, 2);
        if ((threadIdx.x & 3) == 0) nrm[c] = a;
    }
    __syncthreads();
    const int ti = threadIdx.x & 7, tj = threadIdx.x >> 3, i = i0 + ti, j = j0 + tj;
    const double sc = ldexp(1.0, -2 * e);
    if (STEP == 1) { g.x *= sc; g.y *= sc; }
    const double zthr = DBL_EPSILON * DBL_EPSILON * (double)max(m, n) * frob2 * sc;
    double a = nrm[ti], b = nrm[T64 + tj];
    float2 k = make_float2(0.f, 0.f);
    if (i < j && j < n && a > zthr && b > zthr) {
        if (STEP == 0) {
            const double2* E = (const double2*)d.pre_b;
            const double2 f = E[(size_t)j * n + i];
            const double h = 0.5 * (a + b);
            g.x = fma(f.x, h, g.x);
            g.y = fma(f.y, h, g.y);
            a = fma(a, E[(size_t)i * n + i].x, a);
            b = fma(b, E[(size_t)j * n + j].x, b);
        }
        const int es = ((__double2hiint(a > b ? a : b) >> 20) & 0x7ff) - 1023;
        const float gr = f32_scaled(g.x, es), gi = f32_scaled(g.y, es), df = f32_scaled(b - a, es);
        const float h = fmaf(df, df, 4.f * fmaf(gr, gr, gi * gi));
        const float tau = copysignf(__fdividef(2.f, fabsf(df) + sqrtf(h)), df);
        const float2 kk = make_float2(tau * gr, tau * gi);
        if (fmaf(kk.x, kk.x, kk.y * kk.y) <= (STEP ? kRefCap1 * kRefCap1 : kRefCap0 * kRefCap0)) k = kk;
    }
    if (STEP == 1) {
        const float v = fabsf(k.x) + fabsf(k.y);
        mix_rows_add(mix_rows(d, n, 1), v, kRowUnit1, i, j, n, true);
        mix_rows_add(mix_rows(d, n, 2), v <= kRefCap2 ? v : 0.f, kRowUnit1, i, j, n, true);
    }
    float2* K = (float2*)d.pre;
    if (i <= j && j < n) {
        K[(size_t)j * n + i] = k;
        K[(size_t)i * n + j] = make_float2(-k.x, k.y);
    }
}

// K^2 (Hermitian) in FP32 pairs.  Step 0 stores it, step 1 F = K + K^2 / 2, of the angles up
// to kRefCap1, or to kRefCap2, whichever bounds K: a column far smaller than the others can
// have middling angles with many that are smaller still.
template <int STEP>
__global__ void __launch_bounds__(TILE_THREADS) k_mix_sq(const GateDesc* __restrict__ gd) {
    const GateDesc& d = gd[blockIdx.z];
    const int m = 2 * d.chi[d.q], n = 2 * d.chi[d.q + 2];
    if (!mix_active(d, m, n)) return;
    const int i0 = blockIdx.x * T64, j0 = blockIdx.y * T64;
    if (i0 >= n || j0 >= n || i0 > j0 || mix_off(d, n)) return;
    const float2* K = (const float2*)d.pre;
    // step 1: the angles in use, |Re K| + |Im K| at most this
    float cap = 1.f;
    if (STEP == 1 && mix_rows_above(mix_rows(d, n, 1), n, kRowUnit1, kRefRow1))
        cap = mix_rows_above(mix_rows(d, n, 2), n, kRowUnit1, kRefRow1) ? 0.f : kRefCap2;
    auto angle = [&](size_t t) {
        const float2 k = K[t];
        return STEP == 0 || fabsf(k.x) + fabsf(k.y) <= cap ? k : make_float2(0.f, 0.f);
    };
    Df acc = {};
    tile_product<Df, true, true, false, DfMulAdd<false>>(
        n,
        [&](int c, int k) {   // K[i, k] = -conj(K[k, i])
            if (i0 + c >= n) return Df{};
            const float2 v = angle((size_t)(i0 + c) * n + k);
            return Df{-v.x, v.y, 0.f, 0.f};
        },
        [&](int k, int c) {
            if (j0 + c >= n) return Df{};
            const float2 v = angle((size_t)(j0 + c) * n + k);
            return Df{v.x, v.y, 0.f, 0.f};
        },
        acc);
    const int i = i0 + (threadIdx.x & 7), j = j0 + (threadIdx.x >> 3);
    const double2 e2 = from_df(acc);
    const bool in = i < n && j < n;
    if (STEP == 0) {
        const float v = fabsf(acc.x) + fabsf(acc.y);
        mix_rows_add(mix_rows(d, n, 0), in ? v : 0.f, kRowUnit0, i, j, n, i0 != j0);
        if (!in) return;
        double2* D = (double2*)d.pre_d;
        D[(size_t)j * n + i] = e2;
        if (i0 != j0) D[(size_t)i * n + j] = make_double2(e2.x, -e2.y);
    } else {
        if (!in) return;
        const float2 k = angle((size_t)j * n + i);
        Df* F = mix_bufs(d, 1).F;
        const double hx = 0.5 * e2.x, hy = 0.5 * e2.y, kx = (double)k.x, ky = (double)k.y;
        F[(size_t)j * n + i] = df_of(hx + kx, hy + ky);
        if (i0 != j0) F[(size_t)i * n + j] = df_of(hx - kx, ky - hy);
    }
}

// Step 0: I + F = (I + C) (I + B'), C = E/2 + 3/8 E^2 + 5/16 E^3 = (I - E)^{-1/2} - I and
// B' = B - K^4/8 = K + (I + K^2)^{1/2} - I with B = K + K^2/2, without K where K^2 is too
// large for K^6 to vanish.  F = E/2 + B' + E R with R = 3/8 E + B/2 + E (5/16 E + 3/8 B): two
// products of E, in FP32 (E ~ 1e-6, K < 2^-10).  Left out: 35/128 E^4, 5/16 E^3 B, E K^4/16.
// |E|_2 was 2e-6 .. 5e-6 at n = 64 .. 512 and |K|_2 is at most 2.8e-3, so these are below 2e-17;
// at the largest row sums of E that are admitted (kRefRowE) below 2e-15.
__device__ __forceinline__ float2 mix_B(const float2& k, const double2& q, bool skip) {
    return skip ? make_float2(0.f, 0.f) : make_float2(fmaf(0.5f, (float)q.x, k.x), fmaf(0.5f, (float)q.y, k.y));
}
// f M[i, k] = f conj(M[k, i]) for rows i0 + c of a Hermitian matrix
__device__ __forceinline__ float2 mix_herm(const double2* M, float f, int i, int k, int n) {
    if (i >= n) return make_float2(0.f, 0.f);
    const double2 e = M[(size_t)i * n + k];
    return make_float2(f * (float)e.x, -f * (float)e.y);
}
__global__ void __launch_bounds__(TILE_THREADS) k_mix_r(const GateDesc* __restrict__ gd) {
    const GateDesc& d = gd[blockIdx.z];
    const int m = 2 * d.chi[d.q], n = 2 * d.chi[d.q + 2];
    if (!mix_active(d, m, n)) return;
    const int i0 = blockIdx.x * T64, j0 = blockIdx.y * T64;
    if (i0 >= n || j0 >= n || mix_off(d, n)) return;
    const double2 *E = (const double2*)d.pre_b, *Q = (const double2*)d.pre_d;
    const float2* K = (const float2*)d.pre;
    const bool skip = mix_rows_above(mix_rows(d, n, 0), n, kRowUnit0, kRefRow0);
    float2 acc = make_float2(0.f, 0.f);
    tile_product<float2, true, true, true, MulAdd>(
        n, [&](int c, int k) { return mix_herm(E, 1.f, i0 + c, k, n); },
        [&](int k, int c) {
            if (j0 + c >= n) return make_float2(0.f, 0.f);
            const size_t t = (size_t)(j0 + c) * n + k;
            const double2 e = E[t];
            const float2 b = mix_B(K[t], Q[t], skip);
            return make_float2(fmaf(0.375f, b.x, 0.3125f * (float)e.x), fmaf(0.375f, b.y, 0.3125f * (float)e.y));
        },
        acc);
    const int i = i0 + (threadIdx.x & 7), j = j0 + (threadIdx.x >> 3);
    if (i >= n || j >= n) return;
    const size_t t = (size_t)j * n + i;
    const double2 e = E[t];
    const float2 b = mix_B(K[t], Q[t], skip);
    mix_R(d, n)[t] = make_float2(fmaf(0.5f, b.x, fmaf(0.375f, (float)e.x, acc.x)),
                                 fmaf(0.5f, b.y, fmaf(0.375f, (float)e.y, acc.y)));
}
__global__ void __launch_bounds__(TILE_THREADS) k_mix_corr(const GateDesc* __restrict__ gd) {
    const GateDesc& d = gd[blockIdx.z];
    const int m = 2 * d.chi[d.q], n = 2 * d.chi[d.q + 2];
    if (!mix_active(d, m, n)) return;
    const int i0 = blockIdx.x * T64, j0 = blockIdx.y * T64;
    if (i0 >= n || j0 >= n || mix_off(d, n)) return;
    const double2 *E = (const double2*)d.pre_b, *Q = (const double2*)d.pre_d;
    const float2 *K = (const float2*)d.pre, *Rm = mix_R(d, n);
    const bool skip = mix_rows_above(mix_rows(d, n, 0), n, kRowUnit0, kRefRow0);
    float2 acc = make_float2(0.f, 0.f);
    tile_product<float2, true, true, true, MulAdd>(
        n, [&](int c, int k) { return mix_herm(E, 1.f, i0 + c, k, n); },
        [&](int k, int c) { return j0 + c < n ? Rm[(size_t)(j0 + c) * n + k] : make_float2(0.f, 0.f); }, acc);
    if (!skip)
        tile_product<float2, true, true, true, MulAdd>(
            n, [&](int c, int k) { return mix_herm(Q, -0.125f, i0 + c, k, n); },
            [&](int k, int c) {
                if (j0 + c >= n) return make_float2(0.f, 0.f);
                const double2 q = Q[(size_t)(j0 + c) * n + k];
                return make_float2((float)q.x, (float)q.y);
            },
            acc);
    const int i = i0 + (threadIdx.x & 7), j = j0 + (threadIdx.x >> 3);
    if (i >= n || j >= n) return;
    const size_t t = (size_t)j * n + i;
    double2 f = E[t];
    if (!skip) {
        f.x += Q[t].x;
        f.y += Q[t].y;
    }
    f.x = fma(0.5, f.x, (double)acc.x);
    f.y = fma(0.5, f.y, (double)acc.y);
    if (!skip) {
        f.x += (double)K[t].x;
        f.y += (double)K[t].y;
    }
    mix_bufs(d, 0).F[t] = df_of(f.x, f.y);
}

// dst = src + src F: F is at most 1e-3, so products and sums of FP32 pairs (2^-47) are as
// good as FP64 ones
template <int STEP>
__global__ void __launch_bounds__(TILE_THREADS) k_mix_mul(const GateDesc* __restrict__ gd) {
    const GateDesc& d = gd[blockIdx.z];
    const int m = 2 * d.chi[d.q], n = 2 * d.chi[d.q + 2];
    if (!mix_active(d, m, n)) return;
    const int i0 = blockIdx.x * T64, j0 = blockIdx.y * T64;
    if (i0 >= m || j0 >= n || mix_off(d, n)) return;
    const MixBufs b = mix_bufs(d, STEP);
    const int e = mix_exp(d.out->frob2);
    Df acc = {};
    tile_product<Df, false, true, false, DfMulAdd<true>>(
        n, [&](int c, int k) { return i0 + c < m ? to_df(b.src[(size_t)k * m + i0 + c], e, false) : Df{}; },
        [&](int k, int c) { return j0 + c < n ? b.F[(size_t)(j0 + c) * n + k] : Df{}; }, acc);
    const int i = i0 + (threadIdx.x & 7), j = j0 + (threadIdx.x >> 3);
    if (i >= m || j >= n) return;
    const size_t idx = (size_t)j * m + i;
    const double2 x = b.src[idx], y = from_df(acc);
    const double sc = ldexp(1.0, e);
    b.dst[idx] = make_double2(fma(y.x, sc, x.x), fma(y.y, sc, x.y));
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
    if (n_gates <= 0 || n_max < kMixMinCols || plain64(m_max, n_max)) return cudaSuccess;
    const int mt = m_max + n_max < kMixMaxRows ? m_max + n_max : kMixMaxRows;   // of an active gate
    const int mm = m_max < kMixMaxRows ? m_max : kMixMaxRows, nm = n_max < kMixMaxRows ? n_max : kMixMaxRows;
    int bx = (int)(((long long)mt * nm + 1023) / 1024);
    if (bx > 128) bx = 128;
    const int tn = (nm + T64 - 1) / T64, tm = (mm + T64 - 1) / T64;
    k_mix_build<<<dim3(bx, n_gates), 256, 0, s>>>(d, ctl);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = launch_jacobi_mix(d, n_gates, mt, nm, ctl, s, n_lead, spin_limit);
    if (e != cudaSuccess) return e;
    k_mix_first<<<dim3(tm + tn, tn, n_gates), TILE_THREADS, 0, s>>>(d, tm);
    k_mix_angle<0><<<dim3(tn, tn, n_gates), TILE_THREADS, 0, s>>>(d);
    k_mix_sq<0><<<dim3(tn, tn, n_gates), TILE_THREADS, 0, s>>>(d);
    k_mix_r<<<dim3(tn, tn, n_gates), TILE_THREADS, 0, s>>>(d);
    k_mix_corr<<<dim3(tn, tn, n_gates), TILE_THREADS, 0, s>>>(d);
    k_mix_mul<0><<<dim3(tm, tn, n_gates), TILE_THREADS, 0, s>>>(d);
    k_mix_angle<1><<<dim3(tn, tn, n_gates), TILE_THREADS, 0, s>>>(d);
    k_mix_sq<1><<<dim3(tn, tn, n_gates), TILE_THREADS, 0, s>>>(d);
    k_mix_mul<1><<<dim3(tm, tn, n_gates), TILE_THREADS, 0, s>>>(d);
    return cudaGetLastError();
}

}  // namespace tnsim
