// Scheduling and rotation-parameter pieces shared by the two persistent Jacobi
// kernels (k_jacobi.cu: rotations on the columns; k_jacobi_tc.cu: rotations on the
// block pair's Gram matrix with tensor-core block products).
#pragma once
#include <float.h>

#include "tnsim_internal.h"

namespace tnsim {

template <typename T> struct Eps;
template <> struct Eps<float> { static constexpr double v = FLT_EPSILON; };
template <> struct Eps<double> { static constexpr double v = DBL_EPSILON; };

// pair v of round r in the circle method for P players (P even)
__device__ __forceinline__ void rr_pair(int P, int r, int v, int& a, int& b) {
    if (v == 0) {
        a = P - 1;
        b = r;
    } else {
        a = (r + v) % (P - 1);
        b = (r - v + (P - 1)) % (P - 1);
    }
}

// Rotation parameters (c - 1, s e^{i phi}) of a column pair from a, b and g = gr + i gi.
// With tau = t / |g| = 2 sign(b - a) / (|b - a| + sqrt((b - a)^2 + 4 |g|^2)):
//     t^2 = tau^2 |g|^2,   c = (1 + t^2)^{-1/2},   s e^{i phi} = c tau g,
// so the rotation is unitary (c^2 + |s e^{i phi}|^2 = 1) for whatever tau, which only has to
// orthogonalise the pair to within rounding and comes from the approximate reciprocal and
// square root.  c takes one Newton step (its rounding error is then unbiased), and
// c - 1 = -t^2 c^2 / (1 + c) is formed without cancellation with a correctly rounded
// reciprocal: a bias of either would make the norms drift.  Three dependent special-function
// operations instead of eight (with |g|, zeta and 1 / |g| by IEEE square roots and
// reciprocals): the chain from g to the update is what the warps of a step wait for.
__device__ __forceinline__ bool rot_params_fast(float a, float b, float gr, float gi, float tol2, float zthr,
                                                float& cm1, float& sr, float& si, float& tg) {
    const float g2 = fmaf(gr, gr, gi * gi);
    if (!(a > zthr && b > zthr && g2 > (tol2 * a) * b)) return false;
    const float d = b - a, ad = fabsf(d);
    float h = fmaf(d, d, 4.f * g2);
    // sqrt(h); where h overflows, its larger part (norms that are equal leave 2 |g|)
    float rt = h * rsqrtf(h);
    if (h > 3e38f) rt = fmaxf(ad, 2.f * (g2 * rsqrtf(g2)));
    const float tau = copysignf(__fdividef(2.f, ad + rt), d);
    tg = tau * g2;                                        // the norms become a - t|g|, b + t|g|
    const float t2 = tg * tau;
    const float u = 1.f + t2;
    const float c0 = rsqrtf(u);
    const float c = fmaf(0.5f * c0, fmaf(-u * c0, c0, 1.f), c0);
    const float f = c * tau;
    sr = f * gr;
    si = f * gi;
    cm1 = -(t2 * c) * c * __frcp_rn(1.f + c);
    return true;
}

// x 2^-e in FP32 (truncated) and back, by integer operations: FP64 instructions, the
// conversions among them, issue once in 64 cycles per scheduler.
__device__ __forceinline__ float f32_scaled(double x, int e) {
    const int hi = __double2hiint(x), ex = ((hi >> 20) & 0x7ff) - 1023 - e + 127;
    if (ex <= 0) return 0.f;
    const unsigned mant = ((unsigned)(hi & 0xfffff) << 3) | ((unsigned)__double2loint(x) >> 29);
    return __uint_as_float(((unsigned)hi & 0x80000000u) | ((unsigned)min(ex, 254) << 23) | mant);
}
__device__ __forceinline__ double f64_scaled(float x, int e) {
    const unsigned b = __float_as_uint(x);
    const int ex = (int)((b >> 23) & 0xff) - 127 + 1023 + e;
    if (!(b & 0x7f800000u) || ex <= 0) return 0.0;
    return __hiloint2double((int)((b & 0x80000000u) | ((unsigned)min(ex, 2046) << 20) | ((b & 0x7fffffu) >> 3)),
                            (int)(b << 29));
}
// FP64 (gates beyond kPlain64; the others: plain64_sweeps in k_jacobi.cu): the test and a first
// tau in FP32 on values scaled by the larger norm's power of two;
// one Newton step for tau (without it a gate took 0.6 sweeps more) and the quantities that
// make the rotation unitary in FP64: 15 FP64 instructions while t < 2^-10 (where c - 1 is
// its series), 20 beyond, against about 150 with FP64 square roots and divisions.
__device__ __forceinline__ bool rot_params64(double a, double b, double gr, double gi, float tol, double zthr,
                                             double& cm1, double& sr, double& si, double& tg) {
    const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b), iz = __double_as_longlong(zthr);
    if (!(ia > iz && ib > iz)) return false;              // zthr >= 0: ordered like the values
    const int e = (int)((max(ia, ib) >> 52) & 0x7ff) - 1023;
    const float xr = fabsf(f32_scaled(gr, e)), xi = fabsf(f32_scaled(gi, e));
    const float mx = fmaxf(xr, xi);
    if (!(mx > 0.f)) return false;
    const float r = __fdividef(fminf(xr, xi), mx);
    const float gm = mx * sqrtf(fmaf(r, r, 1.f));
    if (!(gm > tol * sqrtf(f32_scaled(a, e) * f32_scaled(b, e)))) return false;
    const double d = b - a;
    const float df = f32_scaled(d, e);
    const float tauf = __fdividef(2.f, fabsf(df) + sqrtf(fmaf(df, df, 4.f * gm * gm)));
    double tau = f64_scaled(copysignf(tauf, df), -e);
    const double g2 = fma(gr, gr, gi * gi);
    // one Newton step on |g|^2 tau^2 + d tau = 1, its slope sqrt(d^2 + 4 |g|^2) in FP32
    const float slope = copysignf(__fdividef(1.f, sqrtf(fmaf(df, df, 4.f * gm * gm))), df);
    tau = fma(-fma(tau, fma(tau, g2, d), -1.0), f64_scaled(slope, -e), tau);
    tg = tau * g2;
    const double t2 = tg * tau;
    if (__double2hiint(t2) < 0x3eb00000) {                // t^2 < 2^-20: the next term is below 2^-61
        cm1 = t2 * fma(0.375, t2, -0.5);
    } else {
        // c = u^{-1/2} from an FP32 estimate c0: with e = 1 - u c0^2 (~1e-7),
        // c = c0 (1 + e/2 + 3/8 e^2 + O(e^3)); c - 1 is exact here
        const double u = 1.0 + t2;
        const double c0 = f64_scaled(rsqrtf(f32_scaled(u, 0)), 0);
        const double ee = fma(-u * c0, c0, 1.0);
        cm1 = fma(c0 * ee, fma(0.375, ee, 0.5), c0) - 1.0;
    }
    const double f = fma(tau, cm1, tau);
    sr = f * gr;
    si = f * gi;
    return true;
}

// Geometry of one gate's tournament: nb column blocks, P players (nb rounded up to
// even), R rounds per sweep and V visits (block pairs) per round.
struct Tour {
    int m, n, nb, P, R, V;
};
// F64: a plain gate is one visit, whatever BC.
template <int BC, bool F64 = false>
__device__ __forceinline__ Tour tour_of(const GateDesc& d) {
    Tour t;
    t.m = 2 * d.chi[d.q];
    t.n = 2 * d.chi[d.q + 2];
    t.nb = F64 && plain64(t.m, t.n) ? 1 : (t.n + BC - 1) / BC;
    t.P = t.nb + (t.nb & 1);
    t.R = (t.nb == 1) ? 1 : t.P - 1;
    t.V = (t.nb == 1) ? 1 : t.P / 2;
    return t;
}

constexpr unsigned kSpinLimit = 1u << 22;   // default idle polls without any progress before giving up
constexpr int kScanTable = 2048;              // gates whose visit count is cached in shared memory

// Warp-parallel claim of one visit (warp 0): each lane checks one gate per pass (one
// L2 round trip), the first claimable gate in descriptor order from gate scan0 on
// (wrapping around) is tried with an atomic.  found = 0 when nothing is claimable now.
template <int BC, bool F64 = false>
__device__ __forceinline__ void claim_scan(const GateDesc* __restrict__ gd, int n_gates, const short* s_V, int scan0,
                                           int lane, int& found, int& fg, int& frnd, int& fv) {
    found = 0;
    fg = -1;
    frnd = 0;
    fv = 0;
    const int nchunks = (n_gates + 31) / 32;
    for (int c = 0; c < nchunks && !found; ++c) {
        const int k = 32 * c + lane;
        const int g = k < n_gates ? (scan0 + k) % n_gates : n_gates;   // every gate once
        bool ok = false;
        int V = 0;
        GateOut* o = nullptr;
        if (g < n_gates) {
            o = gd[g].out;
            V = g < kScanTable ? (int)s_V[g] : tour_of<BC, F64>(gd[g]).V;
            const int fin = *((volatile int*)&o->finished);
            const unsigned long long cur = *((volatile unsigned long long*)&o->claim);
            ok = !fin && (unsigned)(cur & 0xffffffffull) < (unsigned)V;
        }
        unsigned mask = __ballot_sync(0xffffffffu, ok);
        while (mask && !found) {
            const int l = __ffs(mask) - 1;
            int got = 0;
            if (lane == l) {
                const unsigned long long st = atomicAdd(&o->claim, 1ull);
                if ((unsigned)(st & 0xffffffffull) < (unsigned)V) {
                    got = 1;
                    fg = g;
                    frnd = (int)(st >> 32);
                    fv = (int)(st & 0xffffffffull);
                }
            }
            got = __shfl_sync(0xffffffffu, got, l);
            if (got) {
                fg = __shfl_sync(0xffffffffu, fg, l);
                frnd = __shfl_sync(0xffffffffu, frnd, l);
                fv = __shfl_sync(0xffffffffu, fv, l);
                found = 1;
            }
            mask &= mask - 1;
        }
    }
}

// Both blocks of a visit into shared memory with asynchronous 16-byte copies
// (cp.async.cg: through L2, no registers held), so every copy of both blocks is in
// flight at once; the caller's barrier follows the wait.
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem_src) : "memory");
}
template <typename C>
__device__ __forceinline__ void copy_blocks_in(C* dI, const C* sI, int countI, C* dJ, const C* sJ, int countJ) {
    const int uI = (int)((size_t)countI * sizeof(C) / 16), uJ = (int)((size_t)countJ * sizeof(C) / 16);
    const int4* a = reinterpret_cast<const int4*>(sI);
    const int4* b = reinterpret_cast<const int4*>(sJ);
    int4* da = reinterpret_cast<int4*>(dI);
    int4* db = reinterpret_cast<int4*>(dJ);
    for (int i = threadIdx.x; i < uI; i += blockDim.x) cp_async16(da + i, a + i);
    for (int i = threadIdx.x; i < uJ; i += blockDim.x) cp_async16(db + i, b + i);
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}
}  // namespace tnsim
