// Batched one-sided (Hestenes) Jacobi SVD of theta for every gate of a launch.
//
// The paper decomposes theta with a Jacobi SVD (cusolverDnZgesvdj, Sec. IV.A);
// here the one-sided variant orthogonalises the n = 2chi_R columns of the
// m x n column-major working matrix W in place: W <- theta . V with V unitary,
// so at convergence the columns of W are u_j s_j.  V itself is never formed --
// the right site is recovered as U^H theta (see k_gemm.cu).
//
// Rotation of a column pair (i, j) (Hestenes 1958; Demmel & Veselic 1992, with
// the complex phase split off): a = |w_i|^2, b = |w_j|^2, g = w_i^H w_j = |g| e^{i phi}.
// If |g| > tol sqrt(a b):  zeta = (b - a) / (2|g|), t = sign(zeta) / (|zeta| + sqrt(1 + zeta^2)),
// c = 1/sqrt(1+t^2), s = c t, and
//     w_i <- c w_i - s e^{-i phi} w_j,     w_j <- s e^{i phi} w_i + c w_j,
// which makes the pair orthogonal.  Columns whose norm is below
// eps*sqrt(max(m,n))*|theta|_F are numerically zero and are not rotated.
//
// Schedule.  The columns are cut into blocks of BC.  A sweep visits every pair of
// blocks once in round-robin ("circle") order: P - 1 rounds of P/2 disjoint block
// pairs.  A visit stages both blocks in shared memory, rotates the BC x BC cross
// pairs in BC rounds of BC disjoint pairs and, in the first round of a sweep, the pairs
// inside each block as well (Visit32, visit64 below), then writes the
// blocks back.  Each sweep therefore rotates every column pair exactly once.  A sweep
// that rotates nothing ends the gate's iteration; reaching max_sweeps sets ENOCONV.
//
// Three kernels run this schedule with the same arithmetic: k_jacobi_cl, one cluster per gate,
// where all gates are resident at once; else k_jacobi, a queue, and beyond 256 rows in FP32
// k_jacobi_pf, the queue with a prefetching warp.  complex128 gates of up to kPlain64 rows and
// columns run all their sweeps in one visit of either kernel (plain64_sweeps below).
//
// k_jacobi is persistent: as many CTAs as the SMs hold claim visits of
// any gate from a device-side queue, so gates of different sizes and all rounds of
// a layer share the machine without waves.  The visits of a round are independent;
// a gate's next round opens when the last visit of the current one is reported.  An
// idle CTA polls with a sleep; if nothing progresses for spin_limit polls (default
// 2^22, settable per state) it sets an error flag and leaves; every other CTA leaves
// at its next claim, abandoning the claim, and the unfinished gates report status 5
// (the host reports ETIMEOUT).  k_jacobi_pf also polls for its own copies and threads, with
// a fixed limit and the same flag.  No other wait exists, and no CTA leaves with a copy in
// flight.
#include <float.h>

#include <algorithm>
#include <type_traits>

#include <cooperative_groups.h>

#include "jacobi_sched.cuh"
#include "tc_common.cuh"
#include "tnsim_internal.h"

namespace cg = cooperative_groups;

namespace tnsim {

// One visit in FP32.  A pair belongs to a group of LP lanes, each holding RPL rows of a
// column.  16 rows a lane up to m = 512 (LP = m / 16): the shuffles of the inner product
// and the rotation parameters are then shared by 32 / LP pairs of a warp, and a CTA of
// 16 LP threads leaves room for others on its SM that run while this one waits (with a
// whole warp per pair these took ~110 of ~180 issue slots per pair and step at m = 128).
// Shared memory holds a block as 16-byte units (two rows) [RPL / 2][BC columns][LP lanes]
// (a whole warp per pair: columns contiguous, [BC][RPL / 2][LP]), rows padded with zeros to
// RPL LP: the accesses have constant offsets, no bounds and no bank conflicts.
// Block I's columns stay in registers over the BC rounds of the cross pairs; in the first
// round of a sweep the pairs inside each block come first.  Column norms are tracked:
// exact at the start of the visit, then a - t|g| and b + t|g| (the eigenvalues of the
// pair's 2 x 2 Gram matrix).
// Inner products and norms run over the first md rows (EXT: fewer than the stored m).
template <int BC, int LP, int RPL, bool EXT>
struct Visit32 {
    static constexpr int U = RPL / 2, BLOCK = U * BC * LP;   // units per lane and column; units of a block
    static constexpr int COL = LP == 32 ? U * LP : LP;       // from a column to the next
    static constexpr int PITCH = LP == 32 ? LP : BC * LP;    // from a lane's unit to its next
    float4 *XI, *XJ;                                         // the two blocks
    int w, l, kd;   // this thread's group and lane, its units inside the first md rows

    __device__ __forceinline__ Visit32(float4* xi, float4* xj, int md)
        : XI(xi), XJ(xj), w(threadIdx.x / LP), l(threadIdx.x % LP), kd((md / 2 - l + LP - 1) / LP) {}
    // column c of the two blocks (c < 2 BC): this lane's first unit
    __device__ __forceinline__ float4* unit(int c) const {
        return (c >= BC ? XJ : XI) + (c & (BC - 1)) * COL + l;
    }
    // all visiting threads (a prefetching warp may share the CTA)
    static __device__ __forceinline__ void sync() { asm volatile("bar.sync 0, %0;" ::"n"(BC * LP) : "memory"); }
    static __device__ __forceinline__ float sum(float v) {
#pragma unroll
        for (int o = LP / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    }
    __device__ __forceinline__ float norm2(const float4 (&x)[U]) const {
        float a = 0.f;
#pragma unroll
        for (int k = 0; k < U; ++k)
            if (!EXT || k < kd)
                a = fmaf(x[k].x, x[k].x, fmaf(x[k].y, x[k].y, fmaf(x[k].z, x[k].z, fmaf(x[k].w, x[k].w, a))));
        return sum(a);
    }
    __device__ __forceinline__ float norm2(int c) const {
        float4 x[U];
        load(x, c);
        return norm2(x);
    }
    // x + d with the small correction d = (c-1) x + ... summed first and then added to x
    // with a single rounding.  Near convergence |(c-1) x| is below half an ulp of x: added
    // to an already rounded x + ... it would always round away, leaving c = 1 and growing
    // the pair's norm by a factor 1 + t^2 per rotation (a systematic drift of the singular
    // values in FP32).
    static __device__ __forceinline__ void rot2(float& ax, float& ay, float& bx, float& by, float cm1, float sr,
                                                float si) {
        const float ux = ax, uy = ay, vx = bx, vy = by;
        ax = ux + fmaf(-si, vy, fmaf(-sr, vx, cm1 * ux));
        ay = uy + fmaf(si, vx, fmaf(-sr, vy, cm1 * uy));
        bx = vx + fmaf(-si, uy, fmaf(sr, ux, cm1 * vx));
        by = vy + fmaf(si, ux, fmaf(sr, uy, cm1 * vy));
    }
    // The pair of the register column u (norm a) and the shared column cv (norm b), which
    // is read once and written back once; tg: a -> a - tg, b -> b + tg.
    __device__ __forceinline__ bool rotate(float4 (&u)[U], int cv, bool act, float tol2, float zthr, float a, float b,
                                           float& tg) const {
        float4* p = unit(cv);
        float4 v[U];
        float gr = 0.f, gi = 0.f, hr = 0.f, hi = 0.f;   // two chains each: a chain of 2 RPL FMAs waits 4 cycles on each
#pragma unroll
        for (int k = 0; k < U; ++k) {
            v[k] = p[k * PITCH];
            if (!EXT || k < kd) {
                gr = fmaf(u[k].x, v[k].x, fmaf(u[k].y, v[k].y, gr));
                gi = fmaf(u[k].x, v[k].y, fmaf(-u[k].y, v[k].x, gi));
                hr = fmaf(u[k].z, v[k].z, fmaf(u[k].w, v[k].w, hr));
                hi = fmaf(u[k].z, v[k].w, fmaf(-u[k].w, v[k].z, hi));
            }
        }
        gr = sum(gr + hr);
        gi = sum(gi + hi);
        float cm1, sr, si;
        if (!act || !rot_params_fast(a, b, gr, gi, tol2, zthr, cm1, sr, si, tg)) return false;
#pragma unroll
        for (int k = 0; k < U; ++k) {
            rot2(u[k].x, u[k].y, v[k].x, v[k].y, cm1, sr, si);
            rot2(u[k].z, u[k].w, v[k].z, v[k].w, cm1, sr, si);
            p[k * PITCH] = v[k];
        }
        return true;
    }
    __device__ __forceinline__ void load(float4 (&u)[U], int c) const {
        const float4* p = unit(c);
#pragma unroll
        for (int k = 0; k < U; ++k) u[k] = p[k * PITCH];
    }
    __device__ __forceinline__ void store(int c, const float4 (&u)[U]) const {
        float4* p = unit(c);
#pragma unroll
        for (int k = 0; k < U; ++k) p[k * PITCH] = u[k];
    }

    // The pairs inside both blocks, from exact norms.
    __device__ __forceinline__ void inner(int nI, int nJ, float tol2, float zthr, float* __restrict__ nrm,
                                          int& my_rot, int& my_vis) const {
        const float na0 = norm2(w), nb0 = norm2(BC + w);
        if (l == 0) {
            nrm[w] = na0;
            nrm[BC + w] = nb0;
        }
        sync();
        // pairs inside block I (the first half of the groups) and inside block J (the rest)
        constexpr int half = BC / 2;
        const int base = w < half ? 0 : BC, nblk = w < half ? nI : nJ;
        float4 u[U];
#pragma unroll 1
        for (int t = 0; t < BC - 1; ++t) {
            int a, b;
            rr_pair(BC, t, w < half ? w : w - half, a, b);
            const bool act = a < nblk && b < nblk;
            a += base;
            b += base;
            load(u, a);
            const float na = nrm[a], nb = nrm[b];
            float tg;
            const bool rot = rotate(u, b, act, tol2, zthr, na, nb, tg);
            my_vis += act && l == 0;
            __syncwarp();
            if (rot) {
                store(a, u);
                if (l == 0) {
                    ++my_rot;
                    nrm[a] = na - tg;
                    nrm[b] = nb + tg;
                }
            }
            sync();
        }
    }

    // The cross pairs: block I's columns in registers (u, loaded by the caller, and the
    // caller's to store).  The CTA's groups form two halves, each with its own barrier: in
    // the first BC / 2 rounds half h rotates I_h with J_h, in the others with the other half
    // of J.  A half's loads, shuffles and parameters then run beside the other's updates
    // (one barrier for all in every round: 50.2 against 43.6 ms for the chi 256 layer).
    // Exact norms first unless inner() left tracked ones; the first pair of a group are its
    // own columns, so they need no barrier.
    __device__ __forceinline__ void cross(float4 (&u)[U], int nI, int nJ, bool tracked, float tol2, float zthr,
                                          float* __restrict__ nrm, int& my_rot, int& my_vis) const {
        constexpr int H = BC / 2;
        constexpr bool halves = H * LP % 32 == 0;   // named barriers count whole warps
        const int h = w / H;
        float a_i;
        if (tracked) {
            a_i = nrm[w];
        } else {
            a_i = norm2(u);
            const float b0 = norm2(BC + w);
            if (l == 0) nrm[BC + w] = b0;
            __syncwarp();
        }
#pragma unroll 1
        for (int t = 0; t < BC; ++t) {
            const int b = ((w + t) & (H - 1)) + H * (h ^ (t / H));
            const bool act = w < nI && b < nJ;
            const float nb = nrm[BC + b];
            float tg;
            const bool rot = rotate(u, BC + b, act, tol2, zthr, a_i, nb, tg);
            my_vis += act && l == 0;
            __syncwarp();
            if (rot) {
                a_i -= tg;
                if (l == 0) {
                    ++my_rot;
                    nrm[BC + b] = nb + tg;
                }
            }
            if (!halves || (t & (H - 1)) == H - 1) sync();
            else asm volatile("bar.sync %0, %1;" ::"r"(1 + h), "n"(H * LP) : "memory");
        }
    }

    // blocks in: 16-byte asynchronous copies (through L2, no registers held), every copy of
    // both blocks in flight at once; zeros past the stored rows and columns.  The caller's
    // barrier follows the wait.
    __device__ __forceinline__ void copy_in(const float2* WI, int nI, const float2* WJ, int nJ, int m) const {
        const int units = m / 2;
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = BC * LP / 32;
        for (int c = warp; c < 2 * BC; c += nw) {
            const int cc = c & (BC - 1);
            const float2* src = (c < BC ? WI : WJ) + (size_t)cc * m;
            const int have = cc < (c < BC ? nI : nJ) ? units : 0;
            float4* dst = (c >= BC ? XJ : XI) + cc * COL;
#pragma unroll 4
            for (int i = lane; i < U * LP; i += 32) {
                float4* p = dst + (i / LP) * PITCH + i % LP;
                if (i < have) cp_async16(p, src + 2 * i);
                else *p = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");
    }
    // One block by one warp, a bulk copy per column counted on the mbarrier bar, zeros
    // likewise.  (512-byte copies, from [RPL / 2][BC][LP], took 25 k cycles for two blocks.)
    static __device__ __forceinline__ void bulk_in(float4* slot, const float2* W, int nc, int m, uint32_t bar) {
        static_assert(LP == 32, "columns contiguous");
        for (int c = 0; c < BC; ++c) {
            const int have = c < nc ? m / 2 : 0;
            float4* dst = slot + c * COL;
            for (int i = have + (threadIdx.x & 31); i < COL; i += 32) dst[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const int c = threadIdx.x & 31;
        if (c < nc)
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                    smem_u32(slot + c * COL)),
                "l"(W + (size_t)c * m), "r"(m * 8), "r"(bar)
                : "memory");
    }
    // block I's columns straight from the registers
    __device__ __forceinline__ void regs_out(const float4 (&u)[U], float2* WI, int nI, int m) const {
        if (w >= nI) return;
        float4* dst = reinterpret_cast<float4*>(WI + (size_t)w * m);
#pragma unroll
        for (int k = 0; k < U; ++k)
            if (k * LP + l < m / 2) __stcg(dst + k * LP + l, u[k]);
    }
    // blocks out (L2 stores), by the warps from warp0 on
    __device__ __forceinline__ void copy_out(float2* WI, int nI, float2* WJ, int nJ, int m, int warp0) const {
        const int units = m / 2;
        const int warp = (int)(threadIdx.x >> 5) - warp0, lane = threadIdx.x & 31, nw = BC * LP / 32 - warp0;
        for (int c = warp; c < nI + nJ; c += nw) {
            const bool isI = c < nI;
            const int cc = isI ? c : c - nI;
            float4* dst = reinterpret_cast<float4*>((isI ? WI : WJ) + (size_t)cc * m);
            const float4* src = (isI ? XI : XJ) + cc * COL;
#pragma unroll 4
            for (int i = lane; i < units; i += 32) __stcg(dst + i, src[(i / LP) * PITCH + i % LP]);
        }
    }
};

// shared-memory block back to W (L2 stores) by the threads from first_thread on
template <typename C>
__device__ __forceinline__ void copy_block_out_from(C* dst, const C* src, int count, int first_thread) {
    const int units = (int)((size_t)count * sizeof(C) / 16);
    const int4* s = reinterpret_cast<const int4*>(src);
    int4* d = reinterpret_cast<int4*>(dst);
    const int nt = (int)blockDim.x - first_thread;
    for (int i = (int)threadIdx.x - first_thread; i < units; i += nt) __stcg(d + i, s[i]);
}

// One visit in FP64.  Each of an SM's four schedulers issues one FP64 warp instruction in
// 64 cycles, so FP64 instruction counts per scheduler are the time: 8 + 32 per 64 rows and
// pair for the inner product and the update, and everything else is arranged to cost
// little.  The per-lane partial products of the step's BC pairs go to shared memory, and
// one warp per scheduler sums those of BC / 4 pairs and forms their rotation parameters:
// 6 + 12 instructions instead of 10 + ~150 in each of the BC warps (shuffle reductions
// and FP64 square roots and divisions, which took more than half of the time at m = 64).
// Rows past m cost nothing (a register layout like the FP32 visit's padded m = 180 to 256).
// Pairs of step t: the BC - 1 rounds inside both blocks first (intra), then the BC rounds
// of the cross pairs.  All column norms are tracked from exact ones at the start.
constexpr int kRed64 = 33;
struct Par64 {
    double cm1, sr, si;
    int rot, pad_;
};
template <int BC>
__device__ __forceinline__ void pair64(int t, int w, bool intra, int nI, int nJ, int& ca, int& cb, bool& act) {
    if (intra && t < BC - 1) {
        constexpr int half = BC / 2;
        const int base = w < half ? 0 : BC, nblk = w < half ? nI : nJ;
        int a, b;
        rr_pair(BC, t, w < half ? w : w - half, a, b);
        act = a < nblk && b < nblk;
        ca = base + a;
        cb = base + b;
    } else {
        const int b = (w + t - (intra ? BC - 1 : 0)) % BC;
        act = w < nI && b < nJ;
        ca = w;
        cb = BC + b;
    }
}
template <int BC>
__device__ __forceinline__ void visit64(double2* __restrict__ XI, double2* __restrict__ XJ, int m, int nI, int nJ, bool intra, float tol,
                                        double zthr, double2* __restrict__ red, double* __restrict__ nrm,
                                        Par64* __restrict__ par, int& my_rot, int& my_vis) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto col = [&](int c) { return c < BC ? XI + (size_t)c * m : XJ + (size_t)(c - BC) * m; };
    for (int c = warp; c < 2 * BC; c += BC) {
        const double2* x = col(c);
        double a = 0.0;
        if (c < BC ? c < nI : c - BC < nJ)
            for (int r = lane; r < m; r += 32) a = fma(x[r].x, x[r].x, fma(x[r].y, x[r].y, a));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) nrm[c] = a;
    }
    __syncthreads();
    const int steps = (intra ? BC - 1 : 0) + (nI > 0 && nJ > 0 ? BC : 0);
    for (int t = 0; t < steps; ++t) {
        int ca, cb;
        bool act;
        pair64<BC>(t, warp, intra, nI, nJ, ca, cb, act);
        double2* xa = col(ca);
        double2* xb = col(cb);
        double2 g = make_double2(0.0, 0.0);
        if (act) {
#pragma unroll 4
            for (int r = lane; r < m; r += 32) {
                const double2 u = xa[r], v = xb[r];
                g.x = fma(u.x, v.x, fma(u.y, v.y, g.x));
                g.y = fma(u.x, v.y, fma(-u.y, v.x, g.y));
            }
        }
        red[warp * kRed64 + lane] = g;
        __syncthreads();
        if (warp < 4) {
            constexpr int LP = 128 / BC, LC = LP / 2, E = 32 / LC;   // lanes per pair and per component, terms per lane
            const int p = warp * (BC / 4) + lane / LP;
            const bool im = (lane & LC) != 0;
            const double* term = reinterpret_cast<const double*>(red + p * kRed64 + (lane % LC)) + (im ? 1 : 0);
            double s = term[0];
#pragma unroll
            for (int i = 1; i < E; ++i) s += term[2 * LC * i];
#pragma unroll
            for (int o = LC / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            const double so = __shfl_xor_sync(0xffffffffu, s, LC);
            const double gr = im ? so : s, gi = im ? s : so;
            int pa, pb;
            bool on, rot = false;
            pair64<BC>(t, p, intra, nI, nJ, pa, pb, on);
            double cm1, sr, si, tg = 0.0;
            const double a = nrm[pa], b = nrm[pb];
            if (on) rot = rot_params64(a, b, gr, gi, tol, zthr, cm1, sr, si, tg);
            __syncwarp();
            const bool first = lane % LP == 0;
            if (first) par[p].rot = rot;
            if (first && rot) {
                nrm[pa] = a - tg;
                nrm[pb] = b + tg;
                par[p].cm1 = cm1;
                par[p].sr = sr;
                par[p].si = si;
            }
            const unsigned vis = __ballot_sync(0xffffffffu, on && first), rts = __ballot_sync(0xffffffffu, rot && first);
            if (lane == 0) {
                my_vis += __popc(vis);
                my_rot += __popc(rts);
            }
        }
        __syncthreads();
        if (act && par[warp].rot) {
            const double cm1 = par[warp].cm1, sr = par[warp].sr, si = par[warp].si;
#pragma unroll 2
            for (int r = lane; r < m; r += 32) {
                const double2 u = xa[r], v = xb[r];
                double2 nu, nv;
                nu.x = u.x + fma(-si, v.y, fma(-sr, v.x, cm1 * u.x));
                nu.y = u.y + fma(si, v.x, fma(-sr, v.y, cm1 * u.y));
                nv.x = v.x + fma(-si, u.y, fma(sr, u.x, cm1 * v.x));
                nv.y = v.y + fma(si, u.x, fma(sr, u.y, cm1 * v.y));
                xa[r] = nu;
                xb[r] = nv;
            }
        }
        __syncthreads();
    }
}

// A plain gate (plain64: at most 30 rows and columns): all its sweeps in one visit, the
// columns X (n x m) in shared memory.  Column blocks of 16 whatever the launch's: 15 steps
// of the pairs inside the one or two blocks, whose norms are summed again for every pair,
// then 16 of the cross pairs with tracked norms.  Every sum is the lanes' terms by halving
// distances (a lane has row r, in the cross pairs 2 r and 2 r + 1), the parameters are IEEE
// operations: see kPlain64.  A pair's sums are its warp's, four of them in six instead of
// twenty additions.  The parameters of all 16 pairs are one warp's, two lanes each: of seven
// divisions two of a pair share an issue slot three times, and the seventh, in the test, is
// only made within rounding of the limit.  Bound by FP64 issue: 30 instructions per pair and
// step over the schedulers and 75 of the one warp, 64 cycles each.
// sw: the sweeps done; returns whether the last one still rotated.
struct Plain64 {
    double val[16][4];   // a, b, gr, gi of the step's pairs (cross pairs: gr, gi)
    double nrm[32];      // cross pairs: tracked norms
    Par64 par[16];
};
__device__ __forceinline__ void plain_pair(int s, int p, int n, int& ca, int& cb, bool& act) {
    const int nI = min(16, n), nJ = n - nI;
    if (s < 15) {
        const int base = p < 8 ? 0 : 16, nblk = p < 8 ? nI : nJ;
        int a, b;
        rr_pair(16, s, p & 7, a, b);
        act = a < nblk && b < nblk;
        ca = base + a;
        cb = base + b;
    } else {
        const int b = (p + s - 15) & 15;
        act = p < nI && b < nJ;
        ca = p;
        cb = 16 + b;
    }
}
// v[0..NV-1] summed over the warp's lanes: the sum of v[2 (lane >> 4 & 1) + (lane >> 3 & 1)]
// (NV = 4) or v[lane >> 4 & 1] (NV = 2)
template <int NV>
__device__ __forceinline__ double plain_sums(const double (&v)[NV], int lane) {
    const bool u4 = lane & 16, u3 = lane & 8;
    double k;
    if constexpr (NV == 4) {
        double k0 = u4 ? v[2] : v[0], k1 = u4 ? v[3] : v[1];
        k0 += __shfl_xor_sync(0xffffffffu, u4 ? v[0] : v[2], 16);
        k1 += __shfl_xor_sync(0xffffffffu, u4 ? v[1] : v[3], 16);
        k = u3 ? k1 : k0;
        k += __shfl_xor_sync(0xffffffffu, u3 ? k0 : k1, 8);
    } else {
        k = u4 ? v[1] : v[0];
        k += __shfl_xor_sync(0xffffffffu, u4 ? v[0] : v[1], 16);
        k += __shfl_xor_sync(0xffffffffu, k, 8);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
    return k;
}
// g2 / b > lim a without the division unless the product is within rounding of g2
__device__ __forceinline__ bool plain_above(double g2, double b, double la) {
    const double p = la * b;
    const long long ig = __double_as_longlong(g2), ip = __double_as_longlong(p);
    constexpr long long lo = 0x0080000000000000ll, hi = 0x7f00000000000000ll;
    if (ig > lo && ig < hi && ip > lo && ip < hi && (ig > ip + 64 || ig < ip - 64)) return ig > ip;
    return g2 / b > la;
}
__device__ __noinline__ int plain64_sweeps(double2* X, int m, int n, int max_sweeps, double tol2, double zthr, Plain64& S,
                                           int& sw, int& my_rot, int& my_vis) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int steps = n > 16 ? 31 : 15;
    int rot_any = 0;
    for (sw = 0; sw < max_sweeps;) {
        int rots = 0;
        for (int s = 0; s < steps; ++s) {
            if (s == 15) {
                // norms at the start of the cross pairs
                for (int c = warp; c < n; c += nw) {
                    const double2* x = X + (size_t)c * m;
                    double a = 0.0;
                    if (c < 16) {
                        for (int k = 0; k < 2; ++k)
                            if (2 * lane + k < m) {
                                const double2 u = x[2 * lane + k];
                                a = fma(u.x, u.x, fma(u.y, u.y, a));
                            }
                    } else if (lane < m) {
                        const double2 u = x[lane];
                        a = fma(u.x, u.x, fma(u.y, u.y, a));
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
                    if (lane == 0) S.nrm[c] = a;
                }
            }
            for (int p = warp; p < 16; p += nw) {
                int ca, cb;
                bool act;
                plain_pair(s, p, n, ca, cb, act);
                if (!act) continue;
                const double2 *xa = X + (size_t)ca * m, *xb = X + (size_t)cb * m;
                if (s < 15) {
                    double v[4] = {0.0, 0.0, 0.0, 0.0};
                    if (lane < m) {
                        const double2 x = xa[lane], y = xb[lane];
                        v[0] = fma(x.x, x.x, x.y * x.y);
                        v[1] = fma(y.x, y.x, y.y * y.y);
                        v[2] = fma(x.x, y.x, x.y * y.y);
                        v[3] = fma(x.x, y.y, -x.y * y.x);
                    }
                    const double k = plain_sums<4>(v, lane);
                    if ((lane & 7) == 0) S.val[p][lane >> 3] = k;
                } else {
                    double v[2] = {0.0, 0.0};
#pragma unroll
                    for (int k = 0; k < 2; ++k)
                        if (2 * lane + k < m) {
                            const double2 x = xa[2 * lane + k], y = xb[2 * lane + k];
                            v[0] = fma(x.x, y.x, fma(x.y, y.y, v[0]));
                            v[1] = fma(x.x, y.y, fma(-x.y, y.x, v[1]));
                        }
                    const double k = plain_sums<2>(v, lane);
                    if ((lane & 15) == 0) S.val[p][2 + (lane >> 4)] = k;
                }
            }
            __syncthreads();
            if (warp == 0) {
                const int p = lane >> 1;
                const bool h = lane & 1;
                int ca, cb;
                bool act;
                plain_pair(s, p, n, ca, cb, act);
                const double gr = S.val[p][2], gi = S.val[p][3];
                const double a = s < 15 ? S.val[p][0] : act ? S.nrm[ca] : 0.0;
                const double b = s < 15 ? S.val[p][1] : act ? S.nrm[cb] : 0.0;
                double g2 = 0.0;
                bool rot = false;
                if (act) {
                    g2 = gr * gr + gi * gi;
                    rot = a > zthr && b > zthr && plain_above(g2, b, tol2 * a);
                }
                const unsigned on = __ballot_sync(0xffffffffu, rot);
                __syncwarp();
                if (rot) {
                    const double gabs = sqrt(g2);
                    const double q1 = (h ? gr : b - a) / (h ? gabs : 2 * gabs);            // zeta; gr / |g|
                    const double q2 = (h ? gi : copysign(1.0, q1)) /
                                      (h ? gabs : fabs(q1) + sqrt(1.0 + q1 * q1));         // t; gi / |g|
                    const double t = __shfl_sync(on, q2, lane & ~1);
                    const double rr = sqrt(1.0 + t * t);
                    const double q3 = (h ? t : -(t * t)) / (h ? rr : rr * (1.0 + rr));     // c - 1; s
                    if (h) {
                        S.par[p].sr = q3 * q1;
                        S.par[p].si = q3 * q2;
                    } else {
                        S.par[p].cm1 = q3;
                        if (s >= 15) {
                            const double tg = __dmul_rn(t, gabs);   // rounded by itself
                            S.nrm[ca] = __dsub_rn(a, tg);
                            S.nrm[cb] = __dadd_rn(b, tg);
                        }
                    }
                }
                if (!h) S.par[p].rot = rot;
                const int r = __popc(on) / 2, v = __popc(__ballot_sync(0xffffffffu, act && !h));
                rots += r;
                if (lane == 0) {
                    my_rot += r;
                    my_vis += v;
                }
            }
            __syncthreads();
            for (int p = warp; p < 16; p += nw) {
                int ca, cb;
                bool act;
                plain_pair(s, p, n, ca, cb, act);
                if (!act || !S.par[p].rot || lane >= m) continue;
                const double cm1 = S.par[p].cm1, sr = S.par[p].sr, si = S.par[p].si;
                double2 *xa = X + (size_t)ca * m + lane, *xb = X + (size_t)cb * m + lane;
                const double2 u = *xa, v = *xb;
                double2 nu, nv;
                nu.x = u.x + fma(-si, v.y, fma(-sr, v.x, cm1 * u.x));
                nu.y = u.y + fma(si, v.x, fma(-sr, v.y, cm1 * u.y));
                nv.x = v.x + fma(-si, u.y, fma(sr, u.x, cm1 * v.x));
                nv.y = v.y + fma(si, u.x, fma(sr, u.y, cm1 * v.y));
                *xa = nu;
                *xb = nv;
            }
            __syncthreads();
        }
        rot_any = __syncthreads_or(rots);
        ++sw;
        if (!rot_any) break;
    }
    return rot_any;
}

// Persistent kernel: every CTA repeatedly claims one visit (gate g, global round
// number, block pair v) from the gates' claim words, processes it, and reports it.
// The last visit of a round advances that gate to its next round (and, at the end
// of a sweep, decides convergence).  Gates are scanned in descriptor order, which
// the host sorts by decreasing size.  A CTA never waits while holding a claim, so
// a CTA with nothing to claim only waits for work that running CTAs are doing.
// EXT (FP32): the columns of the complex128 gates' preconditioner, [theta; I] in GateDesc::pre
// (k_fp64.cu); rotated over all m + n rows, the inner products and norms over the first m.
// LP, RPL: lanes per pair and rows per lane of the launch's largest m (FP32; 32 and 0 for FP64).
template <typename T, int BC, int LP, int RPL, int MINB, bool EXT>
__global__ void __launch_bounds__(BC * LP, MINB)
k_jacobi(const GateDesc* __restrict__ gd, int n_gates, int n_lead, double tol_in, int max_sweeps,
         JacobiCtl* __restrict__ ctl, unsigned spin_limit) {
    using C = typename CT<T>::type;
    constexpr bool F64 = sizeof(T) == 8;
    static_assert(BC * LP >= 64, "warp 0 claims while the others write back");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* X = reinterpret_cast<C*>(smem_raw);       // FP64: [2*BC][m], column-major
    __shared__ int s_g, s_rnd, s_v, s_exit, s_rot, s_vis;
    __shared__ T s_bn[2 * BC];                   // tracked squared norms (FP32: of block J's columns; FP64: of both)
    __shared__ double2 s_red[sizeof(T) == 8 ? BC * kRed64 : 1];
    __shared__ Par64 s_par[sizeof(T) == 8 ? BC : 1];
    __shared__ typename std::conditional<F64, Plain64, int>::type s_plain;
    __shared__ short s_V[kScanTable];            // visits per round of each gate

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned spins = 0, last_progress = 0;
    // where this CTA starts scanning: spread over the n_lead leading gates (those as large
    // as the first; the descriptors come sorted by decreasing size), so the CTAs share out
    // the largest gates instead of crowding the first ones; afterwards the gate it last
    // claimed, and from there on in descriptor order
    int scan0 = (int)(((long long)blockIdx.x * n_lead) / gridDim.x);
    for (int g = threadIdx.x; g < n_gates && g < kScanTable; g += blockDim.x)
        s_V[g] = (short)tour_of<BC, F64>(gd[g]).V;
    __syncthreads();

    int have_next = 0, nxt_g = -1, nxt_rnd = 0, nxt_v = 0;   // warp 0: a claim made during the last visit
    int nxt_err = 0;                                          // the error flag read during the last visit
    for (;;) {
        if (warp == 0) {
            int found = 0, fg = -1, frnd = 0, fv = 0, err = 0;
            if (have_next) {
                found = 1;
                fg = nxt_g;
                frnd = nxt_rnd;
                fv = nxt_v;
                err = nxt_err;
                have_next = 0;
            } else {
                if (lane == 0) err = *((volatile int*)&ctl->error);
                claim_scan<BC, F64>(gd, n_gates, s_V, scan0, lane, found, fg, frnd, fv);
            }
            if (found) scan0 = fg;
            if (lane == 0) {
                s_exit = 0;
                s_g = found ? fg : -1;
                s_rnd = frnd;
                s_v = fv;
                // after a timeout every CTA leaves, a claim in hand included: the gates
                // left unfinished report status 5
                if (err || (!found && (*((volatile int*)&ctl->n_finished) >= n_gates ||
                                       *((volatile int*)&ctl->error))))
                    s_exit = 1;
                s_rot = 0;
                s_vis = 0;
            }
        }
        __syncthreads();
        if (s_exit) break;
        if (s_g < 0) {
            if (threadIdx.x == 0) {
                const unsigned p = *((volatile unsigned*)&ctl->progress);
                if (p != last_progress) {
                    last_progress = p;
                    spins = 0;
                } else if (++spins > spin_limit) {
                    atomicExch(&ctl->error, 1);
                }
                __nanosleep(256);
            }
            __syncthreads();
            continue;
        }
        __threadfence();   // order the claim before reading the blocks of the previous round

        const int g = s_g, rnd = s_rnd, v = s_v;
        const GateDesc& d = gd[g];
        GateOut* out = d.out;
        const Tour tg = tour_of<BC, F64>(d);
        const int md = tg.m, n = tg.n, nb = tg.nb, P = tg.P, R = tg.R;
        const int m = EXT ? md + n : md;   // rows of a stored column
        int sweep = rnd / R;
        const int round = rnd - sweep * R;
        int last_rot = -1;   // one-block gates: whether the last sweep rotated (-1: see rot_sweep)
        C* Wm = EXT ? (C*)d.pre : (C*)d.W;
        // default tolerance: FP64, sqrt(m) * eps (LAPACK's one-sided Jacobi uses the same
        // scale), floored at 4 eps for tiny m; FP32, 2 eps.  Near convergence the columns
        // are almost orthogonal, so the FP32 partial sums of g stay small and its rounding
        // error is a fraction of eps sqrt(a b): the tighter test is resolvable, and it
        // matters because a pair left non-orthogonal at tol tilts the kept subspace by
        // about tol / (relative gap at the cut).  A column below eps*sqrt(max(m,n))*|theta|_F
        // is zero.
        const double tol = tol_in > 0.0 ? tol_in
                                        : (sizeof(T) == 4 ? 2.0 * Eps<T>::v : fmax(sqrt((double)md), 4.0) * Eps<T>::v);
        const T tol2 = (T)(tol * tol);
        double frob2 = out->frob2;
        if (EXT) {
            const double f = mix_scale(frob2);
            frob2 *= f * f;
        }
        const T zthr = (T)(Eps<T>::v * Eps<T>::v * (double)max(md, n) * frob2);

        int I, J;
        if (nb == 1) {
            I = 0;
            J = -1;
        } else {
            rr_pair(P, round, v, I, J);
            if (I >= nb) { I = J; J = -1; }
            else if (J >= nb) J = -1;
        }
        const bool intra = (round == 0);
        int my_rot = 0, my_vis = 0;
        bool plain = false;
        if constexpr (F64) {
            plain = plain64(md, n);
            if (plain) {
                copy_blocks_in(X, Wm, n * m, X, Wm, 0);
                __syncthreads();
                last_rot = plain64_sweeps(X, m, n, max_sweeps, tol2, zthr, s_plain, sweep, my_rot, my_vis);
                --sweep;   // the last one's number
                if (warp > 0) copy_block_out_from(Wm, X, n * m, 32);
            }
        }
        if (!plain && (J >= 0 || intra)) {
            const int colI = I * BC, nI = min(BC, n - colI);
            const int colJ = J >= 0 ? J * BC : 0, nJ = J >= 0 ? min(BC, n - colJ) : 0;
            using V32 = Visit32<BC, LP, RPL, EXT>;
            float4* const xs = reinterpret_cast<float4*>(smem_raw);
            const V32 vis(xs, xs + V32::BLOCK, md);
            if constexpr (sizeof(T) == 8)
                copy_blocks_in(X, Wm + (size_t)colI * m, nI * m, X + (size_t)BC * m, Wm + (size_t)colJ * m,
                               J >= 0 ? nJ * m : 0);
            else
                vis.copy_in(Wm + (size_t)colI * m, nI, Wm + (size_t)colJ * m, nJ, m);
            __syncthreads();
            // a gate of one block runs all its sweeps in this visit
            for (;;) {
                int rot = 0;
                if constexpr (sizeof(T) == 8) {
                    visit64<BC>(X, X + (size_t)BC * m, m, nI, nJ, intra, (float)tol, zthr, s_red, s_bn, s_par, rot, my_vis);
                } else {
                    if (intra) vis.inner(nI, nJ, tol2, zthr, s_bn, rot, my_vis);
                    if (nJ > 0) {
                        float4 u[V32::U];
                        vis.load(u, vis.w);
                        vis.cross(u, nI, nJ, intra, tol2, zthr, s_bn, rot, my_vis);
                        vis.store(vis.w, u);
                        __syncthreads();
                    }
                }
                my_rot += rot;
                if (nb > 1) break;
                last_rot = __syncthreads_or(rot);
                if (!last_rot || ++sweep >= max_sweeps) break;
            }
            if (warp > 0) {
                if constexpr (sizeof(T) == 8) {
                    copy_block_out_from(Wm + (size_t)colI * m, X, nI * m, 32);
                    if (J >= 0) copy_block_out_from(Wm + (size_t)colJ * m, X + (size_t)BC * m, nJ * m, 32);
                } else {
                    vis.copy_out(Wm + (size_t)colI * m, nI, Wm + (size_t)colJ * m, nJ, m, 1);
                }
            }
        }
        // warp 0 claims the next visit while the other warps write the blocks back (a CTA
        // never waits while holding a claim, so claiming before this visit's report is safe)
        if (warp == 0) {
            int found, fg, frnd, fv;
            if (lane == 0) nxt_err = *((volatile int*)&ctl->error);
            claim_scan<BC, F64>(gd, n_gates, s_V, scan0, lane, found, fg, frnd, fv);
            have_next = found;
            nxt_g = fg;
            nxt_rnd = frnd;
            nxt_v = fv;
        }
        my_rot = __reduce_add_sync(0xffffffffu, my_rot);
        my_vis = __reduce_add_sync(0xffffffffu, my_vis);
        if (lane == 0 && my_rot) atomicAdd(&s_rot, my_rot);
        if (lane == 0 && my_vis) atomicAdd(&s_vis, my_vis);
        __threadfence();   // every thread's block stores before the report
        __syncthreads();
        if (threadIdx.x == 0) {
            if (s_rot) {
                atomicAdd(&out->rot_sweep, s_rot);
                if (!EXT) atomicAdd(&out->rotations, (unsigned long long)s_rot);
            }
            if (s_vis && !EXT) atomicAdd(&out->visits, (unsigned long long)s_vis);
            __threadfence();
            const int dn = atomicAdd(&out->done, 1) + 1;
            if (dn == tg.V) {
                // last visit of this round: advance the gate
                out->done = 0;
                bool fin = false;
                if (round == R - 1) {
                    int rs = atomicExch(&out->rot_sweep, 0);
                    if (last_rot >= 0) rs = last_rot;
                    if (rs == 0 || sweep + 1 >= max_sweeps) {
                        fin = true;
                        out->sweeps = min(sweep + 1, max_sweeps);
                        // keep a timeout the contraction reported (5) before this launch
                        if (rs != 0 && out->status < 4) out->status = 4;
                    }
                }
                __threadfence();
                if (fin) {
                    atomicExch(&out->finished, 1);
                    atomicAdd(&ctl->n_finished, 1);
                } else {
                    atomicExch(&out->claim, (unsigned long long)(rnd + 1) << 32);
                }
                atomicAdd(&ctl->progress, 1u);
            }
        }
        __syncthreads();
    }
}

// The persistent kernel for FP32 columns so long that one CTA fills an SM (m > 256), with a
// warp beside the visiting threads: a visit's claim, copies, fences and report took 20 of its
// 49 k cycles at m = 512, and no other CTA covers them there.  In the cross pairs block I's
// columns are in registers, so its slot and a third one take the next visit's blocks: the
// extra warp claims the visit, has both blocks copied in, stores the finished visit's block
// J from its slot and reports it, while the others are at work on the next.
//   MID    the visiting threads arrive when block I's slot is free, the warp waits
//   READY  all: the visit is through, the next one's blocks are in place
// The warp claims ahead only while there are more visits than CTAs: a claim held while
// another CTA idles would delay its gate's round.  A CTA still never waits while it holds a
// claim, except for its own visit's end and copies.  Registers: 512 threads of 104 and a
// group of four warps (three leave) of 40 are within the launch's 640 x 96; with one extra
// warp and no redistribution 96 a thread spilled (37.5 against 41.4 ms).
// 100 qubits at chi 256, 50 gates of m = n = 512: 44.1 -> 37.5 ms.  At m <= 256 the CTAs of
// an SM cover for each other: this kernel took 4.5 against 4.3 ms for 32 gates at m = 256.
struct VisitInfo {
    float2 *WI, *WJ;             // the two blocks' columns
    GateOut* out;
    int nI, nJ, m;               // their columns (nI = 0: no work, nJ = 0: block I alone) and rows
    int intra, single;           // first round of a sweep; a gate of one block
    float tol2, zthr;
    int V, rnd, R, leave;        // visits of a round, round and rounds of a sweep (report); no more visits
};
template <int BC, int LP, int RPL>
__global__ void __launch_bounds__(BC * LP + 128, 1)
k_jacobi_pf(const GateDesc* __restrict__ gd, int n_gates, int n_lead, double tol_in, int max_sweeps,
            JacobiCtl* __restrict__ ctl, unsigned spin_limit) {
    using V32 = Visit32<BC, LP, RPL, false>;
    constexpr int NT = BC * LP, NW = NT / 32;
    constexpr unsigned kPolls = 1u << 24;   // of a wait for this CTA's own copies or threads
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4* const xs = reinterpret_cast<float4*>(smem_raw);   // slots: block I in 0, block J in 1 and 2 in turn
    __shared__ VisitInfo s_info[2];
    __shared__ int s_rot[2], s_vis[2], s_last[2];   // of a visit: rotations, pairs; one-block gates: 2 sweep + (it rotated)
    __shared__ int s_claimed;                       // the last visit claimed
    __shared__ int s_done;                          // warps whose part is stored and fenced, over all visits
    __shared__ float s_bn[2 * BC];
    __shared__ short s_V[kScanTable];
    __shared__ __align__(8) uint64_t s_full;
    const uint32_t bar = smem_u32(&s_full);
    const int lane = threadIdx.x & 31;
    auto mid_arrive = [] { __syncwarp(); asm volatile("fence.proxy.async.shared::cta;\nbar.arrive 3, %0;" ::"n"(NT + 32) : "memory"); };
    auto mid_wait = [] { __syncwarp(); asm volatile("bar.sync 3, %0;" ::"n"(NT + 32) : "memory"); };
    auto ready = [] { __syncwarp(); asm volatile("fence.proxy.async.shared::cta;\nbar.sync 4, %0;" ::"n"(NT + 32) : "memory"); };
    for (int g = threadIdx.x; g < n_gates && g < kScanTable; g += blockDim.x)
        s_V[g] = (short)tour_of<BC>(gd[g]).V;
    if (threadIdx.x < 2) s_rot[threadIdx.x] = s_vis[threadIdx.x] = s_last[threadIdx.x] = 0;
    if (threadIdx.x == 2) s_done = s_claimed = 0;
    if (threadIdx.x == 3) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\nfence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();

    if (threadIdx.x >= NT) {
        // ---- the prefetching warp (of a group of four: registers move by groups)
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
        if (threadIdx.x >= NT + 32) return;
        int scan0 = (int)(((long long)blockIdx.x * n_lead) / gridDim.x);
        unsigned spins = 0, last_progress = 0;
        uint32_t phase = 0;
        // a finished visit: block J out, then count it, and advance its gate after the
        // round's last one
        auto store_J = [&](int p) {
            const VisitInfo& q = s_info[p];
            if (lane < q.nJ)
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(q.WJ + (size_t)lane * q.m),
                             "r"(smem_u32(xs + (size_t)(1 + p) * V32::BLOCK + lane * V32::COL)), "r"(q.m * 8)
                             : "memory");
            asm volatile("cp.async.bulk.commit_group;\ncp.async.bulk.wait_group 0;\nfence.proxy.async;" ::: "memory");
            __threadfence();
            __syncwarp();
        };
        auto report = [&](int p) {
            if (lane == 0) {
                const VisitInfo& q = s_info[p];
                GateOut* out = q.out;
                if (s_rot[p]) {
                    atomicAdd(&out->rot_sweep, s_rot[p]);
                    atomicAdd(&out->rotations, (unsigned long long)s_rot[p]);
                }
                if (s_vis[p]) atomicAdd(&out->visits, (unsigned long long)s_vis[p]);
                __threadfence();
                if (atomicAdd(&out->done, 1) + 1 == q.V) {
                    out->done = 0;
                    bool fin = false;
                    int sweep = q.rnd / q.R;
                    if (q.rnd - sweep * q.R == q.R - 1) {
                        int rs = atomicExch(&out->rot_sweep, 0);
                        if (q.single) {
                            sweep = s_last[p] >> 1;
                            rs = s_last[p] & 1;
                        }
                        if (rs == 0 || sweep + 1 >= max_sweeps) {
                            fin = true;
                            out->sweeps = min(sweep + 1, max_sweeps);
                            // keep a timeout the contraction reported (5) before this launch
                            if (rs != 0 && out->status < 4) out->status = 4;
                        }
                    }
                    __threadfence();
                    if (fin) {
                        atomicExch(&out->finished, 1);
                        atomicAdd(&ctl->n_finished, 1);
                    } else {
                        atomicExch(&out->claim, (unsigned long long)(q.rnd + 1) << 32);
                    }
                    atomicAdd(&ctl->progress, 1u);
                }
                s_rot[p] = s_vis[p] = s_last[p] = 0;
            }
            __syncwarp();
        };
        for (int i = 0;; ++i) {
            const int p = i & 1;
            bool reported = i == 0;
            if (i > 0) mid_wait();
            int found = 0, fg = -1, frnd = 0, fv = 0, leave = 0;
            for (;;) {
                if (!reported && __all_sync(0xffffffffu, *((volatile int*)&s_done) == i * NW)) {
                    __threadfence();   // their part, before block J is read and reported
                    store_J(p ^ 1);
                    report(p ^ 1);
                    reported = true;
                }
                const int fin = *((volatile int*)&ctl->n_finished), err = *((volatile int*)&ctl->error);
                if (__any_sync(0xffffffffu, err || (reported && fin >= n_gates))) {
                    leave = 1;
                    break;
                }
                // ahead of the running visit's end only with work for every CTA
                if (__all_sync(0xffffffffu, reported || (long long)(n_gates - fin) * s_V[0] * 2 > (long long)gridDim.x * 3))
                    claim_scan<BC>(gd, n_gates, s_V, scan0, lane, found, fg, frnd, fv);
                if (found) break;
                if (reported) {
                    if (lane == 0) {
                        const unsigned pr = *((volatile unsigned*)&ctl->progress);
                        if (pr != last_progress) {
                            last_progress = pr;
                            spins = 0;
                        } else if (++spins > spin_limit) {
                            atomicExch(&ctl->error, 1);
                        }
                    }
                    __syncwarp();
                }
                __nanosleep(256);
            }
            if (found) {
                if (lane == 0) *((volatile int*)&s_claimed) = i;
                __threadfence();   // order the claim before reading the blocks of the previous round
                scan0 = fg;
                const GateDesc& d = gd[fg];
                const int m = 2 * d.chi[d.q], n = 2 * d.chi[d.q + 2];
                const int nb = (n + BC - 1) / BC, P = nb + (nb & 1), R = nb == 1 ? 1 : P - 1, round = frnd % R;
                int I = 0, J = -1;
                if (nb > 1) {
                    rr_pair(P, round, fv, I, J);
                    if (I >= nb) { I = J; J = -1; }
                    else if (J >= nb) J = -1;
                }
                const int nI = J >= 0 || round == 0 ? min(BC, n - I * BC) : 0, nJ = J >= 0 ? min(BC, n - J * BC) : 0;
                float2* W = (float2*)d.W;
                float2 *WI = W + (size_t)I * BC * m, *WJ = W + (size_t)(J >= 0 ? J : 0) * BC * m;
                if (nI > 0) {
                    asm volatile("fence.proxy.async;" ::: "memory");
                    if (lane == 0) mbar_expect_tx(bar, (uint32_t)((nI + nJ) * m) * 8u);
                    __syncwarp();
                    V32::bulk_in(xs, WI, nI, m, bar);
                    V32::bulk_in(xs + (size_t)(1 + p) * V32::BLOCK, WJ, nJ, m, bar);
                }
                if (lane == 0) {
                    VisitInfo& q = s_info[p];
                    q.WI = WI;
                    q.WJ = WJ;
                    q.out = d.out;
                    q.nI = nI;
                    q.nJ = nJ;
                    q.m = m;
                    q.intra = round == 0;
                    q.single = nb == 1;
                    q.V = nb == 1 ? 1 : P / 2;
                    q.rnd = frnd;
                    q.R = R;
                    q.leave = 0;
                    // tolerances: see k_jacobi
                    const double tol = tol_in > 0.0 ? tol_in : 2.0 * Eps<float>::v;
                    q.tol2 = (float)(tol * tol);
                    q.zthr = (float)(Eps<float>::v * Eps<float>::v * (double)max(m, n) * d.out->frob2);
                }
                if (nI > 0) {
                    if (!__all_sync(0xffffffffu, mbar_wait(bar, phase, kPolls))) {
                        if (lane == 0) atomicExch(&ctl->error, 1);
                        leave = 1;
                        mbar_wait(bar, phase, kPolls);   // not before the copies have landed
                    }
                    phase ^= 1;
                }
            }
            if (leave && lane == 0) s_info[p].leave = 1;
            __syncwarp();
            ready();
            if (!reported) {
                store_J(p ^ 1);
                // the visiting threads fence their part early in the next visit or on their way out
                bool done = false;
                for (unsigned k = 0; k < kPolls && !done; ++k) done = *((volatile int*)&s_done) >= i * NW;
                if (__all_sync(0xffffffffu, done)) {
                    __threadfence();
                    report(p ^ 1);
                } else if (lane == 0) {
                    atomicExch(&ctl->error, 1);
                }
            }
            if (leave) return;
        }
    }

    // ---- the visiting threads
    asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
    bool pending = false;   // the last visit's stores are not fenced yet
    auto signal = [&] {
        __threadfence();   // every thread's block stores before the report
        __syncwarp();
        if (lane == 0) atomicAdd(&s_done, 1);
        pending = false;
    };
    ready();
    for (int i = 0;; ++i) {
        const int p = i & 1;
        const VisitInfo& q = s_info[p];
        if (q.leave) {
            if (pending) signal();
            return;
        }
        const V32 vis(xs, xs + (size_t)(1 + p) * V32::BLOCK, q.m);
        int my_rot = 0, my_vis = 0;
        if (q.nJ > 0) {
            const int nI = q.nI, nJ = q.nJ;
            const bool intra = q.intra;
            const float tol2 = q.tol2, zthr = q.zthr;
            if (intra) vis.inner(nI, nJ, tol2, zthr, s_bn, my_rot, my_vis);
            float4 u[V32::U];
            vis.load(u, vis.w);
            mid_arrive();
            if (pending) signal();
            vis.cross(u, nI, nJ, intra, tol2, zthr, s_bn, my_rot, my_vis);
            vis.regs_out(u, q.WI, nI, q.m);
        } else {
            if (pending) signal();
            if (q.nI > 0) {
                // a gate of one block runs all its sweeps in this visit
                for (int sweep = 0;; ++sweep) {
                    int rot = 0;
                    vis.inner(q.nI, 0, q.tol2, q.zthr, s_bn, rot, my_vis);
                    my_rot += rot;
                    if (!q.single) break;
                    unsigned any;
                    asm volatile("{\n.reg .pred a, b;\nsetp.ne.u32 a, %1, 0;\nbarrier.cta.red.or.pred b, 0, %2, a;\nselp.u32 %0, 1, 0, b;\n}"
                                 : "=r"(any) : "r"((unsigned)rot), "n"(NT) : "memory");
                    if (threadIdx.x == 0) s_last[p] = 2 * sweep + (int)any;
                    if (!any || sweep + 1 >= max_sweeps) break;
                }
                vis.copy_out(q.WI, q.nI, q.WJ, 0, q.m, 0);
            }
            mid_arrive();
        }
        my_rot = __reduce_add_sync(0xffffffffu, my_rot);
        my_vis = __reduce_add_sync(0xffffffffu, my_vis);
        if (lane == 0 && my_rot) atomicAdd(&s_rot[p], my_rot);
        if (lane == 0 && my_vis) atomicAdd(&s_vis[p], my_vis);
        // a fence waits until the stores have landed: with the next visit in hand, later
        pending = true;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        // one lane's reading for the warp: the prefetching warp writes it meanwhile, and lanes
        // that read different values would part at signal's __syncwarp and the barrier
        __syncwarp();
        int ahead = lane == 0 ? *((volatile int*)&s_claimed) : 0;
        ahead = __shfl_sync(0xffffffffu, ahead, 0);
        if (ahead != i + 1) signal();
        ready();
    }
}

// One thread-block cluster per gate: the whole iteration with the columns in (distributed)
// shared memory.  In the persistent kernel a visit of a 128-row gate spends 12 k of its 40 k
// cycles on the claim, the copies through L2, the fence, the report and waiting for the
// round's other visits; a layer whose gates all fit on the GPU at once gains nothing from
// its queue.  Here CTA v of the cluster is seat v of the tournament: in round r it holds the
// blocks a = r + v and b = r - v modulo P - 1 (a = P - 1 and b = r for v = 0), rotates
// their pairs as above, and passes a to seat v - 1 and b to seat v + 1 (a turns into seat
// 0's b, the last seat's b into its own a) through distributed shared memory.  After the
// P - 1 rounds of a sweep every block is back, and the seats' rotation counts decide
// whether the iteration ends.  Seats beyond the gate's P / 2 only keep the barriers.
//   FP32: three block slots; b stays in its slot, a's columns are in registers, so two slots
// are free for the next round's blocks once every seat has loaded a (the first cluster
// barrier of a round, arrived at early).  FP64: four slots, two free.
template <typename T, int BC, int LP, int RPL, int MINB, bool EXT>
__global__ void __launch_bounds__(BC * LP, MINB)
k_jacobi_cl(const GateDesc* __restrict__ gd, double tol_in, int max_sweeps) {
    using C = typename CT<T>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ T s_n[2 * BC];
    __shared__ double2 s_red[sizeof(T) == 8 ? BC * kRed64 : 1];
    __shared__ Par64 s_par[sizeof(T) == 8 ? BC : 1];
    __shared__ int s_cnt[2][8];      // the seats' rotations in this sweep, by parity of the sweep
    __shared__ int s_rot, s_vis;
    cg::cluster_group cl = cg::this_cluster();
    const int seats = (int)cl.num_blocks(), v = (int)cl.block_rank();
    const GateDesc& d = gd[blockIdx.x / seats];
    GateOut* out = d.out;
    if (EXT && out->finished) return;   // outside the preconditioner: the whole cluster leaves
    const Tour tg = tour_of<BC>(d);
    const int md = tg.m, n = tg.n, nb = tg.nb, P = tg.P, R = tg.R;
    const int m = EXT ? md + n : md, last = P / 2 - 1;
    C* Wm = EXT ? (C*)d.pre : (C*)d.W;
    const double tol = tol_in > 0.0 ? tol_in
                                    : (sizeof(T) == 4 ? 2.0 * Eps<T>::v : fmax(sqrt((double)md), 4.0) * Eps<T>::v);
    const T tol2 = (T)(tol * tol);
    double frob2 = out->frob2;
    if (EXT) {
        const double f = mix_scale(frob2);
        frob2 *= f * f;
    }
    const T zthr = (T)(Eps<T>::v * Eps<T>::v * (double)max(md, n) * frob2);
    const bool seat = v <= last;
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) s_rot = s_vis = 0;
    if constexpr (sizeof(T) == 8) {
        if (plain64(md, n)) {   // one CTA's work
            if (v > 0) return;
            __shared__ Plain64 s_plain;
            C* const X = reinterpret_cast<C*>(smem_raw);
            int sw, my_rot = 0, my_vis = 0;
            copy_blocks_in(X, Wm, n * m, X, Wm, 0);
            __syncthreads();
            const int rs = plain64_sweeps(X, m, n, max_sweeps, tol2, zthr, s_plain, sw, my_rot, my_vis);
            copy_block_out_from(Wm, X, n * m, 0);
            if (tid == 0) {
                atomicAdd(&out->rotations, (unsigned long long)my_rot);
                atomicAdd(&out->visits, (unsigned long long)my_vis);
                out->sweeps = sw;
                if (rs != 0 && out->status < 4) out->status = 4;
                out->finished = 1;
            }
            return;
        }
    }

    using V32 = Visit32<BC, LP, sizeof(T) == 4 ? RPL : 2, EXT>;
    // a block slot in 16-byte units (a multiple of two elements: m is even)
    const int slot_units = sizeof(T) == 4 ? V32::BLOCK : BC * m;
    float4* const xs = reinterpret_cast<float4*>(smem_raw);
    auto slot = [&](int k) { return xs + (size_t)k * slot_units; };
    auto cols = [&](int b) { return b < nb ? min(BC, n - b * BC) : 0; };
    // seats and slots of this CTA's outgoing blocks
    const int to_a = v == 0 ? 0 : v - 1, to_b = v == last ? v : v + 1;
    const bool a_stays_a = v != 1, b_turns_a = v == last && v > 0;
    int sa = 1, sb = 0;                 // slots of a and b; FP64: pairs (0, 1) and (2, 3) in turn
    int blk_a = P - 1, blk_b = 0;
    if (v > 0) { blk_a = v; blk_b = P - 1 - v; }
    if (seat) {
        if constexpr (sizeof(T) == 4) {
            V32(slot(sa), slot(sb), md)
                .copy_in(Wm + (size_t)blk_a * BC * m, cols(blk_a), Wm + (size_t)blk_b * BC * m, cols(blk_b), m);
        } else {
            copy_blocks_in((C*)slot(sa), Wm + (size_t)blk_a * BC * m, cols(blk_a) * m, (C*)slot(sb),
                           Wm + (size_t)blk_b * BC * m, cols(blk_b) * m);
        }
    }
    cl.sync();   // every seat runs before anything is written into it
    int sweep = 0, my_rot = 0, my_vis = 0, rs = 0;
    for (;; ++sweep) {
        int rot = 0;
        for (int r = 0; r < R; ++r) {
            int a = P - 1, b = r;
            if (v > 0) {
                a = (r + v) % (P - 1);
                b = (r - v + P - 1) % (P - 1);
            }
            const int nA = seat ? cols(a) : 0, nB = seat ? cols(b) : 0;
            if constexpr (sizeof(T) == 4) {
                const V32 vis(slot(sa), slot(sb), md);
                float4 u[V32::U];
                const int na = (sb + 1) % 3, nbs = (sb + 2) % 3;   // slots of the next a and b
                if (seat) {
                    if (r == 0) vis.inner(nA, nB, tol2, zthr, s_n, rot, my_vis);
                    vis.load(u, vis.w);
                }
                asm volatile("barrier.cluster.arrive.release;" ::: "memory");
                if (seat && nA > 0 && nB > 0) vis.cross(u, nA, nB, r == 0, tol2, zthr, s_n, rot, my_vis);
                __syncthreads();
                if (r == R - 1) {
                    // this seat's count, to every CTA
                    const int wr = __reduce_add_sync(0xffffffffu, rot);
                    if (lane == 0 && wr) atomicAdd(&s_rot, wr);
                    __syncthreads();
                    if (tid < seats) cl.map_shared_rank(&s_cnt[sweep & 1][v], tid)[0] = s_rot;
                }
                asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
                if (seat) {
                    float4* da = cl.map_shared_rank(slot(a_stays_a ? na : nbs), to_a) + vis.w * V32::COL + vis.l;
#pragma unroll
                    for (int k = 0; k < V32::U; ++k) da[k * V32::PITCH] = u[k];
                    float4* db = cl.map_shared_rank(slot(b_turns_a ? na : nbs), to_b);
                    const float4* src = slot(sb);
#pragma unroll 4
                    for (int i = tid; i < V32::BLOCK; i += BC * LP) db[i] = src[i];
                }
                sa = na;
                sb = nbs;
            } else {
                const int na = (sa + 2) & 3, nbs = (sb + 2) & 3;
                if (seat) {
                    visit64<BC>((double2*)slot(sa), (double2*)slot(sb), m, nA, nB, r == 0, (float)tol, (double)zthr, s_red,
                                (double*)s_n, s_par, rot, my_vis);
                    float4* da = cl.map_shared_rank(slot(a_stays_a ? na : nbs), to_a);
                    float4* db = cl.map_shared_rank(slot(b_turns_a ? na : nbs), to_b);
                    const float4 *pa = slot(sa), *pb = slot(sb);
#pragma unroll 2
                    for (int i = tid; i < slot_units; i += BC * LP) {
                        da[i] = pa[i];
                        db[i] = pb[i];
                    }
                }
                if (r == R - 1) {
                    const int wr = __reduce_add_sync(0xffffffffu, rot);
                    if (lane == 0 && wr) atomicAdd(&s_rot, wr);
                    __syncthreads();
                    if (tid < seats) cl.map_shared_rank(&s_cnt[sweep & 1][v], tid)[0] = s_rot;
                }
                sa = na;
                sb = nbs;
            }
            __syncwarp();
            cl.sync();   // the next round's blocks have arrived
        }
        my_rot += rot;
        rs = 0;
        for (int k = 0; k < seats; ++k) rs += s_cnt[sweep & 1][k];
        __syncthreads();
        if (tid == 0) s_rot = 0;
        __syncthreads();
        if (rs == 0 || sweep + 1 >= max_sweeps) break;
    }
    // every block is back at its first seat
    if (seat) {
        if constexpr (sizeof(T) == 4) {
            V32(slot(sa), slot(sb), md)
                .copy_out(Wm + (size_t)blk_a * BC * m, cols(blk_a), Wm + (size_t)blk_b * BC * m, cols(blk_b), m, 0);
        } else {
            copy_block_out_from(Wm + (size_t)blk_a * BC * m, (const C*)slot(sa), cols(blk_a) * m, 0);
            copy_block_out_from(Wm + (size_t)blk_b * BC * m, (const C*)slot(sb), cols(blk_b) * m, 0);
        }
        if (!EXT) {
            my_rot = __reduce_add_sync(0xffffffffu, my_rot);
            my_vis = __reduce_add_sync(0xffffffffu, my_vis);
            if (lane == 0 && my_rot) atomicAdd(&s_rot, my_rot);
            if (lane == 0 && my_vis) atomicAdd(&s_vis, my_vis);
            __syncthreads();
            if (tid == 0) {
                atomicAdd(&out->rotations, (unsigned long long)s_rot);
                atomicAdd(&out->visits, (unsigned long long)s_vis);
            }
        }
    }
    if (v == 0 && tid == 0) {
        out->sweeps = sweep + 1;
        if (rs != 0 && out->status < 4) out->status = 4;
        out->finished = 1;
    }
}

constexpr size_t kOneCta = 116 << 10;   // dynamic shared memory that leaves no room for a second CTA

// Launch k_jacobi_cl when all the gates' clusters are resident at once; *used tells.
template <typename T, int BC, int LP, int RPL, int MINB, bool EXT = false>
static cudaError_t launch_cl(const GateDesc* d, int n_gates, int m_max, int n_max, double tol, int max_sweeps,
                             cudaStream_t s, bool* used) {
    using C = typename CT<T>::type;
    *used = false;
    const int nb = (n_max + BC - 1) / BC;
    const int seats = (nb + 1) / 2;
    if (seats > 8) return cudaSuccess;
    const auto kernel = k_jacobi_cl<T, BC, LP, RPL, MINB, EXT>;
    const size_t smem = sizeof(T) == 4 ? (size_t)3 * BC * LP * RPL * sizeof(C) : (size_t)4 * BC * m_max * sizeof(C);
    static SmemLimit limit;
    cudaError_t e = allow_dynamic_smem((const void*)kernel, limit);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = seats;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(n_gates * seats));
    cfg.blockDim = dim3(BC * LP);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int fit = 0, dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if (n_gates * seats <= sms && smem < kOneCta) {
        // one CTA per SM, where every SM's pipes and schedulers are its own: the cluster
        // scheduler otherwise packs two on an SM beside idle ones
        cfg.dynamicSmemBytes = kOneCta;
        if ((e = cudaOccupancyMaxActiveClusters(&fit, kernel, &cfg)) != cudaSuccess) return e;
        if (n_gates > fit) cfg.dynamicSmemBytes = smem;
    }
    if (n_gates > fit && (e = cudaOccupancyMaxActiveClusters(&fit, kernel, &cfg)) != cudaSuccess) return e;
    if (n_gates > fit) return cudaSuccess;
    *used = true;
    return cudaLaunchKernelEx(&cfg, kernel, d, tol, max_sweeps < 1 ? 1 : max_sweeps);
}

template <int BC, int LP, int RPL>
static cudaError_t launch_pf(const GateDesc* d, int n_gates, int n_lead, int n_max, double tol, int max_sweeps,
                             JacobiCtl* ctl, cudaStream_t s, unsigned spin_limit) {
    const auto kernel = k_jacobi_pf<BC, LP, RPL>;
    const size_t smem = (size_t)3 * BC * LP * RPL * sizeof(float2);
    static SmemLimit limit;
    cudaError_t e = allow_dynamic_smem((const void*)kernel, limit);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const int nb = (n_max + BC - 1) / BC;
    const long long visits = (long long)n_gates * ((nb == 1) ? 1 : (nb + (nb & 1)) / 2);
    const int lead = (n_lead < 1 || n_lead > n_gates) ? n_gates : n_lead;
    kernel<<<(unsigned)(visits < sms ? visits : sms), BC * LP + 128, smem, s>>>(
        d, n_gates, lead, tol, max_sweeps < 1 ? 1 : max_sweeps, ctl, spin_limit ? spin_limit : kSpinLimit);
    return cudaGetLastError();
}

template <typename T, int BC, int LP, int RPL, int MINB, bool EXT = false>
static cudaError_t launch_bc(const GateDesc* d, int n_gates, int n_lead, int m_max, int n_max, double tol,
                             int max_sweeps, JacobiCtl* ctl, cudaStream_t s, unsigned spin_limit) {
    using C = typename CT<T>::type;
    const auto kernel = k_jacobi<T, BC, LP, RPL, MINB, EXT>;
    // FP64: two blocks, or all columns of a plain gate
    const size_t smem = sizeof(T) == 8 ? std::max((size_t)2 * BC * m_max, (size_t)std::min(n_max, kPlain64) * std::min(m_max, kPlain64)) * sizeof(C)
                                       : (size_t)2 * BC * LP * RPL * sizeof(C);
    static SmemLimit limit;
    cudaError_t e = allow_dynamic_smem((const void*)kernel, limit);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, BC * LP, smem)) != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorLaunchOutOfResources;
    // no more CTAs than visits that can run at once
    const int nb = (n_max + BC - 1) / BC;
    const long long visits = (long long)n_gates * ((nb == 1) ? 1 : (nb + (nb & 1)) / 2);
    long long grid = (long long)sms * per_sm;
    if (grid > visits) grid = visits;
    if (grid < 1) grid = 1;
    const int lead = (n_lead < 1 || n_lead > n_gates) ? n_gates : n_lead;
    kernel<<<(unsigned)grid, BC * LP, smem, s>>>(d, n_gates, lead, tol, max_sweeps < 1 ? 1 : max_sweeps, ctl,
                                                 spin_limit ? spin_limit : kSpinLimit);
    return cudaGetLastError();
}

// Block width BC and lanes per pair LP per precision: the two staged blocks take
// 2 BC m elements of shared memory (at most 128 KB), and the register columns leave
// 16 warps per SM, in one CTA at m = 512 and in up to eight at m = 64.  Two
// configurations per shape: cfg 0 -- wide blocks (fewer rounds per sweep); cfg 1 --
// half-width blocks, more CTAs per SM (independent barriers, twice the rounds).  FP64
// visits keep no column in registers: 8-column blocks of up to 256
// rows let two or three CTAs share an SM's FP64 pipe and fill each other's waits.  Bit 1 of a
// state's configuration (QR preconditioning, k_qr.cu) does not change this launch.
// tnsim_autotune times every configuration on a real layer.
template <typename T>
cudaError_t launch_jacobi(const GateDesc* d, int n_gates, int m_max, int n_max, double tol,
                          int max_sweeps, JacobiCtl* ctl, cudaStream_t s, int cfg, int n_lead,
                          unsigned spin_limit) {
    if (n_gates <= 0) return cudaSuccess;
    const bool narrow = (cfg & 1) != 0;
#define TNSIM_CL(BC, LP, RPL, MINB) launch_cl<T, BC, LP, RPL, MINB>(d, n_gates, m_max, n_max, tol, max_sweeps, s, &used)
#define TNSIM_JAC(BC, LP, RPL, MINB) launch_bc<T, BC, LP, RPL, MINB>(d, n_gates, n_lead, m_max, n_max, tol, max_sweeps, ctl, s, spin_limit)
    if constexpr (sizeof(T) == 4) {
        if ((cfg & 4) && m_max <= jacobi_tc_max_rows())
            return launch_jacobi_tc(d, n_gates, n_lead, n_max, tol, max_sweeps, ctl, s, spin_limit);
        if (!narrow) {
            bool used = false;
            cudaError_t e = cudaSuccess;
            if (m_max <= 64) e = TNSIM_CL(16, 4, 16, 1);
            else if (m_max <= 128) e = TNSIM_CL(16, 8, 16, 1);
            else if (m_max <= 256) e = TNSIM_CL(16, 16, 16, 2);
            if (e != cudaSuccess || used) return e;
        }
        if (m_max <= 64) return narrow ? TNSIM_JAC(8, 8, 16, 8) : TNSIM_JAC(16, 4, 16, 8);
        if (m_max <= 128) return narrow ? TNSIM_JAC(8, 8, 16, 8) : TNSIM_JAC(16, 8, 16, 4);
        if (m_max <= 256) return narrow ? TNSIM_JAC(8, 16, 16, 4) : TNSIM_JAC(16, 16, 16, 2);
        if (m_max <= 512) return narrow ? TNSIM_JAC(8, 32, 16, 2) : launch_pf<16, 32, 16>(d, n_gates, n_lead, n_max, tol, max_sweeps, ctl, s, spin_limit);
        return TNSIM_JAC(8, 32, 32, 1);
    } else {
        if (!narrow && m_max <= 256) {
            bool used = false;
            const cudaError_t e = TNSIM_CL(8, 32, 0, 1);
            if (e != cudaSuccess || used) return e;
        }
        if (m_max <= 512) return narrow ? TNSIM_JAC(4, 32, 0, 2) : TNSIM_JAC(8, 32, 0, 2);
        return TNSIM_JAC(4, 32, 0, 1);
    }
#undef TNSIM_JAC
}

cudaError_t launch_jacobi_mix(const GateDesc* d, int n_gates, int mt_max, int n_max, JacobiCtl* ctl, cudaStream_t s,
                              int n_lead, unsigned spin_limit) {
    if (n_gates <= 0) return cudaSuccess;
    // sweep cap: more than these do not make the preconditioner better
    constexpr int sweeps = 20;
#define TNSIM_MIXCL(BC, LP, RPL, MINB) launch_cl<float, BC, LP, RPL, MINB, true>(d, n_gates, mt_max, n_max, kMixTol, sweeps, s, &used)
    bool used = false;
    cudaError_t e = cudaSuccess;
    if (mt_max <= 64) e = TNSIM_MIXCL(16, 4, 16, 1);
    else if (mt_max <= 128) e = TNSIM_MIXCL(16, 8, 16, 1);
    else if (mt_max <= 256) e = TNSIM_MIXCL(16, 16, 16, 1);
    else if (mt_max <= 384) e = TNSIM_MIXCL(16, 32, 12, 1);
    else if (mt_max <= 512) e = TNSIM_MIXCL(16, 32, 16, 1);
    if (e != cudaSuccess || used) return e;
#define TNSIM_MIX(BC, LP, RPL, MINB) launch_bc<float, BC, LP, RPL, MINB, true>(d, n_gates, n_lead, mt_max, n_max, kMixTol, sweeps, ctl, s, spin_limit)
    if (mt_max <= 64) return TNSIM_MIX(16, 4, 16, 8);
    if (mt_max <= 128) return TNSIM_MIX(16, 8, 16, 4);
    if (mt_max <= 256) return TNSIM_MIX(16, 16, 16, 2);
    if (mt_max <= 384) return TNSIM_MIX(16, 32, 12, 1);
    if (mt_max <= 512) return TNSIM_MIX(16, 32, 16, 1);
    return TNSIM_MIX(8, 32, 32, 1);
#undef TNSIM_MIX
}

template cudaError_t launch_jacobi<float>(const GateDesc*, int, int, int, double, int, JacobiCtl*, cudaStream_t, int,
                                          int, unsigned);
template cudaError_t launch_jacobi<double>(const GateDesc*, int, int, int, double, int, JacobiCtl*, cudaStream_t, int,
                                           int, unsigned);

}  // namespace tnsim
