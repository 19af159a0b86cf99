// Sums over cells and the control of the reconstruction solve: partial sums to
// norms and Gram-Schmidt coefficients, the Givens step, the start and the end
// of a cycle, and the conditions of the device-controlled graphs.
//
// Partial sums are stored part[q][variable][row] (row: the producer's blocks in
// cell order, R rows in all, rs per cell block), so that the threads of a sum
// read consecutive numbers.
//
// These kernels are a few blocks of latency: FP64 divisions and square roots (285
// and 346 ns for a warp whatever its active lanes; warps on one SM sub-partition
// queue for its FP64 pipe), L2 round trips and the launch.  What follows a sum
// is therefore done by the block that formed it, a block per system, the four of
// a case a cluster that its hardware barrier joins; the cluster (of a batch the
// last one to finish) then sets the graph's condition: one launch for the norm, the Givens
// step, the condition and a single mesh's end of the cycle, one for the residual's norm, the
// masks, g and the condition.  With the per-cell equations the first of the two (8.2 us
// at 41,000 triangles) is a block of the update's launch (control_end): ten steps at
// 41,000 triangles, mixed, 4.89 -> 4.55 ms, at 800, FP64, 5.44 -> 5.14 ms, a batch of 64
// 19.1 -> 18.5 ms.  One block with a case's four systems was slower (10.0 us for the
// first of the two at 41,000 triangles: four FP64 chains on one SM, and 25 us for the
// sums at 1M).
#pragma once

#include <cuda_runtime.h>

#include "gks_solve32.cuh"

namespace gks {
namespace {

constexpr int kReduceThreads = 256;

// sum of at(b) over b = b0 + t, b0 + t + kReduceThreads, ... < b1 (t the
// thread), added in that order as the plain loop does, so the sum is the same
// bit for bit; the loads are issued eight at a time, so a thread waits for a
// few L2 round trips instead of one per term (a case's 4,000 cell blocks at 1M
// are 16 terms per thread)
template <typename F>
__device__ __forceinline__ double strided_sum(int t, int b0, int b1, F &&at)
{
    constexpr int U = 8;
    double acc = 0.0;
    for (int b = b0 + t; b < b1; b += U * kReduceThreads) {
        double x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int bb = b + u * kReduceThreads;
            x[u] = bb < b1 ? at(bb) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (b + u * kReduceThreads < b1) acc += x[u];
    }
    return acc;
}

// The sum of acc over the block, to every lane of the first warp.  sh: one value per warp.
__device__ __forceinline__ double block_total(double acc, double *sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x < 32) {
        s = sh[threadIdx.x & 7];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    return s;
}

// The block's sum of column q of the partial sums for variable v, rows b0..b1:
// every lane of the first warp gets it.  sh: one value per warp.
__device__ __forceinline__ double block_sum(const double *part, int q, int v, int64_t R, int b0, int b1, double *sh)
{
    const double *p = part + ((int64_t)q * 4 + v) * R;
    return block_total(strided_sum(threadIdx.x, b0, b1, [&](int b) { return p[b]; }), sh);
}

// out[s][q] = sum over the rows of case(s) of column q, q < nq, and with vn given
// co[s][q] = sum / vn[s][q]^2 (the Gram-Schmidt coefficient of the unnormalised
// basis vector q; q < nco).  Grid (nq, ns).  on (may be NULL): the systems to sum.
// ran (may be NULL) = run: the running systems, for a kernel that changes run.
__global__ void __launch_bounds__(kReduceThreads) k_reduce(const double *__restrict__ part, int64_t R,
                                                           const int32_t *__restrict__ seg, int rs, double *out,
                                                           int ostride, const double *__restrict__ vn, int vstride,
                                                           double *co, int cstride, int nco,
                                                           const int32_t *__restrict__ on, const int32_t *run,
                                                           int32_t *ran)
{
    __shared__ double sh[kReduceThreads / 32];
    const int q = blockIdx.x, sy = blockIdx.y, c = sy >> 2;
    if (on && !on[sy]) return;
    const double n = q < nco ? vn[sy * vstride + q] : 0.0;
    const double acc = block_sum(part, q, sy & 3, R, rs * seg[c], rs * seg[c + 1], sh);
    if (threadIdx.x == 0) {
        out[sy * ostride + q] = acc;
        if (q == 0 && ran) ran[sy] = run[sy];
        if (q < nco) co[sy * cstride + q] = n > 0.0 ? acc / (n * n) : 0.0;
    }
}

// ---- conditions

// Where a control kernel's answer "any system has the flag" goes once its systems
// are done: the graph's condition h (set), a word for the host (word, may be
// NULL); ctr[slot] (slot >= 0) counts the run.  begin: a new solve, no cycles
// yet; limit > 0: the answer is no once more than limit cycles ran (each cycle
// takes at least one iteration of every active system, which stops at maxit, so
// the limit maxit + 1 is a backstop that a correct solve never reaches).
struct Cond {
    cudaGraphConditionalHandle h;
    int64_t *ctr;
    int64_t limit;
    int32_t *word;
    uint32_t *ticket;       // blocks done, back to 0 by itself
    int set, slot, begin;
};

// Whether any of the ns flags is set, once every block of the launch has written
// its own: known to the case's four blocks for a single mesh, else to the first
// block of the last cluster alone (*last).
__device__ __forceinline__ bool any_flag(const int32_t *flag, int ns, uint32_t *ticket, bool *last)
{
    __shared__ int is_last;
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    const unsigned clusters = gridDim.x / 4;
    *last = true;
    if (clusters > 1) {
        if (threadIdx.x == 0) {
            is_last = 0;
            if ((blockIdx.x & 3) == 0) {
                __threadfence();
                is_last = atomicInc(ticket, clusters - 1) == clusters - 1;
                __threadfence();
            }
        }
        __syncthreads();
        *last = is_last != 0;
        if (!*last) return false;
    }
    int a = 0;
    for (int q = threadIdx.x; q < ns; q += blockDim.x) a |= __ldcg(flag + q);
    return __syncthreads_or(a) != 0;
}

__device__ __forceinline__ void put_cond(const Cond &cd, bool any)
{
    unsigned v = any ? 1u : 0u;
    if (cd.slot >= 0) cd.ctr[cd.slot] += 1;
    if (cd.begin) cd.ctr[kCtrGuard] = 0;
    if (cd.limit > 0 && cd.ctr[kCtrGuard] > cd.limit) v = 0u;
    if (cd.word) *cd.word = (int32_t)v;
    if (cd.set) cudaGraphSetConditional(cd.h, v);
}

// ... by the first thread of a cluster
__device__ __forceinline__ void set_cond(const Cond &cd, bool any)
{
    if (threadIdx.x == 0 && (blockIdx.x & 3) == 0) put_cond(cd, any);
}

// A cycle of the device-controlled solve begins: counted for the launch and work
// totals and against the cycle limit.
__global__ void k_cycle_count(int64_t *ctr)
{
    if (threadIdx.x != 0) return;
    ctr[kCtrCycles] += 1;
    ctr[kCtrGuard] += 1;
}

// ---- small GMRES state of all systems

struct Krylov {
    int m, ns;
    double *H, *cs, *sn, *g, *y, *vn;
    float *y32;             // FP32 copy of y (mixed mode) or NULL
    int32_t *ctl;
    double *bnorm, *beta;
    int32_t *sexp;          // FP32 basis (else NULL): exponents [current][next]
    double rtol, eta;
    int maxit;
};

__device__ __forceinline__ double pow2_exact(int e)
{
    e = e < -1022 ? -1022 : (e > 1023 ? 1023 : e);
    return __longlong_as_double((long long)(e + 1023) << 52);
}

// Arnoldi index j of system sy, by one warp: the new Hessenberg column from the
// raw sums hc (plus h2 of a second Gram-Schmidt pass, if given) and shift on its
// diagonal (1 when V_j was taken off the new vector, else 0), the earlier
// rotations applied, a new rotation, the rotated residual g and the stopping
// test (stop: it ends the cycle here in any case).  The column's divisions are done by the lanes together, and only the
// chain of rotations (four FP64 instructions each) is serial.
__device__ __forceinline__ void givens_step(const Krylov &k, int sy, int j, const double *hc, int hstride,
                                            const double *h2, int h2stride, double shift, double hnext,
                                            bool stop, double (*sh)[kMaxRestart + 1])
{
    const int lane = threadIdx.x & 31, m = k.m;
    // Hessenberg column of the normalised basis: h_kj = <V_k, u_j> / (vn_k vn_j),
    // h_{j+1,j} = |V_{j+1}| / vn_j; the new vector's norm becomes vn_{j+1}
    double *h = sh[0], *c0 = sh[1], *s0 = sh[2], *hr = sh[3];
    const double nj = k.vn[sy * (m + 1) + j];
    for (int q = lane; q <= j + 1; q += 32) {
        const double a = q <= j ? hc[sy * hstride + q] + (h2 ? h2[sy * h2stride + q] : 0.0) : hnext;
        h[q] = a / (q <= j ? k.vn[sy * (m + 1) + q] * nj : nj) + (q == j ? shift : 0.0);
        if (q < j) {
            c0[q] = k.cs[sy * m + q];
            s0[q] = k.sn[sy * m + q];
        }
    }
    __syncwarp();
    const double gj = k.g[sy * (m + 1) + j], bn = k.bnorm[sy], be = k.beta[sy];
    const int it = k.ctl[kCtlIters * k.ns + sy] + 1;
    double t0 = h[0];
#pragma unroll 4
    for (int q = 0; q < j; ++q) {
        const double c = c0[q], s = s0[q], t1 = h[q + 1];
        const double u = c * t0 + s * t1;
        t0 = c * t1 - s * t0;
        if (lane == 0) hr[q] = u;
    }
    const double t1 = h[j + 1];
    // hypot where the squares leave FP64's range
    const double d2 = t0 * t0 + t1 * t1;
    double id, dd;
    if (d2 > 1e-280 && d2 < 1e280) {
        id = rsqrt(d2);
        dd = d2 * id;
    } else {
        dd = hypot(t0, t1);
        id = dd > 0.0 ? 1.0 / dd : 0.0;
    }
    const double c = dd > 0.0 ? t0 * id : 1.0, s = dd > 0.0 ? t1 * id : 0.0;
    __syncwarp();
    for (int q = lane; q < j; q += 32) k.H[((int64_t)sy * (m + 1) + q) * m + j] = hr[q];
    if (lane != 0) return;
    k.H[((int64_t)sy * (m + 1) + j) * m + j] = dd;
    k.vn[sy * (m + 1) + j + 1] = hnext;
    k.cs[sy * m + j] = c;
    k.sn[sy * m + j] = s;
    k.g[sy * (m + 1) + j + 1] = -s * gj;
    k.g[sy * (m + 1) + j] = c * gj;
    k.ctl[kCtlJv * k.ns + sy] = j + 1;
    k.ctl[kCtlIters * k.ns + sy] = it;
    // stop the cycle at the target, or (mixed precision, eta > 0) once the inner
    // residual has dropped by eta: the FP64 refinement residual then restarts it
    const double gn = fabs(s * gj);
    if (gn <= k.rtol * bn || gn <= k.eta * be || !(hnext > 0.0) || it >= k.maxit || j + 1 == m || stop)
        k.ctl[kCtlRunning * k.ns + sy] = 0;
}

// End of a cycle for system sy, by one warp: y = H^{-1} g on the first jv columns
// (upper triangular after the rotations), column by column, the lanes holding
// the right-hand side (the diagonal's reciprocals are formed together); then
// y_k /= vn_k, the coefficients of the unnormalised preconditioned vectors.
// With sexp (FP32 basis, rows [current][next] exponents e of the scale 2^-e of
// the first basis vector): y is also scaled by 2^-e of the current cycle (the
// combination adds 2^e sum y_k Z_k, so its FP32 sums stay near unit size), and
// the next residual's exponent comes from the cycle's estimate |g_jv| of its
// norm (at least 1e-3 rtol |b|).
__device__ __forceinline__ void cycle_solve(const Krylov &k, int sy)
{
    const int lane = threadIdx.x & 31, m = k.m;
    const int jv = k.ctl[kCtlJv * k.ns + sy];
    if (jv <= 0) return;
    // lane l holds the entries l and l + 32 (jv <= kMaxRestart = 64)
    const double *Hs = k.H + (int64_t)sy * (m + 1) * m;
    double rh[2], iv[2], sc[2];
    const double f = k.sexp ? pow2_exact(-k.sexp[sy]) : 1.0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int r = lane + 32 * q;
        rh[q] = r < jv ? k.g[sy * (m + 1) + r] : 0.0;
        iv[q] = r < jv ? 1.0 / Hs[(int64_t)r * m + r] : 0.0;
        sc[q] = r < jv ? f / k.vn[sy * (m + 1) + r] : 0.0;
    }
    for (int c = jv - 1; c >= 0; --c) {
        const double yc = __shfl_sync(0xffffffffu, c >= 32 ? rh[1] * iv[1] : rh[0] * iv[0], c & 31);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int r = lane + 32 * q;
            if (r < c) rh[q] = fma(-Hs[(int64_t)r * m + c], yc, rh[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int r = lane + 32 * q;
        if (r >= jv) continue;
        const double yr = rh[q] * iv[q] * sc[q];
        k.y[sy * m + r] = yr;
        if (k.y32) k.y32[sy * m + r] = float(yr);
    }
    if (k.sexp && lane == 0) {
        const double est = fmax(fabs(k.g[sy * (m + 1) + jv]), 1e-3 * k.rtol * k.bnorm[sy]);
        if (est > 0.0 && est < 1e300) k.sexp[k.ns + sy] = max(-1000, ilogb(est));
    }
}

// ... of every system on its own (batches)
constexpr int kSolveWarps = 4;      // systems per block
__global__ void __launch_bounds__(32 * kSolveWarps) k_cycle_solve(Krylov k)
{
    const int sy = blockIdx.x * kSolveWarps + (threadIdx.x >> 5);
    if (sy < k.ns) cycle_solve(k, sy);
}

// The second Gram-Schmidt pass of a system by one block: h2 = the products' sums,
// w -= sum_k h2_k / vn_k^2 V_k over the case's cells; the first warp gets |w|^2.  A block's
// latency: with the block on one sum after another and a thread per cell, steps on 50 triangles
// stretched 50 : 1 (a pass in two indices of three) took 15.7 ms, now 12.0 (launches 13.0).
struct Solo {
    const double *V;
    double *w;              // NULL: the pass has launches of its own
    int64_t T;
};

__device__ __forceinline__ double solo_pass(const Krylov &k, const Solo &o, int sy, int j, const double *part, int64_t R,
                                            int b0, int b1, int c0, int c1, double *h2, double *hk, double *sh)
{
    // the products' sums: a warp per basis vector
    const int lane = threadIdx.x & 31;
    for (int q = threadIdx.x >> 5; q <= j; q += kReduceThreads / 32) {
        const double *p = part + ((int64_t)q * 4 + (sy & 3)) * R;
        double s = 0.0;
        for (int b = b0 + lane; b < b1; b += 32) s += p[b];
        s = warp_sum(s);
        if (lane == 0) {
            const double n = k.vn[sy * (k.m + 1) + q];
            h2[q] = s;
            hk[q] = n > 0.0 ? s / (n * n) : 0.0;
        }
    }
    __syncthreads();
    // the update: a thread per cell and unknown
    const int64_t vo = (int64_t)(sy & 3) * 5 * o.T, vs = 20 * o.T;
    const int n = int(min((int64_t)c1, o.T) - c0);
    double nr = 0.0;
    for (int e = threadIdx.x; e < 5 * n; e += kReduceThreads) {
        const int l = e / n;
        const int64_t at = vo + l * o.T + c0 + (e - l * n);
        double u = o.w[at];
        for (int q = 0; q <= j; ++q) u = fma(-hk[q], o.V[q * vs + at], u);
        o.w[at] = u;
        nr = fma(u, u, nr);
    }
    return block_total(nr, sh);
}

// End of Arnoldi index j, one block per system: |V_{j+1}| of a running system
// from the summed partials and its Givens step (twice given: only of the systems
// flagged there, which ran the second Gram-Schmidt pass, the others are done; no
// such system: nothing to do); with solo.w the block also does that pass for its
// system, from the products' partial sums on (small meshes: one launch that
// returns as a rule instead of three); then the condition "any system
// still runs" and, for a single mesh, the solve of the cycle once none does.
__global__ void __cluster_dims__(4, 1, 1) __launch_bounds__(kReduceThreads)
    k_arnoldi_end(Krylov k, const double *part, int64_t R, const int32_t *__restrict__ seg, int rs, int j,
                  const double *hc, int hstride, double *h2, int h2stride, const int32_t *twice, double shift, Solo solo,
                  Cond cd)
{
    __shared__ double sh[kReduceThreads / 32];
    __shared__ double shg[4][kMaxRestart + 1];
    const int sy = blockIdx.x, c = sy >> 2;
    if (twice) {
        int a = 0;
        for (int q = threadIdx.x; q < k.ns; q += blockDim.x) a |= twice[q];
        if (__syncthreads_or(a) == 0) return;
    }
    if (k.ctl[kCtlRunning * k.ns + sy] != 0 && (!twice || twice[sy])) {
        const int b0 = rs * seg[c], b1 = rs * seg[c + 1];
        const double acc = solo.w ? solo_pass(k, solo, sy, j, part, R, b0, b1, kBlock * seg[c], kBlock * seg[c + 1],
                                              h2 + sy * h2stride, shg[0], sh)
                                  : block_sum(part, 0, sy & 3, R, b0, b1, sh);
        __syncthreads();
        if (threadIdx.x < 32) givens_step(k, sy, j, hc, hstride, h2, h2stride, shift, sqrt(acc), false, shg);
    }
    bool last;
    const bool any = any_flag(k.ctl + kCtlRunning * k.ns, k.ns, cd.ticket, &last);
    if (!last) return;
    if (gridDim.x == 4 && !any && threadIdx.x < 32) cycle_solve(k, sy);
    set_cond(cd, any);
}

// End of Arnoldi index j inside the update's launch, a block per case with a warp
// per system: the basis holds w = K Z_j - V_j, at least half of whose norm is
// orthogonal to it as a rule (gks_solve64.cuh), so the new vector's norm follows from
// |w|^2 (hs[j + 1]) and the projections, and the Givens step needs no sum over the
// updated vector.  ran: the running systems before this launch.
//  - FP64: the difference of the squares keeps its digits (within a factor of 4);
//    a system with less than half of |w| left gets the second Gram-Schmidt pass and
//    its Givens step from the launches that follow (twice[system] = 1);
//  - mixed: a system with less than 3 % left, where an FP32 basis loses the digits,
//    ends its cycle (twice NULL).  The norm is then good to FP32's digits over |w| / |V_{j+1}|;
//    with it the basis is still nearer to orthonormal than without the shift and with a norm
//    of its own: largest entry of V^T V - 1 over eight indices on 60 systems (32 to 1,800
//    triangles, aspects 1 to 200, no to two sweeps) 4e-8 to 3e-6 against 5e-7 to 0.2.

// |w|^2 of system sy and the part of it that the projections take, to every lane
__device__ __forceinline__ double projected(const double *hs, const double *hc, int hstride, int sy, int j, double *n2)
{
    double s = 0.0;
    for (int q = threadIdx.x & 31; q <= j; q += 32) s = fma(hc[sy * hstride + q], hs[sy * hstride + q], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    *n2 = hs[sy * hstride + j + 1];
    return s;
}

__device__ __forceinline__ bool needs_second(double s, double n2) { return !(n2 > 0.0 && s <= 0.75 * n2); }

typedef double GivensRows[4][kMaxRestart + 1];

__device__ __forceinline__ void control_end(const Krylov &k, int c, int ncase, int j, const double *hs, const double *hc,
                                            int hstride, const int32_t *ran, int32_t *twice, const Cond &cd,
                                            GivensRows *shg)
{
    __shared__ int is_last;
    const int warp = threadIdx.x >> 5, sy = 4 * c + (warp & 3);
    if (warp < 4) {
        bool again = false;
        if (ran[sy] != 0) {
            double n2;
            const double s = projected(hs, hc, hstride, sy, j, &n2), r2 = n2 - s;
            again = twice && needs_second(s, n2);
            if (!again)
                givens_step(k, sy, j, hs, hstride, nullptr, 0, 1.0, sqrt(fmax(r2, 1e-7 * n2)),
                            !twice && !(r2 > 1e-3 * n2), shg[warp]);
        }
        if (twice && (threadIdx.x & 31) == 0) twice[sy] = again;
    }
    bool any;
    __syncthreads();
    if (ncase == 1) {
        any = __syncthreads_or(threadIdx.x < 4 && k.ctl[kCtlRunning * k.ns + threadIdx.x] != 0) != 0;
        if (!any && warp < 4) cycle_solve(k, sy);
    } else {
        if (threadIdx.x == 0) {
            __threadfence();
            is_last = atomicInc(cd.ticket, ncase - 1) == (unsigned)(ncase - 1);
            __threadfence();
        }
        __syncthreads();
        if (!is_last) return;
        int a = 0;
        for (int q = threadIdx.x; q < k.ns; q += blockDim.x) a |= __ldcg(k.ctl + kCtlRunning * k.ns + q);
        any = __syncthreads_or(a) != 0;
    }
    if (threadIdx.x == 0) put_cond(cd, any);
}

// Start (first) or restart of a system, one block each: the norm of the stored
// first basis vector V_0 = 2^-e r from the partials' column 0 (e: the next
// exponent sexp[ns + s], which becomes the current one; 0 when sexp is NULL) and,
// first, |b|^2 from column 1 (FP64 basis) or b2 (see k_sigma).  Systems of
// finished cases stay inactive; a system that stopped keeps its solution, its
// residual and their norm.  Then g = beta e_1 for active systems and the
// condition "any system active".
__global__ void __cluster_dims__(4, 1, 1) __launch_bounds__(kReduceThreads)
    k_cycle_begin(Krylov k, const double *part, int64_t R, const int32_t *__restrict__ seg, int rs, const double *b2,
                  int bstride, const int32_t *__restrict__ done, int first, Cond cd)
{
    __shared__ double sh[kReduceThreads / 32], shb[kReduceThreads / 32], shbe;
    const int sy = blockIdx.x, c = sy >> 2, v = sy & 3;
    const int b0 = rs * seg[c], b1 = rs * seg[c + 1];
    const bool on = first || k.ctl[kCtlActive * k.ns + sy] != 0;
    double r2 = 0.0, bb = 0.0;
    if (on) {
        r2 = block_sum(part, 0, v, R, b0, b1, sh);
        if (first && !k.sexp) bb = block_sum(part, 1, v, R, b0, b1, shb);
    }
    if (threadIdx.x == 0) {
        int act = 0;
        double be = 0.0;
        if (on) {
            const double vn0 = sqrt(r2);
            be = vn0;
            if (k.sexp) {
                be = vn0 * pow2_exact(k.sexp[k.ns + sy]);
                k.sexp[sy] = k.sexp[k.ns + sy];
            }
            const double bn = first ? sqrt(k.sexp ? b2[sy * bstride] : bb) : k.bnorm[sy];
            const int it = first ? 0 : k.ctl[kCtlIters * k.ns + sy];
            if (first) {
                k.bnorm[sy] = bn;
                k.ctl[kCtlIters * k.ns + sy] = 0;
            }
            k.beta[sy] = be;
            k.vn[sy * (k.m + 1)] = vn0;                    // V_0 = 2^-e r, v_0 = r / beta
            act = (!first || !done[c]) && bn > 0.0 && be > k.rtol * bn && it < k.maxit;
        }
        k.ctl[kCtlActive * k.ns + sy] = act;
        k.ctl[kCtlRunning * k.ns + sy] = act;
        k.ctl[kCtlJv * k.ns + sy] = 0;
        shbe = act ? be : 0.0;
    }
    __syncthreads();
    if (threadIdx.x <= k.m) k.g[sy * (k.m + 1) + threadIdx.x] = threadIdx.x == 0 ? shbe : 0.0;
    bool last;
    const bool any = any_flag(k.ctl + kCtlActive * k.ns, k.ns, cd.ticket, &last);
    if (last) set_cond(cd, any);
}

// First Gram-Schmidt update w -= sum_k h_k V_k of the FP64 solve (32 C cells per
// block) and the end of Arnoldi index j (the first ncase blocks); a system that
// needs the second pass also gets the products <V_k, w>.  Dynamic shared memory:
// 4 (j + 1) (kAccStride + 1) doubles, at least four GivensRows.
template <int C>
__global__ void __launch_bounds__(kW64) k64_update(int64_t T, const int32_t *__restrict__ blk_case, Krylov kr, int ncase,
                                                   const double *__restrict__ V, double *__restrict__ wn, int j,
                                                   const double *__restrict__ hs, const double *__restrict__ hc,
                                                   int hstride, const int32_t *__restrict__ ran, int32_t *twice,
                                                   Cond cd, double *__restrict__ part)
{
    extern __shared__ double sh64[];
    if ((int)blockIdx.x < ncase) {
        control_end(kr, blockIdx.x, ncase, j, hs, hc, hstride, ran, twice, cd, reinterpret_cast<GivensRows *>(sh64));
        return;
    }
    const int64_t b = blockIdx.x - ncase, R = gridDim.x - ncase, c0 = b * (32 * C);
    const Warp64 w = warp64(blk_case, ran, c0);
    if (!w.run) return;
    const int K = j + 1;
    double *acc = sh64 + w.v * K * (kAccStride + 1), *h = acc + K * kAccStride, n2;
    const double s0 = projected(hs, hc, hstride, w.sys, j, &n2);
    const bool again = needs_second(s0, n2);
    for (int k = w.lane; k < K; k += 32) h[k] = hc[w.sys * hstride + k];
    for (int k = 0; k < K; ++k) acc[k * kAccStride + w.lane] = 0.0;
    __syncwarp();
    const int64_t vo = (int64_t)w.v * 5 * T, vs = 20 * T;
    for (int c = 0; c < C; ++c) {
        const int64_t i = c0 + 32 * c + w.lane;
        if (i >= T) break;
        double u[5];
#pragma unroll
        for (int l = 0; l < 5; ++l) u[l] = wn[vo + l * T + i];
#pragma unroll 4
        for (int k = 0; k < K; ++k) {
            const double *vk = V + k * vs + vo + i;
            const double hk = -h[k];
#pragma unroll
            for (int l = 0; l < 5; ++l) u[l] = fma(hk, vk[l * T], u[l]);
        }
#pragma unroll
        for (int l = 0; l < 5; ++l) wn[vo + l * T + i] = u[l];
        if (!again) continue;
#pragma unroll 4
        for (int k = 0; k < K; ++k) {
            const double *vk = V + k * vs + vo + i;
            double s = acc[k * kAccStride + w.lane];
#pragma unroll
            for (int l = 0; l < 5; ++l) s = fma(vk[l * T], u[l], s);
            acc[k * kAccStride + w.lane] = s;
        }
    }
    if (!again) return;
    __syncwarp();
    warp_rows(acc, K, w.lane, part + w.v * R + b, 4 * R);
}

// w -= sum_{k<=j} c_k V_k for the running systems, w = 0 for the others, and the end
// of Arnoldi index j: the first ncase blocks are control_end's, the others take
// kBlock cells each.  J as k32_apply_dots (the loads of all vectors first).
template <int J>
__global__ void __launch_bounds__(kBlock) k32_update(int64_t T, const int32_t *__restrict__ blk_case, Krylov kr,
                                                     int ncase, const float *__restrict__ V, float *__restrict__ wn,
                                                     int j, const double *__restrict__ hs_raw,
                                                     const double *__restrict__ hc, int hstride,
                                                     const int32_t *__restrict__ ran, Cond cd)
{
    if (J > 0) j = J - 1;
    __shared__ GivensRows shg[4];
    __shared__ float hs[kMaxRestart][4];
    if ((int)blockIdx.x < ncase) {
        control_end(kr, blockIdx.x, ncase, j, hs_raw, hc, hstride, ran, nullptr, cd, shg);
        return;
    }
    const int64_t b = blockIdx.x - ncase, i = b * kBlock + threadIdx.x;
    const int c = blk_case[b];
    const int4 r = reinterpret_cast<const int4 *>(ran)[c];
    if ((r.x | r.y | r.z | r.w) == 0) return;
    for (int q = threadIdx.x; q < 4 * (j + 1); q += blockDim.x)
        hs[q >> 2][q & 3] = -float(hc[(4 * c + (q & 3)) * hstride + (q >> 2)]);
    const bool on[4] = {r.x != 0, r.y != 0, r.z != 0, r.w != 0};
    __syncthreads();
    if (i >= T) return;
    const int64_t vs = 20 * T;
    float w[5][4];
#pragma unroll
    for (int l = 0; l < 5; ++l) vload(wn, l, T, i, w[l]);
    if constexpr (J > 0) {
        float t[J][5][4];
#pragma unroll
        for (int k = 0; k < J; ++k)
#pragma unroll
            for (int l = 0; l < 5; ++l) vload(V + k * vs, l, T, i, t[k][l]);
#pragma unroll
        for (int k = 0; k < J; ++k)
#pragma unroll
            for (int l = 0; l < 5; ++l)
#pragma unroll
                for (int v = 0; v < 4; ++v) w[l][v] = fmaf(hs[k][v], t[k][l][v], w[l][v]);
    } else {
#pragma unroll 2
        for (int k = 0; k <= j; ++k)
#pragma unroll
            for (int l = 0; l < 5; ++l) {
                float t[4];
                vload(V + k * vs, l, T, i, t);
#pragma unroll
                for (int v = 0; v < 4; ++v) w[l][v] = fmaf(hs[k][v], t[v], w[l][v]);
            }
    }
#pragma unroll
    for (int l = 0; l < 5; ++l) {
#pragma unroll
        for (int v = 0; v < 4; ++v) w[l][v] = on[v] ? w[l][v] : 0.0f;
        vstore(wn, l, T, i, w[l]);
    }
}

// Scale of the first residual of a solve, one block per system: |b|^2 from the
// partials' column 1 into b2, and the next exponent sexp[ns + s] = e with 2^-e B
// in [1, 2), B = max(|b|, |b_prev|) (bnorm = |b| of the previous solve, 0 at
// first): the warm start solved the previous system, so its residual is of the
// order of B at most; e = 0 when B = 0.
__global__ void __launch_bounds__(kReduceThreads) k_sigma(const double *part, int64_t R,
                                                          const int32_t *__restrict__ seg, int rs, double *b2,
                                                          int bstride, const double *__restrict__ bnorm,
                                                          int32_t *sexp, int ns)
{
    __shared__ double sh[kReduceThreads / 32];
    const int sy = blockIdx.x, c = sy >> 2;
    const double s = block_sum(part, 1, sy & 3, R, rs * seg[c], rs * seg[c + 1], sh);
    if (threadIdx.x != 0) return;
    b2[sy * bstride] = s;
    const double bn = fmax(sqrt(s), bnorm[sy]);
    sexp[ns + sy] = bn > 0.0 && bn < 1e300 ? max(-1000, ilogb(bn)) : 0;
}

}  // namespace
}  // namespace gks
