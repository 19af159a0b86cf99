// CLS reconstruction on the device (Sec. III): right-hand side, operator
// application, block ILU(0) preconditioner and restarted GMRES.
//
// Four independent systems (rho, rho u, rho v, E) share one operator.  This file
// holds the generic kernels, a cell and all four variables per thread (extended
// stencils, exact triangular solves, FP64 basis of the mixed mode), the mixed
// mode's right-hand side, residual and correction, and the launches; the per-cell
// equations' own kernels are in gks_solve64.cuh (FP64, a thread per cell and
// variable) and gks_solve32.cuh (mixed), sums and control in gks_control.cuh.
// FP64 vectors are [var][dof][cell] in RCM order, FP32 vectors [dof][cell][var]
// (vload, vstore).  GMRES (Saad & Schultz 1986) is right-preconditioned with
// classical Gram-Schmidt: one pass on the shifted basis in FP64, a second where it is
// needed; two on the extended stencils; one in the mixed mode.  Per-variable state
// stays on the device (running/converged masks); reductions go through
// per-block partial sums and a fixed-order second pass, so results are
// deterministic.  The Krylov basis is stored unnormalised, V_k = vn_k v_k,
// with the norms vn_k on the device: the normalisation is folded into the
// Gram-Schmidt coefficients, the Hessenberg entries and the final combination,
// which saves one read and one write of the new vector per iteration.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "gks_internal.h"
#include "gks_control.cuh"
#include "gks_wait.cuh"

namespace gks {
namespace {

constexpr int NV = 4, ND = 5, NX = 20;
constexpr int kDotThreads = 256;       // threads per block of the dot-product kernel
constexpr int kDotMaxTiles = 65535;    // grid.y limit of the dot-product kernel

// acc += sa [e1 + dx e3 + dy e4 | e2 + dx e4 + dy e5] (g1, g2): the off-diagonal
// block O_ij = alpha [...] applied to the gradient entries (g1, g2) of
// neighbour j, scaled by sa = +-alpha, with sax = sa dx, say = sa dy; all FMAs
template <typename R>
__device__ __forceinline__ void oacc(R sa, R sax, R say, R g1, R g2, R *acc)
{
    acc[0] = fma(sa, g1, acc[0]);
    acc[1] = fma(sa, g2, acc[1]);
    acc[2] = fma(sax, g1, acc[2]);
    acc[3] = fma(say, g1, fma(sax, g2, acc[3]));
    acc[4] = fma(say, g2, acc[4]);
}

// acc[0..1] += sr [x0 + dx x2 + dy x3 | x1 + dx x3 + dy x4] (srx = sr dx, sry =
// sr dy): the transpose form that the global normal equations (Eq. (33)) add
// to an off-diagonal block from the neighbour's own equations, applied to all
// five unknowns x of the neighbour
template <typename R>
__device__ __forceinline__ void racc(R sr, R srx, R sry, const R *x, R *acc)
{
    acc[0] = fma(sr, x[0], fma(srx, x[2], fma(sry, x[3], acc[0])));
    acc[1] = fma(sr, x[1], fma(srx, x[3], fma(sry, x[4], acc[1])));
}

// 2^e exactly (|e| <= 1022)
__device__ __forceinline__ double pow2(int e)
{
    e = e < -1022 ? -1022 : (e > 1023 ? 1023 : e);
    return __longlong_as_double((long long)(e + 1023) << 52);
}

// 2^k in FP32 for k <= 0; 0 below FP32's normal range
__device__ __forceinline__ float pow2f(int k)
{
    return k >= -126 ? __uint_as_float((unsigned)(127 + k) << 23) : 0.0f;
}

// Block reduction of NV values; thread 0 of the block gets the totals.
__device__ __forceinline__ void block_sum4(double *v, double *sh)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < NV; ++q)
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < NV; ++q) sh[warp * NV + q] = v[q];
    __syncthreads();
    if (threadIdx.x == 0) {
        const int nw = blockDim.x >> 5;
        for (int q = 0; q < NV; ++q) {
            double s = 0.0;
            for (int k = 0; k < nw; ++k) s += sh[k * NV + q];
            v[q] = s;
        }
    }
    __syncthreads();
}

// r_i = sum_j a0_ij (ubar_j - ubar_i), Eq. (25) with b_ij = (ubar_j - ubar_i, 0, 0)
// with partial sums of |b|^2 per block and variable in column 1 of part
__global__ void k_rhs(DeviceMesh d, const double *__restrict__ w, double *__restrict__ b, double *__restrict__ part)
{
    __shared__ double sh[32 * NV];
    const int64_t T = d.T;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    double nb[NV] = {0, 0, 0, 0};
    if (i < T) {
        double acc[NX];
#pragma unroll
        for (int q = 0; q < NX; ++q) acc[q] = 0.0;
        double wi[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) wi[v] = w[v * T + i];
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const int j = d.nb[s * T + i];
            if (j < 0) continue;
            double a[ND];
#pragma unroll
            for (int l = 0; l < ND; ++l) a[l] = d.a0[(s * ND + l) * T + i];
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const double du = w[v * T + j] - wi[v];
#pragma unroll
                for (int l = 0; l < ND; ++l) acc[v * ND + l] += a[l] * du;
            }
        }
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int l = 0; l < ND; ++l) {
                const double bv = acc[v * ND + l];
                b[(v * ND + l) * T + i] = bv;
                nb[v] += bv * bv;
            }
    }
    block_sum4(nb, sh);
    if (threadIdx.x == 0)
        for (int v = 0; v < NV; ++v) part[(NV + v) * (int64_t)gridDim.x + blockIdx.x] = nb[v];
}

// acc = (K x)_i, the operator row of cell i applied to x (TM arithmetic).
// Every load (neighbour indices, blocks, the neighbours' gradient entries, own
// data) is issued before the arithmetic; a missing neighbour reads the cell's
// own entries with a zero block.
// G: extended stencil (global normal equations and / or second-derivative
// equations): the transpose form with the reverse-slot coefficients arg, exrg,
// eyrg (racc) and the diagonal coupling bdg of the unknowns 3..5; unused
// otherwise.
template <typename TX, typename TM, bool G = false>
__device__ __forceinline__ void cell_apply(const DeviceMesh &d, const TM *__restrict__ Dg, const TM *__restrict__ alg,
                                           const TM *__restrict__ exg, const TM *__restrict__ eyg,
                                           const TX *__restrict__ x, int64_t i, TM *acc,
                                           const TM *__restrict__ arg = nullptr, const TM *__restrict__ exrg = nullptr,
                                           const TM *__restrict__ eyrg = nullptr, const TM *__restrict__ bdgg = nullptr)
{
    const int64_t T = d.T;
    int64_t jn[3];
    TM sa[3], sax[3], say[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const int j = d.nb[s * T + i];
        jn[s] = j >= 0 ? j : i;
        sa[s] = j >= 0 ? -alg[s * T + i] : TM(0);
        sax[s] = sa[s] * exg[s * T + i];
        say[s] = sa[s] * eyg[s * T + i];
    }
    TM g[3][2][NV];
#pragma unroll
    for (int s = 0; s < 3; ++s)
#pragma unroll
        for (int a = 0; a < 2; ++a) vload(x, a, T, jn[s], g[s][a]);
    TM Dm[15];
#pragma unroll
    for (int q = 0; q < 15; ++q) Dm[q] = Dg[q * T + i];
    TM xo[ND][NV];
#pragma unroll
    for (int l = 0; l < ND; ++l) vload(x, l, T, i, xo[l]);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const TM xv[ND] = {xo[0][v], xo[1][v], xo[2][v], xo[3][v], xo[4][v]};
        // symmetric 5x5 times vector
        acc[v * ND + 0] = Dm[0] * xv[0] + Dm[1] * xv[1] + Dm[2] * xv[2] + Dm[3] * xv[3] + Dm[4] * xv[4];
        acc[v * ND + 1] = Dm[1] * xv[0] + Dm[5] * xv[1] + Dm[6] * xv[2] + Dm[7] * xv[3] + Dm[8] * xv[4];
        acc[v * ND + 2] = Dm[2] * xv[0] + Dm[6] * xv[1] + Dm[9] * xv[2] + Dm[10] * xv[3] + Dm[11] * xv[4];
        acc[v * ND + 3] = Dm[3] * xv[0] + Dm[7] * xv[1] + Dm[10] * xv[2] + Dm[12] * xv[3] + Dm[13] * xv[4];
        acc[v * ND + 4] = Dm[4] * xv[0] + Dm[8] * xv[1] + Dm[11] * xv[2] + Dm[13] * xv[3] + Dm[14] * xv[4];
    }
#pragma unroll
    for (int s = 0; s < 3; ++s)
#pragma unroll
        for (int v = 0; v < NV; ++v) oacc(sa[s], sax[s], say[s], g[s][0][v], g[s][1][v], acc + v * ND);
    if (G) {
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const bool has = jn[s] != i;
            const TM sr = has ? -arg[s * T + i] : TM(0);
            const TM srx = sr * exrg[s * T + i], sry = sr * eyrg[s * T + i];
            const TM sb = has ? -bdgg[s * T + i] : TM(0);
            TM xn[ND][NV];
#pragma unroll
            for (int l = 0; l < ND; ++l) vload(x, l, T, jn[s], xn[l]);
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const TM xj[ND] = {xn[0][v], xn[1][v], xn[2][v], xn[3][v], xn[4][v]};
                racc(sr, srx, sry, xj, acc + v * ND);
#pragma unroll
                for (int l = 2; l < ND; ++l) acc[v * ND + l] = fma(sb, xj[l], acc[v * ND + l]);
            }
        }
    }
}

// y = K x (mode 0), or y = 2^-e (b - K x) with partial sums of |y|^2 of the
// stored y (mode 1), e = sexp[system] (0 when sexp is NULL): an FP32 Krylov
// basis keeps its first vector near unit size whatever the size of b.
// K_ii = D_i (symmetric, 15 stored values), K_ij = -O_ij.  TX: type of x, TM:
// type of the operator data and of the arithmetic (mode 1 is FP64 only), TY:
// type of y.
template <typename TX, typename TM, typename TY, bool G = false>
__global__ void k_spmv(DeviceMesh d, const TM *__restrict__ Dg, const TM *__restrict__ alg,
                       const TM *__restrict__ exg, const TM *__restrict__ eyg, const TX *__restrict__ x,
                       TY *__restrict__ y, int mode, const double *__restrict__ b, double *__restrict__ part,
                       const int32_t *__restrict__ sexp = nullptr, const TM *__restrict__ arg = nullptr,
                       const TM *__restrict__ exrg = nullptr, const TM *__restrict__ eyrg = nullptr,
                       const TM *__restrict__ bdgg = nullptr)
{
    __shared__ double sh[32 * NV];
    const int64_t T = d.T;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    double nr[NV] = {0, 0, 0, 0};
    if (i < T) {
        TM acc[NX];
        cell_apply<TX, TM, G>(d, Dg, alg, exg, eyg, x, i, acc, arg, exrg, eyrg, bdgg);
        if (mode == 0) {
#pragma unroll
            for (int l = 0; l < ND; ++l) {
                const TY o[NV] = {TY(acc[l]), TY(acc[ND + l]), TY(acc[2 * ND + l]), TY(acc[3 * ND + l])};
                vstore(y, l, T, i, o);
            }
        } else {
            const int c = d.blk_case[blockIdx.x];
            double sig[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) sig[v] = sexp ? pow2(-sexp[4 * c + v]) : 1.0;
#pragma unroll
            for (int l = 0; l < ND; ++l) {
                TY o[NV];
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    const double rv = b[(v * ND + l) * T + i] - double(acc[v * ND + l]);
                    o[v] = TY(rv * sig[v]);
                    nr[v] += double(o[v]) * double(o[v]);
                }
                vstore(y, l, T, i, o);
            }
        }
    }
    if (mode >= 1) {
        block_sum4(nr, sh);
        if (threadIdx.x == 0)
            for (int v = 0; v < NV; ++v) part[v * (int64_t)gridDim.x + blockIdx.x] = nr[v];
    }
}

// ---- double-FP32 arithmetic for the refinement residual of the mixed mode.
// A value is the unevaluated sum h + l of two FP32 numbers (about 48
// significant bits; Dekker 1971).  The product of two high parts is exact as
// p + e with e = fma(a, b, -p); sums use Knuth's TwoSum (TAOCP vol. 2, 4.2.2),
// whose rounding error is exact; the small cross terms a_h b_l + a_l b_h are
// plain FP32.  The _rn intrinsics keep the compiler from contracting or
// reordering these steps.  GB300 runs FP32 at 64 times its FP64 rate, so the
// 13 FP32 operations of a product-sum cost far less than one DFMA.

// 2^-e v = h + l on the integer pipe (no FP64 instruction; e is applied to the
// exponent field): h holds the upper 24 significant bits (truncated), l the
// next 29 rounded to 24, so |2^-e v - h - l| <= 2^-47 |2^-e v|.  The residual
// scales each system by 2^-e ~ 1/|b|, against which smaller parts do not
// count: below 2^-74 only h is kept, below 2^-126 nothing (with operator
// entries <= 2^30 either drop is under 2^-68 |2^-e b| per term).  Returns
// false for 2^-e v >= 2^128 or a value that is not finite; that cell then
// takes the FP64 operator.
__device__ __forceinline__ bool df_split(double v, int e, float &h, float &l)
{
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    const unsigned hw = (unsigned)(u >> 32), lw = (unsigned)u;
    const int E = (int)((hw >> 20) & 0x7FFu);           // biased FP64 exponent
    const int Es = E - e;                                // that of 2^-e v
    h = l = 0.0f;
    if (E == 2047 || (E != 0 && Es > 1150)) return false;
    if (E == 0 || Es < 897) return true;                 // zero, FP64 subnormal, or negligible
    const unsigned sgn = hw & 0x80000000u;
    h = __uint_as_float(sgn | ((unsigned)(Es - 896) << 23) | ((hw & 0xFFFFFu) << 3) | (lw >> 29));
    if (Es >= 949) {
        // the remaining 29 bits times 2^(Es - 1075), a normal FP32 power of two here
        const float r = __fmul_rn(__uint2float_rn(lw & 0x1FFFFFFFu), __uint_as_float((unsigned)(Es - 948) << 23));
        l = sgn ? -r : r;
    }
    return true;
}

// (sh, sl) += (ah, al) (bh, bl)
__device__ __forceinline__ void df_mac(float ah, float al, float bh, float bl, float &sh, float &sl)
{
    const float p = __fmul_rn(ah, bh);
    const float e = __fmaf_rn(ah, bh, -p);
    const float t = __fadd_rn(sh, p);
    const float z = __fsub_rn(t, sh);
    const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, z)), __fsub_rn(p, z));
    sh = t;
    sl = __fadd_rn(sl, __fadd_rn(err, __fadd_rn(e, __fmaf_rn(ah, bl, __fmul_rn(al, bh)))));
}

// (bh, bl) - (sh, sl), rounded to FP32
__device__ __forceinline__ float df_sub_round(float bh, float bl, float sh, float sl)
{
    const float t = __fsub_rn(bh, sh);
    const float z = __fsub_rn(t, bh);
    const float err = __fadd_rn(__fsub_rn(bh, __fsub_rn(t, z)), __fsub_rn(-sh, z));
    return __fadd_rn(t, __fadd_rn(err, __fsub_rn(bl, sl)));
}

// FP64 fallback of k_resid_df for variable v of cell i: out = 2^-e (b - K x)
template <bool G>
__device__ __noinline__ void resid64_cell(const DeviceMesh &d, const double *__restrict__ x,
                                          const double *__restrict__ b, int64_t i, int v, int e, float *out)
{
    double acc[NX];
    cell_apply<double, double, G>(d, d.D, d.alpha, d.ex, d.ey, x, i, acc, d.alr, d.exr, d.eyr, d.bdg);
    for (int l = 0; l < ND; ++l) out[l] = float((b[(v * ND + l) * d.T + i] - acc[v * ND + l]) * pow2(-e));
}

constexpr int kResidRows = NV;          // residual blocks (partial-sum rows) per cell block

// (h, l) += (x, y), sums of FP32 numbers to about 48 bits (TwoSum): on GB300 an
// FP64 addition costs a warp 33 ns, this seven FP32 operations
__device__ __forceinline__ void df_add(float x, float y, float &h, float &l)
{
    const float t = __fadd_rn(h, x);
    const float z = __fsub_rn(t, h);
    const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(t, z)), __fsub_rn(x, z));
    l = __fadd_rn(l, __fadd_rn(e, y));
    h = t;
}

// (h, l) of every lane summed over the warp (lane 0 gets the pair)
__device__ __forceinline__ void df_warp_sum(float &h, float &l)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        df_add(__shfl_down_sync(0xffffffffu, h, o), __shfl_down_sync(0xffffffffu, l, o), h, l);
}

// four floats of chunk q of cell i
__device__ __forceinline__ void load4(const float4 *__restrict__ p, int q, int64_t T, int64_t i, float *o)
{
    const float4 t = p[q * T + i];
    o[0] = t.x;
    o[1] = t.y;
    o[2] = t.z;
    o[3] = t.w;
}

// V_0 = 2^-e (b - K x) in FP32 and partial |V_0|^2 (as k_spmv mode 1 with an
// FP32 basis), in double-FP32 arithmetic: the operator as FP32 pairs D2
// ([12][T][4]: the 15 diagonal-block values and their low parts, sa, sa dx, sa dy
// of each neighbour and their low parts), 2^-e x and 2^-e b split on the fly, so
// the sums come out scaled.  One thread per cell and
// variable (the double-FP32 chains are latency-bound: many small threads hide
// it better than one thread per cell), the four variables of a cell in
// neighbouring lanes: one load serves the operator of eight cells for all four,
// and V_0 is written in whole lines.  (With the variables in different blocks
// of 256 cells the operator came from L2 four times; in different warps of a
// block it was no faster.)  A value outside the split range sends
// the thread to the FP64 operator.  Each thread's five squares are summed in
// FP32 (the scaled vector is near unit size), the threads' sums in FP64.
// act (NULL on a solve's first residual): a case without an active system keeps
// its V_0 and norms.  G: global normal equations, the
// transpose form from the reverse-slot pairs SR2 ([6][T][4]: 9 values and their
// low parts, then -beta per slot and its low parts) on all five unknowns of each
// neighbour.
template <bool G>
__global__ void __launch_bounds__(kBlock, 4) k_resid_df(const __grid_constant__ DeviceMesh d,
                                                        const float4 *__restrict__ D2,
                                                        const double *__restrict__ x, float *__restrict__ y,
                                                        const double *__restrict__ b, double *__restrict__ part,
                                                        const int32_t *__restrict__ sexp,
                                                        const int32_t *__restrict__ act,
                                                        const float4 *__restrict__ SR2 = nullptr)
{
    __shared__ double sh[kBlock / 32][NV];
    const int64_t T = d.T;
    const int cs = d.blk_case[blockIdx.x / kResidRows];
    if (act) {
        const int4 r = reinterpret_cast<const int4 *>(act)[cs];
        if ((r.x | r.y | r.z | r.w) == 0) return;
    }
    const int v = threadIdx.x & 3;
    const int64_t i = blockIdx.x * (int64_t)(kBlock / NV) + (threadIdx.x >> 2);
    double nr = 0.0;
    if (i < T) {
        const int e = sexp[4 * cs + v];
        int64_t jn[3];
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const int j = d.nb[s * T + i];
            jn[s] = j >= 0 ? j : i;
        }
        // the cell's own block first, then the neighbours: the two phases keep
        // fewer values live (no spills at the register cap), and the sums run
        // in the same order
        constexpr int NG = G ? ND : 2;                    // neighbour unknowns used
        double xv[ND], gv[3][NG], bv[ND];
        float dp[48], rp[G ? 24 : 1];
#pragma unroll
        for (int l = 0; l < ND; ++l) xv[l] = x[(v * ND + l) * T + i];
#pragma unroll
        for (int q = 0; q < 8; ++q) load4(D2, q, T, i, dp + 4 * q);
        bool ok = true;
        float xh[ND], xl[ND], gh[3][NG], gl[3][NG], ah[ND], al[ND], out[ND];
#pragma unroll
        for (int l = 0; l < ND; ++l) {
            ok &= df_split(xv[l], e, xh[l], xl[l]);
            ah[l] = al[l] = 0.0f;
        }
        // symmetric 5x5 block: entry (a, k) in the upper-triangle order
        constexpr int kIdx[5][5] = {{0, 1, 2, 3, 4}, {1, 5, 6, 7, 8}, {2, 6, 9, 10, 11}, {3, 7, 10, 12, 13},
                                    {4, 8, 11, 13, 14}};
#pragma unroll
        for (int a = 0; a < ND; ++a)
#pragma unroll
            for (int k = 0; k < ND; ++k) df_mac(dp[kIdx[a][k]], dp[15 + kIdx[a][k]], xh[k], xl[k], ah[a], al[a]);
#pragma unroll
        for (int s = 0; s < 3; ++s)
#pragma unroll
            for (int l = 0; l < NG; ++l) gv[s][l] = x[(v * ND + l) * T + jn[s]];
#pragma unroll
        for (int q = 8; q < 12; ++q) load4(D2, q, T, i, dp + 4 * q);
        const float *op = dp + 30, *bp = rp + (G ? 18 : 0);
        if (G)
#pragma unroll
            for (int q = 0; q < 6; ++q) load4(SR2, q, T, i, rp + 4 * q);
#pragma unroll
        for (int l = 0; l < ND; ++l) bv[l] = b[(v * ND + l) * T + i];
#pragma unroll
        for (int s = 0; s < 3; ++s)
#pragma unroll
            for (int l = 0; l < NG; ++l) ok &= df_split(gv[s][l], e, gh[s][l], gl[s][l]);
        // off-diagonal block of neighbour s (see oacc): sa, sax = sa dx, say = sa dy
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const int q = 3 * s;
            df_mac(op[q], op[9 + q], gh[s][0], gl[s][0], ah[0], al[0]);
            df_mac(op[q], op[9 + q], gh[s][1], gl[s][1], ah[1], al[1]);
            df_mac(op[q + 1], op[10 + q], gh[s][0], gl[s][0], ah[2], al[2]);
            df_mac(op[q + 1], op[10 + q], gh[s][1], gl[s][1], ah[3], al[3]);
            df_mac(op[q + 2], op[11 + q], gh[s][0], gl[s][0], ah[3], al[3]);
            df_mac(op[q + 2], op[11 + q], gh[s][1], gl[s][1], ah[4], al[4]);
            if (G) {
                // transpose form (see racc): rows 0 and 1 from all five unknowns
                df_mac(rp[q], rp[9 + q], gh[s][0], gl[s][0], ah[0], al[0]);
                df_mac(rp[q + 1], rp[10 + q], gh[s][NG > 2 ? 2 : 0], gl[s][NG > 2 ? 2 : 0], ah[0], al[0]);
                df_mac(rp[q + 2], rp[11 + q], gh[s][NG > 3 ? 3 : 0], gl[s][NG > 3 ? 3 : 0], ah[0], al[0]);
                df_mac(rp[q], rp[9 + q], gh[s][1], gl[s][1], ah[1], al[1]);
                df_mac(rp[q + 1], rp[10 + q], gh[s][NG > 3 ? 3 : 0], gl[s][NG > 3 ? 3 : 0], ah[1], al[1]);
                df_mac(rp[q + 2], rp[11 + q], gh[s][NG > 4 ? 4 : 0], gl[s][NG > 4 ? 4 : 0], ah[1], al[1]);
                // diagonal coupling of the unknowns 3..5 (second-derivative equations)
#pragma unroll
                for (int l = 2; l < ND; ++l)
                    df_mac(bp[s], bp[3 + s], gh[s][NG > l ? l : 0], gl[s][NG > l ? l : 0], ah[l], al[l]);
            }
        }
#pragma unroll
        for (int l = 0; l < ND; ++l) {
            float bh, bl;
            ok &= df_split(bv[l], e, bh, bl);
            out[l] = df_sub_round(bh, bl, ah[l], al[l]);
        }
        if (!ok) resid64_cell<G>(d, x, b, i, v, e, out);   // a value outside the split range
        float sq = 0.0f;
#pragma unroll
        for (int l = 0; l < ND; ++l) {
            y[(l * T + i) * NV + v] = out[l];
            sq = __fmaf_rn(out[l], out[l], sq);
        }
        nr = double(sq);
    }
    block_quads(nr, sh, part);
}

// 2^e f as an FP64 value, formed on the integer pipe (exact; an FP32 subnormal
// f, below 2^-126 of the scale, counts as zero)
__device__ __forceinline__ double f2d_pow2(float f, int e)
{
    const unsigned u = __float_as_uint(f);
    const int ef = (int)((u >> 23) & 0xFFu);
    if (ef == 0) return 0.0;
    const long long E = (long long)ef - 127 + 1023 + e;
    if (E <= 0 || E >= 2047) return double(f) * pow2(e);
    const unsigned long long bits = ((unsigned long long)(u >> 31) << 63) | ((unsigned long long)E << 52) |
                                    ((unsigned long long)(u & 0x7FFFFFu) << 29);
    return __longlong_as_double((long long)bits);
}

// The right-hand side of k_rhs in double-FP32 arithmetic (the FP32-basis
// solve), one thread per cell and variable.  GB300's FP64 pipe made the FP64
// kernel (92 FP64 operations per cell) its bottleneck; here a cell and variable
// take the power of two 2^e of their largest difference w_j - w_i (formed in
// FP64), split the scaled differences on the integer pipe, multiply them exactly
// by the weights as FP32 pairs a0p ([30][T]: the 15 high parts, then the low
// parts) and sum with compensation (df_mac); the normalised pair (high + low, 48
// bits) is widened on the integer pipe and added in FP64: 8 FP64 instructions
// per cell and variable, b to about 2^-48 relative at any magnitude.  A
// difference that does not split (not finite) sends the thread to FP64.
// Column 1 of part gets the |b|^2 of the block's 32 C cells: the scaled high
// parts squared in FP32, the lanes' sums kept to 48 bits with a power of two of
// their own, rescaled to the warp's largest at the end.  The four warps of a
// block take the four variables of the same cells (the weights come from L1).
template <int C>
__global__ void __launch_bounds__(kW32) k_rhs_df(DeviceMesh d, const float *__restrict__ a0p,
                                                 const double *__restrict__ w, double *__restrict__ b,
                                                 double *__restrict__ part)
{
    const int64_t T = d.T, c0 = blockIdx.x * (int64_t)(32 * C);
    const int lane = threadIdx.x & 31, v = threadIdx.x >> 5;
    const double *wv = w + v * T;
    float nh = 0.0f, nl = 0.0f;                   // 2^(-2 ne) |b|^2 of this lane
    int ne = -1022;
    for (int c = 0; c < C; ++c) {
        const int64_t i = c0 + 32 * c + lane;
        if (i >= T) break;
        int js[3];
#pragma unroll
        for (int s = 0; s < 3; ++s) js[s] = d.nb[s * T + i];
        // the cell's weights: their loads overlap the neighbour gathers
        float ah[3][ND], al[3][ND];
#pragma unroll
        for (int s = 0; s < 3; ++s)
#pragma unroll
            for (int l = 0; l < ND; ++l) {
                ah[s][l] = a0p[(s * ND + l) * T + i];
                al[s][l] = a0p[(15 + s * ND + l) * T + i];
            }
        const double wi = wv[i];
        double du[3];
        int em = 1;
        bool ok = true;
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            du[s] = wv[js[s] >= 0 ? js[s] : i] - wi;       // no neighbour: 0
            const int E = (int)(((unsigned)__double2hiint(du[s]) >> 20) & 0x7FFu);
            em = E > em ? E : em;
            ok &= E < 2047;
        }
        // with 2^e the largest difference, a difference fails to split only when
        // it is not finite: that sends the thread to FP64
        const int e = (em == 2047 ? 1023 : em) - 1023;
        float ss = 0.0f;                                   // 2^(-2 e) |b|^2 of this cell
        if (ok) {
            float sh_[ND], sl_[ND];
#pragma unroll
            for (int l = 0; l < ND; ++l) sh_[l] = sl_[l] = 0.0f;
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                float dh, dl;
                df_split(du[s], e, dh, dl);
#pragma unroll
                for (int l = 0; l < ND; ++l) df_mac(ah[s][l], al[s][l], dh, dl, sh_[l], sl_[l]);
            }
#pragma unroll
            for (int l = 0; l < ND; ++l) {
                // normalise (TwoSum): h + lo = sh + sl exactly
                const float h = __fadd_rn(sh_[l], sl_[l]);
                const float z = __fsub_rn(h, sh_[l]);
                const float lo = __fadd_rn(__fsub_rn(sh_[l], __fsub_rn(h, z)), __fsub_rn(sl_[l], z));
                b[(v * ND + l) * T + i] = f2d_pow2(h, e) + f2d_pow2(lo, e);
                ss = __fmaf_rn(h, h, ss);
            }
        } else {
            // FP64 as in k_rhs; the norm from the values scaled by 2^-e
            double acc[ND] = {0.0, 0.0, 0.0, 0.0, 0.0};
            for (int s = 0; s < 3; ++s) {
                if (js[s] < 0) continue;
                for (int l = 0; l < ND; ++l) acc[l] += d.a0[(s * ND + l) * T + i] * du[s];
            }
            for (int l = 0; l < ND; ++l) {
                b[(v * ND + l) * T + i] = acc[l];
                const float h = float(acc[l] * pow2(-e));
                ss = __fmaf_rn(h, h, ss);
            }
        }
        // to the larger of the two powers of two (terms below 2^-126 of it drop out)
        const int m = max(e, ne);
        const float f0 = pow2f(2 * (ne - m)), f1 = pow2f(2 * (e - m));
        nh *= f0;
        nl *= f0;
        df_add(ss * f1, 0.0f, nh, nl);
        ne = m;
    }
    int m = ne;
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    const float f = pow2f(2 * (ne - m));
    nh *= f;
    nl *= f;
    df_warp_sum(nh, nl);
    if (lane == 0)
        part[(NV + v) * (int64_t)gridDim.x + blockIdx.x] = (double(nh) + double(nl)) * pow2(m) * pow2(m);
}

// Forward block-ILU relation for the listed rows (or all rows when rows == nullptr):
//   z_i = P_i (r_i + sum_{k<i} O_ik zin_k)      (use_nb = 0: z_i = P_i r_i)
// use_nb = 2 (G): the first sweep with the block-diagonal pass folded in, zin_k =
// P_k r_k formed here from the lower neighbours' factors and right-hand sides
// (rounded to TZ as the separate pass stores them), which saves the write and
// the re-read of that pass; the neighbours' data mostly comes from L2.
// TR: type of r, TZ: type of z, TM: type of the factors and of the arithmetic.
// rcopy (G, may be NULL): also store TZ(r_i), so that later sweeps read r in the
// working precision (same values as converting r again).  Own data (r, P) is
// loaded before the neighbour gathers so that the two overlap.
// TP: storage type of the factors (TM, or FP16 for the mixed mode's FP32
// preconditioner), widened to TM on load.
// G: global normal equations, the transpose form with the reverse-slot
// coefficients arg, exrg, eyrg on all five unknowns of the neighbour.
// A bounded wait of the sync-free solves gives up after 1 s (a correct solve
// waits a few microseconds per level).
constexpr uint64_t kWaitLimitNs = 1000000000ull;

// The forward relation of row i (see k_ilu_fwd).  SF: the sync-free exact
// solve, which waits for each lower neighbour's ready tag before reading its
// value (through L2) and publishes its own row's tag after the store.
template <typename TR, typename TZ, typename TM, typename TP, bool G, bool SF>
__device__ __forceinline__ void ilu_fwd_row(const DeviceMesh &d, const TP *__restrict__ Pg,
                                            const TP *__restrict__ alg, const TP *__restrict__ exg,
                                            const TP *__restrict__ eyg, int64_t i, const TR *r, const TZ *zin,
                                            TZ *zout, int use_nb, TZ *__restrict__ rcopy, const TP *__restrict__ arg,
                                            const TP *__restrict__ exrg, const TP *__restrict__ eyrg,
                                            const TP *__restrict__ bdgg, int32_t *sf_flag, int32_t sf_tag,
                                            int32_t *sf_err)
{
    const int64_t T = d.T;
    TM y[NX];
#pragma unroll
    for (int l = 0; l < ND; ++l) {
        TM t[NV];
        vload(r, l, T, i, t);
        if (G && rcopy) vstore(rcopy, l, T, i, t);
#pragma unroll
        for (int v = 0; v < NV; ++v) y[v * ND + l] = t[v];
    }
    TM Pm[25];
#pragma unroll
    for (int k = 0; k < 25; ++k) Pm[k] = TM(Pg[k * T + i]);
    if (SF) {
        // every lower neighbour's tag first (one round trip for all of them)
        const int32_t *wf[3];
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const int j = d.nb[s * T + i];
            wf[s] = (j >= 0 && j < i) ? sf_flag + j : nullptr;
        }
        bounded_wait_all(wf[0], wf[1], wf[2], sf_tag, sf_err, kWaitLimitNs);
    }
    if (use_nb) {
        // unknowns of a neighbour that its off-diagonal block reaches
        constexpr int NA = G ? ND : 2;
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            // every slot's loads are issued (a slot that is not a lower
            // neighbour reads the cell's own data, which is discarded), only the
            // accumulation is conditional: the gathers of the slots overlap
            const int jn = d.nb[s * T + i];
            const bool lower = jn >= 0 && jn < i;
            const int64_t j = lower ? jn : i;
            const TM sa = TM(alg[s * T + i]), sax = sa * TM(exg[s * T + i]), say = sa * TM(eyg[s * T + i]);
            TM zn[NV][NA];
            if (G && use_nb == 2) {
                TM rj[ND][NV];
#pragma unroll
                for (int l = 0; l < ND; ++l) vload(r, l, T, j, rj[l]);
#pragma unroll
                for (int a = 0; a < NA; ++a) {
                    TM pa[ND];
#pragma unroll
                    for (int c = 0; c < ND; ++c) pa[c] = TM(Pg[(a * ND + c) * T + j]);
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        TM t = TM(0);
#pragma unroll
                        for (int c = 0; c < ND; ++c) t = fma(pa[c], rj[c][v], t);
                        zn[v][a] = TM(TZ(t));
                    }
                }
            } else {
#pragma unroll
                for (int a = 0; a < NA; ++a) {
                    TM t[NV];
                    if constexpr (SF) vload_cg(zin, a, T, j, t);
                    else vload(zin, a, T, j, t);
#pragma unroll
                    for (int v = 0; v < NV; ++v) zn[v][a] = t[v];
                }
            }
            if (!lower) continue;
#pragma unroll
            for (int v = 0; v < NV; ++v) oacc(sa, sax, say, zn[v][0], zn[v][1], y + v * ND);
            if constexpr (G) {
                const TM sr = TM(arg[s * T + i]), srx = sr * TM(exrg[s * T + i]), sry = sr * TM(eyrg[s * T + i]);
                const TM sb = TM(bdgg[s * T + i]);
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    racc(sr, srx, sry, zn[v], y + v * ND);
#pragma unroll
                    for (int l = 2; l < ND; ++l) y[v * ND + l] = fma(sb, zn[v][l], y[v * ND + l]);
                }
            }
        }
    }
#pragma unroll
    for (int a = 0; a < ND; ++a) {
        TM o[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            o[v] = TM(0);
#pragma unroll
            for (int c = 0; c < ND; ++c) o[v] = fma(Pm[a * ND + c], y[v * ND + c], o[v]);
        }
        vstore(zout, a, T, i, o);
    }
    if (SF) publish(sf_flag + i, sf_tag);
}

template <typename TR, typename TZ, typename TM, typename TP = TM, bool G = false>
__global__ void k_ilu_fwd(DeviceMesh d, const TP *__restrict__ Pg, const TP *__restrict__ alg,
                          const TP *__restrict__ exg, const TP *__restrict__ eyg, const int32_t *__restrict__ rows,
                          int64_t nrows, const TR *r, const TZ *zin, TZ *zout, int use_nb, TZ *__restrict__ rcopy,
                          const TP *__restrict__ arg = nullptr, const TP *__restrict__ exrg = nullptr,
                          const TP *__restrict__ eyrg = nullptr, const TP *__restrict__ bdgg = nullptr)
{
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= nrows) return;
    const int64_t i = rows ? rows[q] : q;
    ilu_fwd_row<TR, TZ, TM, TP, G, false>(d, Pg, alg, exg, eyg, i, r, zin, zout, use_nb, rcopy, arg, exrg, eyrg,
                                          bdgg, nullptr, 0, nullptr);
}

// Backward block-ILU relation: x_i = z_i + P_i sum_{j>i} O_ij xin_j (own data
// loaded before the neighbour gathers; with no upper neighbour the sum is 0
// and x_i = z_i exactly).
template <typename TZ, typename TM, typename TP, bool G, bool SF>
__device__ __forceinline__ void ilu_bwd_row(const DeviceMesh &d, const TP *__restrict__ Pg,
                                            const TP *__restrict__ alg, const TP *__restrict__ exg,
                                            const TP *__restrict__ eyg, int64_t i, const TZ *z, const TZ *xin,
                                            TZ *xout, const TP *__restrict__ arg, const TP *__restrict__ exrg,
                                            const TP *__restrict__ eyrg, const TP *__restrict__ bdgg,
                                            int32_t *sf_flag, int32_t sf_tag, int32_t *sf_err)
{
    const int64_t T = d.T;
    TM zi[ND][NV], y[NX];
#pragma unroll
    for (int l = 0; l < ND; ++l) vload(z, l, T, i, zi[l]);
#pragma unroll
    for (int k = 0; k < NX; ++k) y[k] = TM(0);
    TM Pm[25];
#pragma unroll
    for (int k = 0; k < 25; ++k) Pm[k] = TM(Pg[k * T + i]);
    if (SF) {
        // every upper neighbour's tag first (one round trip for all of them)
        const int32_t *wf[3];
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const int j = d.nb[s * T + i];
            wf[s] = j > i ? sf_flag + j : nullptr;
        }
        bounded_wait_all(wf[0], wf[1], wf[2], sf_tag, sf_err, kWaitLimitNs);
    }
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const int j = d.nb[s * T + i];
        if (j <= i) continue;
        const TM sa = TM(alg[s * T + i]), sax = sa * TM(exg[s * T + i]), say = sa * TM(eyg[s * T + i]);
        constexpr int NA = G ? ND : 2;       // rows of a neighbour that its block reaches
        TM xn[NA][NV];
#pragma unroll
        for (int a = 0; a < NA; ++a) {
            if constexpr (SF) vload_cg(xin, a, T, j, xn[a]);
            else vload(xin, a, T, j, xn[a]);
        }
#pragma unroll
        for (int v = 0; v < NV; ++v) oacc(sa, sax, say, xn[0][v], xn[1][v], y + v * ND);
        if constexpr (G) {
            const TM sr = TM(arg[s * T + i]), srx = sr * TM(exrg[s * T + i]), sry = sr * TM(eyrg[s * T + i]);
            const TM sb = TM(bdgg[s * T + i]);
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const TM xj[ND] = {xn[0][v], xn[1][v], xn[2][v], xn[3][v], xn[4][v]};
                racc(sr, srx, sry, xj, y + v * ND);
#pragma unroll
                for (int l = 2; l < ND; ++l) y[v * ND + l] = fma(sb, xj[l], y[v * ND + l]);
            }
        }
    }
#pragma unroll
    for (int a = 0; a < ND; ++a) {
        TM o[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            o[v] = zi[a][v];
#pragma unroll
            for (int c = 0; c < ND; ++c) o[v] = fma(Pm[a * ND + c], y[v * ND + c], o[v]);
        }
        vstore(xout, a, T, i, o);
    }
    if (SF) publish(sf_flag + i, sf_tag);
}

template <typename TZ, typename TM, typename TP = TM, bool G = false>
__global__ void __launch_bounds__(kBlock, sizeof(TM) == 4 ? 3 : 1)
    k_ilu_bwd(DeviceMesh d, const TP *__restrict__ Pg, const TP *__restrict__ alg, const TP *__restrict__ exg,
              const TP *__restrict__ eyg, const int32_t *__restrict__ rows, int64_t nrows, const TZ *z, const TZ *xin,
              TZ *xout, const TP *__restrict__ arg = nullptr, const TP *__restrict__ exrg = nullptr,
              const TP *__restrict__ eyrg = nullptr, const TP *__restrict__ bdgg = nullptr)
{
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= nrows) return;
    const int64_t i = rows ? rows[q] : q;
    ilu_bwd_row<TZ, TM, TP, G, false>(d, Pg, alg, exg, eyg, i, z, xin, xout, arg, exrg, eyrg, bdgg, nullptr, 0,
                                      nullptr);
}

// ---- sync-free exact triangular solves (GKS_PC_ILU_EXACT).  One launch per
// relation instead of one per level: persistent blocks take tickets for
// kBlock-row ranges in RCM order (forward: increasing rows, backward:
// decreasing), so a block only ever waits on rows of tickets taken before its
// own, by blocks that are already running; within a range a row waits on
// lower (upper) rows of the same range, which earlier threads finish (threads
// of a warp make independent progress).  Every row waits for its lower
// (upper) neighbours' tags (bounded_wait, at most kWaitLimitNs each), reads
// their values through L2 and publishes its own tag.  The tags of the two
// relations of application e are 2e + 1 and 2e + 2, so no flag is reset
// between applications.  ctl: [0] epoch e, [1] forward and [2] backward
// tickets, [3] sticky wait error.  The arithmetic of a row is that of the
// level-scheduled launches, so the results are the same bit for bit.

constexpr int kSfBlocksPerSm = 2;       // persistent blocks per SM of the sync-free solves

// Next application: new epoch, tickets back to 0 (clear = 1: only the error word).
__global__ void k_sf_begin(int32_t *ctl, int clear)
{
    if (threadIdx.x != 0) return;
    if (clear) {
        ctl[3] = 0;
        return;
    }
    ctl[0] += 1;
    ctl[1] = 0;
    ctl[2] = 0;
}

template <typename TR, typename TZ, typename TM, typename TP, bool G>
__global__ void __launch_bounds__(kBlock) k_ilu_fwd_sf(DeviceMesh d, const TP *__restrict__ Pg,
                                                       const TP *__restrict__ alg, const TP *__restrict__ exg,
                                                       const TP *__restrict__ eyg, const TR *r, TZ *z,
                                                       int32_t *flag, int32_t *ctl,
                                                       const TP *__restrict__ arg = nullptr,
                                                       const TP *__restrict__ exrg = nullptr,
                                                       const TP *__restrict__ eyrg = nullptr,
                                                       const TP *__restrict__ bdgg = nullptr)
{
    __shared__ int32_t ticket;
    const int64_t T = d.T;
    const int64_t nt = (T + kBlock - 1) / kBlock;
    const int32_t tag = 2 * ctl[0] + 1;
    for (;;) {
        if (threadIdx.x == 0) ticket = atomicAdd(ctl + 1, 1);
        __syncthreads();
        const int64_t tk = ticket;
        __syncthreads();
        if (tk >= nt) return;
        const int64_t i = tk * kBlock + threadIdx.x;
        if (i < T)
            ilu_fwd_row<TR, TZ, TM, TP, G, true>(d, Pg, alg, exg, eyg, i, r, z, z, 1, nullptr, arg, exrg, eyrg, bdgg,
                                                 flag, tag, ctl + 3);
    }
}

template <typename TZ, typename TM, typename TP, bool G>
__global__ void __launch_bounds__(kBlock) k_ilu_bwd_sf(DeviceMesh d, const TP *__restrict__ Pg,
                                                       const TP *__restrict__ alg, const TP *__restrict__ exg,
                                                       const TP *__restrict__ eyg, TZ *x, int32_t *flag,
                                                       int32_t *ctl, const TP *__restrict__ arg = nullptr,
                                                       const TP *__restrict__ exrg = nullptr,
                                                       const TP *__restrict__ eyrg = nullptr,
                                                       const TP *__restrict__ bdgg = nullptr)
{
    __shared__ int32_t ticket;
    const int64_t T = d.T;
    const int64_t nt = (T + kBlock - 1) / kBlock;
    const int32_t tag = 2 * ctl[0] + 2;
    for (;;) {
        if (threadIdx.x == 0) ticket = atomicAdd(ctl + 2, 1);
        __syncthreads();
        const int64_t tk = ticket;
        __syncthreads();
        if (tk >= nt) return;
        const int64_t i = T - 1 - (tk * kBlock + threadIdx.x);
        if (i >= 0)
            ilu_bwd_row<TZ, TM, TP, G, true>(d, Pg, alg, exg, eyg, i, x, x, x, arg, exrg, eyrg, bdgg, flag, tag,
                                             ctl + 3);
    }
}

// Partial dot products <V_k, w> of the four variables over one block of
// kBlock cells: grid (k, block), blockIdx.x = k so that the j + 1 blocks of a
// cell block run together and read w once from HBM.  64 threads per variable,
// four cells each (64 apart), all 40 loads issued before the sums (read-only
// kernels need many bytes in flight); the warp sums then the two warps of a
// variable give part[k][v][blk].  Fixed order: the sums are deterministic.
// TB: type of the stored basis.  An FP64 basis is multiplied and summed in
// FP64; an FP32 basis (the inner cycles of the mixed mode) in FP32 within a
// warp (640 products), each warp's sum then widened once and summed across
// warps and blocks in FP64, so that the FP64 pipe sees almost nothing.
template <typename TB>
__global__ void __launch_bounds__(kDotThreads, 3) k_dots(int64_t T, int64_t nblk, const TB *__restrict__ V,
                                                         const TB *__restrict__ w, double *__restrict__ part)
{
    constexpr int kPerVar = kDotThreads / NV;          // 64 threads (two warps) per variable
    constexpr int kCells = kBlock / kPerVar;           // 4 cells per thread
    __shared__ double sh[kDotThreads / 32];
    const int k = blockIdx.x;
    const int v = threadIdx.x / kPerVar, t = threadIdx.x % kPerVar;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const TB *vk = V + (int64_t)k * NX * T + (int64_t)v * ND * T;
    const TB *wv = w + (int64_t)v * ND * T;
    for (int64_t b = blockIdx.y; b < nblk; b += gridDim.y) {
        const int64_t c0 = b * kBlock + t;
        TB st = TB(0);
#pragma unroll
        for (int q = 0; q < kCells; ++q) {
            const int64_t i = c0 + q * kPerVar;
#pragma unroll
            for (int l = 0; l < ND; ++l) st = i < T ? fma(vk[l * T + i], wv[l * T + i], st) : st;
        }
        // warp sum in the basis precision, widened once per warp
        for (int o = 16; o > 0; o >>= 1) st += __shfl_down_sync(0xffffffffu, st, o);
        if (lane == 0) sh[warp] = double(st);
        __syncthreads();
        if (threadIdx.x < NV) part[(k * NV + threadIdx.x) * nblk + b] = sh[2 * threadIdx.x] + sh[2 * threadIdx.x + 1];
        __syncthreads();
    }
}

// The same for an FP32 basis ([dof][cell][variable]): a thread per cell, FP32
// within a warp (160 products), FP64 across warps and blocks.
__global__ void __launch_bounds__(kBlock) k_dots32(int64_t T, const float *__restrict__ V,
                                                   const float *__restrict__ w, double *__restrict__ part)
{
    __shared__ float sh[kBlock / 32][1][4];
    const int64_t b = blockIdx.x, i = b * kBlock + threadIdx.x;
    const int k = blockIdx.y;
    float sv[1][4] = {};
    if (i < T)
#pragma unroll
        for (int l = 0; l < ND; ++l) {
            float a[NV], u[NV];
            vload(V + (int64_t)k * NX * T, l, T, i, a);
            vload(w, l, T, i, u);
#pragma unroll
            for (int v = 0; v < NV; ++v) sv[0][v] = fmaf(a[v], u[v], sv[0][v]);
        }
    block_rows32<1>(sv, sh, part, k);
}

// w -= sum_{k<=j} c[s][k] V_k for running systems s = case * 4 + v (c: the
// Gram-Schmidt coefficients of the unnormalised basis), w = 0 for the others;
// optional partial |w|^2 per block.  The arithmetic is in the basis precision
// TB (FP32 for the inner cycles of the mixed mode); the block's coefficients
// are rounded to TB once, in shared memory.  J > 0: the Arnoldi index j = J - 1
// is a compile-time constant and every load of the four systems is issued
// before the arithmetic (systems that are not running read their vectors too
// and store zeros), for more bytes in flight per thread; the same operations
// in the same order as the loop over k.
template <typename TB, int J = 0>
__global__ void k_orth_update(DeviceMesh d, const TB *__restrict__ V, TB *__restrict__ w, int j,
                              const double *__restrict__ hc, int hstride, const int32_t *__restrict__ ctl, int ns,
                              double *__restrict__ part, int want_norm)
{
    if (J > 0) j = J - 1;
    __shared__ double sh[32 * NV];
    __shared__ TB shc[NV][kMaxRestart];
    const int64_t T = d.T;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t vs = (int64_t)NX * T;
    const int c = d.blk_case[blockIdx.x];
    for (int q = threadIdx.x; q < NV * (j + 1); q += blockDim.x)
        shc[q / (j + 1)][q % (j + 1)] = TB(hc[(4 * c + q / (j + 1)) * hstride + q % (j + 1)]);
    __syncthreads();
    TB nrm[NV] = {0, 0, 0, 0};
    if (J > 0 && i < T) {
        bool run[NV];
        TB wv[ND][NV], vk[J > 0 ? J : 1][ND][NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) run[v] = ctl[kCtlRunning * ns + 4 * c + v] != 0;
#pragma unroll
        for (int l = 0; l < ND; ++l) vload(w, l, T, i, wv[l]);
#pragma unroll
        for (int k = 0; k < J; ++k)
#pragma unroll
            for (int l = 0; l < ND; ++l) vload(V + k * vs, l, T, i, vk[k][l]);
#pragma unroll
        for (int l = 0; l < ND; ++l) {
#pragma unroll
            for (int v = 0; v < NV; ++v) {
#pragma unroll
                for (int k = 0; k < J; ++k) wv[l][v] = fma(-shc[v][k], vk[k][l][v], wv[l][v]);
                wv[l][v] = run[v] ? wv[l][v] : TB(0);
                nrm[v] = fma(wv[l][v], wv[l][v], nrm[v]);
            }
            vstore(w, l, T, i, wv[l]);
        }
    } else if (i < T) {
        TB wv[ND][NV];
#pragma unroll
        for (int l = 0; l < ND; ++l) vload(w, l, T, i, wv[l]);
        for (int k = 0; k <= j; ++k)
#pragma unroll
            for (int l = 0; l < ND; ++l) {
                TB t[NV];
                vload(V + k * vs, l, T, i, t);
#pragma unroll
                for (int v = 0; v < NV; ++v) wv[l][v] = fma(-shc[v][k], t[v], wv[l][v]);
            }
#pragma unroll
        for (int l = 0; l < ND; ++l) {
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                wv[l][v] = ctl[kCtlRunning * ns + 4 * c + v] ? wv[l][v] : TB(0);
                nrm[v] = fma(wv[l][v], wv[l][v], nrm[v]);
            }
            vstore(w, l, T, i, wv[l]);
        }
    }
    if (want_norm) {
        double nd[NV];
        if (std::is_same<TB, float>::value) {
            // warp sums in FP32, widened once per warp
            const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                for (int o = 16; o > 0; o >>= 1) nrm[v] += __shfl_down_sync(0xffffffffu, nrm[v], o);
                if (lane == 0) sh[warp * NV + v] = double(nrm[v]);
            }
            __syncthreads();
            if (threadIdx.x == 0)
                for (int v = 0; v < NV; ++v) {
                    double t = 0.0;
                    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w * NV + v];
                    nd[v] = t;
                }
        } else {
#pragma unroll
            for (int v = 0; v < NV; ++v) nd[v] = double(nrm[v]);
            block_sum4(nd, sh);
        }
        if (threadIdx.x == 0)
            for (int v = 0; v < NV; ++v) part[v * (int64_t)gridDim.x + blockIdx.x] = nd[v];
    }
}

// x += sum_k y[s][k] Z_k, k < jv, with Z_k = M^{-1} V_k kept from the iterations.
// FP64 path (extended stencil; see k64_combine): FP64 sums, one variable per grid row.
__global__ void k_combine_z(DeviceMesh d, const double *__restrict__ Z, const double *__restrict__ y, int m,
                            const int32_t *__restrict__ ctl, int ns, double *__restrict__ x)
{
    const int64_t T = d.T;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= T) return;
    const int v = blockIdx.y;
    const int sy = 4 * d.blk_case[blockIdx.x] + v;
    const int jv = ctl[kCtlJv * ns + sy];
    if (jv <= 0) return;
    const int64_t vs = (int64_t)NX * T;
    double acc[ND] = {0, 0, 0, 0, 0};
    for (int k = 0; k < jv; ++k) {
        const double yk = y[sy * m + k];
#pragma unroll
        for (int l = 0; l < ND; ++l) acc[l] += yk * Z[k * vs + (v * ND + l) * T + i];
    }
#pragma unroll
    for (int l = 0; l < ND; ++l) x[(v * ND + l) * T + i] += acc[l];
}

// Mixed path (FP32 Z): the correction of one inner cycle is formed in FP32 (it
// only has to be accurate to the inner tolerance; the next FP64 residual measures
// what is left) and added to x in FP64, so the FP64 pipe sees one add per value
// instead of one conversion and one FMA per value and Krylov vector.  With sexp
// given (FP32 basis): y carries 2^-e of the cycle (see k_cycle_solve) and the sum
// is scaled back by 2^e exactly, on the integer pipe (f2d_pow2).  A thread per
// cell and variable, the four variables of a cell in neighbouring lanes.
__global__ void __launch_bounds__(kBlock) k_combine32(DeviceMesh d, const float *__restrict__ Z,
                                                      const float *__restrict__ y32, int m,
                                                      const int32_t *__restrict__ ctl, int ns,
                                                      double *__restrict__ x, const int32_t *__restrict__ sexp)
{
    const int64_t T = d.T;
    const int v = threadIdx.x & 3;
    const int64_t i = blockIdx.x * (int64_t)(kBlock / NV) + (threadIdx.x >> 2);
    if (i >= T) return;
    const int sy = 4 * d.blk_case[blockIdx.x / NV] + v;
    const int jv = ctl[kCtlJv * ns + sy];
    if (jv <= 0) return;
    const float *zv = Z + i * NV + v;
    const int64_t ls = NV * T, vs = (int64_t)NX * T;
    double xi[ND];
#pragma unroll
    for (int l = 0; l < ND; ++l) xi[l] = x[(v * ND + l) * T + i];
    float acc[ND] = {0, 0, 0, 0, 0};
#pragma unroll 4
    for (int k = 0; k < jv; ++k) {
        const float yk = y32[sy * m + k];
#pragma unroll
        for (int l = 0; l < ND; ++l) acc[l] = fmaf(yk, zv[k * vs + l * ls], acc[l]);
    }
    const int e = sexp ? sexp[sy] : 0;
#pragma unroll
    for (int l = 0; l < ND; ++l) x[(v * ND + l) * T + i] = xi[l] + (sexp ? f2d_pow2(acc[l], e) : double(acc[l]));
}

// Warm start of solve n (cases not done) from the last solutions
// x = s_{n-1}, xp = s_{n-2}, xpp = s_{n-3}: order 0 keeps x, order 1 takes
// 2 x - xp, order 2 takes 3 x - 3 xp + xpp (polynomial extrapolation in the
// step index).  The history shifts by an exchange of the two buffers' roles,
// which follow the parity of the device's solve count n (k_mark_noconv raises
// it after the solve): the old x goes into xpp's buffer (the next xp), and
// xp's buffer (the next xpp) already holds s_{n-2}, so one vector is written
// instead of two.  Cells of finished cases keep their history: their two
// buffers exchange contents, which the exchange of roles undoes.
__global__ void k_warm(DeviceMesh d, double *__restrict__ x, double *__restrict__ h0, double *__restrict__ h1,
                       const int32_t *__restrict__ done, const int64_t *__restrict__ nsolve, int max_order)
{
    const int64_t T = d.T;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= T) return;
    const int q0 = blockIdx.y * ND;                  // one variable per grid row
    // n solves so far: the two history buffers swap roles after every solve, and
    // the extrapolation uses as many past solutions as exist
    const int64_t n = *nsolve;
    double *__restrict__ xp = (n & 1) ? h1 : h0;
    double *__restrict__ xpp = (n & 1) ? h0 : h1;
    const int order = (max_order >= 2 && n >= 3) ? 2 : (n >= 2 ? 1 : 0);
    if (done[d.blk_case[blockIdx.x]]) {
#pragma unroll
        for (int q = q0; q < q0 + ND; ++q) {
            const double b = xp[q * T + i], c = xpp[q * T + i];
            xp[q * T + i] = c;
            xpp[q * T + i] = b;
        }
        return;
    }
#pragma unroll
    for (int q = q0; q < q0 + ND; ++q) {
        const double a = x[q * T + i];
        if (order == 2) x[q * T + i] = 3.0 * (a - xp[q * T + i]) + xpp[q * T + i];
        else if (order == 1) x[q * T + i] = 2.0 * a - xp[q * T + i];
        xpp[q * T + i] = a;
    }
}

// Condition of the device-controlled step loop (one block): any case not done,
// and the loops of this launch (run_ctl[0]) below its limit (run_ctl[1]).
// entry = 1 before the loop (no loops yet); otherwise at the end of a loop,
// which it counts in run_ctl[0] and in ctr[kCtrRun].
__global__ void k_run_cond(const int32_t *done, int n, int64_t *run_ctl, int64_t *ctr, cudaGraphConditionalHandle h,
                           int entry)
{
    __shared__ int any;
    if (threadIdx.x == 0) any = 0;
    __syncthreads();
    int a = 0;
    for (int c = threadIdx.x; c < n; c += blockDim.x) a |= done[c] == 0;
    if (a) atomicOr(&any, 1);
    __syncthreads();
    if (threadIdx.x != 0) return;
    int64_t loops = 0;
    if (!entry) {
        loops = run_ctl[0] + 1;
        ctr[kCtrRun] += 1;
    }
    run_ctl[0] = loops;
    cudaGraphSetConditional(h, (any && loops < run_ctl[1]) ? 1u : 0u);
}

// x = 0 for systems with b = 0 (|b| compared as integers: an FP64 comparison per
// thread took 10 us at 1M triangles)
__global__ void k_zero_trivial(DeviceMesh d, double *__restrict__ x, const double *__restrict__ bnorm)
{
    const int64_t T = d.T;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= T) return;
    const int c = d.blk_case[blockIdx.x];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const long long b = __double_as_longlong(bnorm[4 * c + v]);
        if (b > 0 && b <= 0x7FF0000000000000ll) continue;      // |b| > 0
#pragma unroll
        for (int l = 0; l < ND; ++l) x[(v * ND + l) * T + i] = 0.0;
    }
}

// status[c] |= noconv for cases with a system that stopped above the tolerance,
// and |= timeout for every active case if a wait of the sync-free ILU solves
// gave up during the solve (sf_err, may be NULL); the solve count of the warm
// start (k_warm) goes up by one; in a run (acc) the solve's iterations it are
// added to the sums acc
__global__ void k_mark_noconv(const double *__restrict__ bnorm, const double *__restrict__ beta,
                              const int32_t *__restrict__ done, int ns, double rtol, int32_t *status,
                              int64_t *nsolve, const int32_t *sf_err, const int32_t *__restrict__ it, int64_t *acc)
{
    const int sy = blockIdx.x * blockDim.x + threadIdx.x;
    if (sy == 0) ++*nsolve;
    if (acc && sy < ns) acc[sy] += it[sy];
    if (sy >= ns || done[sy >> 2]) return;
    if (bnorm[sy] > 0.0 && beta[sy] > rtol * bnorm[sy]) atomicOr(&status[sy >> 2], kStatusNoConv);
    if (sf_err && *sf_err) atomicOr(&status[sy >> 2], kStatusTimeout);
}

inline unsigned nblocks(int64_t n) { return (unsigned)((n + kBlock - 1) / kBlock); }

// k_orth_update with the Arnoldi index unrolled for the first four indices
// (the inner cycles of the mixed mode rarely go further)
template <typename TB>
void launch_orth_update(const DeviceMesh &d, unsigned nb, cudaStream_t q, const TB *V, TB *w, int j,
                        const double *hc, int hstride, const int32_t *ctl, int ns, double *part, int want_norm)
{
    switch (j) {
    case 0: k_orth_update<TB, 1><<<nb, kBlock, 0, q>>>(d, V, w, j, hc, hstride, ctl, ns, part, want_norm); break;
    case 1: k_orth_update<TB, 2><<<nb, kBlock, 0, q>>>(d, V, w, j, hc, hstride, ctl, ns, part, want_norm); break;
    case 2: k_orth_update<TB, 3><<<nb, kBlock, 0, q>>>(d, V, w, j, hc, hstride, ctl, ns, part, want_norm); break;
    case 3: k_orth_update<TB, 4><<<nb, kBlock, 0, q>>>(d, V, w, j, hc, hstride, ctl, ns, part, want_norm); break;
    default: k_orth_update<TB><<<nb, kBlock, 0, q>>>(d, V, w, j, hc, hstride, ctl, ns, part, want_norm);
    }
}

// The reverse-slot coefficients of the global normal equations for the ILU
// kernels (all NULL for the per-cell equations).
template <typename TP>
struct RevSlots {
    const TP *a = nullptr, *x = nullptr, *y = nullptr, *b = nullptr;
};

// dst = M^{-1} src (block ILU(0) on the RCM order).  TZ, TM: storage and
// arithmetic precision of the application; TP: storage of the factors; tA, tB:
// work buffers of type TZ; rev: reverse slots of the global normal equations.
template <typename TR, typename TZ, typename TM, typename TP = TM>
gks_status precond_t(gks_mesh *m, const TP *Pg, const TP *alg, const TP *exg, const TP *eyg, const TR *src,
                     TZ *dst, TZ *tA, TZ *tB, TZ *rz, cudaStream_t s, RevSlots<TP> rev = {})
{
    DeviceMesh &d = m->d;
    const int64_t T = d.T;
    // forward / backward relation, the global variant when reverse slots are given
    auto fwd_global = [&](int64_t n, const int32_t *rows, auto r, const TZ *zin, TZ *zout, int use_nb, TZ *rc) {
        using TRx = std::remove_cv_t<std::remove_pointer_t<decltype(r)>>;
        k_ilu_fwd<TRx, TZ, TM, TP, true><<<nblocks(n), kBlock, 0, s>>>(d, Pg, alg, exg, eyg, rows, n, r, zin, zout,
                                                                      use_nb, rc, rev.a, rev.x, rev.y, rev.b);
        note_launch();
    };
    auto fwd = [&](int64_t n, const int32_t *rows, const TR *r, const TZ *zin, TZ *zout, int use_nb) {
        if (rev.a) return fwd_global(n, rows, r, zin, zout, use_nb, nullptr);
        k_ilu_fwd<TR, TZ, TM, TP, false><<<nblocks(n), kBlock, 0, s>>>(d, Pg, alg, exg, eyg, rows, n, r, zin, zout,
                                                                      use_nb, nullptr);
        note_launch();
    };
    auto bwd = [&](int64_t n, const int32_t *rows, const TZ *z, const TZ *xin, TZ *xout) {
        if (rev.a)
            k_ilu_bwd<TZ, TM, TP, true><<<nblocks(n), kBlock, 0, s>>>(d, Pg, alg, exg, eyg, rows, n, z, xin, xout,
                                                                     rev.a, rev.x, rev.y, rev.b);
        else
            k_ilu_bwd<TZ, TM, TP, false><<<nblocks(n), kBlock, 0, s>>>(d, Pg, alg, exg, eyg, rows, n, z, xin, xout);
        note_launch();
    };
    if (m->cfg.precond == GKS_PC_ILU_EXACT) {
        // sync-free: a new epoch, then one launch per relation
        Work &k = m->wk;
        k_sf_begin<<<1, 32, 0, s>>>(k.sf_ctl, 0);
        note_launch();
        const unsigned g = (unsigned)std::min<int64_t>(nblocks(T), (int64_t)k.sm_count * kSfBlocksPerSm);
        if (rev.a)
            k_ilu_fwd_sf<TR, TZ, TM, TP, true><<<g, kBlock, 0, s>>>(d, Pg, alg, exg, eyg, src, dst, k.sf_flag,
                                                                    k.sf_ctl, rev.a, rev.x, rev.y, rev.b);
        else
            k_ilu_fwd_sf<TR, TZ, TM, TP, false><<<g, kBlock, 0, s>>>(d, Pg, alg, exg, eyg, src, dst, k.sf_flag,
                                                                     k.sf_ctl);
        note_launch();
        if (rev.a)
            k_ilu_bwd_sf<TZ, TM, TP, true><<<g, kBlock, 0, s>>>(d, Pg, alg, exg, eyg, dst, k.sf_flag, k.sf_ctl,
                                                                rev.a, rev.x, rev.y, rev.b);
        else
            k_ilu_bwd_sf<TZ, TM, TP, false><<<g, kBlock, 0, s>>>(d, Pg, alg, exg, eyg, dst, k.sf_flag, k.sf_ctl);
        note_launch();
    } else if (m->cfg.precond == GKS_PC_ILU_LEVELS) {
        const auto &lp = m->lvl_lo_ptr;
        for (size_t l = 0; l + 1 < lp.size(); ++l)
            fwd(lp[l + 1] - lp[l], d.lvl_lo + lp[l], src, dst, dst, 1);
        const auto &up = m->lvl_up_ptr;
        for (size_t l = 0; l + 1 < up.size(); ++l) bwd(up[l + 1] - up[l], d.lvl_up + up[l], dst, dst, dst);
    } else if (m->cfg.precond == GKS_PC_BJACOBI) {
        fwd(T, nullptr, src, nullptr, dst, 0);     // z = P r, the block-diagonal inverse
    } else {
        // sweeps of the global normal equations (those of the per-cell equations:
        // precond64, precond32s): forward z^0 = P r, z^{q+1} = F(z^q); backward x^0 = z, x^{q+1} = B(x^q)
        const int ns = m->cfg.ilu_sweeps;
        const int nsb = m->cfg.ilu_sweeps_bwd < 0 ? ns : m->cfg.ilu_sweeps_bwd;
        // z^0 folded into the first sweep (ilu_fuse_first) or a pass of its own
        const bool fuse = ns > 0 && m->cfg.ilu_fuse_first;
        const int nf = fuse ? ns : ns + 1;   // forward launches
        TZ *za = (nf % 2 == 1) ? tA : dst;   // buffers chosen so that z ends in tA
        TZ *zb = (nf % 2 == 1) ? dst : tA;
        // a wider source is rounded to TZ once, in the first pass, for the sweeps
        TZ *rc = (sizeof(TR) > sizeof(TZ) && ns > 0) ? rz : nullptr;
        fwd_global(T, nullptr, src, nullptr, za, fuse ? 2 : 0, rc);
        for (int q = fuse ? 1 : 0; q < ns; ++q) {
            if (rc)
                fwd_global(T, nullptr, (const TZ *)rc, za, zb, 1, (TZ *)nullptr);
            else
                fwd_global(T, nullptr, src, za, zb, 1, (TZ *)nullptr);
            std::swap(za, zb);
        }
        if (nsb == 0) {
            GKS_CUDA(cudaMemcpyAsync(dst, za, sizeof(TZ) * NX * T, cudaMemcpyDeviceToDevice, s));
        } else {
            TZ *xa = za;                                    // x^0 = z (in za)
            TZ *xb = (nsb % 2 == 1) ? dst : (za == tB ? tA : tB);
            for (int q = 0; q < nsb; ++q) {
                bwd(T, nullptr, za, xa, xb);
                xa = xb;
                xb = (xb == dst) ? tB : dst;
            }
        }
    }
    GKS_CUDA(cudaGetLastError());
    return GKS_OK;
}

// The sweeps of the FP64 solve of the per-cell equations (a thread per cell and
// variable, see gks_solve64.cuh): dst = M^{-1} src with the sweeps of precond_t.
//
// z = P src is in t3 (rows 0 and 1 of it are z^0).  The rows 0 and 1 of the other
// intermediate results go to four pairs of rows, two in t2 and two in dst; what the
// last launch reads of neighbours, z^{ns-1} and x^{nsb-1}, is in t3 or t2.
gks_status precond64(gks_mesh *m, const double *src, double *dst, cudaStream_t s)
{
    const DeviceMesh &d = m->d;
    Work &k = m->wk;
    const int64_t T = d.T;
    const unsigned g = (unsigned)((T + 31) / 32);
    const int32_t *run = k.ctl + kCtlRunning * k.ns;
    const int ns = m->cfg.ilu_sweeps, nsb = m->cfg.ilu_sweeps_bwd < 0 ? ns : m->cfg.ilu_sweeps_bwd;
    // forward sweeps of the rows 0 and 1: z^ns is the start of the backward sweeps
    const int nf = nsb > 0 ? ns : ns - 1;
    double *z = ns + nsb > 0 ? k.t3 : dst;
    double *t2a = k.t2, *t2b = k.t2 + 2 * T, *da = dst, *db = dst + 2 * T;
    // z^q (0 < q <= nf), z^{ns-1} in t2a; z^ns in da (t2b where the last launch reads it as x^0)
    auto zq = [&](int q) { return q == 0 ? z : (q == ns ? (nsb == 1 ? t2b : da) : ((ns - 1 - q) % 2 == 0 ? t2a : da)); };
    // x^q (q < nsb), x^0 = z^ns, x^{nsb-1} in t2b
    auto xq = [&](int q) { return q == 0 ? zq(ns) : ((nsb - 1 - q) % 2 == 0 ? t2b : db); };
    k64_pivot<<<g, kW64, 0, s>>>(T, d.P, d.blk_case, run, src, z);
    note_launch();
    for (int q = 0; q < nf; ++q) {
        k64_sweep<false><<<g, kW64, 0, s>>>(T, d.nb, d.w64, d.blk_case, run, z, zq(q), zq(q + 1));
        note_launch();
    }
    for (int q = 0; q + 1 < nsb; ++q) {
        k64_sweep<true><<<g, kW64, 0, s>>>(T, d.nb, d.w64, d.blk_case, run, zq(ns), xq(q), xq(q + 1));
        note_launch();
    }
    if (ns + nsb > 0) {
        k64_last<<<g, kW64, 0, s>>>(T, d.nb, d.w64, d.blk_case, run, z, ns > 0 ? zq(ns - 1) : nullptr,
                                    nsb > 0 ? xq(nsb - 1) : nullptr, dst);
        note_launch();
    }
    GKS_CUDA(cudaGetLastError());
    return GKS_OK;
}

// Up to this many triangles the second Gram-Schmidt pass of the FP64 solve is a block per
// system inside k_arnoldi_end; above, three launches over the whole GPU, which return at once
// (about 1.3 us each) when no system needs them.  Timed both ways on 148 systems (cells stretched
// up to 300 : 1, no to four sweeps, restarts of 8 and 30; passes in none to two thirds of the
// indices): up to 968 triangles the block is the faster one for every solve that converged
// (0.5 to 8 %; exact triangular solves, bound by their waits, within 4 % either way), at 1,800-1,922 it
// is 2 to 7 % faster where passes are rare and up to 11 % slower where they are not, at 6,400 (a
// shock tube) 30 % slower.
constexpr int64_t kSolo64 = 1000;

// A launch with c cells per thread.
template <typename F>
void with_cells(int c, F &&f)
{
    switch (c) {
    case 1: f(std::integral_constant<int, 1>{}); break;
    case 2: f(std::integral_constant<int, 2>{}); break;
    case 4: f(std::integral_constant<int, 4>{}); break;
    default: f(std::integral_constant<int, 8>{}); break;
    }
    note_launch();
}

inline unsigned rows64(const gks_mesh *m) { return (unsigned)(m->wk.nblk * (kRows64 / m->wk.c64)); }

// dynamic shared memory of the product kernels at Arnoldi index j
inline size_t acc64(int j, int stride) { return sizeof(double) * 4 * (j + 1) * stride; }

// Beyond 48 KiB (restart lengths above 45) the kernels have to ask for it.  The limit
// is the process's, not the handle's: always that of the longest restart, so that a
// handle never lowers it between another's call and launch.
gks_status solve64_shared_limit()
{
    auto set = [&](auto C) -> gks_status {
        constexpr int c = decltype(C)::value;
        GKS_CUDA(cudaFuncSetAttribute(k64_apply_dots<c>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)acc64(kMaxRestart, kAccStride)));
        GKS_CUDA(cudaFuncSetAttribute(k64_update<c>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)acc64(kMaxRestart - 1, kAccStride + 1)));
        return GKS_OK;
    };
    gks_status st = set(std::integral_constant<int, 1>{});
    if (st == GKS_OK) st = set(std::integral_constant<int, 2>{});
    if (st == GKS_OK) st = set(std::integral_constant<int, 4>{});
    if (st == GKS_OK) st = set(std::integral_constant<int, 8>{});
    return st;
}

void solve64_rhs(gks_mesh *m, cudaStream_t q)
{
    const DeviceMesh &d = m->d;
    with_cells(m->wk.c64, [&](auto C) {
        k64_rhs<decltype(C)::value><<<rows64(m), kW64, 0, q>>>(d.T, d.nb, d.a0, m->wk.w, m->wk.b, m->wk.part);
    });
}

void solve64_resid(gks_mesh *m, double *V0, const int32_t *act, cudaStream_t q)
{
    const DeviceMesh &d = m->d;
    with_cells(m->wk.c64, [&](auto C) {
        k64_resid<decltype(C)::value><<<rows64(m), kW64, 0, q>>>(d.T, d.nb, d.D, d.off, d.blk_case, act, m->wk.x,
                                                               m->wk.b, V0, m->wk.part);
    });
}

void solve64_apply_dots(gks_mesh *m, const double *z, const double *V, double *y, int j, cudaStream_t q)
{
    const DeviceMesh &d = m->d;
    with_cells(m->wk.c64, [&](auto C) {
        k64_apply_dots<decltype(C)::value><<<rows64(m), kW64, acc64(j + 1, kAccStride), q>>>(
            d.T, d.nb, d.D, d.off, d.blk_case, m->wk.ctl + kCtlRunning * m->wk.ns, z, y, V, j, m->wk.part);
    });
}

// the first update with the end of Arnoldi index j
void solve64_update(gks_mesh *m, const Krylov &kry, const double *V, double *w, int j, int ps, const Cond &cd,
                    cudaStream_t q)
{
    const DeviceMesh &d = m->d;
    const Work &k = m->wk;
    with_cells(m->wk.c64, [&](auto C) {
        k64_update<decltype(C)::value>
            <<<m->n_case + rows64(m), kW64, std::max(acc64(j, kAccStride + 1), 4 * sizeof(GivensRows)), q>>>(
                d.T, d.blk_case, kry, m->n_case, V, w, j, k.hcol, k.hco, ps, k.ctl + kCtlRan * k.ns,
                k.ctl + kCtlTwice * k.ns, cd, k.part);
    });
}

void solve64_update_norm(gks_mesh *m, const double *V, double *w, int j, int ps, cudaStream_t q)
{
    const DeviceMesh &d = m->d;
    with_cells(m->wk.c64, [&](auto C) {
        k64_update_norm<decltype(C)::value><<<rows64(m), kW64, 0, q>>>(
            d.T, d.blk_case, m->wk.ctl + kCtlRunning * m->wk.ns, m->wk.ctl + kCtlTwice * m->wk.ns, V, w, j, m->wk.hco,
            ps, m->wk.part);
    });
}

template <typename TR>
gks_status precond(gks_mesh *m, const TR *src, double *dst, cudaStream_t s)
{
    DeviceMesh &d = m->d;
    if constexpr (std::is_same_v<TR, double>)
        if (d.w64) return precond64(m, src, dst, s);
    return precond_t<TR, double, double>(m, d.P, d.alpha, d.ex, d.ey, src, dst, m->wk.t2, m->wk.t3, nullptr, s,
                                         {d.alr, d.exr, d.eyr, d.bdg});
}

void solve32_rhs(gks_mesh *m, cudaStream_t q)
{
    const unsigned g = (unsigned)(m->wk.nblk * (kRows64 / m->wk.c32));
    with_cells(m->wk.c32, [&](auto C) {
        k_rhs_df<decltype(C)::value><<<g, kW32, 0, q>>>(m->d, m->d.a0p, m->wk.w, m->wk.b, m->wk.part);
    });
}

void solve32_apply_dots(gks_mesh *m, const float *z, const float *V, float *y, int j, cudaStream_t q)
{
    const DeviceMesh &d = m->d;
    const Work &k = m->wk;
    const int32_t *run = k.ctl + kCtlRunning * k.ns;
    const float4 *op = reinterpret_cast<const float4 *>(d.op32);
#define A32(J) k32_apply_dots<J><<<k.nblk, kBlock, 0, q>>>(d.T, d.nb, op, d.blk_case, run, z, y, V, j, k.part)
    switch (j) {     // the first four Arnoldi indices unrolled (the inner cycles rarely go further)
    case 0: A32(1); break;
    case 1: A32(2); break;
    case 2: A32(3); break;
    case 3: A32(4); break;
    default: A32(0);
    }
#undef A32
    note_launch();
}

// the update with the end of Arnoldi index j
void solve32_update(gks_mesh *m, const Krylov &kry, const float *V, float *w, int j, int ps, const Cond &cd,
                    cudaStream_t q)
{
    const DeviceMesh &d = m->d;
    const Work &k = m->wk;
    const unsigned g = (unsigned)(m->n_case + k.nblk);
    const int32_t *ran = k.ctl + kCtlRan * k.ns;
#define U32(J) \
    k32_update<J><<<g, kBlock, 0, q>>>(d.T, d.blk_case, kry, m->n_case, V, w, j, k.hcol, k.hco, ps, ran, cd)
    switch (j) {
    case 0: U32(1); break;
    case 1: U32(2); break;
    case 2: U32(3); break;
    case 3: U32(4); break;
    default: U32(0);
    }
#undef U32
    note_launch();
}

// The FP32 sweeps of the per-cell equations with packed factors (see precond64
// for the buffers).  A wider source is rounded to FP32 once, in the
// first pass, for the later sweeps.
template <typename TR, typename TP>
gks_status precond32s(gks_mesh *m, const TP *pk, const TR *src, float *dst, cudaStream_t s)
{
    const DeviceMesh &d = m->d;
    Work &k = m->wk;
    const int64_t T = d.T;
    const unsigned g = (unsigned)((T + kW32 - 1) / kW32);
    const int32_t *run = k.ctl + kCtlRunning * k.ns;
    const int ns = m->cfg.ilu_sweeps, nsb = m->cfg.ilu_sweeps_bwd < 0 ? ns : m->cfg.ilu_sweeps_bwd;
    const bool fuse = ns > 0 && m->cfg.ilu_fuse_first;
    float *z = nsb > 0 ? k.t3_32 : dst;
    auto mid = [&](int q, int n) { return (n - 1 - q) % 2 == 0 ? k.t2_32 : dst; };
    float *rc = (sizeof(TR) > sizeof(float) && ns > 0) ? k.r32 : nullptr;
    const int nf = fuse ? ns : ns + 1;                    // forward launches
    const float *prev = nullptr;
    for (int q = 0; q < nf; ++q) {
        const bool last = q + 1 == nf;
        float *out = last ? z : mid(q, nf - 1);
#define F32(NB, FULL, TS, SRC, RC) \
    k32_fwd<NB, FULL, TS, TP><<<g, kW32, 0, s>>>(T, d.nb, pk, d.blk_case, run, SRC, prev, out, RC)
        if (q == 0 && fuse) last ? F32(2, true, TR, src, rc) : F32(2, false, TR, src, rc);
        else if (q == 0) last ? F32(0, true, TR, src, rc) : F32(0, false, TR, src, rc);
        else if (rc) last ? F32(1, true, float, rc, nullptr) : F32(1, false, float, rc, nullptr);
        else last ? F32(1, true, TR, src, nullptr) : F32(1, false, TR, src, nullptr);
#undef F32
        note_launch();
        prev = out;
    }
    // backward: pairs of sweeps (ilu_sweep_pairs), then a single one if nsb is odd
    const int npair = m->cfg.ilu_sweep_pairs ? nsb / 2 : 0, nb = npair + (nsb - 2 * npair);
    const float *x = z;
    for (int q = 0; q < nb; ++q) {
        const bool last = q + 1 == nb;
        float *out = last ? dst : mid(q, nb - 1);
#define B32(K, FULL) K<FULL, TP><<<g, kW32, 0, s>>>(T, d.nb, pk, d.blk_case, run, z, x, out)
        if (q < npair) last ? B32(k32_bwd2, true) : B32(k32_bwd2, false);
        else last ? B32(k32_bwd, true) : B32(k32_bwd, false);
#undef B32
        note_launch();
        x = out;
    }
    GKS_CUDA(cudaGetLastError());
    return GKS_OK;
}

template <typename TR>
gks_status precond32(gks_mesh *m, const TR *src, float *dst, cudaStream_t s)
{
    DeviceMesh &d = m->d;
    if (d.pk16) return precond32s<TR, __half>(m, d.pk16, src, dst, s);
    if (d.pk32) return precond32s<TR, float>(m, d.pk32, src, dst, s);
    if (d.P16)   // FP16 factors (ilu_fp16), FP32 arithmetic
        return precond_t<TR, float, float, __half>(m, d.P16, d.alpha16, d.ex16, d.ey16, src, dst, m->wk.t2_32,
                                                   m->wk.t3_32, m->wk.r32, s, {d.alr16, d.exr16, d.eyr16, d.bdg16});
    return precond_t<TR, float, float>(m, d.P32, d.alpha32, d.ex32, d.ey32, src, dst, m->wk.t2_32, m->wk.t3_32,
                                       m->wk.r32, s, {d.alr32, d.exr32, d.eyr32, d.bdg32});
}

// The control kernels' words (any active, any running system) into the pinned
// host flags (no synchronisation).
gks_status enqueue_flags(gks_mesh *m, cudaStream_t s)
{
    GKS_CUDA(cudaMemcpyAsync(m->wk.h_flags, m->wk.flags, sizeof(int32_t) * 2, cudaMemcpyDeviceToHost, s));
    return GKS_OK;
}

// Add what the device-controlled solves ran since the last call (counters
// already copied to h_ctr, stream synchronised) to the launch and work totals.
void take_counters(gks_mesh *m)
{
    SolveGraphs &g = *m->graphs;
    for (int q = 0; q < kCtrLen; ++q) {
        const int64_t d = g.h_ctr[q] - g.ctr_seen[q];
        g.ctr_seen[q] = g.h_ctr[q];
        if (q < kCtrCycles && d > 0) {
            if (q < (int)g.whole_iter_launches.size()) g_launches.fetch_add(d * g.whole_iter_launches[q]);
            m->prof.arnoldi += d;
            m->prof.precond += d;
            m->prof.arnoldi_jsum += d * (q + 1);
        } else if (q == kCtrCycles && d > 0) {
            g_launches.fetch_add(d * g.whole_cycle_launches);
            m->prof.residuals += d;
        } else if (q == kCtrRun && d > 0) {
            // loops of the step-loop graph: their kernels outside the solve's
            // cycles, and the first residual of each loop's solve
            g_launches.fetch_add(d * g.run_loop_launches);
            m->prof.residuals += d;
        }
    }
}

// Graphs are used unless disabled or the profiler (events between kernels) is on;
// a change of a knob baked into the captured kernel arguments drops them.
bool prepare_graphs(gks_mesh *m)
{
    if (m->cfg.no_graphs == 1 || m->prof.mask) return false;
    if (!m->graphs) m->graphs = new SolveGraphs;
    SolveGraphs &g = *m->graphs;
    if (g.disabled) return false;
    const gks_config &c = m->cfg;
    if (g.sweeps != c.ilu_sweeps || g.sweeps_bwd != c.ilu_sweeps_bwd || g.fuse != c.ilu_fuse_first ||
        g.pairs != c.ilu_sweep_pairs || g.spmv_dots != c.spmv_dots ||
        g.precond != c.precond ||
        g.maxit != c.gmres_maxit || g.eta != c.inner_rtol ||
        g.rtol != c.gmres_rtol || (int)g.iter.size() != m->wk.m) {
        if (g.whole || g.run) flush_solve_counters(m);
        destroy_graph_execs(&g);
        g.sweeps = c.ilu_sweeps;
        g.sweeps_bwd = c.ilu_sweeps_bwd;
        g.fuse = c.ilu_fuse_first;
        g.pairs = c.ilu_sweep_pairs;
        g.spmv_dots = c.spmv_dots;
        g.precond = c.precond;
        g.maxit = c.gmres_maxit;
        g.eta = c.inner_rtol;
        g.rtol = c.gmres_rtol;
        g.iter.assign(m->wk.m, nullptr);
        g.iter_launches.assign(m->wk.m, 0);
    }
    return true;
}

// Capture enq(stream) into *exec on the private stream; *nl = kernels captured.
template <typename F>
gks_status capture_part(gks_mesh *m, cudaGraphExec_t *exec, int64_t *nl, F &&enq)
{
    SolveGraphs &g = *m->graphs;
    if (!g.cap) GKS_CUDA(cudaStreamCreateWithFlags(&g.cap, cudaStreamNonBlocking));
    const int64_t l0 = g_launches.load();
    GKS_CUDA(cudaStreamBeginCapture(g.cap, cudaStreamCaptureModeThreadLocal));
    const gks_status st = enq(g.cap);
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamEndCapture(g.cap, &graph);
    const int64_t n = g_launches.load() - l0;
    g_launches.fetch_sub(n, std::memory_order_relaxed);   // captured, not run
    if (st != GKS_OK || e != cudaSuccess || !graph) {
        if (graph) cudaGraphDestroy(graph);
        cudaGetLastError();
        return st != GKS_OK ? st : GKS_ECUDA;
    }
    e = cudaGraphInstantiate(exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) {
        *exec = nullptr;
        cudaGetLastError();
        return GKS_ECUDA;
    }
    *nl = n;
    return GKS_OK;
}

// Run one part of the solve on s and wait for its host flags: a replay of its
// graph (captured on first use), or the launches themselves.
template <typename F>
gks_status run_part(gks_mesh *m, bool use_graph, cudaGraphExec_t *exec, int64_t *nl, cudaStream_t s, F &&enq)
{
    use_graph = use_graph && !m->graphs->disabled;
    if (use_graph && !*exec && capture_part(m, exec, nl, enq) != GKS_OK) {
        m->graphs->disabled = true;                   // fall back to direct launches for good
        use_graph = false;
    }
    if (use_graph) {
        GKS_CUDA(cudaGraphLaunch(*exec, s));
        g_launches.fetch_add(*nl, std::memory_order_relaxed);
    } else {
        const gks_status st = enq(s);
        if (st != GKS_OK) return st;
    }
    GKS_CUDA(cudaStreamSynchronize(s));
    return GKS_OK;
}

// Append enq(stream) to graph g after the nodes deps[0..nd) by capture on the
// private stream; *sink = the last captured node, *nl = kernels captured.
template <typename F>
gks_status capture_into(gks_mesh *m, cudaGraph_t g, const cudaGraphNode_t *deps, size_t nd, cudaGraphNode_t *sink,
                        int64_t *nl, F &&enq)
{
    SolveGraphs &G = *m->graphs;
    if (!G.cap) GKS_CUDA(cudaStreamCreateWithFlags(&G.cap, cudaStreamNonBlocking));
    const int64_t l0 = g_launches.load();
    GKS_CUDA(cudaStreamBeginCaptureToGraph(G.cap, g, deps, nullptr, nd, cudaStreamCaptureModeThreadLocal));
    const gks_status st = enq(G.cap);
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    const cudaGraphNode_t *tail = nullptr;
    size_t nt = 0;
    const cudaError_t e = cudaStreamGetCaptureInfo(G.cap, &cs, nullptr, nullptr, &tail, nullptr, &nt);
    const cudaGraphNode_t last = (e == cudaSuccess && nt == 1) ? tail[0] : nullptr;
    cudaGraph_t out = nullptr;
    const cudaError_t e2 = cudaStreamEndCapture(G.cap, &out);
    const int64_t n = g_launches.load() - l0;
    g_launches.fetch_sub(n, std::memory_order_relaxed);   // captured, not run
    if (st != GKS_OK || e != cudaSuccess || e2 != cudaSuccess || !last) {
        cudaGetLastError();
        return st != GKS_OK ? st : GKS_ECUDA;
    }
    *sink = last;
    *nl = n;
    return GKS_OK;
}

// Add a conditional node (if / while, one body) on handle h after dep.
gks_status add_cond(cudaGraph_t g, cudaGraphNode_t dep, cudaGraphConditionalHandle h,
                    cudaGraphConditionalNodeType type, cudaGraphNode_t *node, cudaGraph_t *body)
{
    cudaGraphNodeParams p = {};
    p.type = cudaGraphNodeTypeConditional;
    p.conditional.handle = h;
    p.conditional.type = type;
    p.conditional.size = 1;
    GKS_CUDA(cudaGraphAddNode(node, g, &dep, nullptr, 1, &p));
    *body = p.conditional.phGraph_out[0];
    return GKS_OK;
}

// The device counters of the device-controlled graphs (allocated once per handle).
gks_status ensure_counters(gks_mesh *m, cudaStream_t s)
{
    SolveGraphs &G = *m->graphs;
    if (G.ctr) return GKS_OK;
    GKS_CUDA(cudaMalloc(&G.ctr, sizeof(int64_t) * kCtrLen));
    GKS_CUDA(cudaMallocHost(&G.h_ctr, sizeof(int64_t) * kCtrLen));
    GKS_CUDA(cudaMemsetAsync(G.ctr, 0, sizeof(int64_t) * kCtrLen, s));
    G.ctr_seen.assign(kCtrLen, 0);
    return GKS_OK;
}

// A device-controlled solve built as part of a larger graph: into g after dep
// (NULL: with no dependency); sink receives its last node, launches the kernels
// that run once per solve (the start part and what follows the cycle loop).
struct SolveEmbed {
    cudaGraph_t g = nullptr;
    cudaGraphNode_t dep = nullptr;
    cudaGraphNode_t sink = nullptr;
    int64_t launches = 0;
};

// The device-controlled solve as one executable graph (or, with emb, as nodes
// of the caller's graph):
//   start; c = any active
//   while (c) { count the cycle; Arnoldi 0; i_1 = any running
//               if (i_1) { Arnoldi 1; ... if (i_{m-1}) { Arnoldi m-1 } }
//               restart; c = any active (and within the cycle limit) }
// (a cycle starts with every active system running).  The conditions replace the
// host flags of the per-part graphs; those of an index are only evaluated once
// the one before it has run.
template <typename SB, typename IB, typename RB>
gks_status build_whole(gks_mesh *m, cudaStream_t s, SB &&start_body, IB &&iter_body, RB &&restart_body,
                       SolveEmbed *emb = nullptr)
{
    SolveGraphs &G = *m->graphs;
    Work &k = m->wk;
    const int mm = k.m;
    const int64_t limit = (int64_t)m->cfg.gmres_maxit + 1;
    if (const gks_status r = ensure_counters(m, s); r != GKS_OK) return r;
    int64_t *ctr = G.ctr;
    uint32_t *ticket = reinterpret_cast<uint32_t *>(k.flags + 3);
    cudaGraph_t top = emb ? emb->g : nullptr;
    if (!emb) GKS_CUDA(cudaGraphCreate(&top, 0));
    const size_t ndep = emb && emb->dep ? 1 : 0;
    gks_status st = GKS_OK;
    std::vector<int64_t> nl_iter(mm, 0);
    int64_t nl_start = 0, nl_restart = 0;
    do {
        cudaGraphConditionalHandle h_outer, h_next = 0;
        if (cudaGraphConditionalHandleCreate(&h_outer, top, 0, 0) != cudaSuccess) { st = GKS_ECUDA; break; }
        cudaGraphNode_t sink, wnode, inode;
        cudaGraph_t wbody, ibody;
        st = capture_into(m, top, ndep ? &emb->dep : nullptr, ndep, &sink, &nl_start, [&](cudaStream_t q) -> gks_status {
            return start_body(q, Cond{h_outer, ctr, 0, nullptr, ticket, 1, -1, 1});
        });
        if (st != GKS_OK || (st = add_cond(top, sink, h_outer, cudaGraphCondTypeWhile, &wnode, &wbody)) != GKS_OK)
            break;
        ibody = wbody;
        for (int j = 0; j < mm && st == GKS_OK; ++j) {
            const bool more = j + 1 < mm;
            if (more && cudaGraphConditionalHandleCreate(&h_next, ibody, 0, 0) != cudaSuccess) {
                st = GKS_ECUDA;
                break;
            }
            st = capture_into(m, ibody, nullptr, 0, &sink, &nl_iter[j], [&](cudaStream_t q) -> gks_status {
                if (j == 0) {
                    k_cycle_count<<<1, 32, 0, q>>>(ctr);
                    note_launch();
                }
                return iter_body(q, j, Cond{h_next, ctr, 0, nullptr, ticket, more ? 1 : 0, j, 0});
            });
            if (st == GKS_OK && more) {
                cudaGraph_t next;
                st = add_cond(ibody, sink, h_next, cudaGraphCondTypeIf, &inode, &next);
                ibody = next;
            } else {
                inode = sink;
            }
            if (st == GKS_OK && j == 0) {
                // the rest of the loop's body after the first index (and those nested behind it)
                cudaGraphNode_t tail;
                st = capture_into(m, wbody, &inode, 1, &tail, &nl_restart, [&](cudaStream_t q) -> gks_status {
                    return restart_body(q, Cond{h_outer, ctr, limit, nullptr, ticket, 1, -1, 0});
                });
            }
        }
        if (st != GKS_OK) break;
        if (emb) {
            emb->sink = wnode;
        } else if (cudaGraphInstantiate(&G.whole, top, 0) != cudaSuccess) {
            G.whole = nullptr;
            st = GKS_ECUDA;
        }
    } while (false);
    if (!emb) cudaGraphDestroy(top);
    cudaGetLastError();
    if (st != GKS_OK) return st;
    G.whole_start_launches = nl_start;
    nl_iter[0] -= 1;                                     // k_cycle_count: counted with the cycle
    G.whole_cycle_launches = nl_restart + 1;
    G.whole_iter_launches = nl_iter;
    return GKS_OK;
}

// part[k][v][blk] = partial <V_k, w>, k <= j, per cell block
template <typename TB>
gks_status dots(gks_mesh *m, const TB *V, const TB *w, int j, double *part, cudaStream_t s)
{
    const int64_t nblk = m->wk.nblk;
    if constexpr (std::is_same_v<TB, float>) {
        k_dots32<<<dim3((unsigned)nblk, (unsigned)(j + 1)), kBlock, 0, s>>>(m->d.T, V, w, part);
    } else {
        const dim3 g((unsigned)(j + 1), (unsigned)std::min<int64_t>(nblk, kDotMaxTiles));
        k_dots<TB><<<g, kDotThreads, 0, s>>>(m->d.T, nblk, V, w, part);
    }
    note_launch();
    GKS_CUDA(cudaGetLastError());
    return GKS_OK;
}

inline unsigned sblocks(int n) { return (unsigned)((n + 127) / 128); }

}  // namespace

// Solve the CLS systems of every case for the right-hand sides built from
// m->wk.w; the solutions (and warm starts) are m->wk.x.  GMRES cycles of all
// systems run in lockstep: every launch covers all cases, and per-system masks
// stop the systems that have converged.
// The whole solve with the Krylov basis stored as TB (double, or float in the
// mixed mode with basis_fp32).  With emb the device-controlled solve and its
// closing kernel are built into the caller's graph instead of run.
template <typename TB>
gks_status cls_solve_t(gks_mesh *m, TB *V, cudaStream_t s, int32_t *iters, double *relres, int32_t *converged,
                       bool acc, SolveEmbed *emb = nullptr)
{
    DeviceMesh &d = m->d;
    Work &k = m->wk;
    const int64_t T = d.T;
    const int mm = k.m;
    const int ps = mm + 2;
    const int ns = k.ns;
    const unsigned nb = (unsigned)k.nblk;
    const double rtol = m->cfg.gmres_rtol;
    const int maxit = m->cfg.gmres_maxit;
    const int64_t vs = (int64_t)NX * T;
    const bool mixed = m->cfg.precision == GKS_MIXED;
    // mixed precision: an inner GMRES cycle (FP32 operator and ILU) stops once its
    // residual estimate has dropped by inner_rtol; the FP64 residual of the next
    // refinement sweep then measures the true error
    const double eta = mixed ? m->cfg.inner_rtol : 0.0;
    gks_status st;
    // the FP64 solve of the per-cell equations: a thread per cell and variable
    // (gks_solve64.cuh), C64 cells per thread, rs partial-sum rows per cell block
    const int C64 = k.c64;
    if (C64 && mm > 45) {
        if ((st = solve64_shared_limit()) != GKS_OK) return st;
    }

    // FP32 basis: first basis vector scaled by a power of two; exponents per
    // system, [current cycle][next residual]
    int32_t *sx = std::is_same<TB, float>::value ? k.sexp : nullptr;
    const int32_t *sxn = sx ? sx + ns : nullptr;
    // V_0 = 2^-e (b - K x) and partial |V_0|^2: double-FP32 arithmetic into the
    // FP32 basis when the operator has FP32 pairs, FP64 arithmetic otherwise
    // operator applications y = K x (mode 0) or the FP64 residual (mode 1); the
    // global normal equations' variant when the mesh has reverse slots
    auto spmv64 = [&](cudaStream_t q, const double *xs, TB *y, int mode, const double *bb, const int32_t *se) {
        if (d.alr)
            k_spmv<double, double, TB, true><<<nb, kBlock, 0, q>>>(d, d.D, d.alpha, d.ex, d.ey, xs, y, mode, bb,
                                                                   k.part, se, d.alr, d.exr, d.eyr, d.bdg);
        else
            k_spmv<double, double, TB, false><<<nb, kBlock, 0, q>>>(d, d.D, d.alpha, d.ex, d.ey, xs, y, mode, bb,
                                                                    k.part, se);
    };
    auto spmv32 = [&](cudaStream_t q, const float *xs, TB *y) {
        if (d.alr32)
            k_spmv<float, float, TB, true><<<nb, kBlock, 0, q>>>(d, d.D32, d.alpha32, d.ex32, d.ey32, xs, y, 0,
                                                                 nullptr, nullptr, nullptr, d.alr32, d.exr32,
                                                                 d.eyr32, d.bdg32);
        else
            k_spmv<float, float, TB, false><<<nb, kBlock, 0, q>>>(d, d.D32, d.alpha32, d.ex32, d.ey32, xs, y, 0,
                                                                  nullptr, nullptr);
    };
    // the FP32-basis solve forms b in double-FP32 arithmetic when the weights fit
    const bool rhs_df = std::is_same<TB, float>::value && d.a0p;
    // the FP32 basis with the per-cell equations: the operator kernel also forms
    // the Gram-Schmidt products
    const bool fused_dots = std::is_same<TB, float>::value && !d.alr32 && m->cfg.spmv_dots;
    // partial-sum rows per cell block of the kernels in use
    const int rs64 = C64 ? kRows64 / C64 : 1, rs32 = k.c32 ? kRows64 / k.c32 : 1;
    const int rs_rhs = C64 ? rs64 : (rhs_df ? rs32 : 1);
    const int rs_res = C64 ? rs64 : (std::is_same<TB, float>::value && d.D2 ? kResidRows : 1);
    const int rs = rs64;
    const int32_t *twice = C64 ? k.ctl + kCtlTwice * ns : nullptr;
    auto residual = [&](cudaStream_t q, bool first) -> gks_status {
        const int32_t *act = first ? nullptr : k.ctl + kCtlActive * ns;
        if (C64) {
            solve64_resid(m, reinterpret_cast<double *>(V), act, q);
        } else if (std::is_same<TB, float>::value && d.D2) {
            float *v0 = reinterpret_cast<float *>(V);
            const float4 *d2 = reinterpret_cast<const float4 *>(d.D2);
            if (d.SR2)
                k_resid_df<true><<<rs_res * nb, kBlock, 0, q>>>(d, d2, k.x, v0, k.b, k.part, sxn, act,
                                                                   reinterpret_cast<const float4 *>(d.SR2));
            else
                k_resid_df<false><<<rs_res * nb, kBlock, 0, q>>>(d, d2, k.x, v0, k.b, k.part, sxn, act);
            note_launch();
        } else {
            spmv64(q, k.x, V, 1, k.b, sxn);
            note_launch();
        }
        GKS_CUDA(cudaGetLastError());
        return GKS_OK;
    };
    const Krylov kry = {mm, ns, k.H, k.cs, k.sn, k.g, k.y, k.vn, mixed ? k.y32 : nullptr, k.ctl, k.bnorm, k.beta, sx,
                        rtol, eta, maxit};
    auto cycle_begin = [&](cudaStream_t q, int first, const Cond &cd) {
        k_cycle_begin<<<ns, kReduceThreads, 0, q>>>(kry, k.part, rs_res * (int64_t)nb, d.case_blk, rs_res,
                                                        k.hcol + 1, ps, k.done, first, cd);
        note_launch();
    };
    // the three fixed launch sequences (the per-part graphs end each with the
    // flags for the host; in the whole-solve graph their last kernels set the
    // conditions)
    uint32_t *ticket = reinterpret_cast<uint32_t *>(k.flags + 3);
    const Cond host_active = {0, nullptr, 0, k.flags, ticket, 0, -1, 0};
    const Cond host_running = {0, nullptr, 0, k.flags + 1, ticket, 0, -1, 0};
    auto start_body = [&](cudaStream_t q, const Cond &cd) -> gks_status {
        int slot = prof_start(m, kProfCtl, q);
        if (m->cfg.precond == GKS_PC_ILU_EXACT) {
            k_sf_begin<<<1, 32, 0, q>>>(k.sf_ctl, 1);      // a new solve: clear the wait error
            note_launch();
        }
        if (C64) {
            solve64_rhs(m, q);
        } else if (rhs_df) {
            solve32_rhs(m, q);
        } else {
            k_rhs<<<nb, kBlock, 0, q>>>(d, k.w, k.b, k.part);
            note_launch();
        }
        if (sx) {
            // the FP32 basis stores its first vector scaled by a power of two 2^-e
            k_sigma<<<ns, kReduceThreads, 0, q>>>(k.part, rs_rhs * (int64_t)nb, d.case_blk, rs_rhs, k.hcol + 1,
                                                      ps, k.bnorm, k.sexp, ns);
            note_launch();
        }
        prof_stop(m, slot, q);
        slot = prof_start(m, kProfResid, q);
        // residual r = b - K x, written straight into the basis slot V_0 (v_0 = V_0 / beta)
        if (const gks_status r = residual(q, true); r != GKS_OK) return r;
        prof_stop(m, slot, q);
        slot = prof_start(m, kProfCtl, q);
        cycle_begin(q, 1, cd);
        k_zero_trivial<<<nb, kBlock, 0, q>>>(d, k.x, k.bnorm); note_launch();
        prof_stop(m, slot, q);
        GKS_CUDA(cudaGetLastError());
        return GKS_OK;
    };
    auto iter_body = [&](cudaStream_t q, int j, const Cond &cd) -> gks_status {
        TB *vj = V + j * vs, *vj1 = V + (j + 1) * vs;
        gks_status st;
        int slot = prof_start(m, kProfIlu, q);
        // Z_j = M^{-1} V_j, kept for the update of x at the end of the cycle
        if ((st = mixed ? precond32(m, vj, k.Z32 + j * vs, q) : precond(m, vj, k.Z + j * vs, q)) != GKS_OK)
            return st;
        prof_stop(m, slot, q);
        slot = prof_start(m, kProfSpmv, q);
        if (fused_dots) {
            solve32_apply_dots(m, k.Z32 + j * vs, reinterpret_cast<const float *>(V), reinterpret_cast<float *>(vj1),
                               j, q);
        } else if (mixed) {
            spmv32(q, k.Z32 + j * vs, vj1);
        } else if (C64) {
            // V_{j+1} = K Z_j - V_j with the first Gram-Schmidt products
            solve64_apply_dots(m, k.Z + j * vs, reinterpret_cast<const double *>(V), reinterpret_cast<double *>(vj1),
                               j, q);
        } else {
            spmv64(q, k.Z + j * vs, vj1, 0, nullptr, nullptr);
        }
        if (!C64 && !fused_dots) note_launch();
        prof_stop(m, slot, q);
        slot = prof_start(m, kProfOrth, q);
        // classical Gram-Schmidt: twice in FP64 mode (per-cell equations: a second
        // time where it is needed, see gks_solve64.cuh); once in the mixed mode, whose
        // cycles only reduce the residual by inner_rtol before an FP64 restart
        if (!fused_dots && !C64 && (st = dots<TB>(m, V, vj1, j, k.part, q)) != GKS_OK) return st;
        // (C64, fused_dots: and |w|^2)
        k_reduce<<<dim3(j + (C64 || fused_dots ? 2 : 1), ns), kReduceThreads, 0, q>>>(
            k.part, rs * (int64_t)nb, d.case_blk, rs, k.hcol, ps, k.vn, mm + 1, k.hco, ps, j + 1, nullptr,
            k.ctl + kCtlRunning * ns, C64 || fused_dots ? k.ctl + kCtlRan * ns : nullptr);
        note_launch();
        if (C64) {
            solve64_update(m, kry, reinterpret_cast<const double *>(V), reinterpret_cast<double *>(vj1), j, ps, cd, q);
        } else if (fused_dots) {
            solve32_update(m, kry, reinterpret_cast<const float *>(V), reinterpret_cast<float *>(vj1), j, ps, cd, q);
            prof_stop(m, slot, q);
            GKS_CUDA(cudaGetLastError());
            return GKS_OK;
        } else {
            launch_orth_update<TB>(d, nb, q, V, vj1, j, k.hco, ps, k.ctl, ns, k.part, mixed ? 1 : 0);
            note_launch();
        }
        // small meshes: the second pass inside the last kernel
        const bool solo = C64 && T <= kSolo64;
        if (!mixed && !solo) {
            // the second pass (the systems flagged in twice)
            if (!C64 && (st = dots<TB>(m, V, vj1, j, k.part, q)) != GKS_OK) return st;
            k_reduce<<<dim3(j + 1, ns), kReduceThreads, 0, q>>>(k.part, rs * (int64_t)nb, d.case_blk, rs, k.y, mm, k.vn,
                                                                 mm + 1, k.hco, ps, j + 1, twice,
                                                                 nullptr, nullptr);
            note_launch();
            if (C64) {
                solve64_update_norm(m, reinterpret_cast<const double *>(V), reinterpret_cast<double *>(vj1), j, ps, q);
            } else {
                launch_orth_update<TB>(d, nb, q, V, vj1, j, k.hco, ps, k.ctl, ns, k.part, 1);
                note_launch();
            }
        }
        // |V_{j+1}| and the Givens step of every system (and the end of a single mesh's cycle);
        // C64: of the systems with a second pass, the index is counted already
        Cond ce = cd;
        if (C64) ce.slot = -1;
        k_arnoldi_end<<<ns, kReduceThreads, 0, q>>>(kry, k.part, rs * (int64_t)nb, d.case_blk, rs, j, k.hcol, ps,
                                                        mixed ? nullptr : k.y, mm, twice, C64 ? 1.0 : 0.0,
                                                        Solo{reinterpret_cast<const double *>(V),
                                                             solo ? reinterpret_cast<double *>(vj1) : nullptr, T},
                                                        ce);
        note_launch();
        prof_stop(m, slot, q);
        GKS_CUDA(cudaGetLastError());
        return GKS_OK;
    };
    auto restart_body = [&](cudaStream_t q, const Cond &cd) -> gks_status {
        int slot = prof_start(m, kProfCorr, q);
        if (m->n_case > 1) {
            k_cycle_solve<<<(ns + kSolveWarps - 1) / kSolveWarps, 32 * kSolveWarps, 0, q>>>(kry);
            note_launch();
        }
        if (mixed)
            k_combine32<<<NV * nb, kBlock, 0, q>>>(d, k.Z32, k.y32, mm, k.ctl, ns, k.x, sx);
        else if (C64)
            k64_combine<<<(unsigned)((T + 31) / 32), kW64, 0, q>>>(T, d.blk_case, k.Z, k.y, mm, k.ctl + kCtlJv * ns,
                                                                  k.x);
        else
            k_combine_z<<<dim3(nb, NV), kBlock, 0, q>>>(d, k.Z, k.y, mm, k.ctl, ns, k.x);
        note_launch();
        prof_stop(m, slot, q);
        slot = prof_start(m, kProfResid, q);
        if (const gks_status r = residual(q, false); r != GKS_OK) return r;
        prof_stop(m, slot, q);
        slot = prof_start(m, kProfCtl, q);
        cycle_begin(q, 0, cd);
        prof_stop(m, slot, q);
        GKS_CUDA(cudaGetLastError());
        return GKS_OK;
    };
    auto with_flags = [&](cudaStream_t q, gks_status r) { return r != GKS_OK ? r : enqueue_flags(m, q); };
    auto start_part = [&](cudaStream_t q) { return with_flags(q, start_body(q, host_active)); };
    auto iter_part = [&](cudaStream_t q, int j) { return with_flags(q, iter_body(q, j, host_running)); };
    auto restart_part = [&](cudaStream_t q) { return with_flags(q, restart_body(q, host_active)); };

    const bool use_graph = prepare_graphs(m);
    SolveGraphs *G = use_graph ? m->graphs : nullptr;
    bool whole = false;
    // the whole-solve graph holds every Arnoldi index up front: with the
    // level-by-level exact ILU (two launches per level) that is too many nodes
    // on large meshes, whose per-step graphs are built only for the indices used
    const bool few_nodes = m->cfg.precond != GKS_PC_ILU_LEVELS || m->lvl_lo_ptr.size() + m->lvl_up_ptr.size() <= 256;
    if (emb) {
        if (!G || !few_nodes || G->disabled || m->cfg.no_graphs != 0) return GKS_EINVAL;
        if ((st = build_whole(m, s, start_body, iter_body, restart_body, emb)) != GKS_OK) return st;
        int64_t nl = 0;
        st = capture_into(m, emb->g, &emb->sink, 1, &emb->sink, &nl, [&](cudaStream_t q) -> gks_status {
            k_mark_noconv<<<sblocks(ns), 128, 0, q>>>(k.bnorm, k.beta, k.done, ns, rtol, k.status, k.nsolve,
                                                      m->cfg.precond == GKS_PC_ILU_EXACT ? k.sf_ctl + 3 : nullptr,
                                                      k.ctl + kCtlIters * ns, k.iters_acc);
            note_launch();
            GKS_CUDA(cudaGetLastError());
            return GKS_OK;
        });
        emb->launches = G->whole_start_launches + nl;
        return st;
    }
    if (G && few_nodes && !G->disabled && !G->whole_failed && m->cfg.no_graphs != 2) {
        if (!G->whole && build_whole(m, s, start_body, iter_body, restart_body) != GKS_OK) {
            G->whole_failed = true;                     // per-part graphs with host control from now on
            cudaGetLastError();
        }
        whole = G->whole != nullptr;
    }
    cudaGraphExec_t none = nullptr;
    int64_t none_n = 0;
    if (whole) {
        GKS_CUDA(cudaGraphLaunch(G->whole, s));
        g_launches.fetch_add(G->whole_start_launches, std::memory_order_relaxed);
        m->prof.residuals += 1;
    } else {
        if ((st = run_part(m, use_graph, G ? &G->start : &none, G ? &G->start_launches : &none_n, s,
                           start_part)) != GKS_OK)
            return st;
        m->prof.residuals += 1;
    }
    while (!whole && k.h_flags[0]) {
        for (int j = 0; j < mm; ++j) {
            m->prof.precond += 1;
            m->prof.arnoldi += 1;
            m->prof.arnoldi_jsum += j + 1;
            st = run_part(m, use_graph, G ? &G->iter[j] : &none, G ? &G->iter_launches[j] : &none_n, s,
                          [&](cudaStream_t q) { return iter_part(q, j); });
            if (st != GKS_OK) return st;
            if (!k.h_flags[1]) break;
        }
        if ((st = run_part(m, use_graph, G ? &G->restart : &none, G ? &G->restart_launches : &none_n, s,
                           restart_part)) != GKS_OK)
            return st;
        m->prof.residuals += 1;
    }
    k_mark_noconv<<<sblocks(ns), 128, 0, s>>>(k.bnorm, k.beta, k.done, ns, rtol, k.status, k.nsolve,
                                              m->cfg.precond == GKS_PC_ILU_EXACT ? k.sf_ctl + 3 : nullptr,
                                              k.ctl + kCtlIters * ns, acc ? k.iters_acc : nullptr);
    note_launch();
    if (iters || relres || converged) {
        std::vector<int32_t> it(ns);
        std::vector<double> be(ns), bn(ns);
        GKS_CUDA(cudaMemcpyAsync(it.data(), k.ctl + kCtlIters * ns, sizeof(int32_t) * ns, cudaMemcpyDeviceToHost, s));
        GKS_CUDA(cudaMemcpyAsync(be.data(), k.beta, sizeof(double) * ns, cudaMemcpyDeviceToHost, s));
        GKS_CUDA(cudaMemcpyAsync(bn.data(), k.bnorm, sizeof(double) * ns, cudaMemcpyDeviceToHost, s));
        if (whole)
            GKS_CUDA(cudaMemcpyAsync(G->h_ctr, G->ctr, sizeof(int64_t) * kCtrLen, cudaMemcpyDeviceToHost, s));
        GKS_CUDA(cudaStreamSynchronize(s));
        if (whole) take_counters(m);
        int32_t conv = 1;
        for (int q = 0; q < ns; ++q) {
            const double rr = bn[q] > 0.0 ? be[q] / bn[q] : 0.0;
            if (iters) iters[q] = it[q];
            if (relres) relres[q] = rr;
            if (rr > rtol) conv = 0;
        }
        if (converged) *converged = conv;
    }
    return GKS_OK;
}

namespace {

// the extrapolated warm start of the next solve (if configured)
gks_status launch_warm(gks_mesh *m, cudaStream_t s)
{
    Work &k = m->wk;
    if (!m->cfg.warm_extrap) return GKS_OK;
    const int slot = prof_start(m, kProfCtl, s);
    k_warm<<<dim3((unsigned)k.nblk, NV), kBlock, 0, s>>>(m->d, k.x, k.x_prev, k.x_prev2, k.done, k.nsolve, m->cfg.warm_extrap);
    note_launch();
    prof_stop(m, slot, s);
    GKS_CUDA(cudaGetLastError());
    return GKS_OK;
}

// The step loop as a graph (see run_graph_launch):
//   c = any case not done and a loop limit above 0
//   while (c) { CFL step, clipped to the end times; warm start;
//               the device-controlled solve; solve count and convergence marks;
//               iteration sums; limiter; flux; update; per-case clocks;
//               c = any case not done and the loops of this launch below the limit }
gks_status build_run(gks_mesh *m, cudaStream_t s)
{
    SolveGraphs &G = *m->graphs;
    Work &k = m->wk;
    const int n = m->n_case;
    if (const gks_status r = ensure_counters(m, s); r != GKS_OK) return r;
    if (!G.h_run) GKS_CUDA(cudaMallocHost(&G.h_run, sizeof(int64_t)));
    int64_t *ctr = G.ctr;
    cudaGraph_t top = nullptr;
    GKS_CUDA(cudaGraphCreate(&top, 0));
    gks_status st = GKS_OK;
    int64_t nl_entry = 0, nl_a = 0, nl_b = 0;
    SolveEmbed e;
    do {
        cudaGraphConditionalHandle h;
        if (cudaGraphConditionalHandleCreate(&h, top, 0, 0) != cudaSuccess) { st = GKS_ECUDA; break; }
        cudaGraphNode_t sink, wnode;
        cudaGraph_t body;
        st = capture_into(m, top, nullptr, 0, &sink, &nl_entry, [&](cudaStream_t q) -> gks_status {
            k_run_cond<<<1, kBlock, 0, q>>>(k.done, n, k.run_ctl, ctr, h, 1); note_launch();
            return GKS_OK;
        });
        if (st != GKS_OK || (st = add_cond(top, sink, h, cudaGraphCondTypeWhile, &wnode, &body)) != GKS_OK) break;
        st = capture_into(m, body, nullptr, 0, &sink, &nl_a, [&](cudaStream_t q) -> gks_status {
            gks_status r;
            if ((r = launch_cfl_dt(m, k.w, k.dt, q, true)) != GKS_OK) return r;
            return launch_warm(m, q);
        });
        if (st != GKS_OK) break;
        e.g = body;
        e.dep = sink;
        st = k.V32 ? cls_solve_t<float>(m, k.V32, s, nullptr, nullptr, nullptr, true, &e)
                   : cls_solve_t<double>(m, k.V, s, nullptr, nullptr, nullptr, true, &e);
        if (st != GKS_OK) break;
        st = capture_into(m, body, &e.sink, 1, &sink, &nl_b, [&](cudaStream_t q) -> gks_status {
            gks_status r;
            if (m->cfg.limiter && (r = launch_limiter(m, k.w, k.x, q)) != GKS_OK) return r;
            if ((r = launch_flux(m, k.w, m->cfg.limiter ? k.xl : k.x, 0.0, k.dt, k.flux, q)) != GKS_OK) return r;
            if ((r = launch_update(m, k.w, k.flux, q)) != GKS_OK) return r;
            if ((r = launch_after_step(m, q)) != GKS_OK) return r;
            k_run_cond<<<1, kBlock, 0, q>>>(k.done, n, k.run_ctl, ctr, h, 0); note_launch();
            GKS_CUDA(cudaGetLastError());
            return GKS_OK;
        });
        if (st != GKS_OK) break;
        if (cudaGraphInstantiate(&G.run, top, 0) != cudaSuccess) {
            G.run = nullptr;
            st = GKS_ECUDA;
        }
    } while (false);
    cudaGraphDestroy(top);
    cudaGetLastError();
    if (st != GKS_OK) return st;
    G.run_loop_launches = nl_a + e.launches + nl_b;
    G.run_cfg = m->cfg;
    return GKS_OK;
}

}  // namespace

gks_status cls_solve(gks_mesh *m, cudaStream_t s, int32_t *iters, double *relres, int32_t *converged, bool acc)
{
    Work &k = m->wk;
    if (const gks_status st = launch_warm(m, s); st != GKS_OK) return st;
    return k.V32 ? cls_solve_t<float>(m, k.V32, s, iters, relres, converged, acc)
                 : cls_solve_t<double>(m, k.V, s, iters, relres, converged, acc);
}

void plan_solve(gks_mesh *m, int *rows)
{
    const int c = cells64(m->d.T);
    if (m->cfg.precision == GKS_FP64) m->wk.c64 = c;
    else m->wk.c32 = c;
    // the mixed path's residual has rows of its own
    *rows = std::max(kRows64 / c, m->cfg.precision == GKS_MIXED ? kResidRows : 1);
}

gks_status launch_pack(gks_mesh *m)
{
    const DeviceMesh &d = m->d;
    if (d.T == 0) return GKS_OK;
    const unsigned g = nblocks(d.T);
    if (d.off) {
        k64_off<<<g, kBlock>>>(d.T, d.alpha, d.ex, d.ey, d.off);
        note_launch();
    }
    if (d.w64) {
        k64_products<<<g, kBlock>>>(d.T, d.P, d.off, d.w64);
        note_launch();
    }
    if (d.op32) {
        k32_pack_op<<<g, kBlock>>>(d.T, d.D32, d.alpha32, d.ex32, d.ey32, reinterpret_cast<float4 *>(d.op32));
        note_launch();
    }
    if (d.pk16) {
        k32_pack<__half><<<g, kBlock>>>(d.T, d.P16, d.alpha16, d.ex16, d.ey16, d.pk16);
        note_launch();
    } else if (d.pk32) {
        k32_pack<float><<<g, kBlock>>>(d.T, d.P32, d.alpha32, d.ex32, d.ey32, d.pk32);
        note_launch();
    }
    GKS_CUDA(cudaGetLastError());
    return GKS_OK;
}

gks_status run_graph_launch(gks_mesh *m, int64_t max_steps, cudaStream_t s, bool *used)
{
    *used = false;
    if (m->cfg.no_graphs != 0 || !prepare_graphs(m)) return GKS_OK;
    SolveGraphs &G = *m->graphs;
    if (G.run_failed || G.disabled) return GKS_OK;
    if (G.run && std::memcmp(&G.run_cfg, &m->cfg, sizeof(gks_config)) != 0) {
        flush_solve_counters(m);                   // counted with the old graph's launch numbers
        cudaGraphExecDestroy(G.run);
        G.run = nullptr;
    }
    if (!G.run && build_run(m, s) != GKS_OK) {
        G.run_failed = true;                       // the host loop from now on
        cudaGetLastError();
        return GKS_OK;
    }
    *G.h_run = max_steps;
    GKS_CUDA(cudaMemcpyAsync(m->wk.run_ctl + 1, G.h_run, sizeof(int64_t), cudaMemcpyHostToDevice, s));
    GKS_CUDA(cudaGraphLaunch(G.run, s));
    g_launches.fetch_add(1, std::memory_order_relaxed);   // the entry condition
    *used = true;
    return GKS_OK;
}

void flush_solve_counters(gks_mesh *m)
{
    SolveGraphs *g = m->graphs;
    if (!g || !g->ctr) return;
    if (cudaDeviceSynchronize() == cudaSuccess &&
        cudaMemcpy(g->h_ctr, g->ctr, sizeof(int64_t) * kCtrLen, cudaMemcpyDeviceToHost) == cudaSuccess)
        take_counters(m);
    cudaGetLastError();
}

void destroy_graph_execs(SolveGraphs *g)
{
    for (cudaGraphExec_t &e : g->iter)
        if (e) {
            cudaGraphExecDestroy(e);
            e = nullptr;
        }
    if (g->start) cudaGraphExecDestroy(g->start);
    if (g->restart) cudaGraphExecDestroy(g->restart);
    if (g->whole) cudaGraphExecDestroy(g->whole);
    if (g->run) cudaGraphExecDestroy(g->run);
    g->start = g->restart = g->whole = g->run = nullptr;
}

}  // namespace gks
