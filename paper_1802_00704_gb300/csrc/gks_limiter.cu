// Shock detector and DWBAP limiter on the CLS reconstruction (Sec. III.C).
//
// Reading of Eqs. (34)-(38) used here (the CPU checker of the tests follows the
// same reading, written independently):
//  - detector, Eq. (37): IS_i = sum_j |u_i(r_i) - u_j(r_i)| /
//    (J h_i^{(k_i+1)/2} max(ubar_i, ubar_j)) over the J face neighbours, for the
//    density and for the total energy; the cell is limited unless both are
//    below 1 (Eq. (38));
//  - DWBAP, Eqs. (34)-(36): a derivative of a flagged cell becomes
//    u_0 tan(sum_j omega_j arctan(u_j / u_0)) (0 when u_0 = 0), u_0 the cell's
//    own derivative and u_j the same derivative of neighbour j's polynomial at
//    the cell centroid; omega_j = beta_j / sum beta, beta_j = d_j^{-S(chi)},
//    d_j the mean distance from candidate j's centroid (the cell's own for
//    j = 0) to the cell's interior-face midpoints, S(chi) = 1/(sqrt(chi + 1e-8)
//    + 0.05), chi = standard deviation / mean of the neighbours' pressures;
//    second derivatives (from neighbours with k_j = 2, weights renormalised)
//    and first derivatives, all from the unlimited polynomials;
//  - positivity (not in the paper): a cell is also limited when its unlimited
//    polynomial has rho <= 0 or p <= 0 at one of its face Gauss points; a
//    limited cell whose polynomial still has one keeps its cell average only
//    (all coefficients zero);
//  - characteristic variables (limit_char = 1; Sec. IV.B compares them with the
//    conservative ones): each derivative row is limited in the eigenvector
//    basis of the Euler flux Jacobian at the cell average, along x for d/dx and
//    d2/dx2, y for d/dy and d2/dy2 and the diagonal for d2/dxdy;
//  - robust mode (limiter = 2, not in the paper): a limited cell keeps its
//    cell average only (first order), for contacts with density ratios near
//    10, where the DWBAP polynomials let cell averages turn negative.
//
// FP64 throughout, in two kernels: a thread per cell for the detector and the
// positivity of every cell, which copies the coefficients of a smooth cell and
// lists the others, and a group of lanes per listed cell for the limiter.  An FP64
// instruction holds an SM sub-partition for 33 ns whatever its active lanes, and a
// limited cell's weights and means are some 5,000 of them (80 arctangents and
// divisions, 20 tangents): one flagged cell among a warp's 32 cost as much as 32.
// A limiter call on a 12,000-triangle strip (characteristic variables) went from 260 us
// in one kernel to 21 us for the detector and 30 us for the limiter, a step of the
// 6,400-triangle Sod strip from 0.85 to 0.65 ms.
// The unlimited coefficients stay in x (the warm start of the next CLS solve);
// the limited ones are written to a separate array that the flux kernel reads.
#include <algorithm>
#include <cmath>

#include "gks_internal.h"

namespace gks {
namespace {

// The Euler flux Jacobian's eigenvectors at a conservative state: what does not depend
// on the direction, once per cell.
struct EulerState {
    double u, v, ke, c, ic, H, b1, b2;
};

__device__ __forceinline__ EulerState euler_state(const double *W, double gamma)
{
    EulerState e;
    e.u = W[1] / W[0];
    e.v = W[2] / W[0];
    e.ke = 0.5 * (e.u * e.u + e.v * e.v);
    const double p = (gamma - 1.0) * (W[3] - W[0] * e.ke);
    e.c = sqrt(gamma * p / W[0]);
    e.H = (W[3] + p) / W[0];
    e.b1 = (gamma - 1.0) / (e.c * e.c);
    e.b2 = e.b1 * e.ke;
    e.ic = 1.0 / e.c;
    return e;
}

// Row q of the left eigenvectors (eigenvalues q_n - c, q_n, q_n, q_n + c), and row q of
// the right ones (columns), of the Jacobian along the unit direction (nx, ny).
__device__ __forceinline__ void char_rows(const EulerState &e, int q, double nx, double ny, double *R, double *L)
{
    const double qn = e.u * nx + e.v * ny, qt = -e.u * ny + e.v * nx;
    const double s = q == 0 ? e.ic : -e.ic;
    const double bu = e.b1 * e.u, bv = e.b1 * e.v;
    if (q == 0 || q == 3) {
        L[0] = 0.5 * (e.b2 + qn * s);
        L[1] = -0.5 * (bu + nx * s);
        L[2] = -0.5 * (bv + ny * s);
        L[3] = 0.5 * e.b1;
    } else {
        L[0] = q == 1 ? 1.0 - e.b2 : -qt;
        L[1] = q == 1 ? bu : -ny;
        L[2] = q == 1 ? bv : nx;
        L[3] = q == 1 ? -e.b1 : 0.0;
    }
    const double mid = q == 0 ? 1.0 : (q == 1 ? e.u : (q == 2 ? e.v : e.H));
    const double dif = e.c * (q == 0 ? 0.0 : (q == 1 ? nx : (q == 2 ? ny : qn)));
    R[0] = mid - dif;
    R[1] = q == 3 ? e.ke : mid;
    R[2] = q == 0 ? 0.0 : (q == 1 ? -ny : (q == 2 ? nx : qt));
    R[3] = mid + dif;
}

// u_0 tan(sum_j om_j atan(u_j / u_0)) over the candidates (weight 0: none); the own
// candidate's arctangent is pi/4 (NaN for an infinite u_0, as the quotient is)
__device__ __forceinline__ double biased_mean(const double (&u)[4], const double (&om)[4])
{
    if (u[0] == 0.0) return 0.0;
    double acc = om[0] * 0.78539816339744830962 + (u[0] - u[0]);
#pragma unroll
    for (int j = 1; j < 4; ++j)
        if (om[j] != 0.0) acc += om[j] * atan(u[j] / u[0]);
    return u[0] * tan(acc);
}

// rho > 0 and p > 0 at Gauss point (dx, dy) of a cell, U its averages and c its
// coefficients [variable][5].  p > 0 as 2 rho E > |rho u|^2, which has the same sign
// for rho > 0 without a division (9 instructions), unless rho E nears the range's ends
__device__ __forceinline__ bool physical_at(const double *U, const double (*c)[5], double mxx, double mxy, double myy,
                                            double dx, double dy)
{
    const double hx = 0.5 * (dx * dx - mxx), xy = dx * dy - mxy, hy = 0.5 * (dy * dy - myy);
    double q[4];
#pragma unroll
    for (int v = 0; v < 4; ++v)
        q[v] = U[v] + c[v][0] * dx + c[v][1] * dy + c[v][2] * hx + c[v][3] * xy + c[v][4] * hy;
    const double e = 2.0 * q[0] * q[3], k = q[1] * q[1] + q[2] * q[2];
    const int ex = (__double2hiint(e) >> 20) & 0x7ff;      // biased exponent, on the integer pipe
    if (ex < 64 || ex > 1983) return q[0] > 0.0 && q[3] - 0.5 * k / q[0] > 0.0;
    return q[0] > 0.0 && e > k;
}

constexpr int kDetectBlock = 64;       // small blocks: a few thousand cells reach every SM

// Detector (Eqs. (37)-(38)) and positivity of every cell.  A smooth cell keeps its
// coefficients (flag 0); another one goes to list (list_n: its length) or, robust,
// keeps its average only (flag 2).
__global__ void __launch_bounds__(kDetectBlock) k_detect(const DeviceMesh d, const double *__restrict__ w,
                                                         const double *__restrict__ x, double *__restrict__ xl,
                                                         int32_t *__restrict__ flag, int32_t *__restrict__ list,
                                                         int32_t *__restrict__ list_n, int robust)
{
    const int64_t T = d.T, F = d.F;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= T) return;
    double U[4], c[4][5];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        U[v] = w[v * T + i];
#pragma unroll
        for (int l = 0; l < 5; ++l) c[v][l] = x[(v * 5 + l) * T + i];
    }
    const double hi = d.h[i], mxx = d.mxx[i], mxy = d.mxy[i], myy = d.myy[i];
    int J = 0;
    double s0 = 0.0, s3 = 0.0, m0 = U[0], m3 = U[3];
    const double v0 = U[0] - 0.5 * c[0][2] * mxx - c[0][3] * mxy - 0.5 * c[0][4] * myy;
    const double v3 = U[3] - 0.5 * c[3][2] * mxx - c[3][3] * mxy - 0.5 * c[3][4] * myy;
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const int64_t j = d.nb[s * T + i];             // neighbour slots are filled from slot 0
        if (j < 0) continue;
        ++J;
        const double r = hi / d.h[j];
        const double dx = -d.ox[s * T + i] * r, dy = -d.oy[s * T + i] * r;   // r_i in j's scaled frame
        const double hx = 0.5 * (dx * dx - d.mxx[j]), xy = dx * dy - d.mxy[j], hy = 0.5 * (dy * dy - d.myy[j]);
        const double w0 = w[j], w3 = w[3 * T + j];
        const double q0 = w0 + x[j] * dx + x[T + j] * dy + x[2 * T + j] * hx + x[3 * T + j] * xy + x[4 * T + j] * hy;
        const double q3 = w3 + x[15 * T + j] * dx + x[16 * T + j] * dy + x[17 * T + j] * hx + x[18 * T + j] * xy +
                          x[19 * T + j] * hy;
        s0 += fabs(v0 - q0);
        s3 += fabs(v3 - q3);
        m0 = fmax(m0, w0);
        m3 = fmax(m3, w3);
    }
    bool flagged = false;
    if (J > 0) {
        const double scale = J * (d.kord[i] == 2 ? hi * sqrt(hi) : hi);     // J h^{(k+1)/2}
        flagged = !(s0 / (scale * m0) < 1.0 && s3 / (scale * m3) < 1.0);
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const int32_t cf = d.cf[s * T + i];
            if (cf < 0) continue;
            const int64_t f = cf >> 1;
            const double *g = (cf & 1) ? d.gr : d.gl;
#pragma unroll
            for (int k = 0; k < 2; ++k)
                flagged |= !physical_at(U, c, mxx, mxy, myy, g[(2 * k) * F + f], g[(2 * k + 1) * F + f]);
        }
    }
    if (flagged && !robust) {
        list[atomicAdd(list_n, 1)] = (int32_t)i;
        return;
    }
#pragma unroll
    for (int v = 0; v < 4; ++v)
#pragma unroll
        for (int l = 0; l < 5; ++l) xl[(v * 5 + l) * T + i] = flagged ? 0.0 : c[v][l];
    flag[i] = flagged ? 2 : 0;
}

constexpr int kLimitWarps = 4;         // warps per block

// DWBAP limiter (Eqs. (34)-(36)) of the listed cells from e0 on, in steps of the grid,
// G lanes each: the first four lanes of a group take a candidate's weight each, lane
// 4 a + v the derivatives l = a, a + G/4, ... of variable (characteristic) v.
template <int G>
__device__ __forceinline__ void limit_cells(const DeviceMesh &d, const double *__restrict__ w,
                                            const double *__restrict__ x, double *__restrict__ xl,
                                            int32_t *__restrict__ flag, const int32_t *__restrict__ list, int total,
                                            double gamma, int charm, double (*sh)[4][5])
{
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int kPer = 32 / G;               // cells per warp
    const int64_t T = d.T, F = d.F;
    const int lane = threadIdx.x & (G - 1), grp = (threadIdx.x & 31) / G, v = lane & 3;
    double(*c)[5] = sh[grp];
    const int warp = blockIdx.x * kLimitWarps + (threadIdx.x >> 5), nwarp = gridDim.x * kLimitWarps;
    for (int e0 = warp * kPer; e0 < total; e0 += nwarp * kPer) {       // uniform over the warp
        const bool mine = e0 + grp < total;
        const int64_t i = list[mine ? e0 + grp : total - 1];
        const double hi = d.h[i];
        const int ki = d.kord[i];
        // lane s < 3: the pressure of neighbour s, its centroid in i's frame and i's in its
        int J = 0;
        int32_t nbj[3];
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            nbj[s] = d.nb[s * T + i];
            J += nbj[s] >= 0;
        }
        double X = 0.0, rh = 0.0, dx = 0.0, dy = 0.0;
        if (v < J) {
            const int64_t j = v == 0 ? nbj[0] : (v == 1 ? nbj[1] : nbj[2]);
            // in velocities: an infinite density gives no pressure (NaN), as an infinite energy does
            const double rho = w[j], ir = 1.0 / rho, u = w[T + j] * ir, vv = w[2 * T + j] * ir;
            X = (gamma - 1.0) * (w[3 * T + j] - 0.5 * rho * (u * u + vv * vv));
            rh = 1.0 / d.h[j];
            dx = -d.ox[v * T + i] * hi * rh;
            dy = -d.oy[v * T + i] * hi * rh;
        }
        // ---- weights, Eqs. (35)-(36); distances in i's scaled frame times h_i
        const double rJ = 1.0 / J;
        double Xs[3], rhj[3], ddx[3], ddy[3], Xbar = 0.0, var = 0.0;
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            Xs[s] = __shfl_sync(kAll, X, s, G);
            rhj[s] = __shfl_sync(kAll, rh, s, G);
            ddx[s] = __shfl_sync(kAll, dx, s, G);
            ddy[s] = __shfl_sync(kAll, dy, s, G);
            Xbar += s < J ? Xs[s] * rJ : 0.0;
        }
#pragma unroll
        for (int s = 0; s < 3; ++s)
            if (s < J) var += (Xs[s] - Xbar) * (Xs[s] - Xbar) * rJ;
        const double chi = sqrt(var) / Xbar;
        const double S = 1.0 / (sqrt(chi + 1e-8) + 0.05);
        // lane q: the weight of candidate q (0 the cell itself)
        double wt = 0.0;
        if (v <= J) {
            const double px = v == 0 ? 0.0 : d.ox[(v - 1) * T + i], py = v == 0 ? 0.0 : d.oy[(v - 1) * T + i];
            double dist = 0.0;
            int nf = 0;
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                const int32_t cf = d.cf[s * T + i];
                if (cf < 0) continue;
                const int64_t f = cf >> 1;
                if (d.fr[f] < 0) continue;
                const double *g = (cf & 1) ? d.gr : d.gl;   // the two Gauss points straddle the midpoint
                dist += hypot(px - 0.5 * (g[f] + g[2 * F + f]), py - 0.5 * (g[F + f] + g[3 * F + f]));
                ++nf;
            }
            wt = pow(hi * dist / nf, -S);
        }
        // weights of the first derivatives, and of the second ones (the neighbours with k = 2)
        double om[2][4], sum[2] = {0.0, 0.0};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            om[0][q] = __shfl_sync(kAll, wt, q, G);
            om[1][q] = q == 0 || (q <= J && d.kord[nbj[q > 0 ? q - 1 : 0]] == 2) ? om[0][q] : 0.0;
            sum[0] += om[0][q];
            sum[1] += om[1][q];
        }
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const double r = 1.0 / sum[a];
#pragma unroll
            for (int q = 0; q < 4; ++q) om[a][q] *= r;
        }
        // ---- a derivative row at a time: candidates in physical units, the cell's own
        // polynomial and the neighbours' (at r_i)
        const double rhi = 1.0 / hi;
        EulerState es = {};
        if (charm) {
            const double Wi[4] = {w[i], w[T + i], w[2 * T + i], w[3 * T + i]};
            es = euler_state(Wi, gamma);
        }
#pragma unroll 1
        for (int l0 = 0; l0 < 5; l0 += G / 4) {
            const int l = min(l0 + (lane >> 2), 4);        // spare lanes repeat the last row
            const bool high = l >= 2;
            const double own = x[(v * 5 + l) * T + i];
            double cand[4] = {own * (high ? rhi * rhi : rhi), 0.0, 0.0, 0.0}, o[4];
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                if (s >= J) continue;
                const int64_t j = nbj[s];
                if (high) {
                    cand[s + 1] = x[(v * 5 + l) * T + j] * (rhj[s] * rhj[s]);
                } else {
                    const double ua = x[(v * 5 + l) * T + j];          // u1 (l = 0) or u2 (l = 1)
                    const double ub = x[(v * 5 + 2 + l) * T + j];      // u3 or u4
                    const double uc = x[(v * 5 + 3 + l) * T + j];      // u4 or u5
                    cand[s + 1] = (ua + ub * ddx[s] + uc * ddy[s]) * rhj[s];
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) o[q] = high ? om[1][q] : om[0][q];
            double res;
            if (charm) {
                // characteristic variables along x (d/dx, d2/dx2), y (d/dy, d2/dy2), the
                // diagonal (d2/dxdy); lane v of a row takes characteristic v
                const double nx = l == 1 || l == 4 ? 0.0 : (l == 3 ? 0.70710678118654752 : 1.0);
                const double ny = l == 0 || l == 2 ? 0.0 : (l == 3 ? 0.70710678118654752 : 1.0);
                double Lr[4], Rr[4], ch[4];
                char_rows(es, v, nx, ny, Rr, Lr);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    ch[q] = Lr[0] * __shfl_sync(kAll, cand[q], 0, 4) + Lr[1] * __shfl_sync(kAll, cand[q], 1, 4) +
                            Lr[2] * __shfl_sync(kAll, cand[q], 2, 4) + Lr[3] * __shfl_sync(kAll, cand[q], 3, 4);
                const double lim = biased_mean(ch, o);
                res = Rr[0] * __shfl_sync(kAll, lim, 0, 4) + Rr[1] * __shfl_sync(kAll, lim, 1, 4) +
                      Rr[2] * __shfl_sync(kAll, lim, 2, 4) + Rr[3] * __shfl_sync(kAll, lim, 3, 4);
            } else {
                res = biased_mean(cand, o);
            }
            // a linear cell's second derivatives are kept
            c[v][l] = high && ki != 2 ? own : (high ? hi * hi : hi) * res;
        }
        __syncwarp();

        // ---- safeguard at the cell's face Gauss points, a point (2 s + k: k of face s) per lane
        double U[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) U[q] = w[q * T + i];
        bool ok = true;
        for (int t = lane; t < 6; t += G) {
            const int32_t cf = d.cf[(t >> 1) * T + i];
            if (cf < 0) continue;
            const int64_t f = cf >> 1;
            const double *g = (cf & 1) ? d.gr : d.gl;
            const int k = t & 1;
            ok = ok && physical_at(U, c, d.mxx[i], d.mxy[i], d.myy[i], g[(2 * k) * F + f], g[(2 * k + 1) * F + f]);
        }
        const unsigned fails = __ballot_sync(kAll, !ok) >> (G * grp);
        const bool bad = (G == 32 ? fails : fails & ((1u << (G & 31)) - 1u)) != 0u;
        if (mine) {
            for (int l = lane >> 2; l < 5; l += G / 4) xl[(v * 5 + l) * T + i] = bad ? 0.0 : c[v][l];
            if (lane == 0) flag[i] = bad ? 2 : 1;
        }
        __syncwarp();
    }
}

// A warp takes one listed cell or eight.  A cell of its own ends in about 20 us, eight
// in about 45 (five rows per lane), so eight pay once the sub-partitions have more than
// two cells each.  Long lists need the grid's four blocks per SM resident: 128 registers
// with 28 bytes of spills, where 151 left a quarter of the grid for a second round (a call with
// 480,000 flagged cells, conservative / characteristic: 6.4 / 8.0 -> 4.5 / 5.6 ms, 5.8 / 6.3
// with a thread per cell; 240,000: 2.7 / 3.4 -> 2.3 / 2.8, 3.1 / 3.4; 24,000 or fewer the same).
__global__ void __launch_bounds__(32 * kLimitWarps, 4) k_limit(const DeviceMesh d, const double *__restrict__ w,
                                                            const double *__restrict__ x, double *__restrict__ xl,
                                                            int32_t *__restrict__ flag,
                                                            const int32_t *__restrict__ list,
                                                            const int32_t *__restrict__ list_n, double gamma, int charm,
                                                            int one_max)
{
    __shared__ double sh[kLimitWarps][8][4][5];
    const int total = *list_n;
    if (total <= one_max)
        limit_cells<32>(d, w, x, xl, flag, list, total, gamma, charm, sh[threadIdx.x >> 5]);
    else
        limit_cells<4>(d, w, x, xl, flag, list, total, gamma, charm, sh[threadIdx.x >> 5]);
}

// caller[perm[i]] = internal[i] for the limiter flags (padding skipped)
__global__ void k_scatter_flags(const int32_t *__restrict__ src, const int32_t *__restrict__ perm,
                                int32_t *__restrict__ dst, int64_t T)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= T) return;
    const int32_t c = perm[i];
    if (c >= 0) dst[c] = src[i];
}

}  // namespace

gks_status launch_limiter(gks_mesh *m, const double *w, const double *x, cudaStream_t s)
{
    const DeviceMesh &d = m->d;
    if (!d.ox || !d.oy || !d.kord || !m->wk.xl || !m->wk.lflag) {
        set_error("the limiter was not enabled when the mesh was created (gks_config.limiter = 1)");
        return GKS_EINVAL;
    }
    if (d.T == 0) return GKS_OK;
    Work &k = m->wk;
    const bool robust = m->cfg.limiter == 2;
    if (!robust) GKS_CUDA(cudaMemsetAsync(k.llist + d.T, 0, sizeof(int32_t), s));
    k_detect<<<(unsigned)((d.T + kDetectBlock - 1) / kDetectBlock), kDetectBlock, 0, s>>>(
        d, w, x, k.xl, k.lflag, k.llist, robust ? nullptr : k.llist + d.T, robust ? 1 : 0);
    note_launch();
    if (!robust) {
        // every listed cell on a group of its own, up to four warps per SM sub-partition
        const int64_t need = (d.T + kLimitWarps - 1) / kLimitWarps;
        const unsigned g = (unsigned)std::min<int64_t>(need, (int64_t)k.sm_count * 4);
        k_limit<<<g, 32 * kLimitWarps, 0, s>>>(d, w, x, k.xl, k.lflag, k.llist, k.llist + d.T, m->cfg.gamma,
                                               m->cfg.limit_char, 2 * 4 * k.sm_count);
        note_launch();
    }
    GKS_CUDA(cudaGetLastError());
    return GKS_OK;
}

gks_status launch_scatter_flags(gks_mesh *m, int32_t *flags_out, cudaStream_t s)
{
    const DeviceMesh &d = m->d;
    if (d.T == 0) return GKS_OK;
    const unsigned nb = (unsigned)((d.T + kBlock - 1) / kBlock);
    k_scatter_flags<<<nb, kBlock, 0, s>>>(m->wk.lflag, d.perm, flags_out, d.T);
    note_launch();
    GKS_CUDA(cudaGetLastError());
    return GKS_OK;
}

}  // namespace gks
