// Kernels of the FP64 reconstruction solve (per-cell equations), one thread per
// cell and variable.
//
// GB300 runs FP64 at 1/64 of its FP32 rate: a warp's FP64 instruction holds its
// SM sub-partition for 33 ns whatever its active lanes, so a kernel's time is
// the number of FP64 instructions per thread times the warps per sub-partition
// (608 of them).  A thread per cell (all four variables in it) left an
// 800-triangle mesh with 25 warps of 640 instructions per preconditioner
// application.  Here a warp takes 32 cells of one variable: four times the
// warps with a quarter of the instructions each, no block-wide barrier, and the
// warps of a variable whose system has stopped return at once.
//
// What else keeps the instruction count down:
//  - the sweeps work on the products W = P O of the pivot inverse and the
//    off-diagonal blocks (set-up; 5 x 2, a block reads the gradient rows 0 and 1 of a
//    neighbour alone): z = P r once, then rows 0 and 1 of z + sum W z per sweep (12
//    multiply-adds; rows 0 and 1 are all that the next sweep reads), and the last
//    sweep adds the lower and the upper neighbours' terms together, three slots
//    of 10.  With P applied in every sweep, and the lower and upper slots
//    apart (a warp's lanes have up to three of each), two sweeps each way
//    took 152 multiply-adds, now 91;
//  - the operator's off-diagonal blocks are stored multiplied out (off: alpha,
//    alpha dx, alpha dy per slot);
//  - sums over cells start their FMA chains from the running sum in shared
//    memory and are added across the lanes of a warp in transposed order, 7-31
//    additions for all Arnoldi indices together instead of 5 for each;
//  - the basis grows by w = K M^-1 V_j - V_j, which spans the same Krylov space (the
//    Hessenberg diagonal gets its 1 back).  The preconditioner is close to the
//    inverse, so nearly all of K M^-1 V_j is V_j itself: without the shift the part
//    orthogonal to the basis is 0.02-0.36 of the vector, with it 0.3 or more and mostly
//    0.5-0.99 of |w|, so one Gram-Schmidt pass loses few digits and the second runs only
//    where the orthogonal part is below half of |w|.  Largest entry of V^T V - 1 (128 to 800
//    triangles, aspects 1 to 300, no to two sweeps, 28 vectors): 4e-15, with a second pass in
//    none to 13 of the indices; two passes of the unshifted basis 1e-15, one 2e-13 to 1.
//    Three steps at 399,424 triangles 46.2 -> 41.9 ms, ten at 6,400 6.56 -> 6.06 ms, at 800
//    6.05 -> 5.50 ms.
// Measured on GB300 (the solve's classes, per Arnoldi index, events around each
// class) against a thread per cell: preconditioner with two sweeps each way 80 -> 25 us
// at 6,400 triangles and 680 -> 266 us at 399,424 (436 with P in every sweep);
// operator with the first Gram-Schmidt products and the rest of the Gram-Schmidt
// passes 83 -> 39 us and 610 -> 363 us.
#pragma once

#include "gks_internal.h"

namespace gks {
namespace {

constexpr int kW64 = 128;              // threads per block: one warp per variable

// Cells per thread (C) and partial-sum rows per kBlock-cell block (8 / C): more
// cells per thread amortise the sums across lanes once the GPU is full of warps
// (T / 8 of them with one cell per thread), fewer spread a small mesh over it.
inline int cells64(int64_t T) { return T <= 40000 ? 1 : (T <= 80000 ? 2 : (T <= 160000 ? 4 : 8)); }
constexpr int kRows64 = kBlock / 32;   // rows per cell block with one cell per thread

// acc += O (g1, g2) for the stored block (a, ax, ay) = alpha (1, dx, dy)
__device__ __forceinline__ void off_acc(double a, double ax, double ay, double g1, double g2, double *acc)
{
    acc[0] = fma(a, g1, acc[0]);
    acc[1] = fma(a, g2, acc[1]);
    acc[2] = fma(ax, g1, acc[2]);
    acc[3] = fma(ay, g1, fma(ax, g2, acc[3]));
    acc[4] = fma(ay, g2, acc[4]);
}

struct Off64 {
    double a, ax, ay;
};

__device__ __forceinline__ Off64 off_load(const double *__restrict__ off, int64_t T, int s, int64_t i)
{
    return {off[(3 * s) * T + i], off[(3 * s + 1) * T + i], off[(3 * s + 2) * T + i]};
}

// Multiplied-out off-diagonal blocks (set-up): off[3 s + (0, 1, 2)] = alpha (1, dx, dy)
__global__ void k64_off(int64_t T, const double *__restrict__ al, const double *__restrict__ ex,
                        const double *__restrict__ ey, double *__restrict__ off)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= T) return;
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const double a = al[s * T + i];
        off[(3 * s) * T + i] = a;
        off[(3 * s + 1) * T + i] = a * ex[s * T + i];
        off[(3 * s + 2) * T + i] = a * ey[s * T + i];
    }
}

// W = P O per slot (set-up): w[10 s + 2 a + c], row a, column c (the neighbour's row c)
__global__ void k64_products(int64_t T, const double *__restrict__ P, const double *__restrict__ off,
                             double *__restrict__ w)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= T) return;
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const Off64 o = off_load(off, T, s, i);
        for (int a = 0; a < 5; ++a) {
            double p[5];
#pragma unroll
            for (int c = 0; c < 5; ++c) p[c] = P[(a * 5 + c) * T + i];
            w[(10 * s + 2 * a) * T + i] = fma(p[0], o.a, fma(p[2], o.ax, p[3] * o.ay));
            w[(10 * s + 2 * a + 1) * T + i] = fma(p[1], o.a, fma(p[3], o.ax, p[4] * o.ay));
        }
    }
}

// What every kernel of the solve knows about its warp: the variable, the first
// cell of the block, and whether the system still runs.
struct Warp64 {
    int lane, v, sys;
    bool run;
};

__device__ __forceinline__ Warp64 warp64(const int32_t *__restrict__ blk_case, const int32_t *__restrict__ run,
                                         int64_t cell0)
{
    Warp64 w;
    w.lane = threadIdx.x & 31;
    w.v = threadIdx.x >> 5;
    w.sys = 4 * blk_case[cell0 / kBlock] + w.v;
    w.run = !run || run[w.sys] != 0;
    return w;
}

// z = P r.  (Forming the first forward sweep here as well, with the neighbours'
// rows 0 and 1 of z from their r, saved a launch and no time: 20 steps 8.55 against 8.55 ms at
// 800 triangles, 10.8 against 10.5 at 6,500, 16.3 against 15.8 at 15,800.)
__global__ void __launch_bounds__(kW64, 6) k64_pivot(int64_t T, const double *__restrict__ P,
                                                     const int32_t *__restrict__ blk_case,
                                                     const int32_t *__restrict__ run, const double *__restrict__ r,
                                                     double *__restrict__ z)
{
    const int64_t c0 = blockIdx.x * (int64_t)32;
    const Warp64 w = warp64(blk_case, run, c0);
    const int64_t i = c0 + w.lane, vo = (int64_t)w.v * 5 * T;
    if (!w.run || i >= T) return;
    double y[5], Pm[25];
#pragma unroll
    for (int k = 0; k < 5; ++k) y[k] = r[vo + k * T + i];
#pragma unroll
    for (int k = 0; k < 25; ++k) Pm[k] = P[k * T + i];
#pragma unroll
    for (int a = 0; a < 5; ++a) {
        double s = 0.0;
#pragma unroll
        for (int c = 0; c < 5; ++c) s = fma(Pm[a * 5 + c], y[c], s);
        z[vo + a * T + i] = s;
    }
}

// A sweep that only feeds another one, rows 0 and 1: out_i = base_i + sum_j W_ij
// in_j over the lower (UP = false) or upper neighbours j
template <bool UP>
__global__ void __launch_bounds__(kW64) k64_sweep(int64_t T, const int32_t *__restrict__ nb,
                                                  const double *__restrict__ W, const int32_t *__restrict__ blk_case,
                                                  const int32_t *__restrict__ run, const double *__restrict__ base,
                                                  const double *__restrict__ in, double *__restrict__ out)
{
    const int64_t c0 = blockIdx.x * (int64_t)32;
    const Warp64 w = warp64(blk_case, run, c0);
    const int64_t i = c0 + w.lane, vo = (int64_t)w.v * 5 * T;
    if (!w.run || i >= T) return;
    int js[3];
    double wj[3][4], z[3][2], o[2];
#pragma unroll
    for (int s = 0; s < 3; ++s) js[s] = nb[s * T + i];
#pragma unroll
    for (int a = 0; a < 2; ++a) o[a] = base[vo + a * T + i];
    // the loads of all neighbours first, then the sums
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const int64_t j = js[s];
        if (!(UP ? j > i : (j >= 0 && j < i))) continue;
#pragma unroll
        for (int k = 0; k < 4; ++k) wj[s][k] = W[(10 * s + k) * T + i];
#pragma unroll
        for (int a = 0; a < 2; ++a) z[s][a] = in[vo + a * T + j];
    }
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const int64_t j = js[s];
        if (!(UP ? j > i : (j >= 0 && j < i))) continue;
#pragma unroll
        for (int a = 0; a < 2; ++a) o[a] = fma(wj[s][2 * a], z[s][0], fma(wj[s][2 * a + 1], z[s][1], o[a]));
    }
#pragma unroll
    for (int a = 0; a < 2; ++a) out[vo + a * T + i] = o[a];
}

// The last sweep, x_i = z_i + sum_{j<i} W_ij low_j + sum_{j>i} W_ij up_j, all five
// rows (low, up: the last sweep's sources; NULL: no sweeps that way)
__global__ void __launch_bounds__(kW64, 4) k64_last(int64_t T, const int32_t *__restrict__ nb,
                                                 const double *__restrict__ W, const int32_t *__restrict__ blk_case,
                                                 const int32_t *__restrict__ run, const double *__restrict__ z,
                                                 const double *__restrict__ low, const double *__restrict__ up,
                                                 double *__restrict__ x)
{
    const int64_t c0 = blockIdx.x * (int64_t)32;
    const Warp64 w = warp64(blk_case, run, c0);
    const int64_t i = c0 + w.lane, vo = (int64_t)w.v * 5 * T;
    if (!w.run || i >= T) return;
    double o[5], g[3][2], wj[3][10];
    int js[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) js[s] = nb[s * T + i];
#pragma unroll
    for (int a = 0; a < 5; ++a) o[a] = z[vo + a * T + i];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const int64_t j = js[s];
        const double *src = j < 0 ? nullptr : (j < i ? low : up);
#pragma unroll
        for (int a = 0; a < 2; ++a) g[s][a] = src ? src[vo + a * T + j] : 0.0;
#pragma unroll
        for (int k = 0; k < 10; ++k) wj[s][k] = W[(10 * s + k) * T + i];
    }
#pragma unroll
    for (int s = 0; s < 3; ++s)
#pragma unroll
        for (int a = 0; a < 5; ++a) o[a] = fma(wj[s][2 * a], g[s][0], fma(wj[s][2 * a + 1], g[s][1], o[a]));
#pragma unroll
    for (int a = 0; a < 5; ++a) x[vo + a * T + i] = o[a];
}

// acc = (K x)_i of variable v, diagonal block minus the off-diagonal ones, minus
// s_i (s may be NULL)
__device__ __forceinline__ void apply64(int64_t T, const int32_t *__restrict__ nb, const double *__restrict__ D,
                                        const double *__restrict__ off, const double *__restrict__ xv, int64_t i,
                                        double *acc, const double *__restrict__ s0 = nullptr)
{
    int j[3];
    Off64 o[3];
    double g[3][2], Dm[15], x[5];
#pragma unroll
    for (int s = 0; s < 3; ++s) j[s] = nb[s * T + i];
#pragma unroll
    for (int l = 0; l < 5; ++l) x[l] = xv[l * T + i];
#pragma unroll
    for (int q = 0; q < 15; ++q) Dm[q] = D[q * T + i];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        // a missing neighbour has a zero block; it reads the cell's own values
        const int64_t n = j[s] >= 0 ? j[s] : i;
        o[s] = off_load(off, T, s, i);
        g[s][0] = -xv[n];
        g[s][1] = -xv[T + n];
    }
    constexpr int kIdx[5][5] = {{0, 1, 2, 3, 4}, {1, 5, 6, 7, 8}, {2, 6, 9, 10, 11}, {3, 7, 10, 12, 13},
                                {4, 8, 11, 13, 14}};
#pragma unroll
    for (int a = 0; a < 5; ++a) {
        acc[a] = s0 ? fma(Dm[kIdx[a][0]], x[0], -s0[a * T + i]) : Dm[kIdx[a][0]] * x[0];
#pragma unroll
        for (int c = 1; c < 5; ++c) acc[a] = fma(Dm[kIdx[a][c]], x[c], acc[a]);
    }
#pragma unroll
    for (int s = 0; s < 3; ++s) off_acc(o[s].a, o[s].ax, o[s].ay, g[s][0], g[s][1], acc);
}

// Sums over the lanes of a warp of the rows acc[k][lane] (k < K, row stride 33),
// written to out[k os]: each row is split among 32 / (rows per pass) lanes, which
// add its entries in order and then each other's sums.
constexpr int kAccStride = 33;

__device__ __forceinline__ void warp_rows(const double *acc, int K, int lane, double *__restrict__ out, int64_t os)
{
    const int g = K <= 4 ? 8 : (K <= 8 ? 4 : (K <= 16 ? 2 : 1));
    const int sub = lane % g;
    for (int k0 = 0; k0 < K; k0 += 32 / g) {
        const int k = k0 + lane / g;
        double s = 0.0;
        if (k < K)
            for (int t = sub; t < 32; t += g) s += acc[k * kAccStride + t];
        for (int o = g >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (sub == 0 && k < K) out[k * os] = s;
    }
}

// One value per lane summed over the warp (lane 0 gets it)
__device__ __forceinline__ double warp_sum(double s)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    return s;
}

// y = K z - V_j, the products <V_k, y>, k <= j, of the first Gram-Schmidt pass and
// |y|^2 (k = j + 1): part[k][v][row] over the 32 C cells of the block.  Dynamic
// shared memory: 4 (j + 2) kAccStride doubles.
template <int C>
__global__ void __launch_bounds__(kW64) k64_apply_dots(int64_t T, const int32_t *__restrict__ nb,
                                                       const double *__restrict__ D, const double *__restrict__ off,
                                                       const int32_t *__restrict__ blk_case,
                                                       const int32_t *__restrict__ run, const double *__restrict__ z,
                                                       double *__restrict__ y, const double *__restrict__ V, int j,
                                                       double *__restrict__ part)
{
    extern __shared__ double sh64[];
    const int64_t c0 = blockIdx.x * (int64_t)(32 * C);
    const Warp64 w = warp64(blk_case, run, c0);
    if (!w.run) return;
    const int K = j + 1;
    double *acc = sh64 + w.v * (K + 1) * kAccStride;
    for (int k = 0; k < K; ++k) acc[k * kAccStride + w.lane] = 0.0;
    const int64_t vo = (int64_t)w.v * 5 * T, vs = 20 * T;
    double nr = 0.0;
    for (int c = 0; c < C; ++c) {
        const int64_t i = c0 + 32 * c + w.lane;
        if (i >= T) break;
        double u[5];
        apply64(T, nb, D, off, z + vo, i, u, V + j * vs + vo);
#pragma unroll
        for (int l = 0; l < 5; ++l) {
            y[vo + l * T + i] = u[l];
            nr = fma(u[l], u[l], nr);
        }
#pragma unroll 4
        for (int k = 0; k < K; ++k) {
            const double *vk = V + k * vs + vo + i;
            double s = acc[k * kAccStride + w.lane];
#pragma unroll
            for (int l = 0; l < 5; ++l) s = fma(vk[l * T], u[l], s);
            acc[k * kAccStride + w.lane] = s;
        }
    }
    acc[K * kAccStride + w.lane] = nr;
    __syncwarp();
    warp_rows(acc, K + 1, w.lane, part + w.v * (int64_t)gridDim.x + blockIdx.x, 4 * (int64_t)gridDim.x);
}

// The second pass of the systems that need it: w -= sum_k h_k V_k and the partial |w|^2
template <int C>
__global__ void __launch_bounds__(kW64) k64_update_norm(int64_t T, const int32_t *__restrict__ blk_case,
                                                        const int32_t *__restrict__ run,
                                                        const int32_t *__restrict__ twice,
                                                        const double *__restrict__ V, double *__restrict__ wn, int j,
                                                        const double *__restrict__ hc, int hstride,
                                                        double *__restrict__ part)
{
    __shared__ double hs[4][kMaxRestart];
    const int64_t c0 = blockIdx.x * (int64_t)(32 * C);
    const Warp64 w = warp64(blk_case, run, c0);
    if (!w.run || !twice[w.sys]) return;
    const int K = j + 1;
    for (int k = w.lane; k < K; k += 32) hs[w.v][k] = hc[w.sys * hstride + k];
    __syncwarp();
    const int64_t vo = (int64_t)w.v * 5 * T, vs = 20 * T;
    double nr = 0.0;
    for (int c = 0; c < C; ++c) {
        const int64_t i = c0 + 32 * c + w.lane;
        if (i >= T) break;
        double u[5];
#pragma unroll
        for (int l = 0; l < 5; ++l) u[l] = wn[vo + l * T + i];
#pragma unroll 4
        for (int k = 0; k < K; ++k) {
            const double *vk = V + k * vs + vo + i;
            const double hk = -hs[w.v][k];
#pragma unroll
            for (int l = 0; l < 5; ++l) u[l] = fma(hk, vk[l * T], u[l]);
        }
#pragma unroll
        for (int l = 0; l < 5; ++l) {
            wn[vo + l * T + i] = u[l];
            nr = fma(u[l], u[l], nr);
        }
    }
    nr = warp_sum(nr);
    if (w.lane == 0) part[w.v * (int64_t)gridDim.x + blockIdx.x] = nr;
}

// Right-hand side b_i = sum_j a0_ij (w_j - w_i) and the partial |b|^2 (entry 1)
template <int C>
__global__ void __launch_bounds__(kW64) k64_rhs(int64_t T, const int32_t *__restrict__ nb,
                                                const double *__restrict__ a0, const double *__restrict__ wst,
                                                double *__restrict__ b, double *__restrict__ part)
{
    const int64_t c0 = blockIdx.x * (int64_t)(32 * C);
    const int lane = threadIdx.x & 31, v = threadIdx.x >> 5;
    const int64_t vo = (int64_t)v * 5 * T;
    const double *wv = wst + v * T;
    double nr = 0.0;
    for (int c = 0; c < C; ++c) {
        const int64_t i = c0 + 32 * c + lane;
        if (i >= T) break;
        const double wi = wv[i];
        double du[3], a[3][5], s[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int j = nb[q * T + i];
            du[q] = wv[j >= 0 ? j : i] - wi;       // no neighbour: 0
#pragma unroll
            for (int l = 0; l < 5; ++l) a[q][l] = a0[(q * 5 + l) * T + i];
        }
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int l = 0; l < 5; ++l) s[l] = fma(a[q][l], du[q], s[l]);
#pragma unroll
        for (int l = 0; l < 5; ++l) {
            b[vo + l * T + i] = s[l];
            nr = fma(s[l], s[l], nr);
        }
    }
    nr = warp_sum(nr);
    if (lane == 0) part[(4 + v) * (int64_t)gridDim.x + blockIdx.x] = nr;
}

// Residual y = b - K x and the partial |y|^2 (entry 0); act (NULL on a solve's
// first residual): systems that are not active keep theirs
template <int C>
__global__ void __launch_bounds__(kW64) k64_resid(int64_t T, const int32_t *__restrict__ nb,
                                                  const double *__restrict__ D, const double *__restrict__ off,
                                                  const int32_t *__restrict__ blk_case,
                                                  const int32_t *__restrict__ act, const double *__restrict__ x,
                                                  const double *__restrict__ b, double *__restrict__ y,
                                                  double *__restrict__ part)
{
    const int64_t c0 = blockIdx.x * (int64_t)(32 * C);
    const Warp64 w = warp64(blk_case, act, c0);
    if (!w.run) return;
    const int lane = w.lane, v = w.v;
    const int64_t vo = (int64_t)v * 5 * T;
    double nr = 0.0;
    for (int c = 0; c < C; ++c) {
        const int64_t i = c0 + 32 * c + lane;
        if (i >= T) break;
        double u[5];
        apply64(T, nb, D, off, x + vo, i, u);
#pragma unroll
        for (int l = 0; l < 5; ++l) {
            const double rv = b[vo + l * T + i] - u[l];
            y[vo + l * T + i] = rv;
            nr = fma(rv, rv, nr);
        }
    }
    nr = warp_sum(nr);
    if (lane == 0) part[v * (int64_t)gridDim.x + blockIdx.x] = nr;
}

// x += sum_{k<jv} y_k Z_k at the end of a cycle
__global__ void __launch_bounds__(kW64) k64_combine(int64_t T, const int32_t *__restrict__ blk_case,
                                                    const double *__restrict__ Z, const double *__restrict__ y,
                                                    int m, const int32_t *__restrict__ jvs, double *__restrict__ x)
{
    const int64_t c0 = blockIdx.x * (int64_t)32;
    const Warp64 w = warp64(blk_case, nullptr, c0);
    const int64_t i = c0 + w.lane;
    const int jv = jvs[w.sys];
    if (jv <= 0 || i >= T) return;
    const int64_t vo = (int64_t)w.v * 5 * T, vs = 20 * T;
    double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (int k = 0; k < jv; ++k) {
        const double yk = y[w.sys * m + k];
        const double *zk = Z + k * vs + vo + i;
#pragma unroll
        for (int l = 0; l < 5; ++l) acc[l] = fma(yk, zk[l * T], acc[l]);
    }
#pragma unroll
    for (int l = 0; l < 5; ++l) x[vo + l * T + i] += acc[l];
}

}  // namespace
}  // namespace gks
