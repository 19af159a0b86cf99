// Kernels of the mixed-precision reconstruction solve (per-cell equations), one
// thread per cell with its four variables: the FP32 preconditioner sweeps (FP32
// or FP16 factors), the operator with the Gram-Schmidt products, and the update.
//
// FP32 vectors of the solve are stored [dof][cell][variable], so a thread reads
// or writes a dof of its cell, or gathers one of a neighbour's, with one 16-byte
// access; the factors are packed in chunks of eight values per cell and the
// operator in six groups of four.  These kernels were bound by load
// instructions and L1 wavefronts, not by DRAM (the first forward sweep made 167
// 4-byte loads per cell for 240 bytes of DRAM traffic; now 36 loads).  A thread per cell
// and variable, as in FP64 (gks_solve64.cuh), reads the factors four times and
// ran the sweeps at 1,000,000 triangles 1.7 times slower.
#pragma once

#include <type_traits>

#include "gks_solve64.cuh"

namespace gks {
namespace {

constexpr int kW32 = 128;              // threads per block (cells), half a cell block

// ---- vectors: FP32 [dof][cell][4], FP64 [variable][dof][cell]

// the four variables of dof l of cell i
template <typename TX, typename TM>
__device__ __forceinline__ void vload(const TX *__restrict__ x, int l, int64_t T, int64_t i, TM *o)
{
    if constexpr (std::is_same_v<TX, float>) {
        const float4 t = reinterpret_cast<const float4 *>(x)[l * T + i];
        o[0] = TM(t.x);
        o[1] = TM(t.y);
        o[2] = TM(t.z);
        o[3] = TM(t.w);
    } else {
#pragma unroll
        for (int v = 0; v < 4; ++v) o[v] = TM(x[(v * 5 + l) * T + i]);
    }
}

// the same through L2 (a value that another block of the launch has written)
template <typename TX, typename TM>
__device__ __forceinline__ void vload_cg(const TX *x, int l, int64_t T, int64_t i, TM *o)
{
    if constexpr (std::is_same_v<TX, float>) {
        const float4 t = __ldcg(reinterpret_cast<const float4 *>(x) + l * T + i);
        o[0] = TM(t.x);
        o[1] = TM(t.y);
        o[2] = TM(t.z);
        o[3] = TM(t.w);
    } else {
#pragma unroll
        for (int v = 0; v < 4; ++v) o[v] = TM(__ldcg(x + (v * 5 + l) * T + i));
    }
}

template <typename TX, typename TM>
__device__ __forceinline__ void vstore(TX *x, int l, int64_t T, int64_t i, const TM *o)
{
    if constexpr (std::is_same_v<TX, float>) {
        reinterpret_cast<float4 *>(x)[l * T + i] = make_float4(float(o[0]), float(o[1]), float(o[2]), float(o[3]));
    } else {
#pragma unroll
        for (int v = 0; v < 4; ++v) x[(v * 5 + l) * T + i] = TX(o[v]);
    }
}

// ---- packed factors: 34 values per cell in four chunks of eight, [chunk][cell][8],
// and a pair: P 0-7 | P 8-9, alpha 0-2, dx 0-2 | dy 0-2, P 10-14 | P 15-22 | P 23-24 (the pivot
// inverse row-major; rows 0 and 1 and the off-diagonal blocks in the first three)
template <typename TP>
__device__ __forceinline__ void load8(const TP *__restrict__ pk, int c, int64_t T, int64_t i, float *o)
{
    const TP *p = pk + (c * T + i) * 8;
    if constexpr (std::is_same_v<TP, float>) {
        const float4 a = reinterpret_cast<const float4 *>(p)[0], b = reinterpret_cast<const float4 *>(p)[1];
        o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w;
        o[4] = b.x; o[5] = b.y; o[6] = b.z; o[7] = b.w;
    } else {
        const uint4 a = reinterpret_cast<const uint4 *>(p)[0];
        const unsigned u[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&u[q]));
            o[2 * q] = f.x;
            o[2 * q + 1] = f.y;
        }
    }
}

template <typename TP>
__device__ __forceinline__ void load2(const TP *__restrict__ pk, int64_t T, int64_t i, float *o)
{
    const TP *p = pk + 32 * T + 2 * i;
    if constexpr (std::is_same_v<TP, float>) {
        const float2 f = *reinterpret_cast<const float2 *>(p);
        o[0] = f.x; o[1] = f.y;
    } else {
        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(p));
        o[0] = f.x; o[1] = f.y;
    }
}

// set-up: the packed factors from P [25][T] and the off-diagonal blocks [3][T]
template <typename TP>
__global__ void k32_pack(int64_t T, const TP *__restrict__ P, const TP *__restrict__ al, const TP *__restrict__ ex,
                         const TP *__restrict__ ey, TP *__restrict__ pk)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= T) return;
    TP o[34];
#pragma unroll
    for (int q = 0; q < 10; ++q) o[q] = P[q * T + i];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        o[10 + s] = al[s * T + i];
        o[13 + s] = ex[s * T + i];
        o[16 + s] = ey[s * T + i];
    }
#pragma unroll
    for (int q = 10; q < 25; ++q) o[9 + q] = P[q * T + i];
#pragma unroll
    for (int q = 0; q < 32; ++q) pk[((q / 8) * T + i) * 8 + q % 8] = o[q];
    pk[32 * T + 2 * i] = o[32];
    pk[32 * T + 2 * i + 1] = o[33];
}

// set-up: the operator, D [15][T] and the off-diagonal blocks, as [6][cell][4]
__global__ void k32_pack_op(int64_t T, const float *__restrict__ D, const float *__restrict__ al,
                            const float *__restrict__ ex, const float *__restrict__ ey, float4 *__restrict__ op)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= T) return;
    float o[24];
#pragma unroll
    for (int q = 0; q < 15; ++q) o[q] = D[q * T + i];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        o[15 + s] = al[s * T + i];
        o[18 + s] = ex[s * T + i];
        o[21 + s] = ey[s * T + i];
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) op[q * T + i] = make_float4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
}

// rows 0 and 1 of a pivot inverse (p[0..9]) with the off-diagonal blocks of the cell
struct Rows01 {
    float p[10], a[3], x[3], y[3];
};

template <bool OFF, typename TP>
__device__ __forceinline__ void load_rows(const TP *__restrict__ pk, int64_t T, int64_t i, Rows01 &r, float *c2)
{
    float c0[8], c1[8];
    load8(pk, 0, T, i, c0);
    load8(pk, 1, T, i, c1);
#pragma unroll
    for (int q = 0; q < 8; ++q) r.p[q] = c0[q];
    r.p[8] = c1[0];
    r.p[9] = c1[1];
    if (OFF) {
        load8(pk, 2, T, i, c2);
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            r.a[s] = c1[2 + s];
            r.x[s] = c1[5 + s];
            r.y[s] = c2[s];
        }
    }
}

// y[l][v] += O_s (g0[v], g1[v]): the off-diagonal block a (1, dx, dy) on a neighbour's gradient rows
__device__ __forceinline__ void off_acc4(float a, float dx, float dy, const float *g0, const float *g1, float (*y)[4])
{
    const float ax = a * dx, ay = a * dy;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        y[0][v] = fmaf(a, g0[v], y[0][v]);
        y[1][v] = fmaf(a, g1[v], y[1][v]);
        y[2][v] = fmaf(ax, g0[v], y[2][v]);
        y[3][v] = fmaf(ay, g0[v], fmaf(ax, g1[v], y[3][v]));
        y[4][v] = fmaf(ay, g1[v], y[4][v]);
    }
}

// out[v] = start[v] + sum_c p[c] y[c][v]
__device__ __forceinline__ void row_times(const float *p, const float (*y)[4], const float *start, float *out)
{
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        float s = start ? start[v] : 0.0f;
#pragma unroll
        for (int c = 0; c < 5; ++c) s = fmaf(p[c], y[c][v], s);
        out[v] = s;
    }
}

// Whether any of the four systems of this block's case still runs (run NULL: yes)
__device__ __forceinline__ bool case_runs(const int32_t *__restrict__ blk_case, const int32_t *__restrict__ run)
{
    if (!run) return true;
    const int4 r = reinterpret_cast<const int4 *>(run)[blk_case[(blockIdx.x * (int64_t)blockDim.x) / kBlock]];
    return (r.x | r.y | r.z | r.w) != 0;
}

// Forward relation z_i = P_i (r_i + sum_{k<i} O_ik zin_k); NB 0: no neighbours
// (z = P r); 1: zin as given; 2: zin_k = P_k r_k formed here (the first sweep).
// FULL: all five rows of z, else the rows 0 and 1 that the next sweep reads.  rc
// (may be NULL): also store float(r_i) for the later sweeps of a wider source.
template <int NB, bool FULL, typename TR, typename TP>
__global__ void __launch_bounds__(kW32, 5) k32_fwd(int64_t T, const int32_t *__restrict__ nb,
                                                   const TP *__restrict__ pk, const int32_t *__restrict__ blk_case,
                                                   const int32_t *__restrict__ run, const TR *__restrict__ r,
                                                   const float *__restrict__ zin, float *__restrict__ zout,
                                                   float *__restrict__ rc)
{
    if (!case_runs(blk_case, run)) return;
    const int64_t i = blockIdx.x * (int64_t)kW32 + threadIdx.x;
    if (i >= T) return;
    int js[3];
    if (NB)
#pragma unroll
        for (int s = 0; s < 3; ++s) js[s] = nb[s * T + i];
    float y[5][4], c2[8];
    Rows01 own;
#pragma unroll
    for (int l = 0; l < 5; ++l) vload(r, l, T, i, y[l]);
    load_rows<NB != 0 || FULL>(pk, T, i, own, c2);
    if (rc)
#pragma unroll
        for (int l = 0; l < 5; ++l) vstore(rc, l, T, i, y[l]);
    if (NB) {
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            if (!(js[s] >= 0 && js[s] < (int)i)) continue;
            const int64_t j = js[s];
            float z[2][4];
            if (NB == 2) {
                // the neighbour's z^0 = P r, rows 0 and 1, as the separate pass forms it
                float rj[5][4];
                Rows01 n;
#pragma unroll
                for (int l = 0; l < 5; ++l) vload(r, l, T, j, rj[l]);
                load_rows<false>(pk, T, j, n, nullptr);
#pragma unroll
                for (int a = 0; a < 2; ++a) row_times(n.p + 5 * a, rj, nullptr, z[a]);
            } else {
#pragma unroll
                for (int a = 0; a < 2; ++a) vload(zin, a, T, j, z[a]);
            }
            off_acc4(own.a[s], own.x[s], own.y[s], z[0], z[1], y);
        }
    }
    float o[4];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        row_times(own.p + 5 * a, y, nullptr, o);
        vstore(zout, a, T, i, o);
    }
    if (FULL) {
        float p[15], c3[8], c4[2];
        load8(pk, 3, T, i, c3);
        load2(pk, T, i, c4);
#pragma unroll
        for (int q = 0; q < 15; ++q) p[q] = q < 5 ? c2[3 + q] : (q < 13 ? c3[q - 5] : c4[q - 13]);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            row_times(p + 5 * a, y, nullptr, o);
            vstore(zout, 2 + a, T, i, o);
        }
    }
}

// x_i = z_i + P_i y (rows 0 and 1 alone unless FULL), y the sum over the upper neighbours
template <bool FULL, typename TP>
__device__ __forceinline__ void bwd_finish(const TP *__restrict__ pk, int64_t T, int64_t i, const Rows01 &own,
                                           const float *c2, const float (*y)[4], const float *__restrict__ z,
                                           float *__restrict__ xout)
{
    float zi[4], o[4];
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        vload(z, a, T, i, zi);
        row_times(own.p + 5 * a, y, zi, o);
        vstore(xout, a, T, i, o);
    }
    if (FULL) {
        float p[15], c3[8], c4[2];
        load8(pk, 3, T, i, c3);
        load2(pk, T, i, c4);
#pragma unroll
        for (int q = 0; q < 15; ++q) p[q] = q < 5 ? c2[3 + q] : (q < 13 ? c3[q - 5] : c4[q - 13]);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            vload(z, 2 + a, T, i, zi);
            row_times(p + 5 * a, y, zi, o);
            vstore(xout, 2 + a, T, i, o);
        }
    }
}

// Backward relation x_i = z_i + P_i sum_{j>i} O_ij xin_j; FULL as k32_fwd
template <bool FULL, typename TP>
__global__ void __launch_bounds__(kW32, 5) k32_bwd(int64_t T, const int32_t *__restrict__ nb,
                                                   const TP *__restrict__ pk, const int32_t *__restrict__ blk_case,
                                                   const int32_t *__restrict__ run, const float *__restrict__ z,
                                                   const float *__restrict__ xin, float *__restrict__ xout)
{
    if (!case_runs(blk_case, run)) return;
    const int64_t i = blockIdx.x * (int64_t)kW32 + threadIdx.x;
    if (i >= T) return;
    int js[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) js[s] = nb[s * T + i];
    float y[5][4] = {}, c2[8], x[3][2][4];
    Rows01 own;
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        // a slot that is not an upper neighbour reads the cell's own values, discarded
        const int64_t j = js[s] > (int)i ? js[s] : i;
        vload(xin, 0, T, j, x[s][0]);
        vload(xin, 1, T, j, x[s][1]);
    }
    load_rows<true>(pk, T, i, own, c2);
#pragma unroll
    for (int s = 0; s < 3; ++s)
        if (js[s] > (int)i) off_acc4(own.a[s], own.x[s], own.y[s], x[s][0], x[s][1], y);
    bwd_finish<FULL>(pk, T, i, own, c2, y, z, xout);
}

// Two backward sweeps in one launch, x^{q+2} from x^q = xin: each thread forms
// its upper neighbours' x^{q+1} rows 0 and 1 itself, with the arithmetic of
// k32_bwd (the same results bit for bit).
template <bool FULL, typename TP>
__global__ void __launch_bounds__(kW32, 5) k32_bwd2(int64_t T, const int32_t *__restrict__ nb,
                                                    const TP *__restrict__ pk, const int32_t *__restrict__ blk_case,
                                                    const int32_t *__restrict__ run, const float *__restrict__ z,
                                                    const float *__restrict__ xin, float *__restrict__ xout)
{
    if (!case_runs(blk_case, run)) return;
    const int64_t i = blockIdx.x * (int64_t)kW32 + threadIdx.x;
    if (i >= T) return;
    int js[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) js[s] = nb[s * T + i];
    float y[5][4] = {}, c2[8];
    Rows01 own;
    load_rows<true>(pk, T, i, own, c2);
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        if (js[s] <= (int)i) continue;
        const int64_t j = js[s];
        Rows01 n;
        float yj[5][4] = {}, nc2[8], x[3][2][4], x1[2][4], zj[4];
        int ks[3];
#pragma unroll
        for (int t = 0; t < 3; ++t) ks[t] = nb[t * T + j];
        load_rows<true>(pk, T, j, n, nc2);
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            const int64_t k = ks[t] > js[s] ? ks[t] : j;
            vload(xin, 0, T, k, x[t][0]);
            vload(xin, 1, T, k, x[t][1]);
        }
#pragma unroll
        for (int t = 0; t < 3; ++t)
            if (ks[t] > js[s]) off_acc4(n.a[t], n.x[t], n.y[t], x[t][0], x[t][1], yj);
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            vload(z, a, T, j, zj);
            row_times(n.p + 5 * a, yj, zj, x1[a]);
        }
        off_acc4(own.a[s], own.x[s], own.y[s], x1[0], x1[1], y);
    }
    bwd_finish<FULL>(pk, T, i, own, c2, y, z, xout);
}

// ---- operator with the Gram-Schmidt products, update

// u = (K x)_i
__device__ __forceinline__ void apply32(int64_t T, const int32_t *__restrict__ nb, const float4 *__restrict__ op,
                                        const float *__restrict__ x, int64_t i, float (*u)[4])
{
    int js[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) js[s] = nb[s * T + i];
    float xi[5][4], c[24];
#pragma unroll
    for (int l = 0; l < 5; ++l) vload(x, l, T, i, xi[l]);
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        const float4 t = op[q * T + i];
        c[4 * q] = t.x;
        c[4 * q + 1] = t.y;
        c[4 * q + 2] = t.z;
        c[4 * q + 3] = t.w;
    }
    float g[3][2][4];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        // a missing neighbour has a zero block; it reads the cell's own values
        const int64_t j = js[s] >= 0 ? js[s] : i;
        vload(x, 0, T, j, g[s][0]);
        vload(x, 1, T, j, g[s][1]);
    }
    constexpr int kIdx[5][5] = {{0, 1, 2, 3, 4}, {1, 5, 6, 7, 8}, {2, 6, 9, 10, 11}, {3, 7, 10, 12, 13},
                                {4, 8, 11, 13, 14}};
#pragma unroll
    for (int a = 0; a < 5; ++a)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            float s = c[kIdx[a][0]] * xi[0][v];
#pragma unroll
            for (int k = 1; k < 5; ++k) s = fmaf(c[kIdx[a][k]], xi[k][v], s);
            u[a][v] = s;
        }
#pragma unroll
    for (int s = 0; s < 3; ++s) off_acc4(-c[15 + s], c[18 + s], c[21 + s], g[s][0], g[s][1], u);
}

// Block sums of K x 4 FP32 values per thread, sv[k][v]: FP32 within a warp (at
// most 160 products each), FP64 across the warps: part[k0 + k][v][row], k < n.  A warp
// per k adds its four sums, eight lanes each (four FP64 instructions).
template <int K>
__device__ __forceinline__ void block_rows32(float (&sv)[K][4], float (*sh)[K][4], double *__restrict__ part, int k0,
                                             int n = K)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        // the four variables' sums over the warp together: two exchanges that leave
        // each lane one variable, then three that sum it
        const bool hi = lane & 16, odd = lane & 8;
        float a = hi ? sv[k][2] : sv[k][0], b = hi ? sv[k][3] : sv[k][1];
        a += __shfl_xor_sync(0xffffffffu, hi ? sv[k][0] : sv[k][2], 16);
        b += __shfl_xor_sync(0xffffffffu, hi ? sv[k][1] : sv[k][3], 16);
        float s = odd ? b : a;
        s += __shfl_xor_sync(0xffffffffu, odd ? a : b, 8);
        s += __shfl_xor_sync(0xffffffffu, s, 4);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        if ((lane & 7) == 0) sh[warp][k][lane >> 3] = s;
    }
    __syncthreads();
    if (warp < min(K, n)) {
        const int v = lane >> 3;
        double s = double(sh[lane & 7][warp][v]);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((lane & 7) == 0) part[((k0 + warp) * 4 + v) * (int64_t)gridDim.x + blockIdx.x] = s;
    }
}

// Block sums of one value per thread, the variable of a thread being its index mod 4:
// FP64 from the thread on, part[variable][row].
__device__ __forceinline__ void block_quads(double s, double (*sh)[4], double *__restrict__ part)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o >= 4; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane < 4) sh[warp][lane] = s;
    __syncthreads();
    if (warp == 0) {
        s = sh[lane >> 2][lane & 3];
#pragma unroll
        for (int o = 16; o >= 4; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane < 4) part[lane * (int64_t)gridDim.x + blockIdx.x] = s;
    }
}

// y = K z - V_j (gks_solve64.cuh), the products <V_k, y>, k <= j, of the Gram-Schmidt
// pass and |y|^2 (k = j + 1); J > 0: the Arnoldi index j = J - 1 is a compile-time
// constant (all products before one block-wide pass), J = 0: two sums at a time
template <int J>
__global__ void __launch_bounds__(kBlock, 3) k32_apply_dots(int64_t T, const int32_t *__restrict__ nb,
                                                            const float4 *__restrict__ op,
                                                            const int32_t *__restrict__ blk_case,
                                                            const int32_t *__restrict__ run,
                                                            const float *__restrict__ z, float *__restrict__ y,
                                                            const float *__restrict__ V, int j,
                                                            double *__restrict__ part)
{
    constexpr int N = J > 0 ? J + 1 : 2;
    __shared__ float sh[kBlock / 32][N][4];
    if (!case_runs(blk_case, run)) return;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t vs = 20 * T;
    if (J > 0) j = J - 1;
    float u[5][4] = {}, sv[N][4] = {};
    // the last two sums: <V_j, y> and |y|^2
    if (i < T) {
        apply32(T, nb, op, z, i, u);
#pragma unroll
        for (int l = 0; l < 5; ++l) {
            float t[4];
            vload(V + j * vs, l, T, i, t);
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                u[l][v] -= t[v];
                sv[N - 2][v] = fmaf(t[v], u[l][v], sv[N - 2][v]);
                sv[N - 1][v] = fmaf(u[l][v], u[l][v], sv[N - 1][v]);
            }
            vstore(y, l, T, i, u[l]);
        }
    }
    if constexpr (J > 0) {
        if (i < T)
#pragma unroll
            for (int k = 0; k < J - 1; ++k)
#pragma unroll
                for (int l = 0; l < 5; ++l) {
                    float t[4];
                    vload(V + k * vs, l, T, i, t);
#pragma unroll
                    for (int v = 0; v < 4; ++v) sv[k][v] = fmaf(t[v], u[l][v], sv[k][v]);
                }
        block_rows32<N>(sv, sh, part, 0);
    } else {
        block_rows32<N>(sv, sh, part, j);
        for (int k0 = 0; k0 < j; k0 += N) {
            float s2[N][4] = {};
            if (i < T)
#pragma unroll
                for (int k = 0; k < N; ++k) {
                    if (k0 + k >= j) continue;
#pragma unroll
                    for (int l = 0; l < 5; ++l) {
                        float t[4];
                        vload(V + (k0 + k) * vs, l, T, i, t);
#pragma unroll
                        for (int v = 0; v < 4; ++v) s2[k][v] = fmaf(t[v], u[l][v], s2[k][v]);
                    }
                }
            __syncthreads();
            block_rows32<N>(s2, sh, part, k0, j - k0);
        }
    }
}

}  // namespace
}  // namespace gks
