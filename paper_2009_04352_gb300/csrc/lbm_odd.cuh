// Two cells per thread on rows of an odd number of cells.
//
// The one-cell kernel loads and stores one element per direction and thread,
// with a 64-bit address each, and holds half the bytes in flight a warp could
// (FP32 255x65x127: 61 us a step, 76% of the copy rate; FP16 53 us, 44%). Rows are
// padded to 32 elements, so pairs (x0, x0 + 1), x0 even, can be loaded 2-wide
// up to the end; only the last thread of a row holds a single cell, whose right
// neighbour is cell 0. The collision stays collide() cell by cell, so the
// populations are the one-cell kernel's bit for bit; sampled steps and wall nodes
// run that kernel.
#pragma once

#include "lbm_pair.cuh"

namespace lbm {

// row_pair of lbm_pair.cuh where nx is odd.
template <typename T, int SH, bool NC>
__device__ __forceinline__ float2 row_pair_odd(const T *row, int x0, int nx, int lane)
{
    const float2 v = NC ? ld2<T>(row + x0) : ldc2<T>(row + x0);
    if (SH == 0) return v;
    if (SH == 1) {
        float l = __shfl_up_sync(0xffffffffu, v.y, 1);
        if (lane == 0 || x0 == 0) l = ldx<T, NC>(row + (x0 == 0 ? nx - 1 : x0 - 1));
        return make_float2(l, v.x);
    }
    // the right neighbour of the pair, or of a single last cell (cell 0): one
    // predicated load, as branches here would split the gather
    const bool single = x0 + 1 >= nx;
    float r = __shfl_down_sync(0xffffffffu, v.x, 1);
    if (lane == 31 || single) r = ldx<T, NC>(row + (single ? 0 : x0 + 2));
    return make_float2(single ? r : v.y, r);
}

template <typename T, int ROW, int LAY>
__device__ __forceinline__ void gather_odd(const T *src, const Geom &g, int wall, int x0, int y, int z, int zm, int zp,
                                           int lane, float2 (&f)[Q])
{
    constexpr bool NC = LAY == LAY_PULL && pull_nc<T>;
#pragma unroll
    for (int a = 0; a < Q; ++a) {
        const int ex = ex_of(a), ey = ey_of(a), ez = ez_of(a);
        if (LAY == LAY_AA_EVEN) {
            f[a] = ldc2<T>(src + (long long)a * g.plane + ((long long)z * g.ny + y) * g.sx + x0);
            continue;
        }
        const bool crosses = (ROW == ROW_BOTTOM && ey == 1) || (ROW == ROW_TOP && ey == -1);
        const int zs = ez == 1 ? zm : (ez == -1 ? zp : z);
        if (crosses && bb_map(wall)) {
            const int s = LAY == LAY_AA_ODD ? a : opp_of(a);
            f[a] = row_pair_odd<T, 0, NC>(src + (long long)s * g.plane + ((long long)z * g.ny + y) * g.sx, x0, g.nx, lane);
        } else {
            const int m = crosses ? mirror_of(a) : a, s = LAY == LAY_AA_ODD ? opp_of(m) : m;
            const T *row = src + (long long)s * g.plane + ((long long)zs * g.ny + (crosses ? y : y - ey)) * g.sx;
            f[a] = ex == 1 ? row_pair_odd<T, 1, NC>(row, x0, g.nx, lane)
                           : (ex == -1 ? row_pair_odd<T, -1, NC>(row, x0, g.nx, lane)
                                       : row_pair_odd<T, 0, NC>(row, x0, g.nx, lane));
        }
    }
}

// push_row of lbm_pair.cuh where nx is odd: every element is written once, and
// with SH = 0 the first element of the row padding too. All 32 lanes must call it.
template <typename T, int SH>
__device__ __forceinline__ void push_row_odd(T *row, int x0, int nx, int lane, bool valid, float2 v)
{
    const bool two = x0 + 1 < nx, first = lane == 0 || x0 == 0;
    if (SH == 0) {
        if (valid) st2<T>(row + x0, v);
        return;
    }
    if (SH == 1) {   // cells x0, x0 + 1 -> x0 + 1, x0 + 2; the single last cell -> 0
        const float l = __shfl_up_sync(0xffffffffu, v.y, 1);
        if (!valid) return;
        if (two) {
            if (first)
                st<T>(row + x0 + 1, v.x);
            else
                st2<T>(row + x0, make_float2(l, v.x));
            if (lane == 31) st<T>(row + x0 + 2, v.y);
        } else {
            if (!first) st<T>(row + x0, l);
            st<T>(row, v.x);
        }
        return;
    }
    // SH == -1: cells x0, x0 + 1 -> x0 - 1, x0
    const float r = __shfl_down_sync(0xffffffffu, v.x, 1);
    if (!valid) return;
    if (two) {
        if (lane == 31)
            st<T>(row + x0, v.y);
        else
            st2<T>(row + x0, make_float2(v.y, r));
    }
    if (first) st<T>(row + (x0 == 0 ? nx - 1 : x0 - 1), v.x);
}

template <typename T, int ROW>
__device__ __forceinline__ void push_odd(T *dst, const Geom &g, int wall, int x0, int y, int z, int zm, int zp, int lane,
                                         bool valid, const float2 (&f)[Q])
{
#pragma unroll
    for (int a = 0; a < Q; ++a) {
        const int ex = ex_of(a), ey = ey_of(a), ez = ez_of(a);
        const bool crosses = (ROW == ROW_BOTTOM && ey == -1) || (ROW == ROW_TOP && ey == 1);
        const int zt = ez == 1 ? zp : (ez == -1 ? zm : z);
        if (crosses && bb_map(wall)) {
            push_row_odd<T, 0>(dst + (long long)opp_of(a) * g.plane + ((long long)z * g.ny + y) * g.sx, x0, g.nx, lane, valid,
                               f[a]);
        } else {
            T *row = dst + (long long)(crosses ? mirror_of(a) : a) * g.plane +
                     ((long long)zt * g.ny + (crosses ? y : y + ey)) * g.sx;
            if (ex == 1)
                push_row_odd<T, 1>(row, x0, g.nx, lane, valid, f[a]);
            else if (ex == -1)
                push_row_odd<T, -1>(row, x0, g.nx, lane, valid, f[a]);
            else
                push_row_odd<T, 0>(row, x0, g.nx, lane, valid, f[a]);
        }
    }
}

// Resident CTAs per SM the register budget must allow. us a step at 255x65x127, the
// one-cell kernel / 6 / 5 / 4 CTAs: FP32 60.8 / 49.2 / 55.3 / 61.8, AA 61.5 / 49.1 / 51.1
// / 53.8, MRT 65.4 / 56.2 / 51.1 / 64.6; FP16 53.3 / 40.5 / 39.7 / 43.3, AA 53.4 / 46.8 /
// 43.9 / 43.6, MRT 60.7 / 47.1 / 44.6 / 47.0.
template <typename T, int COLL> constexpr int ODD_BLOCKS = sizeof(T) == 4 && COLL == COLL_BGK ? 6 : 5;

// A plain step (halfway walls) over the row set ROWS; grid (row tiles, rows, nz).
template <typename T, int COLL, int LAY, int ROWS, bool REV>
__global__ void __launch_bounds__(128, ODD_BLOCKS<T, COLL>)
    k_step_odd(const T *src, T *dst, Geom g, Phys p, float *__restrict__ tw_out)
{
    pdl_begin();
    int y, z;
    row_of_block<ROWS, REV>(g, y, z);
    const int lane = threadIdx.x & 31;
    const int x0 = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    const bool valid = x0 < g.nx, two = x0 + 1 < g.nx;
    const int xl = valid ? x0 : g.nx - 1;   // lanes past the row end read in bounds and store nothing
    const int zm = z == 0 ? g.nz - 1 : z - 1, zp = z == g.nz - 1 ? 0 : z + 1;
    float2 f[Q];
    if (ROWS != ROWS_INTERIOR && y == 0)
        gather_odd<T, ROW_BOTTOM, LAY>(src, g, p.wall, xl, y, z, zm, zp, lane, f);
    else if (ROWS != ROWS_INTERIOR && y == g.ny - 1)
        gather_odd<T, ROW_TOP, LAY>(src, g, p.wall, xl, y, z, zm, zp, lane, f);
    else
        gather_odd<T, ROW_INTERIOR, LAY>(src, g, p.wall, xl, y, z, zm, zp, lane, f);

    const float smag = row_smag(p, y, g.ny);
    PairState c;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float in[Q], out[Q];
#pragma unroll
        for (int a = 0; a < Q; ++a) in[a] = h ? f[a].y : f[a].x;
        const CellState s = collide<COLL>(in, out, p, smag);
#pragma unroll
        for (int a = 0; a < Q; ++a) (h ? f[a].y : f[a].x) = out[a];
        (h ? c.rho.y : c.rho.x) = s.rho;
        (h ? c.ux.y : c.ux.x) = s.ux;
        (h ? c.uy.y : c.uy.x) = s.uy;
        (h ? c.uz.y : c.uz.x) = s.uz;
    }
    if (ROWS != ROWS_INTERIOR && (y == 0 || y == g.ny - 1)) {
        float2 twx, twz;
        if (!two) {   // the lane past a single last cell solves the same wall law
            c.rho.y = c.rho.x;
            c.ux.y = c.ux.x;
            c.uy.y = c.uy.x;
            c.uz.y = c.uz.x;
        }
        wall_layer_pair(f, c, p, y == 0, twx, twz);
        if (valid) {
            float2 *t = reinterpret_cast<float2 *>(tw_out) + ((long long)((y == 0 ? 0 : 1) * g.nz + z) * g.nx + x0);
            t[0] = make_float2(twx.x, twz.x);
            if (two) t[1] = make_float2(twx.y, twz.y);
        }
    }
    if (LAY == LAY_AA_ODD) {
        if (ROWS != ROWS_INTERIOR && y == 0)
            push_odd<T, ROW_BOTTOM>(dst, g, p.wall, xl, y, z, zm, zp, lane, valid, f);
        else if (ROWS != ROWS_INTERIOR && y == g.ny - 1)
            push_odd<T, ROW_TOP>(dst, g, p.wall, xl, y, z, zm, zp, lane, valid, f);
        else
            push_odd<T, ROW_INTERIOR>(dst, g, p.wall, xl, y, z, zm, zp, lane, valid, f);
    } else {
        T *d = dst + ((long long)z * g.ny + y) * g.sx;
#pragma unroll
        for (int a = 0; a < Q; ++a)
            push_row_odd<T, 0>(d + (LAY == LAY_AA_EVEN ? opp_of(a) : a) * g.plane, xl, g.nx, lane, valid, f[a]);
    }
}

}  // namespace lbm
