// Fields and sums of the current state f(t): density and velocity, the plane
// profile, and the global mass and momentum.
//
// All of them read the 19 populations of every cell once, as the step's gather
// does, so DRAM bounds them as long as the rest stays small. The one-cell gather
// of k_export with FP64 sums did not: FP64 runs at 1/64 of the FP32 rate here, and
// FP16 storage was read 2 bytes at a time. us a call at 512x128x256, before / now
// (floor, the reads and writes at the copy rate): conservation FP32 3980 / 388 (188),
// FP16 3967 / 266 (94); plane profile FP32 739 / 306, AA 721 / 218 (188), FP16 736 /
// 214 (94); moments FP32 234 / 220 (228), FP16 206 / 158, AA 181 / 133 (134). Here a thread gathers V cells of a row with the wide loads of the
// step kernels (gather_pair, gather_quad), and the sums run in compensated FP32:
// every addition is an error-free transformation (Knuth's two-sum; products with
// their FMA residual), the residuals are added up beside it, and after at most
// SUM_RUN additions the pair of sums is moved to FP64. A run's residual sum is
// itself rounded to 2^-24 of at most SUM_RUN half ulps of the run's sum, about
// 2^-46 of it, independently from run to run.
#pragma once

#include <algorithm>

#include "lbm_handle.h"
#include "lbm_quad.cuh"

namespace lbm {

constexpr int SUM_RUN = 32;   // additions to one compensated sum before it goes to FP64

// Compensated sum of two lanes: hi + lo.
struct Sum2 {
    float2 hi, lo;
};

__device__ __forceinline__ void sum_add(Sum2 &s, float2 v)
{
    const float2 t = add2(s.hi, v), b = sub2(t, s.hi);
    s.lo = add2(s.lo, add2(sub2(s.hi, sub2(t, b)), sub2(v, b)));
    s.hi = t;
}

// s += a b with the product's rounding error
__device__ __forceinline__ void sum_mul(Sum2 &s, float2 a, float2 b)
{
    const float2 v = mul2(a, b);
    s.lo = add2(s.lo, fma2(a, b, make_float2(-v.x, -v.y)));
    sum_add(s, v);
}

// The sum over both lanes in FP64; clears s.
__device__ __forceinline__ double sum_take(Sum2 &s)
{
    const float t = __fadd_rn(s.hi.x, s.hi.y), b = __fsub_rn(t, s.hi.x);
    const float e = __fadd_rn(__fsub_rn(s.hi.x, __fsub_rn(t, b)), __fsub_rn(s.hi.y, b));
    const double v = (double)t + (double)__fadd_rn(e, __fadd_rn(s.lo.x, s.lo.y));
    s.hi = s.lo = bc(0.f);
    return v;
}

// f(t) of V cells as gathered: packed pairs, or for V = 4 the raw words of two
// pairs (converted one pair at a time, to hold half the registers).
template <int V> struct Cells {
    float2 f[Q];
    __device__ __forceinline__ void pair(int, float2 (&out)[Q]) const
    {
#pragma unroll
        for (int a = 0; a < Q; ++a) out[a] = f[a];
    }
};
template <> struct Cells<4> {
    uint2 r[Q];
    __device__ __forceinline__ void pair(int h, float2 (&out)[Q]) const
    {
#pragma unroll
        for (int a = 0; a < Q; ++a) out[a] = h2f(h ? r[a].y : r[a].x);
    }
};

// f(t) of the V cells x0 .. x0 + V - 1 (V = 4: FP16 storage; V = 1: one cell in
// lane x) of row y under the storage map of LAY. The quad gather takes bb_map
// walls as WALL_BB.
template <typename T, int V, int LAY>
__device__ __forceinline__ void gather_cells(const T *src, const Geom &g, int wall, int x0, int y, int z, int lane,
                                             Cells<V> &c)
{
    const int zm = z == 0 ? g.nz - 1 : z - 1, zp = z == g.nz - 1 ? 0 : z + 1;
    if constexpr (V == 4) {
        const int w = bb_map(wall) ? (int)WALL_BB : wall;
        if (y == 0)
            gather_quad<ROW_BOTTOM, LAY>(src, g, w, x0, y, z, zm, zp, lane, c.r);
        else if (y == g.ny - 1)
            gather_quad<ROW_TOP, LAY>(src, g, w, x0, y, z, zm, zp, lane, c.r);
        else
            gather_quad<ROW_INTERIOR, LAY>(src, g, w, x0, y, z, zm, zp, lane, c.r);
    } else if constexpr (V == 2) {
        if (y == 0)
            gather_pair<T, ROW_BOTTOM, LAY>(src, g, wall, x0, y, z, zm, zp, lane, c.f);
        else if (y == g.ny - 1)
            gather_pair<T, ROW_TOP, LAY>(src, g, wall, x0, y, z, zm, zp, lane, c.f);
        else
            gather_pair<T, ROW_INTERIOR, LAY>(src, g, wall, x0, y, z, zm, zp, lane, c.f);
    } else {
        constexpr int MAP = LAY == LAY_PULL ? MAP_PULL : (LAY == LAY_AA_EVEN ? MAP_AA0 : MAP_AA1);
        float s[Q];
        gather<T, MAP>(src, g, wall, x0, y, z, s);
#pragma unroll
        for (int a = 0; a < Q; ++a) c.f[a] = make_float2(s[a], 0.f);
    }
}

// velocity(moments_of(f)) of lbm_kernels.cuh for two cells, the same roundings.
__device__ __forceinline__ PairState state_pair(const float2 (&f)[Q], const Phys &p)
{
    const float2 drho =
        add2(add2(add2(add2(add2(add2(f[0], f[1]), add2(f[2], f[3])), add2(add2(f[4], f[5]), add2(f[6], f[7]))),
                       add2(add2(f[8], f[9]), add2(f[10], f[11]))),
                  add2(add2(f[12], f[13]), add2(f[14], f[15]))),
             add2(add2(f[16], f[17]), f[18]));
    const float2 jx = add2(add2(add2(sub2(f[1], f[2]), sub2(f[7], f[8])), add2(sub2(f[9], f[10]), sub2(f[13], f[14]))),
                           sub2(f[15], f[16]));
    const float2 jy = add2(add2(add2(sub2(f[3], f[4]), sub2(f[7], f[8])), add2(sub2(f[11], f[12]), sub2(f[14], f[13]))),
                           sub2(f[17], f[18]));
    const float2 jz = add2(add2(add2(sub2(f[5], f[6]), sub2(f[9], f[10])), add2(sub2(f[11], f[12]), sub2(f[16], f[15]))),
                           sub2(f[18], f[17]));
    PairState c;
    c.rho = add2(bc(1.f), drho);
    const float2 idev = make_float2(-drho.x / c.rho.x, -drho.y / c.rho.y);
    c.ux = add2(jx, fma2(jx, idev, fma2(bc(p.hF[0]), idev, bc(p.hF[0]))));
    c.uy = add2(jy, fma2(jy, idev, fma2(bc(p.hF[1]), idev, bc(p.hF[1]))));
    c.uz = add2(jz, fma2(jz, idev, fma2(bc(p.hF[2]), idev, bc(p.hF[2]))));
    return c;
}

template <int V> __device__ __forceinline__ void store_cells(float *out, const float2 (&v)[(V + 1) / 2], bool wide)
{
    if constexpr (V == 4) {
        if (wide) {
            *reinterpret_cast<float4 *>(out) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
        } else {
            out[0] = v[0].x;
            out[1] = v[0].y;
            out[2] = v[1].x;
            out[3] = v[1].y;
        }
    } else if constexpr (V == 2) {
        if (wide) {
            *reinterpret_cast<float2 *>(out) = v[0];
        } else {
            out[0] = v[0].x;
            out[1] = v[0].y;
        }
    } else {
        out[0] = v[0].x;
    }
}

// Density and velocity, dense FP32 arrays (either may be null). nx is a multiple
// of V; wide: both arrays are aligned to V floats. grid (row tiles, ny, nz).
template <typename T, int V, int LAY>
__global__ void __launch_bounds__(128) k_moments(const T *__restrict__ src, Geom g, Phys p, float *__restrict__ rho_out,
                                                 float *__restrict__ u_out, bool wide)
{
    const int lane = threadIdx.x & 31, y = blockIdx.y, z = blockIdx.z;
    const int x0 = V * (blockIdx.x * blockDim.x + threadIdx.x);
    const bool valid = x0 < g.nx;
    Cells<V> in;
    gather_cells<T, V, LAY>(src, g, p.wall, valid ? x0 : g.nx - V, y, z, lane, in);
    float2 rho[(V + 1) / 2], ux[(V + 1) / 2], uy[(V + 1) / 2], uz[(V + 1) / 2];
#pragma unroll
    for (int h = 0; h < (V + 1) / 2; ++h) {
        float2 f[Q];
        in.pair(h, f);
        const PairState c = state_pair(f, p);
        rho[h] = c.rho;
        ux[h] = c.ux;
        uy[h] = c.uy;
        uz[h] = c.uz;
    }
    if (!valid) return;
    const long long n = (long long)g.nx * g.ny * g.nz, cell = ((long long)z * g.ny + y) * g.nx + x0;
    if (rho_out) store_cells<V>(rho_out + cell, rho, wide);
    if (u_out) {
        store_cells<V>(u_out + cell, ux, wide);
        store_cells<V>(u_out + n + cell, uy, wide);
        store_cells<V>(u_out + 2 * n + cell, uz, wide);
    }
}

// Sum N <= 16 doubles over the block by reduce-scatter (warp_stats_reduce of
// lbm_kernels.cuh in FP64: 16 additions a lane instead of 5 N), then over the
// warps in order; thread k < N returns sum k in v[0]. All threads must call it.
template <int N>
__device__ __forceinline__ double block_sums(double (&v)[16])
{
    __shared__ double red[4][16];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int h = 8, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const double send = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    const double w = v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
    if (!(lane & 1)) red[warp][lane >> 1] = w;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x < N)
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i][threadIdx.x];
    return s;
}

constexpr float VEL_SCALE = 1073741824.f;   // 2^30

// Whether a cell's terms go to the FP32 sums: rho from 1/2, below which rho - 1
// outweighs the density that its sum stands for, to 2^24, above which the 1 falls
// between two FP32 numbers, and velocities whose products FP32 holds. False for NaN.
__device__ __forceinline__ bool profile_in_range(float rho, float ux, float uy, float uz)
{
    return rho >= 0.5f && rho <= 16777216.f && fabsf(ux) + fabsf(uy) + fabsf(uz) < 1e6f;
}

__device__ __forceinline__ void profile_add_fp64(double (&v)[16], float rho, float fx, float fy, float fz)
{
    const double r = rho, ux = fx, uy = fy, uz = fz;
    v[0] += r;
    v[1] += ux;
    v[2] += uy;
    v[3] += uz;
    v[4] += ux * ux;
    v[5] += uy * uy;
    v[6] += uz * uz;
    v[7] += ux * uy;
    v[8] += r * ux;
    v[9] += r * uy;
    v[10] += r * uz;
}

// Sums over the row tiles blockIdx.x, blockIdx.x + gridDim.x, ... of plane
// blockIdx.y (tile t: row z = t / nxb, cells from V blockDim (t % nxb)):
//   PROFILE  rho, u, u_i^2, u_x u_y, rho u (K_STATS columns of lbm_plane_stats)
//   else     sum of f - w and of e f (4 columns), one compensated sum for each
//            direction, combined in FP64
// to out[(y gridDim.x + blockIdx.x) columns]. The order of the additions depends
// on the grid only, so every layout and storage map gives the same bits.
// CTAs per SM the register budget must allow (us at 512x128x256, 3 / 4 / 5): FP32
// profile 342 / 353 / 306, FP16 profile 222 / 214 / 235, conservation FP32 462 / 386 /
// 415, FP16 262 / 265 / 364.
template <typename T, bool PROFILE> constexpr int SUM_BLOCKS = PROFILE && sizeof(T) == 4 ? 5 : 4;

template <typename T, int V, int LAY, bool PROFILE>
__global__ void __launch_bounds__(128, SUM_BLOCKS<T, PROFILE>) k_plane_sums(const T *__restrict__ src, Geom g, Phys p, int nxb,
                                                       double *__restrict__ out)
{
    constexpr int NP = (V + 1) / 2, NS = PROFILE ? K_STATS : Q, NOUT = PROFILE ? K_STATS : 4;
    const int lane = threadIdx.x & 31, y = blockIdx.y;
    const int tiles = nxb * g.nz;
    Sum2 s[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) s[k].hi = s[k].lo = bc(0.f);
    double v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = 0.0;
    auto take = [&]() {
        if constexpr (PROFILE) {
#pragma unroll
            for (int k = 0; k < NS; ++k)
                v[k] += sum_take(s[k]) * (k >= 4 && k < 8 ? 1.0 / ((double)VEL_SCALE * VEL_SCALE) : 1.0);
        } else {
            v[0] += sum_take(s[0]);
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                const int a = 2 * k + 1;
                const double va = sum_take(s[a]), vb = sum_take(s[a + 1]), d = va - vb;
                v[0] += va + vb;
                if (ex_of(a)) v[1] += ex_of(a) > 0 ? d : -d;
                if (ey_of(a)) v[2] += ey_of(a) > 0 ? d : -d;
                if (ez_of(a)) v[3] += ez_of(a) > 0 ? d : -d;
            }
        }
    };
    int run = 0, cells = 0;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int z = t / nxb, x0 = V * ((t - z * nxb) * blockDim.x + threadIdx.x);
        const bool valid = x0 < g.nx;
        Cells<V> in;
        gather_cells<T, V, LAY>(src, g, p.wall, valid ? x0 : g.nx - V, y, z, lane, in);
        if (valid) {
#pragma unroll
            for (int h = 0; h < NP; ++h) {
                float2 f[Q];
                in.pair(h, f);
                if constexpr (PROFILE) {
                    PairState c = state_pair(f, p);
                    if (V == 1) c.rho.y = 1.f, c.ux.y = c.uy.y = c.uz.y = 0.f;   // the unused lane adds nothing
                    if (profile_in_range(c.rho.x, c.ux.x, c.uy.x, c.uz.x) && profile_in_range(c.rho.y, c.ux.y, c.uy.y, c.uz.y)) {
                        // velocities scaled by 2^30, so that the residuals of small squares stay normal
                        const float2 vx = mul2(c.ux, bc(VEL_SCALE)), vy = mul2(c.uy, bc(VEL_SCALE)),
                                     vz = mul2(c.uz, bc(VEL_SCALE));
                        sum_add(s[0], sub2(c.rho, bc(1.f)));   // exact; the count of these cells is added below
                        cells += V == 1 ? 1 : 2;
                        sum_add(s[1], c.ux);
                        sum_add(s[2], c.uy);
                        sum_add(s[3], c.uz);
                        sum_mul(s[4], vx, vx);
                        sum_mul(s[5], vy, vy);
                        sum_mul(s[6], vz, vz);
                        sum_mul(s[7], vx, vy);
                        sum_mul(s[8], c.rho, c.ux);
                        sum_mul(s[9], c.rho, c.uy);
                        sum_mul(s[10], c.rho, c.uz);
                    } else {
                        profile_add_fp64(v, c.rho.x, c.ux.x, c.uy.x, c.uz.x);
                        if (V > 1) profile_add_fp64(v, c.rho.y, c.ux.y, c.uy.y, c.uz.y);
                    }
                } else {
#pragma unroll
                    for (int a = 0; a < Q; ++a) sum_add(s[a], f[a]);
                }
            }
        }
        if (++run * NP >= SUM_RUN) {
            take();
            run = 0;
        }
    }
    take();
    if (PROFILE) v[0] += (double)cells;
    const double r = block_sums<NOUT>(v);
    if (threadIdx.x < NOUT) out[((long long)y * gridDim.x + blockIdx.x) * NOUT + threadIdx.x] = r;
}

// Cells a thread gathers at once on rows of nx cells.
inline int cells_wide(const lbm_handle *h)
{
    return h->g.nx % 2 ? 1 : (h->precision == LBM_FP16_SHIFTED && h->g.nx % 4 == 0 ? 4 : 2);
}

// CTAs of k_plane_sums for each plane: about four rounds of the four CTAs an SM
// holds of the 152 of this GPU over all planes, at most one for each row tile and
// `most`. (More rounds shorten the runs between the FP64 sums, fewer leave SMs
// idle at the end.)
inline int plane_sum_blocks(const lbm_handle *h, int most)
{
    const int v = cells_wide(h), per_row = h->g.nx / v, bx = row_threads(per_row);
    const long long tiles = (long long)((per_row + bx - 1) / bx) * h->g.nz;
    const int want = std::max(1, 4 * 4 * 152 / h->g.ny);
    return (int)std::min<long long>(std::min<long long>(want, most), tiles);
}

template <bool PROFILE, typename T, int V>
void plane_sums_v(const lbm_handle *h, int blocks, double *out)
{
    const int per_row = h->g.nx / V, bx = row_threads(per_row), nxb = (per_row + bx - 1) / bx;
    const dim3 grid(blocks, h->g.ny);
    const T *src = (const T *)lbm_state_ptr(h);
    const int map = lbm_state_map(h);
    if (map == MAP_AA0)
        k_plane_sums<T, V, LAY_AA_EVEN, PROFILE><<<grid, bx, 0, h->stream>>>(src, h->g, h->p, nxb, out);
    else if (map == MAP_AA1)
        k_plane_sums<T, V, LAY_AA_ODD, PROFILE><<<grid, bx, 0, h->stream>>>(src, h->g, h->p, nxb, out);
    else
        k_plane_sums<T, V, LAY_PULL, PROFILE><<<grid, bx, 0, h->stream>>>(src, h->g, h->p, nxb, out);
}

// k_plane_sums over the current state on the handle's stream.
template <bool PROFILE>
void plane_sums(const lbm_handle *h, int blocks, double *out)
{
    const bool half = h->precision == LBM_FP16_SHIFTED;
    switch (cells_wide(h)) {
    case 1: half ? plane_sums_v<PROFILE, __half, 1>(h, blocks, out) : plane_sums_v<PROFILE, float, 1>(h, blocks, out); break;
    case 2: half ? plane_sums_v<PROFILE, __half, 2>(h, blocks, out) : plane_sums_v<PROFILE, float, 2>(h, blocks, out); break;
    default: plane_sums_v<PROFILE, __half, 4>(h, blocks, out);
    }
}

}  // namespace lbm
