// Fields and sums of the current state f(t): density and velocity, the plane
// profile, and the global mass and momentum.
//
// All of them read the 19 populations of every cell once, as the step's gather
// does, so DRAM bounds them as long as the rest stays small. The one-cell gather
// of k_export with FP64 sums did not: FP64 runs at 1/64 of the FP32 rate here, and
// FP16 storage was read 2 bytes at a time. us a call at 512x128x256, before / now
// (floor, the reads and writes at the copy rate): conservation FP32 3980 / 388 (188),
// AA 302, FP16 3967 / 300 (94), AA 229; plane profile FP32 739 / 320, AA 721 / 241 (188),
// FP16 736 / 282 (94), AA 208; moments FP32 234 / 220 (228: a pass that mostly reads
// can beat the copy rate), FP16 206 / 158, AA 181 / 133 (134).
// Here a thread gathers V cells of a row with the wide loads of the step kernels
// (gather_pair, gather_quad), and the sums run in FP32 without loss against FP64:
// every addition is an error-free transformation (Knuth's two-sum; products with
// their FMA residual), its error is added to a second word error-free, and only the
// errors of those additions to a third, with rounding. After n <= SUM_RUN cells the
// three words move to FP64. With M the largest partial sum the second word stays
// below 2 n 2^-24 M, the third below (2 n)^2 2^-48 M, so its roundings add up to less
// than (2 n)^3 2^-72 M (2^-48 M for 128 cells, half the terms where a cell adds no
// product); n additions in FP64 may lose n 2^-53 M, 2^-46 M.
#pragma once

#include <algorithm>

#include "lbm_handle.h"
#include "lbm_quad.cuh"

namespace lbm {

constexpr int SUM_RUN = 128;   // cells in one compensated sum before it goes to FP64

// a + b = s + e exactly, in both lanes.
__device__ __forceinline__ float2 two_sum(float2 a, float2 b, float2 &e)
{
    const float2 s = add2(a, b), t = sub2(s, a);
    e = add2(sub2(a, sub2(s, t)), sub2(b, t));
    return s;
}

// Two sums hi + mid + lo of FP32 terms, one a lane. mid takes the rounding
// errors of hi and lo those of mid.
struct Sum3 {
    float2 hi, mid, lo;
};

__device__ __forceinline__ void sum_residual(Sum3 &s, float2 r)
{
    float2 e;
    s.mid = two_sum(s.mid, r, e);
    s.lo = add2(s.lo, e);
}

__device__ __forceinline__ void sum_add(Sum3 &s, float2 v)
{
    float2 e;
    s.hi = two_sum(s.hi, v, e);
    sum_residual(s, e);
}

// s += a b with the products' rounding errors
__device__ __forceinline__ void sum_mul(Sum3 &s, float2 a, float2 b)
{
    const float2 v = mul2(a, b);
    sum_residual(s, fma2(a, b, make_float2(-v.x, -v.y)));
    sum_add(s, v);
}

// Both sums in FP64; clears s.
__device__ __forceinline__ double2 sum_take(Sum3 &s)
{
    const double2 v = make_double2((double)s.hi.x + ((double)s.mid.x + (double)s.lo.x),
                                   (double)s.hi.y + ((double)s.mid.y + (double)s.lo.y));
    s.hi = s.mid = s.lo = bc(0.f);
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
// between two FP32 numbers, and velocities whose products FP32 holds, and whose
// products' errors it holds exactly: each 0 or at least 2^-81 (2^-51 scaled). False
// for NaN.
__device__ __forceinline__ bool profile_in_range(float rho, float ux, float uy, float uz)
{
    const float ax = fabsf(ux), ay = fabsf(uy), az = fabsf(uz);
    // 0 wraps round to the largest word
    const unsigned least = min(__float_as_uint(ax) - 1u, min(__float_as_uint(ay) - 1u, __float_as_uint(az) - 1u));
    return rho >= 0.5f && rho <= 16777216.f && ax + ay + az < 1e6f && least >= ((127u - 81u) << 23) - 1u;
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
//   else     sum of f - w and of e f (4 columns), one sum for each direction,
//            combined in FP64
// to out[(y gridDim.x + blockIdx.x) columns]. The two lanes of a sum hold two columns
// (or opposite directions) of one cell, not one column of two cells: half the
// registers for the same packed additions. The order of the additions depends on the
// grid only, so every layout and storage map gives the same bits.
// CTAs per SM the register budget must allow (us at 512x128x256 with sixteen CTAs an
// SM in all, 3 / 4 / 5 / 6): FP32 profile 388 / 412 / 337 / 362, AA 232 / 235 / 258 /
// 253, conservation 450 / 459 / 415 / 573, AA 315 / 294 / 328 / 450; FP16 profile 278 /
// 283 / 300 / 304, conservation 302 / 299 / 340 / 400.
template <typename T, int LAY> constexpr int SUM_BLOCKS = sizeof(T) == 4 && LAY == LAY_PULL ? 5 : 4;

template <typename T, int V, int LAY, bool PROFILE>
__global__ void __launch_bounds__(128, SUM_BLOCKS<T, LAY>) k_plane_sums(const T *__restrict__ src, Geom g, Phys p, int nxb,
                                                                         double *__restrict__ out)
{
    constexpr int NP = (V + 1) / 2, NS = PROFILE ? (K_STATS + 1) / 2 : (Q + 1) / 2, NOUT = PROFILE ? K_STATS : 4;
    const int lane = threadIdx.x & 31, y = blockIdx.y;
    const int tiles = nxb * g.nz;
    Sum3 s[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) s[k].hi = s[k].mid = s[k].lo = bc(0.f);
    double v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = 0.0;
    auto take = [&]() {
        if constexpr (PROFILE) {
            const double s1 = 1.0 / (double)VEL_SCALE, s2 = s1 * s1;
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                const double2 t = sum_take(s[k]);
                const double scale = k < 2 ? 1.0 : (k < 4 ? s2 : s1);
                v[2 * k] += t.x * scale;
                if (2 * k + 1 < K_STATS) v[2 * k + 1] += t.y * scale;
            }
        } else {
            const double2 rest = sum_take(s[9]);
            v[0] += rest.x + rest.y;
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                const int a = 2 * k + 1;
                const double2 t = sum_take(s[k]);
                const double d = t.x - t.y;
                v[0] += t.x + t.y;
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
                    const PairState c = state_pair(f, p);
#pragma unroll
                    for (int l = 0; l < (V == 1 ? 1 : 2); ++l) {
                        const float rho = l ? c.rho.y : c.rho.x, ux = l ? c.ux.y : c.ux.x, uy = l ? c.uy.y : c.uy.x,
                                    uz = l ? c.uz.y : c.uz.x;
                        if (profile_in_range(rho, ux, uy, uz)) {
                            // velocities scaled by 2^30, so that the errors of small products stay normal
                            const float2 vxy = make_float2(ux * VEL_SCALE, uy * VEL_SCALE);
                            const float vz = uz * VEL_SCALE;
                            sum_add(s[0], make_float2(__fsub_rn(rho, 1.f), ux));   // exact; these cells are counted in below
                            ++cells;
                            sum_add(s[1], make_float2(uy, uz));
                            sum_mul(s[2], vxy, vxy);
                            sum_mul(s[3], make_float2(vz, vxy.x), make_float2(vz, vxy.y));
                            sum_mul(s[4], bc(rho), vxy);
                            sum_mul(s[5], make_float2(rho, 0.f), make_float2(vz, 0.f));
                        } else {
                            profile_add_fp64(v, rho, ux, uy, uz);
                        }
                    }
                } else {
                    sum_add(s[9], f[0]);
#pragma unroll
                    for (int k = 0; k < 9; ++k) {
                        sum_add(s[k], make_float2(f[2 * k + 1].x, f[2 * k + 2].x));
                        if (V > 1) sum_add(s[k], make_float2(f[2 * k + 1].y, f[2 * k + 2].y));
                    }
                }
            }
        }
        run += V;
        if (run + V > SUM_RUN) {
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

// CTAs of k_plane_sums for each plane: five rounds of the four CTAs an SM holds of
// the 152 of this GPU over all planes (four of the five in two-lattice FP32), at most
// one for each row tile and `most`. The number of SMs is written out, as the order of
// the additions must not depend on the device. us at 512x128x256 with one / two /
// three / four rounds of five: FP32 profile 439 / 352 / 327 / 320, conservation 529 /
// 401 / 391 / 388; of four: FP16 profile 369 / 303 / 286 / 281, conservation 402 / 306 /
// 297 / 296.
inline int plane_sum_blocks(const lbm_handle *h, int most)
{
    const int v = cells_wide(h), per_row = h->g.nx / v, bx = row_threads(per_row);
    const long long tiles = (long long)((per_row + bx - 1) / bx) * h->g.nz;
    const int want = std::max(1, 5 * 4 * 152 / h->g.ny);
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
