// Fields and sums of the current state f(t): density and velocity, the plane
// profile, and the global mass and momentum.
//
// All of them read the 19 populations of every cell once, as the step's gather
// does, so DRAM bounds them as long as the rest stays small. The one-cell gather
// of k_export with FP64 sums did not: FP64 runs at 1/64 of the FP32 rate here, and
// FP16 storage was read 2 bytes at a time. us a call at 512x128x256, before / now
// (floor, the reads and writes at the copy rate): conservation FP32 3980 / 367 (188),
// AA 277, FP16 3967 / 289 (94), AA 225; plane profile FP32 739 / 326, AA 721 / 219 (188),
// FP16 736 / 261 (94), AA 204; moments FP32 234 / 220 (228: a pass that mostly reads
// can beat the copy rate), FP16 206 / 158, AA 181 / 133 (134).
// Here a thread gathers V cells of a row with the wide loads of the step kernels
// (gather_pair, gather_quad), and the sums run in FP32 without loss against FP64:
// every addition is an error-free transformation (Knuth's two-sum; products with
// their FMA residual), its error is added to a second word error-free, and only the
// errors of those additions to a third, with rounding. After n <= SUM_RUN cells the
// three words are renormalised. With M the largest partial sum the second word stays
// below 2 n 2^-24 M, the third below (2 n)^2 2^-48 M, so its roundings in a run add up
// to less than (2 n)^3 2^-72 M (2^-48 M for 128 cells, an eighth where a cell adds no
// product); n additions in FP64 may lose n 2^-53 M, 2^-46 M. Lanes and warps add their
// words the same way, so that a block spends some thirty FP64 instructions: with the
// words of every thread moved to FP64 it spent 165 a warp, 105 us of a call, which small
// grids paid in full (conservation of 256x64x128 FP32 175 us, now 105; profile 90, now 64).
#pragma once

#include <algorithm>

#include "lbm_handle.h"
#include "lbm_quad.cuh"

namespace lbm {

constexpr int SUM_RUN = 128;   // cells added to one sum before it is renormalised

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

// The same sums with mid no more than an ulp of hi and lo of mid, exactly.
__device__ __forceinline__ void sum_renormalise(Sum3 &s)
{
    float2 e;
    s.hi = two_sum(s.hi, s.mid, e);
    s.mid = two_sum(e, s.lo, s.lo);
}

// s += o
__device__ __forceinline__ void sum_merge(Sum3 &s, const Sum3 &o)
{
    float2 e;
    s.hi = two_sum(s.hi, o.hi, e);
    sum_residual(s, e);
    sum_residual(s, o.mid);
    s.lo = add2(s.lo, o.lo);
}

// Both sums in FP64.
__device__ __forceinline__ double2 sum_value(const Sum3 &s)
{
    return make_double2((double)s.hi.x + ((double)s.mid.x + (double)s.lo.x),
                        (double)s.hi.y + ((double)s.mid.y + (double)s.lo.y));
}

__device__ __forceinline__ float2 shfl_xor2(float2 v, int o)
{
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}

// Sum N Sum3 over the warp by reduce-scatter: lane l returns sum l / (32 / P) in
// s[0], P the power of two from N up (lanes beyond sum N - 1 return others' copies).
template <int N>
__device__ __forceinline__ void warp_sums(Sum3 (&s)[N], int lane)
{
    constexpr int P = N > 8 ? 16 : 8;
    static_assert(N > 4 && N <= 16, "six sums of a profile, ten of the directions");
#pragma unroll
    for (int h = P / 2, o = 16; o >= 1; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < (h ? h : 1); ++i) {
            Sum3 send = s[i], keep = s[i];
            if (h && i + h < N) {
                send.hi = up ? s[i].hi : s[i + h].hi, keep.hi = up ? s[i + h].hi : s[i].hi;
                send.mid = up ? s[i].mid : s[i + h].mid, keep.mid = up ? s[i + h].mid : s[i].mid;
                send.lo = up ? s[i].lo : s[i + h].lo, keep.lo = up ? s[i + h].lo : s[i].lo;
            }
            send.hi = shfl_xor2(send.hi, o);
            send.mid = shfl_xor2(send.mid, o);
            send.lo = shfl_xor2(send.lo, o);
            sum_merge(keep, send);
            s[i] = keep;
        }
    }
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
    return rho >= 0.5f && rho <= 16777216.f && ax + ay + az < 65536.f && least >= ((127u - 81u) << 23) - 1u;
}

__device__ __forceinline__ void profile_add_fp64(double (*v)[128], float rho, float fx, float fy, float fz)
{
    const double r = rho, ux = fx, uy = fy, uz = fz;
    const double t[K_STATS] = {r, ux, uy, uz, ux * ux, uy * uy, uz * uz, ux * uy, r * ux, r * uy, r * uz};
#pragma unroll
    for (int k = 0; k < K_STATS; ++k) v[k][threadIdx.x] += t[k];
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
// CTAs per SM the register budget must allow (us at 512x128x256, 4 / 5): FP32 profile
// 326 / 366, AA 231 / 219, conservation 466 / 367, AA 278 / 290; FP16 profile 262 / 270,
// AA 205 / 210, conservation 291 / 302, AA 226 / 250; 6 is slower than both.
template <typename T, int LAY, bool PROFILE> constexpr int SUM_BLOCKS = sizeof(T) == 4 && PROFILE != (LAY == LAY_PULL) ? 5 : 4;

template <typename T, int V, int LAY, bool PROFILE>
__global__ void __launch_bounds__(128, SUM_BLOCKS<T, LAY, PROFILE>) k_plane_sums(const T *__restrict__ src, Geom g, Phys p, int nxb,
                                                                         double *__restrict__ out)
{
    constexpr int NP = (V + 1) / 2, NS = PROFILE ? (K_STATS + 1) / 2 : (Q + 1) / 2, NOUT = PROFILE ? K_STATS : 4;
    __shared__ Sum3 red[4][NS];
    __shared__ int count[4];
    __shared__ double beyond[PROFILE ? K_STATS : 1][128];   // terms that FP32 does not hold, a column a thread
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, y = blockIdx.y;
    const int tiles = nxb * g.nz;
    Sum3 s[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) s[k].hi = s[k].mid = s[k].lo = bc(0.f);
    if (PROFILE) {
#pragma unroll
        for (int k = 0; k < K_STATS; ++k) beyond[k][threadIdx.x] = 0.0;
    }
    bool fp64 = false;
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
                            profile_add_fp64(beyond, rho, ux, uy, uz);
                            fp64 = true;
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
#pragma unroll
            for (int k = 0; k < NS; ++k) sum_renormalise(s[k]);
            run = 0;
        }
    }
    warp_sums<NS>(s, lane);
    constexpr int LANES = NS > 8 ? 2 : 4;   // lanes that return a sum
    if (lane % LANES == 0 && lane / LANES < NS) red[warp][lane / LANES] = s[0];
    if (PROFILE) {
        const int c = __reduce_add_sync(0xffffffffu, cells);
        if (lane == 0) count[warp] = c;
    }
    fp64 = __syncthreads_or(fp64);
    if (warp != 0) return;
    const int warps = blockDim.x >> 5;
    Sum3 t = red[0][min(lane, NS - 1)];
    for (int w = 1; w < warps; ++w) sum_merge(t, red[w][min(lane, NS - 1)]);
    double2 v = sum_value(t);
    out += ((long long)y * gridDim.x + blockIdx.x) * NOUT;
    if constexpr (PROFILE) {
        if (lane >= NS) return;
        const bool last = 2 * lane + 1 >= K_STATS;
        if (lane > 1) {
            const double scale = 1.0 / (double)VEL_SCALE * (lane < 4 ? 1.0 / (double)VEL_SCALE : 1.0);
            v = make_double2(v.x * scale, v.y * scale);
        }
        if (lane == 0)
            for (int w = 0; w < warps; ++w) v.x += (double)count[w];
        if (fp64)
            for (int i = 0; i < (int)blockDim.x; ++i) {
                v.x += beyond[2 * lane][i];
                if (!last) v.y += beyond[2 * lane + 1][i];
            }
        out[2 * lane] = v.x;
        if (!last) out[2 * lane + 1] = v.y;
    } else {
        // sums 0 .. 8 hold directions a = 2 k + 1 and a + 1 = opp(a), sum 9 the rest population of both cells
        const int a = lane < 9 ? 2 * lane + 1 : 0;
        const double d = v.x - v.y;
        double r[4] = {lane < NS ? v.x + v.y : 0.0, ex_of(a) * d, ey_of(a) * d, ez_of(a) * d};
#pragma unroll
        for (int o = 8; o >= 1; o >>= 1)
#pragma unroll
            for (int k = 0; k < 4; ++k) r[k] += __shfl_xor_sync(0xffffffffu, r[k], o);
        if (lane < 4) out[lane] = lane == 0 ? r[0] : (lane == 1 ? r[1] : (lane == 2 ? r[2] : r[3]));
    }
}

// Cells a thread gathers at once on rows of nx cells.
inline int cells_wide(const lbm_handle *h)
{
    return h->g.nx % 2 ? 1 : (h->precision == LBM_FP16_SHIFTED && h->g.nx % 4 == 0 ? 4 : 2);
}

// CTAs of k_plane_sums for each plane: five rounds of the four CTAs an SM holds of
// the 152 of this GPU over all planes, at most one for each row tile and `most`. The
// number of SMs is written out, as the order of the additions must not depend on the
// device. us with 16 / 20 / 24 / 30 CTAs an SM, FP32 on two lattices: 512x128x256 profile
// 335 / 326 / 318 / 313, conservation 388 / 365 / 359 / 362; 446x16x157 43 / 44 / 48 / 50
// and 91 / 93 / 89 / 99; 256x64x128 63 / 64 / 66 / 66 and 106 / 105 / 112 / 114.
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
