// lbfd_step_small.cuh -- a 2-D step in one launch of one-warp blocks
// (lbfd_step_small.cu, and the forward-mode step of lbfd_tangent.cu).
//
// One warp per block: the first blocks take the boundary cells that the tiles
// leave out (by their neighbourhood codes; the longest-latency work starts
// first), the others a small tile each, with one lane or two lanes (one per
// axis of the FD terms) per cell.  What bounds such grids is not the work
// but where it runs: an SM partition issues one FP64 warp instruction per 64
// cycles whatever its lanes do, so 8192 FP64 cells in 256-thread tiles kept
// 32 of the 152 SMs busy for 64 us; in FP32 it is the latency of one
// warp's instruction chain, a boundary kernel of its own and its two
// events.  Spread one warp per partition, with half of the FD chain per
// lane, the step takes 28 us in FP64 and 4.6 us in FP32 (256x32 channel, in
// a graph; 64 and 13.6 us before).
#pragma once
#include "lbfd_internal.h"
#include "lbfd_step_tiled.cuh"

namespace lbfd {

__device__ __forceinline__ float lane_xor16(float v) { return __shfl_xor_sync(0xffffffffu, v, 16); }
__device__ __forceinline__ double lane_xor16(double v) { return __shfl_xor_sync(0xffffffffu, v, 16); }
template <typename T, int N>
__device__ __forceinline__ Dual<T, N> lane_xor16(const Dual<T, N>& a)
{
    Dual<T, N> r;
    r.v = lane_xor16(a.v);
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = lane_xor16(a.d[k]);
    return r;
}

constexpr int SM_TX = 8, SM_TY = 4;        // one cell per lane
constexpr int SP_TX = 8, SP_TY = 2;        // two lanes per cell
// The tiles take the coded cells too, next to their interior lanes, so that
// only the cells they leave out pay a warp of their own (256x32 channel in
// FP64: 28.4 -> 27.6 us per step, mixed in a graph 5.6 -> 4.5; 17 + 33 + 65
// wide channels of 301 cells 1.10x).  In forward mode the selects of the four
// derivatives cost more than the list (512x64 cells: FP64 321 us against
// 348, mixed 25 against 28), which stays.
template <typename R>
constexpr bool SMALL_CODED = std::is_arithmetic<R>::value;

// The two axes' parts of a cell's FD terms, in the lanes c and c + 16 of a
// warp, summed into both.
template <typename R>
__device__ __forceinline__ void join_axes(FDAccum<R>& acc, R gam, int axis)
{
    auto sum = [](R& v) { v += lane_xor16(v); };
    sum(acc.conv_T);
    sum(acc.diff_T);
    sum(acc.along);
    sum(acc.lamY);
#pragma unroll
    for (int k = 0; k < NSP; ++k) sum(acc.rhs_Y[k]);
    const R other = lane_xor16(gam);
    acc.gam[0] = axis ? other : gam;
    acc.gam[1] = axis ? gam : other;
}

// an interior tile of 16 cells, lane = cell + 16 axis: each lane takes the FD
// terms of one axis, both lanes of a cell the rest (one of them stores)
template <typename S, typename R, bool HI1>
__device__ __forceinline__ void split_tile(const StepParams<R>& P, const S* LBFD_RESTRICT g_in, S* LBFD_RESTRICT g_out,
                                           const S* LBFD_RESTRICT T_in, S* LBFD_RESTRICT T_out,
                                           const S* LBFD_RESTRICT Y_in, S* LBFD_RESTRICT Y_out,
                                           const uint8_t* LBFD_RESTRICT interior,
                                           const unsigned long long* LBFD_RESTRICT cell_codes, int bx, int by)
{
    using G = TileGeom<SP_TX, SP_TY>;
    constexpr int SX = G::SX, NPT = G::NPT;
    constexpr bool CODED = SMALL_CODED<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const TileSmem<R> sm = tile_smem<R, SP_TX, SP_TY>(smem_raw);
    const int lane = threadIdx.x, axis = lane >> 4, tx = lane % SP_TX, ty = (lane / SP_TX) % SP_TY;
    const int x0 = bx * SP_TX, y0 = by * SP_TY, x = x0 + tx, y = y0 + ty;
    const long long c = (long long)x + (long long)P.nx * y;
    const bool inside = x < P.nx && y < P.ny;
    R g[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = R(0);
    bool fast = false;
    unsigned long long code = 0;
    if (inside) {
        const int cls = interior[c];
        fast = cls == 1 || (CODED && cls == 2);
        if (CODED && cls == 2) code = cell_codes[c];
        pull_interior<S, R>(P, g_in, c, x, y, g);
    }
    const bool cw = CODED && __any_sync(0xffffffffu, code != 0);
    stage_tile2d<S, R, SP_TX, SP_TY, CODED, 32>(P, sm, x0, y0, lane, T_in, Y_in);
    __syncwarp();
    if (!__any_sync(0xffffffffu, fast)) return;
    const int p0 = (ty + 2) * SX + tx + 2;
    const R T0 = sm.T[p0], invW0 = sm.invW[p0], rho0 = sm.rho[p0];
    const R inv_rho0 = T0 * invW0 * par<R>(P.inv_rho_c);
    if (CODED && code) pull_coded_tile<S, R>(P, x, y, c, (unsigned)code, rho0, inv_rho0, g_in, g);
    LowMoments<2, R> lm;
    low_moments<2>(g, lm);
    const R u[3] = {lm.m1[0] * (K<R>(3) * inv_rho0), lm.m1[1] * (K<R>(3) * inv_rho0), R(0)};
    FDAccum<R> acc;
    acc.clear();
    R gam;
    fd_axis_smem<CODED, R>(P, sm, NPT, p0, axis ? SX : 1, cw, (unsigned)(code >> (axis ? 38 : 32)) & 63u,
                           (unsigned)(code >> (axis ? 52 : 50)) & 3u, axis ? u[1] : u[0], invW0, inv_rho0, &gam, acc);
    join_axes(acc, gam, axis);
    if (!fast) return;
    R Y0[NSP];
#pragma unroll
    for (int k = 0; k < NSP; ++k) Y0[k] = sm.Y[k * NPT + p0];
    const R rc = rho0 * par<R>(P.inv_rho_c);
    const R Lam = update_scalars<S, R>(P, c, T0, Y0, rc * invW0, rc * T0, acc, T_out, Y_out, axis == 0);
    if constexpr (HI1) collide_hi1<2, R>(P, lm, rho0, inv_rho0, u, acc.gam, Lam, g);
    else collide<2, R>(P, g, rho0, inv_rho0, u, acc.gam, Lam);
    if (axis == 0)
#pragma unroll
        for (int i = 0; i < 9; ++i) g_out[(long long)i * P.N + c] = S(g[i]);
}

// a coded boundary cell the same way
template <typename S, typename R, bool HI1>
__device__ __forceinline__ void split_coded(const StepParams<R>& P, long long c, unsigned long long code, bool store,
                                            const S* LBFD_RESTRICT g_in, S* LBFD_RESTRICT g_out,
                                            const S* LBFD_RESTRICT T_in, S* LBFD_RESTRICT T_out,
                                            const S* LBFD_RESTRICT Y_in, S* LBFD_RESTRICT Y_out)
{
    const int axis = (threadIdx.x >> 4) & 1;
    const int p[3] = {(int)(c % P.nx), (int)(c / P.nx), 0};
    const R T0 = R(T_in[c]);
    R Y0[NSP];
#pragma unroll
    for (int k = 0; k < NSP; ++k) Y0[k] = R(Y_in[(long long)k * P.N + c]);
    const R invW0 = inv_molar_mass(P, Y0);
    R rho0, W0;
    eos_w(P, T0, invW0, rho0, W0);
    const R inv_rho0 = T0 * invW0 * par<R>(P.inv_rho_c), inv_T0 = rho0 * invW0 * par<R>(P.inv_rho_c);
    R g[9];
    pull_coded<2, S, R, true>(P, p, c, code, rho0, inv_rho0, g_in, g);
    LowMoments<2, R> lm;
    low_moments<2>(g, lm);
    const R u[3] = {lm.m1[0] * (K<R>(3) * inv_rho0), lm.m1[1] * (K<R>(3) * inv_rho0), R(0)};
    FDAccum<R> acc;
    acc.clear();
    R gam;
    fd_axis_coded<2, S, R, true>(P, p, c, axis, code, T_in, Y_in, axis ? u[1] : u[0], invW0, inv_rho0, &gam, acc);
    join_axes(acc, gam, axis);
    store = store && axis == 0;
    const R Lam = update_scalars<S, R>(P, c, T0, Y0, inv_T0, W0, acc, T_out, Y_out, store);
    if constexpr (HI1) collide_hi1<2, R>(P, lm, rho0, inv_rho0, u, acc.gam, Lam, g);
    else collide<2, R>(P, g, rho0, inv_rho0, u, acc.gam, Lam);
    if (store)
#pragma unroll
        for (int i = 0; i < 9; ++i) g_out[(long long)i * P.N + c] = S(g[i]);
}

template <typename S, typename R, bool HI1, bool SPLIT>
__global__ void __launch_bounds__(32)
    step_kernel_small2d(StepParams<R> P, const S* LBFD_RESTRICT g_in, S* LBFD_RESTRICT g_out,
                        const S* LBFD_RESTRICT T_in, S* LBFD_RESTRICT T_out, const S* LBFD_RESTRICT Y_in,
                        S* LBFD_RESTRICT Y_out, const uint8_t* LBFD_RESTRICT interior,
                        const unsigned long long* LBFD_RESTRICT cell_codes,
                        const long long* LBFD_RESTRICT cells, const unsigned long long* LBFD_RESTRICT codes, int ncells,
                        int list_blocks, int tiles_x)
{
    const int t = (int)blockIdx.x - list_blocks;
    if constexpr (SPLIT) {
        if (t < 0) {
            // idle lanes of the last block repeat its last cell without storing
            const int j = blockIdx.x * 16 + (threadIdx.x & 15), k = j < ncells ? j : ncells - 1;
            split_coded<S, R, HI1>(P, cells[k], codes[k], j < ncells, g_in, g_out, T_in, T_out, Y_in, Y_out);
        } else {
            split_tile<S, R, HI1>(P, g_in, g_out, T_in, T_out, Y_in, Y_out, interior, cell_codes, t % tiles_x,
                                   t / tiles_x);
        }
    } else {
        if (t < 0) {
            const int j = blockIdx.x * 32 + threadIdx.x;
            if (j >= ncells) return;
            const long long c = cells[j];
            const int p[3] = {(int)(c % P.nx), (int)(c / P.nx), 0};
            cell_step_coded<2, S, R, true, HI1>(P, p, c, codes[j], g_in, g_out, T_in, T_out, Y_in, Y_out);
        } else {
            tiled2d_body<S, R, SM_TX, SM_TY, SMALL_CODED<R>, HI1>(P, g_in, g_out, T_in, T_out, Y_in, Y_out, interior,
                                                                  cell_codes, threadIdx.x % SM_TX,
                                                                  threadIdx.x / SM_TX, t % tiles_x, t / tiles_x);
        }
    }
}

// HI1: omega_hi = 1
template <typename S, typename R, bool HI1, bool SPLIT>
cudaError_t launch_small(const StepParams<R>& P, StateView in, StateView out, const BoundaryLists& b,
                         cudaStream_t stream)
{
    constexpr int TX = SPLIT ? SP_TX : SM_TX, TY = SPLIT ? SP_TY : SM_TY, CELLS = TX * TY;
    constexpr size_t smem = tile_smem_bytes<R, TX, TY>();
    const int gx = (P.nx + TX - 1) / TX, gy = (P.ny + TY - 1) / TY;
    const int n = (int)(SMALL_CODED<R> ? b.all2.nout : b.all2.n), lb = (n + CELLS - 1) / CELLS;
    auto kern = step_kernel_small2d<S, R, HI1, SPLIT>;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    kern<<<lb + gx * gy, 32, smem, stream>>>(P, (const S*)in.g, (S*)out.g, (const S*)in.T, (S*)out.T, (const S*)in.Y,
                                             (S*)out.Y, b.interior, b.cell_codes, b.all2.cells, b.all2.codes, n, lb,
                                             gx);
    return cudaGetLastError();
}

// SM partitions, and warps of 32 cells of a grid
constexpr long long PARTITIONS = 4 * 152;
inline long long small_warps(int nx, int ny)
{
    return (long long)((nx + SM_TX - 1) / SM_TX) * ((ny + SM_TY - 1) / SM_TY);
}

}  // namespace lbfd
