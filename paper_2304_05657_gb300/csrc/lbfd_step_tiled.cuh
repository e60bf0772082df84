// lbfd_step_tiled.cuh -- 2-D fused coupled step with shared-memory staging.
//
// A block owns a TX x TY tile of cells.  It stages T, Y_k and the derived
// point values 1/W, X_k and rho of the tile plus a 2-cell halo in shared
// memory (each derived value is computed once per point instead of once per
// stencil use; across periodic faces the halo holds the wrapped cells).
// Interior cells (+-2 FD lines and the 8 LB neighbours are fluid cells of
// the domain; a per-cell flag computed at create) take the fast path: FD
// stencils from shared memory, populations pulled straight from global
// memory (coalesced, one plane at a time).  The wall-tile kernel updates
// the cells next to in-domain solid cells over the listed tiles, from the
// same staging plus the mask; step_kernel_boundary runs the general form
// of lbfd_step_general.cuh over the list of the remaining cells (near
// inlet, outlet and wall faces).
#pragma once
#include "lbfd_step_general.cuh"

namespace lbfd {

template <typename R>
struct TileSmem {
    // layout: [field][point], point = sy * SX + sx
    R* T;
    R* Y;     // NSP planes
    R* X;     // NSP planes
    R* invW;
    R* rho;
    uint8_t* mask;  // 0 fluid, 1 solid, 2 outside the domain
};

template <int TX, int TY>
struct TileGeom {
    static constexpr int SX = TX + 4;
    static constexpr int SY = TY + 4;
    static constexpr int NPT = SX * SY;
};

template <typename R, int TX, int TY>
__host__ __device__ constexpr size_t tile_smem_bytes()
{
    return sizeof(R) * (size_t)TileGeom<TX, TY>::NPT * (3 + 2 * NSP) + (size_t)TileGeom<TX, TY>::NPT;
}

// the tile's arrays in the block's dynamic shared memory
template <typename R, int TX, int TY>
__device__ __forceinline__ TileSmem<R> tile_smem(unsigned char* raw)
{
    constexpr int NPT = TileGeom<TX, TY>::NPT;
    TileSmem<R> sm;
    sm.T = reinterpret_cast<R*>(raw);
    sm.Y = sm.T + NPT;
    sm.X = sm.Y + NSP * NPT;
    sm.invW = sm.X + NSP * NPT;
    sm.rho = sm.invW + NPT;
    sm.mask = reinterpret_cast<uint8_t*>(sm.rho + NPT);
    return sm;
}

// FD terms along one axis of an interior cell from the staged tile:
// `line(f, v)` gathers the five points of the staged field f along the axis
// into v.  R is the compute type (float, double, or F2 for a pair of
// cells), PR the parameters' type.
template <typename R, typename PR, typename SR, typename Line>
__device__ __forceinline__ void fd_axis_tile(const StepParams<PR>& P, const TileSmem<SR>& sm, int npt, Line line,
                                             R u_a, R invW0, R inv_rho0, R* gam_a, FDAccum<R>& acc)
{
    fd_axis<false, R>(
        P, u_a, invW0, inv_rho0, false, false, [&](R* v) { line(sm.rho, v); }, [&](R* v) { line(sm.T, v); },
        [&](R* v) { line(sm.invW, v); }, [&](int k, R* v) { line(sm.X + k * npt, v); },
        [&](int k, R* v) { line(sm.Y + k * npt, v); }, gam_a, acc);
}

// the same with the axis' point stride `st` (1 for x, SX for y) and the
// centre point p0
template <typename R>
__device__ __forceinline__ void fd_axis_smem(const StepParams<R>& P, const TileSmem<R>& sm, int npt, int p0, int st,
                                             R u_a, R invW0, R inv_rho0, R* gam_a, FDAccum<R>& acc)
{
    auto line = [&](const R* f, R* v) {
#pragma unroll
        for (int j = 0; j < 5; ++j) v[j] = f[p0 + (j - 2) * st];
    };
    fd_axis_tile<R>(P, sm, npt, line, u_a, invW0, inv_rho0, gam_a, acc);
}

// FD terms along one axis for a cell next to in-domain solid cells (staircase
// walls), from shared memory: pts are the five line points after the mirror
// rule, `ghost` flags the points that are ghosts (bit j), whose T and rho
// take the Dirichlet form when the solid is isothermal (Y, X, 1/W mirror).
template <typename R>
__device__ __forceinline__ void fd_axis_smem_walls(const StepParams<R>& P, const TileSmem<R>& sm, int npt,
                                                   const int* pts, int ghost, int a, R u_a, R invW0, R inv_rho0,
                                                   FDAccum<R>& acc)
{
    const bool iso = P.solid_isothermal;
    const R TB = P.T_solid;
    auto line = [&](const R* f, R* v) {
#pragma unroll
        for (int j = 0; j < 5; ++j) v[j] = f[pts[j]];
    };
    auto line_rho = [&](R* v) {
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            v[j] = sm.rho[pts[j]];
            if (iso && ((ghost >> j) & 1)) v[j] = R(2) * eos(P, TB, sm.invW[pts[j]]) - v[j];
        }
    };
    auto line_T = [&](R* v) {
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            v[j] = sm.T[pts[j]];
            if (iso && ((ghost >> j) & 1)) v[j] = R(2) * TB - v[j];
        }
    };
    fd_axis<true, R>(
        P, u_a, invW0, inv_rho0, ghost != 0, true, line_rho, line_T, [&](R* v) { line(sm.invW, v); },
        [&](int k, R* v) { line(sm.X + k * npt, v); }, [&](int k, R* v) { line(sm.Y + k * npt, v); }, &acc.gam[a],
        acc);
}

// the five points of an axis line after the mirror rule of Eq. 34 for
// in-domain solid cells (the ghost at distance j mirrors the fluid point at
// distance j-1 across the wall; the centre when that point is solid)
__device__ __forceinline__ int wall_line(const uint8_t* mask, int p0, int st, int* pts)
{
    int ghost = 0;
#pragma unroll
    for (int j = 0; j < 5; ++j) pts[j] = p0 + (j - 2) * st;
#pragma unroll
    for (int side = -1; side <= 1; side += 2) {
        const int w = mask[p0 + side * st] ? 1 : (mask[p0 + 2 * side * st] ? 2 : 0);
        if (!w) continue;
#pragma unroll
        for (int j = 1; j <= 2; ++j) {
            if (j < w) continue;
            const int m = 2 * w - 1 - j;
            int mp;
            if (m >= 0) mp = p0 + side * m * st;
            else mp = mask[p0 - side * st] ? p0 : p0 - side * st;
            pts[2 + side * j] = mp;
            ghost |= 1 << (2 + side * j);
        }
    }
    return ghost;
}

// a1 (Eq. 8) for a cell whose 8 neighbours are fluid cells of the domain:
// plain pull, the x-1, x+1, y-1, y+1 neighbours wrapped on periodic axes
// (the offsets stay inside the domain for any in-range cell)
template <typename S, typename R>
__device__ __forceinline__ void pull_interior(const StepParams<R>& P, const S* LBFD_RESTRICT g_in, long long c, int x,
                                              int y, R* g)
{
    const int oxm = x == 0 ? P.nx - 1 : -1, oxp = x == P.nx - 1 ? 1 - P.nx : 1;
    const int oym = y == 0 ? (P.ny - 1) * P.nx : -P.nx, oyp = y == P.ny - 1 ? (1 - P.ny) * P.nx : P.nx;
    const S* gc = g_in + c;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int ox = cx_of(i) > 0 ? oxm : (cx_of(i) < 0 ? oxp : 0);
        const int oy = cy_of(i) > 0 ? oym : (cy_of(i) < 0 ? oyp : 0);
        g[i] = R(LBFD_LDG(gc + (long long)i * P.N + (ox + oy)));
    }
}

// Stage T, Y_k, X_k, 1/W, rho and the mask of a tile (origin x0, y0) and
// its 2-cell halo with NTHR threads, this one numbered tid.  All of a
// thread's global loads are issued before any of them is used, so that
// their latencies overlap.  WALLS == false (interior tiles, whose cells are
// flagged interior from a per-cell array): no mask; solid points are staged
// like fluid ones, their values are never read.
template <typename S, typename R, int TX, int TY, bool WALLS, int NTHR>
__device__ __forceinline__ void stage_tile2d(const StepParams<R>& P, const TileSmem<R>& sm, int x0, int y0, int tid,
                                             const S* LBFD_RESTRICT T_in, const S* LBFD_RESTRICT Y_in,
                                             const uint8_t* LBFD_RESTRICT solid)
{
    using G = TileGeom<TX, TY>;
    constexpr int SX = G::SX, NPT = G::NPT;
    constexpr int NIT = (NPT + NTHR - 1) / NTHR;
    const long long N = P.N;
    long long cell[NIT];  // -1: outside the domain
    uint8_t s[NIT];
    R T[NIT], Y[NIT][NSP];
#pragma unroll
    for (int it = 0; it < NIT; ++it) {
        const int pt = tid + it * NTHR;
        cell[it] = -1;
        if (pt >= NPT) continue;
        const int sx = pt % SX, sy = pt / SX;
        int gx = x0 + sx - 2, gy = y0 + sy - 2;
        // across a periodic face the halo holds the wrapped cells
        // (at most two periods away: the halo is two cells wide)
        if (P.bc[0] == BC_PERIODIC) {
            if (gx < 0) gx += P.nx;
            if (gx < 0) gx += P.nx;
            if (gx >= P.nx) gx -= P.nx;
            if (gx >= P.nx) gx -= P.nx;
        }
        if (P.bc[2] == BC_PERIODIC) {
            if (gy < 0) gy += P.ny;
            if (gy < 0) gy += P.ny;
            if (gy >= P.ny) gy -= P.ny;
            if (gy >= P.ny) gy -= P.ny;
        }
        if (gx < 0 || gx >= P.nx || gy < 0 || gy >= P.ny) {
            // outside the domain: marked 2 and never read by a fast-path cell
            uint8_t m = 2;
            if constexpr (WALLS) {  // beyond walls that act like the solid cells
                const bool okx = gx >= 0 && gx < P.nx ? true : P.face_solid[gx < 0 ? 0 : 1];
                const bool oky = gy >= 0 && gy < P.ny ? true : P.face_solid[gy < 0 ? 2 : 3];
                if (okx && oky) m = 1;
                sm.mask[pt] = m;
            }
            continue;
        }
        const long long c = (long long)gx + (long long)P.nx * gy;
        cell[it] = c;
        if constexpr (WALLS) s[it] = solid[c];
        T[it] = R(T_in[c]);
#pragma unroll
        for (int k = 0; k < NSP; ++k) Y[it][k] = R(Y_in[(long long)k * N + c]);
    }
#pragma unroll
    for (int it = 0; it < NIT; ++it) {
        if (cell[it] < 0) continue;
        const int pt = tid + it * NTHR;
        if constexpr (WALLS) {
            sm.mask[pt] = s[it] ? 1 : 0;
            if (s[it]) continue;
        }
        const R invW = inv_molar_mass(P, Y[it]);
        R W, rho;
        eos_w(P, T[it], invW, rho, W);
        sm.T[pt] = T[it];
#pragma unroll
        for (int k = 0; k < NSP; ++k) {
            sm.Y[k * NPT + pt] = Y[it][k];
            sm.X[k * NPT + pt] = Y[it][k] * W;  // X_k W_k (1/W_k folded into a12)
        }
        sm.invW[pt] = invW;
        sm.rho[pt] = rho;
    }
}

// the +-2 FD lines and the 8 LB neighbours of point p0 are fluid cells of the domain
template <int SX>
__device__ __forceinline__ bool interior_point(const uint8_t* mask, int p0)
{
    bool fast = !mask[p0];
#pragma unroll
    for (int j = 1; j <= 2; ++j)
        fast = fast && !mask[p0 + j] && !mask[p0 - j] && !mask[p0 + j * SX] && !mask[p0 - j * SX];
    return fast && !mask[p0 + SX + 1] && !mask[p0 + SX - 1] && !mask[p0 - SX + 1] && !mask[p0 - SX - 1];
}

// body of the 2-D tile kernels: the tile (bx, by), this thread at (tx, ty)
// of its TX x TY threads.  WALLS == false: the interior cells of the tile.
// WALLS == true: only the cells next to in-domain solid cells (or walls that
// act like them).  Every thread of the block calls it (it synchronises the
// block once, after the staging).
template <typename S, typename R, int TX, int TY, bool WALLS, bool HI1>
__device__ __forceinline__ void tiled2d_body(const StepParams<R>& P, const S* LBFD_RESTRICT g_in, S* LBFD_RESTRICT g_out,
                                             const S* LBFD_RESTRICT T_in, S* LBFD_RESTRICT T_out,
                                             const S* LBFD_RESTRICT Y_in, S* LBFD_RESTRICT Y_out,
                                             const uint8_t* LBFD_RESTRICT solid,
                                             const uint8_t* LBFD_RESTRICT interior, int tx, int ty, int bx, int by)
{
    using G = TileGeom<TX, TY>;
    constexpr int SX = G::SX, NPT = G::NPT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const TileSmem<R> sm = tile_smem<R, TX, TY>(smem_raw);

    const int x0 = bx * TX, y0 = by * TY;
    const int tid = tx + TX * ty;
    const long long N = P.N;
    const int x = x0 + tx, y = y0 + ty;
    const bool inside = x < P.nx && y < P.ny;
    const long long c = (long long)x + (long long)P.nx * y;
    R g[9];
    // interior tiles: the cell's class (the +-2 lines and the 8 neighbours
    // are fluid cells of the domain, precomputed per cell) and a1, issued
    // before the staging so that the loads are in flight while the tile is
    // staged
    bool fast = false;
    if constexpr (!WALLS) {
        if (inside) {
            fast = interior[c] != 0;
            pull_interior<S, R>(P, g_in, c, x, y, g);
        }
    }
    stage_tile2d<S, R, TX, TY, WALLS, TX * TY>(P, sm, x0, y0, tid, T_in, Y_in, solid);
    __syncthreads();

    if (!inside) return;
    const int p0 = (ty + 2) * SX + tx + 2;
    if constexpr (WALLS) {
        if (sm.mask[p0]) return;  // solid
        fast = interior_point<SX>(sm.mask, p0);
        // next to in-domain solid cells only (staircase walls); the interior
        // cells belong to the plain tile kernel, the rest to the boundary list
        if (fast || P.curved) return;
        bool walls = true;
#pragma unroll
        for (int j = 1; j <= 2; ++j)
            walls = walls && sm.mask[p0 + j] != 2 && sm.mask[p0 - j] != 2 && sm.mask[p0 + j * SX] != 2 &&
                    sm.mask[p0 - j * SX] != 2;
        walls = walls && sm.mask[p0 + SX + 1] != 2 && sm.mask[p0 + SX - 1] != 2 && sm.mask[p0 - SX + 1] != 2 &&
                sm.mask[p0 - SX - 1] != 2;
        if (!walls) return;
    } else {
        if (!fast) return;  // solid, or a boundary cell: another kernel updates it
    }
    // a1 for the wall tiles: pull from the neighbours (Eq. 8), half-way
    // bounce-back from an in-domain solid neighbour (Eq. 28)
    if constexpr (WALLS) {
        const int oxm = x == 0 ? P.nx - 1 : -1, oxp = x == P.nx - 1 ? 1 - P.nx : 1;
        const int oym = y == 0 ? (P.ny - 1) * P.nx : -P.nx, oyp = y == P.ny - 1 ? (1 - P.ny) * P.nx : P.nx;
        const S* gc = g_in + c;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int ox = cx_of(i) > 0 ? oxm : (cx_of(i) < 0 ? oxp : 0);
            const int oy = cy_of(i) > 0 ? oym : (cy_of(i) < 0 ? oyp : 0);
            long long off = (long long)i * N + (ox + oy);
            if (sm.mask[p0 - cx_of(i) - cy_of(i) * SX]) off = (long long)opposite<2>(i) * N;
            g[i] = R(LBFD_LDG(gc + off));
        }
    }
    // a2
    const R T0 = sm.T[p0], invW0 = sm.invW[p0], rho0 = sm.rho[p0];
    const R inv_rho0 = T0 * invW0 * par<R>(P.inv_rho_c);
    LowMoments<2, R> lm;
    low_moments<2>(g, lm);
    const R u[3] = {lm.m1[0] * (K<R>(3) * inv_rho0), lm.m1[1] * (K<R>(3) * inv_rho0), R(0)};
    // a3-a5
    FDAccum<R> acc;
    acc.clear();
    if constexpr (WALLS) {
        int pts[5];
        int gh = wall_line(sm.mask, p0, 1, pts);
        fd_axis_smem_walls<R>(P, sm, NPT, pts, gh, 0, u[0], invW0, inv_rho0, acc);
        gh = wall_line(sm.mask, p0, SX, pts);
        fd_axis_smem_walls<R>(P, sm, NPT, pts, gh, 1, u[1], invW0, inv_rho0, acc);
    } else {
        if constexpr (std::is_arithmetic<R>::value) {
            fd_axis_smem<R>(P, sm, NPT, p0, 1, u[0], invW0, inv_rho0, &acc.gam[0], acc);
            fd_axis_smem<R>(P, sm, NPT, p0, SX, u[1], invW0, inv_rho0, &acc.gam[1], acc);
        } else {  // forward mode: one copy of the FD code (instruction fetch)
#pragma unroll 1
            for (int a = 0; a < 2; ++a) {
                R gam;
                fd_axis_smem<R>(P, sm, NPT, p0, a ? SX : 1, a ? u[1] : u[0], invW0, inv_rho0, &gam, acc);
                if (a) acc.gam[1] = gam;
                else acc.gam[0] = gam;
            }
        }
    }
    // a6-a7
    R Y0[NSP];
#pragma unroll
    for (int k = 0; k < NSP; ++k) Y0[k] = sm.Y[k * NPT + p0];
    const R rc = rho0 * par<R>(P.inv_rho_c);
    const R Lam = update_scalars<S, R>(P, c, T0, Y0, rc * invW0, rc * T0, acc, T_out, Y_out);
    // a8-a10
    if constexpr (HI1) collide_hi1<2, R>(P, lm, rho0, inv_rho0, u, acc.gam, Lam, g);
    else collide<2, R>(P, g, rho0, inv_rho0, u, acc.gam, Lam);
#pragma unroll
    for (int i = 0; i < 9; ++i) g_out[(long long)i * N + c] = S(g[i]);
}

// FP32: four 256-thread blocks (1024 threads) per SM, i.e. <= 64 registers
template <typename S, typename R, int TX, int TY, bool HI1>
__global__ void __launch_bounds__(TX * TY, sizeof(R) == 4 ? 1024 / (TX * TY) : 1)
    step_kernel_tiled2d(StepParams<R> P, const S* LBFD_RESTRICT g_in, S* LBFD_RESTRICT g_out,
                        const S* LBFD_RESTRICT T_in, S* LBFD_RESTRICT T_out, const S* LBFD_RESTRICT Y_in,
                        S* LBFD_RESTRICT Y_out, const uint8_t* LBFD_RESTRICT interior)
{
    tiled2d_body<S, R, TX, TY, false, HI1>(P, g_in, g_out, T_in, T_out, Y_in, Y_out, nullptr, interior, threadIdx.x,
                                      threadIdx.y, blockIdx.x, blockIdx.y);
}

// the cells next to in-domain solid cells, over the tiles that contain any
template <typename S, typename R, int TX, int TY, bool HI1>
__global__ void __launch_bounds__(TX * TY)
    step_kernel_tiled2d_walls(StepParams<R> P, const S* LBFD_RESTRICT g_in, S* LBFD_RESTRICT g_out,
                              const S* LBFD_RESTRICT T_in, S* LBFD_RESTRICT T_out, const S* LBFD_RESTRICT Y_in,
                              S* LBFD_RESTRICT Y_out, const uint8_t* LBFD_RESTRICT solid, const int* LBFD_RESTRICT tiles)
{
    const int t = tiles[blockIdx.x];
    const int gxn = (P.nx + TX - 1) / TX;
    tiled2d_body<S, R, TX, TY, true, HI1>(P, g_in, g_out, T_in, T_out, Y_in, Y_out, solid, nullptr, threadIdx.x,
                                     threadIdx.y, t % gxn, t / gxn);
}

// The cells of a coded list: next to in-domain solids (staircase walls, no
// non-periodic face in reach), or (FACES) near inlet and outlet faces:
// cell_step_coded
template <int DIM, typename S, typename R, bool FACES = false, bool HI1 = false>
__global__ void __launch_bounds__(128) step_kernel_wallcode(StepParams<R> P, const S* LBFD_RESTRICT g_in,
                                                            S* LBFD_RESTRICT g_out, const S* LBFD_RESTRICT T_in,
                                                            S* LBFD_RESTRICT T_out, const S* LBFD_RESTRICT Y_in,
                                                            S* LBFD_RESTRICT Y_out,
                                                            const long long* LBFD_RESTRICT cells,
                                                            const unsigned long long* LBFD_RESTRICT codes,
                                                            long long ncells)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ncells) return;
    const long long c = cells[t];
    int p[3];
    p[0] = (int)(c % P.nx);
    const long long r = c / P.nx;
    p[1] = (int)(r % P.ny);
    p[2] = (int)(r / P.ny);
    cell_step_coded<DIM, S, R, FACES, HI1>(P, p, c, codes[t], g_in, g_out, T_in, T_out, Y_in, Y_out);
}

// The cells the tiled kernel leaves out: general form over a cell list
// (FACES == false: cells whose stencils reach no non-periodic face).
template <int DIM, typename S, typename R, bool FACES, bool HI1>
__global__ void __launch_bounds__(128) step_kernel_boundary(StepParams<R> P, const S* LBFD_RESTRICT g_in,
                                                            S* LBFD_RESTRICT g_out, const S* LBFD_RESTRICT T_in,
                                                            S* LBFD_RESTRICT T_out, const S* LBFD_RESTRICT Y_in,
                                                            S* LBFD_RESTRICT Y_out, const uint8_t* LBFD_RESTRICT solid,
                                                            const long long* LBFD_RESTRICT cells, long long ncells)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ncells) return;
    const long long c = cells[t];
    int p[3];
    p[0] = (int)(c % P.nx);
    const long long r = c / P.nx;
    p[1] = (int)(r % P.ny);
    p[2] = (int)(r / P.ny);
    cell_step_general<DIM, S, R, FACES, HI1>(P, p, c, g_in, g_out, T_in, T_out, Y_in, Y_out, solid);
}

}  // namespace lbfd
