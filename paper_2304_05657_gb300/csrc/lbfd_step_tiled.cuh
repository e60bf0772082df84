// lbfd_step_tiled.cuh -- 2-D fused coupled step with shared-memory staging.
//
// A block owns a TX x TY tile of cells.  It stages T, Y_k and the derived
// point values 1/W, X_k and rho of the tile plus a 2-cell halo in shared
// memory (each derived value is computed once per point instead of once per
// stencil use; across periodic faces the halo holds the wrapped cells).
// Interior cells (+-2 FD lines and the 8 LB neighbours are fluid cells of
// the domain; a per-cell flag computed at create) take the fast path: FD
// stencils from shared memory, populations pulled straight from global
// memory (coalesced, one plane at a time).  The coded form of the tiles
// takes the cells next to staircase walls and domain faces too, by their
// neighbourhood codes (list_codes2d); what the tiles leave out goes through
// lists: step_kernel_wallcode the coded cells, step_kernel_boundary the
// general form of lbfd_step_general.cuh.
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
    return sizeof(R) * (size_t)TileGeom<TX, TY>::NPT * (3 + 2 * NSP);
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

// The line points of a coded cell along one axis (see coded_line): pts[j]
// are the staged points at offsets -2..2, replaced by the mirror points of
// the solids' ghosts (the ghosts beyond a face are staged as such); returns
// the solid ghosts (bit j).  Branch-free: 17 integer instructions per side.
__device__ __forceinline__ unsigned coded_pts(unsigned code, unsigned faces, int* pts)
{
    const int lo = pts[1], hi = pts[3], c0 = pts[2];
    unsigned ghosts = 0;
#pragma unroll
    for (int side = -1; side <= 1; side += 2) {
        const unsigned bits = side < 0 ? (code & 7u) : (code >> 3);
        const unsigned w = (faces >> (side < 0 ? 0 : 1)) & 1u ? 0u : (bits & 3u);
        const int near = side < 0 ? lo : hi, opp = side < 0 ? hi : lo;
        const int far = w == 2 ? near : ((bits & 4u) ? c0 : opp);
        pts[2 + 2 * side] = w == 0 ? pts[2 + 2 * side] : far;
        pts[2 + side] = w == 1 ? c0 : near;
        ghosts |= (w == 1 ? 1u << (2 + side) : 0u) | (w != 0 ? 1u << (2 + 2 * side) : 0u);
    }
    return ghosts;
}

// The FD terms along one axis with the axis' point stride `st` (1 for x, SX
// for y) and the centre point p0.  CODED and cw (a warp-uniform flag: some
// lane is a coded cell): the line points of a coded cell are the mirror
// points of code6 and faces2 (the axis' part of its code), T and rho of the
// ghosts of isothermal solids take the Dirichlet form of Eq. 34, and the
// convection of an axis next to a boundary is centred.
template <bool CODED, typename R>
__device__ __forceinline__ void fd_axis_smem(const StepParams<R>& P, const TileSmem<R>& sm, int npt, int p0, int st,
                                             bool cw, unsigned code6, unsigned faces2, R u_a, R invW0, R inv_rho0,
                                             R* gam_a, FDAccum<R>& acc)
{
    int pts[5];
#pragma unroll
    for (int j = 0; j < 5; ++j) pts[j] = p0 + (j - 2) * st;
    unsigned dir = 0;
    if (CODED && cw) dir = coded_pts(code6, faces2, pts);
    const bool iso = CODED && cw && P.solid_isothermal;
    auto line = [&](const R* f, R* v) {
#pragma unroll
        for (int j = 0; j < 5; ++j) v[j] = f[pts[j]];
    };
    auto line_rho = [&](R* v) {
        line(sm.rho, v);
        if (iso) {
            // 2 EOS(T_solid, Y) - rho at the mirror point, W = rho T / rho_c
            const R rc = K<R>(2) * (P.rho_solid * par<R>(P.inv_rho_c));
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                if (j == 2) continue;
                const R g = rc * (v[j] * sm.T[pts[j]]) - v[j];
                v[j] = (dir >> j) & 1u ? g : v[j];
            }
        }
    };
    auto line_T = [&](R* v) {
        line(sm.T, v);
        if (iso) {
            const R t = K<R>(2) * P.T_solid;
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                if (j == 2) continue;
                const R g = t - v[j];
                v[j] = (dir >> j) & 1u ? g : v[j];
            }
        }
    };
    fd_axis<CODED, R>(
        P, u_a, invW0, inv_rho0, code6 != 0, cw, line_rho, line_T, [&](R* v) { line(sm.invW, v); },
        [&](int k, R* v) { line(sm.X + k * npt, v); }, [&](int k, R* v) { line(sm.Y + k * npt, v); }, gam_a, acc);
}

// a1 of a coded cell of a tile, after the plain pull (g holds what the
// sources x - c_i hold): bounce-back where the code says so (Eq. 28), and the
// inlet (Eq. 31) and constant-pressure outlet rules for what comes from
// beyond an open face.
template <typename S, typename R>
__device__ __forceinline__ void pull_coded_tile(const StepParams<R>& P, int x, int y, long long c, unsigned code,
                                                R rho0, R inv_rho0, const S* LBFD_RESTRICT g_in, R* g)
{
    const bool xlo = x == 0 && P.bc[0] != BC_PERIODIC, xhi = x == P.nx - 1 && P.bc[1] != BC_PERIODIC;
    const bool ylo = y == 0 && P.bc[2] != BC_PERIODIC, yhi = y == P.ny - 1 && P.bc[3] != BC_PERIODIC;
    unsigned cross = 0;  // from beyond a face and not bounced back
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const bool f = (cx_of(i) > 0 && xlo) || (cx_of(i) < 0 && xhi) || (cy_of(i) > 0 && ylo) || (cy_of(i) < 0 && yhi);
        if (f && !((code >> i) & 1u)) cross |= 1u << i;
    }
    const unsigned own = (code & 0x1ffu) | cross;
#pragma unroll
    for (int i = 0; i < 9; ++i)
        if ((own >> i) & 1u) g[i] = R(LBFD_LDG(g_in + (long long)opposite<2>(i) * P.N + c));
    if (!cross) return;
    R u[2] = {R(0), R(0)}, uu = R(0);
    if ((xlo && P.bc[0] == BC_OUTLET_PRESSURE) || (xhi && P.bc[1] == BC_OUTLET_PRESSURE) ||
        (ylo && P.bc[2] == BC_OUTLET_PRESSURE) || (yhi && P.bc[3] == BC_OUTLET_PRESSURE)) {
        R q[9];  // the cell's own velocity before streaming
#pragma unroll
        for (int i = 0; i < 9; ++i) q[i] = R(LBFD_LDG(g_in + (long long)i * P.N + c));
        LowMoments<2, R> m;
        low_moments<2>(q, m);
        u[0] = m.m1[0] * (K<R>(3) * inv_rho0);
        u[1] = m.m1[1] * (K<R>(3) * inv_rho0);
        uu = u[0] * u[0] + u[1] * u[1];
    }
    R mag = P.u_in;  // along the inward normal, as is c_i
    if (P.poiseuille) {
        const R ny = R(P.ny), yc = R(y) + R(0.5);
        mag = R(6) * P.u_in * yc * (ny - yc) / (ny * ny);
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        if (i == 4 || !((cross >> i) & 1u)) continue;
        const int cx = cx_of(i), cy = cy_of(i);
        const bool fx = (cx > 0 && xlo) || (cx < 0 && xhi);
        const int t = fx ? (cx > 0 ? P.bc[0] : P.bc[1]) : (cy > 0 ? P.bc[2] : P.bc[3]);
        const auto w2 = K<R>(2.0 * weight<2, double>(i));
        if (t == BC_INLET) {
            g[i] += w2 * R((fx ? mag : P.u_in) * P.rho_in);
        } else {
            const R cu = R(cx) * u[0] + R(cy) * u[1];
            g[i] = w2 * R(rho0 * (K<R>(1.5) * R(cu * cu) - K<R>(0.5) * uu)) - g[i];
        }
    }
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

// Stage T, Y_k, X_k, 1/W and rho of a tile (origin x0, y0) and its 2-cell
// halo with NTHR threads, this one numbered tid.  All of a thread's global
// loads are issued before any of them is used, so that their latencies
// overlap.  Solid points are staged like fluid ones, their values are never
// read.  CODED: the points beyond a non-periodic face hold the ghosts of
// their lines (Eq. 34).
template <typename S, typename R, int TX, int TY, bool CODED, int NTHR>
__device__ __forceinline__ void stage_tile2d(const StepParams<R>& P, const TileSmem<R>& sm, int x0, int y0, int tid,
                                             const S* LBFD_RESTRICT T_in, const S* LBFD_RESTRICT Y_in)
{
    using G = TileGeom<TX, TY>;
    constexpr int SX = G::SX, NPT = G::NPT;
    constexpr int NIT = (NPT + NTHR - 1) / NTHR;
    const long long N = P.N;
    long long cell[NIT];  // -1: outside the domain
    int face[NIT];        // CODED: the face a ghost point lies beyond, -1 for others
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
        face[it] = -1;
        if constexpr (CODED) {
            // beyond a face: the ghost of its line, from the mirror cell
            if (gx < 0 || gx >= P.nx) {
                if (gx < -2 || gx >= P.nx + 2) continue;
                face[it] = gx < 0 ? 0 : 1;
                gx = gx < 0 ? -1 - gx : 2 * P.nx - 1 - gx;
                gx = gx < 0 ? 0 : (gx >= P.nx ? P.nx - 1 : gx);
            }
            if (gy < 0 || gy >= P.ny) {
                if (gy < -2 || gy >= P.ny + 2 || face[it] >= 0) continue;
                face[it] = gy < 0 ? 2 : 3;
                gy = gy < 0 ? -1 - gy : 2 * P.ny - 1 - gy;
                gy = gy < 0 ? 0 : (gy >= P.ny ? P.ny - 1 : gy);
            }
        }
        if (gx < 0 || gx >= P.nx || gy < 0 || gy >= P.ny) continue;  // never read by a cell of the tile
        const long long c = (long long)gx + (long long)P.nx * gy;
        cell[it] = c;
        T[it] = R(T_in[c]);
#pragma unroll
        for (int k = 0; k < NSP; ++k) Y[it][k] = R(Y_in[(long long)k * N + c]);
    }
#pragma unroll
    for (int it = 0; it < NIT; ++it) {
        if (cell[it] < 0) continue;
        const int pt = tid + it * NTHR;
        R invW = inv_molar_mass(P, Y[it]);
        R W, rho;
        eos_w(P, T[it], invW, rho, W);
        if (CODED && face[it] >= 0) {  // Eq. 34 (zero gradient: the mirror values)
            const int t = face_type(P, face[it]);
            if (t == BC_INLET) {
                T[it] = K<R>(2) * P.T_in - T[it];
#pragma unroll
                for (int k = 0; k < NSP; ++k) Y[it][k] = K<R>(2) * P.Y_in[k] - Y[it][k];
                invW = inv_molar_mass(P, Y[it]);
                W = frcp(invW);
                rho = K<R>(2) * P.rho_in - rho;
            } else if (t == BC_WALL_ISOTHERMAL) {
                const R Tw = face_T_wall(P, face[it]);
                T[it] = K<R>(2) * Tw - T[it];
                rho = K<R>(2) * R(R(par<R>(P.rho_c) * frcp(Tw)) * W) - rho;
            }
        }
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

// body of the 2-D tile kernels: the tile (bx, by), this thread at (tx, ty)
// of its TX x TY threads.  The interior cells, with CODED also the cells of
// class 2 by their codes.  Every thread of the block calls it (it
// synchronises the block once, after the staging).
template <typename S, typename R, int TX, int TY, bool CODED, bool HI1>
__device__ __forceinline__ void tiled2d_body(const StepParams<R>& P, const S* LBFD_RESTRICT g_in, S* LBFD_RESTRICT g_out,
                                             const S* LBFD_RESTRICT T_in, S* LBFD_RESTRICT T_out,
                                             const S* LBFD_RESTRICT Y_in, S* LBFD_RESTRICT Y_out,
                                             const uint8_t* LBFD_RESTRICT interior,
                                             const unsigned long long* LBFD_RESTRICT codes, int tx, int ty, int bx,
                                             int by)
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
    // the cell's class (precomputed per cell) and a1, issued before the
    // staging so that the loads are in flight while the tile is staged
    bool fast = false;
    unsigned long long code = 0;  // of a coded cell
    if (inside) {
        const int cls = interior[c];
        fast = cls == 1 || (CODED && cls == 2 && !P.curved);
        if (CODED && cls == 2 && fast) code = codes[c];
        pull_interior<S, R>(P, g_in, c, x, y, g);
    }
    const bool cw = CODED && __any_sync(0xffffffffu, code != 0);
    stage_tile2d<S, R, TX, TY, CODED, TX * TY>(P, sm, x0, y0, tid, T_in, Y_in);
    __syncthreads();

    if (!fast) return;  // outside, solid, or a cell that another kernel updates
    const int p0 = (ty + 2) * SX + tx + 2;
    // a2
    const R T0 = sm.T[p0], invW0 = sm.invW[p0], rho0 = sm.rho[p0];
    const R inv_rho0 = T0 * invW0 * par<R>(P.inv_rho_c);
    if (CODED && code) pull_coded_tile<S, R>(P, x, y, c, (unsigned)code, rho0, inv_rho0, g_in, g);
    LowMoments<2, R> lm;
    low_moments<2>(g, lm);
    const R u[3] = {lm.m1[0] * (K<R>(3) * inv_rho0), lm.m1[1] * (K<R>(3) * inv_rho0), R(0)};
    // a3-a5
    FDAccum<R> acc;
    acc.clear();
    const unsigned cx6 = (unsigned)(code >> 32) & 63u, cy6 = (unsigned)(code >> 38) & 63u;
    const unsigned fx2 = (unsigned)(code >> 50) & 3u, fy2 = (unsigned)(code >> 52) & 3u;
    if constexpr (std::is_arithmetic<R>::value) {
        fd_axis_smem<CODED, R>(P, sm, NPT, p0, 1, cw, cx6, fx2, u[0], invW0, inv_rho0, &acc.gam[0], acc);
        fd_axis_smem<CODED, R>(P, sm, NPT, p0, SX, cw, cy6, fy2, u[1], invW0, inv_rho0, &acc.gam[1], acc);
    } else {  // forward mode: one copy of the FD code (instruction fetch)
#pragma unroll 1
        for (int a = 0; a < 2; ++a) {
            R gam;
            fd_axis_smem<CODED, R>(P, sm, NPT, p0, a ? SX : 1, cw, a ? cy6 : cx6, a ? fy2 : fx2, a ? u[1] : u[0],
                                   invW0, inv_rho0, &gam, acc);
            if (a) acc.gam[1] = gam;
            else acc.gam[0] = gam;
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
template <typename S, typename R, int TX, int TY, bool CODED, bool HI1>
__global__ void __launch_bounds__(TX * TY, sizeof(R) == 4 ? 1024 / (TX * TY) : 1)
    step_kernel_tiled2d(StepParams<R> P, const S* LBFD_RESTRICT g_in, S* LBFD_RESTRICT g_out,
                        const S* LBFD_RESTRICT T_in, S* LBFD_RESTRICT T_out, const S* LBFD_RESTRICT Y_in,
                        S* LBFD_RESTRICT Y_out, const uint8_t* LBFD_RESTRICT interior,
                        const unsigned long long* LBFD_RESTRICT codes)
{
    tiled2d_body<S, R, TX, TY, CODED, HI1>(P, g_in, g_out, T_in, T_out, Y_in, Y_out, interior, codes, threadIdx.x,
                                           threadIdx.y, blockIdx.x, blockIdx.y);
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
