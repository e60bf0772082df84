// lbfd_step_tiled3d.cuh -- 3-D (D3Q27) fused coupled step, 2.5-D tiling.
//
// A block of TX x TY threads owns a TX x TY column of cells and marches it
// through zc consecutive z-planes.  Shared memory holds a ring of five
// z-planes (z-2 .. z+2) of the tile plus its 2-cell x/y halo, with T, Y_k
// and the derived W, 1/W, rho of every point (X_k = Y_k W / W_k is formed
// when used); each plane is loaded once per column pass.  A 64-bit word per
// cell (cell_words) says what the cell is: interior (every +-2 axis
// neighbour and all 26 LB neighbours are fluid cells of the domain), a cell
// next to in-domain solids or near inlet and outlet faces, with its
// neighbourhood code, or one that another kernel updates.  A warp with coded
// cells takes their ghost points from the staged planes (mirror points and
// Dirichlet forms of Eq. 34) and their bounce-back and face rules from the
// code; the others skip all of that with a warp-uniform branch.  So a step
// is one launch (two when some cells need the general form): as lists of
// their own the 276 000 coded cells of a 256x128x128 packing took 155 us
// beside 463 us for the 3.3 million interior ones, their lanes here being
// idle anyway.
#pragma once
#include "lbfd_step_tiled.cuh"

namespace lbfd {

// the value `off` bytes from a pointer that is uniform over the block: a
// 32-bit offset keeps the 64-bit arithmetic out of the lanes.  In-plane
// offsets of a state array stay below 2^32 bytes on every grid that fits the
// device: 2^30 FP32 cells of 297 bytes each (two states, the split variants'
// planes, word, read-out value, mask) or 2^29 FP64 cells of 577 are 319 and
// 310 GB.
template <typename S>
__device__ __forceinline__ const S* at_bytes(const S* base, unsigned off)
{
    return reinterpret_cast<const S*>(reinterpret_cast<const char*>(base) + off);
}
template <typename S>
__device__ __forceinline__ S* at_bytes(S* base, unsigned off)
{
    return reinterpret_cast<S*>(reinterpret_cast<char*>(base) + off);
}

// the cell whose value lies `off` bytes into a plane of S that starts at cell
// `base`: the words are indexed by it in 64 bits, 8 bytes a cell for either S
// (as a 32-bit byte offset they would wrap from 2^29 cells a plane on)
template <typename S>
__host__ __device__ __forceinline__ long long cell_at(long long base, unsigned off)
{
    return base + off / (unsigned)sizeof(S);
}

template <int TX, int TY>
struct Tile3Geom {
    static constexpr int SX = TX + 4;
    static constexpr int SY = TY + 4;
    static constexpr int NPP = SX * SY;  // points per plane
    static constexpr int NPL = 5;        // planes in the ring
    static constexpr int NPT = NPP * NPL;
};

template <typename R, int TX, int TY>
__host__ __device__ constexpr size_t tile3_smem_bytes()
{
    // T, Y_k, 1/W, W, rho per point (X_k = Y_k W / W_k is formed when used)
    return sizeof(R) * (size_t)Tile3Geom<TX, TY>::NPT * (4 + NSP);
}

// FD terms along one axis from five shared-memory points.  CODED and cw (a
// warp-uniform flag: some lane is a coded cell): dir flags the ghosts of
// isothermal solids, whose T and rho take the Dirichlet form of Eq. 34, and
// `near` the axes next to a boundary, whose convection is centred (Sec. II.D).
template <bool CODED, typename R>
__device__ __forceinline__ void fd_axis_pts(const StepParams<R>& P, const TileSmem<R>& sm, int npt, const int* pts,
                                            bool cw, unsigned dir, bool near, R u_a, R invW0, R inv_rho0, R* gam_a,
                                            FDAccum<R>& acc)
{
    R Wl[5];
    auto line = [&](const R* f, R* v) {
#pragma unroll
        for (int j = 0; j < 5; ++j) v[j] = f[pts[j]];
    };
    auto line_rho = [&](R* v) {
        line(sm.rho, v);
        if (CODED && cw) {
            const R rc = R(2) * P.rho_solid;
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                if (j == 2) continue;
                const R g = rc * sm.X[pts[j]] - v[j];  // 2 EOS(T_solid, Y of the mirror point) - rho
                v[j] = (dir >> j) & 1u ? g : v[j];
            }
        }
    };
    auto line_T = [&](R* v) {
        line(sm.T, v);
        if (CODED && cw) {
            const R t = R(2) * P.T_solid;
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                if (j == 2) continue;
                const R g = t - v[j];
                v[j] = (dir >> j) & 1u ? g : v[j];
            }
        }
    };
    auto line_invW = [&](R* v) {
        line(sm.invW, v);
        line(sm.X, Wl);  // W (the 3-D tile keeps W in the X slot)
    };
    fd_axis<CODED, R>(
        P, u_a, invW0, inv_rho0, near, cw, line_rho, line_T, line_invW,
        [&](int k, R* v) {
#pragma unroll
            for (int j = 0; j < 5; ++j) v[j] = sm.Y[k * npt + pts[j]] * Wl[j];
        },
        [&](int k, R* v) { line(sm.Y + k * npt, v); }, gam_a, acc);
}

// populations whose component along an axis is +1 (cp) or -1, as bits
constexpr unsigned pop_mask(int axis, int c)
{
    unsigned m = 0;
    for (int i = 0; i < 27; ++i)
        if (ccomp<3>(i, axis) == c) m |= 1u << i;
    return m;
}
// the populations of cell p that come from beyond an open face
template <typename R>
__device__ __forceinline__ unsigned face_crossing(const StepParams<R>& P, int x, int y, int z)
{
    unsigned m = 0;
    if (x == 0 && P.bc[0] != BC_PERIODIC) m |= pop_mask(0, 1);
    if (x == P.nx - 1 && P.bc[1] != BC_PERIODIC) m |= pop_mask(0, -1);
    if (y == 0 && P.bc[2] != BC_PERIODIC) m |= pop_mask(1, 1);
    if (y == P.ny - 1 && P.bc[3] != BC_PERIODIC) m |= pop_mask(1, -1);
    if (z == 0 && P.bc[4] != BC_PERIODIC) m |= pop_mask(2, 1);
    if (z == P.nz - 1 && P.bc[5] != BC_PERIODIC) m |= pop_mask(2, -1);
    return m;
}

// Inlet and constant-pressure outlet rules (Eq. 31; anti-bounce-back) of a
// cell at one open face: on entry the crossing populations hold the opposite
// population of the cell itself, as for bounce-back.  Both rules are
//   g_i = +-g_ibar + w_i (k0 + 3 rho (c_i.u)^2),
// inlet: +, k0 = 2 rho_in u_in, u = 0; outlet: -, k0 = -rho u.u, u the cell's
// velocity before streaming.
template <typename S, typename R>
__device__ __forceinline__ void face_rules(const StepParams<R>& P, unsigned cross, const S* LBFD_RESTRICT g_cell,
                                           R rho0, R inv_rho0, R* g)
{
    const int f = cross == pop_mask(0, 1)    ? 0
                  : cross == pop_mask(0, -1) ? 1
                  : cross == pop_mask(1, 1)  ? 2
                  : cross == pop_mask(1, -1) ? 3
                  : cross == pop_mask(2, 1)  ? 4
                                             : 5;
    R u[3] = {R(0), R(0), R(0)}, k0 = R(2) * P.rho_in * P.u_in, sign = R(1);
    if (face_type(P, f) != BC_INLET) {
        R own[27];
#pragma unroll
        for (int j = 0; j < 27; ++j) own[j] = R(g_cell[(long long)j * P.N]);
        LowMoments<3, R> m;
        low_moments<3>(own, m);
#pragma unroll
        for (int b = 0; b < 3; ++b) u[b] = m.m1[b] * (K<R>(3) * inv_rho0);
        k0 = -rho0 * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
        sign = R(-1);
    }
    const R r3 = R(3) * rho0;
#pragma unroll
    for (int i = 0; i < 27; ++i) {
        if (i == 13 || !((cross >> i) & 1u)) continue;
        const R cu = R(cx_of(i)) * u[0] + R(cy_of(i)) * u[1] + R(cz_of(i)) * u[2];
        g[i] = sign * g[i] + weight<3, R>(i) * (k0 + r3 * cu * cu);
    }
}

// Staging of one plane of the tile.  What does not change from plane to
// plane is computed once per thread: the in-plane offsets of its points,
// wrapped across periodic faces.  A point beyond another face is staged as
// the ghost of Eq. 34 of its line there (the mirror cell's values, Dirichlet
// at an inlet; cells near wall faces are not taken from the tile), so that
// cells near open faces read plain lines.  Solid points are staged like
// fluid ones (never read by a fluid cell).
template <int TX, int TY>
struct StagePoints {
    using G = Tile3Geom<TX, TY>;
    static constexpr int NTHR = TX * TY, NIT = (G::NPP + NTHR - 1) / NTHR;
    unsigned off[NIT];  // bytes
    unsigned inlet;  // bit it: beyond an inlet face
};
// coordinate q beyond [0, n): wrapped, or its mirror image; *face = the face
// crossed (-1: none or periodic)
template <typename R>
__device__ __forceinline__ int stage_coord(const StepParams<R>& P, int q, int n, int axis, int* face)
{
    *face = -1;
    if (q >= 0 && q < n) return q;
    const int f = 2 * axis + (q < 0 ? 0 : 1);
    if (face_type(P, f) == BC_PERIODIC) return ((q % n) + n) % n;
    *face = f;
    const int m = q < 0 ? -1 - q : 2 * n - 1 - q;
    return m < 0 ? 0 : (m >= n ? n - 1 : m);
}
template <typename S, typename R, int TX, int TY>
__device__ __forceinline__ void stage_points(const StepParams<R>& P, int x0, int y0, StagePoints<TX, TY>& sp)
{
    using G = Tile3Geom<TX, TY>;
    const int tid = threadIdx.x + TX * threadIdx.y;
    sp.inlet = 0;
#pragma unroll
    for (int it = 0; it < sp.NIT; ++it) {
        const int q = tid + it * sp.NTHR;
        int fx, fy;
        const int gx = stage_coord(P, x0 + q % G::SX - 2, P.nx, 0, &fx);
        const int gy = stage_coord(P, y0 + q / G::SX - 2, P.ny, 1, &fy);
        sp.off[it] = ((unsigned)gx + (unsigned)P.nx * (unsigned)gy) * (unsigned)sizeof(S);
        const int f = fx >= 0 ? fx : fy;
        if (f >= 0 && face_type(P, f) == BC_INLET) sp.inlet |= 1u << it;
    }
}
// stage plane z (grid coordinate) into the ring slot that starts at point `base`
template <typename S, typename R, int TX, int TY>
__device__ __forceinline__ void stage_plane(const StepParams<R>& P, const TileSmem<R>& sm, int base, int z,
                                            const StagePoints<TX, TY>& sp, const S* LBFD_RESTRICT T_in,
                                            const S* LBFD_RESTRICT Y_in)
{
    using G = Tile3Geom<TX, TY>;
    constexpr int NPT = G::NPT, NIT = StagePoints<TX, TY>::NIT, NTHR = TX * TY;
    int fz;
    z = stage_coord(P, z, P.nz, 2, &fz);
    const unsigned inlet = fz >= 0 && face_type(P, fz) == BC_INLET ? 0xffffffffu : sp.inlet;
    const long long zo = (long long)P.nx * P.ny * z;
    const int tid = threadIdx.x + TX * threadIdx.y;
    // all of this thread's global loads first, then the derived values
    R T[NIT], Y[NIT][NSP];
#pragma unroll
    for (int it = 0; it < NIT; ++it) {
        if ((it + 1) * NTHR > G::NPP && tid + it * NTHR >= G::NPP) continue;
        T[it] = R(*at_bytes(T_in + zo, sp.off[it]));
#pragma unroll
        for (int k = 0; k < NSP; ++k) Y[it][k] = R(*at_bytes(Y_in + (k * P.N + zo), sp.off[it]));
    }
#pragma unroll
    for (int it = 0; it < NIT; ++it) {
        if ((it + 1) * NTHR > G::NPP && tid + it * NTHR >= G::NPP) continue;
        const int pt = base + tid + it * NTHR;
        R invW = inv_molar_mass(P, Y[it]);
        R W, rho;
        eos_w(P, T[it], invW, rho, W);
        if ((inlet >> it) & 1u) {  // Dirichlet T_in, Y_in (few blocks)
            T[it] = R(2) * P.T_in - T[it];
#pragma unroll
            for (int k = 0; k < NSP; ++k) Y[it][k] = R(2) * P.Y_in[k] - Y[it][k];
            invW = inv_molar_mass(P, Y[it]);
            W = frcp(invW);
            rho = R(2) * P.rho_in - rho;
        }
        sm.T[pt] = T[it];
#pragma unroll
        for (int k = 0; k < NSP; ++k) sm.Y[k * NPT + pt] = Y[it][k];
        sm.X[pt] = W;  // the 3-D tile keeps W in the X slot
        sm.invW[pt] = invW;
        sm.rho[pt] = rho;
    }
}

// SPLIT: steps a1-a7 only; Lambda and grad rho / rho of every interior cell go
// to aux (four planes) for step_kernel_collide3d, which does a8-a10.
// CODED: the coded cells too, by `coded` (0: none, curved walls; 1: those
// next to in-domain solids; 2: and those near open faces, bit 63 of the word).
template <typename S, typename R, int TX, int TY, bool SPLIT, bool CODED, bool HI1>
__device__ __forceinline__ void tiled3d_body(const StepParams<R>& P, int zc, const S* LBFD_RESTRICT g_in,
                                             S* LBFD_RESTRICT g_out, const S* LBFD_RESTRICT T_in,
                                             S* LBFD_RESTRICT T_out, const S* LBFD_RESTRICT Y_in,
                                             S* LBFD_RESTRICT Y_out, const unsigned long long* LBFD_RESTRICT words,
                                             int coded_cells, R* LBFD_RESTRICT aux)
{
    using G = Tile3Geom<TX, TY>;
    constexpr int SX = G::SX, NPP = G::NPP, NPT = G::NPT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TileSmem<R> sm;
    sm.T = reinterpret_cast<R*>(smem_raw);
    sm.Y = sm.T + NPT;
    sm.X = sm.Y + NSP * NPT;  // one plane: W
    sm.invW = sm.X + NPT;
    sm.rho = sm.invW + NPT;

    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY, zb = blockIdx.z * zc;
    const long long N = P.N;
    const long long plane = (long long)P.nx * P.ny;
    StagePoints<TX, TY> sp;
    stage_points<S>(P, x0, y0, sp);
    // ring[j]: first point of the slot of plane z - 2 + j
    int ring[5];
#pragma unroll
    for (int j = 0; j < 5; ++j) ring[j] = j * NPP;
    for (int j = 0; j < 4; ++j) stage_plane<S, R, TX, TY>(P, sm, j * NPP, zb + j - 2, sp, T_in, Y_in);
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
    const bool inside = x < P.nx && y < P.ny;
    const int q0 = (threadIdx.y + 2) * SX + threadIdx.x + 2;  // in-plane point of this thread
    const int zend = zb + zc < P.nz ? zb + zc : P.nz;
    // in-plane byte offsets of the cell and its neighbours (periodic wrap; the
    // threads beyond the grid take its last cell and store nothing)
    unsigned oxy[3][3];
    {
        const int xc = inside ? x : P.nx - 1, yc = inside ? y : P.ny - 1;
        const unsigned xs[3] = {(unsigned)(xc == 0 ? P.nx - 1 : xc - 1), (unsigned)xc,
                                (unsigned)(xc == P.nx - 1 ? 0 : xc + 1)};
        const unsigned ys[3] = {(unsigned)(yc == 0 ? P.ny - 1 : yc - 1), (unsigned)yc,
                                (unsigned)(yc == P.ny - 1 ? 0 : yc + 1)};
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
            for (int a = 0; a < 3; ++a) oxy[b][a] = (xs[a] + (unsigned)P.nx * ys[b]) * (unsigned)sizeof(S);
    }
    constexpr unsigned long long OTHER = ~0ull;  // solid, or another kernel's cell
    unsigned long long next = inside ? words[cell_at<S>(plane * zb, oxy[1][1])] : OTHER;
    for (int z = zb; z < zend; ++z) {
        // what the cell is; the next plane's word is loaded meanwhile
        unsigned long long word = next;
        if (word != 0 && !(CODED && (coded_cells == 2 || (coded_cells == 1 && !(word >> 63))))) word = OTHER;
        const bool active = word != OTHER, coded = CODED && active && word != 0;
        const bool cw = CODED && __any_sync(0xffffffffu, coded);
        if (z + 1 < zend && inside) next = words[cell_at<S>(plane * (z + 1), oxy[1][1])];
        // a1 issued before the staging of plane z+2, so that the population
        // loads are in flight meanwhile
        const long long zo[3] = {plane * (z == 0 ? P.nz - 1 : z - 1), plane * z, plane * (z == P.nz - 1 ? 0 : z + 1)};
        const long long c = cell_at<S>(zo[1], oxy[1][1]);
        R g[27];
#pragma unroll
        for (int i = 0; i < 27; ++i)
            g[i] = R(LBFD_LDG(at_bytes(g_in + ((long long)i * N + zo[1 - cz_of(i)]), oxy[1 - cy_of(i)][1 - cx_of(i)])));
        unsigned cross = 0;
        if (cw) {
            // from a solid neighbour or beyond a face: the opposite population
            // of the cell itself (Eq. 28; the face rules follow below)
            unsigned own = 0;
            if (coded) {
                if (word >> 63) cross = face_crossing(P, x, y, z);
                own = ((unsigned)word & 0x7ffffffu) | cross;
            }
#pragma unroll
            for (int i = 0; i < 27; ++i)
                if ((own >> i) & 1u) 
                    g[i] = R(LBFD_LDG(at_bytes(g_in + ((long long)opposite<3>(i) * N + zo[1]), oxy[1][1])));
        }
        stage_plane<S, R, TX, TY>(P, sm, ring[4], z + 2, sp, T_in, Y_in);
        __syncthreads();
        const int p0 = ring[2] + q0;
        if (active) {
            const R T0 = sm.T[p0], invW0 = sm.invW[p0], rho0 = sm.rho[p0];
            const R inv_rho0 = T0 * invW0 * par<R>(P.inv_rho_c);
            if constexpr (CODED) {
                if (cross) face_rules<S, R>(P, cross, g_in + c, rho0, inv_rho0, g);
            }
            LowMoments<3, R> lm;
            low_moments<3>(g, lm);
            R u[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) u[a] = lm.m1[a] * (K<R>(3) * inv_rho0);
            FDAccum<R> acc;
            acc.clear();
            // the three axes share one copy of the FD code (a rolled loop keeps
            // the kernel small enough for the instruction cache)
#pragma unroll 1
            for (int a = 0; a < 3; ++a) {
                int pts[5];
                const int st = a == 0 ? 1 : SX;
#pragma unroll
                for (int j = 0; j < 5; ++j) pts[j] = a == 2 ? ring[j] + q0 : p0 + (j - 2) * st;
                unsigned dir = 0, code6 = 0;
                if (CODED && cw) {
                    code6 = (unsigned)(word >> (32 + 6 * a)) & 63u;
                    dir = coded_pts(code6, (unsigned)(word >> (50 + 2 * a)) & 3u, pts);
                    if (!P.solid_isothermal) dir = 0;
                }
                const R u_a = a == 0 ? u[0] : (a == 1 ? u[1] : u[2]);
                R gam;
                fd_axis_pts<CODED, R>(P, sm, NPT, pts, cw, dir, code6 != 0, u_a, invW0, inv_rho0, &gam, acc);
                acc.gam[0] = a == 0 ? gam : acc.gam[0];
                acc.gam[1] = a == 1 ? gam : acc.gam[1];
                acc.gam[2] = a == 2 ? gam : acc.gam[2];
            }
            R Y0[NSP];
#pragma unroll
            for (int k = 0; k < NSP; ++k) Y0[k] = sm.Y[k * NPT + p0];
            const R Lam = update_scalars<S, R>(P, c, T0, Y0, rho0 * invW0 * par<R>(P.inv_rho_c), sm.X[p0], acc, T_out,
                                               Y_out);
            if constexpr (SPLIT) {
                aux[c] = Lam;
#pragma unroll
                for (int a = 0; a < 3; ++a) aux[(long long)(1 + a) * N + c] = acc.gam[a];
            } else {
                if constexpr (HI1) collide_hi1<3, R>(P, lm, rho0, inv_rho0, u, acc.gam, Lam, g);
                else collide<3, R>(P, g, rho0, inv_rho0, u, acc.gam, Lam);
#pragma unroll
                for (int i = 0; i < 27; ++i) *at_bytes(g_out + ((long long)i * N + zo[1]), oxy[1][1]) = S(g[i]);
            }
        }
        __syncthreads();  // the slot of z-2 is restaged next iteration
        const int oldest = ring[0];
#pragma unroll
        for (int j = 0; j < 4; ++j) ring[j] = ring[j + 1];
        ring[4] = oldest;
    }
}

// interior and coded cells; the registers capped so that MINB blocks fit on
// an SM (left to itself the compiler hoists addresses until 255 are used)
template <typename S, typename R, int TX, int TY, int MINB, bool HI1>
__global__ void __launch_bounds__(TX * TY, MINB)
    step_kernel_tiled3d(StepParams<R> P, int zc, const S* LBFD_RESTRICT g_in, S* LBFD_RESTRICT g_out,
                               const S* LBFD_RESTRICT T_in, S* LBFD_RESTRICT T_out, const S* LBFD_RESTRICT Y_in,
                               S* LBFD_RESTRICT Y_out, const unsigned long long* LBFD_RESTRICT words,
                               int coded_cells)
{
    tiled3d_body<S, R, TX, TY, false, true, HI1>(P, zc, g_in, g_out, T_in, T_out, Y_in, Y_out, words, coded_cells,
                                                 nullptr);
}

// a1-a7 of the interior cells (the FD half of a split step); FP32 held to
// four 128-thread blocks per SM
template <typename S, typename R, int TX, int TY>
__global__ void __launch_bounds__(TX * TY, sizeof(R) == 4 ? 512 / (TX * TY) : 1)
    step_kernel_fd3d(StepParams<R> P, int zc, const S* LBFD_RESTRICT g_in, const S* LBFD_RESTRICT T_in,
                     S* LBFD_RESTRICT T_out,
                     const S* LBFD_RESTRICT Y_in, S* LBFD_RESTRICT Y_out,
                     const unsigned long long* LBFD_RESTRICT words, R* LBFD_RESTRICT aux)
{
    tiled3d_body<S, R, TX, TY, true, false, false>(P, zc, g_in, nullptr, T_in, T_out, Y_in, Y_out, words, 0, aux);
}

// a1, a2 and a8-a10 of the interior cells (the LB half of a split step):
// the pull and the density are recomputed exactly as in the FD half, Lambda
// and grad rho / rho read from aux.  One thread per cell, 128 cells of an x-row
// per block.
template <typename S, typename R, bool HI1>
__global__ void __launch_bounds__(128)
    step_kernel_collide3d(StepParams<R> P, const S* LBFD_RESTRICT g_in, S* LBFD_RESTRICT g_out,
                          const S* LBFD_RESTRICT T_in, const S* LBFD_RESTRICT Y_in,
                          const unsigned long long* LBFD_RESTRICT words, const R* LBFD_RESTRICT aux)
{
    const int x = blockIdx.x * 128 + threadIdx.x, y = blockIdx.y, z = blockIdx.z;
    if (x >= P.nx) return;
    const long long N = P.N;
    const long long plane = (long long)P.nx * P.ny;
    const long long c = (long long)x + (long long)P.nx * y + plane * z;
    if (words[c] != 0) return;
    R g[27];
    {
        const int oxm = x == 0 ? P.nx - 1 : -1, oxp = x == P.nx - 1 ? 1 - P.nx : 1;
        const long long oym = y == 0 ? (long long)(P.ny - 1) * P.nx : -(long long)P.nx;
        const long long oyp = y == P.ny - 1 ? (long long)(1 - P.ny) * P.nx : (long long)P.nx;
        const long long ozm = z == 0 ? (P.nz - 1) * plane : -plane;
        const long long ozp = z == P.nz - 1 ? (1 - P.nz) * plane : plane;
        const S* gc = g_in + c;
#pragma unroll
        for (int i = 0; i < 27; ++i) {
            const long long o = (cx_of(i) > 0 ? oxm : (cx_of(i) < 0 ? oxp : 0)) +
                                (cy_of(i) > 0 ? oym : (cy_of(i) < 0 ? oyp : 0)) +
                                (cz_of(i) > 0 ? ozm : (cz_of(i) < 0 ? ozp : 0));
            g[i] = R(LBFD_LDG(gc + (long long)i * N + o));
        }
    }
    // the density as staged by the FD half
    const R T0 = R(T_in[c]);
    R Y0[NSP];
#pragma unroll
    for (int k = 0; k < NSP; ++k) Y0[k] = R(Y_in[(long long)k * N + c]);
    const R invW0 = inv_molar_mass(P, Y0);
    R rho0, W0;
    eos_w(P, T0, invW0, rho0, W0);
    const R inv_rho0 = T0 * invW0 * par<R>(P.inv_rho_c);
    LowMoments<3, R> lm;
    low_moments<3>(g, lm);
    R u[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) u[a] = lm.m1[a] * (K<R>(3) * inv_rho0);
    const R Lam = aux[c];
    R gam[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) gam[a] = aux[(long long)(1 + a) * N + c];
    if constexpr (HI1) collide_hi1<3, R>(P, lm, rho0, inv_rho0, u, gam, Lam, g);
    else collide<3, R>(P, g, rho0, inv_rho0, u, gam, Lam);
#pragma unroll
    for (int i = 0; i < 27; ++i) g_out[(long long)i * N + c] = S(g[i]);
}

}  // namespace lbfd
