// lbfd_adjoint_direct.cu -- the transpose of one 2-D step by hand-derived
// local adjoints: lambda^n += (dF/dx^n)^T lambda^{n+1}, dtheta +=
// (dF/dtheta)^T lambda^{n+1}, theta = (ln A, Ta, T_wall, u_in), in one launch
// and without a tape.
//
// Every cell's step is evaluated at the state of that step in FP64 (an FP32
// state is widened), then differentiated backwards: the outputs' adjoints
// through the collision (collide2_adjoint) to the moments, the velocity, grad
// rho / rho and Lambda, then through the FD terms of each axis to the line
// points, and last through the pull.  The one-warp blocks of the small-grid
// step: the first take the coded boundary cells, the others 8x4 interior
// tiles, whose line adjoints are summed per staged point in shared memory
// (T, Y_k, Y_k W, 1/W and rho apart) and turned into adjoints of T and Y_k
// once per point.  Neighbouring tiles meet in FP64 atomic adds.
//
// The tape it replaces (recorded per operation, swept node by node) moved
// 2.3 GB and took 0.86 ms per step of a 512x64 grid (record and sweep
// overlapped); this takes 0.19 ms, bound by the FP64 pipe: 2 144 FP64
// instructions of 64 cycles per warp of 32 cells, two warps on most SM
// partitions.  The line sums are formed twice (for Lambda, then for their
// adjoints) rather than kept: 180 FP64 instructions against 250 registers.
#include "lbfd_adjoint_cell.cuh"
#include "lbfd_step_small.cuh"

namespace lbfd {

namespace {

// What a cell's reverse pass carries between its parts: values of the
// forward step and adjoints of its intermediate quantities.
struct CellReverse {
    // forward
    double T0, invW0, W0, rho0, irho, iT;
    double Y0[NSP], u[2];
    LowMoments<2, double> lm;
    double D1rho[2], gam[2], diff_T, lamY;
    // adjoints
    double bT0, binvW0, brho0, birho, bY0[NSP], bu[2], bgam[2];
    double lT, lY[NSP];   // of the outputs T and Y_k
    double l, cT, dT, z;  // of lamY, conv_T, diff_T and `along`
    double th[4];
};

// forward FD terms of one axis that Lambda and grad rho need
template <typename Lines>
__device__ __forceinline__ void forward_axis(const StepParams<double>& P, int a, const Lines& L, CellReverse& r)
{
    double v[5];
    L.rho(v);
    r.D1rho[a] = fd_D1(v);
    const double gam = r.D1rho[a] * r.irho * (1.0 / 12.0);
    r.gam[a] = gam;
    L.T(v);
    r.diff_T += P.alpha12 * (fd_D2(v) + gam * fd_D1(v));
    L.invW(v);
    const double dinv = fd_D1(v) * (1.0 / 12.0), b = dinv + r.invW0 * gam;
    double M = 0.0, F = 0.0, lam = 0.0;
#pragma unroll 1
    for (int k = 0; k < NSP; ++k) {
        L.X(k, v);
        const double dX = fd_D1(v), f = P.a12[k] * (r.invW0 * fd_D2(v) + b * dX);
        M += P.a12[k] * dX;
        F += f;
        lam += P.inv_Wk[k] * f;
    }
    r.lamY += (lam - M * r.invW0 * dinv) - r.invW0 * F;
}

// From the forward terms and the outputs' adjoints to the adjoints of the
// moments (bm0, bm1, bm2), of u and grad rho / rho, and of the FD sums.
__device__ __forceinline__ void reverse_centre(const StepParams<double>& P, const double* lg, CellReverse& r,
                                               Collision2& b)
{
    const double yf = pick_species(r.Y0, P.fuel), yo = pick_species(r.Y0, P.oxid);
    const double yfp = yf > 0.0 ? yf : 0.0, yop = yo > 0.0 ? yo : 0.0;
    const double ex = P.A_lat * ::exp(-P.Ta * r.iT), q = ex * yfp * yop;
    const double DT = r.diff_T + P.Q_cp * q, lamq = r.lamY + P.lam_yield * q;
    Collision2 s;
    s.m0 = r.lm.m0;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        s.m1[a] = r.lm.m1[a];
        s.u[a] = r.u[a];
        s.gam[a] = r.gam[a];
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) s.m2[j] = r.lm.m2[j];
    s.rho = r.rho0;
    s.irho = r.irho;
    s.Lam = DT * r.iT + lamq * r.W0;
    collide2_adjoint(s, P.one_minus_omega_s, P.omega_s_minus_b, lg, b, nullptr);
    r.brho0 += b.rho;
    r.birho += b.irho;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        r.bu[a] = b.u[a];
        r.bgam[a] = b.gam[a];
    }
    // Lambda = DT / T0 + (lamY + lam_yield q) / invW0
    r.dT = b.Lam * r.iT + r.lT;
    r.bT0 += r.lT - b.Lam * DT * r.iT * r.iT;
    r.l = b.Lam * r.W0;
    r.binvW0 -= b.Lam * lamq * r.W0 * r.W0;
    // the Euler update
    r.cT = -r.lT;
    double bq = r.l * P.lam_yield + r.dT * P.Q_cp;
    r.z = 0.0;
#pragma unroll
    for (int k = 0; k < NSP; ++k) {
        bq += r.lY[k] * P.yield[k];
        r.z += r.lY[k] * r.Y0[k];
        r.bY0[k] += r.lY[k];
    }
    // the rate
    r.th[0] += bq * q;
    r.th[1] -= bq * q * r.iT;
    r.bT0 += bq * q * P.Ta * r.iT * r.iT;
    const double bf = yf > 0.0 ? bq * ex * yop : 0.0, bo = yo > 0.0 ? bq * ex * yfp : 0.0;
#pragma unroll
    for (int k = 0; k < NSP; ++k) r.bY0[k] += (k == P.fuel ? bf : 0.0) + (k == P.oxid ? bo : 0.0);
}

// The FD terms of one axis backwards.  add.pts(field weights) gets the line
// points' adjoints: add.T(v), add.rho_invW(r, w), add.YX(k, y, x).
template <typename Lines, typename Add>
__device__ __forceinline__ void reverse_axis(const StepParams<double>& P, int a, bool near, const Lines& L, Add& add,
                                             CellReverse& r)
{
    const double c1[5] = {1.0, -8.0, 0.0, 8.0, -1.0}, c2[5] = {-1.0, 16.0, -30.0, 16.0, -1.0};
    const double u = r.u[a], gam = r.gam[a];
    const bool neg = u < 0.0;
    const double ua = neg ? -u : u;
    double v[5], w[5], x[5];
    L.invW(v);
    const double dinv = fd_D1(v) * (1.0 / 12.0), b = dinv + r.invW0 * gam;
    // the species sums of the forward terms
    double Mp = 0.0, F = 0.0, SL = 0.0, yD = 0.0, yL = 0.0;
#pragma unroll 1
    for (int k = 0; k < NSP; ++k) {
        L.X(k, v);
        const double dX = fd_D1(v);
        Mp += P.a12[k] * dX;
        F += P.a12[k] * (r.invW0 * fd_D2(v) + b * dX);
    }
    const double M = Mp * r.invW0;
    const double bF = -r.z - r.l * r.invW0, bSL = r.z * ua;
    double bdinv = -r.l * M, bb = 0.0;
    r.binvW0 -= r.l * F;
    // Y lines first (their adjoint of M enters the X lines)
    double bM = -r.l * dinv;
#pragma unroll 1
    for (int k = 0; k < NSP; ++k) {
        L.Y(k, v);
        const double Lk = conv_partials(v, neg, P.epsY, near, w);
        SL += Lk;
        const double D = fd_D1(v), bD = -r.lY[k] * M * (1.0 / 12.0), bL = bSL - r.lY[k] * ua;
        yD += r.lY[k] * D;
        yL += r.lY[k] * Lk;
#pragma unroll
        for (int j = 0; j < 5; ++j) x[j] = bL * w[j] + bD * c1[j];
        add.Y(k, x);
    }
    bM -= yD * (1.0 / 12.0);
    double bua = r.z * SL - yL;
    const double along = ua * SL - F, bMp = bM * r.invW0;
    r.binvW0 += bM * Mp;
#pragma unroll
    for (int k = 0; k < NSP; ++k) r.bY0[k] += r.lY[k] * along;
#pragma unroll 1
    for (int k = 0; k < NSP; ++k) {
        L.X(k, v);
        const double bf = P.a12[k] * (r.lY[k] + bF + r.l * P.inv_Wk[k]);
        const double dX = fd_D1(v), bd1 = bf * b + bMp * P.a12[k], bd2 = bf * r.invW0;
        r.binvW0 += bf * fd_D2(v);
        bb += bf * dX;
#pragma unroll
        for (int j = 0; j < 5; ++j) x[j] = bd2 * c2[j] + bd1 * c1[j];
        add.X(k, x);
    }
    // T
    L.T(v);
    const double LT = conv_partials(v, neg, P.epsT, near, w);
    bua += r.cT * LT;
    const double bD2 = r.dT * P.alpha12, bD1 = bD2 * gam, bLT = r.cT * ua;
    double bgam = r.bgam[a] + bD2 * fd_D1(v) + bb * r.invW0;
#pragma unroll
    for (int j = 0; j < 5; ++j) x[j] = bLT * w[j] + (bD2 * c2[j] + bD1 * c1[j]);
    add.T(x);
    // b = d(1/W) + invW0 gam, gam = D1 rho / (12 rho0)
    bdinv += bb;
    r.binvW0 += bb * gam;
    r.birho += bgam * r.D1rho[a] * (1.0 / 12.0);
    const double br = bgam * r.irho * (1.0 / 12.0), bw = bdinv * (1.0 / 12.0);
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        x[j] = br * c1[j];
        v[j] = bw * c1[j];
    }
    add.rho_invW(x, v);
    r.bu[a] += neg ? -bua : bua;
}

// u, 1/rho and the pulled populations' adjoints bg
__device__ __forceinline__ void reverse_moments(CellReverse& r, Collision2& b, double* bg)
{
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        b.m1[a] += 3.0 * r.irho * r.bu[a];
        r.birho += 3.0 * r.lm.m1[a] * r.bu[a];
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int cx = cx_of(i), cy = cy_of(i);
        double s = b.m0;
        if (cx) s += cx * b.m1[0] + b.m2[0];
        if (cy) s += cy * b.m1[1] + b.m2[1];
        if (cx && cy) s += cx * cy * b.m2[2];
        bg[i] = s;
    }
}

// adjoints of T, Y_k, Y_k W, 1/W and rho of a point with these values, as
// adjoints of its T and Y_k, added to lambda at cell c
__device__ __forceinline__ void scatter_point(const StepParams<double>& P, long long c, double T, const double* Y,
                                              double invW, double rho, double bT, double* bY, const double* bX,
                                              double binvW, double brho, double* lam)
{
    const double W = rho * T * P.inv_rho_c, iT = rho * invW * P.inv_rho_c;
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < NSP; ++k) {
        s += bX[k] * Y[k];
        bY[k] += bX[k] * W;
    }
    binvW -= W * (W * s + brho * rho);
    bT -= brho * rho * iT;
    atomicAdd(&lam[9 * P.N + c], bT);
#pragma unroll
    for (int k = 0; k < NSP; ++k) atomicAdd(&lam[(10 + k) * P.N + c], bY[k] + binvW * P.inv_Wk[k]);
}

__device__ __forceinline__ void load_cell(const StepParams<double>& P, long long c, const double* lam_next,
                                          CellReverse& r, double* lg)
{
    r.lT = lam_next[9 * P.N + c];
#pragma unroll
    for (int k = 0; k < NSP; ++k) r.lY[k] = lam_next[(10 + k) * P.N + c];
#pragma unroll
    for (int i = 0; i < 9; ++i) lg[i] = lam_next[i * P.N + c];
}

__device__ __forceinline__ void begin_cell(const StepParams<double>& P, const double* g, CellReverse& r)
{
    r.irho = r.T0 * r.invW0 * P.inv_rho_c;
    r.iT = r.rho0 * r.invW0 * P.inv_rho_c;
    low_moments<2>(g, r.lm);
    r.diff_T = r.lamY = 0.0;
    r.bT0 = r.binvW0 = r.brho0 = r.birho = 0.0;
#pragma unroll
    for (int a = 0; a < 2; ++a) r.u[a] = r.lm.m1[a] * (3.0 * r.irho);
#pragma unroll
    for (int k = 0; k < NSP; ++k) r.bY0[k] = 0.0;
}

// 1/rho0 = T0 invW0 / rho_c
__device__ __forceinline__ void end_cell(const StepParams<double>& P, CellReverse& r)
{
    r.bT0 += r.birho * r.invW0 * P.inv_rho_c;
    r.binvW0 += r.birho * r.T0 * P.inv_rho_c;
}

struct TileLines {
    const TileSmem<double>& sm;
    int p0, st;
    static constexpr int NPT = TileGeom<SM_TX, SM_TY>::NPT;
    __device__ __forceinline__ void line(const double* f, double* v) const
    {
#pragma unroll
        for (int j = 0; j < 5; ++j) v[j] = f[p0 + (j - 2) * st];
    }
    __device__ __forceinline__ void rho(double* v) const { line(sm.rho, v); }
    __device__ __forceinline__ void T(double* v) const { line(sm.T, v); }
    __device__ __forceinline__ void invW(double* v) const { line(sm.invW, v); }
    __device__ __forceinline__ void X(int k, double* v) const { line(sm.X + k * NPT, v); }
    __device__ __forceinline__ void Y(int k, double* v) const { line(sm.Y + k * NPT, v); }
};
// Adds line adjoints to the staged points of the block's one warp: for each
// of the five positions in turn the lanes' points are distinct, and the warp
// is synchronised before the next.
struct TileAdd {
    const TileSmem<double>& bs;  // the accumulators, laid out as the staged fields
    int p0, st;
    bool on;
    static constexpr int NPT = TileGeom<SM_TX, SM_TY>::NPT;
    __device__ __forceinline__ void line(double* f, const double* v) const
    {
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            if (on) f[p0 + (j - 2) * st] += v[j];
            __syncwarp();
        }
    }
    __device__ __forceinline__ void T(const double* v) const { line(bs.T, v); }
    __device__ __forceinline__ void Y(int k, const double* v) const { line(bs.Y + k * NPT, v); }
    __device__ __forceinline__ void X(int k, const double* v) const { line(bs.X + k * NPT, v); }
    __device__ __forceinline__ void rho_invW(const double* r, const double* w) const
    {
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            if (on && j != 2) {
                bs.rho[p0 + (j - 2) * st] += r[j];
                bs.invW[p0 + (j - 2) * st] += w[j];
            }
            __syncwarp();
        }
    }
};

template <typename S>
__device__ __forceinline__ void reverse_tile(const StepParams<double>& P, const S* __restrict__ g_in,
                                             const S* __restrict__ T_in, const S* __restrict__ Y_in,
                                             const uint8_t* __restrict__ interior, const double* __restrict__ lam_next,
                                             double* __restrict__ lam, int bx, int by, double* th)
{
    using G = TileGeom<SM_TX, SM_TY>;
    constexpr int SX = G::SX, NPT = G::NPT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const TileSmem<double> sm = tile_smem<double, SM_TX, SM_TY>(smem_raw);
    const TileSmem<double> bs = tile_smem<double, SM_TX, SM_TY>(smem_raw + tile_smem_bytes<double, SM_TX, SM_TY>());
    const int lane = threadIdx.x, tx = lane % SM_TX, ty = lane / SM_TX;
    const int x0 = bx * SM_TX, y0 = by * SM_TY, x = x0 + tx, y = y0 + ty;
    const bool inside = x < P.nx && y < P.ny;
    const long long c = inside ? (long long)x + (long long)P.nx * y : 0;
    const bool on = inside && interior[c] == 1;
    double g[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = 0.0;
    if (on) pull_interior<S, double>(P, g_in, c, x, y, g);
    stage_tile2d<S, double, SM_TX, SM_TY, false, 32>(P, sm, x0, y0, lane, T_in, Y_in);
    for (int j = lane; j < NPT * (3 + 2 * NSP); j += 32) bs.T[j] = 0.0;
    __syncwarp();
    if (!__any_sync(0xffffffffu, on)) return;
    // lanes without an interior cell follow (the warp is synchronised below)
    // on the values of one that has one, and add nothing
    const int src = __ffs(__ballot_sync(0xffffffffu, on)) - 1;
    const int p_own = (ty + 2) * SX + tx + 2, p_any = __shfl_sync(0xffffffffu, p_own, src);
    const int p0 = on ? p_own : p_any;
    CellReverse r;
    double lg[9];
    const long long c_any = __shfl_sync(0xffffffffu, c, src), cc = on ? c : c_any;
    load_cell(P, cc, lam_next, r, lg);
    r.T0 = sm.T[p0];
    r.invW0 = sm.invW[p0];
    r.rho0 = sm.rho[p0];
    r.W0 = r.rho0 * r.T0 * P.inv_rho_c;
#pragma unroll
    for (int k = 0; k < NSP; ++k) r.Y0[k] = sm.Y[k * NPT + p0];
#pragma unroll
    for (int j = 0; j < 4; ++j) r.th[j] = 0.0;
    begin_cell(P, g, r);
    forward_axis(P, 0, TileLines{sm, p0, 1}, r);
    forward_axis(P, 1, TileLines{sm, p0, SX}, r);
    Collision2 b{};
    reverse_centre(P, lg, r, b);
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        TileAdd add{bs, p0, a ? SX : 1, on};
        reverse_axis(P, a, false, TileLines{sm, p0, a ? SX : 1}, add, r);
    }
    double bg[9];
    reverse_moments(r, b, bg);
    end_cell(P, r);
    if (on) {
        bs.T[p0] += r.bT0;
        bs.invW[p0] += r.binvW0;
        bs.rho[p0] += r.brho0;
#pragma unroll
        for (int k = 0; k < NSP; ++k) bs.Y[k * NPT + p0] += r.bY0[k];
        const int oxm = x == 0 ? P.nx - 1 : -1, oxp = x == P.nx - 1 ? 1 - P.nx : 1;
        const int oym = y == 0 ? (P.ny - 1) * P.nx : -P.nx, oyp = y == P.ny - 1 ? (1 - P.ny) * P.nx : P.nx;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int o = (cx_of(i) > 0 ? oxm : (cx_of(i) < 0 ? oxp : 0)) + (cy_of(i) > 0 ? oym : (cy_of(i) < 0 ? oyp : 0));
            atomicAdd(&lam[i * P.N + c + o], bg[i]);
        }
        th[0] = r.th[0];
        th[1] = r.th[1];
    }
    __syncwarp();
    // the staged points' sums, once per point (three per lane)
#pragma unroll 1
    for (int pt = lane; pt < NPT; pt += 32) {
        double bY[NSP], bX[NSP], Yp[NSP];
        const double bT = bs.T[pt], bw = bs.invW[pt], br = bs.rho[pt];
        bool any = bT != 0.0 || bw != 0.0 || br != 0.0;
#pragma unroll
        for (int k = 0; k < NSP; ++k) {
            bY[k] = bs.Y[k * NPT + pt];
            bX[k] = bs.X[k * NPT + pt];
            Yp[k] = sm.Y[k * NPT + pt];
            any |= bY[k] != 0.0 || bX[k] != 0.0;
        }
        if (!any) continue;  // no interior cell's line reaches it
        int gx = x0 + pt % SX - 2, gy = y0 + pt / SX - 2;
        gx = ((gx % P.nx) + P.nx) % P.nx;  // across a periodic face (others are out of an interior cell's reach)
        gy = ((gy % P.ny) + P.ny) % P.ny;
        scatter_point(P, (long long)gx + (long long)P.nx * gy, sm.T[pt], Yp, sm.invW[pt], sm.rho[pt], bT, bY, bX, bw,
                      br, lam);
    }
}

struct CodedLines {
    const double *Tl, (*Yl)[5], *wl, *Wl, *rl;
    __device__ __forceinline__ void copy(const double* f, double* v) const
    {
#pragma unroll
        for (int j = 0; j < 5; ++j) v[j] = f[j];
    }
    __device__ __forceinline__ void rho(double* v) const { copy(rl, v); }
    __device__ __forceinline__ void T(double* v) const { copy(Tl, v); }
    __device__ __forceinline__ void invW(double* v) const { copy(wl, v); }
    __device__ __forceinline__ void X(int k, double* v) const
    {
#pragma unroll
        for (int j = 0; j < 5; ++j) v[j] = Yl[k][j] * Wl[j];
    }
    __device__ __forceinline__ void Y(int k, double* v) const { copy(Yl[k], v); }
};
struct CodedAdd {
    double bT[5], bY[NSP][5], bX[NSP][5], br[5], bw[5];
    __device__ __forceinline__ void T(const double* v)
    {
#pragma unroll
        for (int j = 0; j < 5; ++j) bT[j] = v[j];
    }
    __device__ __forceinline__ void Y(int k, const double* v)
    {
#pragma unroll
        for (int j = 0; j < 5; ++j) bY[k][j] = v[j];
    }
    __device__ __forceinline__ void X(int k, const double* v)
    {
#pragma unroll
        for (int j = 0; j < 5; ++j) bX[k][j] = v[j];
    }
    __device__ __forceinline__ void rho_invW(const double* r, const double* w)
    {
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            br[j] = r[j];
            bw[j] = w[j];
        }
    }
};

template <typename S>
__device__ __forceinline__ void coded_points(const StepParams<double>& P, const int p[3], long long c, int a,
                                             unsigned long long code, const S* __restrict__ T_in,
                                             const S* __restrict__ Y_in, LineDesc<double>& L, double* Tl,
                                             double (*Yl)[5], double* wl, double* Wl, double* rl)
{
    coded_line<2, double>(P, p, c, a, (unsigned)(code >> (32 + 6 * a)) & 63u, (unsigned)(code >> (50 + 2 * a)) & 3u, L);
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        double Yj[NSP];
        line_point<S, double>(P, L, j, T_in, Y_in, Tl[j], Yj, wl[j], Wl[j], rl[j]);
#pragma unroll
        for (int k = 0; k < NSP; ++k) Yl[k][j] = Yj[k];
    }
}

template <typename S>
__device__ __forceinline__ void reverse_coded(const StepParams<double>& P, long long c, unsigned long long code,
                                              const S* __restrict__ g_in, const S* __restrict__ T_in,
                                              const S* __restrict__ Y_in, const double* __restrict__ lam_next,
                                              double* __restrict__ lam, double* th)
{
    const int p[3] = {(int)(c % P.nx), (int)(c / P.nx), 0};
    const long long N = P.N;
    CellReverse r;
    double lg[9], g[9];
    load_cell(P, c, lam_next, r, lg);
    r.T0 = (double)T_in[c];
#pragma unroll
    for (int k = 0; k < NSP; ++k) r.Y0[k] = (double)Y_in[k * N + c];
    r.invW0 = inv_molar_mass(P, r.Y0);
    eos_w(P, r.T0, r.invW0, r.rho0, r.W0);
#pragma unroll
    for (int j = 0; j < 4; ++j) r.th[j] = 0.0;
    pull_coded<2, S, double, true>(P, p, c, code, r.rho0, r.T0 * r.invW0 * P.inv_rho_c, g_in, g);
    begin_cell(P, g, r);
    LineDesc<double> L;
    double Tl[5], Yl[NSP][5], wl[5], Wl[5], rl[5];
#pragma unroll 1
    for (int a = 0; a < 2; ++a) {
        coded_points<S>(P, p, c, a, code, T_in, Y_in, L, Tl, Yl, wl, Wl, rl);
        forward_axis(P, a, CodedLines{Tl, Yl, wl, Wl, rl}, r);
    }
    Collision2 b{};
    reverse_centre(P, lg, r, b);
    // the centre's own sums over both axes
    double cT = 0.0, cw = 0.0, cr = 0.0, cY[NSP] = {}, cX[NSP] = {};
#pragma unroll 1
    for (int a = 0; a < 2; ++a) {
        coded_points<S>(P, p, c, a, code, T_in, Y_in, L, Tl, Yl, wl, Wl, rl);
        CodedAdd add;
        reverse_axis(P, a, L.near != 0, CodedLines{Tl, Yl, wl, Wl, rl}, add, r);
#pragma unroll 1
        for (int j = 0; j < 5; ++j) {
            double bT = add.bT[j], bw = add.bw[j], br = add.br[j], bY[NSP], bX[NSP];
#pragma unroll
            for (int k = 0; k < NSP; ++k) {
                bY[k] = add.bY[k][j];
                bX[k] = add.bX[k][j];
            }
            const int mode = L.mode[j];
            // the point's mirror cell (itself when it is no ghost)
            const long long m = L.src[j];
            const double Tm = (double)T_in[m];
            double Ym[NSP];
#pragma unroll
            for (int k = 0; k < NSP; ++k) Ym[k] = (double)Y_in[k * N + m];
            const double wm = inv_molar_mass(P, Ym), Em = frcp(Tm * wm), rm = P.rho_c * Em;
            if (mode == G_DIRICHLET_T) {  // T = 2 TB - Tm, rho = 2 rho_c / (TB invW) - rho_m
                const double TB = L.TB[j], e = P.rho_c * frcp(TB * wm);
                r.th[2] += 2.0 * bT - 2.0 * br * e * frcp(TB);
                bw -= 2.0 * br * e * (Tm * Em);
                bT = -bT;
                br = -br;
            } else if (mode == G_INLET) {  // T = 2 T_in - Tm, Y = 2 Y_in - Ym (and Y W, 1/W of it), rho = 2 - rho_m
                double s = 0.0;
#pragma unroll
                for (int k = 0; k < NSP; ++k) {
                    s += bX[k] * Yl[k][j];
                    bY[k] += bX[k] * Wl[j];
                    bX[k] = 0.0;
                }
                bw -= Wl[j] * Wl[j] * s;
#pragma unroll
                for (int k = 0; k < NSP; ++k) bY[k] = -(bY[k] + bw * P.inv_Wk[k]);
                bw = 0.0;
                bT = -bT;
                br = -br;
            }
            if (m == c) {
                cT += bT;
                cw += bw;
                cr += br;
#pragma unroll
                for (int k = 0; k < NSP; ++k) {
                    cY[k] += bY[k];
                    cX[k] += bX[k];
                }
            } else {
                scatter_point(P, m, Tm, Ym, wm, rm, bT, bY, bX, bw, br, lam);
            }
        }
    }
    double bg[9];
    reverse_moments(r, b, bg);
    // the pull backwards (the rules of pull_coded)
    const int oxm = p[0] == 0 ? P.nx - 1 : -1, oxp = p[0] == P.nx - 1 ? 1 - P.nx : 1;
    const int oym = p[1] == 0 ? (P.ny - 1) * P.nx : -P.nx, oyp = p[1] == P.ny - 1 ? (1 - P.ny) * P.nx : P.nx;
    double uc[2] = {0.0, 0.0}, buc[2] = {0.0, 0.0}, mc[2] = {0.0, 0.0};
    bool outlet = false;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
        outlet |= p[a] == 0 && P.bc[2 * a] == BC_OUTLET_PRESSURE;
        outlet |= p[a] == (a == 0 ? P.nx : P.ny) - 1 && P.bc[2 * a + 1] == BC_OUTLET_PRESSURE;
    }
    if (outlet) {
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            const double gj = (double)g_in[j * N + c];
            mc[0] += cx_of(j) * gj;
            mc[1] += cy_of(j) * gj;
        }
        uc[0] = 3.0 * mc[0] * r.irho;
        uc[1] = 3.0 * mc[1] * r.irho;
    }
    const double uu = uc[0] * uc[0] + uc[1] * uc[1];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int cx = cx_of(i), cy = cy_of(i), ib = opposite<2>(i);
        int f = -1;
        if (cx > 0 && p[0] == 0 && P.bc[0] != BC_PERIODIC) f = 0;
        if (cx < 0 && p[0] == P.nx - 1 && P.bc[1] != BC_PERIODIC) f = 1;
        if (cy > 0 && p[1] == 0 && P.bc[2] != BC_PERIODIC) f = 2;
        if (cy < 0 && p[1] == P.ny - 1 && P.bc[3] != BC_PERIODIC) f = 3;
        const bool bb = (code >> i) & 1ull;
        if (bb || f < 0) {
            const int o = (cx > 0 ? oxm : (cx < 0 ? oxp : 0)) + (cy > 0 ? oym : (cy < 0 ? oyp : 0));
            atomicAdd(&lam[bb ? ib * N + c : i * N + c + o], bg[i]);
            continue;
        }
        const double wi = weight<2, double>(i);
        if (face_type(P, f) == BC_INLET) {
            double prof = 1.0;
            if (P.poiseuille && f < 2) {
                const double ny = P.ny, y = p[1] + 0.5;
                prof = 6.0 * y * (ny - y) / (ny * ny);
            }
            r.th[3] += bg[i] * 2.0 * wi * P.rho_in * prof;
            atomicAdd(&lam[ib * N + c], bg[i]);
        } else {  // g_i = 2 w rho (3/2 (c.u)^2 - u.u/2) - g_ibar
            const double cu = cx * uc[0] + cy * uc[1];
            r.brho0 += bg[i] * 2.0 * wi * (1.5 * cu * cu - 0.5 * uu);
            buc[0] += bg[i] * 2.0 * wi * r.rho0 * (3.0 * cu * cx - uc[0]);
            buc[1] += bg[i] * 2.0 * wi * r.rho0 * (3.0 * cu * cy - uc[1]);
            atomicAdd(&lam[ib * N + c], -bg[i]);
        }
    }
    if (outlet) {
        r.birho += 3.0 * (mc[0] * buc[0] + mc[1] * buc[1]);
#pragma unroll
        for (int j = 0; j < 9; ++j)
            if (j != 4) atomicAdd(&lam[j * N + c], 3.0 * r.irho * (cx_of(j) * buc[0] + cy_of(j) * buc[1]));
    }
    end_cell(P, r);
#pragma unroll
    for (int k = 0; k < NSP; ++k) cY[k] += r.bY0[k];
    scatter_point(P, c, r.T0, r.Y0, r.invW0, r.rho0, cT + r.bT0, cY, cX, cw + r.binvW0, cr + r.brho0, lam);
#pragma unroll
    for (int j = 0; j < 4; ++j) th[j] = r.th[j];
}

template <typename S>
__global__ void __launch_bounds__(32)
    adjoint_step_kernel(StepParams<double> P, const S* __restrict__ g_in, const S* __restrict__ T_in,
                        const S* __restrict__ Y_in, const uint8_t* __restrict__ interior,
                        const long long* __restrict__ cells, const unsigned long long* __restrict__ codes, int ncells,
                        int list_blocks, int tiles_x, const double* __restrict__ lam_next, double* __restrict__ lam,
                        double* __restrict__ dtheta)
{
    const int t = (int)blockIdx.x - list_blocks;
    double th[4] = {0.0, 0.0, 0.0, 0.0};
    if (t < 0) {
        const int j = blockIdx.x * 32 + threadIdx.x;
        if (j < ncells) reverse_coded<S>(P, cells[j], codes[j], g_in, T_in, Y_in, lam_next, lam, th);
    } else {
        reverse_tile<S>(P, g_in, T_in, Y_in, interior, lam_next, lam, t % tiles_x, t / tiles_x, th);
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) th[k] += __shfl_down_sync(0xffffffffu, th[k], off);
        if (threadIdx.x == 0 && th[k] != 0.0) atomicAdd(&dtheta[k], th[k]);
    }
}

template <typename S>
cudaError_t launch_direct(const StepParams<double>& P, StateView st, const BoundaryLists& b, const double* lam_next,
                          double* lam, double* dtheta, cudaStream_t stream)
{
    constexpr size_t smem = 2 * tile_smem_bytes<double, SM_TX, SM_TY>();
    const int gx = (P.nx + SM_TX - 1) / SM_TX, gy = (P.ny + SM_TY - 1) / SM_TY, lb = (int)((b.all2.n + 31) / 32);
    adjoint_step_kernel<S><<<lb + gx * gy, 32, smem, stream>>>(P, (const S*)st.g, (const S*)st.T, (const S*)st.Y,
                                                               b.interior, b.all2.cells, b.all2.codes, (int)b.all2.n,
                                                               lb, gx, lam_next, lam, dtheta);
    return cudaGetLastError();
}

}  // namespace

bool adjoint_direct_applies(const StepParams<double>& P, const BoundaryLists& b)
{
    bool eq32 = false;
    for (int f = 0; f < 4; ++f) eq32 |= P.bc[f] == BC_OUTLET;
    return P.omega_hi == 1.0 && !P.curved && !eq32 && b.all2.nrest == 0;
}

cudaError_t launch_adjoint_step(const StepParams<double>& P, StateView st, bool fp32, const BoundaryLists& b,
                                const double* lam_next, double* lam, double* dtheta, cudaStream_t stream)
{
    if (fp32) return launch_direct<float>(P, st, b, lam_next, lam, dtheta, stream);
    return launch_direct<double>(P, st, b, lam_next, lam, dtheta, stream);
}

}  // namespace lbfd
