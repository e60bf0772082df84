// lbfd_device.cuh -- device-side building blocks of the fused coupled step:
// lattice constants, boundary classification, pull streaming with boundary
// rules, FD line gathering with ghost nodes, FD operators, and the cumulant
// collision.  Written for sm_103a; templated on the compute type R (double
// for the FP64 form, float for the mixed form, F2 for two cells in packed
// FP32, dual numbers for the tangent forms, Rev for the adjoint).
//
// Method: Hosseini & Thevenin, arXiv 2304.05657, Sec. II-III.
#pragma once
#include <cstdint>
#include <type_traits>

#include "lbfd_dual.cuh"
#include "lbfd_f2.cuh"
#include "lbfd_params.h"

namespace lbfd {

// Fast division and reciprocal, for divisors of normal magnitude.  FP32: the
// hardware reciprocal (about 1 ulp; ftz, so one instruction without the
// range checks that division by a subnormal would need).  FP64: the
// hardware's 20-bit seed x and one third-order Newton (Householder) step,
// x (1 + e + e^2) with e = 1 - b x, whose remaining error e^3 is below the
// rounding: within 1 ulp of 1/b (tests/test_gpu_reciprocal.py) for three
// FP64 instructions, where an IEEE division takes about ten (and the pipe
// issues one per 64 cycles and SM partition).  A zero, subnormal or infinite
// divisor gives NaN, where a division would give inf or 0.
__device__ __forceinline__ float frcp(float b)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b));
    return r;
}
__device__ __forceinline__ float fdiv(float a, float b) { return a * frcp(b); }
__device__ __forceinline__ double frcp(double b)
{
    double x;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(b));
    const double e = fma(-b, x, 1.0);
    return fma(x, fma(e, e, e), x);
}
__device__ __forceinline__ double fdiv(double a, double b) { return a * frcp(b); }
__device__ __forceinline__ F2 frcp(const F2& b) { return F2(frcp(b.v.x), frcp(b.v.y)); }
__device__ __forceinline__ F2 fdiv(const F2& a, const F2& b) { return F2(a * frcp(b)); }
// the other number types (reverse and forward mode)
template <typename R>
__device__ __forceinline__ R frcp(const R& b)
{
    return R(1) / b;
}
template <typename T, int N>
__device__ __forceinline__ Dual<T, N> frcp(const Dual<T, N>& b)
{
    Dual<T, N> r;
    r.v = frcp(b.v);
    Vec<T, N>::scale(r.d, -(r.v * r.v), b.d);
    return r;
}

// a parameter that does not depend on theta, as a constant for values of
// type R
template <typename R, typename PR>
__device__ __forceinline__ const_t<R> par(const PR& p)
{
    return const_t<R>(p);
}
template <typename R, typename T, int N>
__device__ __forceinline__ Cst<T> par(const Dual<T, N>& p)
{
    return Cst<T>(p.v);
}

enum { BC_PERIODIC = 0, BC_WALL_ADIABATIC = 1, BC_WALL_ISOTHERMAL = 2, BC_INLET = 3, BC_OUTLET = 4,
       BC_OUTLET_PRESSURE = 5 };
enum { PT_FLUID = 0, PT_SOLID = 16 };
// ghost modes of an FD line point
enum { G_DIRECT = 0, G_NEUMANN = 1, G_DIRICHLET_T = 2, G_INLET = 3, G_CURVED = 4 };

// ---------------------------------------------------------------------------
// lattice: D1Q3 tensor products, i = (cx+1) + 3(cy+1) + 9(cz+1)
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int cx_of(int i) { return i % 3 - 1; }
__host__ __device__ constexpr int cy_of(int i) { return (i / 3) % 3 - 1; }
__host__ __device__ constexpr int cz_of(int i) { return i / 9 - 1; }
template <typename R>
__host__ __device__ constexpr R w1(int c) { return c == 0 ? R(2) / R(3) : R(1) / R(6); }
template <int DIM, typename R>
__host__ __device__ constexpr R weight(int i)
{
    return DIM == 2 ? w1<R>(cx_of(i)) * w1<R>(cy_of(i))
                    : w1<R>(cx_of(i)) * w1<R>(cy_of(i)) * w1<R>(cz_of(i));
}
template <int DIM>
__host__ __device__ constexpr int ccomp(int i, int a)
{
    return a == 0 ? cx_of(i) : (a == 1 ? cy_of(i) : (DIM == 3 ? cz_of(i) : 0));
}
template <int DIM>
__host__ __device__ constexpr int opposite(int i) { return (DIM == 2 ? 8 : 26) - i; }

// ---------------------------------------------------------------------------
// geometry
// ---------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ int extent(const StepParams<R>& P, int a)
{
    return a == 0 ? P.nx : (a == 1 ? P.ny : P.nz);
}

// type and wall temperature of a face known only at run time, without
// indexing the parameter arrays (which would copy them to local memory)
template <typename R>
__device__ __forceinline__ int face_type(const StepParams<R>& P, int f)
{
    int t = P.bc[0];
#pragma unroll
    for (int j = 1; j < 6; ++j) t = f == j ? P.bc[j] : t;
    return t;
}
template <typename R>
__device__ __forceinline__ R face_T_wall(const StepParams<R>& P, int f)
{
    R t = P.T_wall[0];
#pragma unroll
    for (int j = 1; j < 6; ++j) t = f == j ? P.T_wall[j] : t;
    return t;
}

template <typename R>
__device__ __forceinline__ long long cell_of(const StepParams<R>& P, int x, int y, int z)
{
    return (long long)x + (long long)P.nx * ((long long)y + (long long)P.ny * z);
}

// Classify a point that differs from a fluid cell along one or more axes.
// Periodic axes wrap; a crossed non-periodic face returns its bc type.
// FACES == false: the caller guarantees that no non-periodic face is
// crossed (cells whose stencils stay inside the domain up to periodic wrap).
template <int DIM, typename R, bool FACES = true>
__device__ __forceinline__ int classify(const StepParams<R>& P, int q[3], const uint8_t* LBFD_RESTRICT solid,
                                        long long* idx, int* face)
{
    int wall = -1;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        int n = extent(P, a);
        int f = -1;
        if (q[a] < 0) f = 2 * a;
        else if (q[a] >= n) f = 2 * a + 1;
        if (f < 0) continue;
        if (!FACES || P.bc[f] == BC_PERIODIC) q[a] = ((q[a] % n) + n) % n;  // extents may be < 3
        else if (wall < 0) wall = f;
    }
    if (FACES && wall >= 0) {
        *face = wall;
        return P.bc[wall];
    }
    *idx = cell_of(P, q[0], q[1], DIM == 3 ? q[2] : 0);
    return solid[*idx] ? PT_SOLID : PT_FLUID;
}

// ---------------------------------------------------------------------------
// thermochemistry
// ---------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ R inv_molar_mass(const StepParams<R>& P, const R* Y)
{
    R s = Y[0] * par<R>(P.inv_Wk[0]);
#pragma unroll
    for (int k = 1; k < NSP; ++k) s += Y[k] * par<R>(P.inv_Wk[k]);
    return s;
}

// Y[k] for a species index known only at run time, without indexing a
// register array
template <typename R>
__device__ __forceinline__ R pick_species(const R* Y, int k)
{
    R r = Y[0];
#pragma unroll
    for (int j = 1; j < NSP; ++j) r = k == j ? Y[j] : r;
    return r;
}

// EOS at constant P_0 (Sec. II.A) with rho(T_in, Y_in) = 1
template <typename R>
__device__ __forceinline__ R eos(const StepParams<R>& P, R T, R invW)
{
    return par<R>(P.rho_c) * frcp(R(T * invW));
}
// The same with W = 1 / invW.  1 / rho and 1 / T of a point are products of its
// staged values too: T invW / rho_c, rho invW / rho_c.  W by a reciprocal of
// its own: where Y is uniform, W is then so exactly and the species stay
// uniform.  As T (1 / (T invW)), one reciprocal less, it has the rounding of T in it,
// which the species equations integrate: a uniform mixture with 20 K of noise in
// T spread by up to 19 ulp of Y over 4000 steps, in FP32 and in FP64, and a
// mixed tangent's dJ/dT_wall was 6.5e-5 off FP64 after 1000 steps.
template <typename R, typename PR>
__device__ __forceinline__ void eos_w(const StepParams<PR>& P, R T, R invW, R& rho, R& W)
{
    rho = par<R>(P.rho_c) * frcp(R(T * invW));
    W = frcp(invW);
}

// Single-step rate per unit mass of fuel, per step.  The mixed form
// evaluates it in FP64 where T > T_fp64.
template <typename R>
__device__ __forceinline__ R arrhenius(const StepParams<R>& P, R T, R yf, R yo)
{
    yf = yf > R(0) ? yf : R(0);
    yo = yo > R(0) ? yo : R(0);
    if constexpr (std::is_same<R, float>::value) {
        if (T > P.T_fp64) {
            const double q = P.A_lat_d * (double)yf * (double)yo * ::exp(-P.Ta_d / (double)T);
            return (float)q;
        }
        return P.A_lat * yf * yo * expf(-(P.Ta / T));
    } else if constexpr (std::is_same<R, double>::value) {
        return P.A_lat * yf * yo * ::exp(-(P.Ta / T));
    } else if constexpr (std::is_same<R, Tanf>::value) {
        if (T > P.T_fp64) {  // FP64 rate and derivatives, as the mixed form
            Tan A = widen(P.A_lat), Ta = widen(P.Ta);
            A.v = P.A_lat_d;
            A.d[0] = P.A_lat_d;  // d(A dt)/d(ln A)
            Ta.v = P.Ta_d;
            return narrow(A * widen(yf) * widen(yo) * exp(-(Ta / widen(T))));
        }
        return P.A_lat * yf * yo * exp(-(P.Ta / T));
    } else {
        return P.A_lat * yf * yo * exp(-(P.Ta / T));  // the Dual overload
    }
}

// ---------------------------------------------------------------------------
// FD operators (Sec. II.D), unit spacing, v[0..4] = phi_{i-2..i+2}; the
// 4th-order stencils are evaluated times 12 (their users fold 1/12 into
// coefficients)
// ---------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ R fd_D1(const R* v)  // 12 x the 4th-order central first derivative
{
    return R(v[0] - v[4]) + K<R>(8) * R(v[3] - v[1]);
}
template <typename R>
__device__ __forceinline__ R fd_D2(const R* v)  // 12 x the 4th-order central second derivative
{
    return R(K<R>(16) * R(v[1] + v[3]) - R(v[0] + v[4])) - K<R>(30) * v[2];
}

// a product rounded before it is added to anything
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
template <typename A, typename R>
__device__ __forceinline__ R mul_rn(const A& a, const R& b)
{
    return R(a * b);
}

// Upwind side of a velocity component (u < 0; u = 0 takes the u >= 0 side)
// and the velocity along it: the FD terms use mirrored lines and |u|, since
// u L(v) = |u| L(v mirrored) for u < 0.
template <typename R>
__device__ __forceinline__ bool upwind_neg(const R& u)
{
    return u < R(0);
}
template <typename R>
__device__ __forceinline__ R upwind_abs(const R& u, bool neg)
{
    return neg ? R(-u) : u;
}
template <typename R>
__device__ __forceinline__ R upwind_sel(bool neg, const R& a, const R& b)
{
    return neg ? a : b;
}

// WENO3 derivative along the upwind direction (Jiang-Shu r = 2), the line
// mirrored when neg.  With p, q, s the three differences from the far upwind
// point to the downwind one and A, B, C the squares of eps + p^2, eps + q^2,
// eps + s^2, the two face values' difference is
//   q + B/2 [ (s - q) / (B + C/2) + (q - p) / (B + 2A) ],
// the reconstruction with weights 1/3 : 2/3 over the smoothness, rearranged
// so that no face value is formed and every weight enters once (17 FP32
// instructions and two reciprocals, against 31 and two divisions for the
// two faces).  Plain FP64 takes one reciprocal (three instructions) for both
// terms, eight instructions where two take nine; there the product of two
// smoothness squares cannot leave the range, in FP32 it can.  CENTRED: `near`
// selects the centred 2nd-order derivative
// (any_near: false, uniformly over the warp, when no lane does).
template <bool CENTRED, typename R, typename N>
__device__ __forceinline__ R conv_deriv(const R* v, N neg, const_t<R> eps, bool near, bool any_near)
{
    const R a = upwind_sel(neg, v[4], v[0]), b = upwind_sel(neg, v[3], v[1]), d = upwind_sel(neg, v[1], v[3]);
    const R c = v[2];
    const R p = b - a, q = c - b, s = d - c;
    const R ep = eps + p * p, eq = eps + q * q, es = eps + s * s;
    const R A = ep * ep, B = eq * eq, C = es * es;
    const R d1 = B + K<R>(0.5) * C, d0 = B + K<R>(2) * A;
    const R hB = K<R>(0.5) * B;
    R r;
    if constexpr (std::is_same<R, double>::value) {
        r = q + hB * fdiv((s - q) * d0 + (q - p) * d1, d1 * d0);
    } else if constexpr (std::is_same<R, float>::value || std::is_same<R, F2>::value) {
        r = q + hB * R(R(s - q) * frcp(d1) + R(q - p) * frcp(d0));
    } else {
        // reverse mode: B scales the numerators first, so that the partials of
        // the divisions stay within 1 / eps^2 (of a reciprocal: 1 / eps^4, beyond
        // the FP32 tape's range from eps = 1e-10 down)
        r = q + fdiv(hB * R(s - q), d1) + fdiv(hB * R(q - p), d0);
    }
    if constexpr (CENTRED) {
        if (any_near) return near ? R(K<R>(0.5) * R(d - b)) : r;
    }
    return r;
}
// In forward mode the value and its partials with respect to p, q and s,
// chained to the derivatives of the four points: about 70 operations for
// four directions, where the rule per operation takes 190.
template <bool CENTRED, typename T, int ND>
__device__ __forceinline__ Dual<T, ND> conv_deriv(const Dual<T, ND>* v, bool neg, const Cst<T>& eps, bool near, bool)
{
    const T a = neg ? v[4].v : v[0].v, b = neg ? v[3].v : v[1].v, c = v[2].v, d = neg ? v[1].v : v[3].v;
    const T p = b - a, q = c - b, s = d - c;
    const T ep = eps.v + p * p, eq = eps.v + q * q, es = eps.v + s * s;
    const T B = eq * eq, hB = T(0.5) * B;
    const T i1 = frcp(B + T(0.5) * (es * es)), i0 = frcp(B + T(2) * (ep * ep));
    const T t1 = (s - q) * i1, t0 = (q - p) * i0, w = t1 + t0, qe = q * eq;
    T rp = -(hB * i0) * (T(1) + T(8) * t0 * (p * ep));
    T rs = hB * i1 * (T(1) - T(2) * t1 * (s * es));
    // (i ~ 1 / eps^2 and t ~ eps^-3/2 where the field is nearly uniform: their
    // product would leave the FP32 range from eps = 1e-11 down, hB i is of order 1)
    T rq = T(1) + T(2) * qe * w + hB * (i0 - i1) - T(4) * qe * ((hB * i1) * t1 + (hB * i0) * t0);
    Dual<T, ND> r;
    r.v = q + hB * w;
    if (CENTRED && near) {
        r.v = T(0.5) * (d - b);
        rp = T(0);
        rq = rs = T(0.5);
    }
    const T ca = -rp, cb = rp - rq, cc = rq - rs;
    if constexpr (sizeof(T) == 4) {  // packed, over the five points as they lie
        Vec<T, ND>::comb(r.d, neg ? T(0) : ca, v[0].d, neg ? rs : cb, v[1].d);
        Vec<T, ND>::axpy(r.d, cc, v[2].d);
        Vec<T, ND>::axpy(r.d, neg ? cb : rs, v[3].d);
        Vec<T, ND>::axpy(r.d, neg ? ca : T(0), v[4].d);
    } else {
#pragma unroll
        for (int k = 0; k < ND; ++k)
            r.d[k] = ca * (neg ? v[4].d[k] : v[0].d[k]) + cb * (neg ? v[3].d[k] : v[1].d[k]) + cc * v[2].d[k] +
                     rs * (neg ? v[1].d[k] : v[3].d[k]);
    }
    return r;
}

// Sums of the FD terms over the axes: T's convective and non-convective
// parts, the species' net rate (diffusion - convection) without its part
// along Y_k, the factor `along` of that part (rate of Y_k = rhs_Y[k] +
// Y_k * along), lamY = sum_k (diffusion of Y_k) / W_k (the FD part of
// Lambda's species sum, Eq. 6) and grad rho / rho.
template <typename R>
struct FDAccum {
    R conv_T, diff_T;
    R rhs_Y[NSP];
    R along, lamY;
    R gam[3];
    __device__ __forceinline__ void clear()
    {
        conv_T = diff_T = along = lamY = R(0);
#pragma unroll
        for (int k = 0; k < NSP; ++k) rhs_Y[k] = R(0);
#pragma unroll
        for (int a = 0; a < 3; ++a) gam[a] = R(0);
    }
};

// FD terms along one axis of a cell (Eq. 1, 2, 7, 25-27).  The callables
// fill the five line points of rho, T, 1/W, Y_k W (= X_k W_k) and Y_k.
// With m_k = D_k W_k (1/W) dX_k and M = sum m_k, the mixture-averaged flux
// divergence of Eq. 1-2 is
//   dk = f_k - M dY_k - Y_k F,  f_k = D_k W_k [ (1/W) d2X_k + b dX_k ],
//   b = d(1/W) + (1/W) drho/rho,  F = sum f_k
// (the density terms of the expanded form collected in b), its sum over
// dk / W_k closes with sum_k dY_k / W_k = d(1/W), and the terms along Y_k
// (-F and the convective correction u sum_j L_j of Eq. 26) are kept as one
// factor applied once per cell.  Each axis' share is rounded before it joins
// the sums, so that the two axes may be evaluated by different lanes with
// the same result.  37 FP32 instructions per species and axis
// instead of 58 (counted).  a12 = D_k / 12 (W_k cancels against the Y_k W lines).
template <bool CENTRED, typename R, typename PR, typename LRho, typename LT, typename LW, typename LX, typename LY>
__device__ __forceinline__ void fd_axis(const StepParams<PR>& P, R u_a, R invW0, R inv_rho0, bool near, bool any_near,
                                        LRho line_rho,
                                        LT line_T, LW line_invW, LX line_X, LY line_Y, R* gam_a, FDAccum<R>& acc)
{
    const auto twelfth = K<R>(1.0 / 12.0);
    const auto neg = upwind_neg(u_a);
    const R ua = upwind_abs(u_a, neg);
    R v[5];
    line_rho(v);
    const R gam = R(fd_D1(v)) * R(inv_rho0 * twelfth);
    *gam_a = gam;
    line_T(v);
    acc.conv_T += mul_rn(ua, conv_deriv<CENTRED>(v, neg, par<R>(P.epsT), near, any_near));
    acc.diff_T += mul_rn(par<R>(P.alpha12), R(fd_D2(v) + gam * fd_D1(v)));
    line_invW(v);
    const R dinvW = R(fd_D1(v)) * twelfth;
    const R b = dinvW + invW0 * gam;
    R f[NSP];
    R M = R(0), F = R(0), lam = R(0);
#pragma unroll
    for (int k = 0; k < NSP; ++k) {
        line_X(k, v);
        const R dX = fd_D1(v), d2X = fd_D2(v);
        const auto ak = par<R>(P.a12[k]);
        M += ak * dX;
        f[k] = ak * R(invW0 * d2X + b * dX);
        F += f[k];
        lam += par<R>(P.inv_Wk[k]) * f[k];
    }
    M = M * invW0;
    const R M12 = M * twelfth;
    acc.lamY += R(R(lam - M * dinvW) - invW0 * F);
    R sumL = R(0);
#pragma unroll
    for (int k = 0; k < NSP; ++k) {
        line_Y(k, v);
        const R L = conv_deriv<CENTRED>(v, neg, par<R>(P.epsY), near, any_near);
        sumL += L;
        acc.rhs_Y[k] += R(R(f[k] - M12 * fd_D1(v)) - ua * L);
    }
    acc.along += R(ua * sumL - F);
}

// ---------------------------------------------------------------------------
// central moments (Eq. 21) by axis-wise D1Q3 transforms, and cumulants
// (Eq. 22) with their exact inverse.  Moment index p + 3q + 9r.
// ---------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ void cm3_forward(R& f0, R& f1, R& f2, R u)
{
    R r0 = f0 + f1 + f2;
    R r1 = f2 - f0;
    R r2 = f2 + f0;
    f0 = r0;
    f1 = r1 - u * r0;
    f2 = r2 - R(2) * u * r1 + u * u * r0;
}
template <typename R>
__device__ __forceinline__ void cm3_inverse(R& m0, R& m1, R& m2, R u)
{
    R r0 = m0;
    R r1 = m1 + u * m0;
    R r2 = m2 + R(2) * u * m1 + u * u * m0;
    m0 = R(0.5) * (r2 - r1);
    m1 = r0 - r2;
    m2 = R(0.5) * (r2 + r1);
}

template <int DIM, typename R>
__device__ __forceinline__ void central_forward(R* f, const R* u)
{
    constexpr int NZ = DIM == 3 ? 3 : 1;
#pragma unroll
    for (int c = 0; c < NZ; ++c)
#pragma unroll
        for (int b = 0; b < 3; ++b) cm3_forward(f[3 * b + 9 * c], f[1 + 3 * b + 9 * c], f[2 + 3 * b + 9 * c], u[0]);
#pragma unroll
    for (int c = 0; c < NZ; ++c)
#pragma unroll
        for (int p = 0; p < 3; ++p) cm3_forward(f[p + 9 * c], f[p + 3 + 9 * c], f[p + 6 + 9 * c], u[1]);
    if (DIM == 3) {
#pragma unroll
        for (int j = 0; j < 9; ++j) cm3_forward(f[j], f[j + 9], f[j + 18], u[2]);
    }
}

template <int DIM, typename R>
__device__ __forceinline__ void central_inverse(R* m, const R* u)
{
    constexpr int NZ = DIM == 3 ? 3 : 1;
    if (DIM == 3) {
#pragma unroll
        for (int j = 0; j < 9; ++j) cm3_inverse(m[j], m[j + 9], m[j + 18], u[2]);
    }
#pragma unroll
    for (int c = 0; c < NZ; ++c)
#pragma unroll
        for (int p = 0; p < 3; ++p) cm3_inverse(m[p + 9 * c], m[p + 3 + 9 * c], m[p + 6 + 9 * c], u[1]);
#pragma unroll
    for (int c = 0; c < NZ; ++c)
#pragma unroll
        for (int b = 0; b < 3; ++b) cm3_inverse(m[3 * b + 9 * c], m[1 + 3 * b + 9 * c], m[2 + 3 * b + 9 * c], u[0]);
}

// central -> raw moments (binomial shift by u along each axis), and raw
// moments, each divided by 2 per axis with a non-zero exponent, ->
// populations
template <int DIM, typename R>
__device__ __forceinline__ void central_to_raw(R* m, const R* u)
{
    constexpr int Q = DIM == 3 ? 27 : 9;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const int s = a == 0 ? 1 : (a == 1 ? 3 : 9);
#pragma unroll
        for (int j = 0; j < Q; ++j) {
            if ((j / s) % 3) continue;
            const R r1 = m[j + s] + u[a] * m[j];
            m[j + 2 * s] = m[j + 2 * s] + u[a] * R(m[j + s] + r1);
            m[j + s] = r1;
        }
    }
}
template <int DIM, typename R>
__device__ __forceinline__ void raw_to_populations(R* m)
{
    constexpr int Q = DIM == 3 ? 27 : 9;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const int s = a == 0 ? 1 : (a == 1 ? 3 : 9);
#pragma unroll
        for (int j = 0; j < Q; ++j) {
            if ((j / s) % 3) continue;
            const R h1 = m[j + s], h2 = m[j + 2 * s];
            m[j + s] = m[j] - K<R>(2) * h2;
            m[j] = h2 - h1;
            m[j + 2 * s] = h2 + h1;
        }
    }
}

#define LBFD_M(p, q, r) ((p) + 3 * (q) + 9 * (r))

// In place: central moments -> cumulants (orders >= 4 change).
template <int DIM, typename R>
__device__ __forceinline__ void to_cumulants(R* m)
{
#define C_(p, q, r) m[LBFD_M(p, q, r)]
    if (DIM == 2) {
        C_(2, 2, 0) -= C_(2, 0, 0) * C_(0, 2, 0) + R(2) * C_(1, 1, 0) * C_(1, 1, 0);
        return;
    }
    // sixth order first: it reads the order-4 central moments
    R k222 = C_(2, 2, 2)
        - (C_(2, 0, 0) * C_(0, 2, 2) + C_(0, 2, 0) * C_(2, 0, 2) + C_(0, 0, 2) * C_(2, 2, 0))
        - R(4) * (C_(1, 1, 0) * C_(1, 1, 2) + C_(1, 0, 1) * C_(1, 2, 1) + C_(0, 1, 1) * C_(2, 1, 1))
        - R(4) * C_(1, 1, 1) * C_(1, 1, 1)
        - R(2) * (C_(2, 1, 0) * C_(0, 1, 2) + C_(2, 0, 1) * C_(0, 2, 1) + C_(1, 2, 0) * C_(1, 0, 2))
        + R(2) * C_(2, 0, 0) * C_(0, 2, 0) * C_(0, 0, 2)
        + R(4) * (C_(2, 0, 0) * C_(0, 1, 1) * C_(0, 1, 1) + C_(0, 2, 0) * C_(1, 0, 1) * C_(1, 0, 1)
                  + C_(0, 0, 2) * C_(1, 1, 0) * C_(1, 1, 0))
        + R(16) * C_(1, 1, 0) * C_(1, 0, 1) * C_(0, 1, 1);
    R k122 = C_(1, 2, 2) - C_(0, 0, 2) * C_(1, 2, 0) - C_(0, 2, 0) * C_(1, 0, 2)
        - R(4) * C_(0, 1, 1) * C_(1, 1, 1) - R(2) * (C_(1, 0, 1) * C_(0, 2, 1) + C_(1, 1, 0) * C_(0, 1, 2));
    R k212 = C_(2, 1, 2) - C_(0, 0, 2) * C_(2, 1, 0) - C_(2, 0, 0) * C_(0, 1, 2)
        - R(4) * C_(1, 0, 1) * C_(1, 1, 1) - R(2) * (C_(0, 1, 1) * C_(2, 0, 1) + C_(1, 1, 0) * C_(1, 0, 2));
    R k221 = C_(2, 2, 1) - C_(2, 0, 0) * C_(0, 2, 1) - C_(0, 2, 0) * C_(2, 0, 1)
        - R(4) * C_(1, 1, 0) * C_(1, 1, 1) - R(2) * (C_(1, 0, 1) * C_(1, 2, 0) + C_(0, 1, 1) * C_(2, 1, 0));
    C_(2, 2, 2) = k222;
    C_(1, 2, 2) = k122;
    C_(2, 1, 2) = k212;
    C_(2, 2, 1) = k221;
    C_(2, 2, 0) -= C_(2, 0, 0) * C_(0, 2, 0) + R(2) * C_(1, 1, 0) * C_(1, 1, 0);
    C_(2, 0, 2) -= C_(2, 0, 0) * C_(0, 0, 2) + R(2) * C_(1, 0, 1) * C_(1, 0, 1);
    C_(0, 2, 2) -= C_(0, 2, 0) * C_(0, 0, 2) + R(2) * C_(0, 1, 1) * C_(0, 1, 1);
    C_(2, 1, 1) -= C_(2, 0, 0) * C_(0, 1, 1) + R(2) * C_(1, 1, 0) * C_(1, 0, 1);
    C_(1, 2, 1) -= C_(0, 2, 0) * C_(1, 0, 1) + R(2) * C_(1, 1, 0) * C_(0, 1, 1);
    C_(1, 1, 2) -= C_(0, 0, 2) * C_(1, 1, 0) + R(2) * C_(1, 0, 1) * C_(0, 1, 1);
#undef C_
}

// In place: cumulants -> central moments (exact inverse of to_cumulants).
template <int DIM, typename R>
__device__ __forceinline__ void from_cumulants(R* m)
{
#define C_(p, q, r) m[LBFD_M(p, q, r)]
    if (DIM == 2) {
        C_(2, 2, 0) += C_(2, 0, 0) * C_(0, 2, 0) + R(2) * C_(1, 1, 0) * C_(1, 1, 0);
        return;
    }
    C_(2, 2, 0) += C_(2, 0, 0) * C_(0, 2, 0) + R(2) * C_(1, 1, 0) * C_(1, 1, 0);
    C_(2, 0, 2) += C_(2, 0, 0) * C_(0, 0, 2) + R(2) * C_(1, 0, 1) * C_(1, 0, 1);
    C_(0, 2, 2) += C_(0, 2, 0) * C_(0, 0, 2) + R(2) * C_(0, 1, 1) * C_(0, 1, 1);
    C_(2, 1, 1) += C_(2, 0, 0) * C_(0, 1, 1) + R(2) * C_(1, 1, 0) * C_(1, 0, 1);
    C_(1, 2, 1) += C_(0, 2, 0) * C_(1, 0, 1) + R(2) * C_(1, 1, 0) * C_(0, 1, 1);
    C_(1, 1, 2) += C_(0, 0, 2) * C_(1, 1, 0) + R(2) * C_(1, 0, 1) * C_(0, 1, 1);
    C_(1, 2, 2) += C_(0, 0, 2) * C_(1, 2, 0) + C_(0, 2, 0) * C_(1, 0, 2)
        + R(4) * C_(0, 1, 1) * C_(1, 1, 1) + R(2) * (C_(1, 0, 1) * C_(0, 2, 1) + C_(1, 1, 0) * C_(0, 1, 2));
    C_(2, 1, 2) += C_(0, 0, 2) * C_(2, 1, 0) + C_(2, 0, 0) * C_(0, 1, 2)
        + R(4) * C_(1, 0, 1) * C_(1, 1, 1) + R(2) * (C_(0, 1, 1) * C_(2, 0, 1) + C_(1, 1, 0) * C_(1, 0, 2));
    C_(2, 2, 1) += C_(2, 0, 0) * C_(0, 2, 1) + C_(0, 2, 0) * C_(2, 0, 1)
        + R(4) * C_(1, 1, 0) * C_(1, 1, 1) + R(2) * (C_(1, 0, 1) * C_(1, 2, 0) + C_(0, 1, 1) * C_(2, 1, 0));
    C_(2, 2, 2) += (C_(2, 0, 0) * C_(0, 2, 2) + C_(0, 2, 0) * C_(2, 0, 2) + C_(0, 0, 2) * C_(2, 2, 0))
        + R(4) * (C_(1, 1, 0) * C_(1, 1, 2) + C_(1, 0, 1) * C_(1, 2, 1) + C_(0, 1, 1) * C_(2, 1, 1))
        + R(4) * C_(1, 1, 1) * C_(1, 1, 1)
        + R(2) * (C_(2, 1, 0) * C_(0, 1, 2) + C_(2, 0, 1) * C_(0, 2, 1) + C_(1, 2, 0) * C_(1, 0, 2))
        - R(2) * C_(2, 0, 0) * C_(0, 2, 0) * C_(0, 0, 2)
        - R(4) * (C_(2, 0, 0) * C_(0, 1, 1) * C_(0, 1, 1) + C_(0, 2, 0) * C_(1, 0, 1) * C_(1, 0, 1)
                  + C_(0, 0, 2) * C_(1, 1, 0) * C_(1, 1, 0))
        - R(16) * C_(1, 1, 0) * C_(1, 0, 1) * C_(0, 1, 1);
#undef C_
}

__host__ __device__ constexpr int moment_order(int j) { return j % 3 + (j / 3) % 3 + j / 9; }

// Cumulants of orders >= 2 of g^eq / (rho cs^2) (Eq. 10, 12, 21, 22) in
// closed form.  On the product-weight lattices (D2Q9, D3Q27) the central
// moments of the discrete second-order equilibrium are polynomials in
// e = P_h / (rho cs^2) - 1 and the velocity; taking them through Eq. 22
// gives the expressions below (a, b, c = u_x^2, u_y^2, u_z^2), the same
// numbers as transforming the Q values, up to rounding.  Orders 0 and 1 are
// not relaxed and are left unset.
template <int DIM, typename R>
__device__ __forceinline__ void eq_cumulants(R* fe, R Ph, const R* u)
{
    const auto third = K<R>(1.0 / 3.0), ninth = K<R>(1.0 / 9.0);
    const R e = Ph - K<R>(1);
    const R ux = u[0], uy = u[1];
    const R a = ux * ux, b = uy * uy;
    const R Ph3 = Ph * third, e3 = e * third, E2 = e * e;
    const R s1 = R(3) + e - K<R>(3) * E2, s2 = E2 * third, s3 = e * R(Ph * ninth);
    // second order: kappa_aa = e u_a^2 + Ph/3, kappa_ab = e u_a u_b
    // third: kappa_aab = -u_b (Ph u_a^2 + e/3); fourth: c_aabb = u_a^2 u_b^2 s1 - s2 (u_a^2 + u_b^2) - s3
    fe[LBFD_M(2, 0, 0)] = e * a + Ph3;
    fe[LBFD_M(0, 2, 0)] = e * b + Ph3;
    fe[LBFD_M(1, 1, 0)] = e * R(ux * uy);
    fe[LBFD_M(2, 1, 0)] = -(uy * R(Ph * a + e3));
    fe[LBFD_M(1, 2, 0)] = -(ux * R(Ph * b + e3));
    fe[LBFD_M(2, 2, 0)] = R(a * b) * s1 - R(s2 * R(a + b) + s3);
    if constexpr (DIM == 3) {
        const R uz = u[2];
        const R c = uz * uz;
        fe[LBFD_M(0, 0, 2)] = e * c + Ph3;
        fe[LBFD_M(1, 0, 1)] = e * R(ux * uz);
        fe[LBFD_M(0, 1, 1)] = e * R(uy * uz);
        fe[LBFD_M(2, 0, 1)] = -(uz * R(Ph * a + e3));
        fe[LBFD_M(0, 2, 1)] = -(uz * R(Ph * b + e3));
        fe[LBFD_M(1, 0, 2)] = -(ux * R(Ph * c + e3));
        fe[LBFD_M(0, 1, 2)] = -(uy * R(Ph * c + e3));
        fe[LBFD_M(1, 1, 1)] = -(Ph * R(R(ux * uy) * uz));
        fe[LBFD_M(2, 0, 2)] = R(a * c) * s1 - R(s2 * R(a + c) + s3);
        fe[LBFD_M(0, 2, 2)] = R(b * c) * s1 - R(s2 * R(b + c) + s3);
        // fourth, c_aabc = u_b u_c (u_a^2 s1 - s2)
        fe[LBFD_M(2, 1, 1)] = R(uy * uz) * R(a * s1 - s2);
        fe[LBFD_M(1, 2, 1)] = R(ux * uz) * R(b * s1 - s2);
        fe[LBFD_M(1, 1, 2)] = R(ux * uy) * R(c * s1 - s2);
        // fifth, c_abbcc = u_a (u_b^2 u_c^2 t1 + (u_b^2 + u_c^2) t2 + t3)
        const R t1 = K<R>(-6) + K<R>(9) * e + K<R>(10) * E2;
        const R t2 = (e + K<R>(4) * E2) * third, t3 = (e + K<R>(2) * E2) * ninth;
        fe[LBFD_M(1, 2, 2)] = ux * R(R(b * c) * t1 + R(R(b + c) * t2 + t3));
        fe[LBFD_M(2, 1, 2)] = uy * R(R(a * c) * t1 + R(R(a + c) * t2 + t3));
        fe[LBFD_M(2, 2, 1)] = uz * R(R(a * b) * t1 + R(R(a + b) * t2 + t3));
        // sixth, in the elementary symmetric polynomials of a, b, c
        const R sg1 = a + b + c, sg2 = a * b + R(a * c + b * c), sg3 = R(a * b) * c;
        fe[LBFD_M(2, 2, 2)] = sg3 * R(e * R(K<R>(30) * E2 - K<R>(25) * e - K<R>(64))) +
            R(sg2 * R(e * R(K<R>(2) * E2 - R(K<R>(5) * e + K<R>(7)) * third)) +
              R(sg1 * R(E2 * R(K<R>(2) * e - K<R>(1)) * ninth) + R(e * R(K<R>(2) * e + K<R>(1))) * R(Ph * K<R>(1.0 / 27.0))));
    }
}

// ---------------------------------------------------------------------------
// Collision of one cell (Eq. 9, 10, 12-15, 19, 21-24): g (post-streaming)
// is replaced by g*.  Relaxation toward the cumulants of g^eq/(rho cs^2);
// orders 0-1 carried, second order split into trace (omega_b) and
// deviatoric/off-diagonal (omega_s), orders >= 3 at omega_hi.  gam = grad
// rho / rho, inv_rho = 1 / rho.
// ---------------------------------------------------------------------------
template <int DIM, typename R, typename PR>
__device__ __forceinline__ void collide(const StepParams<PR>& P, R* g, R rho, R inv_rho, const R* u, const R* gam,
                                        R Lam)
{
    using Sc = scalar_t<R>;
    constexpr int Q = DIM == 2 ? 9 : 27;
    const R cs2 = R(Sc(1) / Sc(3));
    R sum_g = R(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) sum_g += g[i];
    const R rcs2 = rho * cs2;
    const R inv_rcs2 = inv_rho * R(3);
    const R Ph = sum_g * inv_rcs2 + R(Sc(0.5)) * Lam;  // Eq. 13a over rho cs2
    const R uu = u[0] * u[0] + u[1] * u[1] + (DIM == 3 ? R(u[2] * u[2]) : R(0));
    R xi[Q], fe[Q];  // xi = Xi / (rho cs2)
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const R wi = R(weight<DIM, Sc>(i));
        R cu = R(0), cg = R(0);
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            const int c = ccomp<DIM>(i, a);
            cu += R(c) * u[a];
            cg += (R(c) - u[a]) * gam[a];
        }
        // f^eq / rho - w, Eq. 10
        const R fw = wi * (R(3) * cu + R(4.5) * cu * cu - R(1.5) * uu);
        xi[i] = fw * cg + wi * Lam;  // Eq. 9
        g[i] = g[i] * inv_rcs2 + R(0.5) * xi[i];  // Eq. 19
    }
    central_forward<DIM>(g, u);
    to_cumulants<DIM>(g);
    // the target: cumulants of g^eq / (rho cs2) = w (P_h/(rho cs2) - 1) + f^eq/rho (Eq. 12)
    eq_cumulants<DIM>(fe, Ph, u);
    // relaxation
    const R ws = R(P.omega_s), wb = R(P.omega_b), wh = R(P.omega_hi);
#pragma unroll
    for (int j = 0; j < Q; ++j) {
        const int o = moment_order(j);
        if (o >= 3) g[j] = fe[j] + (R(1) - wh) * (g[j] - fe[j]);
    }
    if (DIM == 2) {
        const int ixx = LBFD_M(2, 0, 0), iyy = LBFD_M(0, 2, 0), ixy = LBFD_M(1, 1, 0);
        const R tr = g[ixx] + g[iyy], tre = fe[ixx] + fe[iyy];
        const R dv = g[ixx] - g[iyy], dve = fe[ixx] - fe[iyy];
        const R trs = tre + (R(1) - wb) * (tr - tre);
        const R dvs = dve + (R(1) - ws) * (dv - dve);
        g[ixx] = R(0.5) * (trs + dvs);
        g[iyy] = R(0.5) * (trs - dvs);
        g[ixy] = fe[ixy] + (R(1) - ws) * (g[ixy] - fe[ixy]);
    } else {
        const int ixx = LBFD_M(2, 0, 0), iyy = LBFD_M(0, 2, 0), izz = LBFD_M(0, 0, 2);
        const R tr = g[ixx] + g[iyy] + g[izz], tre = fe[ixx] + fe[iyy] + fe[izz];
        const R d1 = g[ixx] - g[iyy], d1e = fe[ixx] - fe[iyy];
        const R d2 = g[ixx] - g[izz], d2e = fe[ixx] - fe[izz];
        const R trs = tre + (R(1) - wb) * (tr - tre);
        const R d1s = d1e + (R(1) - ws) * (d1 - d1e);
        const R d2s = d2e + (R(1) - ws) * (d2 - d2e);
        const R xx = (trs + d1s + d2s) * R(Sc(1) / Sc(3));
        g[ixx] = xx;
        g[iyy] = xx - d1s;
        g[izz] = xx - d2s;
        const int o1 = LBFD_M(1, 1, 0), o2 = LBFD_M(1, 0, 1), o3 = LBFD_M(0, 1, 1);
        g[o1] = fe[o1] + (R(1) - ws) * (g[o1] - fe[o1]);
        g[o2] = fe[o2] + (R(1) - ws) * (g[o2] - fe[o2]);
        g[o3] = fe[o3] + (R(1) - ws) * (g[o3] - fe[o3]);
    }
    from_cumulants<DIM>(g);
    central_inverse<DIM>(g, u);
#pragma unroll
    for (int i = 0; i < Q; ++i) g[i] = rcs2 * (g[i] + R(0.5) * xi[i]);  // Eq. 14
}

// ---------------------------------------------------------------------------
// Collision with omega_hi = 1 (the usual setting; the caller checks), from
// the raw moments of orders 0-2 of the pulled populations alone: the
// relaxation sets every cumulant of order >= 3 to its equilibrium, so the
// populations collapse to 6 (D2Q9) or 10 (D3Q27) numbers as soon as they
// are pulled.  The source Xi enters through its moments, which are closed
// forms on the product-weight lattices (below), so no population of Xi or
// of the equilibrium is formed.  D3Q27: about 600 instructions instead of
// 950 (counted), and 17 fewer live values through the FD terms: the FP32
// 3-D tile kernel needs 128 registers instead of 168.  With the FD terms
// above: 101x53x47 FP64 packing 2 890 -> 1 820 us per step, 1.75 M cells of
// 2-D channels in FP32 95 -> 77 us per step, and the populations' error
// against 64-bit arithmetic falls to a quarter (no equilibrium is
// subtracted from the populations).
// ---------------------------------------------------------------------------
template <int DIM, typename R>
struct LowMoments {
    R m0;                    // sum g_i
    R m1[3];                 // sum c_a g_i
    R m2[DIM == 2 ? 3 : 6];  // sum c_a c_b g_i: xx, yy, xy or xx, yy, zz, xy, xz, yz
};

// from the populations, axis by axis: of each x line the sum, the first and
// the second moment; then of each of these along y (and z) the moments up
// to the order that is left
template <int DIM, typename R>
__device__ __forceinline__ void low_moments(const R* g, LowMoments<DIM, R>& m)
{
    constexpr int NZ = DIM == 3 ? 3 : 1;
    R s00[NZ], s10[NZ], s20[NZ], s01[NZ], s02[NZ], s11[NZ];  // x order, y order, per z layer
#pragma unroll
    for (int c = 0; c < NZ; ++c) {
        R s[3], d[3], e[3];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const R f0 = g[3 * b + 9 * c], f1 = g[1 + 3 * b + 9 * c], f2 = g[2 + 3 * b + 9 * c];
            e[b] = f2 + f0;
            d[b] = f2 - f0;
            s[b] = e[b] + f1;
        }
        const R t = s[2] + s[0];
        s00[c] = t + s[1];
        s01[c] = s[2] - s[0];
        s02[c] = t;
        s10[c] = d[0] + d[1] + d[2];
        s11[c] = d[2] - d[0];
        s20[c] = e[0] + e[1] + e[2];
    }
    if constexpr (DIM == 2) {
        m.m0 = s00[0];
        m.m1[0] = s10[0];
        m.m1[1] = s01[0];
        m.m1[2] = R(0);
        m.m2[0] = s20[0];
        m.m2[1] = s02[0];
        m.m2[2] = s11[0];
    } else {
        const R t = s00[2] + s00[0];
        m.m0 = t + s00[1];
        m.m1[0] = s10[0] + s10[1] + s10[2];
        m.m1[1] = s01[0] + s01[1] + s01[2];
        m.m1[2] = s00[2] - s00[0];
        m.m2[0] = s20[0] + s20[1] + s20[2];
        m.m2[1] = s02[0] + s02[1] + s02[2];
        m.m2[2] = t;
        m.m2[3] = s11[0] + s11[1] + s11[2];
        m.m2[4] = s10[2] - s10[0];
        m.m2[5] = s01[2] - s01[0];
    }
}

// Moments of xi = Xi / (rho cs^2) = (f^eq/rho - w) (c - u).gam + w Lam, with
// p_a = u_a gam_a and S the set of axes of exponent 2 (each a factor 1/3):
//   no exponent 1:    sum p + Lam + sum_S (2 p_a - 3 (sum p) u_a^2)
//   exponent 1 at a:  sum_{b in S} (gam_a u_b^2 + 2 u_a p_b)
//   at a and b:       (u_a gam_b + u_b gam_a) / 3 - (sum p) u_a u_b
//   at x, y and z:    (u_x u_y gam_z + u_x u_z gam_y + u_y u_z gam_x) / 3
// (raw moments; the discrete w has <c^2> = <c^4> = 1/3 per axis).  The
// non-equilibrium part of the second central moment of f' = (g + Xi/2) /
// (rho cs^2) then is
//   n_ab = m2_ab / (rho cs^2) - u_a u_b + (u_a gam_b + u_b gam_a) / 6
//          + delta_ab ((sum p) / 6 - m0 / (3 rho cs^2)),
// and the first raw moment of f'* is u.
template <int DIM, typename R, typename PR>
__device__ __forceinline__ void collide_hi1(const StepParams<PR>& P, const LowMoments<DIM, R>& lm, R rho, R inv_rho,
                                            const R* u, const R* gam, R Lam, R* g)
{
    constexpr int Q = DIM == 2 ? 9 : 27;
    const auto third = K<R>(1.0 / 3.0), sixth = K<R>(1.0 / 6.0), half = K<R>(0.5);
    const R inv_rcs2 = inv_rho * K<R>(3);
    const R m0 = lm.m0 * inv_rcs2;
    const R Ph = m0 + half * Lam;
    R p[DIM], uu[DIM];
    R sp = R(0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        p[a] = u[a] * gam[a];
        uu[a] = u[a] * u[a];
        sp += p[a];
    }
    const R s0 = half * R(sp + Lam);  // half the zeroth moment of xi
    // g: first the target's cumulants, then the relaxed ones
    eq_cumulants<DIM>(g, Ph, u);
    const auto rs = par<R>(P.one_minus_omega_s), rb = par<R>(P.omega_s_minus_b);
    constexpr int NO = DIM == 2 ? 1 : 3;             // off-diagonal pairs xy, xz, yz
    constexpr int PA[3] = {0, 0, 1}, PB[3] = {1, 2, 2};
    R cross[NO];  // (u_a gam_b + u_b gam_a) / 6
#pragma unroll
    for (int j = 0; j < NO; ++j) {
        const int a = PA[j], b = PB[j], at = (a == 0 ? 1 : 3) + (b == 1 ? 3 : 9);
        cross[j] = R(u[a] * gam[b] + u[b] * gam[a]) * sixth;
        const R n = lm.m2[DIM + j] * inv_rcs2 - u[a] * u[b] + cross[j];
        g[at] += rs * n;
    }
    {
        R n[DIM], tr = R(0);
        const R iso = sixth * sp - third * m0;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            n[a] = R(lm.m2[a] * inv_rcs2 - uu[a]) + R(third * p[a] + iso);
            tr += n[a];
        }
        const R trb = R(tr * rb) * K<R>(1.0 / DIM);
#pragma unroll
        for (int a = 0; a < DIM; ++a) g[a == 0 ? 2 : (a == 1 ? 6 : 18)] += rs * n[a] + trb;
    }
    from_cumulants<DIM>(g);
    // orders 0 and 1 are carried: m0 + s0, and u (1 - that) about u
    g[0] = m0 + s0;
    {
        const R k1 = K<R>(1) - g[0];
        g[1] = u[0] * k1;
        g[3] = u[1] * k1;
        if constexpr (DIM == 3) g[9] = u[2] * k1;
    }
    central_to_raw<DIM>(g, u);
    // + half the moments of xi
    {
        R h[DIM];  // p_a - 3/2 (sum p) u_a^2
        const R sp15 = K<R>(1.5) * sp;
#pragma unroll
        for (int a = 0; a < DIM; ++a) h[a] = p[a] - sp15 * uu[a];
        const R hsp = half * sp;
        const auto ninth = K<R>(1.0 / 9.0);
        R tab[DIM][DIM];  // gam_a u_b^2 / 2 + u_a p_b
#pragma unroll
        for (int a = 0; a < DIM; ++a)
#pragma unroll
            for (int b = 0; b < DIM; ++b)
                if (a != b) tab[a][b] = R(half * gam[a]) * uu[b] + u[a] * p[b];
        const R ex = s0 + h[0], ey = s0 + h[1], exy = ex + h[1];
        const R qxy = cross[0] - hsp * R(u[0] * u[1]);
        g[LBFD_M(2, 0, 0)] += third * ex;
        g[LBFD_M(0, 2, 0)] += third * ey;
        g[LBFD_M(2, 2, 0)] += ninth * exy;
        g[LBFD_M(1, 2, 0)] += third * tab[0][1];
        g[LBFD_M(2, 1, 0)] += third * tab[1][0];
        g[LBFD_M(1, 1, 0)] += qxy;
        if constexpr (DIM == 3) {
            const R ez = s0 + h[2];
            const R qxz = cross[1] - hsp * R(u[0] * u[2]), qyz = cross[2] - hsp * R(u[1] * u[2]);
            g[LBFD_M(0, 0, 2)] += third * ez;
            g[LBFD_M(2, 0, 2)] += ninth * R(ex + h[2]);
            g[LBFD_M(0, 2, 2)] += ninth * R(ey + h[2]);
            g[LBFD_M(2, 2, 2)] += K<R>(1.0 / 27.0) * R(exy + h[2]);
            g[LBFD_M(1, 0, 2)] += third * tab[0][2];
            g[LBFD_M(2, 0, 1)] += third * tab[2][0];
            g[LBFD_M(0, 1, 2)] += third * tab[1][2];
            g[LBFD_M(0, 2, 1)] += third * tab[2][1];
            g[LBFD_M(1, 2, 2)] += ninth * R(tab[0][1] + tab[0][2]);
            g[LBFD_M(2, 1, 2)] += ninth * R(tab[1][0] + tab[1][2]);
            g[LBFD_M(2, 2, 1)] += ninth * R(tab[2][0] + tab[2][1]);
            g[LBFD_M(1, 0, 1)] += qxz;
            g[LBFD_M(0, 1, 1)] += qyz;
            g[LBFD_M(1, 1, 2)] += third * qxy;
            g[LBFD_M(1, 2, 1)] += third * qxz;
            g[LBFD_M(2, 1, 1)] += third * qyz;
            g[LBFD_M(1, 1, 1)] += sixth * R(R(u[0] * u[1]) * gam[2] + u[2] * R(u[0] * gam[1] + u[1] * gam[0]));
        }
    }
    // times rho cs^2, to populations (Eq. 14).  Orders 0 and 1 are taken from
    // the pulled moments, not through the product of rho and 1 / rho, whose
    // rounding would act on mass and momentum with the same sign every step.
    const R r0 = rho * third, r1 = half * r0, r2 = half * r1, r3 = half * r2;
#pragma unroll
    for (int j = 0; j < Q; ++j) {
        const int n = (j % 3 != 0) + ((j / 3) % 3 != 0) + (j / 9 != 0);
        if (moment_order(j) >= 2) g[j] = (n == 1 ? r1 : (n == 2 ? r2 : r3)) * g[j];
    }
    g[0] = lm.m0 + r0 * R(s0 + s0);
    g[1] = half * lm.m1[0];
    g[3] = half * lm.m1[1];
    if constexpr (DIM == 3) g[9] = half * lm.m1[2];
    raw_to_populations<DIM>(g);
}

}  // namespace lbfd
