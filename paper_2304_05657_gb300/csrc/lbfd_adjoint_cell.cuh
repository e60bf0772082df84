// lbfd_adjoint_cell.cuh -- hand-derived local adjoints of the D2Q9 step in
// FP64: the WENO3 derivative's weights and the transpose of the collision
// with omega_hi = 1.  Plain arithmetic, for host and device: the CPU test
// (tests/test_adjoint_cell_host.py) compares them with central differences of
// the forward forms.
#pragma once
#include "lbfd_device.cuh"

namespace lbfd {

#ifdef __CUDA_ARCH__
#define LBFD_RCP(x) frcp(x)
#else
#define LBFD_RCP(x) (1.0 / (x))
#endif

// The convection derivative of conv_deriv (along the upwind direction, the
// line mirrored when neg; centred when near) and its partial derivatives w[j]
// with respect to the five line points.
__host__ __device__ __forceinline__ double conv_partials(const double* v, bool neg, double eps, bool near, double* w)
{
    const double a = neg ? v[4] : v[0], b = neg ? v[3] : v[1], c = v[2], d = neg ? v[1] : v[3];
    const double p = b - a, q = c - b, s = d - c;
    const double ep = eps + p * p, eq = eps + q * q, es = eps + s * s;
    const double hB = 0.5 * (eq * eq);
    const double i1 = LBFD_RCP(eq * eq + 0.5 * (es * es)), i0 = LBFD_RCP(eq * eq + 2.0 * (ep * ep));
    const double t1 = (s - q) * i1, t0 = (q - p) * i0, ww = t1 + t0, qe = q * eq;
    double r = q + hB * ww;
    double rp = -(hB * i0) * (1.0 + 8.0 * t0 * (p * ep));
    double rs = hB * i1 * (1.0 - 2.0 * t1 * (s * es));
    double rq = 1.0 + 2.0 * qe * ww + hB * ((i0 - i1) - 4.0 * qe * (t1 * i1 + t0 * i0));
    if (near) {
        r = 0.5 * (d - b);
        rp = 0.0;
        rq = rs = 0.5;
    }
    w[0] = neg ? 0.0 : -rp;
    w[1] = neg ? rs : rp - rq;
    w[2] = rq - rs;
    w[3] = neg ? rp - rq : rs;
    w[4] = neg ? -rp : 0.0;
    return r;
}

// The D2Q9 collision with omega_hi = 1 (collide_hi1: the same closed forms)
// and its transpose.  rs = 1 - omega_s, rb = omega_s - omega_b.
struct Collision2 {
    double m0, m1[2], m2[3];  // moments of the pulled populations (m2: xx, yy, xy)
    double rho, irho, u[2], gam[2], Lam;
};

// lg: adjoints of the nine populations g*; adds the adjoints of the inputs
// (which are arguments of their own here: u, gam, irho are not followed
// further) into b.  g: if not null, gets the populations themselves.
__host__ __device__ __forceinline__ void collide2_adjoint(const Collision2& s, double rs, double rb, const double* lg,
                                                          Collision2& b, double* g)
{
    // ---- forward
    const double ux = s.u[0], uy = s.u[1], gx = s.gam[0], gy = s.gam[1];
    const double h = 3.0 * s.irho, m0n = s.m0 * h, Ph = m0n + 0.5 * s.Lam, e = Ph - 1.0;
    const double px = ux * gx, py = uy * gy, sp = px + py, ux2 = ux * ux, uy2 = uy * uy, uxy = ux * uy;
    const double s0 = 0.5 * (sp + s.Lam);
    const double E2 = e * e, s1 = 3.0 + e - 3.0 * E2, s2 = E2 * (1.0 / 3.0), s3 = e * Ph * (1.0 / 9.0), e3 = e * (1.0 / 3.0);
    const double cross = (ux * gy + uy * gx) * (1.0 / 6.0);
    const double nxy = s.m2[2] * h - uxy + cross, iso = sp * (1.0 / 6.0) - m0n * (1.0 / 3.0);
    const double nx = s.m2[0] * h - ux2 + px * (1.0 / 3.0) + iso, ny = s.m2[1] * h - uy2 + py * (1.0 / 3.0) + iso;
    const double trb = (nx + ny) * (0.5 * rb);
    const double C20 = e * ux2 + Ph * (1.0 / 3.0) + rs * nx + trb, C02 = e * uy2 + Ph * (1.0 / 3.0) + rs * ny + trb;
    const double C11 = e * uxy + rs * nxy;
    const double q21 = Ph * ux2 + e3, q12 = Ph * uy2 + e3, C21 = -uy * q21, C12 = -ux * q12;
    const double C22 = ux2 * uy2 * s1 - (s2 * (ux2 + uy2) + s3) + C20 * C02 + 2.0 * C11 * C11;
    const double C00 = m0n + s0, k1 = 1.0 - C00, C10 = ux * k1, C01 = uy * k1;
    // central -> raw, along x then y
    const double R10 = C10 + ux * C00, R20 = C20 + ux * (C10 + R10);
    const double R11 = C11 + ux * C01, R21 = C21 + ux * (C11 + R11);
    const double R12 = C12 + ux * C02, R22 = C22 + ux * (C12 + R12);
    const double r01 = C01 + uy * C00, r02 = C02 + uy * (C01 + r01);
    const double r11 = R11 + uy * R10, r12 = R12 + uy * (R11 + r11);
    const double r21 = R21 + uy * R20, r22 = R22 + uy * (R21 + r21);
    // + half the raw moments of xi
    const double hx = px - 1.5 * sp * ux2, hy = py - 1.5 * sp * uy2;
    const double txy = 0.5 * gx * uy2 + ux * py, tyx = 0.5 * gy * ux2 + uy * px, q11 = cross - 0.5 * sp * uxy;
    const double x20 = R20 + (s0 + hx) * (1.0 / 3.0), x02 = r02 + (s0 + hy) * (1.0 / 3.0);
    const double x22 = r22 + (s0 + hx + hy) * (1.0 / 9.0), x12 = r12 + txy * (1.0 / 3.0), x21 = r21 + tyx * (1.0 / 3.0);
    const double x11 = r11 + q11, r0 = s.rho * (1.0 / 3.0);
    if (g) {
        double m[9] = {s.m0 + r0 * 2.0 * s0, 0.5 * s.m1[0],  0.5 * r0 * x20, 0.5 * s.m1[1],  0.25 * r0 * x11,
                       0.25 * r0 * x21,      0.5 * r0 * x02, 0.25 * r0 * x12, 0.25 * r0 * x22};
        for (int a = 1; a <= 3; a += 2)
            for (int j = 0; j < 9; ++j) {
                if ((j / a) % 3) continue;
                const double z = m[j], h1 = m[j + a], h2 = m[j + 2 * a];
                m[j] = h2 - h1;
                m[j + a] = z - 2.0 * h2;
                m[j + 2 * a] = h2 + h1;
            }
        for (int j = 0; j < 9; ++j) g[j] = m[j];
    }
    // ---- reverse: populations -> scaled raw moments (y, then x)
    double A[9];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double y0 = lg[a], y1 = lg[a + 3], y2 = lg[a + 6];
        A[a] = y1;
        A[a + 3] = y2 - y0;
        A[a + 6] = y0 - 2.0 * y1 + y2;
    }
#pragma unroll
    for (int q = 0; q < 9; q += 3) {
        const double y0 = A[q], y1 = A[q + 1], y2 = A[q + 2];
        A[q] = y1;
        A[q + 1] = y2 - y0;
        A[q + 2] = y0 - 2.0 * y1 + y2;
    }
    b.m0 += A[0];
    b.m1[0] += 0.5 * A[1];
    b.m1[1] += 0.5 * A[3];
    double bs0 = 2.0 * r0 * A[0];
    b.rho += (1.0 / 3.0) * (2.0 * s0 * A[0] + 0.5 * (A[2] * x20 + A[6] * x02) +
                            0.25 * (A[4] * x11 + A[5] * x21 + A[7] * x12 + A[8] * x22));
    const double a20 = 0.5 * r0 * A[2], a02 = 0.5 * r0 * A[6], a11 = 0.25 * r0 * A[4], a21 = 0.25 * r0 * A[5],
                 a12 = 0.25 * r0 * A[7], a22 = 0.25 * r0 * A[8];
    // xi
    bs0 += (a20 + a02) * (1.0 / 3.0) + a22 * (1.0 / 9.0);
    const double bhx = a20 * (1.0 / 3.0) + a22 * (1.0 / 9.0), bhy = a02 * (1.0 / 3.0) + a22 * (1.0 / 9.0);
    const double btxy = a12 * (1.0 / 3.0), btyx = a21 * (1.0 / 3.0);
    double bsp = -1.5 * (bhx * ux2 + bhy * uy2) - 0.5 * a11 * uxy, bcross = a11;
    double bux2 = -1.5 * sp * bhx + 0.5 * gy * btyx, buy2 = -1.5 * sp * bhy + 0.5 * gx * btxy, buxy = -0.5 * sp * a11;
    double bgx = 0.5 * uy2 * btxy, bgy = 0.5 * ux2 * btyx;
    double bpx = bhx + uy * btyx, bpy = bhy + ux * btxy, bux = py * btxy, buy = px * btyx;
    // raw -> central, y
    const double b01 = uy * a02;                    // adjoint of r01
    double bR00 = uy * b01, bR01 = uy * a02 + b01, bR02 = a02;
    buy += a02 * (C01 + r01) + b01 * C00;
    const double b11 = a11 + uy * a12;
    const double bR10 = uy * b11, bR11 = uy * a12 + b11, bR12 = a12;
    buy += a12 * (R11 + r11) + b11 * R10;
    const double b21 = a21 + uy * a22;
    const double bR20 = a20 + uy * b21, bR21 = uy * a22 + b21, bR22 = a22;
    buy += a22 * (R21 + r21) + b21 * R20;
    // x
    const double c10 = bR10 + ux * bR20;
    double bC20 = bR20, bC10 = ux * bR20 + c10, bC00 = bR00 + ux * c10;
    bux += bR20 * (C10 + R10) + c10 * C00;
    const double c11 = bR11 + ux * bR21;
    double bC11 = ux * bR21 + c11, bC01 = bR01 + ux * c11;
    bux += bR21 * (C11 + R11) + c11 * C01;
    const double c12 = bR12 + ux * bR22;
    const double bC12 = ux * bR22 + c12, bC21 = bR21, bC22 = bR22;
    double bC02 = bR02 + ux * c12;
    bux += bR22 * (C12 + R12) + c12 * C02;
    // orders 0 and 1
    bux += bC10 * k1;
    buy += bC01 * k1;
    const double bK0 = bC00 - (bC10 * ux + bC01 * uy);
    double bm0n = bK0;
    bs0 += bK0;
    // fourth order
    bC20 += bC22 * C02;
    bC02 += bC22 * C20;
    bC11 += 4.0 * bC22 * C11;
    bux2 += bC22 * (uy2 * s1 - s2);
    buy2 += bC22 * (ux2 * s1 - s2);
    const double bs1 = bC22 * ux2 * uy2, bs2 = -bC22 * (ux2 + uy2), bs3 = -bC22;
    // third
    buy -= bC21 * q21;
    bux -= bC12 * q12;
    const double v21 = -bC21 * uy, v12 = -bC12 * ux;
    double bPh = v21 * ux2 + v12 * uy2;
    bux2 += v21 * Ph;
    buy2 += v12 * Ph;
    const double be3 = v21 + v12;
    // second
    double be = bC11 * uxy + bC20 * ux2 + bC02 * uy2;
    buxy += bC11 * e;
    bux2 += bC20 * e;
    buy2 += bC02 * e;
    bPh += (bC20 + bC02) * (1.0 / 3.0);
    const double bt = (bC20 + bC02) * (0.5 * rb), bnxy = bC11 * rs, bnx = bC20 * rs + bt, bny = bC02 * rs + bt;
    b.m2[0] += bnx * h;
    b.m2[1] += bny * h;
    b.m2[2] += bnxy * h;
    double bh = bnx * s.m2[0] + bny * s.m2[1] + bnxy * s.m2[2];
    bux2 -= bnx;
    buy2 -= bny;
    buxy -= bnxy;
    bcross += bnxy;
    bpx += bnx * (1.0 / 3.0);
    bpy += bny * (1.0 / 3.0);
    bsp += (bnx + bny) * (1.0 / 6.0) + 0.5 * bs0;
    bm0n -= (bnx + bny) * (1.0 / 3.0);
    const double c6 = bcross * (1.0 / 6.0);
    bux += c6 * gy;
    bgx += c6 * uy;
    buy += c6 * gx;
    bgy += c6 * ux;
    bpx += bsp;
    bpy += bsp;
    bux += bpx * gx + 2.0 * ux * bux2 + uy * buxy;
    buy += bpy * gy + 2.0 * uy * buy2 + ux * buxy;
    bgx += bpx * ux;
    bgy += bpy * uy;
    be += bs1 * (1.0 - 6.0 * e) + bs2 * (2.0 / 3.0) * e + bs3 * Ph * (1.0 / 9.0) + be3 * (1.0 / 3.0);
    bPh += bs3 * e * (1.0 / 9.0) + be;
    bm0n += bPh;
    b.Lam += 0.5 * bs0 + 0.5 * bPh;
    b.m0 += bm0n * h;
    bh += bm0n * s.m0;
    b.irho += 3.0 * bh;
    b.u[0] += bux;
    b.u[1] += buy;
    b.gam[0] += bgx;
    b.gam[1] += bgy;
}

}  // namespace lbfd
