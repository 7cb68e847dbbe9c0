// step64.cuh -- FP64 arithmetic of one cell for the tile kernel (step_tile.cuh).
//
// GB300 issues an FP64 warp instruction once per 64 cycles and sub-partition (measured, one warp or
// four), so an FP64 step costs its number of FP64 operations and little else.  The algebra is that
// of pp_collide_v / fe_collide_v / fe_mu (lbm_kernels.cuh) and fe_collide_iwb_v (step_iwb_pair.cuh) with the
// population and stencil sums formed once as pair sums and differences, rho u taken as j + F/2, the
// rest population eliminated from the non-equilibrium parts (rho = f_0 + sum of the others), and
// every constant factor folded on the host (StepParams::d): per cell 141 operations for the
// pseudopotential (164 with the width-control tensor), 155 for the free energy, against about 260
// and 300 before.
#pragma once
#include <cuda_runtime.h>

#include "lbm_kernels.cuh"

namespace lbmk {

__device__ __forceinline__ double fmav(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double abs_v(double a) { return fabs(a); }
__device__ __forceinline__ double sum9_v(const double v[9]) { return sum9(v); }

// 1/x: the hardware's approximation (relative error e < 2^-20) and one step of the third-order iteration
// r (1 + e + e^2), e = 1 - x r (Chebyshev's, the geometric series cut after two terms), for a normal x with a
// normal reciprocal: 2^-60 before the last rounding, so correctly rounded but for 3 in 10,000 arguments, and
// these to an ulp (tests/test_gpu_math.py).
__device__ __forceinline__ double rcp_d(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// sqrt(x) from the hardware's 1/sqrt(x) by one coupled step (Goldschmidt 1964) and Markstein's (1990) correction
// by the residual x - g^2; correctly rounded for a normal x.  0 and subnormal numbers give 0, x < 0 NaN.
__device__ __forceinline__ double sqrt_d(double x) {
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    if ((unsigned)__double2hiint(x) < 0x00100000u) r = 0.0;  // below the normal numbers r is infinite
    double g = x * r, h = 0.5 * r;
    const double e = fma(-g, h, 0.5);
    g = fma(g, e, g);
    h = fma(h, e, h);
    return fma(fma(-g, g, x), h, g);
}

// Eq. (11): psi = sqrt(2 (rho/3 - p)), p of Eq. (28)
__device__ __forceinline__ double tile_psi(double rho, const StepParams<double>& P) {
    const double u = fma(-P.b4, rho, 1.0), e = P.b4 * rho;
    const double num = fma(e, fma(e, u, 1.0), 1.0);
    const double r = rcp_d(u);
    return sqrt_d(rho * fma(P.m2RT, num * (r * r * r), fma(P.a2, rho, 2.0 / 3.0)));
}

// ln x by a table (Tang 1990) of 32 intervals of the significand m, one per lane: c close to 1/m with 20 bits,
// chosen (Gal 1986) so that T = -ln c is a multiple of 2^-48 to 6e-18.  With r = m c - 1, |r| < 1/64,
//   ln x = k ln2 + T + ln(1 + r),
// ln2 = hi + lo with k hi + T exact, and ln(1 + r) - r interpolated in degree 7 to 1.3e-17.  13 FP64 operations
// and shuffles where log() takes about 30; its largest and rms error over 60,000 arguments from 1e-4 to 4,
// in the sum below, are log()'s (against 200-bit arithmetic).  A 256 x 128 step of
// the free-energy model: 20.4 us with log(), 18.2 with this.
static __device__ const int kLogC[32] = {
    0x3fef8299, 0x3fee9135, 0x3fedaf4b, 0x3fecd5a6, 0x3fec0bbf, 0x3feb4c41, 0x3fea99ca, 0x3fe9ed41, 0x3fe949ca, 0x3fe8abb8,
    0x3fe817d6, 0x3fe78afa, 0x3fe702c2, 0x3fe681fe, 0x3fe60468, 0x3fe58ee7, 0x3fe51eea, 0x3fe4b13e, 0x3fe44723, 0x3fe3e009,
    0x3fe3819d, 0x3fe324fb, 0x3fe2c9dd, 0x3fe2721d, 0x3fe21d17, 0x3fe1d0d4, 0x3fe180e8, 0x3fe1379b, 0x3fe0ecb9, 0x3fe0a5cd,
    0x3fe060ee, 0x3fe020b9};
static __device__ const double kLogT[32] = {
    0x1.f97d019432000p-7, 0x1.774213635e600p-5, 0x1.339f0d5536900p-4, 0x1.aaa4d1740b500p-4, 0x1.0e1e7792c6380p-3,
    0x1.457bb2c541a00p-3, 0x1.7a76cf2f49380p-3, 0x1.af0586a57fc80p-3, 0x1.e2178ed0bc400p-3, 0x1.0a5bfb0050640p-2,
    0x1.229f18cc04780p-2, 0x1.3a474ac3356c0p-2, 0x1.51b01f765abc0p-2, 0x1.6851dd426d8c0p-2, 0x1.7ee2a0febb3c0p-2,
    0x1.94756543ee8c0p-2, 0x1.a97378bc13d00p-2, 0x1.be6f5f35ea4c0p-2, 0x1.d3278068e2ec0p-2, 0x1.e7b25c8b8c480p-2,
    0x1.fae0d6ad1a880p-2, 0x1.0706ac5755c40p-1, 0x1.10a273a56eae0p-1, 0x1.1a0fc79cb26e0p-1, 0x1.235d491d4b2e0p-1,
    0x1.2bdad27324000p-1, 0x1.34e807e158ac0p-1, 0x1.3d59e646fd9c0p-1, 0x1.461fdfee846a0p-1, 0x1.4e9321d064ba0p-1,
    0x1.56ea91a876f20p-1, 0x1.5ed1390a15a40p-1};
struct LogTable {
    int c;
    double T;
    __device__ __forceinline__ void load() {
        c = __ldg(kLogC + (threadIdx.x & 31));
        T = __ldg(kLogT + (threadIdx.x & 31));
    }
};
// called by all lanes of a warp
__device__ __forceinline__ double log_d(double x, const LogTable& tab) {
    const int hi = __double2hiint(x), j = (hi >> 15) & 31;
    const double c = __hiloint2double(__shfl_sync(0xffffffffu, tab.c, j), 0), T = __shfl_sync(0xffffffffu, tab.T, j);
    if ((unsigned)(hi - 0x00100000) >= 0x7fe00000u) return log(x);  // not a positive normal number
    const double m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(x));
    const double k = __hiloint2double(0x43300000, hi >> 20) - (4503599627370496.0 + 1023.0);
    const double r = fma(m, c, -1.0);
    double p = 0x1.24a72f7efdbe5p-3;
    p = fma(p, r, -0x1.556cd8738489ap-3);
    p = fma(p, r, 0x1.9999991ec4c98p-3);
    p = fma(p, r, -0x1.ffffff75d0cecp-3);
    p = fma(p, r, 0x1.55555555558adp-2);
    p = fma(p, r, -0x1.00000000001e1p-1);
    double q = fma(p, r * r, r);
    q = fma(k, 0x1.e6af278ece601p-50, q);
    return fma(k, 0x1.62e42fefa39e0p-1, T) + q;
}

// Eq. (29) up to a constant, with the Eq. (24) Laplacian from the sums of the neighbours
__device__ __forceinline__ double tile_mu(double rho, const double n[9], const StepParams<double>& P,
                                          const LogTable& tab) {
    const double sax = (n[1] + n[3]) + (n[2] + n[4]), sdg = (n[5] + n[7]) + (n[6] + n[8]);
    const double u = fma(-P.b4, rho, 1.0);
    const double r = rcp_d(u);
    const double s = fma(u + 2.0, (r * r) * r, log_d(rho, tab));  // (3 - e) / (1 - e)^3 + ln rho
    return fma(P.k23, sax, fma(P.k16, sdg, fma(P.kc, rho, P.RT * s)));
}

// Pair sums and differences of the populations, and the moments both models share.
struct Pairs {
    double a13, a24, a57, a68, d13, d24, t, s, jx, jy, sax, sdg, pxx, pxy;
};
__device__ __forceinline__ Pairs pairs_of(const double v[9]) {
    Pairs p;
    p.a13 = v[1] + v[3];
    p.a24 = v[2] + v[4];
    p.a57 = v[5] + v[7];
    p.a68 = v[6] + v[8];
    p.d13 = v[1] - v[3];
    p.d24 = v[2] - v[4];
    const double d57 = v[5] - v[7], d86 = v[8] - v[6];
    p.t = d57 + d86;  // f5 - f6 - f7 + f8
    p.s = d57 - d86;  // f5 + f6 - f7 - f8
    p.jx = p.d13 + p.t;
    p.jy = p.d24 + p.s;
    p.sax = p.a13 + p.a24;
    p.sdg = p.a57 + p.a68;
    p.pxx = p.a13 - p.a24;
    p.pxy = p.a57 - p.a68;
    return p;
}

// 12 times the Eq. (24) gradient (equally the force stencil of Eq. 10)
__device__ __forceinline__ void grad12(const double n[9], double& gx, double& gy) {
    const double d57 = n[5] - n[7], d86 = n[8] - n[6];
    gx = fma(4.0, n[1] - n[3], d57 + d86);
    gy = fma(4.0, n[2] - n[4], d57 - d86);
}

// A cell's collision by two warps (where a tile has fewer rows than the SM sub-partitions): role 0 takes the
// energy moments and updates f_0 .. f_4, role 1 the fluxes and stresses and f_5 .. f_8; both form the force
// and the velocity.  x: the pair's exchange in shared memory, 32 per value and the lane's own; bar: its
// barrier.  The operations on each number are those of one warp alone (role -1), so the bits are too.
struct Exchange {
    int bar;
    double* x;
    __device__ __forceinline__ void meet() const { asm volatile("bar.sync %0, 64;" ::"r"(bar) : "memory"); }
};

// Populations from the moment increments; P4 = d pxx / 4, Z = d pxy / 4 (M^-1 of Eq. S49).
__device__ __forceinline__ void apply_pairs(double v[9], double de, double dz, double Fx, double dqx, double Fy,
                                            double dqy, double P4, double Z) {
    const double A = fma(de, -1.0 / 36.0, dz * (-1.0 / 18.0)), B = fma(de, 1.0 / 18.0, dz * (1.0 / 36.0));
    const double X1 = Fx - dqx, Y1 = Fy - dqy;  // times 6
    const double X2 = fma(dqx, 1.0 / 12.0, Fx * (1.0 / 6.0)), Y2 = fma(dqy, 1.0 / 12.0, Fy * (1.0 / 6.0));
    const double Ap = A + P4, Am = A - P4, Bp = B + Z, Bm = B - Z, Sp = X2 + Y2, Sm = X2 - Y2;
    v[0] = fma(dz - de, 1.0 / 9.0, v[0]);
    v[1] += fma(X1, 1.0 / 6.0, Ap);
    v[3] += fma(X1, -1.0 / 6.0, Ap);
    v[2] += fma(Y1, 1.0 / 6.0, Am);
    v[4] += fma(Y1, -1.0 / 6.0, Am);
    v[5] += Bp + Sp;
    v[7] += Bp - Sp;
    v[6] += Bm - Sm;
    v[8] += Bm + Sm;
}

__device__ __forceinline__ void apply_energy(double v[9], double de, double dz, const Exchange& E) {
    const double A = fma(de, -1.0 / 36.0, dz * (-1.0 / 18.0)), B = fma(de, 1.0 / 18.0, dz * (1.0 / 36.0));
    E.x[0] = B;
    v[0] = fma(dz - de, 1.0 / 9.0, v[0]);
    E.meet();
    const double P4 = E.x[32], X1 = E.x[64], Y1 = E.x[96];
    const double Ap = A + P4, Am = A - P4;
    v[1] += fma(X1, 1.0 / 6.0, Ap);
    v[3] += fma(X1, -1.0 / 6.0, Ap);
    v[2] += fma(Y1, 1.0 / 6.0, Am);
    v[4] += fma(Y1, -1.0 / 6.0, Am);
}
__device__ __forceinline__ void apply_flux(double v[9], double Fx, double dqx, double Fy, double dqy, double P4,
                                           double Z, const Exchange& E) {
    E.x[32] = P4;
    E.x[64] = Fx - dqx;
    E.x[96] = Fy - dqy;
    const double X2 = fma(dqx, 1.0 / 12.0, Fx * (1.0 / 6.0)), Y2 = fma(dqy, 1.0 / 12.0, Fy * (1.0 / 6.0));
    const double Sp = X2 + Y2, Sm = X2 - Y2;
    E.meet();
    const double B = E.x[0], Bp = B + Z, Bm = B - Z;
    v[5] += Bp + Sp;
    v[7] += Bp - Sp;
    v[6] += Bm - Sm;
    v[8] += Bm + Sm;
}

template <int ROLE>
__device__ __forceinline__ void apply_role(double v[9], double de, double dz, double Fx, double dqx, double Fy,
                                           double dqy, double P4, double Z, const Exchange& E) {
    if (ROLE < 0)
        apply_pairs(v, de, dz, Fx, dqx, Fy, dqy, P4, Z);
    else if (ROLE == 0)
        apply_energy(v, de, dz, E);
    else
        apply_flux(v, Fx, dqx, Fy, dqy, P4, Z, E);
}

// Pseudopotential collision (Eqs. 1, 4, 6, 10, 13, 30-32); pn: psi at the cell and at x + c_i.
template <int ROLE>
__device__ __forceinline__ void tile_collide_pp(double v[9], double rho, const double pn[9], double fx, double fy,
                                                unsigned&, const StepParams<double>& P, const Exchange& E) {
    const double pc = pn[0];
    const Pairs p = pairs_of(v);
    double Sx, Sy;
    grad12(pn, Sx, Sy);
    Sx *= 1.0 / 12.0;
    Sy *= 1.0 / 12.0;
    const double Fx = fma(pc, Sx, fx), Fy = fma(pc, Sy, fy);
    double Ls = P.li * fma(Sx, Sx, Sy * Sy), dQ = 0.0, Qxy = 0.0;
    if (P.kA != 0.0 || P.kB != 0.0) {  // Q vanishes identically for kappa_P = 1, kappa_Li = 0
        const double a13 = pn[1] + pn[3], a24 = pn[2] + pn[4], a57 = pn[5] + pn[7], a68 = pn[6] + pn[8];
        const double dd = fma(-4.0, pc, a57 + a68) * (1.0 / 12.0);
        const double sxx = fma(fma(-2.0, pc, a13), 1.0 / 3.0, dd), syy = fma(fma(-2.0, pc, a24), 1.0 / 3.0, dd);
        const double tr = sxx + syy, pk = pc * P.kB;
        dQ = pk * (sxx - syy);
        Qxy = pk * ((a57 - a68) * (1.0 / 12.0));
        // 1.5 (Qxx + Qyy) = psi (3 kA (tr - dd) + 1.5 kB tr)
        Ls = fma(pc, fma(P.kA3, tr - dd, P.kB15 * tr), Ls);
    }
    const double r = rcp_d(rho);
    const double hx = fma(0.5, Fx, p.jx), hy = fma(0.5, Fy, p.jy);  // rho u
    const double ux = hx * r, uy = hy * r;
    // (sums and differences of products as explicit fma, so that every role rounds them alike)
    const double Y = hy * uy, uFy = uy * Fy, ruu = fma(hx, ux, Y), uF = fma(ux, Fx, uFy);
    // e - e_eq = -2 f0 + sax + 4 sdg - 3 rho uu, zeta - zeta_eq = 3 (f0 - sax + rho uu)
    // (what a role has no use for is not computed)
    const double ene = fma(-3.0, ruu, fma(4.0, p.sdg, fma(-2.0, v[0], p.sax)));
    const double zne = fma(3.0, (v[0] - p.sax) + ruu, Ls);
    const double de = fma(P.h6_e, uF, P.s_e * (Ls - ene));
    const double dz = -fma(P.h6_z, uF, P.s_z * zne);
    const double dqx = -fma(P.h_q, Fx, P.s_q * (fma(-2.0, p.d13, p.t) + hx));
    const double dqy = -fma(P.h_q, Fy, P.s_q * (fma(-2.0, p.d24, p.s) + hy));
    const double P4 = fma(P.hn2, fma(ux, Fx, -uFy), P.sn4 * (fma(hx, ux, -Y) - p.pxx - dQ));
    const double Z = fma(P.hn4, fma(ux, Fy, uy * Fx), P.sn4 * (fma(hx, uy, -p.pxy) - Qxy));
    apply_role<ROLE>(v, de, dz, Fx, dqx, Fy, dqy, P4, Z, E);
}

// Free-energy collision (Eqs. 1, 6, 20, 21, 24) from the cell's force F, its velocity and the
// neighbours' rho.  IWB: the A and p_g terms of the full model (fe_collide_iwb).
struct Iwb64 {
    double dxux, dyux, dxuy, dyuy;  // 12 times the velocity derivatives
    double pg, dpg, A;
};
template <bool IWB, int ROLE>
__device__ __forceinline__ void fe_collide_d(double v[9], double rho, const double rn[9], double hx, double hy,
                                             double ux, double uy, double Fx, double Fy, const Pairs& p,
                                             const Iwb64& W, const StepParams<double>& P, const Exchange& E) {
    double gx, gy;
    grad12(rn, gx, gy);
    const double Y = hy * uy, ruu = fma(hx, ux, Y);
    const double Fg = IWB ? Fy - W.dpg : Fy;
    const double s = fma(ux, gx, uy * gy);                               // 12 u . grad rho
    const double Gx = fma(gx, 1.0 / 36.0, Fx), Gy = fma(gy, 1.0 / 36.0, Fg);  // F + c_s^2 grad rho
    const double fe = fma(6.0, fma(ux, Fx, uy * Fg), s * (1.0 / 3.0));   // 6 u.F + 4 u.grad rho
    // (e - e_eq) / 3 = sax + 2 sdg - rho uu, -(zeta - zeta_eq) / 3 = 2 sax + sdg - rho uu
    double ene = fma(2.0, p.sdg, p.sax) - ruu, zne = fma(2.0, p.sax, p.sdg) - ruu;
    double Nx = fma(hx, ux, -Y) - p.pxx, Nxy = fma(hx, uy, -p.pxy);
    if (IWB) {
        // rho A tr S / 3, rho A (S_xx - S_yy) / 3, rho A S_xy / 3
        const double rA = rho * (W.A * (1.0 / 36.0)), rA2 = rA + rA;
        const double as = rA2 * (W.dxux + W.dyuy);
        ene = fma(-2.0, W.pg, ene - as);
        zne = fma(-3.0, W.pg, zne - as);
        Nx = fma(rA2, W.dxux - W.dyuy, Nx);
        Nxy = fma(rA, W.dxuy + W.dyux, Nxy);
    }
    // (what a role has no use for is not computed)
    const double de = fma(P.h_e, fe, P.me3 * ene);
    const double dz = fma(-P.h_z, fe, P.sz3 * zne);
    const double dqx = -fma(P.h_q, Fx, P.s_q * (fma(-2.0, p.d13, p.t) + hx));
    const double dqy = -fma(P.h_q, Fy, P.s_q * (fma(-2.0, p.d24, p.s) + hy));
    const double P4 = fma(P.hn2, fma(ux, Gx, -(uy * Gy)), P.sn4 * Nx);
    const double Z = fma(P.hn4, fma(ux, Gy, uy * Gx), P.sn4 * Nxy);
    apply_role<ROLE>(v, de, dz, Fx, dqx, Fy, dqy, P4, Z, E);
}
template <int ROLE>
__device__ __forceinline__ void tile_collide_fe(double v[9], double rho, const double mn[9], const double rn[9],
                                                double fx, double fy, unsigned&, const StepParams<double>& P,
                                                const Exchange& E) {
    const Pairs p = pairs_of(v);
    double gx, gy;
    grad12(mn, gx, gy);
    const double m = rho * (-1.0 / 12.0);
    const double Fx = fma(m, gx, fx), Fy = fma(m, gy, fy);
    const double hx = fma(0.5, Fx, p.jx), hy = fma(0.5, Fy, p.jy), r = rcp_d(rho);
    fe_collide_d<false, ROLE>(v, rho, rn, hx, hy, hx * r, hy * r, Fx, Fy, p, Iwb64{}, P, E);
}
__device__ __forceinline__ void tile_velocity(const double v[9], double rho, const double mn[9], double fx, double fy,
                                              double& ux, double& uy, double& Fx, double& Fy) {
    const Pairs p = pairs_of(v);
    double gx, gy;
    grad12(mn, gx, gy);
    const double m = rho * (-1.0 / 12.0);
    Fx = fma(m, gx, fx);
    Fy = fma(m, gy, fy);
    const double r = rcp_d(rho);
    ux = fma(0.5, Fx, p.jx) * r;
    uy = fma(0.5, Fy, p.jy) * r;
}
__device__ __forceinline__ void tile_collide_iwb(double v[9], double rho, const double rn[9], const double un[9],
                                                 const double wn[9], double ux, double uy, double Fx, double Fy,
                                                 double pg, double dpg, double A, unsigned&,
                                                 const StepParams<double>& P) {
    const Pairs p = pairs_of(v);
    Iwb64 W;
    grad12(un, W.dxux, W.dyux);
    grad12(wn, W.dxuy, W.dyuy);
    W.pg = pg;
    W.dpg = dpg;
    W.A = A;
    fe_collide_d<true, -1>(v, rho, rn, fma(0.5, Fx, p.jx), fma(0.5, Fy, p.jy), ux, uy, Fx, Fy, p, W, P, Exchange{});
}

}  // namespace lbmk
