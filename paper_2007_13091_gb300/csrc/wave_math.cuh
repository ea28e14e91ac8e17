// The wave flux of a face in the lab frame (Sec. 2.1, 2.3): second order for an
// interior face, first order for a boundary face or a first-order step, and for each
// the product of its Jacobian's transpose with a given face vector (hand-written
// reverse pass).  Plain functions of scalars, used by the step's flux kernels and by
// the adjoint kernels; they compile for the host as well.
//
// Every slope moment of the flux is the derivative of a Maxwellian moment
// along the gradient of the primitive state (rho, U, theta = RT): for a
// direction x and a moment function Q(rho, U, theta),
//   <.. (a_x . psi) psi> rho = dQ/drho rho_x + dQ/dU . U_x + dQ/dtheta theta_x.
// The half-space moments N_k = int_half u_n^k g1 of the normal velocity obey
//   dN_0/dU_n = s phi,  dN_k/dU_n = k N_{k-1},  dN_k/dtheta = k (k - 1) N_{k-2} / 2
//   (dN_1/dtheta = s phi / 2),  s phi = +- g1(u_n = 0),
// and the tangential velocity integrates over all of its range, so that no
// face frame, no micro-slope solve and no moment tables are needed: with the
// tangential mean velocity V = U - U_n n the slopes enter through their normal
// derivative n.grad, their derivative V.grad along V, grad U_n and the
// divergence of U.  Per face this takes about 0.6 of the binary64 operations of
// micro slopes and moment tables in a face frame.
#pragma once
#include <math.h>

#ifdef __CUDACC__
#define UGKWP_HD __host__ __device__ __forceinline__
#else
#define UGKWP_HD inline
#endif

namespace ugkwp {
namespace wm {

// Constants of K internal degrees of freedom (rho E = rho |U|^2/2 + (3+K)/2 p).
struct Gas {
    double K, c23;  // K, 2/(3+K)
};
UGKWP_HD Gas gas_of(int K) { return Gas{(double)K, 2.0 / (3.0 + (double)K)}; }

UGKWP_HD double dot(const double* a, const double* b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; }

// 1/sqrt(x)
UGKWP_HD double rsqrt_(double x) {
#ifdef __CUDA_ARCH__
    return ::rsqrt(x);
#else
    return 1.0 / ::sqrt(x);
#endif
}

// e^{x^2} erfc(x), x >= 0
UGKWP_HD double erfcx_(double x) {
#ifdef __CUDA_ARCH__
    return ::erfcx(x);
#else
    return exp(x * x) * erfc(x);
#endif
}

// N_0..N_4 and s phi of the unit Maxwellian of mean U_n and variance theta over
// u_n > 0 (s = 1) or u_n < 0 (s = -1).  erfc(|a|) = e^{-a^2} erfcx(|a|) shares
// its exponential with phi (57 binary64 instructions instead of 77 for erfc and
// exp on their own), and the two terms of N_1, which cancel in a supersonic
// tail, then carry the same rounding of it.
struct Half {
    double N[5], sphi;
};
UGKWP_HD Half half_moments(double Un, double th, double s) {
    Half h;
    const double rs = rsqrt_(th + th);
    const double a = Un * rs;
    const double e = exp(-a * a);
    h.sphi = s * (e * rs * 0.56418958354775628695);  // 1/sqrt(pi)
    const double t = 0.5 * e * erfcx_(fabs(a));
    h.N[0] = s * a > 0.0 ? 1.0 - t : t;
    h.N[1] = Un * h.N[0] + th * h.sphi;
    h.N[2] = Un * h.N[1] + th * h.N[0];
    h.N[3] = Un * h.N[2] + 2.0 * th * h.N[1];
    h.N[4] = Un * h.N[3] + 3.0 * th * h.N[2];
    return h;
}

// Primitive state of a conservative one.
struct Prim {
    double rho, ir, U[3], U2, p, th;
};
UGKWP_HD Prim prim_of(const double* W, const Gas& gas) {
    Prim s;
    s.rho = W[0];
    s.ir = 1.0 / W[0];
    for (int d = 0; d < 3; ++d) s.U[d] = W[1 + d] * s.ir;
    s.U2 = dot(s.U, s.U);
    s.p = (W[4] - 0.5 * s.rho * s.U2) * gas.c23;
    s.th = s.p * s.ir;
    return s;
}

// Gradients of U and theta from those of W (g [5][3]): gU[j][d], gt[d].
struct PrimGrad {
    double gU[3][3], gt[3];
};
UGKWP_HD PrimGrad prim_grad(const Prim& s, const double g[5][3], double scale, const Gas& gas) {
    // scale multiplies g (the mean of two gradients comes as their sum and 1/2)
    PrimGrad o;
    const double irs = s.ir * scale, c = gas.c23 * irs, tr = s.th * irs, hU2 = 0.5 * s.U2;
    for (int d = 0; d < 3; ++d) {
        double t = g[4][d] + hU2 * g[0][d];
        for (int j = 0; j < 3; ++j) {
            o.gU[j][d] = (g[1 + j][d] - s.U[j] * g[0][d]) * irs;
            t -= s.U[j] * g[1 + j][d];
        }
        o.gt[d] = c * t - tr * g[0][d];
    }
    return o;
}

// One side of a face: the moments of its half space for the reconstructed
// state: H = <psi>, G = <u_n psi> (unit density) and
// S = sum_d <u_n u_d (a_d . psi) psi> of the hydrodynamic wave (density rh,
// slopes gh of its density, U and theta of the total W).
struct SideFlux {
    double H[5], G[5], S[5];
};
template <bool SLOPES>
UGKWP_HD SideFlux side_flux(const Prim& s, const PrimGrad& pg, double rh, const double gh[3], const double n[3],
                            double sgn, const Gas& gas) {
    SideFlux o;
    const double Un = dot(s.U, n);
    double V[3];
    for (int d = 0; d < 3; ++d) V[d] = s.U[d] - Un * n[d];
    const double th = s.th;
    const Half h = half_moments(Un, th, sgn);
    const double* N = h.N;
    const double q = dot(V, V) + (2.0 + gas.K) * th;
    o.H[0] = N[0];
    o.G[0] = N[1];
    for (int d = 0; d < 3; ++d) {
        o.H[1 + d] = N[1] * n[d] + N[0] * V[d];
        o.G[1 + d] = N[2] * n[d] + N[1] * V[d];
    }
    o.H[4] = 0.5 * (N[2] + N[0] * q);
    o.G[4] = 0.5 * (N[3] + N[1] * q);
    if constexpr (SLOPES) {
        // normal derivatives, derivatives along V, grad U_n
        double Uj_n[3], DU[3], gUn[3];
        for (int j = 0; j < 3; ++j) {
            Uj_n[j] = dot(pg.gU[j], n);
            DU[j] = dot(pg.gU[j], V);
        }
        for (int d = 0; d < 3; ++d) gUn[d] = n[0] * pg.gU[0][d] + n[1] * pg.gU[1][d] + n[2] * pg.gU[2][d];
        const double rn = dot(gh, n), Dr = dot(gh, V), tn = dot(pg.gt, n), Dt = dot(pg.gt, V);
        const double Unn = dot(Uj_n, n), DUn = dot(DU, n);
        const double dv = (pg.gU[0][0] + pg.gU[1][1] + pg.gU[2][2]) - Unn;  // tangential divergence
        const double r0 = rh * N[0], r1 = rh * N[1], r2 = rh * N[2], r3 = rh * N[3];
        const double rf = 0.5 * rh * h.sphi;
        const double X2 = rn * N[2] + 2.0 * r1 * Unn + r0 * tn;
        const double X3 = rn * N[3] + 3.0 * (r2 * Unn + r1 * tn);
        const double X4 = rn * N[4] + 4.0 * r3 * Unn + 6.0 * r2 * tn;
        const double Y1 = Dr * N[1] + r0 * DUn + rf * Dt + r1 * dv;
        const double Y2 = Dr * N[2] + 2.0 * r1 * DUn + r0 * Dt + r2 * dv;
        const double Y3 = Dr * N[3] + 3.0 * (r2 * DUn + r1 * Dt) + r3 * dv;
        const double a3 = th * N[1], a4 = th * r0, a5 = th * rf + r1;
        const double XY = X2 + Y1;
        const double nZ = r2 * Unn + r1 * DUn + a3 * rn + a4 * Unn + a5 * tn;
        const double c = (X3 + Y2) - nZ;
        o.S[0] = XY;
        for (int d = 0; d < 3; ++d)
            o.S[1 + d] = XY * V[d] + r2 * Uj_n[d] + r1 * DU[d] + a3 * gh[d] + a4 * gUn[d] + a5 * pg.gt[d] + c * n[d];
        o.S[4] = 0.5 * (X4 + Y3 + XY * q + 2.0 * (Y1 * th + r2 * dot(V, Uj_n) + r1 * dot(V, DU)) +
                        r2 * ((2.0 + gas.K) * tn) + r1 * ((4.0 + gas.K) * Dt));
    } else {
        for (int k = 0; k < 5; ++k) o.S[k] = 0.0;
    }
    return o;
}

// q1..q5, a4, a5 (time integrals of Sec. 2.1) from one expm1.  q1, q4 and a4 are
// differences of terms of size dt, and carry absolute errors of some 2^-52 dt; q2, q3,
// q5 and a5 are differences of terms of size tau dt, with errors of some
// 2^-52 dt max(tau, dt): far below dt^2, the scale at which they enter the flux, as long as
// tau/dt is far below 2^52 (1e-12 dt^2 at dt/tau = 1e-4, 1e-8 dt^2 at 1e-8), but not
// relative to their own values, which fall as dt^3/tau.
struct QC {
    double q1, q2, q3, q4, q5, a4, a5, e;
};
UGKWP_HD QC time_coeffs_all(double dt, double tau) {
    QC c;
    const double em1 = expm1(-dt / tau);
    const double e = 1.0 + em1;
    const double tdt = tau * dt;
    c.e = e;
    c.q4 = -tau * em1;
    c.q1 = dt - c.q4;
    c.a4 = c.q4 - dt * e;
    c.q2 = 2.0 * tau * c.q4 - tdt - tdt * e;
    c.q3 = 0.5 * dt * dt - tdt + tau * c.q4;
    c.q5 = tdt * e - tau * c.q4;
    c.a5 = c.q5 + 0.5 * dt * dt * e;
    return c;
}

// q1, q4 and a4 = q4 - dt e^{-dt/tau} of the first-order flux, with x = dt/tau:
// below x = 1 all from s1 = e^{-x} - 1 + x by its Taylor series (18 terms, the
// last below 2^-56 of the sum), which keeps their relative accuracy:
// q1 = tau s1, q4 = tau (x - s1), a4 = tau (x^2 - (1 + x) s1).
struct QC1 {
    double q1, q4, a4, e;
};
UGKWP_HD QC1 time_coeffs(double dt, double tau) {
    QC1 c;
    const double x = dt / tau;
    if (x < 1.0) {
        // s1 / x^2 = sum_k (-x)^k / (k + 2)!, from k = 17 down
        double p = 1.0 / 121645100408832000.0;
        const double f[17] = {1.0 / 6402373705728000.0, 1.0 / 355687428096000.0, 1.0 / 20922789888000.0,
                              1.0 / 1307674368000.0, 1.0 / 87178291200.0, 1.0 / 6227020800.0, 1.0 / 479001600.0,
                              1.0 / 39916800.0, 1.0 / 3628800.0, 1.0 / 362880.0, 1.0 / 40320.0, 1.0 / 5040.0,
                              1.0 / 720.0, 1.0 / 120.0, 1.0 / 24.0, 1.0 / 6.0, 0.5};
        for (int k = 0; k < 17; ++k) p = f[k] - p * x;
        const double s1 = p * x * x;
        c.q1 = tau * s1;
        c.q4 = tau * (x - s1);
        c.a4 = tau * (x * x - (1.0 + x) * s1);
        c.e = (1.0 - x) + s1;
    } else {
        const double em1 = expm1(-x);
        c.e = 1.0 + em1;
        c.q4 = -tau * em1;
        c.q1 = dt - c.q4;
        c.a4 = c.q4 - dt * c.e;
    }
    return c;
}
UGKWP_HD double time_coeffs_adj1(const QC1& c, double dt, double tau, double q1b, double q4b, double a4b) {
    const double x = dt / tau, d = c.a4 / tau;
    return (q4b - q1b + a4b) * d - a4b * (x * x * c.e);
}

// The gas constants a face flux needs.
struct FaceGas {
    Gas gas;
    double mu_ref, omega, iRT, C2;  // iRT = 1 / (R T_ref)
};
UGKWP_HD double face_tau0(const Prim& s, const FaceGas& g) { return g.mu_ref * exp(g.omega * log(s.th * g.iRT)) / s.p; }

// First-order flux between two states (normal n from L to R): ghost: R emits
// no particles, so that its half carries the whole q4; gks: both halves do.
UGKWP_HD void flux_o1(const Prim& L, double rhL, const Prim& R, double rhR, bool ghost, bool gks, const double n[3],
                      double dt, const FaceGas& g, double F[5]) {
    const PrimGrad none{};
    const double z[3] = {0.0, 0.0, 0.0};
    const SideFlux a = side_flux<false>(L, none, rhL, z, n, 1.0, g.gas), b = side_flux<false>(R, none, rhR, z, n, -1.0, g.gas);
    double W0[5];
    for (int k = 0; k < 5; ++k) W0[k] = L.rho * a.H[k] + R.rho * b.H[k];
    const Prim c = prim_of(W0, g.gas);
    double tau = face_tau0(c, g);
    if (g.C2 > 0.0) tau += g.C2 * fabs(L.p - R.p) / fabs(L.p + R.p) * dt;
    const QC1 q = time_coeffs(dt, tau);
    const double cL = rhL * (gks ? q.q4 : q.a4), cR = rhR * (ghost || gks ? q.q4 : q.a4);
    const double m = dot(W0 + 1, n), Un = dot(c.U, n);
    F[0] = q.q1 * m + cL * a.G[0] + cR * b.G[0];
    for (int d = 0; d < 3; ++d) F[1 + d] = q.q1 * (m * c.U[d] + c.p * n[d]) + cL * a.G[1 + d] + cR * b.G[1 + d];
    F[4] = q.q1 * (Un * (W0[4] + c.p)) + cL * a.G[4] + cR * b.G[4];
}

// Equilibrium part q1 g0 + q2 u.g_x + q3 g_t of the flux along n: g0 the
// Maxwellian of W0, g_x from the gradient `scale` B of W, g_t from
// W_t = -div F.  In primitive form, with D = U.grad and C = D rho + rho div U:
//   rho_t = -C, U_t = -(D U + grad(rho theta)/rho), theta_t = -(D theta + c23 theta div U).
// pr_fix: (1/Pr - 1) times the heat flux of this part relative to U0 is added
// to the energy flux; e1 = q3 - q2 of its full moments.
UGKWP_HD void equilibrium_flux(const double* W0, const Prim& s, const double B[5][3], double scale, const double n[3],
                               const QC& c, double pr_fix, const Gas& gas, double F[5]) {
    const PrimGrad pg = prim_grad(s, B, scale, gas);
    const double rho = s.rho, th = s.th;
    double gr[3], gP[3];
    for (int d = 0; d < 3; ++d) {
        gr[d] = scale * B[0][d];
        gP[d] = th * gr[d] + rho * pg.gt[d];  // grad(rho theta)
    }
    const double Un = dot(s.U, n);
    const double dv = pg.gU[0][0] + pg.gU[1][1] + pg.gU[2][2];
    double DU[3], Uj_n[3], gUn[3];
    for (int j = 0; j < 3; ++j) {
        DU[j] = dot(pg.gU[j], s.U);
        Uj_n[j] = dot(pg.gU[j], n);
    }
    for (int d = 0; d < 3; ++d) gUn[d] = n[0] * pg.gU[0][d] + n[1] * pg.gU[1][d] + n[2] * pg.gU[2][d];
    const double Dr = dot(gr, s.U), Dt = dot(pg.gt, s.U), tn = dot(pg.gt, n), Pn = dot(gP, n);
    const double C = Dr + rho * dv, DUn = dot(DU, n);
    const double P = rho * th, rUn = rho * Un;
    // q2 <u_n u.(a psi) psi>
    const double M = Un * C + rho * DUn;
    const double A7 = s.U2 + (7.0 + gas.K) * th, A5 = s.U2 + (5.0 + gas.K) * th;
    const double cn = th * C + rho * Dt;
    const double UDU = dot(s.U, DU), UUn = dot(s.U, Uj_n);
    double T[5];
    T[0] = M + Pn;
    for (int k = 0; k < 3; ++k)
        T[1 + k] = T[0] * s.U[k] + rUn * DU[k] + Un * gP[k] + P * (gUn[k] + Uj_n[k]) + cn * n[k];
    T[4] = 0.5 * (M * A7 + rUn * (2.0 * UDU + (7.0 + gas.K) * Dt) + Pn * A5 + P * (2.0 * UUn + (5.0 + gas.K) * tn));
    // time derivatives
    const double rt = -C, tt = -(Dt + gas.c23 * (th * dv));
    double Ut[3];
    for (int k = 0; k < 3; ++k) Ut[k] = -(DU[k] + gP[k] * s.ir);
    const double Unt = dot(Ut, n), UUt = dot(s.U, Ut);
    const double h5 = 0.5 * A5;
    double R[5];
    R[0] = rt * Un + rho * Unt;
    const double ct = rt * th + rho * tt;
    for (int k = 0; k < 3; ++k) R[1 + k] = R[0] * s.U[k] + rUn * Ut[k] + ct * n[k];
    R[4] = R[0] * h5 + rUn * (UUt + 0.5 * (5.0 + gas.K) * tt);
    double Fe[5];
    Fe[0] = c.q1 * rUn + c.q2 * T[0] + c.q3 * R[0];
    for (int k = 0; k < 3; ++k) Fe[1 + k] = c.q1 * (rUn * s.U[k] + P * n[k]) + c.q2 * T[1 + k] + c.q3 * R[1 + k];
    Fe[4] = c.q1 * (Un * (W0[4] + P)) + c.q2 * T[4] + c.q3 * R[4];
    if (pr_fix != 0.0) {
        // q_n = Fe_E - U0.Fe_m + |U0|^2/2 Fe_rho - U0_n (E' - U0.M' + |U0|^2/2 rho'),
        // the full moments (rho', M', E') = q1 W0 + (q3 - q2) W_t:
        // relative to U0 they are q1 and (q3 - q2) times (3+K)/2 of P and of P_t
        const double qf = (Fe[4] - dot(s.U, Fe + 1)) + 0.5 * s.U2 * Fe[0];
        const double qm = (c.q1 * P + (c.q3 - c.q2) * (rt * th + rho * tt)) / gas.c23;
        Fe[4] += pr_fix * (qf - Un * qm);
    }
    for (int k = 0; k < 5; ++k) F[k] += Fe[k];
}

// ------------------------------------------------------------ reverse pass
// Adjoint of a value x is written x_b: the derivative of a scalar along x.

// Adjoint of a side's half-space moments: from N_b, sphi_b to U_n and theta.
UGKWP_HD void half_moments_adj(const Half& h, double Un, double th, const double Nb[5], double fb, double& Un_b,
                               double& th_b) {
    const double* N = h.N;
    const double f = h.sphi, z = Un / th;
    Un_b += Nb[0] * f + Nb[1] * N[0] + 2.0 * Nb[2] * N[1] + 3.0 * Nb[3] * N[2] + 4.0 * Nb[4] * N[3] - fb * f * z;
    th_b += 0.5 * f * (Nb[1] - Nb[0] * z) + Nb[2] * N[0] + 3.0 * Nb[3] * N[1] + 6.0 * Nb[4] * N[2] +
            fb * f * 0.5 * (z * z - 1.0 / th);
}

// Adjoints of a primitive state (U, theta, 1/rho, rho and p as they were used).
struct PrimAdj {
    double U[3], th, ir, rho, p;
};
UGKWP_HD PrimAdj prim_adj_zero() { return PrimAdj{{0.0, 0.0, 0.0}, 0.0, 0.0, 0.0, 0.0}; }

// Wb += the adjoint of the conservative state (a is used up).
UGKWP_HD void prim_adj(const Prim& s, PrimAdj a, const Gas& gas, double Wb[5]) {
    a.p += a.th * s.ir;
    a.ir += a.th * s.p;
    const double pe = gas.c23 * a.p;
    a.rho -= 0.5 * pe * s.U2;
    for (int d = 0; d < 3; ++d) a.U[d] -= pe * s.rho * s.U[d];
    a.ir += dot(a.U, s.U) * s.rho;
    Wb[0] += a.rho - a.ir * s.ir * s.ir;
    for (int d = 0; d < 3; ++d) Wb[1 + d] += a.U[d] * s.ir;
    Wb[4] += pe;
}

// Adjoint of prim_grad: gb += (adjoint of g), a += (adjoint of the state).
UGKWP_HD void prim_grad_adj(const Prim& s, const double g[5][3], double scale, const PrimGrad& pg, const PrimGrad& b,
                            const Gas& gas, double gb[5][3], PrimAdj& a) {
    const double irs = s.ir * scale, c = gas.c23 * irs, tr = s.th * irs, hU2 = 0.5 * s.U2;
    double w = 0.0, t0 = 0.0;
    for (int d = 0; d < 3; ++d) {
        double ug = 0.0;
        for (int j = 0; j < 3; ++j) {
            gb[1 + j][d] += b.gU[j][d] * irs - s.U[j] * (c * b.gt[d]);
            ug += s.U[j] * b.gU[j][d];
            w += b.gU[j][d] * pg.gU[j][d];
        }
        gb[0][d] += b.gt[d] * (c * hU2 - tr) - irs * ug;
        gb[4][d] += c * b.gt[d];
        w += b.gt[d] * pg.gt[d];
        t0 += b.gt[d] * g[0][d];
    }
    for (int j = 0; j < 3; ++j)
        a.U[j] += c * (t0 * s.U[j] - dot(b.gt, g[1 + j])) - irs * dot(b.gU[j], g[0]);
    a.th -= irs * t0;
    a.ir += w * s.rho;
}

// Adjoint of side_flux: a += the state's, pgb, rh_b, gh_b the slopes'.
template <bool SLOPES>
UGKWP_HD void side_flux_adj(const Prim& s, const PrimGrad& pg, double rh, const double gh[3], const double n[3],
                            double sgn, const Gas& gas, const double Hb[5], const double Gb[5], const double Sb[5],
                            PrimAdj& a, PrimGrad& pgb, double& rh_b, double gh_b[3]) {
    const double Un = dot(s.U, n);
    double V[3];
    for (int d = 0; d < 3; ++d) V[d] = s.U[d] - Un * n[d];
    const double th = s.th;
    const Half h = half_moments(Un, th, sgn);
    const double* N = h.N;
    const double K = gas.K, q = dot(V, V) + (2.0 + K) * th;
    double Nb[5], fb = 0.0, th_b = 0.0, Un_b = 0.0, Vb[3];
    // H and G
    Nb[0] = Hb[0] + dot(Hb + 1, V) + 0.5 * Hb[4] * q;
    Nb[1] = Gb[0] + dot(Hb + 1, n) + dot(Gb + 1, V) + 0.5 * Gb[4] * q;
    Nb[2] = 0.5 * Hb[4] + dot(Gb + 1, n);
    Nb[3] = 0.5 * Gb[4];
    Nb[4] = 0.0;
    double q_b = 0.5 * (Hb[4] * N[0] + Gb[4] * N[1]);
    for (int d = 0; d < 3; ++d) Vb[d] = N[0] * Hb[1 + d] + N[1] * Gb[1 + d];
    if constexpr (SLOPES) {
        double Uj_n[3], DU[3], gUn[3];
        for (int j = 0; j < 3; ++j) {
            Uj_n[j] = dot(pg.gU[j], n);
            DU[j] = dot(pg.gU[j], V);
        }
        for (int d = 0; d < 3; ++d) gUn[d] = n[0] * pg.gU[0][d] + n[1] * pg.gU[1][d] + n[2] * pg.gU[2][d];
        const double rn = dot(gh, n), Dr = dot(gh, V), tn = dot(pg.gt, n), Dt = dot(pg.gt, V);
        const double Unn = dot(Uj_n, n), DUn = dot(DU, n);
        const double dv = (pg.gU[0][0] + pg.gU[1][1] + pg.gU[2][2]) - Unn;
        const double r0 = rh * N[0], r1 = rh * N[1], r2 = rh * N[2], r3 = rh * N[3], rf = 0.5 * rh * h.sphi;
        const double a3 = th * N[1], a4 = th * r0, a5 = th * rf + r1;
        const double Y1 = Dr * N[1] + r0 * DUn + rf * Dt + r1 * dv;
        const double XY = rn * N[2] + 2.0 * r1 * Unn + r0 * tn + Y1;
        const double* bv = Sb + 1;
        const double b4 = 0.5 * Sb[4];
        const double cb = dot(bv, n);  // adjoint of X3, Y2 and -nZ
        const double XYb = Sb[0] + dot(bv, V) + b4 * q;
        const double VU = dot(V, Uj_n), VD = dot(V, DU);
        q_b += b4 * XY;
        const double Y1b = XYb + 2.0 * b4 * th;
        // coefficients of the vector part
        const double a3b = dot(bv, gh) - cb * rn, a4b = dot(bv, gUn) - cb * Unn, a5b = dot(bv, pg.gt) - cb * tn;
        double r0b = a4b * th + XYb * tn + Y1b * DUn + cb * Dt;
        double r1b = dot(bv, DU) + b4 * (2.0 * VD + (4.0 + K) * Dt) - cb * DUn + a5b + 2.0 * XYb * Unn +
                     3.0 * cb * tn + Y1b * dv + 2.0 * cb * DUn + 3.0 * b4 * Dt;
        double r2b = dot(bv, Uj_n) + b4 * (2.0 * VU + (2.0 + K) * tn) - cb * Unn + 3.0 * cb * Unn + 6.0 * b4 * tn +
                     cb * dv + 3.0 * b4 * DUn;
        const double r3b = 4.0 * b4 * Unn + b4 * dv;
        const double rfb = a5b * th + Y1b * Dt;
        th_b += 2.0 * b4 * Y1 + a3b * N[1] + a4b * r0 + a5b * rf;
        Nb[1] += a3b * th + Y1b * Dr;
        Nb[2] += XYb * rn + cb * Dr;
        Nb[3] += cb * rn + b4 * Dr;
        Nb[4] += b4 * rn;
        const double rn_b = XYb * N[2] + cb * (N[3] - a3) + b4 * N[4];
        const double Dr_b = Y1b * N[1] + cb * N[2] + b4 * N[3];
        const double tn_b = b4 * r2 * (8.0 + K) - cb * a5 + 3.0 * cb * r1 + XYb * r0;
        const double Dt_b = b4 * r1 * (7.0 + K) + cb * r0 + Y1b * rf;
        const double dv_b = b4 * r3 + cb * r2 + Y1b * r1;
        const double Unn_b = -cb * (r2 + a4) + 4.0 * b4 * r3 + 3.0 * cb * r2 + 2.0 * XYb * r1 - dv_b;
        const double DUn_b = -cb * r1 + 3.0 * b4 * r2 + 2.0 * cb * r1 + Y1b * r0;
        rh_b += 0.5 * rfb * h.sphi + r0b * N[0] + r1b * N[1] + r2b * N[2] + r3b * N[3];
        fb = 0.5 * rfb * rh;
        Nb[0] += r0b * rh;
        Nb[1] += r1b * rh;
        Nb[2] += r2b * rh;
        Nb[3] += r3b * rh;
        double DUb[3], Ujb[3];
        for (int j = 0; j < 3; ++j) {
            const double t = bv[j] + 2.0 * b4 * V[j];
            DUb[j] = r1 * t + DUn_b * n[j];
            Ujb[j] = r2 * t + Unn_b * n[j];
        }
        for (int d = 0; d < 3; ++d) {
            gh_b[d] += a3 * bv[d] + rn_b * n[d] + Dr_b * V[d];
            pgb.gt[d] += a5 * bv[d] + tn_b * n[d] + Dt_b * V[d];
            Vb[d] += XY * bv[d] + 2.0 * b4 * (r2 * Uj_n[d] + r1 * DU[d]) + Dr_b * gh[d] + Dt_b * pg.gt[d] +
                     (DUb[0] * pg.gU[0][d] + DUb[1] * pg.gU[1][d] + DUb[2] * pg.gU[2][d]);
            for (int j = 0; j < 3; ++j) pgb.gU[j][d] += n[j] * (a4 * bv[d]) + DUb[j] * V[d] + Ujb[j] * n[d];
            pgb.gU[d][d] += dv_b;
        }
    }
    for (int d = 0; d < 3; ++d) Vb[d] += 2.0 * q_b * V[d];
    th_b += (2.0 + K) * q_b;
    half_moments_adj(h, Un, th, Nb, fb, Un_b, th_b);
    Un_b -= dot(Vb, n);
    for (int d = 0; d < 3; ++d) a.U[d] += Vb[d] + Un_b * n[d];
    a.th += th_b;
}

// Adjoint of flux_o1 (with particles): the states' adjoints are added to aL, aR,
// those of rhL, rhR to rhLb, rhRb.
UGKWP_HD void flux_o1_adj(const Prim& L, double rhL, const Prim& R, double rhR, bool ghost, const double n[3],
                          double dt, const FaceGas& g, const double Fb[5], PrimAdj& aL, double& rhLb, PrimAdj& aR,
                          double& rhRb) {
    const PrimGrad none{};
    const double z[3] = {0.0, 0.0, 0.0};
    const SideFlux a = side_flux<false>(L, none, rhL, z, n, 1.0, g.gas), b = side_flux<false>(R, none, rhR, z, n, -1.0, g.gas);
    double W0[5];
    for (int k = 0; k < 5; ++k) W0[k] = L.rho * a.H[k] + R.rho * b.H[k];
    const Prim c = prim_of(W0, g.gas);
    const double tau0 = face_tau0(c, g);
    double tau = tau0, rD = 0.0;
    const double D = L.p - R.p, iS = 1.0 / fabs(L.p + R.p);
    if (g.C2 > 0.0) {
        rD = fabs(D) * iS;
        tau += g.C2 * rD * dt;
    }
    const QC1 q = time_coeffs(dt, tau);
    const double m = dot(W0 + 1, n), Un = dot(c.U, n);
    const double* bv = Fb + 1;
    const double bU = dot(bv, c.U), bn = dot(bv, n), Ep = W0[4] + c.p;
    double q1b = Fb[0] * m + m * bU + c.p * bn + Fb[4] * Un * Ep, GL = 0.0, GR = 0.0;
    for (int k = 0; k < 5; ++k) {
        GL += Fb[k] * a.G[k];
        GR += Fb[k] * b.G[k];
    }
    const double cL = q.a4, cR = ghost ? q.q4 : q.a4;
    const double a4b = rhL * GL + (ghost ? 0.0 : rhR * GR), q4b = ghost ? rhR * GR : 0.0;
    const double taub = time_coeffs_adj1(q, dt, tau, q1b, q4b, a4b);
    // W0 through the Euler flux and tau0 = mu_ref (T0/T_ref)^omega / p0
    PrimAdj s = prim_adj_zero();
    s.p = q.q1 * (bn + Fb[4] * Un) - taub * tau0 / c.p;
    s.th = taub * g.omega * tau0 / c.th;
    const double mb = q.q1 * (Fb[0] + bU), Unb = q.q1 * Fb[4] * Ep;
    for (int d = 0; d < 3; ++d) s.U[d] = q.q1 * m * bv[d] + Unb * n[d];
    double W0b[5] = {0.0, mb * n[0], mb * n[1], mb * n[2], q.q1 * Fb[4] * Un};
    prim_adj(c, s, g.gas, W0b);
    double Hb[5], Gb[5], Sb[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, unused[3] = {0.0, 0.0, 0.0};
    PrimGrad nb{};
    for (int k = 0; k < 5; ++k) {
        Hb[k] = L.rho * W0b[k];
        Gb[k] = cL * rhL * Fb[k];
        aL.rho += W0b[k] * a.H[k];
        aR.rho += W0b[k] * b.H[k];
    }
    rhLb += cL * GL;
    rhRb += cR * GR;
    side_flux_adj<false>(L, none, rhL, z, n, 1.0, g.gas, Hb, Gb, Sb, aL, nb, rhLb, unused);
    for (int k = 0; k < 5; ++k) {
        Hb[k] = R.rho * W0b[k];
        Gb[k] = cR * rhR * Fb[k];
    }
    side_flux_adj<false>(R, none, rhR, z, n, -1.0, g.gas, Hb, Gb, Sb, aR, nb, rhRb, unused);
    if (g.C2 > 0.0) {
        const double t = taub * g.C2 * dt * iS, sg = D > 0.0 ? 1.0 : D < 0.0 ? -1.0 : 0.0;
        aL.p += t * (sg - rD);
        aR.p -= t * (sg + rD);
    }
}

// d/dtau of the time coefficients, contracted with their adjoints.  Absolute errors of
// some 2^-52 dt in the derivatives of q2, q3 and a5, of 2^-52 dt/tau in those of q1, q4
// and a4, by the same differences.
UGKWP_HD double time_coeffs_adj(const QC& c, double dt, double tau, double q1b, double q2b, double q3b, double q4b,
                                double a4b, double a5b) {
    const double x = dt / tau, xe = x * c.e, dq4 = c.a4 / tau;
    const double dq5 = dt * c.e + dt * xe - c.q4 - tau * dq4;
    return (q4b - q1b) * dq4 + q2b * (2.0 * (c.q4 + tau * dq4) - dt * (1.0 + c.e) - dt * xe) +
           q3b * (c.q4 + tau * dq4 - dt) + a4b * (dq4 - x * xe) + a5b * (dq5 + 0.5 * dt * x * xe);
}

// Adjoint of equilibrium_flux: a += (the adjoint of the primitive state), E_b += (of the
// energy W0[4]), Bb += (of B itself), qb += (of q1, q2, q3).
UGKWP_HD void equilibrium_flux_adj(const double* W0, const Prim& s, const double B[5][3], double scale,
                                   const double n[3], const QC& c, double pr_fix, const Gas& gas, const double Fb[5],
                                   PrimAdj& a, double& E_b, double Bb[5][3], double qb[3]) {
    const PrimGrad pg = prim_grad(s, B, scale, gas);
    const double K = gas.K, rho = s.rho, th = s.th;
    double gr[3], gP[3];
    for (int d = 0; d < 3; ++d) {
        gr[d] = scale * B[0][d];
        gP[d] = th * gr[d] + rho * pg.gt[d];
    }
    const double Un = dot(s.U, n);
    const double dv = pg.gU[0][0] + pg.gU[1][1] + pg.gU[2][2];
    double DU[3], Uj_n[3], gUn[3];
    for (int j = 0; j < 3; ++j) {
        DU[j] = dot(pg.gU[j], s.U);
        Uj_n[j] = dot(pg.gU[j], n);
    }
    for (int d = 0; d < 3; ++d) gUn[d] = n[0] * pg.gU[0][d] + n[1] * pg.gU[1][d] + n[2] * pg.gU[2][d];
    const double Dr = dot(gr, s.U), Dt = dot(pg.gt, s.U), tn = dot(pg.gt, n), Pn = dot(gP, n);
    const double C = Dr + rho * dv, DUn = dot(DU, n), P = rho * th, rUn = rho * Un;
    const double M = Un * C + rho * DUn;
    const double A7 = s.U2 + (7.0 + K) * th, A5 = s.U2 + (5.0 + K) * th;
    const double cn = th * C + rho * Dt, UDU = dot(s.U, DU), UUn = dot(s.U, Uj_n);
    const double k7 = 2.0 * UDU + (7.0 + K) * Dt, k5 = 2.0 * UUn + (5.0 + K) * tn;
    const double rt = -C, tt = -(Dt + gas.c23 * (th * dv));
    double Ut[3];
    for (int k = 0; k < 3; ++k) Ut[k] = -(DU[k] + gP[k] * s.ir);
    const double Unt = dot(Ut, n), UUt = dot(s.U, Ut), ct = rt * th + rho * tt, ke = UUt + 0.5 * (5.0 + K) * tt;
    double E[5], T[5], R[5];
    E[0] = rUn;
    T[0] = M + Pn;
    R[0] = rt * Un + rho * Unt;
    for (int k = 0; k < 3; ++k) {
        E[1 + k] = rUn * s.U[k] + P * n[k];
        T[1 + k] = T[0] * s.U[k] + rUn * DU[k] + Un * gP[k] + P * (gUn[k] + Uj_n[k]) + cn * n[k];
        R[1 + k] = R[0] * s.U[k] + rUn * Ut[k] + ct * n[k];
    }
    E[4] = Un * (W0[4] + P);
    T[4] = 0.5 * (M * A7 + rUn * k7 + Pn * A5 + P * k5);
    R[4] = 0.5 * R[0] * A5 + rUn * ke;
    double b[5], Ub[3] = {0.0, 0.0, 0.0}, U2_b = 0.0, Un_b = 0.0, P_b = 0.0, ct_b = 0.0, th_b = 0.0, rho_b = 0.0,
                 ir_b = 0.0;
    for (int k = 0; k < 5; ++k) b[k] = Fb[k];
    if (pr_fix != 0.0) {
        const double i23 = 1.0 / gas.c23, g = pr_fix * Fb[4];
        double Fe[5];
        for (int k = 0; k < 4; ++k) Fe[k] = c.q1 * E[k] + c.q2 * T[k] + c.q3 * R[k];
        const double qm = (c.q1 * P + (c.q3 - c.q2) * ct) * i23, qm_b = -g * Un * i23;
        Un_b -= g * qm;
        b[4] += g;
        b[0] += 0.5 * s.U2 * g;
        for (int k = 0; k < 3; ++k) {
            b[1 + k] -= g * s.U[k];
            Ub[k] -= g * Fe[1 + k];
        }
        U2_b += 0.5 * g * Fe[0];
        qb[0] += qm_b * P;
        P_b += qm_b * c.q1;
        ct_b += qm_b * (c.q3 - c.q2);
        qb[2] += qm_b * ct;
        qb[1] -= qm_b * ct;
    }
    for (int k = 0; k < 5; ++k) {
        qb[0] += b[k] * E[k];
        qb[1] += b[k] * T[k];
        qb[2] += b[k] * R[k];
    }
    const double* bv = b + 1;
    const double bU = dot(bv, s.U), bn = dot(bv, n);
    // q1 E
    double rUn_b = c.q1 * (b[0] + bU);
    P_b += c.q1 * (bn + b[4] * Un);
    Un_b += c.q1 * b[4] * (W0[4] + P);
    E_b += c.q1 * b[4] * Un;
    // q2 T
    const double t4 = 0.5 * c.q2 * b[4];
    const double T0b = c.q2 * (b[0] + bU);
    rUn_b += c.q2 * dot(bv, DU) + t4 * k7;
    Un_b += c.q2 * dot(bv, gP);
    P_b += c.q2 * (dot(bv, gUn) + dot(bv, Uj_n)) + t4 * k5;
    const double cn_b = c.q2 * bn, M_b = T0b + t4 * A7, Pn_b = T0b + t4 * A5;
    double A7_b = t4 * M, A5_b = t4 * Pn;
    const double UDU_b = 2.0 * t4 * rUn, UUn_b = 2.0 * t4 * P;
    double Dt_b = t4 * rUn * (7.0 + K), tn_b = t4 * P * (5.0 + K);
    // q3 R
    const double r4 = c.q3 * b[4], R0b = c.q3 * (b[0] + bU) + 0.5 * r4 * A5;
    rUn_b += c.q3 * dot(bv, Ut) + r4 * ke;
    ct_b += c.q3 * bn;
    A5_b += 0.5 * r4 * R[0];
    const double UUt_b = r4 * rUn;
    double tt_b = r4 * rUn * 0.5 * (5.0 + K) + ct_b * rho;
    const double rt_b = R0b * Un + ct_b * th;
    Un_b += R0b * rt;
    rho_b += R0b * Unt + ct_b * tt;
    th_b += ct_b * rt;
    const double Unt_b = R0b * rho;
    double Utb[3], DUb[3], Ujb[3], gPb[3], gUnb[3];
    for (int k = 0; k < 3; ++k) {
        Ub[k] += (c.q1 * rUn + c.q2 * T[0] + c.q3 * R[0]) * bv[k] + UUt_b * Ut[k] + UDU_b * DU[k] + UUn_b * Uj_n[k];
        Utb[k] = c.q3 * rUn * bv[k] + UUt_b * s.U[k] + Unt_b * n[k];
        DUb[k] = c.q2 * rUn * bv[k] - Utb[k] + UDU_b * s.U[k] + M_b * rho * n[k];
        gPb[k] = c.q2 * Un * bv[k] - Utb[k] * s.ir + Pn_b * n[k];
        gUnb[k] = c.q2 * P * bv[k];
        Ujb[k] = c.q2 * P * bv[k] + UUn_b * s.U[k];
    }
    ir_b -= dot(Utb, gP);
    Dt_b -= tt_b;
    th_b -= tt_b * gas.c23 * dv;
    double dv_b = -tt_b * gas.c23 * th;
    double C_b = -rt_b + cn_b * th + M_b * Un;
    U2_b += A7_b + A5_b;
    th_b += (7.0 + K) * A7_b + (5.0 + K) * A5_b + cn_b * C;
    rho_b += cn_b * Dt + M_b * DUn + C_b * dv;
    Dt_b += cn_b * rho;
    Un_b += M_b * C;
    dv_b += C_b * rho;
    rho_b += P_b * th + rUn_b * Un;
    th_b += P_b * rho;
    Un_b += rUn_b * rho;
    PrimGrad pgb;
    for (int d = 0; d < 3; ++d) {
        const double grb = C_b * s.U[d] + th * gPb[d];
        Bb[0][d] += scale * grb;
        pgb.gt[d] = tn_b * n[d] + Dt_b * s.U[d] + rho * gPb[d];
        Ub[d] += Dt_b * pg.gt[d] + C_b * gr[d] + DUb[0] * pg.gU[0][d] + DUb[1] * pg.gU[1][d] + DUb[2] * pg.gU[2][d] +
                 Un_b * n[d] + 2.0 * U2_b * s.U[d];
        for (int j = 0; j < 3; ++j) pgb.gU[j][d] = DUb[j] * s.U[d] + Ujb[j] * n[d] + n[j] * gUnb[d] + (j == d ? dv_b : 0.0);
    }
    th_b += dot(gPb, gr);
    rho_b += dot(gPb, pg.gt);
    for (int d = 0; d < 3; ++d) a.U[d] += Ub[d];
    a.th += th_b;
    a.rho += rho_b;
    a.ir += ir_b;
    prim_grad_adj(s, B, scale, pg, pgb, gas, Bb, a);
}

}  // namespace wm
}  // namespace ugkwp
