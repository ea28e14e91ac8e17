// Adjoint of the wave part of the step with the particle part frozen (Sec. 2.1,
// 2.3, 2.4 (d), (e)).
//
// Frozen map: with the recorded time steps dt^n, particle densities rho^p_n
// (rho^h = rho - rho^p) and particle fluxes pf^n of K real steps,
//   W^{n+1}_i = W^n_i - sum_f (+/-) F_f(W^n; theta) |S_f| / |Omega_i| + pf^n_i / |Omega_i|,
// and a wall functional J = sum_n sum_{listed boundary faces} F_f[c] |S_f|
// (c = 1: x momentum delivered to the walls, drag; c = 4: energy, wall heat
// flux).  theta = (rho_inf, U_inf, T_w) parameterises every far-field state
// equal to the first one (density, speed along its direction, its own
// temperature) and the temperature of the listed diffuse walls.
//
// Reverse sweep: lambda^K = 0 and for n = K-1..0
//   g_f      = -|S_f|/|Omega_o| lambda^{n+1}_o + |S_f|/|Omega_nb| lambda^{n+1}_nb
//              + |S_f| e_c  (listed boundary faces),
//   lambda^n = lambda^{n+1} + sum_f (dF_f/dW^n)^T g_f,
//   dJ/dtheta += sum_f (dF_f/dtheta)^T g_f.
// Face states are recomputed from the checkpointed W^n; each face's products
// with its local Jacobians come from the hand-written reverse pass of the face's
// flux (wave_math.cuh), one evaluation for all inputs, where forward-mode duals
// took two (first order) or ten (second order) evaluations of five directions
// each.  A face writes the products of each side as one row; a cell gathers its
// faces' rows in their fixed order.
//
// Bound by the binary64 pipe.  The face kernel per step: first order, channel of
// 40,500 tets, 0.19 ms (duals: 1.97 ms); second order, 20,736 tets, 0.32 ms
// (duals: 21.8 ms).  The sums over faces run over the boundary faces alone (0.006
// ms; over all faces 0.16-0.47 ms).
#include "recon.cuh"
#include "ugkwp_internal.hpp"

namespace ugkwp {

namespace {

__device__ __forceinline__ bool listed_face(const DevMesh& m, const AdjParams& ap, int f) {
    const int nb = m.f_nbr[f];
    return nb < 0 && ap.b[m.bf_tag[-1 - nb]].listed;
}

// far-field state of tag b at theta (or as given)
__device__ __forceinline__ void farfield_state(const DevParams& P, const AdjParams& ap, int tag, const double* th,
                                               double* Win) {
    const DevBc& bc = P.bc[tag];
    const AdjBc& ab = ap.b[tag];
    if (ab.param_ff) {
        Win[0] = th[0];
        for (int d = 0; d < 3; ++d) Win[1 + d] = th[0] * th[1] * ab.e[d];
        Win[4] = th[0] * (0.5 * th[1] * th[1] + 1.5 * ab.RT);
    } else {
        for (int q = 0; q < 5; ++q) Win[q] = bc.W_in[q];
    }
}

// The Maxwellian re-emitted by a diffuse wall (unit density).
__device__ __forceinline__ wm::Prim wall_state(const DevBc& bc, double R, double T_w) {
    wm::Prim w;
    w.rho = w.ir = 1.0;
    for (int d = 0; d < 3; ++d) w.U[d] = bc.U_w[d];
    w.U2 = wm::dot(w.U, w.U);
    w.th = w.p = R * T_w;
    return w;
}

// First-order flux of a face from the owner's state (and the neighbour's, or the
// boundary condition at theta).
__device__ __forceinline__ void face_o1(const DevMesh& m, const DevParams& P, const AdjParams& ap, int nb,
                                        const wm::Prim& L, double rhL, const double* WR, double rpR, const double* th,
                                        const double* n, double dt, const wm::FaceGas& fg, double F[5]) {
    if (nb >= 0) {
        wm::flux_o1(L, rhL, wm::prim_of(WR, fg.gas), WR[0] - rpR, false, false, n, dt, fg, F);
        return;
    }
    const int tag = m.bf_tag[-1 - nb];
    const DevBc& bc = P.bc[tag];
    if (bc.type == UGKWP_BC_DIFFUSE_WALL) {
        const wm::QC1 c = wm::time_coeffs(dt, wm::face_tau0(L, fg));
        const double c1 = c.q1 * L.rho + c.a4 * rhL;
        const wm::PrimGrad none{};
        const double z[3] = {0.0, 0.0, 0.0};
        const wm::Prim w = wall_state(bc, P.R, ap.b[tag].param_wall ? th[2] : bc.T_w);
        const wm::SideFlux a = wm::side_flux<false>(L, none, 0.0, z, n, 1.0, fg.gas);
        const wm::SideFlux b = wm::side_flux<false>(w, none, 0.0, z, n, -1.0, fg.gas);
        const double r = a.G[0] / b.G[0];
        F[0] = 0.0;
        for (int k = 1; k < 5; ++k) F[k] = c1 * (a.G[k] - r * b.G[k]);
        return;
    }
    wm::Prim R = L;
    double rhR = rhL;
    if (bc.type == UGKWP_BC_SPECULAR) {
        const double Un = wm::dot(L.U, n);
        for (int d = 0; d < 3; ++d) R.U[d] = L.U[d] - 2.0 * Un * n[d];
    } else {
        if (bc.type == UGKWP_BC_FARFIELD) {
            double Win[5];
            farfield_state(P, ap, tag, th, Win);
            R = wm::prim_of(Win, fg.gas);
        }
        rhR = R.rho;
    }
    wm::flux_o1(L, rhL, R, rhR, bc.type != UGKWP_BC_SPECULAR, false, n, dt, fg, F);
    if (bc.type == UGKWP_BC_SPECULAR) {
        const double fn = wm::dot(F + 1, n);
        F[0] = 0.0;
        F[4] = 0.0;
        for (int d = 0; d < 3; ++d) F[1 + d] = fn * n[d];
    }
}

// The adjoint of face_o1 along g: Lb, Rb (of the conservative states; of the
// neighbour's only for an interior face) and thb of theta (boundary faces), all
// added to.
__device__ __forceinline__ void face_o1_adj(const DevMesh& m, const DevParams& P, const AdjParams& ap, int nb,
                                            const wm::Prim& L, double rhL, const double* WR, double rpR,
                                            const double* th, const double* n, double dt, const wm::FaceGas& fg,
                                            const double* g, double* Lb, double* Rb, double* thb) {
    wm::PrimAdj aL = wm::prim_adj_zero(), aR = wm::prim_adj_zero();
    double rhLb = 0.0, rhRb = 0.0;
    if (nb >= 0) {
        const wm::Prim R = wm::prim_of(WR, fg.gas);
        wm::flux_o1_adj(L, rhL, R, WR[0] - rpR, false, n, dt, fg, g, aL, rhLb, aR, rhRb);
        aR.rho += rhRb;  // rho^h = rho - rho^p
        wm::prim_adj(R, aR, fg.gas, Rb);
    } else {
        const int tag = m.bf_tag[-1 - nb];
        const DevBc& bc = P.bc[tag];
        const AdjBc& ab = ap.b[tag];
        if (bc.type == UGKWP_BC_DIFFUSE_WALL) {
            // F_k = c1 (a_k - r b_k), r = a_0 / b_0, c1 = q1 rho + a4 rho^h (F_0 = 0)
            const double tau = wm::face_tau0(L, fg);
            const wm::QC1 c = wm::time_coeffs(dt, tau);
            const double c1 = c.q1 * L.rho + c.a4 * rhL;
            const wm::PrimGrad none{};
            const double z[3] = {0.0, 0.0, 0.0};
            const wm::Prim w = wall_state(bc, P.R, ab.param_wall ? th[2] : bc.T_w);
            const wm::SideFlux a = wm::side_flux<false>(L, none, 0.0, z, n, 1.0, fg.gas);
            const wm::SideFlux b = wm::side_flux<false>(w, none, 0.0, z, n, -1.0, fg.gas);
            const double ib = 1.0 / b.G[0], r = a.G[0] * ib;
            double c1b = 0.0, rb = 0.0, ab_[5], bb[5], Hb[5] = {}, Sb[5] = {};
            for (int k = 1; k < 5; ++k) {
                c1b += g[k] * (a.G[k] - r * b.G[k]);
                rb -= c1 * g[k] * b.G[k];
                ab_[k] = c1 * g[k];
                bb[k] = -c1 * r * g[k];
            }
            ab_[0] = rb * ib;
            bb[0] = -rb * r * ib;
            double u1 = 0.0, u3[3] = {0.0, 0.0, 0.0};
            wm::PrimGrad ub{};
            wm::side_flux_adj<false>(L, none, 0.0, z, n, 1.0, fg.gas, Hb, ab_, Sb, aL, ub, u1, u3);
            aL.rho += c1b * c.q1;
            rhLb += c1b * c.a4;
            const double taub = wm::time_coeffs_adj1(c, dt, tau, c1b * L.rho, 0.0, c1b * rhL);
            aL.th += taub * fg.omega * tau / L.th;
            aL.p -= taub * tau / L.p;
            if (ab.param_wall) {
                wm::side_flux_adj<false>(w, none, 0.0, z, n, -1.0, fg.gas, Hb, bb, Sb, aR, ub, u1, u3);
                thb[2] += aR.th * P.R;
            }
        } else if (bc.type == UGKWP_BC_SPECULAR) {
            wm::Prim R = L;
            const double Un = wm::dot(L.U, n), gn = g[1] * n[0] + g[2] * n[1] + g[3] * n[2];
            for (int d = 0; d < 3; ++d) R.U[d] = L.U[d] - 2.0 * Un * n[d];
            const double gs[5] = {0.0, gn * n[0], gn * n[1], gn * n[2], 0.0};
            wm::flux_o1_adj(L, rhL, R, rhL, false, n, dt, fg, gs, aL, rhLb, aR, rhRb);
            const double rn = wm::dot(aR.U, n);
            for (int d = 0; d < 3; ++d) aL.U[d] += aR.U[d] - 2.0 * rn * n[d];
            aL.th += aR.th;
            aL.rho += aR.rho;
            aL.p += aR.p;
            rhLb += rhRb;
        } else {
            wm::Prim R = L;
            double Win[5];
            if (bc.type == UGKWP_BC_FARFIELD) {
                farfield_state(P, ap, tag, th, Win);
                R = wm::prim_of(Win, fg.gas);
            }
            wm::flux_o1_adj(L, rhL, R, R.rho, true, n, dt, fg, g, aL, rhLb, aR, rhRb);
            aR.rho += rhRb;  // all of the ghost is hydrodynamic
            if (bc.type == UGKWP_BC_OUTFLOW) {
                for (int d = 0; d < 3; ++d) aL.U[d] += aR.U[d];
                aL.th += aR.th;
                aL.rho += aR.rho;
                aL.p += aR.p;
            } else if (ab.param_ff) {
                double b[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
                wm::prim_adj(R, aR, fg.gas, b);
                const double be = b[1] * ab.e[0] + b[2] * ab.e[1] + b[3] * ab.e[2];
                thb[0] += b[0] + th[1] * be + b[4] * (0.5 * th[1] * th[1] + 1.5 * ab.RT);
                thb[1] += th[0] * (be + b[4] * th[1]);
            }
        }
    }
    aL.rho += rhLb;
    wm::prim_adj(L, aL, fg.gas, Lb);
}

// Limited least-squares gradients of W and rho^h = rho - rho^p as rows (second
// order); with record the limiter values are stored in phi [6][nc], otherwise
// phi is used as given (the limiter frozen at theta).  Far-field ghosts hold the
// state at theta.
__global__ void __launch_bounds__(128) k_adj_grad(DevMesh m, DevParams P, AdjParams ap, const double* W,
                                                  const double* rho_p, const double* theta, double* phi, int record,
                                                  double* rec) {
    const int nc = m.nc;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 3 * nc) return;
    const int pair = t >= 2 * nc ? 2 : t >= nc ? 1 : 0, i = t - pair * nc;
    const double th[3] = {theta[0], theta[1], theta[2]};
    limited_pair(
        m, P, i, pair, [&](int q, int j) { return q < 5 ? W[(size_t)q * nc + j] : W[j] - rho_p[j]; },
        [&](int tag, int q) {
            double Win[5];
            farfield_state(P, ap, tag, th, Win);
            return Win[q < 5 ? q : 0];
        },
        [&](int q, double ph) {
            double& v = phi[(size_t)q * nc + i];
            if (record) v = ph;
            return record ? ph : v;
        },
        rec + (size_t)REC_N * i);
}

// ---- forward: fluxes and the functional's terms (boundary faces) at theta
template <bool O2>
__global__ void __launch_bounds__(128) k_adj_fwd_flux(DevMesh m, DevParams P, AdjParams ap, const double* W,
                                                      const double* rho_p, const double* dt_n, const double* theta,
                                                      const double* rec, double* F, double* jf) {
    const int nc = m.nc, nf = m.nf;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nf) return;
    const double dt = dt_n[0];
    const int f = m.face_order[t];  // interior faces first
    const double n[3] = {m.f_n[f], m.f_n[nf + f], m.f_n[2 * nf + f]};
    const int o = m.f_own[f], nb = m.f_nbr[f];
    double Fv[5];
    if (O2 && nb >= 0) {
        interior_flux_o2(m, rec, P, f, o, nb, n, dt, Fv);
    } else {
        const double th[3] = {theta[0], theta[1], theta[2]};
        const wm::FaceGas fg = face_gas(P);
        double WL[5], WR[5];
        for (int q = 0; q < 5; ++q) {
            WL[q] = W[(size_t)q * nc + o];
            WR[q] = nb >= 0 ? W[(size_t)q * nc + nb] : 0.0;
        }
        face_o1(m, P, ap, nb, wm::prim_of(WL, fg.gas), WL[0] - rho_p[o], WR, nb >= 0 ? rho_p[nb] : 0.0, th, n, dt, fg, Fv);
    }
    for (int q = 0; q < 5; ++q) F[(size_t)q * nf + f] = Fv[q];
    if (nb < 0) jf[-1 - nb] = listed_face(m, ap, f) ? Fv[ap.comp] * m.f_area[f] : 0.0;
}

__global__ void k_adj_update(DevMesh m, const double* W, const double* F, const double* pf, double* Wn) {
    const int nc = m.nc, nf = m.nf;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nc) return;
    const int own = m.cfs[i];
    const double ivol = m.ivol[i];
    int f[4];
    double s[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        f[k] = m.cf[k * nc + i];
        s[k] = ((own >> k) & 1) ? m.f_area[f[k]] : -m.f_area[f[k]];
    }
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < 4; ++k) acc += F[(size_t)q * nf + f[k]] * s[k];
        Wn[(size_t)q * nc + i] = (W[(size_t)q * nc + i] - acc * ivol) + pf[(size_t)q * nc + i] * ivol;
    }
}

// out[c] = sum_j x[c n + j] (+ y[c n + j]), c < ncomp: one block per component,
// fixed order.  The summands are one per boundary face, so that a block of 256
// threads is enough.
__global__ void __launch_bounds__(256) k_adj_sum(const double* x, const double* y, int n, double* out) {
    __shared__ double sh[256];
    const size_t at = (size_t)blockIdx.x * n;
    double a = 0.0;
    for (int j = threadIdx.x; j < n; j += 256) a += y ? x[at + j] + y[at + j] : x[at + j];
    sh[threadIdx.x] = a;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = sh[0];
}

// The reverse pass of an interior face at second order: the products of g with
// the Jacobians with respect to both cells' rows, written as rows of the same
// shape (place 5 unused: rho^h's product is added to rho's).
__device__ __forceinline__ void store_row(double* out, const double* Wb, const double gb[5][3], const double* ghb) {
    double v[REC_N];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        v[q] = Wb[q];
        for (int d = 0; d < 3; ++d) v[6 + 3 * q + d] = gb[q][d];
    }
    v[5] = 0.0;
    for (int d = 0; d < 3; ++d) v[21 + d] = ghb[d];
    double2* o = reinterpret_cast<double2*>(out);
#pragma unroll
    for (int j = 0; j < REC_N / 2; ++j) o[j] = make_double2(v[2 * j], v[2 * j + 1]);
}

__device__ __forceinline__ void side_o2_adj(const double* rec, int c, const double* dx, const double* n, double sgn,
                                            const wm::Gas& gas, const double* g, const double* W0b, double c4,
                                            double c5, double gG, double WH, double p_b, const double Bb[5][3],
                                            double* out) {
    const Row r = load_row(rec, c, dx);
    const wm::Prim s = wm::prim_of(r.W, gas);
    const wm::PrimGrad pg = wm::prim_grad(s, r.g, 1.0, gas);
    double Hb[5], Gb[5], Sb[5];
    for (int k = 0; k < 5; ++k) {
        Hb[k] = s.rho * W0b[k];
        Gb[k] = c4 * r.rh * g[k];
        Sb[k] = c5 * g[k];
    }
    wm::PrimAdj a = wm::prim_adj_zero();
    wm::PrimGrad pgb{};
    double rhb = c4 * gG, ghb[3] = {0.0, 0.0, 0.0}, gb[5][3], Wb[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int q = 0; q < 5; ++q)
        for (int d = 0; d < 3; ++d) gb[q][d] = Bb[q][d];
    a.rho = WH;
    a.p = p_b;
    wm::side_flux_adj<true>(s, pg, r.rh, r.gh, n, sgn, gas, Hb, Gb, Sb, a, pgb, rhb, ghb);
    wm::prim_grad_adj(s, r.g, 1.0, pg, pgb, gas, gb, a);
    wm::prim_adj(s, a, gas, Wb);
    // the reconstruction: W = W_c + grad W dx, rho^h = rho^h_c + grad rho^h dx;
    // a side that fell back to its cell values does not depend on its slopes
    if (r.o2) {
        for (int d = 0; d < 3; ++d) {
            for (int q = 0; q < 5; ++q) gb[q][d] += Wb[q] * dx[d];
            ghb[d] += rhb * dx[d];
        }
    } else {
        for (int d = 0; d < 3; ++d) {
            for (int q = 0; q < 5; ++q) gb[q][d] = 0.0;
            ghb[d] = 0.0;
        }
    }
    Wb[0] += rhb;  // rho^h = rho - rho^p
    store_row(out, Wb, gb, ghb);
}

__device__ __forceinline__ void interior_o2_adj(const DevMesh& m, const double* rec, const DevParams& p, int f, int o,
                                                int nb, const double* n, double dt, const double* g, double* out) {
    const int nf = m.nf;
    double dx[6];
#pragma unroll
    for (int d = 0; d < 6; ++d) dx[d] = m.f_dx[(size_t)d * nf + f];
    const wm::FaceGas fg = face_gas(p);
    const wm::Gas& gas = fg.gas;
    double B[5][3], W0[5], H[2][5], gG[2], c4b = 0.0, c5b = 0.0, ps[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const Row r = load_row(rec, e == 0 ? o : nb, dx + 3 * e);
        const wm::Prim c = wm::prim_of(r.W, gas);
        const wm::SideFlux h =
            wm::side_flux<true>(c, wm::prim_grad(c, r.g, 1.0, gas), r.rh, r.gh, n, e == 0 ? 1.0 : -1.0, gas);
        double t = 0.0;
        for (int k = 0; k < 5; ++k) {
            W0[k] = e == 0 ? c.rho * h.H[k] : W0[k] + c.rho * h.H[k];
            H[e][k] = h.H[k];
            t += g[k] * h.G[k];
            c5b += g[k] * h.S[k];
            for (int d = 0; d < 3; ++d) B[k][d] = e == 0 ? r.g[k][d] : B[k][d] + r.g[k][d];
        }
        gG[e] = t;
        c4b += r.rh * t;
        ps[e] = c.p;
    }
    const wm::Prim c0 = wm::prim_of(W0, gas);
    const double tau0 = wm::face_tau0(c0, fg);
    double tau = tau0, rD = 0.0;
    const double D = ps[0] - ps[1], iS = 1.0 / fabs(ps[0] + ps[1]);
    if (fg.C2 > 0.0) {
        rD = fabs(D) * iS;
        tau += fg.C2 * rD * dt;
    }
    const wm::QC qc = wm::time_coeffs_all(dt, tau);
    double qb[3] = {0.0, 0.0, 0.0}, Bb[5][3] = {}, W0b[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, Eb = 0.0;
    wm::PrimAdj a = wm::prim_adj_zero();
    wm::equilibrium_flux_adj(W0, c0, B, 0.5, n, qc, p.pr_fix, gas, g, a, Eb, Bb, qb);
    const double taub = wm::time_coeffs_adj(qc, dt, tau, qb[0], qb[1], qb[2], 0.0, c4b, c5b);
    a.th += taub * fg.omega * tau0 / c0.th;
    a.p -= taub * tau0 / c0.p;
    wm::prim_adj(c0, a, gas, W0b);
    W0b[4] += Eb;
    double pb[2] = {0.0, 0.0};
    if (fg.C2 > 0.0) {
        const double t = taub * fg.C2 * dt * iS, sg = D > 0.0 ? 1.0 : D < 0.0 ? -1.0 : 0.0;
        pb[0] = t * (sg - rD);
        pb[1] = -t * (sg + rD);
    }
#pragma unroll 1
    for (int e = 0; e < 2; ++e) {
        double WH = 0.0;
        for (int k = 0; k < 5; ++k) WH += W0b[k] * (e == 0 ? H[0][k] : H[1][k]);
        side_o2_adj(rec, e == 0 ? o : nb, e == 0 ? dx : dx + 3, n, e == 0 ? 1.0 : -1.0, gas, g, W0b, qc.a4, qc.a5,
                    e == 0 ? gG[0] : gG[1], WH, e == 0 ? pb[0] : pb[1], Bb, out + e * REC_N);
    }
}

// Row of a side of a face at first order (the fifth value pads it to 48 bytes).
constexpr int ROW1 = 6;

// ---- reverse: per face, g_f and its products with the local Jacobians, as one
// row per side (second order: REC_N values, first order: ROW1) at
// fb[(2 f + side) row]; the products with theta of a boundary face at
// thbar[3][nbf].
template <bool O2>
__global__ void __launch_bounds__(128) k_adj_face(DevMesh m, DevParams P, AdjParams ap, const double* W,
                                                  const double* rho_p, const double* dt_n, const double* theta,
                                                  const double* rec, const double* lam_next, double* fb,
                                                  double* thbar) {
    constexpr int ROW = O2 ? REC_N : ROW1;
    const int nc = m.nc, nf = m.nf;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nf) return;
    const double dt = dt_n[0];
    const int f = m.face_order[t];  // interior faces first
    const int o = m.f_own[f], nb = m.f_nbr[f];
    const double n[3] = {m.f_n[f], m.f_n[nf + f], m.f_n[2 * nf + f]};
    const double area = m.f_area[f];
    const double so = area * m.ivol[o], sn = nb >= 0 ? area * m.ivol[nb] : 0.0;
    double g[5];
    for (int q = 0; q < 5; ++q) {
        g[q] = -so * lam_next[(size_t)q * nc + o];
        if (nb >= 0) g[q] += sn * lam_next[(size_t)q * nc + nb];
    }
    if (listed_face(m, ap, f)) g[ap.comp] += area;
    double* out = fb + (size_t)(2 * ROW) * f;
    if (O2 && nb >= 0) {
        interior_o2_adj(m, rec, P, f, o, nb, n, dt, g, out);
        return;
    }
    const double th[3] = {theta[0], theta[1], theta[2]};
    const wm::FaceGas fg = face_gas(P);
    double WL[5], WR[5], Lb[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, Rb[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, tb[3] = {0.0, 0.0, 0.0};
    for (int q = 0; q < 5; ++q) {
        WL[q] = W[(size_t)q * nc + o];
        WR[q] = nb >= 0 ? W[(size_t)q * nc + nb] : 0.0;
    }
    face_o1_adj(m, P, ap, nb, wm::prim_of(WL, fg.gas), WL[0] - rho_p[o], WR, nb >= 0 ? rho_p[nb] : 0.0, th, n, dt, fg, g,
                Lb, Rb, tb);
    if (O2) {  // a boundary face at second order: first order, no products with slopes
        const double z5[5][3] = {}, z3[3] = {0.0, 0.0, 0.0};
        store_row(out, Lb, z5, z3);
    } else {
        double2* r = reinterpret_cast<double2*>(out);
        r[0] = make_double2(Lb[0], Lb[1]);
        r[1] = make_double2(Lb[2], Lb[3]);
        r[2] = make_double2(Lb[4], 0.0);
        if (nb >= 0) {
            r[3] = make_double2(Rb[0], Rb[1]);
            r[4] = make_double2(Rb[2], Rb[3]);
            r[5] = make_double2(Rb[4], 0.0);
        }
    }
    if (nb < 0)
        for (int k = 0; k < 3; ++k) thbar[(size_t)k * m.nbf - 1 - nb] = tb[k];
}

// lambda^n = lambda^{n+1} + the products of the cell's faces with its W; second
// order: also gg = phi * (the sum of the products with its limited gradients)
// as a row [18] per cell, 3q + d (q = 5: rho^h).
template <bool O2>
__global__ void __launch_bounds__(128) k_adj_gather(DevMesh m, const double* lam_next, const double* fb,
                                                    const double* phi, double* lam, double* gg) {
    constexpr int ROW = O2 ? REC_N : ROW1;
    const int nc = m.nc;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nc) return;
    const int own = m.cfs[i];
    double a[ROW];
#pragma unroll
    for (int j = 0; j < ROW; ++j) a[j] = j < 5 ? lam_next[(size_t)j * nc + i] : 0.0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int f = m.cf[k * nc + i];
        const double2* r = reinterpret_cast<const double2*>(fb + ((size_t)2 * f + (((own >> k) & 1) ? 0 : 1)) * ROW);
#pragma unroll
        for (int j = 0; j < ROW / 2; ++j) {
            const double2 v = r[j];
            a[2 * j] += v.x;
            a[2 * j + 1] += v.y;
        }
    }
#pragma unroll
    for (int q = 0; q < 5; ++q) lam[(size_t)q * nc + i] = a[q];
    if constexpr (O2) {
        double2* o = reinterpret_cast<double2*>(gg + (size_t)18 * i);
        double ph[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) ph[q] = phi[(size_t)q * nc + i];
#pragma unroll
        for (int j = 0; j < 9; ++j) o[j] = make_double2(ph[2 * j / 3] * a[6 + 2 * j], ph[(2 * j + 1) / 3] * a[7 + 2 * j]);
    }
}

// Second order: the gradients' dependence on the cells' W, added to lambda^n:
// gradient_c,q = phi sum_k c_k (val_k - self_q) is linear in the cell's own value
// (-c_k), in its neighbours' values (+c_k at the neighbour's side) and in the
// ghost values (specular: mirrored momentum; far field: the state at theta, whose
// theta products go to thc [3][nbf]).
__global__ void __launch_bounds__(128) k_adj_cell(DevMesh m, DevParams P, AdjParams ap, const double* theta,
                                                  const double* gg, double* lam, double* thc) {
    const int nc = m.nc, nbf = m.nbf;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nc) return;
    const int4 nbv = m.trk_f ? m.trk_f[i].nb : m.trk_d[i].nb;
    const int code[4] = {nbv.x, nbv.y, nbv.z, nbv.w};
    double l[5], own[18];
    for (int q = 0; q < 5; ++q) l[q] = lam[(size_t)q * nc + i];
    {
        const double2* r = reinterpret_cast<const double2*>(gg + (size_t)18 * i);
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            const double2 v = r[j];
            own[2 * j] = v.x;
            own[2 * j + 1] = v.y;
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        double c[3];
        for (int d = 0; d < 3; ++d) c[d] = m.lsq_c[(size_t)(3 * k + d) * nc + i];
        if (code[k] >= 0) {
            const int other = code[k] >> 2, ko = code[k] & 3;
            double co[3], t[18];
            for (int d = 0; d < 3; ++d) co[d] = m.lsq_c[(size_t)(3 * ko + d) * nc + other];
            const double2* r = reinterpret_cast<const double2*>(gg + (size_t)18 * other);
#pragma unroll
            for (int j = 0; j < 9; ++j) {
                const double2 v = r[j];
                t[2 * j] = v.x;
                t[2 * j + 1] = v.y;
            }
#pragma unroll
            for (int q = 0; q < 6; ++q) l[q < 5 ? q : 0] += wm::dot(t + 3 * q, co) - wm::dot(own + 3 * q, c);
            continue;
        }
        const int b = -1 - code[k];
        const int tag = m.bf_tag[b];
        const int type = P.bc[tag].type;
        double tc[2] = {0.0, 0.0};
        if (type == UGKWP_BC_SPECULAR) {
            double nn[3], sn = 0.0;
            for (int d = 0; d < 3; ++d) nn[d] = m.bf_n[(size_t)d * nbf + b];
            for (int q = 1; q < 4; ++q) sn += wm::dot(own + 3 * q, c) * nn[q - 1];
            for (int d = 0; d < 3; ++d) l[1 + d] -= 2.0 * sn * nn[d];
        } else if (type == UGKWP_BC_FARFIELD) {
            const AdjBc& ab = ap.b[tag];
            const double th0 = theta[0], th1 = theta[1];
            for (int q = 0; q < 6; ++q) {
                const double s = wm::dot(own + 3 * q, c);
                const int qq = q < 5 ? q : 0;  // rho^h = rho - rho^p
                l[qq] -= s;
                if (!ab.param_ff) continue;
                // d W_in / d theta: rho = th0, m = th0 th1 e, E = th0 (th1^2/2 + 3/2 RT)
                double d0, d1;
                if (qq == 0) { d0 = 1.0; d1 = 0.0; }
                else if (qq <= 3) { d0 = th1 * ab.e[qq - 1]; d1 = th0 * ab.e[qq - 1]; }
                else { d0 = 0.5 * th1 * th1 + 1.5 * ab.RT; d1 = th0 * th1; }
                tc[0] += s * d0;
                tc[1] += s * d1;
            }
        }
        thc[b] = tc[0];
        thc[(size_t)nbf + b] = tc[1];
        thc[2 * (size_t)nbf + b] = 0.0;
    }
    for (int q = 0; q < 5; ++q) lam[(size_t)q * nc + i] = l[q];
}

// recorded particle data of the step just taken
__global__ void k_adj_record(DevMesh m, DevState s, DevParams P, double* rho_p, double* pf) {
    const int nc = m.nc;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nc) return;
    rho_p[i] = s.prim[i] - s.rhoh[i];
    for (int q = 0; q < 5; ++q) pf[(size_t)q * nc + i] = (double)s.pflux[(size_t)q * nc + i] * P.qscale[q];
}

}  // namespace

size_t adjoint_face_row(int order) { return order == 2 ? REC_N : ROW1; }

void launch_adj_record(const DevMesh& m, const DevState& s, const DevParams& p, double* rho_p, double* pf,
                       cudaStream_t st) {
    k_adj_record<<<(m.nc + 255) / 256, 256, 0, st>>>(m, s, p, rho_p, pf);
}

// Blocks of 64: the launches are a few waves of a binary64-bound kernel, and the
// smaller block fills the last one better (second order, channel of 21,168 tets,
// 4 steps: 3.62 ms with 128, 3.55 with 64 and with 32; first order, 40,500 tets,
// 10 steps: 7.06, 7.05, 7.14).
void launch_adj_forward(const DevMesh& m, const DevParams& p, const AdjParams& ap, const double* W, const double* rho_p,
                        const double* pf, const double* dt, const double* theta, const AdjO2& o2, double* F, double* jf,
                        double* Jn, double* Wn, cudaStream_t st) {
    const int gf = (m.nf + 63) / 64, gc = (m.nc + 63) / 64;
    if (p.order == 2) {
        k_adj_grad<<<(3 * m.nc + 63) / 64, 64, 0, st>>>(m, p, ap, W, rho_p, theta, o2.phi, 1, o2.rec);
        k_adj_fwd_flux<true><<<gf, 64, 0, st>>>(m, p, ap, W, rho_p, dt, theta, o2.rec, F, jf);
    } else {
        k_adj_fwd_flux<false><<<gf, 64, 0, st>>>(m, p, ap, W, rho_p, dt, theta, nullptr, F, jf);
    }
    k_adj_sum<<<1, 256, 0, st>>>(jf, nullptr, m.nbf, Jn);
    k_adj_update<<<gc, 64, 0, st>>>(m, W, F, pf, Wn);
}

void launch_adj_reverse(const DevMesh& m, const DevParams& p, const AdjParams& ap, const double* W,
                        const double* rho_p, const double* dt, const double* theta, const AdjO2& o2, const double* lam_next,
                        double* lam, double* fb, double* thbar, double* th_out, cudaStream_t st) {
    const int gf = (m.nf + 63) / 64, gc = (m.nc + 63) / 64;
    if (p.order == 2) {
        k_adj_grad<<<(3 * m.nc + 63) / 64, 64, 0, st>>>(m, p, ap, W, rho_p, theta, o2.phi, 0, o2.rec);
        k_adj_face<true><<<gf, 64, 0, st>>>(m, p, ap, W, rho_p, dt, theta, o2.rec, lam_next, fb, thbar);
        k_adj_gather<true><<<gc, 64, 0, st>>>(m, lam_next, fb, o2.phi, lam, o2.gg);
        k_adj_cell<<<gc, 64, 0, st>>>(m, p, ap, theta, o2.gg, lam, o2.thc);
    } else {
        k_adj_face<false><<<gf, 64, 0, st>>>(m, p, ap, W, rho_p, dt, theta, nullptr, lam_next, fb, thbar);
        k_adj_gather<false><<<gc, 64, 0, st>>>(m, lam_next, fb, nullptr, lam, nullptr);
    }
    k_adj_sum<<<3, 256, 0, st>>>(thbar, p.order == 2 ? o2.thc : nullptr, m.nbf, th_out);
}

}  // namespace ugkwp
