// Device code that the step's wave kernels and the adjoint's share: the limited
// least-squares gradients of a cell and the wave flux of an interior face from
// the cells' rows.
#pragma once
#include "ugkwp_internal.hpp"
#include "wave_math.cuh"

namespace ugkwp {

__device__ __forceinline__ wm::FaceGas face_gas(const DevParams& p) {
    return wm::FaceGas{wm::gas_of(p.K), p.mu_ref, p.omega, 1.0 / (p.R * p.T_ref), p.C2};
}

// Limited gradients of two of the six quantities (0..4: W, 5: rho^h) of cell i,
// quantities 2 pair and 2 pair + 1, written with the values themselves into the
// cell's row (REC_N values, see DevState::rec), which the flux kernel reads whole
// for each side of a face.  One thread per pair and cell: a thread's two
// quantities share the reconstruction weights, the centroid-to-face vectors and
// the neighbour codes and fill whole 16-byte pieces of the row, and three
// threads per cell keep enough of them in flight on small meshes.
// Venkatakrishnan's function of the allowed difference d1 and the extrapolated
// difference d2 (same sign, d2 != 0), divided through by d2:
// num/den = (A + 2 s) / (A + s + 2 d2^2), A = d1^2 + eps^2, s = d1 d2 >= 0.
// The extrema of the differences are taken on their bit patterns (integer
// pipes): among non-negative doubles the larger one has the larger signed bit
// pattern, among negative ones the smaller one the larger unsigned pattern.
// Bound by the binary64 pipe (~75 operations per quantity).
// val(q, j): quantity q of cell j; far(tag, q): of the far-field state of a
// boundary condition; lim(q, phi): the limiter value to use, given the computed
// one (an adjoint pass records or replaces it).
template <class Val, class Far, class Lim>
__device__ __forceinline__ void limited_pair(const DevMesh& m, const DevParams& p, int i, int pair, Val&& val, Far&& far, Lim&& lim,
                                            double* row_of_i) {
    const int nc = m.nc;
    const int4 nbv = m.trk_f ? m.trk_f[i].nb : m.trk_d[i].nb;
    const int code[4] = {nbv.x, nbv.y, nbv.z, nbv.w};
    double c[12], x[12];
#pragma unroll
    for (int j = 0; j < 12; ++j) {
        c[j] = m.lsq_c[(size_t)j * nc + i];
        x[j] = m.lsq_dxf[(size_t)j * nc + i];
    }
    const double eps2 = m.eps2[i];
    double2* row = reinterpret_cast<double2*>(row_of_i);
    double out[4];  // values waiting for a whole pair
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int q = 2 * pair + e;
        const double self = val(q, i);
        double v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (code[k] >= 0) {
                v[k] = val(q, code[k] >> 2) - self;
            } else {
                const int b = -1 - code[k];
                const int tag = m.bf_tag[b];
                const int type = p.bc[tag].type;
                v[k] = 0.0;
                if (type == UGKWP_BC_SPECULAR && q >= 1 && q <= 3) {
                    const int nbf = m.nbf;
                    double n[3];
                    for (int d = 0; d < 3; ++d) n[d] = m.bf_n[(size_t)d * nbf + b];
                    const double mn = val(1, i) * n[0] + val(2, i) * n[1] + val(3, i) * n[2];
                    v[k] = -2.0 * mn * n[q - 1];
                } else if (type == UGKWP_BC_FARFIELD) {
                    v[k] = far(tag, q) - self;
                }
            }
        }
        double g[3] = {0.0, 0.0, 0.0};
        long long hi = 0;
        unsigned long long lo = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            for (int d = 0; d < 3; ++d) g[d] += c[3 * k + d] * v[k];
            const long long bits = __double_as_longlong(v[k]);
            hi = bits > hi ? bits : hi;
            lo = (unsigned long long)bits > lo ? (unsigned long long)bits : lo;
        }
        const double dmax = __longlong_as_double(hi);
        const double dmin = (long long)lo < 0 ? __longlong_as_double((long long)lo) : 0.0;
        const double Amax = dmax * dmax + eps2, Amin = dmin * dmin + eps2;
        // phi = min(1, min_k num_k/den_k), compared by cross products (den > 0)
        // so that only the chosen ratio is divided
        double bn = 1.0, bd = 1.0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double d2 = g[0] * x[3 * k] + g[1] * x[3 * k + 1] + g[2] * x[3 * k + 2];
            if (d2 == 0.0) continue;
            const bool up = d2 > 0.0;
            const double A = up ? Amax : Amin, sd = (up ? dmax : dmin) * d2;
            const double num = A + 2.0 * sd, den = (A + sd) + 2.0 * (d2 * d2);
            if (num * bd < bn * den) { bn = num; bd = den; }
        }
        const double phi = lim(q, bn / bd);
        // the row: W (5), rho^h, grad W [3 q + d], grad rho^h; three gradient
        // values per quantity from an even place on: two quantities make three pairs
        const double v3[3] = {phi * g[0], phi * g[1], phi * g[2]};
        if (e == 0) {
            out[0] = self;
            out[1] = v3[0]; out[2] = v3[1]; out[3] = v3[2];
        } else {
            row[pair] = make_double2(out[0], self);
            const int at = 3 + 3 * pair;
            row[at] = make_double2(out[1], out[2]);
            row[at + 1] = make_double2(out[3], v3[0]);
            row[at + 2] = make_double2(v3[1], v3[2]);
        }
    }
}

// One side of an interior face at second order: its row, reconstructed at the
// face centroid (dx from the cell's); the cell values and zero slopes if the
// reconstruction is not positive.
struct Row {
    double W[5], rh, g[5][3], gh[3];
    bool o2;  // reconstructed
};
__device__ __forceinline__ Row load_row(const double* rec, int c, const double* dx) {
    const double2* r = reinterpret_cast<const double2*>(rec + (size_t)REC_N * c);
    Row o;
    double v[REC_N];
#pragma unroll
    for (int j = 0; j < REC_N / 2; ++j) {
        const double2 t = r[j];
        v[2 * j] = t.x;
        v[2 * j + 1] = t.y;
    }
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        for (int d = 0; d < 3; ++d) o.g[q][d] = v[6 + 3 * q + d];
        o.W[q] = v[q] + wm::dot(o.g[q], dx);
    }
    for (int d = 0; d < 3; ++d) o.gh[d] = v[21 + d];
    o.rh = v[5] + wm::dot(o.gh, dx);
    // p > 0 as rho E - |rho U|^2/(2 rho) > 0, times rho > 0
    o.o2 = o.W[0] > 0.0 && o.W[4] * o.W[0] - 0.5 * wm::dot(o.W + 1, o.W + 1) > 0.0;
    if (!o.o2) {
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            o.W[q] = v[q];
            for (int d = 0; d < 3; ++d) o.g[q][d] = 0.0;
        }
        o.rh = v[5];
        for (int d = 0; d < 3; ++d) o.gh[d] = 0.0;
    }
    return o;
}

// Wave flux per unit area of interior face f at second order (wave_math.cuh).
__device__ __forceinline__ void interior_flux_o2(const DevMesh& m, const double* rec, const DevParams& p, int f, int o,
                                                 int nb, const double* n, double dt, double F[5]) {
    const int nf = m.nf;
    double dx[6];
#pragma unroll
    for (int d = 0; d < 6; ++d) dx[d] = m.f_dx[(size_t)d * nf + f];
    const wm::FaceGas fg = face_gas(p);
    const wm::Gas& gas = fg.gas;
    double B[5][3], W0[5], G[5], S[5], pL, pR;
    {
        const Row r = load_row(rec, o, dx);
        const wm::Prim c = wm::prim_of(r.W, gas);
        const wm::SideFlux h = wm::side_flux<true>(c, wm::prim_grad(c, r.g, 1.0, gas), r.rh, r.gh, n, 1.0, gas);
        for (int k = 0; k < 5; ++k) {
            W0[k] = c.rho * h.H[k];
            G[k] = r.rh * h.G[k];
            S[k] = h.S[k];
            for (int d = 0; d < 3; ++d) B[k][d] = r.g[k][d];
        }
        pL = c.p;
    }
    {
        const Row r = load_row(rec, nb, dx + 3);
        const wm::Prim c = wm::prim_of(r.W, gas);
        const wm::SideFlux h = wm::side_flux<true>(c, wm::prim_grad(c, r.g, 1.0, gas), r.rh, r.gh, n, -1.0, gas);
        for (int k = 0; k < 5; ++k) {
            W0[k] += c.rho * h.H[k];
            G[k] += r.rh * h.G[k];
            S[k] += h.S[k];
            for (int d = 0; d < 3; ++d) B[k][d] += r.g[k][d];
        }
        pR = c.p;
    }
    const wm::Prim c0 = wm::prim_of(W0, gas);
    double tau = wm::face_tau0(c0, fg);
    if (p.C2 > 0.0) tau += p.C2 * fabs(pL - pR) / fabs(pL + pR) * dt;
    const wm::QC qc = wm::time_coeffs_all(dt, tau);
    // free transport of the hydrodynamic wave, upwind, with slopes; without
    // particles (GKS step) the whole free transport, q4 and q5, is the wave's
    const double c4 = p.gks ? qc.q4 : qc.a4, c5 = p.gks ? qc.q5 : qc.a5;
    for (int k = 0; k < 5; ++k) F[k] = c4 * G[k] + c5 * S[k];
    // the mean of both sides' slopes of W
    wm::equilibrium_flux(W0, c0, B, 0.5, n, qc, p.pr_fix, gas, F);
}

}  // namespace ugkwp
