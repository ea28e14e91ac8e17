// a3, a4: limited gradients (order 2) and the time-integrated wave flux per face,
// F = F^eq + F^{fr,wave} (per unit area, normal from owner to neighbour).  First
// order:
//
//  * W0 from the compatibility condition with the upwind initial state
//    (Sec. 2.1): W0 = rho_L <psi>_{u.n>0, L} + rho_R <psi>_{u.n<0, R};
//  * F^eq = q1 int u.n g0 psi (g_x = g_t = 0 at first order);
//  * F^{fr,wave} = (q4 - dt e^{-dt/tau}) int u.n g0^h psi (Sec. 2.3) with the
//    upwind hydrodynamic Maxwellian g0^h = (rho^h/rho) g of each side;
//  * tau at the face = mu(T0)/p0 + C2 |pL - pR|/|pL + pR| dt (Sec. 2.4 (d));
//  * q1..q5 are the time integrals of c1..c5 (Sec. 2.1);
//  * boundaries: diffuse wall (Sec. 2.4 (e), zero net wave mass flux), mirror
//    ghost for specular planes, all-hydrodynamic ghosts for far field and
//    zero-gradient outflow (their incoming half carries q4: no particles are
//    emitted from a ghost).
// The arithmetic of a face is in wave_math.cuh.
//
// Both flux kernels are bound by the binary64 pipe (77% busy in the second-order
// one).  Second order: 963 binary64 instructions per interior face against 1,595
// with moment tables and micro slopes in a face frame; alone on the 24^3 cavity
// (165,888 faces) 0.35 ms against 0.54 ms.  First order (channel of 393,216
// tets, 790,528 faces): 0.63 ms against 0.78 ms.
#include "ugkwp_internal.hpp"
#include "recon.cuh"

// A few warps per SM keep the binary64 pipe busy; the second-order flux runs
// as a persistent grid (by default one block per SM, see LaunchCfg) so that the
// particle kernels running beside it keep most of each SM's registers and warp
// slots.
#ifndef UGKWP_WAVE_THREADS
#define UGKWP_WAVE_THREADS 128
#endif
#ifndef UGKWP_WAVE_MIN_BLOCKS
#define UGKWP_WAVE_MIN_BLOCKS 1
#endif

namespace ugkwp {

namespace {

// Gradient kernel: three threads per cell, a persistent grid.  Two blocks per SM
// leave room for the sampling kernel and the first half of the tracking grid,
// which then spreads evenly over the SMs and leaves each its room for a block
// of the wave flux: two steps of the settled 24^3 cavity take 2.22 ms in a row
// and 2.26 ms on their own, against 2.19 and 2.57 with three blocks per SM and
// 2.24 and 2.57 with four.  In the start-up steps and with
// first-order g_p sampling, which waits for the gradients, nothing runs beside it:
// four (four start-up steps of a channel of 96,000 tets 2.01 against 2.03 ms, two
// g_p-sampled steps of the 16^3 cavity 478 -> 467 us).
constexpr int GRAD_THREADS = 128, GRAD_BLOCKS_PER_SM = 2;

// Constants of K internal degrees of freedom (rho E = rho |U|^2/2 + (3+K)/2 p,
// <|xi|^2> = K theta, theta = 1/(2 lambda)); for K = 0 each is the monatomic
// literal (4/3, 1/3, 3, 5/2) exactly.
struct KC {
    double c43, c13, e3, e5h;
};
__device__ __forceinline__ KC kconst(int K) {
    const double e3 = 3.0 + (double)K;
    return KC{4.0 / e3, 1.0 / e3, e3, 0.5 * (5.0 + (double)K)};
}

__device__ __forceinline__ double dot3(const double* a, const double* b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; }

// ------------------------------------------------------------- order 2
// a3: least-squares gradients over the 4 face neighbours (host-precomputed
// coefficients c_k, ghosts mirrored across boundary faces) limited with
// Venkatakrishnan's function, per conservative component and for rho^h.

__device__ __forceinline__ void gradients_body(const DevMesh& m, const DevState& s, const DevParams& p, Blk bk) {
    const int nc = m.nc;
    // pair-major, so that neighbouring threads read neighbouring cells of one array
    for (int t = bk.id * blockDim.x + threadIdx.x; t < 3 * nc; t += bk.n * blockDim.x) {
        const int pair = t >= 2 * nc ? 2 : t >= nc ? 1 : 0, i = t - pair * nc;
        limited_pair(
            m, p, i, pair, [&](int q, int j) { return q < 5 ? s.W[(size_t)q * nc + j] : s.rhoh[j]; },
            [&](int tag, int q) { return p.bc[tag].W_in[q < 5 ? q : 0]; }, [](int, double phi) { return phi; },
            s.rec + (size_t)REC_N * i);
    }
}
__global__ void __launch_bounds__(GRAD_THREADS) k_gradients(DevMesh m, DevState s, DevParams p) {
    gradients_body(m, s, p, Blk{(int)blockIdx.x, (int)gridDim.x});
}

// Micro slope a with <psi psi^T> a = b for the unit Maxwellian (U, lambda),
// in closed form: with theta = 1/(2 lambda), R_i = b_i - U_i b_0,
// R_4 = 2 b_4 - (|U|^2 + 3 theta) b_0:  a_4 = 4 lambda^2/3 (R_4 - 2 U.R),
// a_i = 2 lambda R_i - U_i a_4,  a_0 = b_0 - U.a - a_4 (|U|^2 + 3 theta)/2.
__device__ __forceinline__ void micro(const double* U, double lam, double th, const double* b, double* a,
                                      const KC& kc) {
    const double R1 = b[1] - U[0] * b[0], R2 = b[2] - U[1] * b[0], R3 = b[3] - U[2] * b[0];
    const double U2 = U[0] * U[0] + U[1] * U[1] + U[2] * U[2];
    const double R4 = 2.0 * b[4] - (U2 + kc.e3 * th) * b[0];
    a[4] = kc.c43 * lam * lam * (R4 - 2.0 * (U[0] * R1 + U[1] * R2 + U[2] * R3));
    a[1] = 2.0 * lam * R1 - U[0] * a[4];
    a[2] = 2.0 * lam * R2 - U[1] * a[4];
    a[3] = 2.0 * lam * R3 - U[2] * a[4];
    a[0] = b[0] - (U[0] * a[1] + U[1] * a[2] + U[2] * a[3]) - 0.5 * a[4] * (U2 + kc.e3 * th);
}

// Equilibrium slope terms in closed form.  For the unit-density Maxwellian
// (U, theta = 1/(2 lambda)) and a micro slope a with <psi psi^T> a = b, the
// product (a.psi) g is the derivative of g(W) along b, so every slope moment is
// the derivative of a Maxwellian moment along b, with
// d rho = b0, dU = b_{1..3} - U b0, d theta = (2 b4 - (|U|^2 + 3 theta) b0 - 2 U.dU)/3:
//   <u_D (a.psi) psi>     = dF_D(b), F_D the Euler flux along D,
//   <u_n u_D (a.psi) psi> = dQ_D(b), Q_D = <u_n u_D psi g> with
//   <u_i u_j> = U_i U_j + theta d_ij,
//   <u_i u_j u_k> = U_i U_j U_k + theta (U_i d_jk + U_j d_ik + U_k d_ij),
//   <u_i u_j |u|^2/2> = (U_i U_j (|U|^2 + 7 theta) + d_ij theta (|U|^2 + 5 theta))/2.
// The face frame has the normal as direction 0.
struct DPrim { double dr, dU[3], dth, UdU; };

__device__ __forceinline__ DPrim dprim(const double* U, double th, double U2, const double* b, const KC& kc) {
    DPrim q;
    q.dr = b[0];
    for (int j = 0; j < 3; ++j) q.dU[j] = b[1 + j] - U[j] * b[0];
    q.UdU = U[0] * q.dU[0] + U[1] * q.dU[1] + U[2] * q.dU[2];
    q.dth = ((2.0 * b[4] - (U2 + kc.e3 * th) * b[0]) - 2.0 * q.UdU) * kc.c13;
    return q;
}

// dF_D(b) (Euler flux Jacobian along frame direction D applied to b)
template <int D>
__device__ __forceinline__ void euler_jac(const double* U, double th, double U2, const double* b, const DPrim& q,
                                          const KC& kc, double out[5]) {
    out[0] = b[1 + D];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        double v = q.dr * (U[D] * U[j]) + q.dU[D] * U[j] + U[D] * q.dU[j];
        if (j == D) v += q.dr * th + q.dth;
        out[1 + j] = v;
    }
    out[4] = b[1 + D] * (0.5 * U2 + kc.e5h * th) + U[D] * (q.UdU + kc.e5h * q.dth);
}

// First-order g_p sampling (Sec. 2.2), per cell: g_p = g - c (u.grad g + g_t),
// c = tau - dt e^{-dt/tau}/(1 - e^{-dt/tau}), with grad g from the limited
// gradient and g_t from W_t = -sum_d dF_d/dx_d; as a polynomial phi of
// X = (u - U)/sqrt(RT) in g_p = rho N(X)(1 + phi), bounded over |X| <= 5 and
// scaled down where that bound Phi exceeds 1; stores GP_NC values per cell.
__device__ __forceinline__ void gp_coef_body(const DevMesh& m, const DevState& s, const DevParams& p, Blk bk) {
    const int nc = m.nc;
    const int i = bk.id * blockDim.x + threadIdx.x;
    if (i >= nc) return;
    const double rho = s.prim[i];
    const double U[3] = {s.prim[nc + i], s.prim[2 * nc + i], s.prim[3 * nc + i]};
    const double th = p.R * s.prim[4 * nc + i];
    const double lam = 0.5 / th;
    const double sig = sqrt(th);
    const double U2 = dot3(U, U);
    const double ir = 1.0 / rho;
    const KC kc = kconst(p.K);
    double bd[3][5], a[3][5], Wt[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, t5[5];
    for (int d = 0; d < 3; ++d)
        for (int q = 0; q < 5; ++q) bd[d][q] = s.rec[(size_t)REC_N * i + 6 + 3 * q + d] * ir;
    {
        const DPrim q = dprim(U, th, U2, bd[0], kc);
        euler_jac<0>(U, th, U2, bd[0], q, kc, t5);
        for (int k = 0; k < 5; ++k) Wt[k] -= t5[k];
    }
    {
        const DPrim q = dprim(U, th, U2, bd[1], kc);
        euler_jac<1>(U, th, U2, bd[1], q, kc, t5);
        for (int k = 0; k < 5; ++k) Wt[k] -= t5[k];
    }
    {
        const DPrim q = dprim(U, th, U2, bd[2], kc);
        euler_jac<2>(U, th, U2, bd[2], q, kc, t5);
        for (int k = 0; k < 5; ++k) Wt[k] -= t5[k];
    }
    double B[5];
    for (int d = 0; d < 3; ++d) micro(U, lam, th, bd[d], a[d], kc);
    micro(U, lam, th, Wt, B, kc);
    // P(u) = B0 + v.u + u^T K u + (h/2)|u|^2 + (|u|^2/2)(beta.u), K[d][j] = a_d,1+j
    double v[3], beta[3];
    const double h = B[4];
    for (int j = 0; j < 3; ++j) {
        v[j] = B[1 + j] + a[j][0];
        beta[j] = a[j][4];
    }
    const double bU = dot3(beta, U);
    double KU[3], UKU = 0.0;
    for (int d = 0; d < 3; ++d) {
        KU[d] = 0.0;
        for (int j = 0; j < 3; ++j) {
            KU[d] += (a[d][1 + j] + a[j][1 + d]) * U[j];
            UKU += U[d] * a[d][1 + j] * U[j];
        }
    }
    double co[13];
    co[0] = B[0] + dot3(v, U) + UKU + 0.5 * h * U2 + 0.5 * U2 * bU;
    for (int d = 0; d < 3; ++d) {
        co[1 + d] = sig * (v[d] + KU[d] + h * U[d] + 0.5 * U2 * beta[d] + bU * U[d]);
        co[10 + d] = 0.5 * sig * sig * sig * beta[d];
    }
    const int qi[6] = {0, 1, 2, 0, 0, 1}, qj[6] = {0, 1, 2, 1, 2, 2};
    for (int k = 0; k < 6; ++k) {
        const int d = qi[k], j = qj[k];
        co[4 + k] = sig * sig * (0.5 * (a[d][1 + j] + a[j][1 + d]) + 0.5 * (U[d] * beta[j] + U[j] * beta[d]) +
                                 (d == j ? 0.5 * h + 0.5 * bU : 0.0));
    }
    const double dt = s.dt[0];
    const double e = exp(-(dt / s.tau[i]));
    const double c = s.tau[i] - dt * e / (1.0 - e);
    for (int k = 0; k < 13; ++k) co[k] = -c * co[k];
    const double nL = sqrt(co[1] * co[1] + co[2] * co[2] + co[3] * co[3]);
    const double nQ = sqrt(co[4] * co[4] + co[5] * co[5] + co[6] * co[6] + 2.0 * (co[7] * co[7] + co[8] * co[8] + co[9] * co[9]));
    const double nC = sqrt(co[10] * co[10] + co[11] * co[11] + co[12] * co[12]);
    double Phi = fabs(co[0]) + 5.0 * nL + 25.0 * nQ + 125.0 * nC;
    if (Phi > 1.0) {
        for (int k = 0; k < 13; ++k) co[k] = co[k] / Phi;
        Phi = 1.0;
    }
    for (int k = 0; k < 13; ++k) s.gpc[(size_t)k * nc + i] = co[k];
    s.gpc[(size_t)13 * nc + i] = 1.0 + Phi;
}
__global__ void __launch_bounds__(128) k_gp_coef(DevMesh m, DevState s, DevParams p) {
    gp_coef_body(m, s, p, Blk{(int)blockIdx.x, (int)gridDim.x});
}

__device__ __forceinline__ void face_flux_o1(const DevMesh& m, const DevState& s, const DevParams& p, int t);

// The faces face_order[first..nf) in tiles of 32, one warp each.  SHARED: a grid that
// does not cover them takes the tiles from a counter, reserved one ahead, instead of
// a fixed stride: the tracking's blocks can keep some flux blocks off the SMs until
// the others are done, and with fixed shares those then start theirs.  Two steps of
// a batch of 14 instances, second order, 7.33 -> 7.08 ms; of a channel of 393,216
// tets, first order, 5.12 -> 5.07 ms.  Not SHARED: the second-order kernel of one
// simulation, whose replayed steps place every block at once (24^3 cavity 1.59
// against 1.61 ms, start-up steps 2.014 against 2.021).
template <bool SHARED>
struct FaceTiles {
    unsigned long long* next_tile;
    long long next;
    int n;
    int stride;
    bool shared;
    __device__ __forceinline__ FaceTiles(const DevState& s, int nf, int first, Blk bk) {
        next_tile = reinterpret_cast<unsigned long long*>(s.cnt64 + CNT_FLUX);
        n = nf;
        stride = bk.n * blockDim.x;
        shared = SHARED && stride < nf - first;
        base = first;
        next = first + (shared ? reserve() : (long long)bk.id * blockDim.x + (threadIdx.x & ~31u));
    }
    __device__ __forceinline__ bool take(int& t) {
        const long long t0 = SHARED ? __shfl_sync(0xffffffffu, next, 0) : next;
        if (t0 >= n) return false;
        t = (int)t0 + (int)(threadIdx.x & 31);
        next = shared ? base + reserve() : next + stride;
        return true;
    }

   private:
    int base;
    __device__ __forceinline__ long long reserve() {  // (lane 0's counts)
        return (threadIdx.x & 31) == 0 ? (long long)atomicAdd(next_tile, 32ull) : 0;
    }
};

// Second-order flux of the interior faces (the first nif entries of face_order),
// then the first-order flux of the boundary faces that follow them.
// With local time steps (GKS step) each face is integrated over the smaller
// step of its cells and stores the mean flux rate F / dt_f.
template <bool SHARED>
__device__ __forceinline__ void face_flux_o2_body(const DevMesh& m, const DevState& s, const DevParams& p, Blk bk) {
    const int nf = m.nf;
    const double dt = s.dt[0];
    FaceTiles<SHARED> tiles(s, nf, 0, bk);
    for (int t; tiles.take(t);) {
        if (t >= nf) continue;
        if (t >= m.nif) {  // the boundary faces follow, at first order, in the same grid
            face_flux_o1(m, s, p, t);
            continue;
        }
        const int f = m.face_order[t];
        const int o = m.f_own[f], nb = m.f_nbr[f];
        const double n[3] = {m.f_n[f], m.f_n[nf + f], m.f_n[2 * nf + f]};
        const double dtf = p.gks == 2 ? fmin(s.dtc[o], s.dtc[nb]) : dt;
        double F[5];
        interior_flux_o2(m, s.rec, p, f, o, nb, n, dtf, F);
        if (p.gks == 2)
            for (int q = 0; q < 5; ++q) F[q] = F[q] / dtf;
        for (int q = 0; q < 5; ++q) s.F[(size_t)q * nf + f] = F[q];
    }
}
__global__ void __launch_bounds__(UGKWP_WAVE_THREADS, UGKWP_WAVE_MIN_BLOCKS) k_face_flux_o2(DevMesh m, DevState s, DevParams p) {
    face_flux_o2_body<false>(m, s, p, Blk{(int)blockIdx.x, (int)gridDim.x});
}

// First-order flux of face face_order[t].
__device__ __forceinline__ void face_flux_o1(const DevMesh& m, const DevState& s, const DevParams& p, int t) {
    const int nc = m.nc, nf = m.nf;
    const int f = m.face_order[t];  // interior faces first, then boundary faces by type
    const double n[3] = {m.f_n[f], m.f_n[nf + f], m.f_n[2 * nf + f]};
    const int o = m.f_own[f], nb = m.f_nbr[f];
    // local time steps (GKS step): the smaller step of the face's cells
    const double dt = p.gks == 2 ? (nb >= 0 ? fmin(s.dtc[o], s.dtc[nb]) : s.dtc[o]) : s.dt[0];
    const wm::FaceGas fg = face_gas(p);
    double W[5];
    for (int q = 0; q < 5; ++q) W[q] = s.W[(size_t)q * nc + o];
    const wm::Prim L = wm::prim_of(W, fg.gas);
    const double rhL = s.rhoh[o];
    double F[5];
    if (nb < 0 && p.bc[m.bf_tag[-1 - nb]].type == UGKWP_BC_DIFFUSE_WALL) {
        // Sec. 2.4 (e): incoming half with the cell's tau, re-emitted half of the
        // wall's Maxwellian with zero net wave mass flux
        const DevBc& bc = p.bc[m.bf_tag[-1 - nb]];
        const wm::QC1 c = wm::time_coeffs(dt, s.tau[o]);
        const double c1 = c.q1 * L.rho + (p.gks ? c.q4 : c.a4) * rhL;
        wm::Prim w;
        for (int d = 0; d < 3; ++d) w.U[d] = bc.U_w[d];
        w.th = p.R * bc.T_w;
        const wm::PrimGrad none{};
        const double z[3] = {0.0, 0.0, 0.0};
        const wm::SideFlux a = wm::side_flux<false>(L, none, 0.0, z, n, 1.0, fg.gas);
        const wm::SideFlux b = wm::side_flux<false>(w, none, 0.0, z, n, -1.0, fg.gas);
        const double r = a.G[0] / b.G[0];
        F[0] = 0.0;
        for (int k = 1; k < 5; ++k) F[k] = c1 * (a.G[k] - r * b.G[k]);
    } else {
        const int type = nb >= 0 ? 0 : p.bc[m.bf_tag[-1 - nb]].type;
        wm::Prim R = L;
        double rhR = rhL;
        bool ghost = false;
        if (nb >= 0) {
            for (int q = 0; q < 5; ++q) W[q] = s.W[(size_t)q * nc + nb];
            R = wm::prim_of(W, fg.gas);
            rhR = s.rhoh[nb];
        } else if (type == UGKWP_BC_SPECULAR) {
            const double Un = wm::dot(L.U, n);
            for (int d = 0; d < 3; ++d) R.U[d] = L.U[d] - 2.0 * Un * n[d];
        } else {
            if (type == UGKWP_BC_FARFIELD) R = wm::prim_of(p.bc[m.bf_tag[-1 - nb]].W_in, fg.gas);
            rhR = R.rho;
            ghost = true;
        }
        wm::flux_o1(L, rhL, R, rhR, ghost, p.gks != 0, n, dt, fg, F);
        if (type == UGKWP_BC_SPECULAR) {
            const double fn = wm::dot(F + 1, n);
            F[0] = 0.0;
            F[4] = 0.0;
            for (int d = 0; d < 3; ++d) F[1 + d] = fn * n[d];
        }
    }
    if (p.gks == 2)
        for (int q = 0; q < 5; ++q) F[q] = F[q] / dt;
    for (int q = 0; q < 5; ++q) s.F[(size_t)q * nf + f] = F[q];
}

// First-order flux of the faces face_order[first..nf).
__device__ __forceinline__ void face_flux_body(const DevMesh& m, const DevState& s, const DevParams& p, int first, Blk bk) {
    FaceTiles<true> tiles(s, m.nf, first, bk);
    for (int t; tiles.take(t);)
        if (t < m.nf) face_flux_o1(m, s, p, t);
}
__global__ void __launch_bounds__(256) k_face_flux(DevMesh m, DevState s, DevParams p, int first) {
    face_flux_body(m, s, p, first, Blk{(int)blockIdx.x, (int)gridDim.x});
}

// ---- fused batches: member i of the chunk runs on the blocks
// off[cls][i] .. off[cls][i + 1] - 1.
__device__ __forceinline__ int member_of(const int32_t* off, int n) {
    int lo = 0, hi = n;  // off[lo] <= blockIdx.x < off[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= (int)blockIdx.x) lo = mid;
        else hi = mid;
    }
    return lo;
}
__device__ __forceinline__ Blk member_blk(const int32_t* off, int i) {
    return Blk{(int)blockIdx.x - off[i], off[i + 1] - off[i]};
}
// The flux of a block's own member i, then what is left of the others' tiles (a
// member whose blocks cover its faces has none).
template <class F> __device__ __forceinline__ void for_members(const BatchChunk& c, const int32_t* off, int i, F&& flux) {
    for (int k = 0, j = i; k < c.n; ++k, j = j + 1 < c.n ? j + 1 : 0)
        if (j == i || (long long)(off[j + 1] - off[j]) * blockDim.x < c.mem[j].m.nf)
            flux(j, Blk{(int)blockIdx.x - off[j], off[j + 1] - off[j]});
}
__global__ void __launch_bounds__(GRAD_THREADS) k_gradients_b(const __grid_constant__ BatchChunk c) {
    const int i = member_of(c.off[BCL_GRAD], c.n);
    gradients_body(c.mem[i].m, c.mem[i].s, c.mem[i].p, member_blk(c.off[BCL_GRAD], i));
}
__global__ void __launch_bounds__(128) k_gp_coef_b(const __grid_constant__ BatchChunk c) {
    const int i = member_of(c.off[BCL_GPC], c.n);
    gp_coef_body(c.mem[i].m, c.mem[i].s, c.mem[i].p, member_blk(c.off[BCL_GPC], i));
}
__global__ void __launch_bounds__(UGKWP_WAVE_THREADS, UGKWP_WAVE_MIN_BLOCKS)
    k_face_flux_o2_b(const __grid_constant__ BatchChunk c) {
    const int i = member_of(c.off[BCL_FLUX_O2], c.n);
    for_members(c, c.off[BCL_FLUX_O2], i, [&](int k, Blk bk) { face_flux_o2_body<true>(c.mem[k].m, c.mem[k].s, c.mem[k].p, bk); });
}
__global__ void __launch_bounds__(256) k_face_flux_b(const __grid_constant__ BatchChunk c) {
    const int i = member_of(c.off[BCL_FLUX], c.n);
    for_members(c, c.off[BCL_FLUX], i, [&](int k, Blk bk) { face_flux_body(c.mem[k].m, c.mem[k].s, c.mem[k].p, 0, bk); });
}

}  // namespace

// Block size of a persistent grid of at most `blocks` blocks of `threads`: where
// n items do not fill one such block per SM, smaller blocks spread them over more
// SMs, each of which has its own binary64 pipe.
static int wave_block(long long n, int threads) {
    const int sms = sm_count();
    while (threads > 32 && n <= (long long)sms * (threads / 2)) threads /= 2;
    return threads;
}
static int wave_grid(long long n, int threads, int blocks) {
    const long long need = (n + threads - 1) / threads;
    return need < blocks ? (int)need : blocks;
}

// A persistent grid of GRAD_BLOCKS_PER_SM blocks per SM, which leaves room
// beside it for the first half of the tracking grid.
void launch_gradients(const DevMesh& m, const DevState& s, const DevParams& p, cudaStream_t st) {
    const int t = wave_block(3LL * m.nc, GRAD_THREADS);
    k_gradients<<<wave_grid(3LL * m.nc, t, (p.gks || p.sampling == UGKWP_SAMPLE_GP1 ? 4 : GRAD_BLOCKS_PER_SM) * sm_count() * (GRAD_THREADS / t)), t, 0, st>>>(m, s, p);
}

void launch_gp_coef(const DevMesh& m, const DevState& s, const DevParams& p, cudaStream_t st) {
    k_gp_coef<<<blocks_gp_coef(m.nc), 128, 0, st>>>(m, s, p);
}

void launch_face_flux_o2(const DevMesh& m, const DevState& s, const DevParams& p, int blocks, cudaStream_t st) {
    const int t = wave_block(m.nf, UGKWP_WAVE_THREADS);
    k_face_flux_o2<<<wave_grid(m.nf, t, blocks * (UGKWP_WAVE_THREADS / t)), t, 0, st>>>(m, s, p);
}

int wave_threads() { return UGKWP_WAVE_THREADS; }

cudaError_t configure_wave_kernels(int carveout) {
    cudaError_t e = cudaSuccess;
    auto set = [&](auto f) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, carveout);
    };
    set(k_gradients);
    set(k_gp_coef);
    set(k_face_flux_o2);
    set(k_face_flux);
    set(k_gradients_b);
    set(k_gp_coef_b);
    set(k_face_flux_o2_b);
    set(k_face_flux_b);
    return e;
}

// blocks > 0 bounds the grid (a step of the method: the flux shares the GPU
// with the particle kernels launched beside it); 0: one thread per face.
void launch_face_flux(const DevMesh& m, const DevState& s, const DevParams& p, int first, int blocks,
                      cudaStream_t st) {
    const long long n = m.nf - first;
    const int t = wave_block(n, 256);
    const int need = (int)((n + t - 1) / t);
    k_face_flux<<<blocks > 0 ? wave_grid(n, t, blocks * (256 / t)) : need, t, 0, st>>>(m, s, p, first);
}

int blocks_gp_coef(int nc) { return (nc + 127) / 128; }
int gradient_threads() { return GRAD_THREADS; }
int gradient_blocks_per_sm() { return GRAD_BLOCKS_PER_SM; }

void launch_gradients_batch(const BatchChunk& c, int blocks, cudaStream_t st) {
    k_gradients_b<<<blocks, GRAD_THREADS, 0, st>>>(c);
}
void launch_gp_coef_batch(const BatchChunk& c, int blocks, cudaStream_t st) { k_gp_coef_b<<<blocks, 128, 0, st>>>(c); }
void launch_face_flux_o2_batch(const BatchChunk& c, int blocks, cudaStream_t st) {
    k_face_flux_o2_b<<<blocks, UGKWP_WAVE_THREADS, 0, st>>>(c);
}
void launch_face_flux_batch(const BatchChunk& c, int blocks, cudaStream_t st) {
    k_face_flux_b<<<blocks, 256, 0, st>>>(c);
}

}  // namespace ugkwp
