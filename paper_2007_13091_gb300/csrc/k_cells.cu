// Per-cell kernels of the UGKWP step: primitives, relaxation time and the
// time-step reduction (a1, a2), hydro-particle counts (a5), the exclusive scan
// that places each cell's samples after the survivors (a11), and the
// conservative update (a10).  Compiled with --fmad=false: tau, dt, N_sam and m_sam decide integer
// outcomes of the particle path and must be reproducible bit for bit.
#include <cfloat>

#include "dmath.cuh"
#include "fixed.cuh"
#include "ugkwp_internal.hpp"

namespace ugkwp {

namespace {

__device__ __forceinline__ void set_err(const DevState& s, int32_t bits) {
    atomicOr(reinterpret_cast<unsigned long long*>(&s.cnt64[CNT_ERR]), (unsigned long long)bits);
}

// Inclusive scan of two ints per thread (count, N_sam) over one block.
__device__ __forceinline__ int2 block_scan_incl2(int2 v, int2* sh_warp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int ox = __shfl_up_sync(0xffffffffu, v.x, d);
        const int oy = __shfl_up_sync(0xffffffffu, v.y, d);
        if (lane >= d) { v.x += ox; v.y += oy; }
    }
    if (lane == 31) sh_warp[warp] = v;
    __syncthreads();
    if (warp == 0) {
        int2 w = (lane < (int)(blockDim.x >> 5)) ? sh_warp[lane] : make_int2(0, 0);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int ox = __shfl_up_sync(0xffffffffu, w.x, d);
            const int oy = __shfl_up_sync(0xffffffffu, w.y, d);
            if (lane >= d) { w.x += ox; w.y += oy; }
        }
        sh_warp[lane] = w;
    }
    __syncthreads();
    if (warp > 0) { v.x += sh_warp[warp - 1].x; v.y += sh_warp[warp - 1].y; }
    return v;
}

// a1 + a2: primitives, tau = mu_ref/p (T/T_ref)^omega, rho^p from the survivors'
// fixed-point mass, rho^h = rho - rho^p, and min_i |Omega_i| / sum_d Lambda_i^d.
__device__ __forceinline__ void cell_prep_body(const DevMesh& m, const DevState& s, const DevParams& p, Blk bk) {
    const int nc = m.nc;
    const int i = bk.id * blockDim.x + threadIdx.x;
    double r = __longlong_as_double(0x7ff0000000000000LL);
    if (i < nc) {
        // the sums this step's tracking adds to
#pragma unroll
        for (int q = 0; q < 5; ++q) s.pflux[(size_t)q * nc + i] = 0;
        s.fill[i] = 0;
        if (i < scan_groups(nc)) s.gsum[i] = make_longlong2(0, 0);
        if (i == 0) s.cnt64[CNT_FLUX] = 0;
        const double rho = s.W[i];
        const double Ux = s.W[nc + i] / rho, Uy = s.W[2 * nc + i] / rho, Uz = s.W[3 * nc + i] / rho;
        const double U2 = (Ux * Ux + Uy * Uy) + Uz * Uz;
        const double pr = (s.W[4 * nc + i] - 0.5 * (rho * U2)) / (1.5 + 0.5 * (double)p.K);
        const double T = pr / (rho * p.R);
        double tau = 1.0;
        if (!(rho > 0.0) || !(pr > 0.0) || !isfinite(pr)) {
            set_err(s, ERRB_NONFINITE);
        } else {
            tau = (p.mu_ref / pr) * dm::d_exp(p.omega * dm::d_log(T / p.T_ref));
            const double c = 3.0 * sqrt(p.R * T);
            const double lam = ((fabs(Ux) + c) * m.dS[i] + (fabs(Uy) + c) * m.dS[nc + i]) + (fabs(Uz) + c) * m.dS[2 * nc + i];
            r = m.vol[i] / lam;
        }
        if (p.gks == 2) s.dtc[i] = p.CFL * r;
        const double rhop = ((double)s.smass[i] * p.qscale[0]) / m.vol[i];
        s.prim[i] = rho;
        s.prim[nc + i] = Ux;
        s.prim[2 * nc + i] = Uy;
        s.prim[3 * nc + i] = Uz;
        s.prim[4 * nc + i] = T;
        s.tau[i] = tau;
        s.tauf[i] = (float)tau;
        if (p.precision == UGKWP_MIXED)
            s.usig[i] = make_float4((float)Ux, (float)Uy, (float)Uz, (float)sqrt(p.R * T));
        s.rhop[i] = rhop;
        s.rhoh[i] = rho - rhop;
    }
    // block minimum, then one atomic on the ordered bit pattern (r > 0)
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) r = fmin(r, __shfl_xor_sync(0xffffffffu, r, d));
    __shared__ double sh[32];
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = r;
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : __longlong_as_double(0x7ff0000000000000LL);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, d));
        if (threadIdx.x == 0 && v < __longlong_as_double(0x7ff0000000000000LL) && v > 0.0)
            atomicMin(reinterpret_cast<unsigned long long*>(&s.cnt64[CNT_DT_BITS]),
                      (unsigned long long)__double_as_longlong(v));
    }
}
__global__ void k_cell_prep(DevMesh m, DevState s, DevParams p) {
    cell_prep_body(m, s, p, Blk{(int)blockIdx.x, (int)gridDim.x});
}

// a5 counts: rho^hp = e^{-dt/tau} rho^h, m_ref = (rho^p + rho^hp)|Omega|/N_ref,
// N_sam = 2 ceil(rho^hp |Omega| / (2 m_ref)), N_sam >= N_min - N_left,
// m_sam = rho^hp |Omega| / N_sam (Sec. 2.4 (b)).  Also the survivor bucket
// the cell gets in the buffer this step's survivors are written to (a11:
// sized from the particles that start the step in the cell), and the
// per-block sums of the bucket sizes and of N_sam.
__device__ __forceinline__ void sample_count_body(const DevMesh& m, const DevState& s, const DevParams& p, Blk bk) {
    __shared__ int2 shw[32];
    const int nc = m.nc;
    const int i = bk.id * blockDim.x + threadIdx.x;
    const double dt = p.CFL * __longlong_as_double(s.cnt64[CNT_DT_BITS]);
    if (p.gks) {  // GKS step: the time step only, nothing is sampled
        if (i == 0) s.dt[0] = dt;
        return;
    }
    int wcap = 0, nsam = 0;
    if (i < nc) {
        const double vol = m.vol[i];
        const double ex = dm::d_exp(-(dt / s.tau[i]));
        const double rh = s.rhoh[i] > 0.0 ? s.rhoh[i] : 0.0;
        const double rhp = ex * rh;
        const double Mhp = rhp * vol;
        long long ns = 0;
        double ms = 0.0;
        if (Mhp > (s.prim[i] * vol) * 0x1p-30) {
            const double mref = ((s.rhop[i] + rhp) * vol) / (double)p.N_ref;
            ns = 2 * (long long)ceil(Mhp / (2.0 * mref));
            const long long need = (long long)p.N_min - (long long)s.nleft[i];
            if (need > ns) ns = need + (need & 1);
            if (ns > 65534) {
                set_err(s, ERRB_SAMPLE_LIMIT);
                ns = 0;
            } else {
                ms = Mhp / (double)ns;
            }
        }
        // the survivors' mass of this step starts from every particle of the cell;
        // the tracking takes out what is removed or leaves and adds what arrives
        long long qm = 0;
        if (ns > 0 && !fixed_of_mass(ms, p.exps[0], qm)) set_err(s, ERRB_FIXED_OVERFLOW);
        s.smass_next[i] = s.smass[i] + ns * qm;
        // collision threshold on the first 32 random bits of a particle's draw:
        // -tau ln eta < dt needs eta > e^{-dt/tau} up to the roundings of tau, dt and
        // of the logarithm in the particle precision (below 3e-7 in eta) and of eta
        // itself (2^-24); 2^-18 = 3.8e-6 below it no particle collides
        const double th = (ex - 0x1p-18) * 0x1p32;
        s.cthr[i] = th > 0.0 ? (uint32_t)th : 0u;
        s.nsam[i] = (int)ns;
        s.msam[i] = ms;
        nsam = (int)ns;
        const int count = s.nleft[i] + nsam;
        s.nleft_next[i] = count;
        wcap = bucket_slots(count);
        s.wcap[i] = wcap;
    }
    const int2 incl = block_scan_incl2(make_int2(wcap, nsam), shw);
    if (threadIdx.x == blockDim.x - 1) {
        s.bsum[bk.id] = incl;
        unsigned long long* g = reinterpret_cast<unsigned long long*>(s.gsum + bk.id / SCAN_GROUP);
        atomicAdd(g, (unsigned long long)incl.x);
        atomicAdd(g + 1, (unsigned long long)incl.y);
    }
    if (i == 0) s.dt[0] = dt;
}
__global__ void k_sample_count(DevMesh m, DevState s, DevParams p) {
    sample_count_body(m, s, p, Blk{(int)blockIdx.x, (int)gridDim.x});
}

// Offsets of the survivor buckets of the buffer written this step and of the
// sampled particles (they follow the N_A slots of the current buffer): every
// block sums the sums of the groups of blocks before its own group and of the
// blocks before its own in it (a few per thread) instead of waiting for a scan
// kernel (with the block sums alone, 64 cells each, a step of 2,239,488 tets took 8.79 ms
// instead of 8.43, one of 384,000 1.49 instead of 1.48); the last block has the totals, checks the capacity
// and clears the counters that the tracking adds to.
__device__ __forceinline__ void scan_apply_body(const DevMesh& m, const DevState& s, const DevParams& p, Blk bk) {
    __shared__ int2 shw[32];
    __shared__ long long part[2][32];
    long long px = 0, py = 0;
    const int group = bk.id / SCAN_GROUP;
    for (int j = threadIdx.x; j < group; j += blockDim.x) {
        const longlong2 v = s.gsum[j];
        px += v.x;
        py += v.y;
    }
    for (int j = group * SCAN_GROUP + threadIdx.x; j < bk.id; j += blockDim.x) {
        const int2 v = s.bsum[j];
        px += v.x;
        py += v.y;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        px += __shfl_xor_sync(0xffffffffu, px, d);
        py += __shfl_xor_sync(0xffffffffu, py, d);
    }
    if ((threadIdx.x & 31) == 0) {
        part[0][threadIdx.x >> 5] = px;
        part[1][threadIdx.x >> 5] = py;
    }
    const int i = bk.id * blockDim.x + threadIdx.x;
    const int2 v = i < m.nc ? make_int2(s.wcap[i], s.nsam[i]) : make_int2(0, 0);
    const int2 incl = block_scan_incl2(v, shw);  // (its barriers publish part)
    px = py = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        px += part[0][w];
        py += part[1][w];
    }
    if (i < m.nc) {
        s.soff[i] = (int)py + incl.y - v.y;
        const int woff = (int)px + incl.x - v.x;
        s.woff[i] = woff;
        s.cinfo[i] = make_int4((int)s.cthr[i], woff, v.x, __float_as_int(m.margin[i]));
    }
    if (bk.id == bk.n - 1 && threadIdx.x == blockDim.x - 1) {
        const long long wtot = px + incl.x, nsam = py + incl.y, slots = s.cnt64[CNT_N_A], left = s.cnt64[CNT_SURV];
        const long long live = left + nsam, cur = s.cnt64[CNT_CUR], age = s.cnt64[CNT_AGE] + 1;
        // steps in place leave holes: where the samples do not fit behind the slots,
        // but behind the particles, these are packed into the other buffer first
        const bool pack = p.in_place && slots + nsam > p.capacity && live <= p.capacity;
        const long long total = pack ? live : slots + nsam;
        const bool fits = total <= p.capacity && wtot <= p.capacity;
        if (!fits) set_err(s, ERRB_CAPACITY);
        s.cnt64[CNT_N_B] = fits ? total : 0;
        s.cnt64[CNT_NSAM] = fits ? nsam : 0;
        s.cnt64[CNT_SAMPLED] = nsam;
        s.cnt64[CNT_WTOT] = wtot;
        const bool in_place = p.in_place && fits && !pack && age < RESORT &&
                              total + 4 * nsam + 4LL * m.nc <= p.capacity && 8 * nsam <= live && 4 * (total - live) <= live;
        const long long src = pack ? 1 - cur : cur;
        s.cnt64[CNT_PACK] = pack && fits ? slots : 0;
        s.cnt64[CNT_PACKED] = 0;
        if (pack) s.cnt64[CNT_N_A] = left;
        s.cnt64[CNT_SRC] = src;
        s.cnt64[CNT_IN_PLACE] = in_place ? 1 : 0;
        s.cnt64[CNT_CUR] = in_place ? src : 1 - src;
        s.cnt64[CNT_AGE] = in_place ? age : 0;
        s.cnt64[CNT_COLLIDED] = 0;
        s.cnt64[CNT_EXITED] = 0;
        s.cnt64[CNT_LOST] = 0;
        s.cnt64[CNT_CROSSINGS] = 0;
        s.cnt64[CNT_WALL] = 0;
        s.cnt64[CNT_MOVERS] = 0;
        s.cnt64[CNT_TRACKED] = 0;
        s.cnt64[CNT_TILE] = 0;
        s.cnt64[CNT_OVF] = 0;
        s.cnt64[CNT_SURV] = 0;
    }
}
__global__ void k_scan_apply(DevMesh m, DevState s, DevParams p) {
    scan_apply_body(m, s, p, Blk{(int)blockIdx.x, (int)gridDim.x});
}

// a10: W^{n+1} = W^n - 1/|Omega| sum_k (+-F_k |S_k|) + F^{fr,p}/|Omega|, faces
// gathered in local order 0..3 (Eq. update_macro_variables).
__device__ __forceinline__ void cell_update_body(const DevMesh& m, const DevState& s, const DevParams& p, const PartBufs& bufs, Blk bk) {
    const int nc = m.nc, nf = m.nf;
    const int i = bk.id * blockDim.x + threadIdx.x;
    if (p.gks) {
        // GKS step (no particles): W -= sum_k (+-F_k |S_k|) / |Omega|; with local
        // steps F_k holds the flux rate and the cell advances by its own dt
        if (i == 0) {
            if (p.gks == 1) s.t[0] = s.t[0] + s.dt[0];
            s.cnt64[CNT_DT_BITS] = DT_BITS_NONE;
        }
        if (i >= nc) return;
        const int own = m.cfs[i];
        const double vol = m.vol[i];
        for (int q = 0; q < 5; ++q) {
            double acc = 0.0;
            for (int k = 0; k < 4; ++k) {
                const int f = m.cf[k * nc + i];
                const double v = s.F[(size_t)q * nf + f] * m.f_area[f];
                acc = acc + (((own >> k) & 1) ? v : -v);
            }
            double& w = s.W[(size_t)q * nc + i];
            w = p.gks == 2 ? w - (s.dtc[i] * acc) / vol : w - acc / vol;
        }
        return;
    }
    // past the capacity the slots of this step were not all written: no particle is left
    const bool lost = s.cnt64[CNT_ERR] & ERRB_CAPACITY;
    if (i == 0) {
        s.t[0] = s.t[0] + s.dt[0];
        if (p.averaging) s.tsum[0] += s.dt[0];
        s.cnt64[CNT_STEP] += 1;
        s.cnt64[CNT_DT_BITS] = DT_BITS_NONE;  // for the next step's minimum
        // sorted: the survivor buckets and the overflow slots; in place: every slot
        const long long ovf = s.cnt64[CNT_OVF];
        const long long room = p.capacity - s.cnt64[CNT_WTOT];
        s.cnt64[CNT_N_A] =
            lost ? 0 : s.cnt64[CNT_IN_PLACE] ? s.cnt64[CNT_N_B] : s.cnt64[CNT_WTOT] + (ovf < room ? ovf : room);
        if (lost) s.cnt64[CNT_SURV] = 0;
    }
    if (i >= nc) return;
    if (lost) {
        s.nleft_next[i] = 0;
        s.smass_next[i] = 0;
    } else if (!s.cnt64[CNT_IN_PLACE]) {  // a11: the bucket slots no survivor took are holes
        int32_t* wcell =
            reinterpret_cast<int32_t*>(reinterpret_cast<char*>(bufs.b0.cell) + (bufs.dyn ? s.cnt64[CNT_CUR] : 1) * bufs.delta);
        const int cap = s.wcap[i], fill = s.fill[i];
        s.nleft_next[i] = fill;  // the bucket's survivors, those in overflow slots included
        if ((long long)s.woff[i] + cap <= p.capacity)
            for (int k = fill < cap ? fill : cap; k < cap; ++k) wcell[(size_t)s.woff[i] + k] = -1;
    }
    // the particle part, added to W - sum_k (+-F_k |S_k|) / |Omega| that
    // k_wave_update left in W: (W - acc/|Omega|) + F^{fr,p}/|Omega|
    const double ivol = m.ivol[i];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const double fp = (double)s.pflux[(size_t)q * nc + i] * p.qscale[q];
        double& w = s.W[(size_t)q * nc + i];
        w = w + fp * ivol;
        if (p.averaging) s.wsum[(size_t)q * nc + i] += s.dt[0] * w;
    }
}

// a10, the wave part of a step with particles: W <- W - sum_k (+-F_k |S_k|)
// |Omega|^-1, faces gathered in local order 0..3.  It runs as soon as the
// wave flux is done, beside the tracking (no particle kernel reads W);
// k_cell_update adds the particle part once the tracking has summed its flux.
__device__ __forceinline__ void wave_update_body(const DevMesh& m, const DevState& s, Blk bk) {
    const int nc = m.nc, nf = m.nf;
    const int i = bk.id * blockDim.x + threadIdx.x;
    if (i >= nc) return;
    int f[4];
    const int own = m.cfs[i];
#pragma unroll
    for (int k = 0; k < 4; ++k) f[k] = m.cf[k * nc + i];
    // 1/|Omega| once per cell (the factor of the update) instead of ten
    // binary64 divisions
    const double ivol = m.ivol[i];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double v = s.F[(size_t)q * nf + f[k]] * m.f_area[f[k]];
            acc = acc + (((own >> k) & 1) ? v : -v);
        }
        double& w = s.W[(size_t)q * nc + i];
        w = w - acc * ivol;
    }
}
__global__ void k_wave_update(DevMesh m, DevState s) {
    wave_update_body(m, s, Blk{(int)blockIdx.x, (int)gridDim.x});
}
__global__ void k_cell_update(DevMesh m, DevState s, DevParams p, PartBufs bufs) {
    cell_update_body(m, s, p, bufs, Blk{(int)blockIdx.x, (int)gridDim.x});
}

// ---- fused batches: member i of the chunk runs on the blocks
// off[cls][i] .. off[cls][i + 1] - 1, the grid its own launch would have.
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

__global__ void k_cell_prep_b(const __grid_constant__ BatchChunk c) {
    const int i = member_of(c.off[BCL_CELLS], c.n);
    cell_prep_body(c.mem[i].m, c.mem[i].s, c.mem[i].p, member_blk(c.off[BCL_CELLS], i));
}
__global__ void k_sample_count_b(const __grid_constant__ BatchChunk c) {
    const int i = member_of(c.off[BCL_SCAN], c.n);
    sample_count_body(c.mem[i].m, c.mem[i].s, c.mem[i].p, member_blk(c.off[BCL_SCAN], i));
}
__global__ void k_scan_apply_b(const __grid_constant__ BatchChunk c) {
    const int i = member_of(c.off[BCL_SCAN], c.n);
    scan_apply_body(c.mem[i].m, c.mem[i].s, c.mem[i].p, member_blk(c.off[BCL_SCAN], i));
}
__global__ void k_cell_update_b(const __grid_constant__ BatchChunk c) {
    const int i = member_of(c.off[BCL_CELLS], c.n);
    cell_update_body(c.mem[i].m, c.mem[i].s, c.mem[i].p, c.mem[i].bufs, member_blk(c.off[BCL_CELLS], i));
}
__global__ void k_wave_update_b(const __grid_constant__ BatchChunk c) {
    const int i = member_of(c.off[BCL_CELLS], c.n);
    wave_update_body(c.mem[i].m, c.mem[i].s, member_blk(c.off[BCL_CELLS], i));
}

// Time average W-bar = sum dt^n W^n / sum dt^n (Sec. 2.4 (c)).
__global__ void k_wbar(DevMesh m, DevState s, double* out) {
    const long long n = 5LL * m.nc;
    const double T = s.tsum[0];
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) out[i] = s.wsum[i] / T;
}

// Kn_GLL = l |grad rho| / rho with the unlimited least-squares gradient of rho
// and the VHS mean free path l = 2(5-2w)(7-2w)/15 mu / (rho sqrt(2 pi R T)).
__global__ void k_kn_gll(DevMesh m, DevState s, DevParams p, double* out) {
    const int nc = m.nc;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nc) return;
    const double rho = s.W[i];
    const int own = m.cfs[i];
    double g[3] = {0.0, 0.0, 0.0};
    for (int k = 0; k < 4; ++k) {
        const int f = m.cf[k * nc + i];
        const int o = ((own >> k) & 1) ? m.f_nbr[f] : m.f_own[f];
        double v = rho;
        if (o >= 0) v = s.W[o];
        else if (p.bc[m.bf_tag[-1 - o]].type == UGKWP_BC_FARFIELD) v = p.bc[m.bf_tag[-1 - o]].W_in[0];
        for (int d = 0; d < 3; ++d) g[d] += m.lsq_c[(size_t)(3 * k + d) * nc + i] * (v - rho);
    }
    const double Ux = s.W[nc + i] / rho, Uy = s.W[2 * nc + i] / rho, Uz = s.W[3 * nc + i] / rho;
    const double pr = (s.W[4 * nc + i] - 0.5 * (rho * ((Ux * Ux + Uy * Uy) + Uz * Uz))) / (1.5 + 0.5 * (double)p.K);
    const double T = pr / (rho * p.R);
    const double mu = p.mu_ref * dm::d_exp(p.omega * dm::d_log(T / p.T_ref));
    const double w = p.omega;
    const double l = (2.0 * (5.0 - 2.0 * w) * (7.0 - 2.0 * w) / 15.0) * mu / (rho * sqrt(2.0 * 3.141592653589793 * p.R * T));
    out[i] = l * sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]) / rho;
}

// The survivors' count and fixed-point mass per cell of an imported buffer.
// Imported particles mostly come sorted by cell, so each warp sums over runs
// of equal cells in its 32 slots and adds once per run (integer sums: the
// result does not depend on how they are grouped).
template <class Real>
__global__ void k_rebuild(DevMesh m, DevState s, DevParams p, PartBufRaw a) {
    const long long n = s.cnt64[CNT_N_A];
    const int32_t* cell = a.cell;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const long long stride = (long long)gridDim.x * blockDim.x;
    // warp-uniform bounds: every lane takes part in the run sums
    for (long long base = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
        const long long i = base + lane;
        int c = -1;
        long long q = 0;
        if (i < n) {
            c = cell[i];
            // (a mass outside the fixed-point range is reported, as in the step)
            if (c >= 0 && !fixed_of_mass(a.m[i], p.exps[0], q)) set_err(s, ERRB_FIXED_OVERFLOW);
        }
        const int prev = __shfl_up_sync(FULL, c, 1);
        const unsigned heads = __ballot_sync(FULL, lane == 0 || prev != c);
        const int start = 31 - __clz(heads & (FULL >> (31 - lane)));
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const long long o = __shfl_up_sync(FULL, q, d);
            if (lane - d >= start) q += o;
        }
        const bool tail = lane == 31 || ((heads >> (lane + 1)) & 1u);
        if (tail && c >= 0) {
            atomicAdd(&s.nleft[c], lane - start + 1);
            atomicAdd(reinterpret_cast<unsigned long long*>(&s.smass[c]), (unsigned long long)q);
        }
    }
}

// A state image's particles, checked and brought into the particle
// precision in the spare buffer b (its cell, m and id arrays already hold the
// image's; so do x, u and e when they come in the particle precision).
// CONVERT (mixed mode, binary64 image): x, u and e come in binary64 (staged
// [3][n], [3][n], [n]); a position becomes its offset from the anchor of its
// tet, which must be exact in binary32 and give back the position when added
// to the anchor, and the velocity and internal energy must be binary32
// values.  *err receives the smallest i << 3 | kind over the particles that
// fail, kind being the first failed check of particle i: 1 cell outside
// [0, nc), 2 internal energy negative or not a number, 3 internal energy not
// a binary32 value, 4 position or velocity not representable.
template <class Real, bool CONVERT>
__global__ void k_import(int nc, long long n, const double* anc, const double* xs, const double* us,
                         const double* es, PartBufRaw b, unsigned long long* err) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const int c = b.cell[i];
        unsigned kind = 0;
        if (c < 0 || c >= nc) {
            kind = 1;
        } else if constexpr (CONVERT) {
            if (es) {
                const double ev = es[i];
                const float ef = __double2float_rn(ev);
                if (!(ev >= 0.0)) kind = 2;
                else if ((double)ef != ev) kind = 3;
                else static_cast<float*>(b.e)[i] = ef;
            }
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const double xv = xs[(size_t)d * n + i], uv = us[(size_t)d * n + i];
                const double A = anc[3 * (size_t)c + d];
                const double xl = xv - A;
                const float xf = __double2float_rn(xl), uf = __double2float_rn(uv);
                if (kind == 0 && ((double)xf != xl || A + xl != xv || (double)uf != uv)) kind = 4;
                static_cast<float*>(b.x[d])[i] = xf;
                static_cast<float*>(b.u[d])[i] = uf;
            }
        } else {
            if (b.e && !(static_cast<const Real*>(b.e)[i] >= (Real)0)) kind = 2;
        }
        if (kind) atomicMin(err, ((unsigned long long)i << 3) | kind);
    }
}

// Fixed-point sums of phi per cell.  A lane takes four slots in a row (16-byte
// loads; the arrays hold whole multiples of 256 slots) and sums while the cell
// stays the same; a warp then sums over lanes of equal cells and adds once per
// run.  Bound by the binary64 pipe: phi takes 10 binary64 instructions, the
// widening and the conversion to fixed point run on the integer pipes.  7.97e6
// particles: 0.185 ms (one thread and five atomics per particle: 0.44 ms).
template <class Real>
__global__ void __launch_bounds__(256) k_wp_acc(DevMesh m, DevState s, DevParams p, PartBufs bufs) {
    PartBufRaw a = bufs.b0;  // the buffer that holds the particles
    {
        const long long d = bufs.dyn ? s.cnt64[CNT_CUR] * bufs.delta : 0;
        for (int k = 0; k < 3; ++k) a.u[k] = static_cast<char*>(a.u[k]) + d;
        a.m = reinterpret_cast<double*>(reinterpret_cast<char*>(a.m) + d);
        a.cell = reinterpret_cast<int32_t*>(reinterpret_cast<char*>(a.cell) + d);
        if (a.e) a.e = static_cast<char*>(a.e) + d;
    }
    const unsigned n = (unsigned)s.cnt64[CNT_N_A];
    const int nc = m.nc, lane = threadIdx.x & 31;
    const unsigned FULL = 0xffffffffu;
    unsigned long long* wacc = reinterpret_cast<unsigned long long*>(s.wacc);
    const unsigned warps = gridDim.x * (blockDim.x / 32);
    for (unsigned base = (blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32) * 128u; base < n; base += warps * 128u) {
        const unsigned i = base + 4 * lane;
        const int4 cv = *reinterpret_cast<const int4*>(a.cell + i);
        const int cell[4] = {cv.x, cv.y, cv.z, cv.w};
        Real u[3][4], e[4] = {(Real)0, (Real)0, (Real)0, (Real)0};
        double mm[4];
        struct alignas(16) Four { Real v[4]; };
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const Four f = *reinterpret_cast<const Four*>(static_cast<const Real*>(a.u[d]) + i);
            for (int k = 0; k < 4; ++k) u[d][k] = f.v[k];
        }
        {
            const double2 v0 = reinterpret_cast<const double2*>(a.m + i)[0], v1 = reinterpret_cast<const double2*>(a.m + i)[1];
            mm[0] = v0.x; mm[1] = v0.y; mm[2] = v1.x; mm[3] = v1.y;
        }
        if (a.e) {
            const Four f = *reinterpret_cast<const Four*>(static_cast<const Real*>(a.e) + i);
            for (int k = 0; k < 4; ++k) e[k] = f.v[k];
        }
        long long acc[5] = {0, 0, 0, 0, 0};
        int key = -1;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c = i + k < n ? cell[k] : -1;
            if (c < 0) continue;  // a hole, or past the end
            if (c != key) {
                if (key >= 0)
                    for (int q = 0; q < 5; ++q) atomicAdd(&wacc[(size_t)q * nc + key], (unsigned long long)acc[q]);
                for (int q = 0; q < 5; ++q) acc[q] = 0;
                key = c;
            }
            const double u0 = widen(u[0][k]), u1 = widen(u[1][k]), u2 = widen(u[2][k]), mk = mm[k];
            const double phi[5] = {mk, mk * u0, mk * u1, mk * u2, mk * (((u0 * u0 + u1 * u1) + u2 * u2) + widen(e[k]))};
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                long long v;
                // (the energy's factor 1/2 as an exponent shift; a value outside the
                // range of the integer conversion takes the saturating one)
                if (!fixed_of(phi[q], p.exps[q] + (q == 4 ? 1 : 0), v)) v = __double2ll_rn((q == 4 ? 0.5 * phi[q] : phi[q]) * p.qinv[q]);
                acc[q] += v;
            }
        }
        const int prev = __shfl_up_sync(FULL, key, 1);
        const unsigned heads = __ballot_sync(FULL, lane == 0 || prev != key);
        const int start = 31 - __clz(heads & (FULL >> (31 - lane)));
        const bool tail = lane == 31 || ((heads >> (lane + 1)) & 1u);
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            long long v = acc[q];
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const long long o = __shfl_up_sync(FULL, v, d);
                if (lane - d >= start) v += o;
            }
            if (tail && key >= 0) atomicAdd(&wacc[(size_t)q * nc + key], (unsigned long long)v);
        }
    }
}

__global__ void k_zero_wacc(DevMesh m, DevState s) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < 5LL * m.nc; i += stride) s.wacc[i] = 0;
}

// which: 1 = W^p, 2 = W^h = W - W^p
__global__ void k_wp_out(DevMesh m, DevState s, DevParams p, int which, double* out) {
    const int nc = m.nc;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nc) return;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const double wp = ((double)s.wacc[(size_t)q * nc + i] * p.qscale[q]) / m.vol[i];
        out[(size_t)q * nc + i] = which == 1 ? wp : s.W[(size_t)q * nc + i] - wp;
    }
}

__global__ void k_prim_out(DevMesh m, DevState s, DevParams p, double* out) {
    const int nc = m.nc;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nc) return;
    const double rho = s.W[i];
    const double Ux = s.W[nc + i] / rho, Uy = s.W[2 * nc + i] / rho, Uz = s.W[3 * nc + i] / rho;
    const double U2 = (Ux * Ux + Uy * Uy) + Uz * Uz;
    const double pr = (s.W[4 * nc + i] - 0.5 * (rho * U2)) / (1.5 + 0.5 * (double)p.K);
    out[i] = rho;
    out[nc + i] = Ux;
    out[2 * nc + i] = Uy;
    out[3 * nc + i] = Uz;
    out[4 * nc + i] = pr / (rho * p.R);
}

inline int cdiv(long long a, int b) { return (int)((a + b - 1) / b); }

}  // namespace

int sm_count() {
    static int g = 0;
    if (!g) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 152;
        g = sms;
    }
    return g;
}

int particle_grid() { return sm_count() * 8; }

cudaError_t configure_cell_kernels(int carveout) {
    cudaError_t e = cudaSuccess;
    auto set = [&](auto f) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, carveout);
    };
    set(k_cell_prep);
    set(k_sample_count);
    set(k_scan_apply);
    set(k_cell_update);
    set(k_cell_prep_b);
    set(k_sample_count_b);
    set(k_scan_apply_b);
    set(k_cell_update_b);
    set(k_wave_update);
    set(k_wave_update_b);
    return e;
}

void launch_cell_prep(const DevMesh& m, const DevState& s, const DevParams& p, cudaStream_t st) {
    k_cell_prep<<<blocks_cells(m.nc), CELL_BLOCK, 0, st>>>(m, s, p);
}
void launch_sample_count(const DevMesh& m, const DevState& s, const DevParams& p, cudaStream_t st) {
    k_sample_count<<<scan_blocks(m.nc), SCAN_BLOCK, 0, st>>>(m, s, p);
}
void launch_scan(const DevMesh& m, const DevState& s, const DevParams& p, cudaStream_t st) {
    k_scan_apply<<<scan_blocks(m.nc), SCAN_BLOCK, 0, st>>>(m, s, p);
}
void launch_cell_update(const DevMesh& m, const DevState& s, const DevParams& p, const PartBufs& b, cudaStream_t st) {
    k_cell_update<<<blocks_cells(m.nc), CELL_BLOCK, 0, st>>>(m, s, p, b);
}
void launch_wave_update(const DevMesh& m, const DevState& s, cudaStream_t st) {
    k_wave_update<<<blocks_cells(m.nc), CELL_BLOCK, 0, st>>>(m, s);
}
int blocks_cells(int nc) { return cdiv(nc, CELL_BLOCK); }

void launch_cell_prep_batch(const BatchChunk& c, int blocks, cudaStream_t st) {
    k_cell_prep_b<<<blocks, CELL_BLOCK, 0, st>>>(c);
}
void launch_sample_count_batch(const BatchChunk& c, int blocks, cudaStream_t st) {
    k_sample_count_b<<<blocks, SCAN_BLOCK, 0, st>>>(c);
}
void launch_scan_batch(const BatchChunk& c, int blocks, cudaStream_t st) {
    k_scan_apply_b<<<blocks, SCAN_BLOCK, 0, st>>>(c);
}
void launch_cell_update_batch(const BatchChunk& c, int blocks, cudaStream_t st) {
    k_cell_update_b<<<blocks, CELL_BLOCK, 0, st>>>(c);
}
void launch_wave_update_batch(const BatchChunk& c, int blocks, cudaStream_t st) {
    k_wave_update_b<<<blocks, CELL_BLOCK, 0, st>>>(c);
}
void launch_rebuild_survivors(const DevMesh& m, const DevState& s, const DevParams& p, const PartBufRaw& a,
                              cudaStream_t st) {
    if (p.precision == UGKWP_MIXED) k_rebuild<float><<<particle_grid(), 256, 0, st>>>(m, s, p, a);
    else k_rebuild<double><<<particle_grid(), 256, 0, st>>>(m, s, p, a);
}
void launch_import(int nc, long long n, bool mixed, bool convert, const double* anc, const double* xs,
                   const double* us, const double* es, const PartBufRaw& b, unsigned long long* err,
                   cudaStream_t st) {
    if (n <= 0) return;
    if (mixed && convert) k_import<float, true><<<particle_grid(), 256, 0, st>>>(nc, n, anc, xs, us, es, b, err);
    else if (mixed) k_import<float, false><<<particle_grid(), 256, 0, st>>>(nc, n, anc, xs, us, es, b, err);
    else k_import<double, false><<<particle_grid(), 256, 0, st>>>(nc, n, anc, xs, us, es, b, err);
}
void launch_wp_moments(const DevMesh& m, const DevState& s, const DevParams& p, const PartBufs& b, cudaStream_t st) {
    k_zero_wacc<<<cdiv(5LL * m.nc, 256), 256, 0, st>>>(m, s);
    if (p.precision == UGKWP_MIXED) k_wp_acc<float><<<particle_grid(), 256, 0, st>>>(m, s, p, b);
    else k_wp_acc<double><<<particle_grid(), 256, 0, st>>>(m, s, p, b);
}
void launch_wbar(const DevMesh& m, const DevState& s, double* out, cudaStream_t st) {
    k_wbar<<<cdiv(5LL * m.nc, 256) < 4096 ? cdiv(5LL * m.nc, 256) : 4096, 256, 0, st>>>(m, s, out);
}
void launch_kn_gll(const DevMesh& m, const DevState& s, const DevParams& p, double* out, cudaStream_t st) {
    k_kn_gll<<<cdiv(m.nc, 256), 256, 0, st>>>(m, s, p, out);
}
void launch_prim_moments(const DevMesh& m, const DevState& s, const DevParams& p, int which, double* out,
                         cudaStream_t st) {
    if (which == UGKWP_PRIM) k_prim_out<<<cdiv(m.nc, 256), 256, 0, st>>>(m, s, p, out);
    else k_wp_out<<<cdiv(m.nc, 256), 256, 0, st>>>(m, s, p, which, out);
}

}  // namespace ugkwp
