// Particle kernels of the UGKWP step, templated on the particle precision
// (double: FP64 mode; float: MIXED mode).  Compiled with --fmad=false so that
// every particle trajectory and fixed-point flux is reproducible bit for bit.
//
//   k_sample_write  a5: N_sam hydro particles per cell, in pairs U +/- sqrt(RT) X
//                   with X ~ N(0, I) (Box-Muller), uniform in the tet.
//   k_track         a6-a9, a11: t_f = min(-tau ln eta, dt), face-by-face streaming
//                   of the cell-sorted particles, boundary interaction, the
//                   counting flux of the particles that left their cell or met a
//                   wall, removal; each survivor is written into the bucket of
//                   its end cell in the next buffer.
#include <algorithm>
#include <type_traits>

#include "dmath.cuh"
#include "fixed.cuh"
#include "ugkwp_internal.hpp"

namespace ugkwp {

namespace {

constexpr unsigned FULL = 0xffffffffu;

enum : unsigned long long { TAG_TF = 1, TAG_SVEL = 2, TAG_SPOS = 3, TAG_WALL = 4, TAG_GP = 5, TAG_SINT = 6, TAG_WINT = 7 };

__device__ __forceinline__ void set_err(const DevState& s, int32_t bits) {
    atomicOr(reinterpret_cast<unsigned long long*>(&s.cnt64[CNT_ERR]), (unsigned long long)bits);
}

// A failed self-check of a kernel: the error bit, and the first failure's
// check number and value (the access it guards is skipped).
__device__ __forceinline__ void check_failed(const DevState& s, int check, unsigned long long value) {
    atomicCAS(reinterpret_cast<unsigned long long*>(&s.cnt64[CNT_CHECK]), 0ULL,
              ((unsigned long long)check << 48) | (value & 0xffffffffffffULL));
    set_err(s, ERRB_CHECK);
}

__device__ __forceinline__ unsigned long long make_id(long long step, int cell, int k) {
    return ((unsigned long long)step << 40) | ((unsigned long long)cell << 16) | (unsigned long long)k;
}

// The arrays of buffer 0 shifted by `d` bytes (0 or the distance to buffer 1).
template <class Real> __device__ __forceinline__ PartView<Real> view(const PartBufRaw& r, long long d) {
    auto at = [d](void* q) { return static_cast<void*>(static_cast<char*>(q) + d); };
    PartView<Real> v;
    for (int c = 0; c < 3; ++c) {
        v.x[c] = (Real*)at(r.x[c]);
        v.u[c] = (Real*)at(r.u[c]);
    }
    v.m = (double*)at(r.m);
    v.cell = (int32_t*)at(r.cell);
    v.id = (uint64_t*)at(r.id);
    v.e = r.e ? (Real*)at(r.e) : nullptr;
    return v;
}

// ------------------------------------------------------------------ sampling
// The three normals X of the pair whose first member has id `ida`: Box-Muller
// in the particle precision (binary32 in the mixed mode).  The pair's two members
// sit in neighbouring lanes (side 0, 1) and each evaluates one of the two
// Box-Muller pairs of the draw (the fourth normal is not used); every lane of the
// warp takes part in the exchange.
template <class Real>
__device__ __forceinline__ void pair_normals(unsigned long long ida, long long step, unsigned long long seed, int side,
                                             Real X[3]) {
    const dm::U4 r = dm::philox(ida, (unsigned long long)step, TAG_SVEL, 0ULL, seed, 0ULL);
    const unsigned long long ru = side == 0 ? r.a : r.c, ra = side == 0 ? r.b : r.d;
    Real rad, sn, cs;
    if constexpr (sizeof(Real) == 4) {
        rad = sqrtf(-2.0f * dm::f_log(dm::u01f(ru)));
        dm::f_sincos2pi(dm::u01f(ra), &sn, &cs);
    } else {
        rad = sqrt(-2.0 * dm::d_log(dm::u01d(ru)));
        dm::d_sincos2pi(dm::u01d(ra), &sn, &cs);
    }
    const Real c = rad * cs, d = rad * sn;
    const Real oc = __shfl_xor_sync(FULL, c, 1), od = __shfl_xor_sync(FULL, d, 1);
    X[0] = side == 0 ? c : oc;
    X[1] = side == 0 ? d : od;
    X[2] = side == 0 ? oc : c;
}

// Internal energy of a particle with K internal degrees of freedom at spread
// sig = sqrt(RT): e = sum_{i<K} (sig N_i)^2, the normals by Box-Muller from
// Philox counters (id, step, tag, idx0 + j), four per counter, summed in
// order in the particle precision.
template <class Real>
__device__ __forceinline__ Real internal_energy(unsigned long long id, long long step, unsigned long long tag,
                                                unsigned long long idx0, int K, Real sig, unsigned long long seed) {
    Real e = (Real)0;
    for (int j = 0; 4 * j < K; ++j) {
        const dm::U4 r = dm::philox(id, (unsigned long long)step, tag, idx0 + (unsigned long long)j, seed, 0ULL);
        Real N[4];
        if constexpr (sizeof(Real) == 4) {
            float sn, cs;
            float rad = sqrtf(-2.0f * dm::f_log(dm::u01f(r.a)));
            dm::f_sincos2pi(dm::u01f(r.b), &sn, &cs);
            N[0] = rad * cs;
            N[1] = rad * sn;
            rad = sqrtf(-2.0f * dm::f_log(dm::u01f(r.c)));
            dm::f_sincos2pi(dm::u01f(r.d), &sn, &cs);
            N[2] = rad * cs;
            N[3] = rad * sn;
        } else {
            double sn, cs;
            double rad = sqrt(-2.0 * dm::d_log(dm::u01d(r.a)));
            dm::d_sincos2pi(dm::u01d(r.b), &sn, &cs);
            N[0] = rad * cs;
            N[1] = rad * sn;
            rad = sqrt(-2.0 * dm::d_log(dm::u01d(r.c)));
            dm::d_sincos2pi(dm::u01d(r.d), &sn, &cs);
            N[2] = rad * cs;
            N[3] = rad * sn;
        }
        for (int i = 0; i < 4 && 4 * j + i < K; ++i) {
            const Real si = sig * N[i];
            e = e + si * si;
        }
    }
    return e;
}

// First-order g_p sampling: X ~ N(0, I) (1 + phi(X)) for particle `id` by
// acceptance-rejection in the particle precision: attempt k draws three normals
// by Box-Muller from Philox counter (id, step, TAG_GP, 2k) and eta from
// (id, step, TAG_GP, 2k + 1); accepted if eta M <= 1 + phi(X), the last draw
// kept after GP_ATTEMPTS attempts.  Coefficients: the cell's GP_NC values.
template <class Real>
__device__ __forceinline__ void gp_normals(const double* gpc, int nc, int cell, unsigned long long id, long long step,
                                           unsigned long long seed, Real X[3]) {
    Real c[GP_NC];
#pragma unroll
    for (int k = 0; k < GP_NC; ++k) c[k] = (Real)gpc[(size_t)k * nc + cell];
    X[0] = X[1] = X[2] = (Real)0;
    for (int k = 0; k < GP_ATTEMPTS; ++k) {
        const dm::U4 r = dm::philox(id, (unsigned long long)step, TAG_GP, (unsigned long long)(2 * k), seed, 0ULL);
        const dm::U4 r2 = dm::philox(id, (unsigned long long)step, TAG_GP, (unsigned long long)(2 * k + 1), seed, 0ULL);
        Real eta;
        if constexpr (sizeof(Real) == 4) {
            float sn, cs;
            float rad = sqrtf(-2.0f * dm::f_log(dm::u01f(r.a)));
            dm::f_sincos2pi(dm::u01f(r.b), &sn, &cs);
            X[0] = rad * cs;
            X[1] = rad * sn;
            rad = sqrtf(-2.0f * dm::f_log(dm::u01f(r.c)));
            dm::f_sincos2pi(dm::u01f(r.d), &sn, &cs);
            X[2] = rad * cs;
            eta = dm::u01f(r2.a);
        } else {
            double sn, cs;
            double rad = sqrt(-2.0 * dm::d_log(dm::u01d(r.a)));
            dm::d_sincos2pi(dm::u01d(r.b), &sn, &cs);
            X[0] = rad * cs;
            X[1] = rad * sn;
            rad = sqrt(-2.0 * dm::d_log(dm::u01d(r.c)));
            dm::d_sincos2pi(dm::u01d(r.d), &sn, &cs);
            X[2] = rad * cs;
            eta = dm::u01d(r2.a);
        }
        // phi = a0 + L.X + X^T Q X + (C.X) |X|^2, in this order
        const Real lin = (c[1] * X[0] + c[2] * X[1]) + c[3] * X[2];
        const Real qd = ((c[4] * X[0]) * X[0] + (c[5] * X[1]) * X[1]) + (c[6] * X[2]) * X[2];
        const Real qo = ((c[7] * X[0]) * X[1] + (c[8] * X[0]) * X[2]) + (c[9] * X[1]) * X[2];
        const Real cub = ((c[10] * X[0] + c[11] * X[1]) + c[12] * X[2]) * ((X[0] * X[0] + X[1] * X[1]) + X[2] * X[2]);
        const Real phi = ((c[0] + lin) + (qd + (qo + qo))) + cub;
        if (eta * c[13] <= (Real)1 + phi) break;
    }
}

// a5 positions: a uniform point in the tet from three uniforms folded cube ->
// prism -> tet (Rocchini & Cignoni, J. Graphics Tools 5(4), 2000).  The
// uniforms are odd multiples of 2^-48 (47 bits of one Philox draw each) and
// the folding runs on their integer numerators, so both precisions start from
// the same exact barycentric weights w_k = N_k 2^-48.
__device__ __forceinline__ void tet_weights(const dm::U4& r, long long N[3]) {
    constexpr long long ONE = 1LL << 48;
    long long a = (long long)(((r.a >> 17) << 1) | 1ULL), b = (long long)(((r.b >> 17) << 1) | 1ULL),
              c = (long long)(((r.c >> 17) << 1) | 1ULL);
    if (a + b > ONE) { a = ONE - a; b = ONE - b; }
    if (b + c > ONE) {
        const long long t = c;
        c = ONE - a - b;
        b = ONE - t;
    } else if (a + b + c > ONE) {
        const long long t = c;
        c = a + b + c - ONE;
        a = ONE - b - t;
    }
    N[0] = a; N[1] = b; N[2] = c;
}

// Error-free sum of two binary32 numbers: s + e = a + b exactly (Knuth).
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// Mixed-mode position coordinate: (p0 - A) + ((w1 E1 + w2 E2) + w3 E3) in
// binary32 pairs (high + low, about 44 bits), then rounded to binary32.  f
// points at the coordinate's 8 table entries (stride nc): p0 - A, E1, E2, E3
// as (high, low).  Each product keeps the exact error of its high parts (FMA)
// and the two cross terms; the sums carry their exact errors in the low part.
__device__ __forceinline__ float ff_position(const float* f, int nc, const float wh[3], const float wl[3]) {
    float p[3], e[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float eh = f[(size_t)(2 + 2 * k) * nc], el = f[(size_t)(3 + 2 * k) * nc];
        p[k] = wh[k] * eh;
        e[k] = __fmaf_rn(wh[k], eh, -p[k]) + (wh[k] * el + wl[k] * eh);
    }
    float s1, r1;
    two_sum(p[0], p[1], s1, r1);
    float lo = r1 + (e[0] + e[1]);
    float s2, r2;
    two_sum(s1, p[2], s2, r2);
    lo = r2 + (lo + e[2]);
    float s3, r3;
    two_sum(f[0], s2, s3, r3);
    lo = r3 + (lo + f[nc]);
    return s3 + lo;
}

// The live slots of the buffer that holds the particles (CNT_PACK slots, holes among
// them) go to the start of the other one (their order changes no result): the rare
// step in place too many, see CNT_PACK.  The samples' slots follow theirs, so that one
// kernel writes both.
template <class Real>
__device__ __forceinline__ void pack_slots(const DevState& s, const PartBufs& bufs, Blk bk) {
    const long long n = s.cnt64[CNT_PACK], left = s.cnt64[CNT_N_A];
    if (n == 0) return;
    // (one address per buffer, the arrays at their distances from the first one:
    // the kernel takes 64 registers, the sampling alone 60; with an address per array 80)
    char* const to = static_cast<char*>(bufs.b0.x[0]) + s.cnt64[CNT_SRC] * bufs.delta;
    char* const from = static_cast<char*>(bufs.b0.x[0]) + s.cnt64[CNT_CUR] * bufs.delta;
    auto at = [&](char* buffer, const void* array) {
        return buffer + (static_cast<const char*>(array) - static_cast<const char*>(bufs.b0.x[0]));
    };
    auto move = [&](const void* array, auto type, long long i, long long j) {
        using T = decltype(type);
        reinterpret_cast<T*>(at(to, array))[j] = reinterpret_cast<const T*>(at(from, array))[i];
    };
    const int32_t* cells = reinterpret_cast<const int32_t*>(at(from, bufs.b0.cell));
    const int lane = threadIdx.x & 31;
    const long long stride = (long long)bk.n * blockDim.x;
#pragma unroll 1
    for (long long base = (long long)bk.id * blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
        const long long i = base + lane;
        const bool live = i < n && cells[i] >= 0;
        const unsigned mask = __ballot_sync(FULL, live);
        unsigned long long first = 0;
        if (lane == 0 && mask)
            first = atomicAdd(reinterpret_cast<unsigned long long*>(&s.cnt64[CNT_PACKED]), (unsigned long long)__popc(mask));
        const long long j = (long long)__shfl_sync(FULL, first, 0) + __popc(mask & ((1u << lane) - 1u));
        if (!live) continue;
        if (j >= left) {
            check_failed(s, 10, (unsigned long long)j);
            continue;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            move(bufs.b0.x[c], Real(), i, j);
            move(bufs.b0.u[c], Real(), i, j);
        }
        move(bufs.b0.m, double(), i, j);
        move(bufs.b0.cell, int32_t(), i, j);
        move(bufs.b0.id, uint64_t(), i, j);
        if (bufs.b0.e) move(bufs.b0.e, Real(), i, j);
    }
}

// One lane per sample; cells sample even numbers, so that the two members of a
// pair are lanes 2i and 2i + 1 and share the work of their normals (first-order
// g_p: each particle on its own).  With energy-matched sampling a pair's
// velocities hold its normals X until k_sample_scale has the cell's factor.  Bound
// by the binary64 pipe in binary64 (logarithms, square roots, sines and cosines),
// by the integer pipes (Philox4x64) in mixed mode.  20 binary64 steps of a tube of
// 9,600 tets, energy-matched: 2.94 ms; with both members evaluating all of the
// pair's normals, and the scale kernel all of them once more, 4.13 ms.
template <class Real>
__device__ __forceinline__ void sample_write_body(const DevMesh& m, const DevState& s, const DevParams& p,
                                                  const PartBufs& bufs, Blk bk) {
    if (__syncthreads_or(threadIdx.x == 0 && (s.cnt64[CNT_ERR] & ERRB_CAPACITY))) return;
    const PartView<Real> b = view<Real>(bufs.b0, bufs.dyn ? s.cnt64[CNT_SRC] * bufs.delta : 0);
    const int nc = m.nc, lane = threadIdx.x & 31;
    const long long total = s.cnt64[CNT_NSAM];
    const long long step = s.cnt64[CNT_STEP];
    const long long n_a = s.cnt64[CNT_N_A];
    const long long stride = (long long)bk.n * blockDim.x;
    const bool gp = p.sampling == UGKWP_SAMPLE_GP1, matched = p.sampling == UGKWP_SAMPLE_ENERGY_MATCHED;
    // warp-uniform bounds: every lane takes part in the exchange of normals
    for (long long base = (long long)bk.id * blockDim.x + (threadIdx.x & ~31); base < total; base += stride) {
        const long long g = min(base + lane, total - 1);  // (a lane past the end repeats the last sample)
        // owning cell: the last c with soff[c] <= g (cells with N_sam = 0 share
        // the offset of the next cell and are never the last such c)
        int lo = 0, hi = nc;  // invariant: soff[lo] <= g < soff[hi] (soff[nc] = +inf)
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (s.soff[mid] <= g) lo = mid; else hi = mid;
        }
        const int cell = lo;
        const int k = (int)(g - s.soff[cell]);
        const int side = lane & 1;  // = k & 1 for g < total
        const unsigned long long ida = make_id(step, cell, k & ~1);
        const unsigned long long id = ida + (unsigned long long)side;
        Real X[3];
        if (!gp) pair_normals<Real>(ida, step, p.seed, side, X);
        // the samples follow the current buffer's survivor slots, in cell order
        const long long j = n_a + g;
        if (base + lane >= total) continue;
        if (j >= p.capacity || cell < 0 || cell >= nc) {
            check_failed(s, 9, (unsigned long long)j);
            continue;
        }
        if (gp) gp_normals<Real>(s.gpc, nc, cell, id, step, p.seed, X);  // every particle on its own
        Real U[3], sig;
        if constexpr (sizeof(Real) == 4) {
            // mixed mode: velocities in binary32 from U and the spread rounded to binary32
            const float4 us = s.usig[cell];
            U[0] = us.x; U[1] = us.y; U[2] = us.z;
            sig = us.w;
        } else {
            for (int c = 0; c < 3; ++c) U[c] = s.prim[(size_t)(1 + c) * nc + cell];
            sig = sqrt(p.R * s.prim[(size_t)4 * nc + cell]);
        }
        long long N[3];
        tet_weights(dm::philox(id, (unsigned long long)step, TAG_SPOS, 0ULL, p.seed, 0ULL), N);
        if constexpr (sizeof(Real) == 4) {
            // the position offset from the tet's anchor in binary32 pairs, rounded once
            float wh[3], wl[3];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                wh[q] = (float)(N[q] >> 24) * 0x1p-24f;
                wl[q] = (float)(N[q] & 0xffffffLL) * 0x1p-48f;
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) b.x[c][j] = ff_position(m.smp_f + (size_t)(8 * c) * nc + cell, nc, wh, wl);
        } else {
            const double a = (double)N[0] * 0x1p-48, bb = (double)N[1] * 0x1p-48, cc = (double)N[2] * 0x1p-48;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double P0 = m.vtx[(size_t)c * nc + cell];
                const double E1 = m.vtx[(size_t)(3 + c) * nc + cell] - P0;
                const double E2 = m.vtx[(size_t)(6 + c) * nc + cell] - P0;
                const double E3 = m.vtx[(size_t)(9 + c) * nc + cell] - P0;
                b.x[c][j] = P0 + ((a * E1 + bb * E2) + cc * E3);
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (matched) b.u[c][j] = X[c];
            else b.u[c][j] = (gp || side == 0) ? U[c] + sig * X[c] : U[c] - sig * X[c];
        }
        if (p.K > 0) b.e[j] = internal_energy<Real>(id, step, TAG_SINT, 0ULL, p.K, sig, p.seed);
        b.m[j] = s.msam[cell];
        b.cell[j] = cell;
        b.id[j] = id;
    }
}
// DYN: the simulation may step in place.
template <class Real, bool DYN>
__global__ void __launch_bounds__(256) k_sample_write(DevMesh m, DevState s, DevParams p, PartBufs bufs) {
    const Blk bk{(int)blockIdx.x, (int)gridDim.x};
    if constexpr (DYN) pack_slots<Real>(s, bufs, bk);
    sample_write_body<Real>(m, s, p, bufs, bk);
}

// Energy-matched sampling: one factor per cell, s^2 sum_j |X_j|^2 = 3 N_sam / 2,
// so the pairs' thermal energy is exactly rho^hp |Omega| (3/2) R T.  The sum
// runs over the cell's pairs in order in binary64; the velocities are
// U +- s sqrt(RT) X.  A block takes CELL_BLOCK cells: a thread sums its cell's
// normals, which k_sample_write left in the velocities, then the block goes over
// its cells' samples, which lie in a row.
template <class Real>
__device__ __forceinline__ void sample_scale_body(const DevMesh& m, const DevState& s, const DevParams& p,
                                                  const PartBufs& bufs, Blk bk) {
    __shared__ int off[CELL_BLOCK + 1];
    __shared__ Real spread[CELL_BLOCK];
    if (__syncthreads_or(threadIdx.x == 0 && (s.cnt64[CNT_ERR] & ERRB_CAPACITY))) return;
    const PartView<Real> b = view<Real>(bufs.b0, bufs.dyn ? s.cnt64[CNT_SRC] * bufs.delta : 0);
    const int nc = m.nc, t = threadIdx.x, cell = bk.id * CELL_BLOCK + t;
    const long long n_a = s.cnt64[CNT_N_A];
    int ns = 0, so = 0;
    if (cell < nc) {
        ns = s.nsam[cell];
        so = s.soff[cell];
        double sig = sqrt(p.R * s.prim[(size_t)4 * nc + cell]);
        if (ns >= 2) {
            double S = 0.0;
            for (int j = 0; j < ns / 2; ++j) {
                const long long at = n_a + so + 2 * j;
                const double x0 = (double)b.u[0][at], x1 = (double)b.u[1][at], x2 = (double)b.u[2][at];
                S = S + ((x0 * x0 + x1 * x1) + x2 * x2);
            }
            if (S > 0.0) sig = sig * sqrt((double)(3 * (ns / 2)) / S);
        }
        spread[t] = (Real)sig;
    }
    const int last = min(CELL_BLOCK, nc - bk.id * CELL_BLOCK) - 1;
    off[t] = so;
    __syncthreads();
    if (t == last) off[last + 1] = so + ns;
    __syncthreads();
    const int first = off[0], end = off[last + 1];
    for (int g = first + t; g < end; g += CELL_BLOCK) {
        int lo = 0, hi = last + 1;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (off[mid] <= g) lo = mid; else hi = mid;
        }
        const int c0 = bk.id * CELL_BLOCK + lo;
        const Real sg = spread[lo];
        Real U[3];
        if constexpr (sizeof(Real) == 4) {
            const float4 us = s.usig[c0];
            U[0] = us.x; U[1] = us.y; U[2] = us.z;
        } else {
            for (int c = 0; c < 3; ++c) U[c] = s.prim[(size_t)(1 + c) * nc + c0];
        }
        const long long j = n_a + g;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const Real X = b.u[c][j];
            b.u[c][j] = ((g - off[lo]) & 1) == 0 ? U[c] + sg * X : U[c] - sg * X;
        }
    }
}
template <class Real>
__global__ void __launch_bounds__(CELL_BLOCK) k_sample_scale(DevMesh m, DevState s, DevParams p, PartBufs bufs) {
    sample_scale_body<Real>(m, s, p, bufs, Blk{(int)blockIdx.x, (int)gridDim.x});
}

// ------------------------------------------------------------------ tracking
template <class Real> struct Trk;
template <> struct Trk<float> {
    __device__ static __forceinline__ void plane(const DevMesh& m, int tet, int k, float& nx, float& ny, float& nz,
                                                 float& d) {
        const float4 v = m.trk_f[tet].pl[k];
        nx = v.x; ny = v.y; nz = v.z; d = v.w;
    }
    __device__ static __forceinline__ int4 nbv(const DevMesh& m, int tet) { return m.trk_f[tet].nb; }
    __device__ static __forceinline__ float tau(const DevState& s, int c) { return s.tauf[c]; }
    __device__ static __forceinline__ float tf(float tau, unsigned long long r) {
        return -(tau * dm::f_log(dm::u01f(r)));
    }
};
template <> struct Trk<double> {
    __device__ static __forceinline__ void plane(const DevMesh& m, int tet, int k, double& nx, double& ny,
                                                 double& nz, double& d) {
        const Dbl4 v = m.trk_d[tet].pl[k];
        nx = v.x; ny = v.y; nz = v.z; d = v.w;
    }
    __device__ static __forceinline__ int4 nbv(const DevMesh& m, int tet) { return m.trk_d[tet].nb; }
    __device__ static __forceinline__ double tau(const DevState& s, int c) { return s.tau[c]; }
    __device__ static __forceinline__ double tf(double tau, unsigned long long r) {
        return -(tau * dm::d_log(dm::u01d(r)));
    }
};

// ---- the walk of one particle, one tet at a time
// Walk state along x0 + u (t - t0): the tet it is in, the face it entered
// through (or last reflected from, skipped in the exit test), its counters.
template <class Real> struct Walk {
    Real x0[3], u[3], t0, t_end;
    int tet, last, ncross, nrefl, nwall, status;
};

// Binary32 of a walk's value by truncation, with integer operations only (a
// conversion would run on the binary64 pipe, which bounds the binary64 mode);
// values below 2^-126 become 0, values of 2^128 and more, infinities and NaNs
// become infinity (no test holds for those).
__device__ __forceinline__ float truncated(float v) { return v; }
__device__ __forceinline__ float truncated(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), mag = hi & 0x7fffffffu;
    unsigned f = ((mag - 0x38000000u) << 3) | ((unsigned)__double2loint(v) >> 29);
    f = mag < 0x38100000u ? 0u : mag >= 0x47f00000u ? 0x7f800000u : f;
    return __uint_as_float(f | (hi & 0x80000000u));
}

// The exit face of a tet decided in binary32 (binary64 mode): k >= 0 the face, -1
// the walk stops in the tet, -2 undecided.  un_k = u.n_k and num_k = d_k - n_k.x0
// carry absolute errors below eu = 2^-20 |u|_1 (truncated u, rounded n, three
// products: 8 2^-24 |u|_1) and en = the inside test's margin; a comparison counts
// only beyond these and beyond 2^-20 of its own products, so that it agrees with
// the binary64 comparison, whose roundings are 2^-29 of that.  About one visit in
// 300 is undecided (21^3 cavity); one visit in binary64 costs ~70 instructions of
// the pipe that bounds this mode.
struct Ray32 {
    float x[3], u[3], eu;
};
template <class Real> __device__ __forceinline__ void ray_start(Ray32& r, const Real* x0, const Real* u) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        r.x[c] = truncated(x0[c]);
        r.u[c] = truncated(u[c]);
    }
    r.eu = (fabsf(r.u[0]) + fabsf(r.u[1]) + fabsf(r.u[2])) * 0x1p-20f;
}
__device__ __forceinline__ int exit_face32(const DevMesh& m, const Ray32& r, int tet, int last, float rem) {
    const float4* pl = m.pln_f + (size_t)4 * tet;
    const float en = m.margin[tet];
    float un[4], num[4];
    bool sure = true;
    int best = -1;
    float bn = 0.0f, bu = 1.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float4 P = pl[k];
        un[k] = __fmaf_rn(r.u[0], P.x, __fmaf_rn(r.u[1], P.y, r.u[2] * P.z));
        num[k] = __fmaf_rn(-r.x[0], P.x, __fmaf_rn(-r.x[1], P.y, __fmaf_rn(-r.x[2], P.z, P.w)));
        if (k == last) un[k] = -1.0f;
        else sure = sure && fabsf(un[k]) > r.eu;
        if (un[k] > 0.0f && (best < 0 || num[k] * bu < bn * un[k])) {
            best = k;
            bn = num[k];
            bu = un[k];
        }
    }
    if (!sure) return -2;
    if (best < 0) return -1;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (k == best || un[k] < 0.0f) continue;
        const float a = num[k] * bu, b = bn * un[k];
        const float tol = en * (bu + un[k]) + r.eu * (fabsf(num[k]) + fabsf(bn)) + 0x1p-20f * (fabsf(a) + fabsf(b));
        sure = sure && a - b > tol;
    }
    const float t = rem * bu, tol = en + r.eu * rem + 0x1p-20f * (t + fabsf(bn));
    if (!(sure && fabsf(bn - t) > tol)) return -2;
    return bn < t ? best : -1;
}

// One tet of the face-by-face walk (Sec. 2.2 streaming): the exit face is the
// one with u.n > 0 and the smallest crossing time (d - n.x0)/(u.n), compared
// by cross products (positive denominators) with one division; ties keep the
// lower local face.  Returns true when the walk goes on (into the neighbour,
// or restarted at a wall); false when it ended: stopped inside the tet (xe the
// end point), left the domain (status 2) or passed max_crossings (status 4).
template <class Real, bool KE>
__device__ __forceinline__ bool visit(const DevMesh& m, const DevParams& p, long long step, unsigned long long id,
                                      Walk<Real>& w, Ray32& ray, Real xe[3], Real& ee) {
    if constexpr (sizeof(Real) == 8) {
        // an interior face or an open boundary leaves the ray as it is: the face is
        // all that is needed, and binary32 decides it
        const Real rem = w.t_end - w.t0;
        const int k = exit_face32(m, ray, w.tet, w.last, truncated(rem));
        if (k == -1) {
#pragma unroll
            for (int c = 0; c < 3; ++c) xe[c] = w.x0[c] + w.u[c] * rem;
            return false;
        }
        if (k >= 0 && w.ncross < p.max_crossings) {
            const int4 nbv = Trk<Real>::nbv(m, w.tet);
            const int code = k == 0 ? nbv.x : k == 1 ? nbv.y : k == 2 ? nbv.z : nbv.w;
            if (code >= 0) {
                ++w.ncross;
                w.tet = code >> 2;
                w.last = code & 3;
                return true;
            }
        }
    }
    // the tet's neighbour codes, loaded with its planes (they sit in
    // another sector of the tet's record)
    const int4 nbv = Trk<Real>::nbv(m, w.tet);
    int best = -1;
    Real nbest = (Real)0, dbest = (Real)1;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (k == w.last) continue;
        Real nx, ny, nz, d;
        Trk<Real>::plane(m, w.tet, k, nx, ny, nz, d);
        const Real un = (w.u[0] * nx + w.u[1] * ny) + w.u[2] * nz;
        if (un > (Real)0) {
            const Real xn = (w.x0[0] * nx + w.x0[1] * ny) + w.x0[2] * nz;
            const Real num = d - xn;
            if (best < 0 || num * dbest < nbest * un) { best = k; nbest = num; dbest = un; }
        }
    }
    Real sbest = best >= 0 ? nbest / dbest : (Real)0;
    const Real rem = w.t_end - w.t0;
    if (best < 0 || sbest >= rem) {
#pragma unroll
        for (int c = 0; c < 3; ++c) xe[c] = w.x0[c] + w.u[c] * rem;
        return false;
    }
    if (sbest < (Real)0) sbest = (Real)0;
    ++w.ncross;
    if (w.ncross > p.max_crossings) {
        w.status |= 4;
#pragma unroll
        for (int c = 0; c < 3; ++c) xe[c] = w.x0[c];
        return false;
    }
    const int code = best == 0 ? nbv.x : best == 1 ? nbv.y : best == 2 ? nbv.z : nbv.w;
    if (code >= 0) {
        const int nt = code >> 2;
        if constexpr (sizeof(Real) == 4) {
            // mixed mode: the segment start moves into the next tet's frame
            // (the anchors' difference, exact in binary32, sits in the
            // record's line loaded for the planes)
            const float* da = m.trk_f[w.tet].da + 3 * best;
            w.x0[0] = w.x0[0] + da[0];
            w.x0[1] = w.x0[1] + da[1];
            w.x0[2] = w.x0[2] + da[2];
        }
        w.tet = nt;
        w.last = code & 3;
        return true;
    }
    const int bi = -1 - code;
    const DevBc& bc = p.bc[m.bf_tag[bi]];
    if (bc.type == UGKWP_BC_FARFIELD || bc.type == UGKWP_BC_OUTFLOW) {
        w.status |= 2;
        return false;
    }
    Real xh[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) xh[c] = w.x0[c] + w.u[c] * sbest;
    if (bc.type == UGKWP_BC_SPECULAR) {
        Real nx, ny, nz, d;
        Trk<Real>::plane(m, w.tet, best, nx, ny, nz, d);
        const Real un = (w.u[0] * nx + w.u[1] * ny) + w.u[2] * nz;
        const Real two = un + un;
        w.u[0] = w.u[0] - two * nx;
        w.u[1] = w.u[1] - two * ny;
        w.u[2] = w.u[2] - two * nz;
    } else {
        // diffuse re-emission, full accommodation: |u_n| = sqrt(-2 R T_w ln eta),
        // tangential components U_w,t + sqrt(R T_w) N(0,1)
        const dm::U4 r = dm::philox(id, (unsigned long long)step, TAG_WALL, (unsigned long long)w.nwall, p.seed, 0ULL);
        if constexpr (sizeof(Real) == 4) {
            // mixed mode: binary32 from the wall constants and the face frame
            // rounded to binary32
            const float vn = sqrtf(bc.c2rt_f * dm::f_log(dm::u01f(r.a)));
            const float rad = sqrtf(-2.0f * dm::f_log(dm::u01f(r.b)));
            float sn, cs;
            dm::f_sincos2pi(dm::u01f(r.c), &sn, &cs);
            const int nbf = m.nbf;
            const float v1 = m.bf_f[(size_t)9 * nbf + bi] + bc.sw_f * (rad * cs);
            const float v2 = m.bf_f[(size_t)10 * nbf + bi] + bc.sw_f * (rad * sn);
#pragma unroll
            for (int c = 0; c < 3; ++c)
                w.u[c] = ((-vn) * m.bf_f[(size_t)c * nbf + bi] + v1 * m.bf_f[(size_t)(3 + c) * nbf + bi]) +
                         v2 * m.bf_f[(size_t)(6 + c) * nbf + bi];
            if constexpr (KE)
                ee = internal_energy<float>(id, step, TAG_WINT, 2ULL * (unsigned long long)w.nwall, p.K, bc.sw_f, p.seed);
        } else {
            const double vn = sqrt(-2.0 * p.R * bc.T_w * dm::d_log(dm::u01d(r.a)));
            const double rad = sqrt(-2.0 * dm::d_log(dm::u01d(r.b)));
            double sn, cs;
            dm::d_sincos2pi(dm::u01d(r.c), &sn, &cs);
            const double sw = sqrt(p.R * bc.T_w);
            const int nbf = m.nbf;
            double n3[3], t1[3], t2[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                n3[c] = m.bf_n[(size_t)c * nbf + bi];
                t1[c] = m.bf_t1[(size_t)c * nbf + bi];
                t2[c] = m.bf_t2[(size_t)c * nbf + bi];
            }
            const double v1 = ((bc.U_w[0] * t1[0] + bc.U_w[1] * t1[1]) + bc.U_w[2] * t1[2]) + sw * (rad * cs);
            const double v2 = ((bc.U_w[0] * t2[0] + bc.U_w[1] * t2[1]) + bc.U_w[2] * t2[2]) + sw * (rad * sn);
#pragma unroll
            for (int c = 0; c < 3; ++c) w.u[c] = (Real)(((-vn) * n3[c] + v1 * t1[c]) + v2 * t2[c]);
            if constexpr (KE)
                ee = (Real)internal_energy<double>(id, step, TAG_WINT, 2ULL * (unsigned long long)w.nwall, p.K, sw, p.seed);
        }
        ++w.nwall;
    }
    ++w.nrefl;
#pragma unroll
    for (int c = 0; c < 3; ++c) w.x0[c] = xh[c];
    w.t0 = w.t0 + sbest;
    w.last = best;
    if constexpr (sizeof(Real) == 8) ray_start(ray, w.x0, w.u);
    return true;
}

// Entries of a warp's queue of particles that may leave their tet: fewer than 32
// wait before a tile is taken and a tile adds at most 32.
constexpr int WALK_QUEUE = 64;
// Lanes of a tile above the collision threshold up to which binary64 defers their
// logarithm to the queue: two steps of the 21^3 cavity in binary64 2.22 ms with 4,
// 8 or 16 against 2.52 ms with none.
constexpr int DEFER_LOG = 8;
// Slots of a run of tiles at most.
constexpr unsigned TRACK_RUN_MAX = 512;
// Threads per SM the tracking kernel is compiled for: 64 registers in mixed mode
// (80: 1.82 ms against 1.69 ms for two steps of the 24^3 cavity, whose wave flux
// leaves room for four such blocks per SM); in binary64 five blocks of 128 threads
// with 96 registers (a 20-step run of a tube of 9,600 tets 4.43 ms against 4.71 ms
// with 64), or two of 256 with up to 128.
template <class Real> constexpr int TRACK_PER_SM = sizeof(Real) == 4 ? 1024 : 640;

// The planes of a tet in binary32, for the inside test: in mixed mode those of
// the tracking record (relative to the anchor), else rounded from binary64.
template <class Real> __device__ __forceinline__ const float4* test_planes(const DevMesh& m, int c) {
    if constexpr (sizeof(Real) == 4) return m.trk_f[c].pl;
    else return m.pln_f + (size_t)4 * c;
}

// One warp's share of the tracking.  Warps work on their own (no block barrier):
// each takes runs of 32-slot tiles from a global counter, one atomic per run,
// reserved one run ahead.
//
// Per tile, one slot per lane:
//  * the collision test compares the t_f draw with a per-cell threshold that lies
//    below e^{-dt/tau}; only the lanes above it need -tau ln eta, and a warp
//    without such a lane skips the logarithm (DevState::cinfo);
//  * the end point x0 + u t is tested against the tet's four planes in binary32.
//    If it lies inside all of them by more than the cell's margin, which bounds
//    the rounding of that test and of the walk's own exit test, then the walk
//    (visit) would stop in this tet at the same point, bit for bit;
//  * the others wait in the warp's queue until 32 of them have gathered, and
//    are then walked face by face in a full warp.
// Nine tenths of the particles of a rarefied cavity end in the tile pass.  They
// change no sum: a cell's survivor mass starts the step from its survivors and
// samples (k_sample_count), and only what is removed or moves is added to it.
//
// Mixed mode is bound by memory latency: beside the wave flux 15 warps per SM are
// active and issue is 27% busy, long-scoreboard stalls 6.8 cycles per issue (16^3
// cavity).  Binary64 is bound by its pipe: what is left there per particle are the
// end point (6 instructions), and per queued particle the logarithm, the last
// segment, walls and the counting flux; the exit faces are decided in binary32
// (exit_face32).  Two steps of the settled 24^3 cavity, mixed, 1.60 ms; of the 21^3
// cavity in binary64 2.17 ms; with the walk of every first tet, block-wide output
// rounds and a mover list for a flux kernel of its own 2.20 and 7.33 ms, with
// every exit face decided in binary64 and no prefetch of the next tile's lines
// 1.78 and 2.99 ms.
//
// IN_PLACE (k_scan_apply chooses per step): a particle keeps its slot, a stayer
// writes its position only, a removed one leaves a hole.  Otherwise each survivor
// is written into the bucket of its end cell in the other buffer.
template <class Real, int THREADS> struct TrackShared {
    int q_slot[THREADS / 32][WALK_QUEUE];
    Real q_end[THREADS / 32][WALK_QUEUE];  // t_f, or dt; -1: not drawn yet
    unsigned red[THREADS / 32][8];
};
// Number: the type of the runs' numbers (fewer than 2^27, see track_blocks).  32 bits in
// the kernel of one simulation (20 binary64 steps of a tube of 9,600 tets 1% faster than
// with 64), 64 in the fused one, which then spills less (a batch of 14 members 7.08
// against 7.18 ms).
template <class Real, bool KE, int THREADS, bool IN_PLACE, class Number>
__device__ __forceinline__ void track_mode(const DevMesh& m, const DevState& s, const DevParams& p, const PartBufs& bufs,
                                           long long src, TrackShared<Real, THREADS>& sh) {
    constexpr int NW = THREADS / 32;
    auto& q_slot = sh.q_slot;
    auto& q_end = sh.q_end;
    auto& sh_red = sh.red;
    const PartBufRaw& br = bufs.b0;
    const PartView<Real> b = view<Real>(br, src);                 // this step's particles (holes: cell -1)
    // sorting: the next step's (src is 0 or delta; without DYN always 0)
    const PartView<Real> nxt = view<Real>(br, bufs.delta - src);
    const unsigned n = (unsigned)s.cnt64[CNT_N_B];
    const long long step = s.cnt64[CNT_STEP];
    const long long wtot = s.cnt64[CNT_WTOT];  // overflow slots start after the buckets
    const Real dtR = (Real)s.dt[0];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u, upto = FULL >> (31 - lane);
    const int nc = m.nc;
    Number* tile_ctr = reinterpret_cast<Number*>(&s.cnt64[CNT_TILE]);  // (or its low word)
    unsigned long long* smass = reinterpret_cast<unsigned long long*>(s.smass_next);
    unsigned long long* pf = reinterpret_cast<unsigned long long*>(s.pflux);
    // warp-uniform counters
    unsigned c_valid = 0, c_coll = 0, c_surv = 0, c_mover = 0;
    unsigned c_exit = 0, c_lost = 0, c_cross = 0, c_wall = 0;  // per lane
    int qn = 0;

    // the slot of a survivor in its end cell's bucket (rank: its place among the
    // cell's survivors), or in the overflow region behind the buckets; -1: none
    const int cap = (int)p.capacity;  // < 2^31
    auto slot_of = [&](int rank, int woff, int wcap) -> int {
        int j = woff + rank;
        if (rank >= wcap) {
            const long long o = (long long)atomicAdd(reinterpret_cast<unsigned long long*>(&s.cnt64[CNT_OVF]), 1ULL);
            j = -1;
            if (o < cap - wtot) j = (int)(wtot + o);
            else set_err(s, ERRB_CAPACITY);
        }
        if (j >= cap) {
            check_failed(s, 6, (unsigned long long)j);
            j = -1;
        }
        return j;
    };

    // ---- the last `take` (<= 32) particles of the queue: the walk, the counting
    // flux (-phi at the start cell, +phi at the end cell unless the particle left
    // the domain; a particle that ends in its start cell with its velocity
    // unchanged contributes nothing), the survivors' mass, removal (a9)
    auto drain = [&](int take) {
        const int k = qn - take + lane;
        const bool act = lane < take;
        qn -= take;
        __syncwarp();
        Walk<Real> w;
        Real us[3] = {(Real)0, (Real)0, (Real)0}, xe[3] = {(Real)0, (Real)0, (Real)0}, es = (Real)0, ee = (Real)0;
        double mm = 0.0;
        int c0 = -1, i = 0;
        unsigned long long id = 0;
        bool survivor = false, mover = false, exited = false;
        w.tet = -1;
        w.u[0] = w.u[1] = w.u[2] = (Real)0;
        w.nrefl = 0;
        if (act) {
            i = q_slot[warp][k];
            w.t_end = q_end[warp][k];
            c0 = b.cell[i];
            id = b.id[i];
            mm = b.m[i];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                w.x0[c] = b.x[c][i];
                w.u[c] = us[c] = b.u[c][i];
            }
            if constexpr (KE) es = ee = b.e[i];
            if constexpr (sizeof(Real) == 8) {
                if (w.t_end < (Real)0) {  // deferred
                    const unsigned long long r =
                        dm::philox32_2((unsigned)id, (unsigned)(id >> 32), (unsigned)step, (unsigned)TAG_TF,
                                       (unsigned)p.seed, (unsigned)(p.seed >> 32));
                    const Real tf = Trk<Real>::tf(Trk<Real>::tau(s, c0), r);
                    w.t_end = tf < dtR ? tf : dtR;
                }
            }
            const bool coll = w.t_end < dtR;
            w.t0 = (Real)0;
            w.tet = c0;
            w.last = -1;
            w.ncross = w.nwall = w.status = 0;
            Ray32 ray;
            if constexpr (sizeof(Real) == 8) ray_start(ray, w.x0, w.u);
            while (visit<Real, KE>(m, p, step, id, w, ray, xe, ee)) {
            }
            exited = w.status & 2;
            const bool lost = w.status & 4;
            survivor = !exited && (!coll || lost);
            mover = exited || w.tet != c0 || w.nrefl > 0;
            c_exit += exited;
            c_lost += lost;
            c_cross += w.ncross;
            c_wall += w.nwall;
            c_coll += coll && !lost && !exited;
        }
        __syncwarp();
        c_mover += __popc(__ballot_sync(FULL, mover));
        long long q0[5] = {0, 0, 0, 0, 0};
        if (__any_sync(FULL, mover)) {
            if (mover) {
                if (!phi_q(us, es, mm, p, q0)) set_err(s, ERRB_FIXED_OVERFLOW);
                if (!exited) {
                    if (w.nrefl == 0) {
#pragma unroll
                        for (int q = 0; q < 5; ++q) atomicAdd(&pf[(size_t)q * nc + w.tet], (unsigned long long)q0[q]);
                    } else {
                        long long q1[5];
                        if (!phi_q(w.u, ee, mm, p, q1)) set_err(s, ERRB_FIXED_OVERFLOW);
#pragma unroll
                        for (int q = 0; q < 5; ++q) atomicAdd(&pf[(size_t)q * nc + w.tet], (unsigned long long)q1[q]);
                    }
                }
            }
            if (mover) {
#pragma unroll
                for (int q = 0; q < 5; ++q) atomicAdd(&pf[(size_t)q * nc + c0], (unsigned long long)(-q0[q]));
            }
        }
        // survivors' mass: out of the start cell, into the end cell
        const bool stays = survivor && w.tet == c0;
        if (act && !mover && !stays && !fixed_of_mass(mm, p.exps[0], q0[0])) set_err(s, ERRB_FIXED_OVERFLOW);
        if (act && !stays) {
            atomicAdd(&smass[c0], (unsigned long long)(-q0[0]));
            if constexpr (IN_PLACE) atomicAdd(&s.nleft_next[c0], -1);
        }
        if (survivor && !stays) {
            atomicAdd(&smass[w.tet], (unsigned long long)q0[0]);
            if constexpr (IN_PLACE) atomicAdd(&s.nleft_next[w.tet], 1);
        }
        c_surv += __popc(__ballot_sync(FULL, survivor));
        if constexpr (IN_PLACE) {
            if (act) {
                if (!stays) b.cell[i] = survivor ? w.tet : -1;
                if (survivor) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) b.x[c][i] = xe[c];
                    if (w.nrefl > 0) {
#pragma unroll
                        for (int c = 0; c < 3; ++c) b.u[c][i] = w.u[c];
                        if constexpr (KE) b.e[i] = ee;
                    }
                }
            }
            return;
        }
        // a11: lanes with the same end cell take consecutive places of its bucket
        const int key = survivor ? w.tet : -1;
        const unsigned peers = __match_any_sync(FULL, key);
        const int leader = __ffs(peers) - 1;
        int first = 0;
        if (lane == leader && key >= 0) first = atomicAdd(&s.fill[key], __popc(peers));
        first = __shfl_sync(FULL, first, leader);
        if (survivor) {
            const int j = slot_of(first + __popc(peers & lt), s.woff[key], s.wcap[key]);
            if (j >= 0) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    nxt.x[c][j] = xe[c];
                    nxt.u[c][j] = w.u[c];
                }
                nxt.m[j] = mm;
                nxt.cell[j] = key;
                nxt.id[j] = id;
                if constexpr (KE) nxt.e[j] = ee;
            }
        }
    };

    // tiles per run: long enough that the counter is off the path, short enough
    // that a small simulation spreads over the whole grid
    const unsigned run = min(max(n / (32u * 8192u), 1u), TRACK_RUN_MAX / 32u) * 32u;
    Number ahead = 0;
    unsigned base = 0, end = 0;
    if (lane == 0) ahead = atomicAdd(tile_ctr, Number(1));
    base = (unsigned)__shfl_sync(FULL, ahead, 0) * run;
    end = base + run;
    if (lane == 0) ahead = atomicAdd(tile_ctr, Number(1));
    // the first lanes prefetch the lines of the next tile's x, u, m and id (its
    // cells are loaded), one line per lane, with one instruction per tile
    constexpr int XL = sizeof(Real) / 4;  // lines per coordinate array
    const char* pptr = nullptr;
    unsigned pstr = 0;
    if (lane < 6 * XL) {
        const int a = lane / XL;
        pptr = reinterpret_cast<const char*>(a < 3 ? br.x[a] : br.u[a - 3]) + src + (lane % XL) * 128;
        pstr = sizeof(Real);
    } else if (!IN_PLACE && lane < 6 * XL + 2) {
        pptr = reinterpret_cast<const char*>(br.m) + src + (lane - 6 * XL) * 128;
        pstr = 8;
    } else if (lane >= 6 * XL + 2 && lane < 6 * XL + 4) {
        pptr = reinterpret_cast<const char*>(br.id) + src + (lane - 6 * XL - 2) * 128;
        pstr = 8;
    }
    int cell_i = -1;
    if (base < n) cell_i = b.cell[base + lane];
    while (base < n) {
        const unsigned i = base + lane;
        const int c0 = i < n ? cell_i : -1;
        const bool valid = c0 >= 0;
        // the whole slot at once (the arrays hold whole tiles, so slots past n
        // are inside them and ignored); a start cell of -1 marks a hole
        const unsigned long long id = b.id[i];
        Real x0[3], u[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            x0[c] = b.x[c][i];
            u[c] = b.u[c][i];
        }
        double mm = 0.0;
        Real es = (Real)0;
        if constexpr (!IN_PLACE) {
            mm = b.m[i];
            if constexpr (KE) es = b.e[i];
        }
        const int cc = valid ? c0 : 0;
        const int4 info = s.cinfo[cc];
        const float4* pl = test_planes<Real>(m, cc);
        float4 P[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) P[k] = pl[k];
        // the next tile's cells (its other loads follow at the top of its turn)
        unsigned nbase = base + 32;
        if (nbase == end) {
            nbase = (unsigned)__shfl_sync(FULL, ahead, 0) * run;
            end = nbase + run;
            if (lane == 0 && nbase < n) ahead = atomicAdd(tile_ctr, Number(1));
        }
        if (nbase < n) {
            cell_i = b.cell[nbase + lane];
            if (pptr) asm volatile("prefetch.global.L1 [%0];" ::"l"(pptr + (size_t)nbase * pstr));
        }
        // a6: t_f = min(-tau ln eta, dt) for the particles left from the last step;
        // Philox4x32-10, counter (id low, id high, step, TAG_TF), key (seed low, seed high)
        Real t_end = dtR;
        const bool old = valid && (long long)(id >> 40) != step;
        unsigned long long r = 0;
        if (old)
            r = dm::philox32_2((unsigned)id, (unsigned)(id >> 32), (unsigned)step, (unsigned)TAG_TF, (unsigned)p.seed,
                               (unsigned)(p.seed >> 32));
        const bool maybe = old && (unsigned)(r >> 32) >= (unsigned)info.x;
        // a few lanes: in binary64 they wait for the queue, so that the logarithm
        // takes the binary64 pipe once per 32 of them
        const int n_maybe = __popc(__ballot_sync(FULL, maybe));
        const bool defer = sizeof(Real) == 8 && n_maybe <= DEFER_LOG && maybe;
        if (n_maybe > (sizeof(Real) == 8 ? DEFER_LOG : 0)) {
            if (maybe) {
                const Real tf = Trk<Real>::tf(Trk<Real>::tau(s, c0), r);
                if (tf < dtR) t_end = tf;
            }
        }
        const bool coll = t_end < dtR;
        // a7: the end point and the inside test
        Real xe[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) xe[c] = x0[c] + u[c] * t_end;
        const float f0 = truncated(xe[0]), f1 = truncated(xe[1]), f2 = truncated(xe[2]), margin = __int_as_float(info.w);
        float gap = 1.0f;
        bool inside = true;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            gap = __fmaf_rn(-P[k].x, f0, __fmaf_rn(-P[k].y, f1, __fmaf_rn(-P[k].z, f2, P[k].w)));
            inside = inside && gap > margin;
        }
        inside = inside && !defer;
        const bool slow = valid && !inside;
        const bool surv = valid && inside && !coll, gone = valid && inside && coll;
        const unsigned smask = __ballot_sync(FULL, surv), qmask = __ballot_sync(FULL, slow);
        int first = 0, start = 0;
        unsigned mine = 0;
        if constexpr (!IN_PLACE) {
            // runs of equal cells: one place in the bucket per survivor
            const int prev = __shfl_up_sync(FULL, c0, 1);
            const unsigned heads = __ballot_sync(FULL, lane == 0 || prev != c0);
            start = 31 - __clz(heads & upto);
            const unsigned above = heads & ~upto;
            const unsigned members = (above ? (above & (0u - above)) - 1u : FULL) & (FULL << start);
            mine = smask & members;
            if (lane == start && mine) first = atomicAdd(&s.fill[c0], __popc(mine));
        }
        c_valid += __popc(__ballot_sync(FULL, valid));
        c_surv += __popc(smask);
        if (slow) {
            const int k = qn + __popc(qmask & lt);
            q_slot[warp][k] = (int)i;
            q_end[warp][k] = defer ? (Real)-1 : t_end;
        }
        qn += __popc(qmask);
        if (gone) {  // removed in its cell (a9)
            long long q = 0;
            c_coll += 1;
            if constexpr (IN_PLACE) mm = b.m[i];
            if (!fixed_of_mass(mm, p.exps[0], q)) set_err(s, ERRB_FIXED_OVERFLOW);
            atomicAdd(&smass[c0], (unsigned long long)(-q));
            if constexpr (IN_PLACE) {
                atomicAdd(&s.nleft_next[c0], -1);
                b.cell[i] = -1;
            }
        }
        if constexpr (IN_PLACE) {
            if (surv) {
#pragma unroll
                for (int c = 0; c < 3; ++c) b.x[c][i] = xe[c];
            }
        } else {
            first = __shfl_sync(FULL, first, start);
            if (surv) {
                const int j = slot_of(first + __popc(mine & lt), info.y, info.z);
                if (j >= 0) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        nxt.x[c][j] = xe[c];
                        nxt.u[c][j] = u[c];
                    }
                    nxt.m[j] = mm;
                    nxt.cell[j] = c0;
                    nxt.id[j] = id;
                    if constexpr (KE) nxt.e[j] = es;
                }
            }
        }
        base = nbase;
        if (qn >= 32) drain(32);
    }
    if (qn > 0) drain(qn);
    // ---- counters: one atomic per block and counter
    c_coll = __reduce_add_sync(FULL, c_coll);
    c_exit = __reduce_add_sync(FULL, c_exit);
    c_lost = __reduce_add_sync(FULL, c_lost);
    c_cross = __reduce_add_sync(FULL, c_cross);
    c_wall = __reduce_add_sync(FULL, c_wall);
    if (lane == 0) {
        const unsigned vals[8] = {c_valid, c_coll, c_exit, c_lost, c_cross, c_wall, c_surv, c_mover};
#pragma unroll
        for (int k = 0; k < 8; ++k) sh_red[warp][k] = vals[k];
    }
    __syncthreads();
    if (threadIdx.x < 8) {
        unsigned long long t = 0;
        for (int w = 0; w < NW; ++w) t += sh_red[w][threadIdx.x];
        const int slot[8] = {CNT_TRACKED, CNT_COLLIDED, CNT_EXITED, CNT_LOST, CNT_CROSSINGS, CNT_WALL, CNT_SURV, CNT_MOVERS};
        if (t) {
            atomicAdd(reinterpret_cast<unsigned long long*>(&s.cnt64[slot[threadIdx.x]]), t);
            if (threadIdx.x == 0) atomicAdd(reinterpret_cast<unsigned long long*>(&s.cnt64[CNT_MOVES]), t);
            if (threadIdx.x == 3) set_err(s, ERRB_TRACK_LIMIT);
        }
    }
}
// DYN: the simulation may step in place.
template <class Real, bool KE, int THREADS, bool DYN, class Number>
__device__ __forceinline__ void track_body(const DevMesh& m, const DevState& s, const DevParams& p, const PartBufs& bufs) {
    __shared__ TrackShared<Real, THREADS> sh;
    // (block-uniform: another block may set the bit while this one starts)
    if (__syncthreads_or(threadIdx.x == 0 && (s.cnt64[CNT_ERR] & ERRB_CAPACITY))) return;
    if constexpr (DYN) {
        const long long src = s.cnt64[CNT_SRC] * bufs.delta;
        if (s.cnt64[CNT_IN_PLACE]) track_mode<Real, KE, THREADS, true, Number>(m, s, p, bufs, src, sh);
        else track_mode<Real, KE, THREADS, false, Number>(m, s, p, bufs, src, sh);
    } else {
        track_mode<Real, KE, THREADS, false, Number>(m, s, p, bufs, 0, sh);
    }
}
template <class Real, bool KE, int THREADS, bool DYN>
__global__ void __launch_bounds__(THREADS, TRACK_PER_SM<Real> / THREADS) k_track(DevMesh m, DevState s, DevParams p,
                                                                                 PartBufs bufs) {
    track_body<Real, KE, THREADS, DYN, unsigned>(m, s, p, bufs);
}

// ---- fused batches
__device__ __forceinline__ int member_of(const int32_t* off, int n) {
    int lo = 0, hi = n;  // off[lo] <= blockIdx.x < off[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= (int)blockIdx.x) lo = mid;
        else hi = mid;
    }
    return lo;
}
template <class Real>
__global__ void __launch_bounds__(CELL_BLOCK) k_sample_scale_b(const __grid_constant__ BatchChunk c) {
    const int32_t* off = c.off[BCL_CELLS];
    const int i = member_of(off, c.n);
    sample_scale_body<Real>(c.mem[i].m, c.mem[i].s, c.mem[i].p, c.mem[i].bufs, Blk{(int)blockIdx.x - off[i], off[i + 1] - off[i]});
}
// The particle kernels take every member of the chunk in turn on the whole grid.
template <class Real>
__global__ void __launch_bounds__(256) k_sample_write_b(const __grid_constant__ BatchChunk c) {
    for (int k = 0; k < c.n; ++k)
        sample_write_body<Real>(c.mem[k].m, c.mem[k].s, c.mem[k].p, c.mem[k].bufs, Blk{(int)blockIdx.x, (int)gridDim.x});
}
// Tiles come from each member's own counter; a block starts at member
// blockIdx.x mod n, so that the blocks spread over the members' counters.
// A batch's members always sort (ugkwp_batch_create).
template <class Real, bool KE, int THREADS>
__global__ void __launch_bounds__(THREADS, TRACK_PER_SM<Real> / THREADS) k_track_b(const __grid_constant__ BatchChunk c) {
    for (int k = 0; k < c.n; ++k) {
        const BatchMember& e = c.mem[((int)blockIdx.x + k) % c.n];
        track_body<Real, KE, THREADS, false, unsigned long long>(e.m, e.s, e.p, e.bufs);
        __syncthreads();
    }
}

}  // namespace

void launch_sample_write(const DevMesh& m, const DevState& s, const DevParams& p, const PartBufs& b,
                         int blocks, cudaStream_t st) {
    (void)m;
    if (p.precision != UGKWP_MIXED) k_sample_write<double, false><<<blocks, 256, 0, st>>>(m, s, p, b);
    else if (b.dyn) k_sample_write<float, true><<<blocks, 256, 0, st>>>(m, s, p, b);
    else k_sample_write<float, false><<<blocks, 256, 0, st>>>(m, s, p, b);
}

void launch_sample_scale(const DevMesh& m, const DevState& s, const DevParams& p, const PartBufs& b, cudaStream_t st) {
    if (p.precision == UGKWP_MIXED) k_sample_scale<float><<<blocks_cells(m.nc), CELL_BLOCK, 0, st>>>(m, s, p, b);
    else k_sample_scale<double><<<blocks_cells(m.nc), CELL_BLOCK, 0, st>>>(m, s, p, b);
}

// Calls f with (a value of) the particle type, K > 0, the block size and whether
// the tracking may be in place (binary64 never is).
namespace {
template <class Real, bool KE, int THREADS, bool DYN> struct TrackKind {
    using R = Real;
    static constexpr bool ke = KE, dyn = DYN;
    static constexpr int threads = THREADS;
};
template <class F> void track_kind(int precision, bool ke, bool dyn, int threads, F&& f) {
    auto shape = [&](auto real, auto kev, auto dynv) {
        using R = decltype(real);
        if (threads == 256) f(TrackKind<R, decltype(kev)::value, 256, decltype(dynv)::value>{});
        else f(TrackKind<R, decltype(kev)::value, 128, decltype(dynv)::value>{});
    };
    using T = std::true_type;
    using N = std::false_type;
    if (precision != UGKWP_MIXED) ke ? shape(0.0, T{}, N{}) : shape(0.0, N{}, N{});
    else if (dyn) ke ? shape(0.0f, T{}, T{}) : shape(0.0f, N{}, T{});
    else ke ? shape(0.0f, T{}, N{}) : shape(0.0f, N{}, N{});
}
// Blocks of one of a step's two tracking launches.  A warp reserves up to two runs
// past the end, so that the slots of all runs stay below n + 2 TRACK_RUN_MAX per warp
// (n < 2^31): two launches of fewer than 2^20 warps keep them below 2^32, in which the
// kernel counts.  (With a check in the kernel a step pair of the batch of 14 members
// took 7.20 ms instead of 7.11, of the 16^3 cavity with g_p sampling 564 us instead of 561.)
int track_blocks(int blocks, int threads) {
    constexpr int WARPS = int((1u << 31) / (4 * TRACK_RUN_MAX));
    return std::min(blocks, (WARPS - 1) / (threads / 32));
}
}  // namespace

void launch_track(const DevMesh& m, const DevState& s, const DevParams& p, const PartBufs& b, const TrackShape& sh,
                  int blocks, cudaStream_t st) {
    track_kind(p.precision, p.K > 0, b.dyn != 0, sh.threads, [&](auto k) {
        using T = decltype(k);
        k_track<typename T::R, T::ke, T::threads, T::dyn><<<track_blocks(blocks, T::threads), T::threads, 0, st>>>(m, s, p, b);
    });
}

namespace {
// The preferred carveout of the particle kernels of one particle type.
template <class Real, bool KE> cudaError_t configure_type(int carveout) {
    cudaError_t e = cudaSuccess;
    auto set = [&](auto f) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, carveout);
    };
    for (int threads : {128, 256})
        for (bool dyn : {false, true})
            track_kind(sizeof(Real) == 4 ? UGKWP_MIXED : UGKWP_FP64, KE, dyn, threads, [&](auto k) {
                using T = decltype(k);
                set(k_track<typename T::R, T::ke, T::threads, T::dyn>);
                set(k_track_b<typename T::R, T::ke, T::threads>);
            });
    set(k_sample_write<Real, false>);
    if constexpr (sizeof(Real) == 4) set(k_sample_write<Real, true>);
    set(k_sample_scale<Real>);
    set(k_sample_write_b<Real>);
    set(k_sample_scale_b<Real>);
    return e;
}
}  // namespace

cudaError_t configure_particle_kernels(const DevParams& p, int carveout) {
    if (p.precision == UGKWP_MIXED) return p.K > 0 ? configure_type<float, true>(carveout) : configure_type<float, false>(carveout);
    return p.K > 0 ? configure_type<double, true>(carveout) : configure_type<double, false>(carveout);
}

void launch_sample_scale_batch(const BatchChunk& c, int blocks, int precision, cudaStream_t st) {
    if (precision == UGKWP_MIXED) k_sample_scale_b<float><<<blocks, CELL_BLOCK, 0, st>>>(c);
    else k_sample_scale_b<double><<<blocks, CELL_BLOCK, 0, st>>>(c);
}
void launch_sample_write_batch(const BatchChunk& c, int blocks, int precision, cudaStream_t st) {
    if (precision == UGKWP_MIXED) k_sample_write_b<float><<<blocks, 256, 0, st>>>(c);
    else k_sample_write_b<double><<<blocks, 256, 0, st>>>(c);
}
void launch_track_batch(const BatchChunk& c, int precision, bool ke, const TrackShape& sh, int blocks,
                        cudaStream_t st) {
    track_kind(precision, ke, false, sh.threads, [&](auto k) {
        using T = decltype(k);
        k_track_b<typename T::R, T::ke, T::threads><<<track_blocks(blocks, T::threads), T::threads, 0, st>>>(c);
    });
}

}  // namespace ugkwp
