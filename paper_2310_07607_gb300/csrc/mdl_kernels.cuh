// mdl_kernels.cuh -- CUDA kernels of one barrier step (Alg. 1) for one (precision, dim, order).
//
// Data layout in HBM (structure of arrays, element-blocked DOFs):
//   V0, V1  [ne * NPS] two slots of V; element e's current value is in slot
//                      par_e ^ (updates this barrier & 1) -- a per-element ping-pong,
//                      so a tick reads the values at its start and writes the other slot
//   v       [ne * NPS] Aliev-Panfilov recovery variable (element-local, in place)
//   Ia, ga  [ne * NPS] I(u_a, t_a) and g(u_a) at the barrier start (only for S_e > 1)
//                      (NPS: the row stride, NP rounded up to 28 for Q2 3D; pad value 0)
//   lvl     [ne]       b_e (bits 0-2) | parity par_e (bit 3) | ordering class (bit 4)
//   info    [ne]       4 bits per face: kind (0 bnd, 1 same, 2 coarser, 3 finer) | pos << 2;
//                      bits 24-27 refinement level; bit 28 in a stimulus box; bit 29 probes pending
//   nbr     [ne * 2d]  neighbour element (same/coarser) or first hang[] index (finer)
//   hang    [*]        2^(d-1) fine neighbours per hanging face
//   order   [ne]       element ids sorted by b descending (regular elements first within a level
//                      on 3D Q2 and curved meshes): tick i updates a prefix
//   acc     [ne]       FP64 RV-T accumulator; eta_t, eta_s [ne] FP64
//   lat     [n_probe]  FP64 activation time per probe (+INF pending)
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "../../include/mdl.h"
#include "mdl_boxop.cuh"
#include "mdl_element.cuh"

namespace mdl {

constexpr uint32_t INFO_STIM = 1u << 28;
constexpr uint32_t INFO_PENDING = 1u << 29;

// Device-resident bookkeeping of one context: every kernel reads its element count
// and the sticky error word from here, so a barrier needs no host round trip.
struct DevMeta {
    int64_t ne;              // elements of the current mesh
    int64_t ne_new;          // elements after this barrier's adaptation
    int64_t nbar;            // completed barriers
    int64_t need;            // element capacity requested on overflow
    unsigned int err;        // sticky: 1 non-finite, 2 CFL, 4 capacity, 8 mesh
    unsigned int changed;    // the adaptation changed the mesh
    unsigned int nf_pending; // non-finite values seen by this barrier's epilogue
    unsigned int cur_set;    // index of the state set holding the current values
    unsigned int done_blocks;// blocks arrived at a kernel's last-block pass (0 between kernels)
    unsigned int cnt[8];     // elements per level b in this barrier
    int32_t nact[128];       // due elements per tick
    int64_t elem_updates;    // accumulated element steps
    int64_t rebuilds;        // barriers whose mesh changed
    int64_t fac_updates;     // curved meshes: elements whose factors were computed
    double integral;         // FP64 int V after the last barrier
    unsigned int nfac;       // curved meshes: elements whose factors the adaptation recomputes
    unsigned int adapted;    // this barrier's new mesh is committed and its state not yet transferred
    unsigned int gbar;       // cooperative sweep: arrivals at its grid barriers (zeroed before each launch)
};

// ERR_WAIT: a bounded wait of a kernel gave up (tensor-core mbarrier, cooperative grid barrier)
constexpr unsigned ERR_NONFINITE = 1u, ERR_CFL = 2u, ERR_CAPACITY = 4u, ERR_MESH = 8u, ERR_WAIT = 16u;

// Programmatic dependent launch: wait until the preceding grid on the stream has completed
// and its writes are visible, then let the following grid be scheduled.  Each kernel of a
// barrier step calls this first; launched without the attribute it returns at once.
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ int64_t gstride() { return (int64_t)gridDim.x * blockDim.x; }
__device__ __forceinline__ int64_t gtid() { return blockIdx.x * (int64_t)blockDim.x + threadIdx.x; }

template <typename R>
struct DevArrays {
    R* V0;
    R* V1;
    R* v;
    R* Ia;
    R* ga;
    double* acc;
    double* eta_t;
    double* eta_s;
    double* lat;
    double* partial;
    uint8_t* lvl;
    const uint8_t* bcfl;
    uint32_t* info;
    const int32_t* nbr;
    const int32_t* hang;
    const int32_t* order;
    const int32_t* root;
    const uint32_t* loc;
    const uint32_t* smask[MDL_MAX_STIM];
    DevMeta* meta;
    const R* qvol;      // Q1 class blocks (see q1_blocks): volume, face, Kelly
    const R* qface;
    const R* qkelly;
    const R* gvol;      // mapped meshes: per-element geometric factors (mdl_mapped.cuh)
    const R* gface;
    const double* mq;   // mapped meshes: per-element GL masses (null on boxes)
};

// Vector width for rows of NP values of type R: 16-byte loads when a row is a whole number
// of them (every table block and element vector below starts on a 16-byte boundary).
template <typename R, int NP>
struct Vec {
    static constexpr int W = (16 / (int)sizeof(R));
    static constexpr bool ok = (NP % W) == 0;
};

// out[0..n) = p[0..n), 16-byte loads where the width allows (p 16-byte aligned then).
template <typename R, int N>
__device__ __forceinline__ void ld_row(const R* __restrict__ p, R* out) {
    if constexpr (Vec<R, N>::ok && sizeof(R) == 4) {
#pragma unroll
        for (int i = 0; i < N / 4; ++i) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(p) + i);
            out[4 * i] = v.x; out[4 * i + 1] = v.y; out[4 * i + 2] = v.z; out[4 * i + 3] = v.w;
        }
    } else if constexpr (Vec<R, N>::ok && sizeof(R) == 8) {
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            const double2 v = __ldg(reinterpret_cast<const double2*>(p) + i);
            out[2 * i] = v.x; out[2 * i + 1] = v.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) out[i] = __ldg(p + i);
    }
}

// Plain (coherent) vector load / store of an element's N values.
template <typename R, int N>
__device__ __forceinline__ void ld_vec(const R* p, R* out) {
    if constexpr (Vec<R, N>::ok && sizeof(R) == 4) {
#pragma unroll
        for (int i = 0; i < N / 4; ++i) {
            const float4 v = reinterpret_cast<const float4*>(p)[i];
            out[4 * i] = v.x; out[4 * i + 1] = v.y; out[4 * i + 2] = v.z; out[4 * i + 3] = v.w;
        }
    } else if constexpr (Vec<R, N>::ok && sizeof(R) == 8) {
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            const double2 v = reinterpret_cast<const double2*>(p)[i];
            out[2 * i] = v.x; out[2 * i + 1] = v.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) out[i] = p[i];
    }
}

template <typename R, int N>
__device__ __forceinline__ void st_vec(R* p, const R* x) {
    if constexpr (Vec<R, N>::ok && sizeof(R) == 4) {
#pragma unroll
        for (int i = 0; i < N / 4; ++i)
            reinterpret_cast<float4*>(p)[i] = make_float4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]);
    } else if constexpr (Vec<R, N>::ok && sizeof(R) == 8) {
#pragma unroll
        for (int i = 0; i < N / 2; ++i) reinterpret_cast<double2*>(p)[i] = make_double2(x[2 * i], x[2 * i + 1]);
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) p[i] = x[i];
    }
}

// One element row of a per-DOF state array: NP values at row stride NPS.  With NPS a whole
// number of 16-byte vectors the row moves in vectors (the pad value read is dropped; a
// store writes the pad as 0), else value by value.
template <typename R, int NP, int NPS>
__device__ __forceinline__ void ld_dofs(const R* p, R* out) {
    if constexpr (NPS == NP) {
        ld_vec<R, NP>(p, out);
    } else {
        R t[NPS];
        ld_vec<R, NPS>(p, t);
#pragma unroll
        for (int q = 0; q < NP; ++q) out[q] = t[q];
    }
}

template <typename R, int NP, int NPS>
__device__ __forceinline__ void st_dofs(R* p, const R* x) {
    if constexpr (NPS == NP) {
        st_vec<R, NP>(p, x);
    } else {
        R t[NPS];
#pragma unroll
        for (int q = 0; q < NPS; ++q) t[q] = q < NP ? x[q] : R(0);
        st_vec<R, NPS>(p, t);
    }
}

// j[t] += sum_q K[t][q] x[q] for a row-major NT x NP block (read-only path).
template <typename R, int NT, int NP>
__device__ __forceinline__ void block_jump(const R* __restrict__ K, const R* x, R* j) {
#pragma unroll
    for (int t = 0; t < NT; ++t) {
        R row[NP];
        ld_row<R, NP>(K + t * NP, row);
        R acc = j[t];
#pragma unroll
        for (int q = 0; q < NP; ++q) acc += row[q] * x[q];
        j[t] = acc;
    }
}

// r[q] += sum_j A[q][j] x[j] for a row-major NP x NP block in global memory (read-only path).
template <typename R, int NP>
__device__ __forceinline__ void block_mv(const R* __restrict__ A, const R* x, R* r) {
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        R row[NP];
        ld_row<R, NP>(A + q * NP, row);
        R acc = r[q];
#pragma unroll
        for (int j = 0; j < NP; ++j) acc += row[j] * x[j];
        r[q] = acc;
    }
}

// 2^-sh exactly, for 0 <= sh < 64 (built from the IEEE-754 exponent field).
template <typename R>
__device__ __forceinline__ R pow2_neg(int sh);
template <>
__device__ __forceinline__ float pow2_neg<float>(int sh) { return __int_as_float((127 - sh) << 23); }
template <>
__device__ __forceinline__ double pow2_neg<double>(int sh) {
    return __longlong_as_double((long long)(1023 - sh) << 52);
}

struct StimArgs {
    int n;
    double t0[MDL_MAX_STIM], t1[MDL_MAX_STIM], amp[MDL_MAX_STIM];
};

template <typename R>
__device__ __forceinline__ R r_exp(R x);
template <>
__device__ __forceinline__ float r_exp<float>(float x) { return expf(x); }
template <>
__device__ __forceinline__ double r_exp<double>(double x) { return exp(x); }

// a / b: FP32 through the fast reciprocal (within 2 ulp; b >= 1e-6 here), FP64 exact.
template <typename R>
__device__ __forceinline__ R r_div(R a, R b);
template <>
__device__ __forceinline__ float r_div<float>(float a, float b) { return __fdividef(a, b); }
template <>
__device__ __forceinline__ double r_div<double>(double a, double b) { return a / b; }

// e^x - 1 in FP32 without the cancellation of expf(x) - 1: for |x| < 1/16 the Taylor series
// of the exponential through x^6 (truncation below 1e-12 relative), else expf(x) - 1.
__device__ __forceinline__ float expm1_f32(float x) {
    if (fabsf(x) < 0.0625f)
        return x * (1.0f + x * (0.5f + x * (1.0f / 6.0f + x * (1.0f / 24.0f + x * (1.0f / 120.0f + x * (1.0f / 720.0f))))));
    return expf(x) - 1.0f;
}

template <typename R>
__device__ __forceinline__ R ap_iion(const Phys<R>& ph, R V, R w) {
    if (ph.ionic < 0) return R(0);
    return (ph.k * V * (V - ph.a) * (V - R(1)) + V * w) * ph.inv_ts;
}

template <typename R>
__device__ __forceinline__ R ap_eps(const Phys<R>& ph, R V, R w) {
    R den = V + ph.mu2;
    den = den > R(1e-6) ? den : R(1e-6);
    return ph.eps0 + r_div<R>(ph.mu1 * w, den);
}

template <typename R>
__device__ __forceinline__ R ap_g(const Phys<R>& ph, R V, R w) {
    if (ph.ionic < 0) return R(0);
    const R vinf = -ph.k * V * (V - ph.a - R(1));
    return ap_eps(ph, V, w) * (vinf - w) * ph.inv_ts;
}

// One step of the state: forward Euler, or the exponential step v_inf + (v - v_inf) e^(-eps dt)
// with eps and v_inf frozen at the step start.  In FP32 the exponential step is evaluated as
// v + (v - v_inf) (e^(-eps dt) - 1): on explicit substeps eps dt is far below 1 (about
// 1e-8 .. 1e-4 for substeps of 1e-6 .. 1e-2 ms), where e^(-eps dt) rounded to FP32 would
// lose most of the increment.
template <typename R>
__device__ __forceinline__ R ap_step_state(const Phys<R>& ph, R V, R w, R dt) {
    if (ph.ionic < 0) return w;
    const R vinf = -ph.k * V * (V - ph.a - R(1));
    const R eps = ap_eps(ph, V, w);
    if (ph.integrator == 0) return w + dt * eps * (vinf - w) * ph.inv_ts;
    if constexpr (sizeof(R) == 4) return w + (w - vinf) * expm1_f32(-eps * dt * ph.inv_ts);
    return vinf + (w - vinf) * r_exp<R>(-eps * dt * ph.inv_ts);
}

// Values of element nb as seen at tick `tick`, given its level byte: its current value if
// it is due (or finer), else the linear time interpolant of its last step (Alg. 1).
template <typename R, int NP, int NPS = NP>
__device__ __forceinline__ void load_seen_lv(const DevArrays<R>& d, int tick, int B, int nb, uint8_t lv, R* un) {
    const int b = lv & 7, par = (lv >> 3) & 1;
    const int sh = B - b;
    const int j = tick >> sh;
    const int rem = tick & ((1 << sh) - 1);
    const int nw = par ^ ((j + (rem ? 1 : 0)) & 1);
    ld_dofs<R, NP, NPS>((nw ? d.V1 : d.V0) + (size_t)nb * NPS, un);
    if (rem) {
        R so[NP];
        ld_dofs<R, NP, NPS>((nw ? d.V0 : d.V1) + (size_t)nb * NPS, so);
        const R th = R(rem) * pow2_neg<R>(sh);
#pragma unroll
        for (int q = 0; q < NP; ++q) un[q] = so[q] + th * (un[q] - so[q]);
    }
}

template <typename R, int NP, int NPS = NP>
__device__ __forceinline__ void load_seen(const DevArrays<R>& d, int tick, int B, int nb, R* un) {
    load_seen_lv<R, NP, NPS>(d, tick, B, nb, d.lvl[nb], un);
}

// Probe activation check for element e after a step from u (at t_old) to un (t_old + dte).
// The probes inside the leaf are the root GL nodes a with pfl[lev][a_k] == the leaf's cell
// in every direction k; a pending probe's values before and after the step are the leaf
// polynomial at its position, evaluated by sum factorisation.
// lc, rid: the leaf's cell in its root and the root id (loc[e], root[e]).
// pend: bit q set if probe q of the root may still be pending (from a read of lat before
// the step; a probe it marks that has meanwhile activated fails the crossing test below).
template <typename R, int DIM, int P>
__device__ void lat_check_at(const DevArrays<R>& d, const Tables<R>& T, const Phys<R>& ph, int e, uint32_t inf,
                             int lev, uint32_t lc, int64_t rid, const R* u, const R* un, double t_old, double dte,
                             uint32_t pend = 0xffffffffu, bool known = false) {
    using S = Shape<DIM, P>;
    constexpr int N1 = S::N1, NP = S::NP;
    const int lx[3] = {(int)(lc & 255u), (int)((lc >> 8) & 255u), (int)((lc >> 16) & 255u)};
    unsigned inside_k[3] = {1u, 1u, 1u};
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
        inside_k[k] = 0u;
#pragma unroll
        for (int a = 0; a < N1; ++a)
            if (T.pfl[lev][a] == lx[k]) inside_k[k] |= 1u << a;
    }
    uint32_t im = 0u;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        bool in = true;
#pragma unroll
        for (int k = 0; k < DIM; ++k) in = in && ((inside_k[k] >> digit<N1>(q, k)) & 1u);
        if (in) im |= 1u << q;
    }
    bool pending = false;
    im &= pend;
    while (im) {
        const int q = __ffs(im) - 1;
        im &= im - 1u;
        double* lp = d.lat + rid * NP + q;
        if (!known && !isinf(*lp)) continue;
        R Pk[3][3];
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int j = 0; j < N1; ++j) Pk[k][j] = (k < DIM) ? T.pphi[lev][digit<N1>(q, k)][j] : R(1);
        R po = 0, pn = 0;
#pragma unroll
        for (int j2 = 0; j2 < (DIM == 3 ? N1 : 1); ++j2) {
            R t1o = 0, t1n = 0;
#pragma unroll
            for (int j1 = 0; j1 < N1; ++j1) {
                R t0o = 0, t0n = 0;
#pragma unroll
                for (int j0 = 0; j0 < N1; ++j0) {
                    const int idx = j0 + N1 * j1 + N1 * N1 * j2;
                    t0o += Pk[0][j0] * u[idx];
                    t0n += Pk[0][j0] * un[idx];
                }
                t1o += Pk[1][j1] * t0o;
                t1n += Pk[1][j1] * t0n;
            }
            po += Pk[2][j2] * t1o;
            pn += Pk[2][j2] * t1n;
        }
        if (po <= ph.act && pn > ph.act) {
            *lp = t_old + dte * (double)((ph.act - po) / (pn - po));
        } else {
            pending = true;
        }
    }
    if (!pending) d.info[e] = inf & ~INFO_PENDING;
}

template <typename R, int DIM, int P>
__device__ void lat_check(const DevArrays<R>& d, const Tables<R>& T, const Phys<R>& ph, int e,
                          uint32_t inf, int lev, const R* u, const R* un, double t_old, double dte) {
    lat_check_at<R, DIM, P>(d, T, ph, e, inf, lev, d.loc[e], (int64_t)d.root[e], u, un, t_old, dte);
}

template <typename R>
struct TickArgs {
    DevArrays<R> d;
    StimArgs stim;
    double dt;         // barrier step
    double tscale;     // dt * 2^-B: t at tick i of barrier n is (n 2^B + i) * tscale (exact)
    double dte[8];     // dt * 2^-b per level b (exact), and the same rounded to R
    R dteR[8];
    int tick, B;
};

// Canonical time of tick `tick` in the current barrier, ((n 2^B + i) dt) / 2^B (the
// division by 2^B is exact, so scaling dt first gives the same value).  Evaluated only
// where a time is needed (stimulus windows, activation times): FP64 is slow on this part.
template <typename R>
__device__ __forceinline__ double tick_time(const TickArgs<R>& a, int tick) {
    return ((double)a.d.meta->nbar * (double)(1 << a.B) + (double)tick) * a.tscale;
}

// Per-element data that stays fixed during a sweep: the element, its level byte and face
// info, its face neighbours and their level bytes.  A tick reads it before waiting for
// the previous tick (programmatic dependent launch), so after the wait only the values are
// loaded, all at once.  (info's probe-pending bit may be cleared by an earlier tick of the
// sweep; a stale bit only repeats a probe check that finds nothing left to do.)
template <int DIM, int P>
struct TickMeta {
    static constexpr int NF = 2 * DIM;
    static constexpr bool HP = DIM == 2;  // 2D: the finer neighbours of hanging faces too
    static constexpr bool PR = P == 1;    // Q1: the probe lookup too
    int e;
    uint32_t inf;
    uint8_t lv;
    int nbf[NF];
    uint8_t lvn[NF];
    int hg[HP ? NF : 1][2];               // fine neighbours of a hanging face and their level bytes
    uint8_t hgl[HP ? NF : 1][2];
    uint32_t lc;                          // probe lookup: cell in the root, root id
    int rid;
    uint32_t pend;                        // probes of the root with no activation time yet
};

template <typename R, int DIM, int P>
__device__ __forceinline__ void tick_fetch(const DevArrays<R>& d, int idx, TickMeta<DIM, P>& m) {
    using M = TickMeta<DIM, P>;
    constexpr int NF = 2 * DIM;
    m.e = d.order[idx];
    m.lv = d.lvl[m.e];
    m.inf = d.info[m.e];
    if constexpr (DIM == 2) {
        const int4 n = *reinterpret_cast<const int4*>(d.nbr + (size_t)m.e * 4);
        m.nbf[0] = n.x; m.nbf[1] = n.y; m.nbf[2] = n.z; m.nbf[3] = n.w;
    } else {
#pragma unroll
        for (int f = 0; f < NF; f += 2) {
            const int2 n = *reinterpret_cast<const int2*>(d.nbr + (size_t)m.e * NF + f);
            m.nbf[f] = n.x;
            m.nbf[f + 1] = n.y;
        }
    }
    if constexpr (M::PR) {
        m.lc = d.loc[m.e];
        m.rid = d.root[m.e];
        // activation times of the root's probes (only this leaf writes those inside it, at its
        // own steps; a value read before the previous tick's write only repeats a check)
        m.pend = 0u;
        if (m.inf & INFO_PENDING) {
            constexpr int NP = Shape<DIM, P>::NP;
#pragma unroll
            for (int q = 0; q < NP; ++q)
                if (isinf(d.lat[(int64_t)m.rid * NP + q])) m.pend |= 1u << q;
        }
    }
    if constexpr (M::HP) {
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const bool hanging = ((m.inf >> (4 * f)) & 3) == 3;
#pragma unroll
            for (int sb = 0; sb < 2; ++sb) {
                m.hg[f][sb] = hanging ? d.hang[m.nbf[f] + sb] : m.e;
                m.hgl[f][sb] = d.lvl[m.hg[f][sb]];
            }
        }
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const int kind = (m.inf >> (4 * f)) & 3;
        m.lvn[f] = d.lvl[(kind == 1 || kind == 2) ? m.nbf[f] : m.e];
    }
}

// The row of element nb (level byte lv) that holds its value at tick `tick`; `old` is the row of
// its step's start and th the interpolation weight when it is mid-interval (th = 0 otherwise).
template <typename R, int NPS>
__device__ __forceinline__ const R* seen_row(const DevArrays<R>& d, int tick, int B, int nb, uint8_t lv, const R*& old,
                                             R& th) {
    const int sh = B - (lv & 7), par = (lv >> 3) & 1;
    const int rem = tick & ((1 << sh) - 1);
    const int nw = par ^ (((tick >> sh) + (rem ? 1 : 0)) & 1);
    th = R(rem) * pow2_neg<R>(sh);
    const size_t o = (size_t)nb * NPS;
    old = (nw ? d.V0 : d.V1) + o;
    return (nw ? d.V1 : d.V0) + o;
}

// v = (1 - th) old + th v for a neighbour mid-interval (Alg. 1's linear interpolant).
template <typename R, int NP, int NPS>
__device__ __forceinline__ void interp_row(const R* old, R th, R* v) {
    R so[NP];
    ld_dofs<R, NP, NPS>(old, so);
#pragma unroll
    for (int q = 0; q < NP; ++q) v[q] = so[q] + th * (v[q] - so[q]);
}

// Q1: r = (A u)_e with the neighbours seen at tick `tick`, from the dense blocks: constants of the
// kernel for same-level faces (level 0, scaled by 2^((2-d) lev), exact), the class blocks in memory
// for the others.
template <typename R, int DIM>
__device__ __forceinline__ void residual_q1(const DevArrays<R>& d, const Q1Op<R, DIM>& op, int tick, int B,
                                            const TickMeta<DIM, 1>& m, int lev, const R* u, R* r) {
    using S = Shape<DIM, 1>;
    constexpr int NP = S::NP, NF = S::NF, NSUB = S::NSUB, NREL = 1 + 2 * NSUB;
    R un[NF][NP];
    const R* old[NF];
    R th[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const int kind = (m.inf >> (4 * f)) & 3;
        const bool use = kind == 1 || kind == 2;
        ld_vec<R, NP>(seen_row<R, NP>(d, tick, B, use ? m.nbf[f] : m.e, use ? m.lvn[f] : m.lv, old[f], th[f]), un[f]);
    }
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        R s = R(0);
#pragma unroll
        for (int j = 0; j < NP; ++j) s += op.vol[q][j] * u[j];
        r[q] = s;
    }
    bool irr = false;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const int kind = (m.inf >> (4 * f)) & 3;
        irr = irr || kind >= 2;
        if (th[f] > R(0)) interp_row<R, NP, NP>(old[f], th[f], un[f]);
        if (kind == 1) {
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                R s = r[q];
#pragma unroll
                for (int j = 0; j < NP; ++j) s += op.face[f][0][q][j] * u[j];
#pragma unroll
                for (int j = 0; j < NP; ++j) s += op.face[f][1][q][j] * un[f][j];
                r[q] = s;
            }
        }
    }
    if (DIM == 3) {
        const R sc = pow2_neg<R>(lev);
#pragma unroll
        for (int q = 0; q < NP; ++q) r[q] *= sc;
    }
    if (!irr) return;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const int kind = (m.inf >> (4 * f)) & 3;
        if (kind < 2) continue;
        const R* A0 = d.qface + (((size_t)f * 8 + lev) * NREL * 2) * NP * NP;
        if (kind == 2) {
            const R* A = A0 + (size_t)(1 + ((m.inf >> (4 * f + 2)) & 3)) * 2 * NP * NP;
            block_mv<R, NP>(A, u, r);
            block_mv<R, NP>(A + NP * NP, un[f], r);
        } else {
#pragma unroll 1
            for (int sb = 0; sb < NSUB; ++sb) {
                R uh[NP];
                int n;
                uint8_t lv;
                if constexpr (TickMeta<DIM, 1>::HP) {
                    n = sb ? m.hg[f][1] : m.hg[f][0];
                    lv = sb ? m.hgl[f][1] : m.hgl[f][0];
                } else {
                    n = d.hang[m.nbf[f] + sb];
                    lv = d.lvl[n];
                }
                const R* o;
                R t;
                ld_vec<R, NP>(seen_row<R, NP>(d, tick, B, n, lv, o, t), uh);
                if (t > R(0)) interp_row<R, NP, NP>(o, t, uh);
                const R* A = A0 + (size_t)(1 + NSUB + sb) * 2 * NP * NP;
                block_mv<R, NP>(A, u, r);
                block_mv<R, NP>(A + NP * NP, uh, r);
            }
        }
    }
}

// rho = (M^-1 A u)_e in level-0 units (times 4^level; see mdl_boxop.cuh) with the neighbours
// seen at tick `tick`, for 2D Q2 elements: every neighbour row is loaded before the arithmetic.
template <typename R, int DIM, int P>
__device__ __forceinline__ void box_residual(const DevArrays<R>& d, const BoxOp<R>& op, int tick, int B,
                                             const TickMeta<DIM, P>& m, const R* u, R* rho) {
    using S = Shape<DIM, P>;
    constexpr int NP = S::NP, NF = S::NF, NT = S::NT, NPS = S::NPS;
    const uint32_t inf = m.inf;
    const R c = u[NP / 2];
    R un[NF][NP];
    const R* old[NF];
    R th[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const int kind = (inf >> (4 * f)) & 3;
        const bool use = kind == 1 || kind == 2;
        ld_dofs<R, NP, NPS>(seen_row<R, NPS>(d, tick, B, use ? m.nbf[f] : m.e, use ? m.lvn[f] : m.lv, old[f], th[f]),
                            un[f]);
    }
    R y[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) y[q] = u[q] - c;
    box_own<R, DIM, P>(op, y, rho, op.cross != 0);
    bool irr = false;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const int kind = (inf >> (4 * f)) & 3;
        irr = irr || kind != 1;
        if (th[f] > R(0)) interp_row<R, NP, NPS>(old[f], th[f], un[f]);
#pragma unroll
        for (int q = 0; q < NP; ++q) un[f][q] -= c;
        if (kind == 1) {
            R TN[NT], DN[NT];
            box_trace<R, DIM, P>(op, f >> 1, 1 - (f & 1), un[f], TN, DN);
            if (op.cross) {
                R Xv[NT];
                box_mixed<R, DIM, P>(op, f >> 1, f & 1, TN, Xv);
                box_lift<R, DIM, P, true>(op, f >> 1, f & 1, TN, DN, Xv, rho);
            } else {
                box_lift<R, DIM, P, false>(op, f >> 1, f & 1, TN, DN, nullptr, rho);
            }
        }
    }
    if (!irr) return;
    // boundary, coarser and finer neighbours
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const int kind = (inf >> (4 * f)) & 3;
        if (kind == 1) continue;
        auto nb = [&](int sb, R* v) {
            if (kind == 2) {
#pragma unroll
                for (int q = 0; q < NP; ++q) v[q] = un[f][q];
                return;
            }
            int n;
            uint8_t lv;
            if constexpr (TickMeta<DIM, P>::HP) {
                n = sb ? m.hg[f][1] : m.hg[f][0];
                lv = sb ? m.hgl[f][1] : m.hgl[f][0];
            } else {
                n = d.hang[m.nbf[f] + sb];
                lv = d.lvl[n];
            }
            const R* o;
            R t;
            ld_dofs<R, NP, NPS>(seen_row<R, NPS>(d, tick, B, n, lv, o, t), v);
            if (t > R(0)) interp_row<R, NP, NPS>(o, t, v);
#pragma unroll
            for (int q = 0; q < NP; ++q) v[q] -= c;
        };
        R TN[NT], DN[NT], Xv[NT];
        box_face_irregular<R, DIM, P>(op, f >> 1, f & 1, kind, (inf >> (4 * f + 2)) & 3, y, nb, TN, DN, Xv,
                                       op.cross != 0);
        box_lift<R, DIM, P, true>(op, f >> 1, f & 1, TN, DN, Xv, rho);
    }
}

// The same for Q2 3D elements (27 values a row: all six neighbours would spill).  The axis is
// unrolled, the side a loop: the straight-line form of the whole step is 50 KB of code, which
// every warp streams through the instruction cache once per element, and waited there for
// most of its time (8.3 of 15.4 cycles per instruction on a 29k-element block).
template <typename R>
__device__ __forceinline__ void box_residual_q23(const DevArrays<R>& d, const BoxOp<R>& op, int tick, int B,
                                                 const TickMeta<3, 2>& m, const R* u, R* rho) {
    constexpr int NP = 27, NPS = 28, NT = 9;
    const uint32_t inf = m.inf;
    const R c = u[NP / 2];
    R y[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) y[q] = u[q] - c;
    box_own<R, 3, 2>(op, y, rho, op.cross != 0);
    auto row = [&](int n, uint8_t lv, R* v) {
        const R* o;
        R t;
        ld_dofs<R, NP, NPS>(seen_row<R, NPS>(d, tick, B, n, lv, o, t), v);
        if (t > R(0)) interp_row<R, NP, NPS>(o, t, v);
#pragma unroll
        for (int q = 0; q < NP; ++q) v[q] -= c;
    };
#pragma unroll
    for (int k = 0; k < 3; ++k) {
#pragma unroll 1
        for (int side = 0; side < 2; ++side) {
            const uint32_t fi = inf >> (8 * k + 4 * side);
            const int kind = fi & 3;
            const int nbf = side ? m.nbf[2 * k + 1] : m.nbf[2 * k];
            const uint8_t lvn = side ? m.lvn[2 * k + 1] : m.lvn[2 * k];
            R TN[NT], DN[NT];
            if (kind == 1) {
                R v[NP];
                row(nbf, lvn, v);
                box_trace<R, 3, 2>(op, k, 1 - side, v, TN, DN);
                if (!op.cross) {
                    box_lift<R, 3, 2, false>(op, k, side, TN, DN, nullptr, rho);
                    continue;
                }
            }
            R Xv[NT];
            if (kind == 1) {
                box_mixed<R, 3, 2>(op, k, side, TN, Xv);
            } else {
                auto nb = [&](int sb, R* v) {
                    const int n = kind == 2 ? nbf : d.hang[nbf + sb];
                    row(n, kind == 2 ? lvn : d.lvl[n], v);
                };
                box_face_irregular<R, 3, 2>(op, k, side, kind, (fi >> 2) & 3, y, nb, TN, DN, Xv, op.cross != 0);
            }
            box_lift<R, 3, 2, true>(op, k, side, TN, DN, Xv, rho);
        }
    }
}

// Stimulus currents of DOF q of element e at the step start (so) and at the step midpoint
// (sm): -amplitude for every stimulus box holding the node whose window [t0, t1) holds the
// time (the midpoint value enters the RV-T term).
template <typename R>
__device__ __forceinline__ void dof_stim(const TickArgs<R>& a, int e, int tick, double dte_d, int q, R& so, R& sm) {
    so = sm = R(0);
    const double t_i = tick_time(a, tick);
    const double t_mid = t_i + 0.5 * dte_d;
    for (int s = 0; s < a.stim.n; ++s) {
        const bool on_o = (a.stim.t0[s] <= t_i) && (t_i < a.stim.t1[s]);
        const bool on_m = (a.stim.t0[s] <= t_mid) && (t_mid < a.stim.t1[s]);
        if (!on_o && !on_m) continue;
        if (!((a.d.smask[s][e] >> q) & 1u)) continue;
        const R amp = (R)a.stim.amp[s];
        if (on_o) so -= amp;
        if (on_m) sm -= amp;
    }
}

// The same for a whole element: bit q of mo[s] (mm[s]) is set where stimulus s acts on node q
// at the step start (midpoint).  The time windows are tested once per element and stimulus: an
// FP64 comparison per DOF costs more than the rest of the DOF's step (FP64 is slow on this part).
struct StimMasks {
    uint32_t mo[MDL_MAX_STIM], mm[MDL_MAX_STIM];
    bool any;
};

template <typename R>
__device__ __forceinline__ void elem_stim(const TickArgs<R>& a, int e, uint32_t inf, int tick, double dte_d,
                                          StimMasks& sm) {
    sm.any = false;
#pragma unroll
    for (int s = 0; s < MDL_MAX_STIM; ++s) sm.mo[s] = sm.mm[s] = 0u;
    if (!(inf & INFO_STIM)) return;
    const double t_i = tick_time(a, tick);
    const double t_mid = t_i + 0.5 * dte_d;
#pragma unroll
    for (int s = 0; s < MDL_MAX_STIM; ++s) {
        if (s >= a.stim.n) break;
        const bool on_o = (a.stim.t0[s] <= t_i) && (t_i < a.stim.t1[s]);
        const bool on_m = (a.stim.t0[s] <= t_mid) && (t_mid < a.stim.t1[s]);
        if (!on_o && !on_m) continue;
        const uint32_t m = a.d.smask[s][e];
        sm.mo[s] = on_o ? m : 0u;
        sm.mm[s] = on_m ? m : 0u;
        sm.any = sm.any || m;
    }
}

// Stimulus currents of node q (step start, midpoint).
template <typename R>
__device__ __forceinline__ void node_stim(const TickArgs<R>& a, const StimMasks& sm, int q, R& so, R& smd) {
    so = smd = R(0);
    if (!sm.any) return;
#pragma unroll
    for (int s = 0; s < MDL_MAX_STIM; ++s) {
        const R amp = (R)a.stim.amp[s];
        if ((sm.mo[s] >> q) & 1u) so -= amp;
        if ((sm.mm[s] >> q) & 1u) smd -= amp;
    }
}

// Update of one DOF given its residual r = (A u)_q, its GL mass Mq = w_q det J and the
// inverse Minv: forward Euler on V, the exponential/FE step on v, and the DOF's share
// Mq [dI^2 + dg^2] of the RV-T midpoint term (returned).  At the element's first step of
// the barrier (ke == 0), Ia/ga receive I and g at the barrier start.
template <typename R>
__device__ __forceinline__ R dof_update(const Phys<R>& ph, R Mq, R Minv, int ke, R dte, R so, R sm, R u, R w, R r,
                                        R& Ia, R& ga, R& un, R& wn) {
    if (ke == 0) {
        Ia = ap_iion(ph, u, w) + so;
        ga = ap_g(ph, u, w);
    }
    const R I = ap_iion(ph, u, w) + so;
    un = u + dte * (-r * Minv - I);
    wn = ap_step_state(ph, u, w, dte);
    const R Vm = R(0.5) * (u + un);
    const R wm = R(0.5) * (w + wn);
    const R dI = ap_iion(ph, Vm, wm) + sm - Ia;
    const R dg = ap_g(ph, Vm, wm) - ga;
    return Mq * (dI * dI + dg * dg);
}

// Constants of the FP32 Aliev-Panfilov step.
struct ApConst {
    float k, a, it, eps0, mu1, mu2;
    __device__ __forceinline__ explicit ApConst(const Phys<float>& ph)
        : k(ph.k), a(ph.a), it(ph.inv_ts), eps0(ph.eps0), mu1(ph.mu1), mu2(ph.mu2) {}
};

// The Aliev-Panfilov reaction I (without its time scale) and z = v_inf - w, which share k u and u - a.
// The cubic stays a product of its factors: expanded to u (k (u (u - a - 1) + a) + w) it cancels near
// u = 1 and u = a (largest FP32 error for u in 0.98 .. 1.02 3.2e-7 against 1.7e-8), and the state's
// fixed points are none.
template <typename R>
__device__ __forceinline__ void ap_forms(R k, R a, R u, R w, R& I, R& z) {
    const R ku = k * u, ua = u - a;
    I = ku * ua * (u - R(1)) + u * w;
    z = -ku * (ua - R(1)) - w;
}

// dof_update of W DOFs under the Aliev-Panfilov model (ionic 0) with the exponential state step
// (integrator 1) in FP32: straight-line code, so that the DOFs interleave.  V and w are updated by
// one addition of their increment, and the midpoints take half of it.  e^x - 1
// (x = -eps dt / time scale) is the exponential's Taylor series: through
// x^4 while every |x| < 2^-7 (truncation below 4e-11 relative; all explicit substeps in practice),
// else expm1_f32.  first: the elements' first step of the barrier, which sets Ia and ga to I and g
// at the step start; otherwise they are inputs.  r: M^-1 A u up to the factor sc.  Returns the sum
// of mq [dI^2 + dg^2].
template <int W>
__device__ __forceinline__ float ap_step(const ApConst& c, const bool first, const float* mq, float sc, float dte,
                                         const float* so, const float* sm, const float* u, const float* w,
                                         const float* r, float* Ia, float* ga, float* un, float* wn) {
    float I[W], z[W], x[W], mx = 0.0f;
    const float xt = -dte * c.it;
#pragma unroll
    for (int j = 0; j < W; ++j) {
        float i0;
        ap_forms(c.k, c.a, u[j], w[j], i0, z[j]);
        I[j] = i0 * c.it + so[j];
        const float den = fmaxf(u[j] + c.mu2, 1e-6f);
        const float eps = c.eps0 + __fdividef(c.mu1 * w[j], den);
        x[j] = eps * xt;
        mx = fmaxf(mx, fabsf(x[j]));
        if (first) {
            Ia[j] = I[j];
            ga[j] = eps * z[j] * c.it;
        }
    }
    if (mx < 0.0078125f) {
#pragma unroll
        for (int j = 0; j < W; ++j) {
            const float t = x[j];
            x[j] = t * (1.0f + t * (0.5f + t * (1.0f / 6.0f + t * (1.0f / 24.0f))));
        }
    } else {
#pragma unroll
        for (int j = 0; j < W; ++j) x[j] = expm1_f32(x[j]);
    }
    float term = 0.0f;
#pragma unroll
    for (int j = 0; j < W; ++j) {
        const float du = dte * (-r[j] * sc - I[j]);
        const float dw = -z[j] * x[j];
        un[j] = u[j] + du;
        wn[j] = w[j] + dw;
        const float Vm = u[j] + 0.5f * du, wm = w[j] + 0.5f * dw;
        float i1, z1;
        ap_forms(c.k, c.a, Vm, wm, i1, z1);
        const float dI = i1 * c.it + (sm[j] - Ia[j]);
        const float den = fmaxf(Vm + c.mu2, 1e-6f);
        const float eps = c.eps0 + __fdividef(c.mu1 * wm, den);
        const float dg = eps * z1 * c.it - ga[j];
        term += mq[j] * (dI * dI + dg * dg);
    }
    return term;
}

static __device__ __noinline__ double expm1_call(double x) { return expm1(x); }   // (out of line: rarely taken)

// e^x - 1 in FP64: the Taylor series of the exponential through x^8 for |x| < 2^-7 (truncation
// below 1e-20 relative), else expm1.
__device__ __forceinline__ double expm1_f64(double x) {
    if (fabs(x) < 0.0078125)
        return x * (1.0 + x * (0.5 + x * (1.0 / 6.0 + x * (1.0 / 24.0 + x * (1.0 / 120.0 + x * (1.0 / 720.0 +
               x * (1.0 / 5040.0 + x * (1.0 / 40320.0))))))));
    return expm1_call(x);
}

// The FP64 Aliev-Panfilov step of one DOF with the products shared as in ap_step, for either state
// integrator: FP64 instructions issue at 1/64 of the FP32 rate, and the separate forms of I, g and
// the state step took about 110 of them.  Returns mq [dI^2 + dg^2].
__device__ __forceinline__ double ap_step_f64(const Phys<double>& ph, const bool first, double mq, double sc, double dte,
                                              double so, double sm, double u, double w, double r, double& Ia,
                                              double& ga, double& un, double& wn) {
    const double it = ph.inv_ts;
    auto eps_of = [&](double V, double s) {
        double den = V + ph.mu2;
        den = den > 1e-6 ? den : 1e-6;
        return ph.eps0 + ph.mu1 * s / den;
    };
    double i0, z, i1, z1;
    ap_forms(ph.k, ph.a, u, w, i0, z);
    const double I = i0 * it + so;
    const double eps = eps_of(u, w) * it;
    if (first) {
        Ia = I;
        ga = eps * z;
    }
    const double du = dte * (-r * sc - I);
    const double dw = ph.integrator == 0 ? dte * eps * z : -z * expm1_f64(-eps * dte);
    un = u + du;
    wn = w + dw;
    const double Vm = u + 0.5 * du, wm = w + 0.5 * dw;
    ap_forms(ph.k, ph.a, Vm, wm, i1, z1);
    const double dI = i1 * it + sm - Ia;
    const double dg = eps_of(Vm, wm) * it * z1 - ga;
    return mq * (dI * dI + dg * dg);
}

// dof_update through the shared forms where they apply.
template <typename R>
__device__ __forceinline__ R dof_update_any(const Phys<R>& ph, R Mq, R Minv, int ke, R dte, R so, R sm, R u, R w, R r,
                                            R& Ia, R& ga, R& un, R& wn) {
    if constexpr (sizeof(R) == 8) {
        if (ph.ionic == 0) return ap_step_f64(ph, ke == 0, Mq, Minv, dte, so, sm, u, w, r, Ia, ga, un, wn);
    }
    return dof_update<R>(ph, Mq, Minv, ke, dte, so, sm, u, w, r, Ia, ga, un, wn);
}

// Pointwise part of one element step (Alg. 1) given the residual: Q1 r = (A u)_e (the GL
// masses of an element are equal), Q2 rho = (M^-1 A u)_e in level-0 units (4^lev scales it); returns the element's RV-T term, vmax = max_q |V_new|.
template <typename R, int DIM, int P>
__device__ __forceinline__ R elem_pointwise(const TickArgs<R>& a, const Phys<R>& ph, const OpT<R, DIM, P>& op, int tick,
                                            int e, uint32_t inf, int b, int ke, int lev, const R* u, const R* w,
                                            const R* r, R* Ia, R* ga, R* un, R* wn, R& vmax) {
    constexpr int NP = Shape<DIM, P>::NP;
    const double dte_d = a.dte[b];
    const R dte = a.dteR[b];
    const R sc = P == 1 ? ph.Minv[lev][0] : R(1 << (2 * lev));
    R term = R(0);
    vmax = R(0);
    StimMasks stm;
    elem_stim<R>(a, e, inf, tick, dte_d, stm);
    if constexpr (sizeof(R) == 4) {
        // Aliev-Panfilov, exponential state step: the straight-line update, so that the element's
        // DOFs interleave
        if (ph.ionic == 0 && ph.integrator == 1) {
            R so[NP], smd[NP];
#pragma unroll
            for (int q = 0; q < NP; ++q) node_stim<R>(a, stm, q, so[q], smd[q]);
            term = ph.Wvol[lev] * ap_step<NP>(ApConst(ph), ke == 0, op.wq, sc, dte, so, smd, u, w, r, Ia, ga, un, wn);
#pragma unroll
            for (int q = 0; q < NP; ++q) vmax = fmaxf(vmax, fabsf(un[q]));
            return term;
        }
    }
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        R so, smd;
        node_stim<R>(a, stm, q, so, smd);
        term += dof_update_any<R>(ph, ph.Wvol[lev] * op.wq[q], sc, ke, dte, so, smd, u[q], w[q], r[q], Ia[q], ga[q], un[q],
                              wn[q]);
        const R av = un[q] < R(0) ? -un[q] : un[q];
        vmax = av > vmax ? av : vmax;
    }
    return term;
}

// Four consecutive values of a row (16-byte vectors; FP64 as two).
template <typename R>
__device__ __forceinline__ void ld4(const R* p, R* x) { ld_vec<R, 4>(p, x); }
template <typename R>
__device__ __forceinline__ void st4(R* p, const R* x) { st_vec<R, 4>(p, x); }

// Pointwise part of a Q2 3D element step, four DOFs at a time in a loop (unrolled, its code alone
// is 20 KB): rho in `rw` (28 values, pad 0), the rows of the element streamed with the next four
// DOFs' loads in flight.  The pad value steps too and stays 0 (its weight is 0).
template <typename R>
__device__ __forceinline__ R pointwise_q23(const TickArgs<R>& a, const Phys<R>& ph, const BoxOp<R>& op, int tick, int e,
                                           uint32_t inf, int b, int ke, int lev, const R* Vc, R* Vd, const R* rw,
                                           R& vmax) {
    constexpr int NPS = 28;
    const DevArrays<R>& d = a.d;
    const size_t o = (size_t)e * NPS;
    R* const vp = d.v + o;
    R* const Ip = d.Ia + o;
    R* const gp = d.ga + o;
    const R dte = a.dteR[b], sc = R(1 << (2 * lev)), Wv = ph.Wvol[lev];
    const bool first = ke == 0, keep = first && b > 0;
    const bool ap = sizeof(R) == 4 && ph.ionic == 0 && ph.integrator == 1;   // (one for all threads)
    StimMasks stm;
    elem_stim<R>(a, e, inf, tick, a.dte[b], stm);
    R term = R(0);
    vmax = R(0);
    R u[4], w[4], Ia[4], ga[4];
    auto load = [&](int i, R* u_, R* w_, R* I_, R* g_) {
        ld4<R>(Vc + 4 * i, u_);
        ld4<R>(vp + 4 * i, w_);
        if (!first) {
            ld4<R>(Ip + 4 * i, I_);
            ld4<R>(gp + 4 * i, g_);
        }
    };
#pragma unroll
    for (int k = 0; k < 4; ++k) Ia[k] = ga[k] = R(0);
    load(0, u, w, Ia, ga);
#pragma unroll 1
    for (int i = 0; i < 7; ++i) {
        R u2[4], w2[4], I2[4], g2[4], r[4], un[4], wn[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) I2[k] = g2[k] = R(0);
        if (i < 6) load(i + 1, u2, w2, I2, g2);
        else {
#pragma unroll
            for (int k = 0; k < 4; ++k) u2[k] = w2[k] = R(0);
        }
        ld4<R>(rw + 4 * i, r);
        R so[4], smd[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) node_stim<R>(a, stm, 4 * i + k, so[k], smd[k]);
        if constexpr (sizeof(R) == 4) {
            if (ap)
                term += ap_step<4>(ApConst(ph), first, op.wq + 4 * i, sc, dte, so, smd, u, w, r, Ia, ga, un, wn);
        }
        if (!ap) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                term += dof_update_any<R>(ph, op.wq[4 * i + k], sc, ke, dte, so[k], smd[k], u[k], w[k], r[k], Ia[k],
                                      ga[k], un[k], wn[k]);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const R av = un[k] < R(0) ? -un[k] : un[k];
            vmax = av > vmax ? av : vmax;
        }
        st4<R>(Vd + 4 * i, un);
        st4<R>(vp + 4 * i, wn);
        if (keep) {
            st4<R>(Ip + 4 * i, Ia);
            st4<R>(gp + 4 * i, ga);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            u[k] = u2[k];
            w[k] = w2[k];
            Ia[k] = I2[k];
            ga[k] = g2[k];
        }
    }
    return Wv * term;
}

// One element step of Alg. 1 at tick `tick`: forward Euler on V, exponential/FE step on
// v, the RV-T accumulation and the element's probe check.
template <typename R, int DIM, int P>
__device__ __forceinline__ void tick_elem(const TickArgs<R>& a, const Tables<R>& T, const Phys<R>& ph,
                                          const OpT<R, DIM, P>& op, int tick, const TickMeta<DIM, P>& m,
                                          double t_tick) {
    using S = Shape<DIM, P>;
    constexpr int NP = S::NP, NPS = S::NPS;
    const DevArrays<R>& d = a.d;
    const int e = m.e;
    const uint32_t inf = m.inf;
    const int b = m.lv & 7, par = (m.lv >> 3) & 1;
    const int ke = tick >> (a.B - b);
    const int cur = par ^ (ke & 1);
    const int lev = (inf >> 24) & 15;
    const R* Vc = (cur ? d.V1 : d.V0) + (size_t)e * NPS;
    R* Vd = (cur ? d.V0 : d.V1) + (size_t)e * NPS;
    R* vp = d.v + (size_t)e * NPS;
    const double dte_d = a.dte[b];
    const double acc0 = ke != 0 ? d.acc[e] : 0.0;
    const bool pend = (inf & INFO_PENDING) != 0;
    R vmax;
    if constexpr (DIM == 3 && P == 2) {
        R rl[NPS];                      // rho, read back in a loop: local memory
        {
            R u[NP], rho[NP];
            ld_dofs<R, NP, NPS>(Vc, u);
            box_residual_q23<R>(d, op, tick, a.B, m, u, rho);
#pragma unroll
            for (int q = 0; q < NPS; ++q) rl[q] = q < NP ? rho[q] : R(0);
        }
        const R term = pointwise_q23<R>(a, ph, op, tick, e, inf, b, ke, lev, Vc, Vd, rl, vmax);
        d.acc[e] = acc0 + dte_d * (double)term;
        if (pend && vmax >= ph.lat_gate)
            lat_check<R, DIM, P>(d, T, ph, e, inf, lev, Vc, Vd, t_tick >= 0.0 ? t_tick : tick_time(a, tick), dte_d);
    } else {
        // every value this step needs is addressed by now: issue the loads together
        R u[NP], w[NP], r[NP], Ia[NP], ga[NP];
        ld_dofs<R, NP, NPS>(Vc, u);
        ld_dofs<R, NP, NPS>(vp, w);
        if (ke != 0) {
            ld_dofs<R, NP, NPS>(d.Ia + (size_t)e * NPS, Ia);
            ld_dofs<R, NP, NPS>(d.ga + (size_t)e * NPS, ga);
        }
        if constexpr (P == 1) residual_q1<R, DIM>(d, op, tick, a.B, m, lev, u, r);
        else box_residual<R, DIM, P>(d, op, tick, a.B, m, u, r);
        R un[NP], wn[NP];
        const R term = elem_pointwise<R, DIM, P>(a, ph, op, tick, e, inf, b, ke, lev, u, w, r, Ia, ga, un, wn, vmax);
        if (ke == 0 && b > 0) {
            st_dofs<R, NP, NPS>(d.Ia + (size_t)e * NPS, Ia);
            st_dofs<R, NP, NPS>(d.ga + (size_t)e * NPS, ga);
        }
        st_dofs<R, NP, NPS>(Vd, un);
        st_dofs<R, NP, NPS>(vp, wn);
        d.acc[e] = acc0 + dte_d * (double)term;
        if (pend && vmax >= ph.lat_gate) {
            const double tt = t_tick >= 0.0 ? t_tick : tick_time(a, tick);
            if constexpr (P == 1)
                lat_check_at<R, DIM, P>(d, T, ph, e, inf, lev, m.lc, m.rid, u, un, tt, dte_d, m.pend, true);
            else lat_check<R, DIM, P>(d, T, ph, e, inf, lev, u, un, tt, dte_d);
        }
    }
}

// One tick of Alg. 1 over the due elements (a prefix of `order`), for callers that
// already waited for the previous tick.
template <typename R, int DIM, int P>
__device__ __forceinline__ void tick_work(const TickArgs<R>& a, const Tables<R>& T, const Phys<R>& ph,
                                          const OpT<R, DIM, P>& op, int tick) {
    const int n_act = a.d.meta->nact[tick];
    const double t_tick = -1.0;   // computed where a probe check needs it
    for (int idx = (int)gtid(); idx < n_act; idx += (int)gstride()) {
        TickMeta<DIM, P> m;
        tick_fetch<R, DIM, P>(a.d, idx, m);
        tick_elem<R, DIM, P>(a, T, ph, op, tick, m, t_tick);
    }
}

// (The bound's "1" lets the Q1 2D FP32 step keep its 168 registers: under the default heuristic
// the compiler held it to 128 and spilled 40 bytes, and the C2 sweep ran 11% slower.)
template <typename R, int DIM, int P>
__global__ void __launch_bounds__(256, 1) k_tick(
    const TickArgs<R> a, const Tables<R> T, const Phys<R> ph, const OpT<R, DIM, P> op) {
    // the due count and the first element's metadata are fixed during the sweep: read them
    // while the previous tick drains, then wait for its values (the first tick of a sweep
    // is launched without overlap, after the ordering that writes them)
    // (so are the tick's time and the error word: ticks do not set errors)
    const int n_act = a.d.meta->nact[a.tick];
    const bool bad = a.d.meta->err != 0;
    const int idx0 = (int)gtid();
    TickMeta<DIM, P> m;
    if (idx0 < n_act) tick_fetch<R, DIM, P>(a.d, idx0, m);
    // the tick's time (FP64, a slow pipe here) only where a probe check may need it
    const double t_tick = (idx0 < n_act && (m.inf & INFO_PENDING)) ? tick_time(a, a.tick) : -1.0;
    pdl_enter();
    if (bad) return;
    for (int idx = idx0; idx < n_act; idx += (int)gstride()) {
        if (idx != idx0) tick_fetch<R, DIM, P>(a.d, idx, m);
        tick_elem<R, DIM, P>(a, T, ph, op, a.tick, m, t_tick);
    }
}

// Refinement marks of an adapting barrier, set by the kernel that computes the indicator: a leaf
// whose eta^s reaches tau is marked unless it is at full depth, and under the 2:1 closure a marked
// leaf marks its coarser face neighbours, theirs in turn, and so on.  Chains only go coarser, from a
// leaf below full depth: up to max_refine - 1 leaves.  Two are followed here (a stack for longer ones
// would give the kernel local memory, which cost 5 us a launch); k_amr_close takes the rest, a pass
// per step.  The marks r are 0 at the start of the kernel (the level pass of the previous barrier
// clears them); two threads that mark a leaf at once write the same.
constexpr int MARK_CHAIN = 2;
struct MarkArgs {
    uint8_t* r;          // null: no adaptation
    double tau;
    int L;
};

template <int DIM>
__device__ __forceinline__ void mark_leaf(const MarkArgs& a, const uint32_t* info, const int32_t* nbr, int64_t e,
                                          uint32_t inf, double eta) {
    constexpr int NF = 2 * DIM;
    if (!(eta >= a.tau) || (int)((inf >> 24) & 15) >= a.L) return;
    a.r[e] = 1;
#pragma unroll 1
    for (int f = 0; f < NF; ++f) {
        if (((inf >> (4 * f)) & 3u) != 2u) continue;
        const int32_t c = nbr[(size_t)e * NF + f];
        const uint32_t ic = info[c];
        a.r[c] = 1;
#pragma unroll 1
        for (int g = 0; g < NF; ++g)
            if (((ic >> (4 * g)) & 3u) == 2u) a.r[nbr[(size_t)c * NF + g]] = 1;
    }
}

// Kelly-type spatial indicator per element (Eq. dg-error-estimate) on the barrier-start
// values; same-level and coarser neighbours are gathered before the face arithmetic.  In
// FP32 the face-point sums are FP32 and the faces accumulate in FP64 (FP64 arithmetic per
// face point would bound the kernel by the FP64 pipe).  Q1; see k_eta_s_q2 and k_eta_q23 for Q2.
template <typename R, int DIM, int P>
__global__ void k_eta_s(const DevArrays<R> d, const Tables<R> T, const Phys<R> ph, const MarkArgs mark) {
    static_assert(P == 1, "Q1");
    pdl_enter();
    using S = Shape<DIM, P>;
    constexpr int NP = S::NP, NF = S::NF, NSUB = S::NSUB, NPS = S::NPS;
    if (d.meta->err) return;
    if (gtid() == 0) d.meta->changed = 0u;
    const int64_t ne = d.meta->ne;
    for (int64_t e = gtid(); e < ne; e += gstride()) {
        const uint32_t inf = d.info[e];
        const int lev = (inf >> 24) & 15;
        const int par = (d.lvl[e] >> 3) & 1;
        const R* Vc = (par ? d.V1 : d.V0) + (size_t)e * NPS;
        R u[NP];
        ld_dofs<R, NP, NPS>(Vc, u);
        // squared face jumps in the working precision, summed in FP64 (the indicator decides
        // refinement, so its reduction keeps FP64 as on the host)
        double acc = 0.0;
        int nbf[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) nbf[f] = d.nbr[(size_t)e * NF + f];
        int src[NF];
        uint8_t lvn[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const int kind = (inf >> (4 * f)) & 3;
            src[f] = (kind == 1 || kind == 2) ? nbf[f] : (int)e;
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) lvn[f] = d.lvl[src[f]];
        R un[NF][NP];
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const R* srcp = (((lvn[f] >> 3) & 1) ? d.V1 : d.V0) + (size_t)src[f] * NPS;
            ld_dofs<R, NP, NPS>(srcp, un[f]);
        }
        constexpr int NT = S::NT, NREL = 1 + 2 * NSUB;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const int kind = (inf >> (4 * f)) & 3;
            if (kind != 1 && kind != 2) continue;
            const int rel = kind == 1 ? 0 : 1 + ((inf >> (4 * f + 2)) & 3);
            const R* K = d.qkelly + ((((size_t)f * 8 + lev) * NREL + rel) * 2) * NT * NP;
            R j[NT];
#pragma unroll
            for (int t = 0; t < NT; ++t) j[t] = R(0);
            block_jump<R, NT, NP>(K, u, j);
            block_jump<R, NT, NP>(K + NT * NP, un[f], j);
            R fsum = R(0);
#pragma unroll
            for (int t = 0; t < NT; ++t) fsum += j[t] * j[t];
            acc += (double)fsum;
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const int kind = (inf >> (4 * f)) & 3;
            if (kind != 3) continue;
            for (int sb = 0; sb < NSUB; ++sb) {
                const int nb = d.hang[nbf[f] + sb];
                const int pn = (d.lvl[nb] >> 3) & 1;
                const R* src = (pn ? d.V1 : d.V0) + (size_t)nb * NPS;
                R un[NP];
                ld_dofs<R, NP, NPS>(src, un);
                const R* K = d.qkelly + ((((size_t)f * 8 + lev) * NREL + 1 + NSUB + sb) * 2) * NT * NP;
                R j[NT];
#pragma unroll
                for (int t = 0; t < NT; ++t) j[t] = R(0);
                block_jump<R, NT, NP>(K, u, j);
                block_jump<R, NT, NP>(K + NT * NP, un, j);
                R fsum = R(0);
#pragma unroll
                for (int t = 0; t < NT; ++t) fsum += j[t] * j[t];
                acc += (double)fsum;
            }
        }
        const double eta = sqrt(acc);
        d.eta_s[e] = eta;
        if (mark.r) mark_leaf<DIM>(mark, d.info, d.nbr, e, inf, eta);
    }
}

// Kelly term of one (sub)face of a Q2 element, sum_t w_t jump_t^2 (times the face weight of the
// finer side's level, 4^lo and kfac): the flux jump at the face points from the traces of both
// sides, one-dimensional derivatives along the face and, across a change of level, the
// interpolation to the finer side's points.  to, dno: own trace and normal derivative; v: the
// neighbour's values; kind 3: of subface pos.
template <typename R, int DIM>
__device__ __forceinline__ R kelly_face(const BoxOp<R>& op, const Tables<R>& T, int k, int side, int kind, int pos,
                                        const R* to, const R* dno, const R* v) {
    constexpr int NT = Shape<DIM, 2>::NT;
    R tn[NT], dn[NT], dt[NT], dd[NT];
    box_trace<R, DIM, 2>(op, k, 1 - side, v, tn, dn);
    R ft = R(1);                       // tangential derivatives in the finer side's length
    if (kind == 1) {
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            dd[t] = dno[t] - dn[t];
            dt[t] = to[t] - tn[t];
        }
    } else {
        // the coarser side's values at the finer side's points
        R a[NT], b[NT];
        const int c0 = pos & 1, c1 = (pos >> 1) & 1;
        if (kind == 2) {
            face_map<R, DIM, 2>(op.PR[0], c0, c1, tn, a);
            face_map<R, DIM, 2>(op.PR[0], c0, c1, dn, b);
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                dd[t] = dno[t] - R(0.5) * b[t];
                dt[t] = to[t] - a[t];
            }
        } else {
            face_map<R, DIM, 2>(op.PR[0], c0, c1, to, a);
            face_map<R, DIM, 2>(op.PR[0], c0, c1, dno, b);
            ft = R(2);
#pragma unroll
            for (int t = 0; t < NT; ++t) {
                dd[t] = b[t] - R(2) * dn[t];
                dt[t] = a[t] - tn[t];
            }
        }
    }
    R j[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) j[t] = op.FK[k][k] * dd[t];
    if (op.cross) {
        int tg[2] = {0, 0};
        tangents<DIM>(k, tg);
#pragma unroll
        for (int ti = 0; ti < DIM - 1; ++ti) face_line<R, DIM, 2>(op.D1, ti, ft * op.FK[k][tg[ti]], dt, j, true);
    }
    R s = R(0);
#pragma unroll
    for (int t = 0; t < NT; ++t) {
        const R w = DIM == 3 ? T.w[t % 3] * T.w[t / 3] : T.w[t];
        s += w * j[t] * j[t];
    }
    return s;
}

// The indicator's terms of the two axis-K faces of a Q2 element from its values y; row(n, v): values of element n, both shifted
// by a value of the element (the flux jump does not see a constant).  nbv(k, side, v): those of the
// same-level neighbour of a face.
template <typename R, int DIM, int K, typename ROW, typename NBV>
__device__ __forceinline__ double kelly_axis(const DevArrays<R>& d, const BoxOp<R>& op, const Tables<R>& T,
                                             const Phys<R>& ph, int64_t e, uint32_t inf, int lev, const R* y, ROW row,
                                             NBV nbv) {
    using S = Shape<DIM, 2>;
    constexpr int NP = S::NP, NF = S::NF, NT = S::NT;
    constexpr int k = K;
    double acc = 0.0;
    const R sc = R(1 << (2 * lev));
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {
            const uint32_t fi = inf >> (8 * k + 4 * side);
            const int kind = fi & 3;
            if (kind == 0) continue;
            R to[NT], dno[NT], v[NP];
            box_trace<R, DIM, 2>(op, k, side, y, to, dno);
            const int sb0 = kind == 3 ? 0 : (fi >> 2) & 3, sb1 = kind == 3 ? S::NSUB : sb0 + 1;
            const int lf = kind == 3 ? lev + 1 : lev;
            R s = R(0);
#pragma unroll 1
            for (int sb = sb0; sb < sb1; ++sb) {
                if (kind == 1) nbv(k, side, v);
                else {
                    const int nbi = d.nbr[(size_t)e * NF + 2 * k + side];
                    row(kind == 2 ? nbi : d.hang[nbi + sb], v);
                }
                s += kelly_face<R, DIM>(op, T, k, side, kind, sb, to, dno, v);
            }
            acc += ph.kfac[lf][k] * (double)(ph.Wface[lf][k] * sc * s);
        }
    return acc;
}

template <typename R, int DIM>
__global__ void __launch_bounds__(128) k_eta_s_q2(const DevArrays<R> d, const Tables<R> T, const Phys<R> ph,
                                                  const BoxOp<R> op, const MarkArgs mark) {
    pdl_enter();
    using S = Shape<DIM, 2>;
    constexpr int NP = S::NP, NPS = S::NPS, NF = S::NF;
    if (d.meta->err) return;
    if (gtid() == 0) d.meta->changed = 0u;
    const int64_t ne = d.meta->ne;
    for (int64_t e = gtid(); e < ne; e += gstride()) {
        const uint32_t inf = d.info[e];
        R y[NP];
        ld_dofs<R, NP, NPS>((((d.lvl[e] >> 3) & 1) ? d.V1 : d.V0) + (size_t)e * NPS, y);
        const R c = y[NP / 2];
        auto row = [&](int n, R* v) {
            ld_dofs<R, NP, NPS>((((d.lvl[n] >> 3) & 1) ? d.V1 : d.V0) + (size_t)n * NPS, v);
#pragma unroll
            for (int q = 0; q < NP; ++q) v[q] -= c;
        };
#pragma unroll
        for (int q = 0; q < NP; ++q) y[q] -= c;
        auto nbv = [&](int k, int side, R* v) { row(d.nbr[(size_t)e * NF + 2 * k + side], v); };
        const int lev = (inf >> 24) & 15;
        double acc = kelly_axis<R, DIM, 0>(d, op, T, ph, e, inf, lev, y, row, nbv);
        acc += kelly_axis<R, DIM, 1>(d, op, T, ph, e, inf, lev, y, row, nbv);
        if constexpr (DIM == 3) acc += kelly_axis<R, DIM, DIM - 1>(d, op, T, ph, e, inf, lev, y, row, nbv);
        const double eta = sqrt(acc);
        d.eta_s[e] = eta;
        if (mark.r) mark_leaf<DIM>(mark, d.info, d.nbr, e, inf, eta);
    }
}

// Square root of a >= 0 in FP64 from an FP32 seed and two Newton steps (each squares the relative
// error, 2^-22 to start with): 5 FP64 operations, which issue at 1/64 of the FP32 rate here.  With the
// seed up to 2 ulp off the result is the rounded root for all but 5e-5 of 2e7 random arguments, and
// the value next to it for those; FP32 contexts only, whose a carries 1e-7.
__device__ __forceinline__ double sqrt_seeded(double a) {
    if (a == 0.0) return 0.0;
    const float f = (float)a;
    if (!(f > 1e-30f && f < 1e30f)) return sqrt(a);
    const double y = (double)rsqrtf(f), h = 0.5 * y;
    double s = a * y;
    s = fma(fma(-s, s, a), h, s);
    return fma(fma(-s, s, a), h, s);
}

// Weights of int V on box elements of level 0: GL weight products times the volume factor (0 past the
// last node).  Level l scales them by 2^(-d l), exact.
struct EpiWeights {
    double w[28];
};

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Sum over the block (of at most 1024 threads), valid in thread 0.
__device__ __forceinline__ double block_sum(double x) {
    __shared__ double part[32];
    x = warp_sum(x);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x < 32) x = warp_sum(threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.0);
    __syncthreads();
    return x;
}

// Barrier epilogue: eta^t = sqrt(acc)/dt, parity flip of single-step elements, non-finite
// check, per-block partial sums of int V = sum_q M_q V_q in FP64, in either precision of the field.
// The FP64 pipe bounds it (1.25 TFLOP/s; a conversion and a multiply-add a DOF): sums in pairs of
// FP32 values took 0.21 ms less of a 6.2 ms barrier step on 2.79 M Q2 3D elements, but their error
// grows with the elements a thread takes (3e-13 of the integral of a constant field at nine).  FP32
// rows of 27 values are read by whole warps (see mdl_q23.cuh): a lane holds four consecutive values of
// a row and adds their weighted sum; shorter rows, FP64 ones and those of curved elements
// (per-element masses) are read by their element's thread.
template <typename R, int DIM, int P>
__global__ void __launch_bounds__(256) k_epilogue(const DevArrays<R> d, const double* __restrict__ mtab,
                                                 const EpiWeights ew, double dt, double inv_dt, int inv_dt_exact,
                                                 int mass_per_elem) {
    using S = Shape<DIM, P>;
    constexpr int NP = S::NP, NPS = S::NPS;
    constexpr bool F32 = sizeof(R) == 4, COOP = F32 && NPS != NP;
    __shared__ double sw[28];
    if (COOP) {
        if (threadIdx.x < 28) sw[threadIdx.x] = ew.w[threadIdx.x];
        __syncthreads();
    }
    pdl_enter();
    if (d.meta->err) return;
    const int64_t ne = d.meta->ne;
    double loc = 0.0;
    float nf = 0.0f;                 // not 0 once a value was not finite
    const int lane = threadIdx.x & 31;
    for (int64_t base = gtid() - lane; base < ne; base += gstride()) {
        const int64_t e = base + lane;
        const bool in = e < ne;
        uint8_t lv = 0;
        int lev = -1;
        if (in) {
            // eta^t = sqrt(acc) / dt in FP64 (it sets b^cell); the product with 1/dt equals the
            // quotient whenever dt is a power of two, as the automatic barrier step is
            const double a = d.acc[e], r = F32 ? sqrt_seeded(a) : sqrt(a);
            d.eta_t[e] = inv_dt_exact ? r * inv_dt : r / dt;
            lv = d.lvl[e];
            if ((lv & 7) == 0) {
                lv ^= 8;
                d.lvl[e] = lv;
            }
            lev = (d.info[e] >> 24) & 15;
        }
        const R* Vc = (((lv >> 3) & 1) ? d.V1 : d.V0) + (size_t)(in ? e : base) * NPS;
        const R* w = d.v + (size_t)(in ? e : base) * NPS;
        if (COOP && !mass_per_elem) {
            if constexpr (COOP) {
#pragma unroll
                for (int j = 0; j < 7; ++j) {
                    const int t = 32 * j + lane, r = t / 7, c = t - 7 * r;
                    const float4 x = reinterpret_cast<const float4*>(__shfl_sync(0xffffffffu, (long long)Vc, r))[c];
                    const float4 y = reinterpret_cast<const float4*>(__shfl_sync(0xffffffffu, (long long)w, r))[c];
                    const int lr = __shfl_sync(0xffffffffu, lev, r);
                    const double sum = sw[4 * c] * (double)x.x + sw[4 * c + 1] * (double)x.y +
                                       sw[4 * c + 2] * (double)x.z + sw[4 * c + 3] * (double)x.w;
                    if (lr >= 0) loc += pow2_neg<double>(DIM * lr) * sum;
                    nf += 0.0f * x.x + 0.0f * x.y + 0.0f * x.z + 0.0f * x.w;
                    nf += 0.0f * y.x + 0.0f * y.y + 0.0f * y.z + 0.0f * y.w;
                }
            }
        } else if (in) {
            R x[NP], y[NP];
            ld_dofs<R, NP, NPS>(Vc, x);
            ld_dofs<R, NP, NPS>(w, y);
            // GL masses: per (level, node) on box elements, per (element, node) on mapped ones
            const double* Mq = mtab + (mass_per_elem ? (size_t)e * NP : (size_t)lev * NP);
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                loc += Mq[q] * (double)x[q];
                if (!isfinite(x[q]) || !isfinite(y[q])) nf = 1.0f;
            }
        }
    }
    if (!(nf == 0.0f)) atomicOr(&d.meta->nf_pending, 1u);
    loc = block_sum(loc);
    __shared__ bool last;
    if (threadIdx.x == 0) {
        d.partial[blockIdx.x] = loc;
        __threadfence();
        last = atomicAdd(&d.meta->done_blocks, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    // the last block: fixed-order sum of the partials, barrier count, non-finite flag
    __threadfence();
    double s2 = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) s2 += __ldcg(d.partial + i);
    s2 = block_sum(s2);
    if (threadIdx.x == 0) {
        DevMeta* m = d.meta;
        m->integral = s2;
        m->nbar += 1;
        m->done_blocks = 0;
        if (*(volatile unsigned*)&m->nf_pending) {
            m->err |= ERR_NONFINITE;
            m->nf_pending = 0;
        }
    }
}



// Q1 tick with a group of G = (p+1)^d lanes per element (4 in 2D, 8 in 3D), lane g owning
// DOF g: it computes row g of the residual from the class blocks (r_g = A_vol[g] u +
// sum_f A_own,f[g] u + A_nb,f[g] u_nb,f) and the pointwise step of DOF g, so G times more
// threads are in flight than with a thread per element and each runs a short chain.
// Everything fixed during the sweep -- the element, its level byte and face info, its
// neighbours and their level bytes, and in 2D the block rows -- is read before waiting for
// the previous tick; after the wait every value load is issued at once.
template <typename R, int DIM>
struct GroupMeta {
    static constexpr int NP = Shape<DIM, 1>::NP, NF = 2 * DIM;
    static constexpr bool ROWS = DIM == 2;     // block rows held in registers (2D only)
    int e;
    uint32_t inf;
    uint8_t lv;
    int nbf[NF];
    uint8_t lvn[NF];
    R vrow[NP];
    R orow[ROWS ? NF : 1][NP];
    R nrow[ROWS ? NF : 1][NP];
};

template <typename R, int DIM>
__device__ __forceinline__ void group_fetch(const DevArrays<R>& d, int64_t idx, int g, GroupMeta<R, DIM>& m) {
    using M = GroupMeta<R, DIM>;
    constexpr int NP = M::NP, NF = M::NF, NREL = 1 + 2 * Shape<DIM, 1>::NSUB;
    m.e = d.order[idx];
    m.lv = d.lvl[m.e];
    m.inf = d.info[m.e];
#pragma unroll
    for (int f = 0; f < NF; ++f) m.nbf[f] = d.nbr[(size_t)m.e * NF + f];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const int kind = (m.inf >> (4 * f)) & 3;
        m.lvn[f] = d.lvl[(kind == 1 || kind == 2) ? m.nbf[f] : m.e];
    }
    const int lev = (m.inf >> 24) & 15;
    ld_row<R, NP>(d.qvol + ((size_t)lev * NP + g) * NP, m.vrow);
    if constexpr (M::ROWS) {
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const int kind = (m.inf >> (4 * f)) & 3;
            const int rel = kind == 2 ? 1 + ((m.inf >> (4 * f + 2)) & 3) : 0;
            const R* A = d.qface + ((((size_t)f * 8 + lev) * NREL + rel) * 2) * NP * NP;
            ld_row<R, NP>(A + g * NP, m.orow[f]);
            ld_row<R, NP>(A + NP * NP + g * NP, m.nrow[f]);
        }
    }
}

template <typename R, int DIM>
__global__ void __launch_bounds__(256) k_tick_group(const TickArgs<R> a, const Phys<R> ph, const Tables<R> T) {
    using S = Shape<DIM, 1>;
    using M = GroupMeta<R, DIM>;
    constexpr int N1 = S::N1, NP = S::NP, NF = S::NF, NSUB = S::NSUB, NREL = 1 + 2 * NSUB;
    constexpr int G = NP;
    const DevArrays<R>& d = a.d;
    const int tick = a.tick, B = a.B;
    const int lane = threadIdx.x & 31;
    const int g = lane % G;
    const unsigned gmask = ((1u << G) - 1u) << (lane - g);
    const int64_t gsz = gstride() / G;
    // per (level, node) GL mass and inverse in shared memory (lanes read different nodes)
    __shared__ R sMq[8 * NP], sMinv[8 * NP];
    for (int i = threadIdx.x; i < 8 * NP; i += blockDim.x) {
        const int l = i / NP, q = i - l * NP;
        R w = ph.Wvol[l];
#pragma unroll
        for (int k = 0; k < DIM; ++k) w *= T.w[digit<N1>(q, k)];
        sMq[i] = w;
        sMinv[i] = ph.Minv[l][q];
    }
    // the due count, the element order and the error word do not change during a sweep
    // (the first tick of a sweep is launched without overlap, after the ordering)
    const int n_act = d.meta->nact[tick];
    const bool bad = d.meta->err != 0;
    int64_t idx = gtid() / G;
    M m;
    if (idx < n_act) group_fetch<R, DIM>(d, idx, g, m);
    __syncthreads();
    pdl_enter();
    if (bad) return;
    for (bool first = true; idx < n_act; idx += gsz, first = false) {
        if (!first) group_fetch<R, DIM>(d, idx, g, m);
        const int e = m.e;
        const uint32_t inf = m.inf;
        const int b = m.lv & 7, par = (m.lv >> 3) & 1;
        const int ke = tick >> (B - b);
        const int cur = par ^ (ke & 1);
        const int lev = (inf >> 24) & 15;
        // every value this step needs: own row, neighbours as seen, state, barrier-start terms
        R u[NP];
        constexpr int NPS = S::NPS;
        ld_dofs<R, NP, NPS>((cur ? d.V1 : d.V0) + (size_t)e * NPS, u);
        const R w = d.v[(size_t)e * NPS + g];
        R un[NF][NP];
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const int kind = (inf >> (4 * f)) & 3;
            load_seen_lv<R, NP>(d, tick, B, (kind == 1 || kind == 2) ? m.nbf[f] : e, m.lvn[f], un[f]);
        }
        R Ia = R(0), ga = R(0);
        double acc0 = 0.0;
        if (ke != 0) {
            Ia = d.Ia[(size_t)e * NPS + g];
            ga = d.ga[(size_t)e * NPS + g];
            if (g == 0) acc0 = d.acc[e];
        }
        // row g of the residual
        R rg = R(0);
#pragma unroll
        for (int j = 0; j < NP; ++j) rg += m.vrow[j] * u[j];
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const int kind = (inf >> (4 * f)) & 3;
            if (kind == 1 || kind == 2) {
                if constexpr (M::ROWS) {
#pragma unroll
                    for (int j = 0; j < NP; ++j) rg += m.orow[f][j] * u[j] + m.nrow[f][j] * un[f][j];
                } else {
                    const int rel = kind == 2 ? 1 + ((inf >> (4 * f + 2)) & 3) : 0;
                    const R* A = d.qface + ((((size_t)f * 8 + lev) * NREL + rel) * 2) * NP * NP;
                    R ro[NP], rn[NP];
                    ld_row<R, NP>(A + g * NP, ro);
                    ld_row<R, NP>(A + NP * NP + g * NP, rn);
#pragma unroll
                    for (int j = 0; j < NP; ++j) rg += ro[j] * u[j] + rn[j] * un[f][j];
                }
            }
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const int kind = (inf >> (4 * f)) & 3;
            if (kind != 3) continue;
            for (int sb = 0; sb < NSUB; ++sb) {
                R uh[NP], ro[NP], rn[NP];
                load_seen<R, NP>(d, tick, B, d.hang[m.nbf[f] + sb], uh);
                const R* A = d.qface + ((((size_t)f * 8 + lev) * NREL + 1 + NSUB + sb) * 2) * NP * NP;
                ld_row<R, NP>(A + g * NP, ro);
                ld_row<R, NP>(A + NP * NP + g * NP, rn);
#pragma unroll
                for (int j = 0; j < NP; ++j) rg += ro[j] * u[j] + rn[j] * uh[j];
            }
        }
        // pointwise step of DOF g
        const double dte_d = a.dte[b];
        R so = R(0), smd = R(0);
        if (inf & INFO_STIM) dof_stim<R>(a, e, tick, dte_d, g, so, smd);
        R my_u = u[0];
#pragma unroll
        for (int q = 1; q < NP; ++q)
            if (q == g) my_u = u[q];
        R un_g, wn_g;
        R term = dof_update_any<R>(ph, sMq[lev * NP + g], sMinv[lev * NP + g], ke, a.dteR[b], so, smd, my_u, w, rg, Ia,
                               ga, un_g, wn_g);
        R vmax = un_g < R(0) ? -un_g : un_g;
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) {
            term += __shfl_xor_sync(gmask, term, o, G);
            const R om = __shfl_xor_sync(gmask, vmax, o, G);
            vmax = om > vmax ? om : vmax;
        }
        ((cur ? d.V0 : d.V1) + (size_t)e * NPS)[g] = un_g;
        d.v[(size_t)e * NPS + g] = wn_g;
        if (ke == 0 && b > 0) {
            d.Ia[(size_t)e * NPS + g] = Ia;
            d.ga[(size_t)e * NPS + g] = ga;
        }
        if (g == 0) d.acc[e] = acc0 + dte_d * (double)term;
        if ((inf & INFO_PENDING) && vmax >= ph.lat_gate) {
            R unv[NP];
#pragma unroll
            for (int q = 0; q < NP; ++q) unv[q] = __shfl_sync(gmask, un_g, q, G);
            if (g == 0) lat_check<R, DIM, 1>(d, T, ph, e, inf, lev, u, unv, tick_time(a, tick), dte_d);
        }
    }
}

// Grid-wide barrier number `round` (1, 2, ...) of a cooperative launch (every block resident):
// each block's thread 0 counts its arrival in m->gbar (zeroed before the launch) and waits,
// with at most `limit` polls 64 ns apart (~1 s by default), until every block of the round has
// arrived.  A wait that gives up sets ERR_WAIT (the host reports it) and lets the block go on:
// no hang.
constexpr uint32_t GRID_WAIT_LIMIT = 1u << 24;
__device__ __forceinline__ void grid_barrier(DevMeta* m, unsigned round, uint32_t limit = GRID_WAIT_LIMIT) {
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned target = round * gridDim.x;
        __threadfence();
        atomicAdd(&m->gbar, 1u);
        uint32_t it = 0;
        while (*(volatile unsigned*)&m->gbar < target) {
            if (++it > limit) {
                atomicOr(&m->err, ERR_WAIT);
                break;
            }
            __nanosleep(64);
        }
        __threadfence();
    }
    __syncthreads();
}

// The whole sweep of a barrier in one cooperative launch: every tick of Alg. 1 with a
// grid-wide barrier between ticks (the Jacobi reading needs all of tick i before tick
// i+1), then the epilogue with a fixed-order final reduction by block 0.  The grid is
// sized from the occupancy API so that every block is resident.
template <typename R, int DIM, int P>
__global__ void __launch_bounds__(256) k_sweep(const TickArgs<R> a, const Tables<R> T, const Phys<R> ph,
                                              const OpT<R, DIM, P> op, const double* __restrict__ mtab) {
    using S = Shape<DIM, P>;
    constexpr int NP = S::NP;
    const DevArrays<R>& d = a.d;
    if (d.meta->err) return;             // uniform: nothing below changes err before the end
    const int nt = 1 << a.B;
    for (int i = 0; i < nt; ++i) {
        tick_work<R, DIM, P>(a, T, ph, op, i);
        grid_barrier(d.meta, (unsigned)(i + 1));
    }
    __shared__ double red[256];
    const int64_t ne = d.meta->ne;
    double loc = 0.0;
    bool bad = false;
    for (int64_t e = gtid(); e < ne; e += gstride()) {
        d.eta_t[e] = sqrt(d.acc[e]) / a.dt;
        uint8_t lv = d.lvl[e];
        if ((lv & 7) == 0) {
            lv ^= 8;
            d.lvl[e] = lv;
        }
        const int par = (lv >> 3) & 1;
        const R* Vc = (par ? d.V1 : d.V0) + (size_t)e * S::NPS;
        const R* w = d.v + (size_t)e * S::NPS;
        const int lev = (d.info[e] >> 24) & 15;
        const double* Mq = mtab + lev * NP;
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            const R x = Vc[q];
            loc += Mq[q] * (double)x;
            bad = bad || !isfinite(x) || !isfinite(w[q]);
        }
    }
    if (bad) atomicOr(&d.meta->nf_pending, 1u);
    red[threadIdx.x] = loc;
    __syncthreads();
    for (int s2 = blockDim.x / 2; s2 > 0; s2 >>= 1) {
        if (threadIdx.x < s2) red[threadIdx.x] += red[threadIdx.x + s2];
        __syncthreads();
    }
    if (threadIdx.x == 0) d.partial[blockIdx.x] = red[0];
    grid_barrier(d.meta, (unsigned)(nt + 1));
    if (blockIdx.x != 0) return;
    double s3 = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) s3 += d.partial[i];
    red[threadIdx.x] = s3;
    __syncthreads();
    for (int s2 = blockDim.x / 2; s2 > 0; s2 >>= 1) {
        if (threadIdx.x < s2) red[threadIdx.x] += red[threadIdx.x + s2];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        DevMeta* m = d.meta;
        m->integral = red[0];
        m->nbar += 1;
        if (m->nf_pending) {
            m->err |= ERR_NONFINITE;
            m->nf_pending = 0;
        }
    }
}

// Copy V (current slot by parity) or v to a compact output (NP values per element).
template <typename R, int NP, int NPS, typename Out>
__global__ void k_gather(const DevArrays<R> d, int64_t ne, int which, Out* out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= ne * NP) return;
    const int64_t e = i / NP, j = e * NPS + (i - e * NP);
    if (which == 0) {
        const int par = (d.lvl[e] >> 3) & 1;
        out[i] = (Out)((par ? d.V1 : d.V0)[j]);
    } else {
        out[i] = (Out)d.v[j];
    }
}

// V (current slot) and the state variable into one compact FP32 buffer [V | v].
template <typename R, int NP, int NPS>
__global__ void k_gather_f32(const DevArrays<R> d, int64_t ne, float* outV, float* outS) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= ne * NP) return;
    const int64_t e = i / NP, j = e * NPS + (i - e * NP);
    const int par = (d.lvl[e] >> 3) & 1;
    if (outV) outV[i] = (float)((par ? d.V1 : d.V0)[j]);
    if (outS) outS[i] = (float)d.v[j];
}

// The same for page-locked host buffers read or written over the host link: four consecutive
// compact values per thread as one 16-byte access (buffers 16-byte aligned; the last partial
// group value by value), which keeps more bytes in flight per request than 4-byte accesses.
template <typename R, int NP, int NPS>
__global__ void k_gather_f32x4(const DevArrays<R> d, int64_t ne, float* outV, float* outS) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, n = ne * NP, i0 = 4 * t;
    if (i0 >= n) return;
    float va[4] = {0.0f, 0.0f, 0.0f, 0.0f}, sa[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int64_t i = i0 + k;
        if (i < n) {
            const int64_t e = i / NP, j = e * NPS + (i - e * NP);
            const int par = (d.lvl[e] >> 3) & 1;
            va[k] = (float)((par ? d.V1 : d.V0)[j]);
            sa[k] = (float)d.v[j];
        }
    }
    if (i0 + 3 < n) {
        if (outV) reinterpret_cast<float4*>(outV)[t] = make_float4(va[0], va[1], va[2], va[3]);
        if (outS) reinterpret_cast<float4*>(outS)[t] = make_float4(sa[0], sa[1], sa[2], sa[3]);
    } else {
        for (int k = 0; i0 + k < n; ++k) {
            if (outV) outV[i0 + k] = va[k];
            if (outS) outS[i0 + k] = sa[k];
        }
    }
}

template <typename R, int NP, int NPS>
__global__ void k_scatter_initial_x4(DevArrays<R> d, int64_t ne, const float* V, const float* w) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, n = ne * NP, i0 = 4 * t;
    if (i0 < n) {
        float va[4] = {0.0f, 0.0f, 0.0f, 0.0f}, wa[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (i0 + 3 < n) {
            const float4 a = reinterpret_cast<const float4*>(V)[t];
            va[0] = a.x; va[1] = a.y; va[2] = a.z; va[3] = a.w;
            if (w) {
                const float4 b = reinterpret_cast<const float4*>(w)[t];
                wa[0] = b.x; wa[1] = b.y; wa[2] = b.z; wa[3] = b.w;
            }
        } else {
            for (int k = 0; i0 + k < n; ++k) {
                va[k] = V[i0 + k];
                if (w) wa[k] = w[i0 + k];
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int64_t i = i0 + k;
            if (i < n) {
                const int64_t e = i / NP, j = e * NPS + (i - e * NP);
                d.V0[j] = (R)va[k];
                if (w) d.v[j] = (R)wa[k];
            }
        }
    }
    // element t: the pad values of its padded rows, and its level byte's parity reset
    if (t < ne) {
#pragma unroll
        for (int q = NP; q < NPS; ++q) {
            d.V0[t * NPS + q] = R(0);
            if (w) d.v[t * NPS + q] = R(0);
        }
        d.lvl[t] &= 7;
    }
}

// Set V (into slot 0, parity reset) and optionally v from compact FP64 or FP32 input; the
// pad values of padded rows are set to 0.
template <typename R, int NP, int NPS, typename In>
__global__ void k_scatter_initial(DevArrays<R> d, int64_t ne, const In* V, const In* w) {
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j >= ne * NPS) return;
    const int64_t e = j / NPS, q = j - e * NPS, i = e * NP + q;
    const bool pad = q >= NP;
    d.V0[j] = pad ? R(0) : (R)V[i];
    if (w) d.v[j] = pad ? R(0) : (R)w[i];
    if (q == 0) d.lvl[e] &= 7;
}

// Activation at the current time for probes already above threshold, and the
// per-element pending flag (any probe of the element not yet activated).
template <typename R, int DIM, int P>
__global__ void k_lat_refresh(DevArrays<R> d, const Tables<R> T, const Phys<R> ph, double t, int mark_now,
                              int force) {
    pdl_enter();
    using S = Shape<DIM, P>;
    constexpr int N1 = S::N1, NP = S::NP;
    if (d.meta->err || !(force || d.meta->changed)) return;
    const int64_t ne = d.meta->ne;
    for (int64_t e = gtid(); e < ne; e += gstride()) {
    uint32_t inf = d.info[e];
    const int lev = (inf >> 24) & 15;
    const int par = (d.lvl[e] >> 3) & 1;
    const R* Vc = (par ? d.V1 : d.V0) + (size_t)e * S::NPS;
    R u[NP];
    ld_dofs<R, NP, S::NPS>(Vc, u);
    const uint32_t lc = d.loc[e];
    const int lx[3] = {(int)(lc & 255u), (int)((lc >> 8) & 255u), (int)((lc >> 16) & 255u)};
    const int64_t rid = d.root[e];
    bool pending = false;
    for (int q = 0; q < NP; ++q) {
        bool inside = true;
#pragma unroll
        for (int k = 0; k < DIM; ++k) inside = inside && (T.pfl[lev][digit<N1>(q, k)] == lx[k]);
        if (!inside) continue;
        double* lp = d.lat + rid * NP + q;
        if (!isinf(*lp)) continue;
        if (mark_now) {
            R pv = 0;
            for (int j = 0; j < NP; ++j) {
                R w = R(1);
#pragma unroll
                for (int k = 0; k < DIM; ++k) w *= T.pphi[lev][digit<N1>(q, k)][digit<N1>(j, k)];
                pv += w * u[j];
            }
            if (pv > ph.act) {
                *lp = t;
                continue;
            }
        }
        pending = true;
    }
    inf = pending ? (inf | INFO_PENDING) : (inf & ~INFO_PENDING);
    d.info[e] = inf;
    }
}

}  // namespace mdl

