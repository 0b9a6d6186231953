// mdl_mapped.cuh -- the element step on curved (mapped) meshes: thread per element.
//
// The geometric factors of every element (mdl_geometry.h) are stored per GL point, in groups of
// 32 elements with the element fastest (value i of element e at [e / 32][i][e % 32]): a warp takes
// consecutive elements, and a row of 704 bytes per element (Q1 3D) read value by value by its own
// thread is 32 cache lines an instruction.  At volume
// node q the symmetric metric G_q and the mass M_q, at face point t the flux vector c, the
// area weight dS and the penalty kappa.  The residual of element e (Eq. monodomain-primal-
// formulation with the flux of Eq. monodomain-numerical-flux, all faces conforming):
//   volume:  r_i += sum_q grad_xi psi_i(q) . G_q grad_xi u(q)
//   face f:  at each point t, with the own trace u_o, the neighbour's trace u_n (its opposite
//            face), flux = c . grad_xi u on each side and jump = u_o - u_n,
//            r_i += dS [ (-(flux_o + flux_n)/2 + kappa jump) psi_i(t) - jump/2 c . grad_xi psi_i(t) ]
// The pointwise update, RV-T term and probe check are those of the box elements with the
// element's own GL mass M_q.
#pragma once

#include "mdl_geofactors.cuh"
#include "mdl_kernels.cuh"

namespace mdl {

template <int DIM, int P>
struct MapShape {
    static constexpr int N1 = P + 1;
    static constexpr int NP = DIM == 2 ? N1 * N1 : N1 * N1 * N1;
    static constexpr int NF = 2 * DIM;
    static constexpr int NPF = DIM == 2 ? N1 : N1 * N1;
    static constexpr int NS = DIM * (DIM + 1) / 2;
    static constexpr int VPN = NS + 1;        // values per volume node: G, M
    static constexpr int FPV = DIM + 2;       // values per face point: c, dS, kappa
    static constexpr int NV = NP * VPN, NFV = NF * NPF * FPV;   // factor values per element
};

// Factors of element e, `per` values each, FS apart.
constexpr int FS = 32;
template <typename R>
__device__ __forceinline__ R* factors_of(R* base, int64_t e, int per) {
    return base + (size_t)(e >> 5) * per * FS + (e & 31);
}

// Entry (k, l) of the symmetric metric stored as (xx, yy, xy) or (xx, yy, zz, xy, xz, yz).
template <int DIM>
__device__ __forceinline__ int sym_index(int k, int l) {
    if (k == l) return k;
    if (DIM == 2) return 2;
    const int a = k < l ? k : l, b = k < l ? l : k;
    return a == 0 ? (b == 1 ? 3 : 4) : 5;
}

// Tangential axes of a normal-k face, increasing.
template <int DIM>
__device__ __forceinline__ void face_tangents(int k, int* tg) {
    int z = 0;
#pragma unroll
    for (int l = 0; l < DIM; ++l)
        if (l != k) tg[z++] = l;
}

// At the points t of face f = 2k + sd (sd = 1: the +k side), own and neighbour traces (to, tn)
// and the normal fluxes c . grad_xi u of both sides (flo, fln): the normal derivative from
// the 1D derivative values at the face, the tangential ones from the traces by the 1D
// derivative matrix.  The neighbour is seen through its opposite face.
template <typename R, int DIM, int P>
__device__ __forceinline__ void mapped_face_fluxes(const Tables<R>& T, const R* u, const R* un, int k, int sd,
                                                   const R* gf, R* to, R* tn, R* flo, R* fln) {
    using M = MapShape<DIM, P>;
    constexpr int N1 = M::N1, NPF = M::NPF, FPV = M::FPV;
    const R* bs = sd ? T.bR : T.bL;
    const R* ds = sd ? T.dR : T.dL;
    const R* bn = sd ? T.bL : T.bR;
    const R* dn = sd ? T.dL : T.dR;
    int tg[2] = {0, 0};
    face_tangents<DIM>(k, tg);
    R go[NPF], gn[NPF];
#pragma unroll
    for (int t = 0; t < NPF; ++t) {
        const int at0 = t % N1, at1 = t / N1;
        int q0 = at0 * stride<N1>(tg[0]);
        if (DIM == 3) q0 += at1 * stride<N1>(tg[1]);
        R a = 0, b = 0, c = 0, g2 = 0;
#pragma unroll
        for (int m = 0; m < N1; ++m) {
            const int q = q0 + m * stride<N1>(k);
            a += bs[m] * u[q];
            c += ds[m] * u[q];
            b += bn[m] * un[q];
            g2 += dn[m] * un[q];
        }
        to[t] = a;
        go[t] = c;
        tn[t] = b;
        gn[t] = g2;
    }
#pragma unroll
    for (int t = 0; t < NPF; ++t) {
        const int at[2] = {t % N1, t / N1};
        const R* c = gf + t * FPV * FS;
        R fo = c[k * FS] * go[t], fn = c[k * FS] * gn[t];
#pragma unroll
        for (int z = 0; z < DIM - 1; ++z) {
            const int st = z == 0 ? 1 : N1;            // face-point stride of tangent z
            R so = 0, sn = 0;
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                const int t2 = t + (a - at[z]) * st;
                so += T.D1[at[z]][a] * to[t2];
                sn += T.D1[at[z]][a] * tn[t2];
            }
            fo += c[tg[z] * FS] * so;
            fn += c[tg[z] * FS] * sn;
        }
        flo[t] = fo;
        fln[t] = fn;
    }
}

// Trace and normal derivative of v at the nodes of its face (axis k, side sd).
template <typename R, int DIM, int P>
__device__ __forceinline__ void mapped_trace(const Tables<R>& T, int k, int sd, const R* v, R* tr, R* dn) {
    using M = MapShape<DIM, P>;
    const R* bs = sd ? T.bR : T.bL;
    const R* ds = sd ? T.dR : T.dL;
#pragma unroll
    for (int m = 0; m < M::NPF; ++m) {
        R a = 0, b = 0;
#pragma unroll
        for (int j = 0; j < M::N1; ++j) {
            const R x = v[line_node<DIM, P>(k, m, j)];
            a += bs[j] * x;
            b += ds[j] * x;
        }
        tr[m] = a;
        dn[m] = b;
    }
}

// The coarse side of a hanging face at the finer side's GL points (half `bits` per tangent of its
// own face), from its face's traces tr0 and normal derivatives dn0: the trace and cscale c . grad_xi,
// c the flux vector stored at each point (FS apart).  One-dimensional interpolation, and derivatives
// along the face from the interpolated trace (its own coordinate runs twice as fast): an eighth of
// the operations of the sums over the element's nodes at every point, which the FP64 pipe bounds.
template <typename R, int DIM, int P>
__device__ __forceinline__ void half_face_eval(const Tables<R>& T, const R* tr0, const R* dn0, int k, const int* tg,
                                               int bits, const R* gf, R cscale, R* tr, R* fl) {
    using M = MapShape<DIM, P>;
    constexpr int NPF = M::NPF, FPV = M::FPV;
    R dn[NPF];
    face_map<R, DIM, P>(T.Pi, bits & 1, (bits >> 1) & 1, tr0, tr);
    face_map<R, DIM, P>(T.Pi, bits & 1, (bits >> 1) & 1, dn0, dn);
#pragma unroll
    for (int t = 0; t < NPF; ++t) fl[t] = gf[(t * FPV + k) * FS] * dn[t];
#pragma unroll
    for (int z = 0; z < DIM - 1; ++z) {
        R g[NPF];
        face_line<R, DIM, P>(T.D1, z, R(2), tr, g, false);
#pragma unroll
        for (int t = 0; t < NPF; ++t) fl[t] += gf[(t * FPV + tg[z]) * FS] * g[t];
    }
#pragma unroll
    for (int t = 0; t < NPF; ++t) fl[t] *= cscale;
}

// The adjoint: test values A and cscale Bc c . grad_xi at the points, added to the coefficients
// trc, dnc of the coarse side's face traces and normal derivatives.
template <typename R, int DIM, int P>
__device__ __forceinline__ void half_face_adjoint(const Tables<R>& T, int k, const int* tg, int bits, const R* gf,
                                                  R cscale, const R* A, const R* Bc, R* trc, R* dnc) {
    using M = MapShape<DIM, P>;
    constexpr int NPF = M::NPF, FPV = M::FPV;
    R a[NPF], n[NPF];
#pragma unroll
    for (int t = 0; t < NPF; ++t) {
        a[t] = A[t];
        n[t] = cscale * Bc[t] * gf[(t * FPV + k) * FS];
    }
#pragma unroll
    for (int z = 0; z < DIM - 1; ++z) {
        R g[NPF];
#pragma unroll
        for (int t = 0; t < NPF; ++t) g[t] = cscale * Bc[t] * gf[(t * FPV + tg[z]) * FS];
        face_line_t<R, DIM, P>(T.D1, z, R(2), g, a, true);
    }
    face_map_t_add<R, DIM, P>(T.Pi, bits & 1, (bits >> 1) & 1, a, trc);
    face_map_t_add<R, DIM, P>(T.Pi, bits & 1, (bits >> 1) & 1, n, dnc);
}

// The faces of element e with finer neighbours (kind 3 on face f): each subface sb is the
// opposite face of neighbour j = hang[sb], integrated at j's GL points with j's stored factors
// (flux vector c_j along j's outward normal, area weight, penalty).  This element's flux vector
// there is -c_j / 2 (the opposite normal, twice the extent); its trace and gradient come from
// its own values on the half of its face the subface covers.
template <typename R, int DIM, int P>
__device__ __forceinline__ void mapped_hanging_coarse(const DevArrays<R>& d, const Tables<R>& T, int tick, int B,
                                                      int e, int k, int sd, const R* u, R* r) {
    using M = MapShape<DIM, P>;
    constexpr int NP = M::NP, NF = M::NF, NPF = M::NPF, FPV = M::FPV, NSUB = 1 << (DIM - 1);
    constexpr int NPS = Shape<DIM, P>::NPS;
    const int f = 2 * k + sd;
    int tg[2] = {0, 0};
    face_tangents<DIM>(k, tg);
    const int base = d.nbr[(size_t)e * NF + f];
    R tr0[NPF], dn0[NPF], trc[NPF], dnc[NPF];
    mapped_trace<R, DIM, P>(T, k, sd, u, tr0, dn0);
#pragma unroll
    for (int t = 0; t < NPF; ++t) trc[t] = dnc[t] = R(0);
#pragma unroll 1
    for (int sb = 0; sb < NSUB; ++sb) {
        const int j = d.hang[base + sb];
        R uj[NP];
        load_seen<R, NP, NPS>(d, tick, B, j, uj);
        const R* gfj = factors_of(d.gface, j, M::NFV) + (f ^ 1) * NPF * FPV * FS;
        R tj[NPF], tx[NPF], fj[NPF], fx[NPF], tro[NPF], flo[NPF], A[NPF], Bc[NPF];
        mapped_face_fluxes<R, DIM, P>(T, uj, uj, k, sd ^ 1, gfj, tj, tx, fj, fx);
        half_face_eval<R, DIM, P>(T, tr0, dn0, k, tg, sb, gfj, R(-0.5), tro, flo);
#pragma unroll
        for (int t = 0; t < NPF; ++t) {
            const R* c = gfj + t * FPV * FS;
            const R fln = -fj[t];
            const R dS = c[DIM * FS], kap = c[(DIM + 1) * FS];
            const R jump = tro[t] - tj[t];
            A[t] = dS * (R(-0.5) * (flo[t] + fln) + kap * jump);
            Bc[t] = R(-0.5) * dS * jump;
        }
        half_face_adjoint<R, DIM, P>(T, k, tg, sb, gfj, R(-0.5), A, Bc, trc, dnc);
    }
    const R* bs = sd ? T.bR : T.bL;
    const R* ds = sd ? T.dR : T.dL;
#pragma unroll
    for (int m = 0; m < NPF; ++m)
#pragma unroll
        for (int j = 0; j < M::N1; ++j) r[line_node<DIM, P>(k, m, j)] += bs[j] * trc[m] + ds[j] * dnc[m];
}

template <typename R, int DIM, int P>
__device__ __forceinline__ void mapped_residual(const DevArrays<R>& d, const Tables<R>& T, int tick, int B,
                                                const TickMeta<DIM, P>& mt, const R* u, R* r) {
    using M = MapShape<DIM, P>;
    constexpr int N1 = M::N1, NP = M::NP, NF = M::NF, NPF = M::NPF, VPN = M::VPN, FPV = M::FPV;
    constexpr int NPS = Shape<DIM, P>::NPS;
    const int e = mt.e;
    const uint32_t inf = mt.inf;
    // the neighbours' rows: FP32 Q1 all at once (48 registers), else face by face
    constexpr bool ALL = sizeof(R) == 4 && P == 1;
    R un_[ALL ? NF : 1][NP];
    if constexpr (ALL) {
        const R* ol[NF];
        R th[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const int kind = (inf >> (4 * f)) & 3;
            const bool use = kind == 1 || kind == 2;
            ld_dofs<R, NP, NPS>(
                seen_row<R, NPS>(d, tick, B, use ? mt.nbf[f] : e, use ? mt.lvn[f] : mt.lv, ol[f], th[f]), un_[f]);
        }
#pragma unroll
        for (int f = 0; f < NF; ++f)
            if (th[f] > R(0)) interp_row<R, NP, NPS>(ol[f], th[f], un_[f]);
    }
#pragma unroll
    for (int q = 0; q < NP; ++q) r[q] = R(0);
    // volume: flux G_q grad u at every node, then r_i = sum_k sum_m D1[m][a_k(i)] flux_k(node m of i's line)
    {
        const R* gv = factors_of(d.gvol, e, M::NV);
        R fl[NP][DIM];
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            R g[DIM];
#pragma unroll
            for (int k = 0; k < DIM; ++k) {
                const int ak = digit<N1>(q, k);
                R s = R(0);
#pragma unroll
                for (int m = 0; m < N1; ++m) s += T.D1[ak][m] * u[q + (m - ak) * stride<N1>(k)];
                g[k] = s;
            }
#pragma unroll
            for (int k = 0; k < DIM; ++k) {
                R s = R(0);
#pragma unroll
                for (int l = 0; l < DIM; ++l) s += gv[(q * VPN + sym_index<DIM>(k, l)) * FS] * g[l];
                fl[q][k] = s;
            }
        }
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            R s = R(0);
#pragma unroll
            for (int k = 0; k < DIM; ++k) {
                const int ak = digit<N1>(i, k);
#pragma unroll
                for (int m = 0; m < N1; ++m) s += T.D1[m][ak] * fl[i + (m - ak) * stride<N1>(k)][k];
            }
            r[i] = s;
        }
    }
    // faces: the side a loop where the rows are not all in registers, the subfaces always (unrolled
    // over 6 faces, 4 subfaces and 4 points the FP64 Q1 step was 700 KB of code, fetched from L2)
    auto face = [&](int k, int sd, R* un) {
        const int f = 2 * k + sd, kind = (inf >> (4 * f)) & 3;
        if (kind == 0 || kind == 3) return;
        if constexpr (!ALL) {
            const int n = sd ? mt.nbf[2 * k + 1] : mt.nbf[2 * k];
            const R* ol;
            R th;
            ld_dofs<R, NP, NPS>(seen_row<R, NPS>(d, tick, B, n, sd ? mt.lvn[2 * k + 1] : mt.lvn[2 * k], ol, th), un);
            if (th > R(0)) interp_row<R, NP, NPS>(ol, th, un);
        }
        const R* bs = sd ? T.bR : T.bL;
        const R* ds = sd ? T.dR : T.dL;
        int tg[2] = {0, 0};
        face_tangents<DIM>(k, tg);
        R to[NPF], tn[NPF], flo[NPF], fln[NPF];
        const R* gf = factors_of(d.gface, e, M::NFV) + f * NPF * FPV * FS;
        mapped_face_fluxes<R, DIM, P>(T, u, un, k, sd, gf, to, tn, flo, fln);
        if (kind == 2) {
            // a coarser neighbour: its trace and flux at this element's points, on the half of
            // its face given by the position bits; its flux vector is half this element's
            R trn[NPF], dnn[NPF];
            mapped_trace<R, DIM, P>(T, k, sd ^ 1, un, trn, dnn);
            half_face_eval<R, DIM, P>(T, trn, dnn, k, tg, (inf >> (4 * f + 2)) & 3, gf, R(0.5), tn, fln);
        }
#pragma unroll
        for (int t = 0; t < NPF; ++t) {
            const int at[2] = {t % N1, t / N1};
            const R* c = gf + t * FPV * FS;
            const R dS = c[DIM * FS], kap = c[(DIM + 1) * FS];
            const R jump = to[t] - tn[t];
            const R A = dS * (R(-0.5) * (flo[t] + fln[t]) + kap * jump);
            const R Bc = R(-0.5) * dS * jump;
            int q0 = at[0] * stride<N1>(tg[0]);
            if (DIM == 3) q0 += at[1] * stride<N1>(tg[1]);
#pragma unroll
            for (int m = 0; m < N1; ++m) {
                const int i = q0 + m * stride<N1>(k);
                r[i] += A * bs[m] + Bc * c[k * FS] * ds[m];
#pragma unroll
                for (int z = 0; z < DIM - 1; ++z) {
                    const R w = Bc * c[tg[z] * FS] * bs[m];
#pragma unroll
                    for (int a = 0; a < N1; ++a) r[i + (a - at[z]) * stride<N1>(tg[z])] += w * T.D1[at[z]][a];
                }
            }
        }
    };
    if constexpr (ALL) {
#pragma unroll
        for (int f = 0; f < NF; ++f) face(f >> 1, f & 1, un_[f]);
    } else {
#pragma unroll
        for (int k = 0; k < DIM; ++k)
#pragma unroll 1
            for (int sd = 0; sd < 2; ++sd) face(k, sd, un_[0]);
    }
#pragma unroll
    for (int k = 0; k < DIM; ++k)
#pragma unroll 1
        for (int sd = 0; sd < 2; ++sd)
            if (((inf >> (8 * k + 4 * sd)) & 3) == 3) mapped_hanging_coarse<R, DIM, P>(d, T, tick, B, e, k, sd, u, r);
}

// One element step of Alg. 1 on a mapped mesh (see tick_elem for the box elements).
template <typename R, int DIM, int P>
__device__ __forceinline__ void tick_elem_mapped(const TickArgs<R>& a, const Tables<R>& T, const Phys<R>& ph,
                                                 int tick, const TickMeta<DIM, P>& mt) {
    using M = MapShape<DIM, P>;
    constexpr int NP = M::NP, VPN = M::VPN;
    constexpr int NPS = Shape<DIM, P>::NPS;
    const DevArrays<R>& d = a.d;
    const int e = mt.e;
    const uint32_t inf = mt.inf;
    const int b = mt.lv & 7, par = (mt.lv >> 3) & 1;
    const int ke = tick >> (a.B - b);
    const int cur = par ^ (ke & 1);
    const R* Vc = (cur ? d.V1 : d.V0) + (size_t)e * NPS;
    R* Vd = (cur ? d.V0 : d.V1) + (size_t)e * NPS;
    R* vp = d.v + (size_t)e * NPS;
    R u[NP], w[NP], r[NP], Ia[NP], ga[NP];
    ld_dofs<R, NP, NPS>(Vc, u);
    ld_dofs<R, NP, NPS>(vp, w);
    mapped_residual<R, DIM, P>(d, T, tick, a.B, mt, u, r);
    double acc0 = 0.0;
    if (ke != 0) {
        ld_dofs<R, NP, NPS>(d.Ia + (size_t)e * NPS, Ia);
        ld_dofs<R, NP, NPS>(d.ga + (size_t)e * NPS, ga);
        acc0 = d.acc[e];
    }
    bool stim = false;
    for (int s = 0; s < a.stim.n; ++s) stim = stim || d.smask[s][e] != 0u;
    const double dte_d = a.dte[b];
    const R dte = a.dteR[b];
    StimMasks stm;
    elem_stim<R>(a, e, stim ? INFO_STIM : 0u, tick, dte_d, stm);   // (info's bit is the box elements')
    const R* gv = factors_of(d.gvol, e, M::NV);
    R un[NP], wn[NP], Mq[NP], so[NP], sm[NP];
    R term = R(0), vmax = R(0);
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        Mq[q] = gv[(q * VPN + VPN - 1) * FS];
        node_stim<R>(a, stm, q, so[q], sm[q]);
    }
    bool ap = false;
    if constexpr (sizeof(R) == 4) {
        ap = ph.ionic == 0 && ph.integrator == 1;
        if (ap) {
#pragma unroll
            for (int q = 0; q < NP; ++q) r[q] *= R(1) / Mq[q];
            term = ap_step<NP>(ApConst(ph), ke == 0, Mq, R(1), dte, so, sm, u, w, r, Ia, ga, un, wn);
        }
    }
    if (!ap) {
#pragma unroll
        for (int q = 0; q < NP; ++q)
            term += dof_update_any<R>(ph, Mq[q], R(1) / Mq[q], ke, dte, so[q], sm[q], u[q], w[q], r[q], Ia[q], ga[q], un[q],
                                  wn[q]);
    }
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        const R av = un[q] < R(0) ? -un[q] : un[q];
        vmax = av > vmax ? av : vmax;
    }
    if (ke == 0 && b > 0) {
        st_dofs<R, NP, NPS>(d.Ia + (size_t)e * NPS, Ia);
        st_dofs<R, NP, NPS>(d.ga + (size_t)e * NPS, ga);
    }
    st_dofs<R, NP, NPS>(Vd, un);
    st_dofs<R, NP, NPS>(vp, wn);
    d.acc[e] = acc0 + dte_d * (double)term;
    if ((inf & INFO_PENDING) && vmax >= ph.lat_gate) {
        const int lev = (inf >> 24) & 15;
        lat_check<R, DIM, P>(d, T, ph, e, inf, lev, u, un, tick_time(a, tick), dte_d);
    }
}

// Kelly-type spatial indicator (Eq. dg-error-estimate) on the mapped mesh, on the barrier-start
// values: per interior face, with the flux jump J_t = (c . grad_xi u)_own - (c . grad_xi u)_nb,
// the face area |F| = sum_t dS_t, h_F = |F|^(1/(d-1)) and the face map's Jacobian at the point
// W_F(t) = dS_t / (reference GL weight of t): h_F / (2p) sum_t dS_t (W_F(t) J_t)^2.  Face-point
// sums in the working precision, faces accumulated in FP64.
template <typename R, int DIM, int P>
__global__ void __launch_bounds__(128) k_eta_s_mapped(const DevArrays<R> d, const Tables<R> T,
                                                       const MarkArgs mark) {
    pdl_enter();
    using M = MapShape<DIM, P>;
    constexpr int N1 = M::N1, NP = M::NP, NF = M::NF, NPF = M::NPF, FPV = M::FPV;
    constexpr int NPS = Shape<DIM, P>::NPS;
    if (d.meta->err) return;
    if (gtid() == 0) d.meta->changed = 0u;
    const int64_t ne = d.meta->ne;
    for (int64_t e = gtid(); e < ne; e += gstride()) {
        const uint32_t inf = d.info[e];
        const int par = (d.lvl[e] >> 3) & 1;
        R u[NP];
        ld_dofs<R, NP, NPS>((par ? d.V1 : d.V0) + (size_t)e * NPS, u);
        double acc = 0.0;
        // one (sub)face: h_F / (2p) sum_t dS_t (W_F(t) J_t)^2 from its points' area weights and jumps
        auto face_sum = [&](const R* dS, const R* jmp) {
            R area = R(0), sum = R(0);
#pragma unroll
            for (int t = 0; t < NPF; ++t) {
                const R wref = T.w[t % N1] * (DIM == 3 ? T.w[t / N1] : R(1));
                const R x = dS[t] / wref * jmp[t];
                area += dS[t];
                sum += dS[t] * x * x;
            }
            const double hF = DIM == 3 ? sqrt((double)area) : (double)area;
            acc += hF / (2.0 * P) * (double)sum;
        };
#pragma unroll
        for (int k = 0; k < DIM; ++k)
#pragma unroll 1
        for (int sd = 0; sd < 2; ++sd) {
            const int f = 2 * k + sd, kind = (inf >> (4 * f)) & 3;
            if (kind == 0) continue;
            int tg[2] = {0, 0};
            face_tangents<DIM>(k, tg);
            const int nb = d.nbr[(size_t)e * NF + f];
            if (kind == 3) {
                // the finer neighbours' subfaces, at their points with their factors
                R tr0[NPF], dn0[NPF];
                mapped_trace<R, DIM, P>(T, k, sd, u, tr0, dn0);
#pragma unroll 1
                for (int sb = 0; sb < (1 << (DIM - 1)); ++sb) {
                    const int j = d.hang[nb + sb];
                    R uj[NP];
                    ld_dofs<R, NP, NPS>((((d.lvl[j] >> 3) & 1) ? d.V1 : d.V0) + (size_t)j * NPS, uj);
                    const R* gfj = factors_of(d.gface, j, M::NFV) + (f ^ 1) * NPF * FPV * FS;
                    R tj[NPF], tx[NPF], fj[NPF], fx[NPF], tro[NPF], flo[NPF], dS[NPF], jmp[NPF];
                    mapped_face_fluxes<R, DIM, P>(T, uj, uj, k, sd ^ 1, gfj, tj, tx, fj, fx);
                    half_face_eval<R, DIM, P>(T, tr0, dn0, k, tg, sb, gfj, R(-0.5), tro, flo);
#pragma unroll
                    for (int t = 0; t < NPF; ++t) {
                        jmp[t] = flo[t] + fj[t];
                        dS[t] = gfj[(t * FPV + DIM) * FS];
                    }
                    face_sum(dS, jmp);
                }
                continue;
            }
            R un[NP];
            ld_dofs<R, NP, NPS>((((d.lvl[nb] >> 3) & 1) ? d.V1 : d.V0) + (size_t)nb * NPS, un);
            const R* gf = factors_of(d.gface, e, M::NFV) + f * NPF * FPV * FS;
            R to[NPF], tn[NPF], flo[NPF], fln[NPF], dS[NPF], jmp[NPF];
            mapped_face_fluxes<R, DIM, P>(T, u, un, k, sd, gf, to, tn, flo, fln);
            if (kind == 2) {
                R trn[NPF], dnn[NPF];
                mapped_trace<R, DIM, P>(T, k, sd ^ 1, un, trn, dnn);
                half_face_eval<R, DIM, P>(T, trn, dnn, k, tg, (inf >> (4 * f + 2)) & 3, gf, R(0.5), tn, fln);
            }
#pragma unroll
            for (int t = 0; t < NPF; ++t) {
                jmp[t] = flo[t] - fln[t];
                dS[t] = gf[(t * FPV + DIM) * FS];
            }
            face_sum(dS, jmp);
        }
        const double eta = sqrt(acc);
        d.eta_s[e] = eta;
        if (mark.r) mark_leaf<DIM>(mark, d.info, d.nbr, e, inf, eta);
    }
}

// Inputs of the device factor pass: the map and diffusion, FP64 tables, GL nodes, level-0
// extents, stimulus boxes (slack applied), the barrier step and the LTS budget.
struct MapArgs {
    GeoArgs g;
    double xg[3];
    double h0[3];
    int nstim;
    double slo[MDL_MAX_STIM][3], shi[MDL_MAX_STIM][3];
    double dt;
    int B, lts;
};

// Smallest b >= 0 with dt 2^-b <= bound (15 if none below 60; Eq. num-substeps, exact).
__device__ __forceinline__ int b_from_bound_dev(double dt, double bound) {
    for (int b = 0; b <= 60; ++b)
        if (ldexp(dt, -b) <= bound) return b > 15 ? 15 : b;
    return 15;
}

// Factors of the current mesh after an adaptation, part 1.  An element kept by the adaptation
// (pkind 0) with the face kinds it had takes its old factors, GL masses, signature (face kinds
// in bits 0-11, level in bits 12-15, b^CFL in bits 16-19) and stimulus masks (source psrc in the
// old set); a warp walks 32 consecutive elements.  Every other element is appended to `todo` (count m->nfac, zeroed by
// the scan that commits the new mesh) for k_mapped_factors.  Without an old set (o* null)
// every element is appended.
template <typename R, int DIM, int P>
__global__ void __launch_bounds__(256) k_mapped_keep(
        const uint32_t* info, const int nstim, R* gvol, R* gface, double* mass, uint32_t* fsig, uint32_t* f0,
        uint32_t* f1, uint32_t* f2, uint32_t* f3, uint8_t* bcfl, uint32_t* sm0, uint32_t* sm1, uint32_t* sm2,
        uint32_t* sm3, const R* ogvol, const R* ogface, const double* omass, const uint32_t* ofsig,
        const uint32_t* of0, const uint32_t* of1, const uint32_t* of2, const uint32_t* of3, const int8_t* pkind,
        const int32_t* psrc, int32_t* todo, DevMeta* m) {
    pdl_enter();
    using M = MapShape<DIM, P>;
    constexpr int NP = M::NP, NF = M::NF;
    constexpr int NV = NP * M::VPN, NFV = NF * M::NPF * M::FPV;
    if (m->err) return;
    uint32_t* smask[4] = {sm0, sm1, sm2, sm3};
    uint32_t* fsm[4] = {f0, f1, f2, f3};
    const uint32_t* ofsm[4] = {of0, of1, of2, of3};
    const int64_t ne = m->ne;
    const int lane = threadIdx.x & 31;
    const int64_t nwarp = gstride() >> 5;
    for (int64_t base = (gtid() >> 5) * 32; base < ne; base += nwarp * 32) {
        const int64_t e = base + lane;
        bool keep = false;
        int64_t o = 0;
        if (e < ne && ofsig) {
            const uint32_t inf = info[e];
            uint32_t kbits = 0;
            for (int f = 0; f < NF; ++f) kbits |= ((inf >> (4 * f)) & 3u) << (2 * f);
            if (pkind[e] == 0) {
                o = psrc[e];
                const uint32_t sg = ofsig[o];
                keep = (sg & 0xfffu) == kbits;
                if (keep) {
                    fsig[e] = sg;
                    bcfl[e] = (uint8_t)((sg >> 16) & 15u);
                    for (int s = 0; s < nstim; ++s) smask[s][e] = fsm[s][e] = ofsm[s][o];
                }
            }
        }
        const unsigned need = __ballot_sync(0xffffffffu, e < ne && !keep);
        if (need) {
            int slot = 0;
            if (lane == 0) slot = (int)atomicAdd(&m->nfac, (unsigned)__popc(need));
            slot = __shfl_sync(0xffffffffu, slot, 0);
            if ((need >> lane) & 1u) todo[slot + __popc(need & ((1u << lane) - 1u))] = (int32_t)e;
        }
        if (keep) {
            // lanes over the elements: the new places are consecutive, the old ones nearly so
            const R* gvo = factors_of(ogvol, o, NV);
            const R* gfo = factors_of(ogface, o, NFV);
            R* gv = factors_of(gvol, e, NV);
            R* gf = factors_of(gface, e, NFV);
#pragma unroll 8
            for (int i = 0; i < NV; ++i) gv[i * FS] = gvo[i * FS];
#pragma unroll 8
            for (int i = 0; i < NFV; ++i) gf[i * FS] = gfo[i * FS];
#pragma unroll
            for (int i = 0; i < NP; ++i) mass[(size_t)e * NP + i] = omass[(size_t)o * NP + i];
        }
    }
}

// One element's factors computed by a whole warp: the arithmetic of geo_element, with the lanes
// over the element's GL points (map, metric, face factors; chunks of 32 points) and over the
// entries of its own block B (registers; every entry summed over the points in geo_element's
// order).  FP64 issues at a small fraction of the FP32 rate on this GPU, so one element's
// instructions are spread over 32 lanes rather than run by one.
template <int DIM, int P>
struct GeoWarp {
    static constexpr int N1 = P + 1;
    static constexpr int NP = DIM == 2 ? N1 * N1 : N1 * N1 * N1;
    static constexpr int NF = 2 * DIM, NPF = DIM == 2 ? N1 : N1 * N1, NSUB = 1 << (DIM - 1);
    static constexpr int NS = DIM * (DIM + 1) / 2, VPN = NS + 1, FPV = DIM + 2;
    static constexpr int CH = 32;                   // points per chunk (one per lane)
    static constexpr int PS = 2 * NP + 2;           // doubles per point: psi, c.grad psi, dS, kappa (face);
                                                    // the metric K (volume node)
    static constexpr int NE = (NP * NP + 31) / 32;  // block entries per lane
    static_assert(PS >= DIM * DIM && CH * PS >= NP * NP, "point record too small");
};

// Returns the Gershgorin bound (every lane); writes the element's volume factors and GL masses
// (gvol, gface: the element's factors, FS apart; mass: its row) and returns its stimulus masks in sk (every lane).
// spt: CH * PS doubles and sm: NP doubles of shared memory owned by the warp.
template <typename R, int DIM, int P>
__device__ double geo_element_warp(const GeoArgs& g, const Tables<double>& T, const double* xg, const double* h0,
                                   int lev, const int* cc, const int* kinds, int nstim, const double (*slo)[3],
                                   const double (*shi)[3], double* spt, double* sm, R* gvol, R* gface, double* mass,
                                   uint32_t* sk) {
    using W = GeoWarp<DIM, P>;
    constexpr int N1 = W::N1, NP = W::NP, NF = W::NF, NPF = W::NPF, NS = W::NS, VPN = W::VPN, FPV = W::FPV;
    constexpr int CH = W::CH, PS = W::PS, NE = W::NE;
    const int lane = threadIdx.x & 31;
    double h[3] = {1.0, 1.0, 1.0}, Xc[3] = {0.0, 0.0, 0.0}, s2h[3] = {2.0, 2.0, 2.0};
    const double sc = 1.0 / (double)(1 << lev);
    for (int k = 0; k < DIM; ++k) {
        h[k] = h0[k] * sc;
        Xc[k] = cc[k] * h[k];
        s2h[k] = 2.0 / h[k];
    }
    // points: the NP volume nodes, then per face with a neighbour its GL points (kind 3: the
    // finer neighbours' points, subface outer)
    int off[NF + 1];
    off[0] = NP;
    for (int f = 0; f < NF; ++f) off[f + 1] = off[f] + (kinds[f] ? NPF * (kinds[f] == 3 ? W::NSUB : 1) : 0);
    const int npt = off[NF];
    for (int f = 0; f < NF; ++f)
        if (kinds[f] == 0 || kinds[f] == 3)
            for (int i = lane; i < NPF * FPV; i += 32) gface[(f * NPF * FPV + i) * FS] = (R)0;
    uint32_t mk[MDL_MAX_STIM] = {0u, 0u, 0u, 0u};
    double bacc[NE];
#pragma unroll
    for (int u = 0; u < NE; ++u) bacc[u] = 0.0;
    for (int c0 = 0; c0 < npt; c0 += CH) {
        const int p = c0 + lane;
        double* rec = spt + lane * PS;
        if (p < NP) {
            const int q = p;
            double X[3] = {0.0, 0.0, 0.0}, x[3], J[3][3], Ji[3][3], D[3][3];
            double Wq = 1.0;
            for (int k = 0; k < DIM; ++k) {
                const int a = digit<N1>(q, k);
                X[k] = Xc[k] + (xg[a] + 1.0) * 0.5 * h[k];
                Wq *= T.w[a] * h[k] * 0.5;
            }
            geo_eval(g, X, x, J);
            const double det = geo_inverse(DIM, J, Ji);
            geo_tensor(g, J, D);
            double K[3][3];
            for (int i = 0; i < DIM; ++i)
                for (int j = 0; j < DIM; ++j) {
                    double s = 0.0;
                    for (int a = 0; a < DIM; ++a)
                        for (int b = 0; b < DIM; ++b) s += Ji[i][a] * D[a][b] * Ji[j][b];
                    K[i][j] = Wq * fabs(det) * s2h[i] * s * s2h[j];
                    rec[i * DIM + j] = K[i][j];
                }
            R* gv = gvol + q * VPN * FS;
            if (DIM == 2) {
                gv[0] = (R)K[0][0]; gv[FS] = (R)K[1][1]; gv[2 * FS] = (R)K[0][1];
            } else {
                gv[0] = (R)K[0][0]; gv[FS] = (R)K[1][1]; gv[2 * FS] = (R)K[2][2];
                gv[3 * FS] = (R)K[0][1]; gv[4 * FS] = (R)K[0][2]; gv[5 * FS] = (R)K[1][2];
            }
            const double mq = Wq * fabs(det);
            mass[q] = mq;
            gv[NS * FS] = (R)mq;
            sm[q] = mq;
            for (int s = 0; s < nstim; ++s) {
                bool in = true;
                for (int k = 0; k < DIM; ++k) in = in && x[k] >= slo[s][k] && x[k] <= shi[s][k];
                if (in) mk[s] |= 1u << q;
            }
        } else if (p < npt) {
            int f = 0;
            while (off[f + 1] <= p) ++f;
            const int kind = kinds[f], r = p - off[f], sb = r / NPF, t = r - sb * NPF;
            const int k = f >> 1, sd = f & 1;
            const double sgn = sd ? 1.0 : -1.0;
            int tg[2] = {0, 0}, nt = 0;
            for (int l = 0; l < DIM; ++l)
                if (l != k) tg[nt++] = l;
            const double* bs = sd ? T.bR : T.bL;
            const double* ds = sd ? T.dR : T.dL;
            const double pen = kind == 2 ? 0.75 : (kind == 3 ? 1.5 : 1.0);   // (1 + h_own / h_nb) / 2
            const int at[2] = {t % N1, t / N1};
            double X[3] = {0.0, 0.0, 0.0};
            double Wt = 1.0;
            double xi_t[2] = {0.0, 0.0};
            X[k] = Xc[k] + (sd ? h[k] : 0.0);
            for (int z = 0; z < nt; ++z) {
                const int l = tg[z];
                if (kind == 3) {
                    const int bit = (sb >> z) & 1;
                    const double xf = (xg[at[z]] + 2.0 * bit - 1.0) * 0.5;
                    X[l] = Xc[l] + (xf + 1.0) * 0.5 * h[l];
                    Wt *= T.w[at[z]] * h[l] * 0.25;
                    xi_t[z] = xf;
                } else {
                    X[l] = Xc[l] + (xg[at[z]] + 1.0) * 0.5 * h[l];
                    Wt *= T.w[at[z]] * h[l] * 0.5;
                    xi_t[z] = xg[at[z]];
                }
            }
            double c[3] = {0.0, 0.0, 0.0}, adet = 0.0, ln = 0.0, nDn = 0.0;
            geo_face_point(g, X, h, k, sgn, c, &adet, &ln, &nDn);
            const double dS = Wt * adet * ln;
            const double kap = g.gamma * nDn * ln / h[k] * pen;
            if (sb == 0 && kind != 3) {
                R* gf = gface + (f * NPF + t) * FPV * FS;
                for (int i = 0; i < DIM; ++i) gf[i * FS] = (R)c[i];
                gf[DIM * FS] = (R)dS;
                gf[(DIM + 1) * FS] = (R)kap;
            }
            double lt[2][3], dlt[2][3];
            for (int z = 0; z < nt; ++z) geo_lagrange<N1>(xg, xi_t[z], lt[z], dlt[z]);
            for (int i = 0; i < NP; ++i) {
                const int ak = digit<N1>(i, k);
                double tv = 1.0;
                for (int z = 0; z < nt; ++z) tv *= lt[z][digit<N1>(i, tg[z])];
                double cgi = c[k] * ds[ak] * tv;
                for (int z = 0; z < nt; ++z) {
                    double dz = bs[ak] * dlt[z][digit<N1>(i, tg[z])];
                    for (int z2 = 0; z2 < nt; ++z2)
                        if (z2 != z) dz *= lt[z2][digit<N1>(i, tg[z2])];
                    cgi += c[tg[z]] * dz;
                }
                rec[i] = bs[ak] * tv;
                rec[NP + i] = cgi;
            }
            rec[2 * NP] = dS;
            rec[2 * NP + 1] = kap;
        }
        __syncwarp();
        // block entries (i, j) = (ent / NP, ent % NP), ent = lane + 32 u, summed over the chunk's points
        const int pe = min(CH, npt - c0);
        for (int pp = 0; pp < pe; ++pp) {
            const double* d = spt + pp * PS;
            if (c0 + pp < NP) {
                // volume node q: B_ij += g_i^T K g_j, g_i = grad psi_i at q (nonzero when i and q
                // differ in at most one digit k: D1[q_k][i_k] there)
                const int q = c0 + pp;
#pragma unroll
                for (int u = 0; u < NE; ++u) {
                    const int ent = lane + 32 * u;
                    if (ent >= NP * NP) continue;
                    const int i = ent / NP, j = ent - (ent / NP) * NP;
                    int di = 0, ki = 0, dj = 0, kj = 0;
                    for (int k = 0; k < DIM; ++k) {
                        if (digit<N1>(i, k) != digit<N1>(q, k)) { ++di; ki = k; }
                        if (digit<N1>(j, k) != digit<N1>(q, k)) { ++dj; kj = k; }
                    }
                    if (di > 1 || dj > 1) continue;
                    double s = bacc[u];
                    for (int k = 0; k < DIM; ++k) {
                        if (di == 1 && k != ki) continue;
                        const double gik = T.D1[digit<N1>(q, k)][digit<N1>(i, k)];
                        for (int l = 0; l < DIM; ++l) {
                            if (dj == 1 && l != kj) continue;
                            s += gik * d[k * DIM + l] * T.D1[digit<N1>(q, l)][digit<N1>(j, l)];
                        }
                    }
                    bacc[u] = s;
                }
            } else {
                const double dS = d[2 * NP], kap = d[2 * NP + 1];
#pragma unroll
                for (int u = 0; u < NE; ++u) {
                    const int ent = lane + 32 * u;
                    if (ent >= NP * NP) continue;
                    const int i = ent / NP, j = ent - (ent / NP) * NP;
                    const double pi = d[i], ci = d[NP + i];
                    if (pi == 0.0 && ci == 0.0) continue;
                    bacc[u] += dS * (-0.5 * d[NP + j] * pi - 0.5 * ci * d[j] + kap * pi * d[j]);
                }
            }
        }
        __syncwarp();
    }
    // Gershgorin: max_i sum_j |B_ij| / M_i
#pragma unroll
    for (int u = 0; u < NE; ++u) {
        const int ent = lane + 32 * u;
        if (ent < NP * NP) spt[ent] = fabs(bacc[u]);
    }
    __syncwarp();
    double mx = 0.0;
    if (lane < NP) {
        double row = 0.0;
        for (int j = 0; j < NP; ++j) row += spt[lane * NP + j];
        mx = row / sm[lane];
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    for (int s = 0; s < nstim; ++s) sk[s] = __reduce_or_sync(0xffffffffu, mk[s]);
    __syncwarp();
    return 1.0 / mx;
}

// Part 2: the factors of the listed elements (todo[0 .. m->nfac)), one warp per element
// (geo_element_warp), with their b^CFL, signature and stimulus masks.  List entry j goes to
// warp j mod (number of warps), the warps numbered block-fastest, so that a run of neighbouring
// elements (a refined patch) spreads over every SM.
template <typename R, int DIM, int P>
__global__ void __launch_bounds__(64) k_mapped_factors(
        const int4* coord, const uint32_t* info, const MapArgs a, const Tables<double> Td, R* gvol, R* gface,
        double* mass, uint32_t* fsig, uint32_t* f0, uint32_t* f1, uint32_t* f2, uint32_t* f3, uint8_t* bcfl,
        uint32_t* sm0, uint32_t* sm1, uint32_t* sm2, uint32_t* sm3, const int32_t* todo, DevMeta* m) {
    pdl_enter();
    using W = GeoWarp<DIM, P>;
    constexpr int NP = W::NP, NF = W::NF;
    constexpr int NV = NP * W::VPN, NFV = NF * W::NPF * W::FPV;
    __shared__ double s_pt[2][W::CH * W::PS];
    __shared__ double s_m[2][NP];
    if (m->err) return;
    uint32_t* smask[4] = {sm0, sm1, sm2, sm3};
    uint32_t* fsm[4] = {f0, f1, f2, f3};
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t n = m->nfac;
    if (blockIdx.x == 0 && threadIdx.x == 0) m->fac_updates += n;
    for (int64_t j = blockIdx.x + (int64_t)gridDim.x * wib; j < n; j += 2 * (int64_t)gridDim.x) {
        const int64_t e = todo[j];
        const int4 c4 = coord[e];
        const uint32_t inf = info[e];
        uint32_t kbits = 0;
        int kinds[6] = {0, 0, 0, 0, 0, 0};
        for (int f = 0; f < NF; ++f) {
            kinds[f] = (inf >> (4 * f)) & 3;
            kbits |= (uint32_t)kinds[f] << (2 * f);
        }
        const int cc[3] = {c4.x, c4.y, c4.z};
        uint32_t sk[MDL_MAX_STIM] = {0u, 0u, 0u, 0u};
        const double cfl = geo_element_warp<R, DIM, P>(a.g, Td, a.xg, a.h0, c4.w, cc, kinds, a.nstim, a.slo, a.shi,
                                                       s_pt[wib], s_m[wib], factors_of(gvol, e, NV),
                                                       factors_of(gface, e, NFV), mass + (size_t)e * NP, sk);
        if (lane == 0) {
            const int b = a.lts ? b_from_bound_dev(a.dt, cfl) : 0;
            bcfl[e] = (uint8_t)b;
            fsig[e] = kbits | ((uint32_t)c4.w << 12) | ((uint32_t)b << 16);
            for (int s = 0; s < a.nstim; ++s) smask[s][e] = fsm[s][e] = sk[s];
        }
    }
}

template <typename R, int DIM, int P>
__global__ void __launch_bounds__(128) k_tick_mapped(const TickArgs<R> a, const Tables<R> T, const Phys<R> ph) {
    // as k_tick: the due count and the first element's metadata before the dependent wait
    const int n_act = a.d.meta->nact[a.tick];
    const bool bad = a.d.meta->err != 0;
    const int idx0 = (int)gtid();
    TickMeta<DIM, P> m;
    if (idx0 < n_act) tick_fetch<R, DIM, P>(a.d, idx0, m);
    pdl_enter();
    if (bad) return;
    for (int idx = idx0; idx < n_act; idx += (int)gstride()) {
        if (idx != idx0) tick_fetch<R, DIM, P>(a.d, idx, m);
        tick_elem_mapped<R, DIM, P>(a, T, ph, a.tick, m);
    }
}

}  // namespace mdl
