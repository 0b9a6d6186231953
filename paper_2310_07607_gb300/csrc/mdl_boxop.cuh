// mdl_boxop.cuh -- the SIPG operator of box elements as sums of one-dimensional lines.
//
// On a box element the GL collocation mass is diagonal and a product over the directions, so
// rho = M^-1 A u (the operator of Eq. monodomain-primal-formulation with the flux of
// Eq. monodomain-numerical-flux) needs no quadrature at run time:
//   own part   along every line of p+1 nodes in direction k, rho += S_k y: the volume term and
//              both own face terms with same-level neighbours, one (p+1) x (p+1) matrix per
//              direction; for every non-zero D_kl, rho -= X_kl (D~_k D~_l + D_k D_l) y with
//              D the derivative matrix and D~ = w^-1 D^T w (the volume's and the faces' mixed
//              terms together, by summation by parts of the GL rule);
//   face (k,s) with the neighbour's trace TN and normal derivative DN at the face's nodes (in
//              units of the element's own reference length), rho += LT TN + LD DN along the
//              lines of direction k, and beta Xv with Xv the mixed terms of D_kl.
// Faces that are not same-level interior faces enter through the same TN and DN:
//   boundary         TN = own trace, DN = - own normal derivative (no jump, no mean flux);
//   coarser          TN, DN interpolated to the face's nodes (DN halved: its length is double);
//   finer            TN, DN restricted from the subfaces by the fine GL rule (DN doubled);
// with beta kappa (kr - 1) (own trace - TN) for the changed penalty, kr = 3/4 for a coarser
// and 3/2 for a finer neighbour.  (The own part over the subfaces of a finer neighbour is the
// same-level one: the fine GL rule restricts an interpolated polynomial exactly.)
// At refinement level l every value is 4^l times the level-0 one (h halves), an exact scale:
// one set of constants serves all levels.  They are kernel arguments, which the FP32 and FP64
// instructions read as constant operands.
// A annihilates constants, so callers pass values shifted by a value of the element: the sums
// then round relative to the local variation of the field.
#pragma once

#include "mdl_element.cuh"

namespace mdl {

template <typename R>
struct BoxOp {
    R S[3][3][3];       // [k][a][j] own line matrix of direction k
    R LT[3][2][3];      // [k][side][a] weight of TN
    R LD[3][2][3];      // [k][side][a] weight of DN
    R be[3][2][3];      // [k][side][a] beta: lift of a face value
    R kap[3];           // same-level penalty of a normal-k face
    R X[3];             // D_kl (2/h_k)(2/h_l) of the pairs (0,1), (0,2), (1,2)
    R XF[3][2][3];      // [k][side][l] -s D_kl (2/h_l): mixed face term
    R FK[3][3];         // [k][l] D_kl (2/h_l): flux of the spatial indicator
    R b[2][3], dn[2][3];// [side] traces and normal derivatives of a line
    R D1[3][3], Dt[3][3];
    R C[3][3];          // (D1 - Dt) / 2
    R E[3][3];          // D1 + Dt
    R PR[2][2][3][3];   // 0 [half][fine node][coarse node]: interpolation to a half of the face;
                        // 1 [half][coarse node][fine node]: restriction from it by the fine rule
    R wq[28];           // GL weight product of every node, 0 past the last
    int32_t cross;      // bit i: pair i of X is non-zero
};

// Q1 elements take the dense blocks of the operator instead (4 or 8 values: the lines save little),
// from level-0 constants for same-level faces: r = A_vol u + sum_f (A_own u + A_nb u_nb), times
// 2^((2-d) l) at level l.  The coefficients are those of the class blocks in memory, which the
// other face kinds use.
template <typename R, int DIM>
struct Q1Op {
    static constexpr int NP = 1 << DIM, NF = 2 * DIM;
    R vol[NP][NP];
    R face[NF][2][NP][NP];   // [face][0 own, 1 neighbour]
    R wq[NP];                // GL weight product of every node
};

template <typename R, int DIM, int P>
struct OpOf {
    using type = BoxOp<R>;
};
template <typename R, int DIM>
struct OpOf<R, DIM, 1> {
    using type = Q1Op<R, DIM>;
};
template <typename R, int DIM, int P>
using OpT = typename OpOf<R, DIM, P>::type;

// Node of line m (over the tangential nodes, the lower axis fastest) at position j of axis k.
template <int DIM, int P>
MDL_HD int line_node(int k, int m, int j) {
    constexpr int N1 = P + 1;
    int tg[2] = {0, 0};
    tangents<DIM>(k, tg);
    int q = j * stride<N1>(k) + (m % N1) * stride<N1>(tg[0]);
    if (DIM == 3) q += (m / N1) * stride<N1>(tg[1]);
    return q;
}

// rho = own part.  cross: op.cross != 0, which a kernel of its own for diagonal tensors knows.
template <typename R, int DIM, int P>
MDL_HD void box_own(const BoxOp<R>& op, const R* y, R* rho, bool cross) {
    using S = Shape<DIM, P>;
    constexpr int N1 = S::N1, NP = S::NP, NT = S::NT;
#pragma unroll
    for (int k = 0; k < DIM; ++k)
#pragma unroll
        for (int m = 0; m < NT; ++m)
#pragma unroll
            for (int a = 0; a < N1; ++a) {
                const int q = line_node<DIM, P>(k, m, a);
                R s = k == 0 ? R(0) : rho[q];
#pragma unroll
                for (int j = 0; j < N1; ++j) s += op.S[k][a][j] * y[line_node<DIM, P>(k, m, j)];
                rho[q] = s;
            }
    if (cross) {
#pragma unroll
        for (int k = 0; k < DIM; ++k)
#pragma unroll
            for (int l = k + 1; l < DIM; ++l) {
                const int pr = k + l - 1;
                if (!((op.cross >> pr) & 1)) continue;
#pragma unroll
                for (int v = 0; v < 2; ++v) {
                    R t[NP];
#pragma unroll
                    for (int m = 0; m < NT; ++m)
#pragma unroll
                        for (int a = 0; a < N1; ++a) {
                            R s = 0;
#pragma unroll
                            for (int j = 0; j < N1; ++j)
                                s += (v ? op.D1[a][j] : op.Dt[a][j]) * y[line_node<DIM, P>(l, m, j)];
                            t[line_node<DIM, P>(l, m, a)] = op.X[pr] * s;
                        }
#pragma unroll
                    for (int m = 0; m < NT; ++m)
#pragma unroll
                        for (int a = 0; a < N1; ++a) {
                            const int q = line_node<DIM, P>(k, m, a);
                            R s = rho[q];
#pragma unroll
                            for (int j = 0; j < N1; ++j)
                                s -= (v ? op.D1[a][j] : op.Dt[a][j]) * t[line_node<DIM, P>(k, m, j)];
                            rho[q] = s;
                        }
                }
            }
    }
}

// Trace and normal derivative of y on its side-`side` face of axis k.
template <typename R, int DIM, int P>
MDL_HD void box_trace(const BoxOp<R>& op, int k, int side, const R* y, R* tr, R* dn) {
    using S = Shape<DIM, P>;
#pragma unroll
    for (int m = 0; m < S::NT; ++m) {
        R a = 0, b = 0;
#pragma unroll
        for (int j = 0; j < S::N1; ++j) {
            const R x = y[line_node<DIM, P>(k, m, j)];
            a += op.b[side][j] * x;
            b += op.dn[side][j] * x;
        }
        tr[m] = a;
        dn[m] = b;
    }
}

// out (+)= f A along tangent ti (0 or 1) of a face's values in.
template <typename R, int DIM, int P>
MDL_HD void face_line(const R (&A)[3][3], int ti, R f, const R* in, R* out, bool add) {
    using S = Shape<DIM, P>;
    constexpr int N1 = S::N1;
    const int st = ti == 0 ? 1 : N1;
#pragma unroll
    for (int t = 0; t < S::NT; ++t) {
        const int tt = (t / st) % N1, base = t - tt * st;
        R s = 0;
#pragma unroll
        for (int m = 0; m < N1; ++m) s += A[tt][m] * in[base + m * st];
        out[t] = add ? out[t] + f * s : f * s;
    }
}

// out = (A_c0 x A_c1) in over a face's values: interpolation to (A = PR[0]) or restriction from
// (A = PR[1]) the subface of halves c0, c1.
template <typename R, int DIM, int P>
MDL_HD void face_map(const R (&A)[2][3][3], int c0, int c1, const R* in, R* out) {
    using S = Shape<DIM, P>;
    if (DIM == 2) {
        face_line<R, DIM, P>(A[c0], 0, R(1), in, out, false);
    } else {
        R t[S::NT];
        face_line<R, DIM, P>(A[c0], 0, R(1), in, t, false);
        face_line<R, DIM, P>(A[c1], 1, R(1), t, out, false);
    }
}

// The transposes: out (+)= f A^T along tangent ti, out += (A_c0 x A_c1)^T in.
template <typename R, int DIM, int P>
MDL_HD void face_line_t(const R (&A)[3][3], int ti, R f, const R* in, R* out, bool add) {
    using S = Shape<DIM, P>;
    constexpr int N1 = S::N1;
    const int st = ti == 0 ? 1 : N1;
#pragma unroll
    for (int t = 0; t < S::NT; ++t) {
        const int tt = (t / st) % N1, base = t - tt * st;
        R s = 0;
#pragma unroll
        for (int m = 0; m < N1; ++m) s += A[m][tt] * in[base + m * st];
        out[t] = add ? out[t] + f * s : f * s;
    }
}
template <typename R, int DIM, int P>
MDL_HD void face_map_t_add(const R (&A)[2][3][3], int c0, int c1, const R* in, R* out) {
    using S = Shape<DIM, P>;
    if (DIM == 2) {
        face_line_t<R, DIM, P>(A[c0], 0, R(1), in, out, true);
    } else {
        R t[S::NT];
        face_line_t<R, DIM, P>(A[c0], 0, R(1), in, t, false);
        face_line_t<R, DIM, P>(A[c1], 1, R(1), t, out, true);
    }
}

// Mixed terms of a same-level or coarser neighbour: Xv = sum_l XF_kl C_l TN.
template <typename R, int DIM, int P>
MDL_HD void box_mixed(const BoxOp<R>& op, int k, int side, const R* TN, R* Xv) {
    int tg[2] = {0, 0};
    tangents<DIM>(k, tg);
#pragma unroll
    for (int ti = 0; ti < DIM - 1; ++ti) face_line<R, DIM, P>(op.C, ti, op.XF[k][side][tg[ti]], TN, Xv, ti > 0);
}

// rho += LT TN + LD DN (+ beta Xv) along the lines of axis k.
template <typename R, int DIM, int P, bool XV>
MDL_HD void box_lift(const BoxOp<R>& op, int k, int side, const R* TN, const R* DN, const R* Xv, R* rho) {
    using S = Shape<DIM, P>;
#pragma unroll
    for (int m = 0; m < S::NT; ++m)
#pragma unroll
        for (int a = 0; a < S::N1; ++a) {
            const int q = line_node<DIM, P>(k, m, a);
            R s = rho[q] + op.LT[k][side][a] * TN[m];
            s += op.LD[k][side][a] * DN[m];
            if (XV) s += op.be[k][side][a] * Xv[m];
            rho[q] = s;
        }
}

// TN, DN and beta's factor Xv (mixed terms and changed penalty) of a face that is not a
// same-level interior face.  y: the own values; nb(i, v): values i of the neighbour (coarser:
// i = 0; finer: i = the subface) on the caller's shift.
template <typename R, int DIM, int P, typename NB>
MDL_HD void box_face_irregular(const BoxOp<R>& op, int k, int side, int kind, int pos, const R* y, NB nb, R* TN, R* DN,
                               R* Xv, bool cross) {
    using S = Shape<DIM, P>;
    constexpr int NT = S::NT, NP = S::NP;
    int tg[2] = {0, 0};
    tangents<DIM>(k, tg);
    R to[NT], dno[NT];
    box_trace<R, DIM, P>(op, k, side, y, to, dno);
    if (kind == 0) {
#pragma unroll
        for (int m = 0; m < NT; ++m) {
            TN[m] = to[m];
            DN[m] = -dno[m];
            Xv[m] = R(0);
        }
        if (cross) {
            // no flux through the boundary: + s/2 D_kl (2/h_l) E_l times the own trace
#pragma unroll
            for (int ti = 0; ti < DIM - 1; ++ti)
                face_line<R, DIM, P>(op.E, ti, R(-0.5) * op.XF[k][side][tg[ti]], to, Xv, true);
        }
        return;
    }
    // a coarser neighbour and the subfaces of finer ones through one loop (the code is what the
    // kernels fetch): A = Pi or Rs, the normal derivative and the tangential one of the
    // neighbour's own length scaled to the element's
    const int fine = kind == 3 ? 1 : 0;
    const R fd = fine ? R(2) : R(0.5), fx = fine ? R(1) : R(0.25);
#pragma unroll
    for (int m = 0; m < NT; ++m) TN[m] = DN[m] = Xv[m] = R(0);
    const int sb0 = fine ? 0 : pos, sb1 = fine ? S::NSUB : pos + 1;
#pragma unroll 1
    for (int sb = sb0; sb < sb1; ++sb) {
        R v[NP], t[NT], dv[NT], z[NT];
        nb(fine ? sb : 0, v);
        box_trace<R, DIM, P>(op, k, 1 - side, v, t, dv);
        const int c0 = sb & 1, c1 = (sb >> 1) & 1;
        face_map<R, DIM, P>(op.PR[fine], c0, c1, t, z);
#pragma unroll
        for (int m = 0; m < NT; ++m) TN[m] += z[m];
        face_map<R, DIM, P>(op.PR[fine], c0, c1, dv, z);
#pragma unroll
        for (int m = 0; m < NT; ++m) DN[m] += fd * z[m];
        if (cross) {
#pragma unroll
            for (int ti = 0; ti < DIM - 1; ++ti)
                face_line<R, DIM, P>(op.D1, ti, fx * op.XF[k][side][tg[ti]], t, dv, ti > 0);
            face_map<R, DIM, P>(op.PR[fine], c0, c1, dv, z);
#pragma unroll
            for (int m = 0; m < NT; ++m) Xv[m] += z[m];
        }
    }
    if (cross) {
#pragma unroll
        for (int ti = 0; ti < DIM - 1; ++ti)
            face_line<R, DIM, P>(op.Dt, ti, R(-0.5) * op.XF[k][side][tg[ti]], TN, Xv, true);
    }
    const R kr = fine ? R(0.5) : R(-0.25);
#pragma unroll
    for (int m = 0; m < NT; ++m) Xv[m] += op.kap[k] * kr * (to[m] - TN[m]);
}

// Host construction (FP64) and conversion.
void make_boxop(const Tables<double>& T, const Phys<double>& ph, int dim, int p, BoxOp<double>* op);
template <typename R>
void convert_boxop(const BoxOp<double>& a, BoxOp<R>* b);

}  // namespace mdl
