// mdl_q23.cuh -- the sweep tick of Q2 3D FP32 contexts (MDL_SWEEP_THREAD, their default).
//
// A thread per due element, with the operator of mdl_boxop.cuh (about 1,000 multiply-adds) and
// ap_step (about 1,450 operations for the 27 DOFs).  A step reads the element's row of 27 values
// and six neighbour rows, and the element's state and barrier-start rows.  Loaded by the thread
// that uses them these are 16-byte accesses to 32 rows per instruction, whose 32 cache lines the
// L1 looks up one by one.  So a warp copies its rows together: 7 consecutive lanes take one row
// (7 x 16 bytes), a cp.async moves 32 chunks of 4 to 5 rows, and the block of 32 rows lands in
// shared memory as it is used: each thread reads its own row at a stride of 28 words, which is
// free of bank conflicts for 16-byte accesses (eight lanes cover the 32 banks).  The copies run
// ahead of their use: both neighbours of an axis while the previous axis is worked on, the state
// and the barrier-start terms during the last axes.  The results go back the same way.  The
// metadata (face info, neighbours, level bytes) of the warp's next 32 elements is fetched a step
// ahead.
#pragma once

#include "mdl_kernels.cuh"

namespace mdl {
namespace q23 {

constexpr int NP = 27, NPS = 28, NT = 9, NF = 6;
constexpr int ROWS = 5;                                   // blocks of 32 rows: A0, A1, B0, B1, own values
constexpr int BLK = 32 * NPS;                             // floats of a block
constexpr int smem_bytes(int threads) { return ROWS * NPS * 4 * threads; }
constexpr int eta_smem_bytes(int threads) { return 4 * NPS * 4 * threads; }

// Row r of the warp's block dst from lane r's `row`: chunk t = 32 j + lane is chunk t % 7 of row
// t / 7, and the block is contiguous.
__device__ __forceinline__ void copy_rows(float* dst, const float* row, int lane) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst) + 16 * lane;
#pragma unroll
    for (int j = 0; j < 7; ++j) {
        const int t = 32 * j + lane, r = t / 7, c = t - 7 * r;
        const float* src = reinterpret_cast<const float*>(__shfl_sync(0xffffffffu, (long long)row, r)) + 4 * c;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 512 * j), "l"(src) : "memory");
    }
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// All but the last N groups of every lane have landed.
template <int N>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
    __syncwarp();
}
// Lane r's `row` (not null) from row r of the block.
__device__ __forceinline__ void store_rows(float* row, const float* src, int lane) {
#pragma unroll
    for (int j = 0; j < 7; ++j) {
        const int t = 32 * j + lane, r = t / 7, c = t - 7 * r;
        float* dst = reinterpret_cast<float*>(__shfl_sync(0xffffffffu, (long long)row, r));
        const float4 v = *reinterpret_cast<const float4*>(src + 4 * t);
        if (dst) reinterpret_cast<float4*>(dst)[c] = v;
    }
}

// Metadata of the next element of the thread, in flight.
struct Next {
    int e;
    uint32_t inf;
    uint8_t lv;
    int nbf[NF];
};

__device__ __forceinline__ void fetch_next(const DevArrays<float>& d, Next& n) {
    n.inf = d.info[n.e];
    n.lv = d.lvl[n.e];
#pragma unroll
    for (int f = 0; f < NF; f += 2) {
        const int2 x = *reinterpret_cast<const int2*>(d.nbr + (size_t)n.e * NF + f);
        n.nbf[f] = x.x;
        n.nbf[f + 1] = x.y;
    }
}
__device__ __forceinline__ void fetch_levels(const DevArrays<float>& d, const Next& n, uint8_t* lvn) {
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const int kind = (n.inf >> (4 * f)) & 3;
        lvn[f] = d.lvl[(kind == 1 || kind == 2) ? n.nbf[f] : n.e];
    }
}

}  // namespace q23

// (The bound of 384 threads gives 168 registers, three blocks of 128 threads per SM, without
// spills; 128 registers spill and were 16% slower.)
template <int DIM, int P, bool CROSS>
__global__ void __launch_bounds__(384, 1) k_tick_q23(const TickArgs<float> a, const Tables<float> T,
                                                    const Phys<float> ph, const BoxOp<float> op) {
    static_assert(DIM == 3 && P == 2, "Q2 3D only");
    using namespace q23;
    extern __shared__ __align__(16) float rows[];
    const DevArrays<float>& d = a.d;
    const int tick = a.tick, B = a.B;
    const int n_act = d.meta->nact[tick];
    const bool bad = d.meta->err != 0;
    const int lane = threadIdx.x & 31;
    const int G = (int)gstride();
    int base = (int)gtid() - lane;                         // the warp's first due element
    // a warp without an element leaves its SM to other work; a tick without any must still end after
    // the tick before it (the next one waits for this one only)
    if (base >= n_act) {
        if (n_act == 0) pdl_enter();
        return;
    }
    // a warp's blocks of rows, and the thread's row in each
    float* const A0 = rows + (size_t)(threadIdx.x >> 5) * ROWS * BLK;
    float *const A1 = A0 + BLK, *const B0 = A0 + 2 * BLK, *const B1 = A0 + 3 * BLK, *const U = A0 + 4 * BLK;
    const int my = lane * NPS;
    // metadata is fixed during a sweep: the first elements' is read before the dependent wait
    // (lanes past the last due element repeat it and store nothing)
    TickMeta<3, 2> m;
    Next nx;
    nx.e = d.order[min(base + lane, n_act - 1)];
    fetch_next(d, nx);
    fetch_levels(d, nx, m.lvn);
    int e_next = base + G < n_act ? d.order[min(base + G + lane, n_act - 1)] : nx.e;
    pdl_enter();
    if (bad) return;
    const bool first = tick == 0;                          // of the barrier, for every due element
    const bool ap = ph.ionic == 0 && ph.integrator == 1;
    const ApConst apc(ph);
    for (;;) {
        const int e = m.e = nx.e;
        const uint32_t inf = m.inf = nx.inf;
        m.lv = nx.lv;
#pragma unroll
        for (int f = 0; f < NF; ++f) m.nbf[f] = nx.nbf[f];
        const bool valid = base + lane < n_act;
        const int b = m.lv & 7, par = (m.lv >> 3) & 1;
        const int ke = tick >> (B - b);
        const int cur = par ^ (ke & 1);
        const int lev = (inf >> 24) & 15;
        const size_t o = (size_t)e * NPS;
        const float* Vc = (cur ? d.V1 : d.V0) + o;
        // the row that holds the value seen of the face's neighbour (a row of its own where the
        // face is not a same-level one: those faces load in their own path)
        auto seen = [&](int f, const float*& ol, float& t) {
            const bool same = ((inf >> (4 * f)) & 3) == 1;
            return seen_row<float, NPS>(d, tick, B, same ? m.nbf[f] : e, same ? m.lvn[f] : m.lv, ol, t);
        };
        auto stage_axis = [&](int k, float* r0) {
            const float* ol;
            float t;
            copy_rows(r0, seen(2 * k, ol, t), lane);
            copy_rows(r0 + BLK, seen(2 * k + 1, ol, t), lane);
            copy_commit();
        };
        copy_rows(U, Vc, lane);
        copy_commit();
        stage_axis(0, A0);
        stage_axis(1, B0);
        nx.e = e_next;
        fetch_next(d, nx);
        const double acc0 = first ? 0.0 : d.acc[e];
        copy_wait<2>();
        float c, y[NP], rho[NP];
        {
            float t[NPS];
            ld_vec<float, NPS>(U + my, t);
            c = t[NP / 2];
#pragma unroll
            for (int q = 0; q < NP; ++q) y[q] = t[q] - c;
        }
        box_own<float, 3, 2>(op, y, rho, CROSS);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            copy_wait<1>();
            float* const r0 = k == 1 ? B0 : A0;
#pragma unroll 1
            for (int side = 0; side < 2; ++side) {
                const uint32_t fi = inf >> (8 * k + 4 * side);
                const int kind = fi & 3;
                const int nbf = side ? m.nbf[2 * k + 1] : m.nbf[2 * k];
                const uint8_t lvn = side ? m.lvn[2 * k + 1] : m.lvn[2 * k];
                float TN[NT], DN[NT];
                if (kind == 1) {
                    float v[NPS];
                    ld_vec<float, NPS>(r0 + side * BLK + my, v);
                    const int rem = tick & ((1 << (B - (lvn & 7))) - 1);
                    if (rem) {
                        const float* ol;
                        float t;
                        seen_row<float, NPS>(d, tick, B, nbf, lvn, ol, t);
                        interp_row<float, NP, NPS>(ol, t, v);
                    }
#pragma unroll
                    for (int q = 0; q < NP; ++q) v[q] -= c;
                    box_trace<float, 3, 2>(op, k, 1 - side, v, TN, DN);
                    if constexpr (CROSS) {
                        float Xv[NT];
                        box_mixed<float, 3, 2>(op, k, side, TN, Xv);
                        box_lift<float, 3, 2, true>(op, k, side, TN, DN, Xv, rho);
                    } else {
                        box_lift<float, 3, 2, false>(op, k, side, TN, DN, nullptr, rho);
                    }
                } else {
                    auto nb = [&](int sb, float* v) {
                        const int n = kind == 2 ? nbf : d.hang[nbf + sb];
                        const float* ol;
                        float t;
                        ld_dofs<float, NP, NPS>(seen_row<float, NPS>(d, tick, B, n, kind == 2 ? lvn : d.lvl[n], ol, t), v);
                        if (t > 0.0f) interp_row<float, NP, NPS>(ol, t, v);
#pragma unroll
                        for (int q = 0; q < NP; ++q) v[q] -= c;
                    };
                    float Xv[NT];
                    box_face_irregular<float, 3, 2>(op, k, side, kind, (fi >> 2) & 3, y, nb, TN, DN, Xv, CROSS);
                    box_lift<float, 3, 2, true>(op, k, side, TN, DN, Xv, rho);
                }
                if (k == 2 && side == 0) {
                    __syncwarp();
                    if (!first) copy_rows(A0, d.ga + o, lane);   // block A0 is read: the barrier-start g
                    copy_commit();
                }
            }
            __syncwarp();
            if (k == 0) stage_axis(2, A0);
            if (k == 1) {
                copy_rows(B0, d.v + o, lane);
                if (!first) copy_rows(B1, d.Ia + o, lane);
                copy_commit();
            }
        }
        {
            float t[NPS];
#pragma unroll
            for (int q = 0; q < NPS; ++q) t[q] = q < NP ? rho[q] : 0.0f;
            st_vec<float, NPS>(A1 + my, t);
        }
        // the next elements' level bytes (their neighbours have arrived)
        fetch_levels(d, nx, m.lvn);
        e_next = base + 2 * G < n_act ? d.order[min(base + 2 * G + lane, n_act - 1)] : nx.e;
        copy_wait<0>();

        // pointwise step, four DOFs at a time (the pad value steps too and stays 0); the results
        // replace the values in the blocks
        const float dte = a.dteR[b], sc = (float)(1 << (2 * lev));
        StimMasks stm;
        elem_stim<float>(a, e, inf, tick, a.dte[b], stm);
        float term = 0.0f, vmax = 0.0f;
#pragma unroll 1
        for (int i = my; i < my + NPS; i += 4) {
            float u[4], w[4], r[4], Ia[4], ga[4], un[4], wn[4], so[4], smd[4];
            ld4<float>(U + i, u);
            ld4<float>(B0 + i, w);
            ld4<float>(A1 + i, r);
            if (first) {
#pragma unroll
                for (int j = 0; j < 4; ++j) Ia[j] = ga[j] = 0.0f;
            } else {
                ld4<float>(B1 + i, Ia);
                ld4<float>(A0 + i, ga);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) so[j] = smd[j] = 0.0f;
            if (stm.any) {
#pragma unroll
                for (int j = 0; j < 4; ++j) node_stim<float>(a, stm, i - my + j, so[j], smd[j]);
            }
            if (ap) {
                term += ap_step<4>(apc, first, op.wq + (i - my), sc, dte, so, smd, u, w, r, Ia, ga, un, wn);
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    term += dof_update<float>(ph, op.wq[i - my + j], sc, ke, dte, so[j], smd[j], u[j], w[j], r[j],
                                              Ia[j], ga[j], un[j], wn[j]);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) vmax = fmaxf(vmax, fabsf(un[j]));
            st4<float>(U + i, un);
            st4<float>(B0 + i, wn);
            if (first) {
                st4<float>(B1 + i, Ia);
                st4<float>(A0 + i, ga);
            }
        }
        __syncwarp();
        store_rows(valid ? (cur ? d.V0 : d.V1) + o : nullptr, U, lane);
        store_rows(valid ? d.v + o : nullptr, B0, lane);
        if (first) {
            store_rows(valid && b > 0 ? d.Ia + o : nullptr, B1, lane);
            store_rows(valid && b > 0 ? d.ga + o : nullptr, A0, lane);
        }
        if (valid) {
            d.acc[e] = acc0 + a.dte[b] * (double)(ph.Wvol[lev] * term);
            if ((inf & INFO_PENDING) && vmax >= ph.lat_gate)
                lat_check<float, 3, 2>(d, T, ph, e, inf, lev, Vc, U + my, tick_time(a, tick), a.dte[b]);
        }
        base += G;
        if (base >= n_act) return;
        __syncwarp();                                      // the blocks are read: the next rows may land
    }
}

// The spatial indicator of Q2 3D FP32 contexts (k_eta_s_q2's sums) with the same row copies: the
// own rows and axis 0, then two axes ahead in turn.
template <int DIM, int P>
__global__ void __launch_bounds__(128, 4) k_eta_q23(const DevArrays<float> d, const Tables<float> T,
                                                   const Phys<float> ph, const BoxOp<float> op, const MarkArgs mark) {
    static_assert(DIM == 3 && P == 2, "Q2 3D only");
    using namespace q23;
    extern __shared__ __align__(16) float rows[];
    pdl_enter();
    if (d.meta->err) return;
    if (gtid() == 0) d.meta->changed = 0u;
    const int64_t ne = d.meta->ne;
    const int lane = threadIdx.x & 31;
    float* const A0 = rows + (size_t)(threadIdx.x >> 5) * 4 * BLK;
    const int my = lane * NPS;
    for (int64_t base = gtid() - lane; base < ne; base += gstride()) {
        const bool valid = base + lane < ne;
        const int e = (int)(valid ? base + lane : ne - 1);
        const uint32_t inf = d.info[e];
        const int lev = (inf >> 24) & 15;
        int nbf[NF];
        uint8_t lvn[NF];
#pragma unroll
        for (int f = 0; f < NF; f += 2) {
            const int2 x = *reinterpret_cast<const int2*>(d.nbr + (size_t)e * NF + f);
            nbf[f] = ((inf >> (4 * f)) & 3) == 1 ? x.x : e;
            nbf[f + 1] = ((inf >> (4 * f + 4)) & 3) == 1 ? x.y : e;
        }
        const uint8_t lv = d.lvl[e];
#pragma unroll
        for (int f = 0; f < NF; ++f) lvn[f] = d.lvl[nbf[f]];
        auto value_row = [&](int n, uint8_t l) { return (((l >> 3) & 1) ? d.V1 : d.V0) + (size_t)n * NPS; };
        auto stage_axis = [&](int k, float* r0) {
            copy_rows(r0, value_row(nbf[2 * k], lvn[2 * k]), lane);
            copy_rows(r0 + BLK, value_row(nbf[2 * k + 1], lvn[2 * k + 1]), lane);
            copy_commit();
        };
        __syncwarp();                                   // the blocks of the last elements are read
        copy_rows(A0 + 2 * BLK, value_row(e, lv), lane);
        stage_axis(0, A0);
        copy_wait<0>();
        float t[NPS], y[NP];
        ld_vec<float, NPS>(A0 + 2 * BLK + my, t);
        const float c = t[NP / 2];
#pragma unroll
        for (int q = 0; q < NP; ++q) y[q] = t[q] - c;
        __syncwarp();
        stage_axis(1, A0 + 2 * BLK);
        auto row = [&](int n, float* v) {
            ld_dofs<float, NP, NPS>(value_row(n, d.lvl[n]), v);
#pragma unroll
            for (int q = 0; q < NP; ++q) v[q] -= c;
        };
        auto nbv = [&](int k, int side, float* v) {
            float x[NPS];
            ld_vec<float, NPS>(A0 + (k == 1 ? 2 * BLK : 0) + side * BLK + my, x);
#pragma unroll
            for (int q = 0; q < NP; ++q) v[q] = x[q] - c;
        };
        double acc = kelly_axis<float, DIM, 0>(d, op, T, ph, e, inf, lev, y, row, nbv);
        __syncwarp();
        stage_axis(2, A0);
        copy_wait<1>();
        acc += kelly_axis<float, DIM, 1>(d, op, T, ph, e, inf, lev, y, row, nbv);
        copy_wait<0>();
        acc += kelly_axis<float, DIM, 2>(d, op, T, ph, e, inf, lev, y, row, nbv);
        if (valid) {
            const double eta = sqrt_seeded(acc);
            d.eta_s[e] = eta;
            if (mark.r) mark_leaf<DIM>(mark, d.info, d.nbr, e, inf, eta);
        }
    }
}

}  // namespace mdl
