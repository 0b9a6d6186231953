// mdl_amr.cuh -- device-side forest adaptation, mesh tables and level ordering.
//
// One refine-then-coarsen step of Alg. 1 on the device, bit-identical to the
// forest bookkeeping it replaces:
//   (mark_leaf, in the indicator kernels) refine flags r_e = (eta_e >= tau_refine && level <
//                  max_refine) with their 2:1 closure: a refined leaf forces its coarser face
//                  neighbours; k_amr_mark for replayed indicators, k_amr_close for long chains
//   k_scan_blocks  complete families of consecutive siblings with every eta <= tau_coarsen, none
//                  refined, no outside face neighbour finer or refined -> coarsen; new leaves per
//                  old leaf (2^d, 1 or 0), their scan and the commit of the new mesh
//   k_scan_emit    new leaf coordinates in (root, Morton) order, the sort key of every new leaf (its
//                  lower corner on the finest grid: root id, then Morton index inside the root) for
//                  neighbour search, and the transfer plan
//   k_mesh_tables  face kinds/positions, neighbours, hanging lists, levels, probe and
//                  stimulus data, CFL class levels of the new mesh (only if it changed)
//   k_transfer     the state, and the elements' substep levels with their counts
// and the level ordering (a stable multi-split by b descending) with the due counts
// of every tick.  Every kernel loops over the device-resident element count, so the
// barrier runs without a host round trip.
#pragma once

#include <cuda_runtime.h>

#include "mdl_kernels.cuh"

namespace mdl {

// Geometry of the base grid and the finest grid.
struct Grid {
    int32_t base[3];
    int64_t fine[3];
    int32_t L;
    int32_t dim;
};

// Stimulus boxes with the inclusion slack already applied, and the GL nodes.
struct StimBoxes {
    int n;
    double lo[MDL_MAX_STIM][3], hi[MDL_MAX_STIM][3];
    double xi[3];
};

// --------------------------------------------------------------------------
// Marks of replayed indicators (the library's own are marked where they are computed).
template <int DIM>
__global__ void k_amr_mark(const uint32_t* info, const int32_t* nbr, const double* eta, DevMeta* m, const MarkArgs mark) {
    pdl_enter();
    if (m->err) return;
    const int64_t ne = m->ne;
    for (int64_t e = gtid(); e < ne; e += gstride()) mark_leaf<DIM>(mark, info, nbr, e, info[e], eta[e]);
    if (gtid() == 0) m->changed = 0;
}

// One more step of the 2:1 closure.
template <int DIM>
__global__ void k_amr_close(const uint32_t* info, const int32_t* nbr, uint8_t* r, const DevMeta* m) {
    pdl_enter();
    if (m->err) return;
    constexpr int NF = 2 * DIM;
    const int64_t ne = m->ne;
    for (int64_t e = gtid(); e < ne; e += gstride()) {
        if (!r[e]) continue;
        const uint32_t inf = info[e];
        for (int f = 0; f < NF; ++f)
            if (((inf >> (4 * f)) & 3u) == 2u) r[nbr[(size_t)e * NF + f]] = 1;
    }
}

// Whether leaf e may coarsen with its siblings: eta <= tau_c, not refined, no face neighbour
// outside the family finer or refined.  Packed with its place: 0 no, else 1 + child index << 1 +
// level << 4.  (A family is 2^d consecutive leaves of one level with child indices 0, 1, ...: the
// leaves tile the domain in Morton order, so the leaf after child b is its sibling b + 1 if it has
// that level and index.)
template <int DIM>
__device__ __forceinline__ int may_coarsen(const int4* coord, const uint32_t* info, const int32_t* nbr,
                                           const double* eta, const uint8_t* r, int64_t e, double tau_c) {
    constexpr int NF = 2 * DIM;
    const int4 a = coord[e];
    const uint32_t ic = info[e];
    if (a.w == 0 || r[e] || !(eta[e] <= tau_c)) return 0;
    const int b = (a.x & 1) | ((a.y & 1) << 1) | (DIM == 3 ? ((a.z & 1) << 2) : 0);
    bool ok = true;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        if (((f & 1) != 0) != (((b >> (f >> 1)) & 1) != 0)) continue;      // a sibling's face
        const unsigned kind = (ic >> (4 * f)) & 3u;
        if (kind == 3u || (kind == 1u && r[nbr[(size_t)e * NF + f]])) ok = false;
    }
    return ok ? 1 | (b << 1) | (a.w << 4) : 0;
}

// Exclusive scan of cnt[0..ne) in chunks of SCAN_CHUNK per block: block sums, a one-block
// scan of the sums, then per-block scans with the block offset.  Writes the total to ne_new.
constexpr int SCAN_THREADS = 256, SCAN_ITEMS = 2, SCAN_CHUNK = SCAN_THREADS * SCAN_ITEMS;

__device__ __forceinline__ int64_t block_excl_scan(int64_t v, int64_t* sh, int64_t* total) {
    // inclusive warp scans then a scan over warp totals
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int64_t x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        const int nw = blockDim.x >> 5;
        int64_t t = lane < nw ? sh[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < nw) sh[lane] = t;
    }
    __syncthreads();
    const int64_t woff = w > 0 ? sh[w - 1] : 0;
    *total = sh[(blockDim.x >> 5) - 1];
    __syncthreads();
    return woff + x - v;
}

// New leaves per old leaf: 2^d if refined, 1 if kept or child 0 of a coarsened family
// (which becomes the parent), 0 for the other children of a coarsened family.
template <int DIM>
__device__ __forceinline__ int new_count(const int4* coord, const uint8_t* r, const uint8_t* c0, int64_t e) {
    if (r[e]) return 1 << DIM;
    if (c0[e]) return 1;
    const int4 a = coord[e];
    if (a.w > 0) {
        const int b = (a.x & 1) | ((a.y & 1) << 1) | (DIM == 3 ? ((a.z & 1) << 2) : 0);
        if (b > 0 && e - b >= 0 && c0[e - b]) return 0;
    }
    return 1;
}

// Coarsening families, new leaves per old leaf and their sums per chunk.  A chunk tests the leaves up
// to 2^d - 1 before and after it too: families that cross its ends.  (The scan of the sums is a launch
// of its own: done by the last block to arrive, its fence, its counter and one block's pass after the
// others cost 1 to 3 us more than a launch.)
template <int DIM>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_blocks(const int4* coord, const uint32_t* info,
                                                              const int32_t* nbr, const double* eta, const uint8_t* r,
                                                              uint8_t* c0, int64_t* bsum, DevMeta* m, double tau_c) {
    pdl_enter();
    if (m->err) return;
    constexpr int NC = 1 << DIM, HALO = NC - 1;
    __shared__ int64_t sh[32];
    __shared__ uint8_t may[SCAN_CHUNK + 2 * HALO];
    __shared__ uint8_t fam[SCAN_CHUNK + HALO];
    const int64_t ne = m->ne;
    const int64_t base = (int64_t)blockIdx.x * SCAN_CHUNK;
    if (base < ne) {
        for (int i = threadIdx.x; i < SCAN_CHUNK + 2 * HALO; i += SCAN_THREADS) {
            const int64_t e = base - HALO + i;
            may[i] = (uint8_t)(e >= 0 && e < ne ? may_coarsen<DIM>(coord, info, nbr, eta, r, e, tau_c) : 0);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < SCAN_CHUNK + HALO; i += SCAN_THREADS) {
            bool c = (may[i] & 0xf) == 1;
#pragma unroll
            for (int b = 1; b < NC; ++b) c = c && may[i + b] == (may[i] | (b << 1));
            fam[i] = c ? 1 : 0;
            const int64_t e = base - HALO + i;
            if (e >= base && e < ne) c0[e] = c ? 1 : 0;
        }
        __syncthreads();
        int64_t s = 0;
        bool ch = false;
        for (int i = 0; i < SCAN_ITEMS; ++i) {
            const int li = threadIdx.x * SCAN_ITEMS + i;
            const int64_t e = base + li;
            if (e < ne) {
                int n = 1;
                if (r[e]) {
                    n = NC;
                } else if (!fam[HALO + li]) {
                    const int4 a = coord[e];
                    const int b = a.w > 0 ? (a.x & 1) | ((a.y & 1) << 1) | (DIM == 3 ? ((a.z & 1) << 2) : 0) : 0;
                    if (b > 0 && fam[HALO + li - b]) n = 0;
                }
                s += n;
                ch = ch || n != 1 || fam[HALO + li];
            }
        }
        if (ch) m->changed = 1;
        int64_t tot;
        block_excl_scan(s, sh, &tot);
        if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
    }
}

// Exclusive scan of the block sums (one block) and the commit of the new mesh.
static __global__ void k_scan_top(int64_t* bsum, DevMeta* m, int64_t cap) {
    pdl_enter();
    if (m->err) return;
    __shared__ int64_t sh[32];
    const int64_t ne = m->ne;
    const int64_t nb = (ne + SCAN_CHUNK - 1) / SCAN_CHUNK;
    int64_t carry = 0;
    for (int64_t s0 = 0; s0 < nb; s0 += blockDim.x) {
        const int64_t i = s0 + threadIdx.x;
        const int64_t v = i < nb ? bsum[i] : 0;
        int64_t tot;
        const int64_t ex = block_excl_scan(v, sh, &tot);
        if (i < nb) bsum[i] = carry + ex;
        carry += tot;
    }
    if (threadIdx.x == 0) {
        if (carry > cap) {
            m->need = carry;
            atomicOr(&m->err, ERR_CAPACITY);
        } else {
            // commit: the new count becomes current, the other set becomes current
            m->ne_new = ne;          // old count, read by the emit pass
            m->ne = carry;
            m->cur_set ^= 1u;
            m->nfac = 0u;
            m->adapted = 1u;
            if (m->changed) m->rebuilds++;
        }
    }
}

// Sort key of a finest-grid cell: its root's id (x fastest over the base grid) above the
// Morton index of the cell inside the root (x bit lowest).  Leaves are stored in this order
// (their lower corner's key), so the leaf holding a cell is the last leaf whose key does not
// exceed the cell's: a search over 8 bytes per leaf instead of an owner map of 4 bytes per
// finest cell (2^(d L) per root).
template <int DIM>
__device__ __forceinline__ uint64_t cell_key(const Grid& g, int64_t fx, int64_t fy, int64_t fz) {
    const int L = g.L;
    const int64_t rx = fx >> L, ry = fy >> L, rz = DIM == 3 ? (fz >> L) : 0;
    const uint64_t rid = (uint64_t)(rx + g.base[0] * (ry + (int64_t)g.base[1] * rz));
    const uint32_t lx = (uint32_t)(fx - (rx << L)), ly = (uint32_t)(fy - (ry << L)),
                   lz = DIM == 3 ? (uint32_t)(fz - (rz << L)) : 0u;
    uint64_t mort = 0;
    for (int b = 0; b < L; ++b) {
        mort |= (uint64_t)((lx >> b) & 1u) << (DIM * b);
        mort |= (uint64_t)((ly >> b) & 1u) << (DIM * b + 1);
        if (DIM == 3) mort |= (uint64_t)((lz >> b) & 1u) << (DIM * b + 2);
    }
    return (rid << (DIM * L)) | mort;
}

// Exclusive offsets of the new leaves, written directly as the new coordinates, their sort keys
// and the transfer plan (0 keep, 1 child, 2 parent).  Runs after the commit: the old count is
// in ne_new.
template <int DIM>
__global__ void k_scan_emit(const int4* coord, const uint8_t* r, const uint8_t* c0, const int64_t* bsum,
                            int4* ncoord, uint64_t* lkey, Grid g, int8_t* pkind, int32_t* psrc, int8_t* pbits,
                            const DevMeta* m) {
    pdl_enter();
    if (m->err) return;
    constexpr int NC = 1 << DIM;
    __shared__ int64_t sh[32];
    const int64_t ne = m->ne_new;
    const int64_t base = (int64_t)blockIdx.x * SCAN_CHUNK;
    if (base >= ne) return;
    int v[SCAN_ITEMS];
    int64_t s = 0;
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        const int64_t e = base + (int64_t)threadIdx.x * SCAN_ITEMS + i;
        v[i] = e < ne ? new_count<DIM>(coord, r, c0, e) : 0;
        s += v[i];
    }
    int64_t tot;
    int64_t o = block_excl_scan(s, sh, &tot) + bsum[blockIdx.x];
    const bool keys = m->changed != 0;     // the mesh tables are rebuilt
    auto put = [&](int64_t i, const int4& x) {
        ncoord[i] = x;
        if (keys) {
            const int sl = g.L - x.w;
            lkey[i] = cell_key<DIM>(g, (int64_t)x.x << sl, (int64_t)x.y << sl, (int64_t)x.z << sl);
        }
    };
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        const int64_t e = base + (int64_t)threadIdx.x * SCAN_ITEMS + i;
        if (e >= ne) break;
        const int4 a = coord[e];
        if (v[i] == NC) {
            for (int b = 0; b < NC; ++b) {
                put(o + b, make_int4(2 * a.x + (b & 1), 2 * a.y + ((b >> 1) & 1),
                                     DIM == 3 ? 2 * a.z + ((b >> 2) & 1) : 0, a.w + 1));
                pkind[o + b] = 1;
                psrc[o + b] = (int32_t)e;
                pbits[o + b] = (int8_t)b;
            }
        } else if (v[i] == 1) {
            if (c0[e]) {
                put(o, make_int4(a.x >> 1, a.y >> 1, DIM == 3 ? a.z >> 1 : 0, a.w - 1));
                pkind[o] = 2;
            } else {
                put(o, a);
                pkind[o] = 0;
            }
            psrc[o] = (int32_t)e;
            pbits[o] = 0;
        }
        o += v[i];
    }
}

template <int DIM>
__global__ void k_leaf_keys(const int4* coord, uint64_t* lkey, Grid g, const DevMeta* m) {
    pdl_enter();
    if (m->err) return;
    const int64_t ne = m->ne;
    for (int64_t e = gtid(); e < ne; e += gstride()) {
        const int4 a = coord[e];
        const int sh = g.L - a.w;
        lkey[e] = cell_key<DIM>(g, (int64_t)a.x << sh, (int64_t)a.y << sh, (int64_t)a.z << sh);
    }
}

// The leaf holding the cell of key k: the last e with lkey[e] <= k (lkey[0] = 0), found by a
// galloping search from `hint` (face neighbours are mostly near in the Morton order), then
// bisection.
__device__ __forceinline__ int32_t find_leaf(const uint64_t* __restrict__ lkey, int64_t ne, int64_t hint,
                                             uint64_t k) {
    int64_t lo, hi;   // lkey[lo] <= k < lkey[hi] (hi == ne: past the end)
    if (lkey[hint] <= k) {
        lo = hint;
        hi = ne;
        for (int64_t step = 1;; step <<= 1) {
            const int64_t j = lo + step;
            if (j >= ne) break;
            if (lkey[j] <= k) {
                lo = j;
            } else {
                hi = j;
                break;
            }
        }
    } else {
        hi = hint;
        lo = 0;
        for (int64_t step = 1;; step <<= 1) {
            const int64_t j = hi - step;
            if (j <= 0) break;
            if (lkey[j] <= k) {
                lo = j;
                break;
            }
            hi = j;
        }
    }
    while (hi - lo > 1) {
        const int64_t mid = (lo + hi) >> 1;
        if (lkey[mid] <= k) lo = mid;
        else hi = mid;
    }
    return (int32_t)lo;
}

// Face tables of the mesh in `coord` from the leaf keys (same rules as the forest
// bookkeeping: neighbour at the same level, one coarser with the tangential position
// bits, or the 2^(d-1) finer children touching the face).
template <typename R, int DIM, int P>
__global__ void k_mesh_tables(const int4* coord, const uint64_t* lkey, Grid g, uint32_t* info, int32_t* nbr,
                              int32_t* hang, int32_t* root, uint32_t* loc, uint8_t* bcfl,
                              const uint8_t* class_b, uint32_t* smask0, uint32_t* smask1, uint32_t* smask2,
                              uint32_t* smask3, StimBoxes sb, Phys<double> phd, const Tables<R> T,
                              const double* lat, DevMeta* m, int force) {
    // element extents per level in FP32 for the stimulus-box pre-test below
    __shared__ float hf[8][3];
    if (threadIdx.x < 24) hf[threadIdx.x / 3][threadIdx.x % 3] = (float)phd.h[threadIdx.x / 3][threadIdx.x % 3];
    __syncthreads();
    pdl_enter();
    if (m->err || !(force || m->changed)) return;
    using S = Shape<DIM, P>;
    constexpr int N1 = S::N1, NP = S::NP, NF = S::NF, NSUB = S::NSUB;
    const int64_t ne = m->ne;
    uint32_t* smask[4] = {smask0, smask1, smask2, smask3};
    for (int64_t e = gtid(); e < ne; e += gstride()) {
        const int4 a = coord[e];
        const int l = a.w, sh = g.L - l;
        const int c[3] = {a.x, a.y, a.z};
        uint32_t inf = (uint32_t)l << 24;
        uint32_t cfg = 0;
        for (int f = 0; f < NF; ++f) {
            const int axis = f >> 1, side = (f & 1) ? 1 : -1;
            int64_t cn[3] = {c[0], c[1], DIM == 3 ? c[2] : 0};
            cn[axis] += side;
            const int64_t ncell = (int64_t)g.base[axis] << l;
            int kind = 0, pos = 0;
            int32_t nb = -1;
            if (cn[axis] >= 0 && cn[axis] < ncell) {
                int64_t fc[3];
                for (int k = 0; k < 3; ++k) fc[k] = (k < DIM) ? (cn[k] << sh) : 0;
                if (side < 0) fc[axis] = ((cn[axis] + 1) << sh) - 1;
                const int32_t o = find_leaf(lkey, ne, e, cell_key<DIM>(g, fc[0], fc[1], fc[2]));
                const int lo = coord[o].w;
                int tg[2] = {0, 0}, nt = 0;
                for (int k = 0; k < DIM; ++k)
                    if (k != axis) tg[nt++] = k;
                if (lo == l) {
                    kind = 1;
                    nb = o;
                } else if (lo != l - 1 && lo != l + 1) {
                    atomicOr(&m->err, ERR_MESH);
                } else if (lo == l - 1) {
                    kind = 2;
                    nb = o;
                    for (int t = 0; t < nt; ++t) pos |= (c[tg[t]] & 1) << t;
                } else {
                    kind = 3;
                    nb = (int32_t)((e * NF + f) * NSUB);
                    for (int b = 0; b < NSUB; ++b) {
                        int64_t ch[3] = {0, 0, 0};
                        ch[axis] = 2 * cn[axis] + (side > 0 ? 0 : 1);
                        for (int t = 0; t < nt; ++t) ch[tg[t]] = 2 * (int64_t)c[tg[t]] + ((b >> t) & 1);
                        int64_t f2[3];
                        for (int k = 0; k < 3; ++k) f2[k] = (k < DIM) ? (ch[k] << (sh - 1)) : 0;
                        hang[nb + b] = find_leaf(lkey, ne, o, cell_key<DIM>(g, f2[0], f2[1], f2[2]));
                    }
                }
            }
            inf |= (uint32_t)(kind | (pos << 2)) << (4 * f);
            cfg |= (uint32_t)kind << (2 * f);
            nbr[e * NF + f] = nb;
        }
        // probes and root
        int32_t rt[3] = {0, 0, 0};
        uint32_t lc = (uint32_t)l << 24;
        for (int k = 0; k < DIM; ++k) {
            rt[k] = c[k] >> l;
            lc |= (uint32_t)(c[k] - (rt[k] << l)) << (8 * k);
        }
        root[e] = rt[0] + g.base[0] * (rt[1] + g.base[1] * rt[2]);
        loc[e] = lc;
        bcfl[e] = class_b[(size_t)l * (1u << (2 * NF)) + cfg];
        // stimulus masks: node coordinates in FP64 without contraction (same bits as the host).
        // GL nodes lie at least 0.11 h inside the element along each axis, so an element whose
        // extent misses the box by 0.05 h (FP32 test: its rounding is below 1e-4 h) holds no
        // node of the box and skips the FP64 evaluation (a slow pipe on this part).
        bool any = false;
        for (int s = 0; s < sb.n; ++s) {
            uint32_t msk = 0;
            bool may = true;
            for (int k = 0; k < DIM; ++k) {
                const float h = hf[l][k], x0 = (float)c[k] * h;
                if (x0 + h < (float)sb.lo[s][k] - 0.05f * h || x0 > (float)sb.hi[s][k] + 0.05f * h) may = false;
            }
            for (int q = 0; may && q < NP; ++q) {
                bool in = true;
                for (int k = 0; k < DIM; ++k) {
                    const double h = phd.h[l][k];
                    const double xi = sb.xi[digit<N1>(q, k)];
                    const double x = __dadd_rn(__dmul_rn((double)c[k], h), __dmul_rn(__dmul_rn(__dadd_rn(xi, 1.0), 0.5), h));
                    if (x < sb.lo[s][k] || x > sb.hi[s][k]) in = false;
                }
                if (in) msk |= 1u << q;
            }
            smask[s][e] = msk;
            any = any || msk;
        }
        if (any) inf |= INFO_STIM;
        // probes of the leaf with no activation time yet (k_lat_refresh without marking)
        if (!force) {
            const int64_t rid = root[e];
            const int lx[3] = {(int)(lc & 255u), (int)((lc >> 8) & 255u), (int)((lc >> 16) & 255u)};
            for (int q = 0; q < NP; ++q) {
                bool inside = true;
#pragma unroll
                for (int k = 0; k < DIM; ++k) inside = inside && (T.pfl[l][digit<N1>(q, k)] == lx[k]);
                if (inside && isinf(lat[rid * NP + q])) inf |= INFO_PENDING;
            }
        }
        info[e] = inf;
    }
}

// --------------------------------------------------------------------------
// Level ordering: stable multi-split of the element ids by b descending, within a level the
// elements with regular faces before the others, with the due count of every tick (tick 0: all;
// tick i > 0: b >= B - ctz(i)).  The sweeps give a warp consecutive due elements: a hanging face
// costs up to ten times a same-level one, and in mesh order most warps near a change of level held
// one.  Bit 4 of the level byte keeps the class; key = 2 b + class.
constexpr int ORD_THREADS = 256, ORD_KEYS = 16;
constexpr uint8_t LVL_IRR = 16;

// Substep levels b_e = max(b^CFL_e, b^cell_e) (Eq. num-substeps), or the replayed levels, with the
// class bit of the ordering.
struct LevelArgs {
    const int8_t* ovr;         // replayed levels (null: the library's own)
    const double* eta_ovr;     // replayed eta^t (null: the elements' own)
    double tau_cell;
    int bcell, B, lts;
    int32_t* bcnt;             // ORD_KEYS columns: elements per key of every block of ORD_THREADS
    int stride;                // column stride of bcnt
    uint32_t fmask, fsame;     // an element is irregular where (info & fmask) != fsame
    uint8_t* r;                // refinement marks, cleared here for the next barrier (null: none)
};

template <typename R>
__device__ __forceinline__ int elem_level(const DevArrays<R>& d, const LevelArgs& a, int64_t e, double eta_t) {
    int b;
    if (a.ovr) b = a.ovr[e];
    else if (!a.lts) b = 0;
    else {
        b = d.bcfl[e];
        const int bt = ((a.eta_ovr ? a.eta_ovr[e] : eta_t) > a.tau_cell) ? a.bcell : 0;
        b = bt > b ? bt : b;
    }
    if (b > a.B || b < 0) {
        atomicOr(&d.meta->err, ERR_CFL);
        b = b < 0 ? 0 : a.B;
    }
    return b | ((d.info[e] & a.fmask) != a.fsame ? LVL_IRR : 0);
}

__device__ __forceinline__ int order_key(int lv) { return 2 * (lv & 7) + ((lv & LVL_IRR) ? 1 : 0); }

// Exclusive scan over the blocks of the per-block key counts, a warp per column (a lane takes 8
// consecutive blocks at a time), then the keys' base offsets (b descending, regular first; after
// the columns) and the due counts of every tick.
static __global__ void k_order_top(int32_t* bcnt, int stride, DevMeta* m, int B) {
    pdl_enter();
    if (threadIdx.x == 0) m->adapted = 0u;
    if (m->err) return;
    __shared__ int32_t tot[ORD_KEYS];
    const int nb = (int)((m->ne + ORD_THREADS - 1) / ORD_THREADS);
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int k = threadIdx.x >> 5; k < ORD_KEYS; k += nw) {
        int32_t carry = 0;
        int32_t* col = bcnt + (size_t)k * stride;
        for (int b0 = 0; k < 2 * (B + 1) && b0 < nb; b0 += 256) {
            const int i = b0 + 8 * lane;
            int4 v[2] = {make_int4(0, 0, 0, 0), make_int4(0, 0, 0, 0)};
            if (i < nb) {
                v[0] = reinterpret_cast<const int4*>(col + i)[0];
                v[1] = reinterpret_cast<const int4*>(col + i)[1];
            }
            int32_t x[8] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w};
            int32_t s = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                if (i + q >= nb) x[q] = 0;     // (blocks past the mesh)
                const int32_t t = x[q];
                x[q] = s;
                s += t;
            }
            int32_t sc = s;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t y = __shfl_up_sync(0xffffffffu, sc, o);
                if (lane >= o) sc += y;
            }
            const int32_t ex = carry + sc - s;
            if (i < nb) {
                reinterpret_cast<int4*>(col + i)[0] = make_int4(ex + x[0], ex + x[1], ex + x[2], ex + x[3]);
                reinterpret_cast<int4*>(col + i)[1] = make_int4(ex + x[4], ex + x[5], ex + x[6], ex + x[7]);
            }
            carry += __shfl_sync(0xffffffffu, sc, 31);
        }
        if (lane == 0) tot[k] = carry;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t off = 0;
        int32_t* lo = bcnt + (size_t)ORD_KEYS * stride;
        int32_t lev[8];
        for (int b = 7; b >= 0; --b) {
            lo[2 * b] = off;
            lo[2 * b + 1] = off + tot[2 * b];
            lev[b] = tot[2 * b] + tot[2 * b + 1];
            off += lev[b];
            m->cnt[b] = (unsigned)lev[b];
        }
        const int nt = 1 << B;
        int64_t eu = 0;
        for (int i = 0; i < nt; ++i) {
            int64_t na = 0;
            if (i == 0) na = m->ne;
            else {
                const int tz = __ffs(i) - 1;
                for (int b = B - tz; b <= B; ++b) na += lev[b];
            }
            m->nact[i] = (int32_t)na;
            eu += na;
        }
        m->elem_updates += eu;
    }
}

template <typename R>
__global__ void __launch_bounds__(ORD_THREADS) k_levels_count(const DevArrays<R> d, const LevelArgs a) {
    pdl_enter();
    __shared__ int sc[ORD_KEYS];
    if (threadIdx.x < ORD_KEYS) sc[threadIdx.x] = 0;
    __syncthreads();
    const int64_t e = (int64_t)blockIdx.x * ORD_THREADS + threadIdx.x;
    if (!d.meta->err && e < d.meta->ne) {
        const int b = elem_level<R>(d, a, e, d.eta_t[e]);
        d.lvl[e] = (uint8_t)(b | (d.lvl[e] & 8));
        atomicAdd(&sc[order_key(b)], 1);
    }
    __syncthreads();
    if (threadIdx.x < ORD_KEYS) a.bcnt[(size_t)threadIdx.x * a.stride + blockIdx.x] = sc[threadIdx.x];
}

// Solution transfer after adaptation (Alg. 1 adapt steps): keep, prolong (parent
// polynomial at the child nodes) or restrict (L2 projection with the children's GL
// rule, exact for the diagonal GL mass).  Old arrays in `o`, new in `n` (slot 0).  Kept
// elements (most of them) with rows of 27 values are copied by whole warps: a warp takes 32
// consecutive new elements and copies their rows lane-parallel over the values, the old row
// of each element broadcast from its lane; shorter rows, refined and coarsened elements take
// a thread each.  The elements' levels follow in the same pass (their eta^t is at hand), with the
// counts of the ordering.
template <typename R, int DIM, int P>
__global__ void __launch_bounds__(ORD_THREADS) k_transfer(const DevArrays<R> o, DevArrays<R> n, const int8_t* pkind,
                                                          const int32_t* psrc, const int8_t* pbits, const Tables<R> T,
                                                          const LevelArgs lev) {
    pdl_enter();
    using S = Shape<DIM, P>;
    constexpr int N1 = S::N1, NP = S::NP, NC = 1 << DIM, NPS = S::NPS;
    __shared__ int sc[ORD_KEYS];
    if (threadIdx.x < ORD_KEYS) sc[threadIdx.x] = 0;
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * ORD_THREADS + threadIdx.x;
    // (not the error word: an element without a level sets it during this kernel, and the state
    // moves to the committed mesh all the same)
    if (n.meta->adapted) {
    const int64_t nne = n.meta->ne;
    const int kd = i < nne ? pkind[i] : -1;
    const int src = i < nne ? psrc[i] : 0;
    double et = kd == 0 || kd == 1 ? o.eta_t[src] : 0.0;
    if constexpr (NP < 27) {
        // short rows (Q1, 2D Q2): a thread per kept element
        if (kd == 0) {
            const int par = (o.lvl[src] >> 3) & 1;
            R x[NP], y[NP];
            ld_dofs<R, NP, NPS>((par ? o.V1 : o.V0) + (size_t)src * NPS, x);
            ld_dofs<R, NP, NPS>(o.v + (size_t)src * NPS, y);
            st_dofs<R, NP, NPS>(n.V0 + (size_t)i * NPS, x);
            st_dofs<R, NP, NPS>(n.v + (size_t)i * NPS, y);
        }
    } else {
        const int lane = threadIdx.x & 31;
        const int64_t base = i - lane;
        if (base < nne) {
            long long vrow = 0, wrow = 0;   // old rows of a kept element (0: not kept)
            if (kd == 0) {
                const int par = (o.lvl[src] >> 3) & 1;
                vrow = (long long)((par ? o.V1 : o.V0) + (size_t)src * NPS);
                wrow = (long long)(o.v + (size_t)src * NPS);
            }
            // value idx = lane + 32 j of the warp's block of padded rows: row r = idx / NPS,
            // column q (the pad copied too); every load of the block is issued before the
            // first store
            R xv[NPS], xw[NPS];
            bool keep[NPS];
            int r = lane / NPS, q = lane - (lane / NPS) * NPS;
#pragma unroll
            for (int j = 0; j < NPS; ++j) {
                const long long vr = __shfl_sync(0xffffffffu, vrow, r);
                const long long wr = __shfl_sync(0xffffffffu, wrow, r);
                keep[j] = vr != 0;
                xv[j] = keep[j] ? reinterpret_cast<const R*>(vr)[q] : R(0);
                xw[j] = keep[j] ? reinterpret_cast<const R*>(wr)[q] : R(0);
                q += 32 % NPS;
                r += 32 / NPS;
                if (q >= NPS) {
                    q -= NPS;
                    ++r;
                }
            }
            const size_t o0 = (size_t)base * NPS + lane;
#pragma unroll
            for (int j = 0; j < NPS; ++j) {
                if (keep[j]) {
                    n.V0[o0 + 32 * j] = xv[j];
                    n.v[o0 + 32 * j] = xw[j];
                }
            }
        }
    }
    if (kd > 0) {
    R* Vn = n.V0 + (size_t)i * NPS;
    R* wn = n.v + (size_t)i * NPS;
#pragma unroll
    for (int q = NP; q < NPS; ++q) Vn[q] = wn[q] = R(0);
    if (kd == 1) {
        const int bits = pbits[i];
        const int par = (o.lvl[src] >> 3) & 1;
        const R* Vo = (par ? o.V1 : o.V0) + (size_t)src * NPS;
        const R* wo = o.v + (size_t)src * NPS;
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            R a = 0, c = 0;
            for (int j = 0; j < NP; ++j) {
                R w = R(1);
#pragma unroll
                for (int k = 0; k < DIM; ++k) w *= T.Pi[(bits >> k) & 1][digit<N1>(q, k)][digit<N1>(j, k)];
                a += w * Vo[j];
                c += w * wo[j];
            }
            Vn[q] = a;
            wn[q] = c;
        }
    } else {
        R a[NP], c[NP];
#pragma unroll
        for (int q = 0; q < NP; ++q) a[q] = c[q] = R(0);
        for (int cb = 0; cb < NC; ++cb) {
            const int ch = src + cb;
            const int par = (o.lvl[ch] >> 3) & 1;
            const R* Vo = (par ? o.V1 : o.V0) + (size_t)ch * NPS;
            const R* wo = o.v + (size_t)ch * NPS;
            et += o.eta_t[ch];
            for (int qc = 0; qc < NP; ++qc) {
                // the child's GL weight in the parent's measure; on a mapped mesh the child's
                // own GL mass (divided by the parent's below)
                R wc = R(1);
                if (o.mq) {
                    wc = (R)o.mq[(size_t)ch * NP + qc];
                } else {
#pragma unroll
                    for (int k = 0; k < DIM; ++k) wc *= T.w[digit<N1>(qc, k)] * R(0.5);
                }
                const R xv = wc * Vo[qc], xw = wc * wo[qc];
#pragma unroll
                for (int q = 0; q < NP; ++q) {
                    R w = R(1);
#pragma unroll
                    for (int k = 0; k < DIM; ++k) w *= T.Pi[(cb >> k) & 1][digit<N1>(qc, k)][digit<N1>(q, k)];
                    a[q] += w * xv;
                    c[q] += w * xw;
                }
            }
        }
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            R wq = R(1);
            if (n.mq) {
                wq = (R)n.mq[(size_t)i * NP + q];
            } else {
#pragma unroll
                for (int k = 0; k < DIM; ++k) wq *= T.w[digit<N1>(q, k)];
            }
            Vn[q] = a[q] / wq;
            wn[q] = c[q] / wq;
        }
        et /= NC;
    }
    }
    if (kd >= 0) {
        n.eta_t[i] = et;
        const int b = elem_level<R>(n, lev, i, et);
        n.lvl[i] = (uint8_t)b;
        atomicAdd(&sc[order_key(b)], 1);
    }
    if (i < nne || i < n.meta->ne_new) lev.r[i] = 0;   // (ne_new: the old mesh's count)
    }
    __syncthreads();
    if (threadIdx.x < ORD_KEYS) lev.bcnt[(size_t)threadIdx.x * lev.stride + blockIdx.x] = sc[threadIdx.x];
}

static __global__ void __launch_bounds__(ORD_THREADS) k_order_scatter(const uint8_t* lvl, const int32_t* bcnt,
                                                                      int stride, int32_t* order, const DevMeta* m) {
    pdl_enter();
    if (m->err) return;
    __shared__ int wc[ORD_THREADS / 32][ORD_KEYS];
    const int64_t ne = m->ne;
    const int64_t e = (int64_t)blockIdx.x * ORD_THREADS + threadIdx.x;
    if ((int64_t)blockIdx.x * ORD_THREADS >= ne) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const bool valid = e < ne;
    const int k = valid ? order_key(lvl[e]) : ORD_KEYS;
    const unsigned peers = __match_any_sync(0xffffffffu, k);
    const int rank = __popc(peers & ((1u << lane) - 1u));
    if (lane < ORD_KEYS) wc[w][lane] = 0;
    __syncwarp();
    if (valid && rank == 0) wc[w][k] = __popc(peers);
    __syncthreads();
    if (!valid) return;
    int woff = 0;
    for (int x = 0; x < w; ++x) woff += wc[x][k];
    const int32_t* lo = bcnt + (size_t)ORD_KEYS * stride;
    order[lo[k] + bcnt[(size_t)k * stride + blockIdx.x] + woff + rank] = (int32_t)e;
}

}  // namespace mdl
