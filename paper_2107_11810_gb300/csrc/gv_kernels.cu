// gv_kernels.cu -- kernels of the level-wise voting search (Algorithm 2 of
// arXiv 2107.11810 with canonization, Sec. 3.2, and B&B pruning, Sec. 3.3).
//
//   k_lift        root records of the original surfaces (Eq. 1 in the frame of the
//                 domain centre), snapped for level 0
//   k_prep        per cell of a chunk: pruning re-check and the change of the
//                 family's basis functions from the cell centre to each child
//                 centre (own sin/cos, FP64, from tables); per tile its cell
//   (k_count, k_emit: the proximity test itself, in gv_count.cu and gv_emit.cu)
//   k_tile_scan   per child its counts, per tile and child its records' place, best
//                 lower bound, all from the count pass's ballots
//   k_child_*     pruning, allocation of surviving children, leaf argmax as a packed
//                 64-bit atomicMax
//   k_path_geo,   replay of every original surface along one root-to-cell path:
//   k_replay      inlier mask of the best leaf and per-cell counts
#include <cstdio>
#include <map>
#include <mutex>

#include "gv_tile.cuh"

namespace gv {

__device__ __forceinline__ unsigned prune_threshold(const Problem &P, const Scalars *sc, int prune) {
    if (!prune) return 1u;
    // plain (cached) loads: every thread of a kernel reads them, and an older value is valid
    unsigned lb = sc->best_lb;
    unsigned long long bk = sc->best_key;
    unsigned leaf = (unsigned)(bk >> P.coord_bits);
    unsigned t = lb > leaf ? lb : leaf;
    return t > 1u ? t : 1u;
}

// ---------------------------------------------------------------------------
// A0 lift
// ---------------------------------------------------------------------------
// Basis of the root cell's centre (once per context).
template <int FAM>
__global__ void k_root_basis(Problem P, Level lev0, double *psi) {
    double c[Fam<FAM>::D], v[Fam<FAM>::NB];
#pragma unroll
    for (int j = 0; j < Fam<FAM>::D; ++j) c[j] = cell_center(P, lev0.h, j, 0);
    Fam<FAM>::basis(P, c, v);
#pragma unroll
    for (int m = 0; m < Fam<FAM>::NB; ++m) psi[m] = v[m];
}

// Rounds to the nearest step; bad unless below 2^30 steps (integer tests: the FP64 pipe,
// one instruction per 32 clocks and SM, bounds this kernel).
__device__ __forceinline__ int lift_q(double x, double inv_s, bool &bad) {
    const double v = dmul(x, inv_s);
    const int q = __double2int_rn(v);                // saturates
    bad |= (__double2hiint(v) & 0x7ff00000) == 0x7ff00000 || (unsigned)q + 0x3fffffffu > 0x7ffffffeu;
    return bad ? 0 : q;
}

// Root records of the surfaces.  48 bytes move per surface of a 3-DoF pose and 16 FP64
// instructions run; blocks take several surfaces per thread so that the largest |q| of
// each field (it sets the screen's band and the record formats) costs one atomic per
// block: 167 us per 1e6 surfaces with a basis per surface and an atomic per warp and
// field, 44 us now.
template <int FAM>
__global__ void __launch_bounds__(256) k_lift(Problem P, Level lev0, const double *psi0, const double *prm, int64_t n,
                                              RecView out, CellView root, Scalars *sc) {
    grid_start();
    using F = Fam<FAM>;
    constexpr int NW = rec_words(F::NFP, false), NQ = F::ND + F::LE;
    const int lane = threadIdx.x & 31;
    __shared__ unsigned s_max[NQ];
    unsigned qa[NQ];
#pragma unroll
    for (int x = 0; x < NQ; ++x) qa[x] = 0u;
    if (threadIdx.x < NQ) s_max[threadIdx.x] = 0u;
    bool bad = false;
    const int64_t first = blockIdx.x * 256ll + threadIdx.x;
    if (first == 0) {                                // the root cell holds every surface
        root.key[0] = 0ull;
        root.rbeg[0] = 0ull;
        root.rcnt[0] = root.ub[0] = (uint32_t)n;
        root.lb[0] = 0u;
    }
    double c[F::D], psi[F::NB];
#pragma unroll
    for (int j = 0; j < F::D; ++j) c[j] = cell_center(P, lev0.h, j, 0);
#pragma unroll
    for (int m = 0; m < F::NB; ++m) psi[m] = psi0[m];
    __syncthreads();
    for (int64_t i = first; i < n; i += gridDim.x * 256ll) {
        double f[F::ND], t[F::LE];
        F::lift(prm, n, i, c, psi, f, t);
        uint32_t w[NW];
#pragma unroll
        for (int x = 0; x < NW; ++x) w[x] = 0u;
#pragma unroll
        for (int x = 0; x < NQ; ++x) {
            const int q = x < F::ND ? lift_q(f[x], P.inv_s_f[x], bad) : lift_q(t[x - F::ND], lev0.inv_s_t[x - F::ND], bad);
            w[x] = (uint32_t)q;
            const unsigned aq = (unsigned)abs(q);
            qa[x] = aq > qa[x] ? aq : qa[x];
        }
        store_words<NW>(out.rec, i, w);
        if (out.mult) out.mult[i] = 1u;
        if ((i & 31) == 0) out.tile_cell[i >> 5] = 0u;
    }
#pragma unroll
    for (int x = 0; x < NQ; ++x) {
        const unsigned m = __reduce_max_sync(kFull, qa[x]);
        if (lane == 0 && m) atomicMax(&s_max[x], m);
    }
    if (bad) atomicOr(&sc->err, 1u);
    __syncthreads();
    if (threadIdx.x < NQ && s_max[threadIdx.x]) atomicMax(&sc->qmax[threadIdx.x], s_max[threadIdx.x]);
}

// ---------------------------------------------------------------------------
// A1 cell geometry: basis change from the parent centre to each child centre
// ---------------------------------------------------------------------------
template <int FAM>
__device__ __forceinline__ void child_dpsi(const Problem &P, const Level &lev, uint64_t key, int fs,
                                           const double *psi_par, double *dpsi) {
    using F = Fam<FAM>;
    if constexpr (F::LINEAR_BASIS) {
        // psi is the free coordinates themselves: their changes are the exact child shifts
#pragma unroll
        for (int m = 0; m < F::NB; ++m) {
            const bool split = (lev.split_mask >> m) & 1;
            dpsi[m] = split ? (((fs >> m) & 1) ? lev.h1[m] : -lev.h1[m]) : 0.0;
        }
        return;
    } else {
    double cch[F::D];
#pragma unroll
    for (int j = 0; j < F::K; ++j) {
        int64_t i = cell_coord(P, key, lev.l, j);
        bool split = (lev.split_mask >> j) & 1;
        int64_t ic = split ? 2 * i + ((fs >> j) & 1) : i;
        cch[j] = cell_center(P, lev.h1, j, ic);
    }
    double psi_ch[F::NB];
    F::basis(P, cch, psi_ch);
#pragma unroll
    for (int m = 0; m < F::NB; ++m) dpsi[m] = dsub(psi_ch[m], psi_par[m]);
    if constexpr (F::LINEAR_TAIL) {
        // the last basis value is the last free coordinate: its change is the exact shift
        constexpr int j = F::K - 1;
        const bool split = (lev.split_mask >> j) & 1;
        dpsi[F::NB - 1] = split ? (((fs >> j) & 1) ? lev.h1[j] : -lev.h1[j]) : 0.0;
    }
    }
}

template <int FAM>
__device__ __forceinline__ void parent_psi(const Problem &P, const Level &lev, uint64_t key, double *psi) {
    using F = Fam<FAM>;
    double cpar[F::D];
#pragma unroll
    for (int j = 0; j < F::K; ++j) cpar[j] = cell_center(P, lev.h, j, cell_coord(P, key, lev.l, j));
    if (!F::LINEAR_BASIS) F::basis(P, cpar, psi);
}

// (sin, cos) of every cell centre of an angular coordinate, by the same operations as
// Fam::basis: a cell's geometry then takes table reads and a few FP64 operations instead
// of two evaluations per child slot (the FP64 pipe issues one lane per clock and SM and
// bounded this pass: 84 % busy).
__global__ void k_sincos_table(Problem P, int j, double2 *tab, int64_t n) {
    const int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (x >= n) return;
    const int e = 63 - __clzll(x + 1);
    const int64_t i = x + 1 - (1ll << e);
    double h[GV_MAXD], sn, cs;
    h[j] = ldexp(P.W[j], -(e + 1));                  // the half-width after e splits
    vsincos(cell_center(P, h, j, i), &sn, &cs);
    tab[x] = make_double2(sn, cs);
}

// Rotation families: the rotations of the child centres that no earlier step has filled
// in.  A thread per (cell, geometry slot) claims its entry; claimed entries are complete
// at the end of the kernel.  Cells that share their rotation coordinates share them.
template <int FAM>
__global__ void __launch_bounds__(256) k_rot_fill(const __grid_constant__ Chunk c) {
    grid_start();
    const int64_t gid = blockIdx.x * 256ll + threadIdx.x;
    const Problem &P = c.P;
    const Level &lev = c.lev;
    if (gid == 0 && lev.l == 0) {                    // the root's own
        double ph[3];
        for (int j = 0; j < 3; ++j) ph[j] = cell_center(P, lev.h, j, 0);
        Fam<FAM_POSE6DOF>::rotation(P, ph, c.rot_par);
    }
    const int64_t cell = gid >> c.kg;
    if (cell >= chunk_cells(c) || c.cells.ub[c.c0 + cell] < prune_threshold(P, c.sc, c.prune)) return;
    int64_t ix[3];
    geo_coords<FAM>(c, c.cells.key[c.c0 + cell], (int)(gid & (c.ng - 1)), true, ix);
    const int64_t e = rot_entry(P, lev.l + 1, ix);
    const unsigned bit = 1u << (e & 31);
    if (c.rot_flag[e >> 5] & bit) return;
    if (atomicOr(c.rot_flag + (e >> 5), bit) & bit) return;
    double ph[3];
    for (int j = 0; j < 3; ++j) ph[j] = cell_center(P, lev.h1, j, ix[j]);
    Fam<FAM_POSE6DOF>::rotation(P, ph, c.rot_ch + 9 * e);
}

// Cells and tiles of a chunk.  Per cell whether it is still above the threshold; per
// (cell, geometry slot) the FP32 basis changes and remainders (G64 = change times a power
// of two; the screen's coefficient is the rounded change times that power), and per basis
// value the largest magnitude (rounded up), which bounds the snap's band; in plain FP64
// mode, and where there are no tables, the FP64 changes too.  Per tile its cell (-1: pruned), how many of its 32 lanes
// hold records, whether it is its cell's first or last tile, and the cell's allowance: of N
// records all but the threshold may fail a child's test.  Of cells with more than four times
// the threshold the count pass could leave a tenth untested at most: they are counted whole.
__device__ __forceinline__ void tile_info(const Chunk &c, int64_t i, unsigned thr) {
    const int64_t nt = chunk_tiles(c);
    if (i >= nt + 2) return;
    // two entries of padding: the count pass loads ahead; after an emit pass gave up its
    // tiles name no cells
    int2 ti = make_int2(-1, 0);
    if (i < nt && !(c.sc->err & kErrTimeout)) {
        const int64_t t = c.t0 + i, cell = (int64_t)c.in.tile_cell[t];
        const int cl = (int)(cell - c.in_c0);
        const unsigned N = c.in_rcnt[cell];
        const int64_t r0 = (int64_t)c.in_rbeg[cell], left = r0 + (int64_t)N - 32 * t;
        const unsigned allow = c.early && N >= thr && N / 4 <= thr && N - thr < 8u * (kAllowNone - 1u)
                                   ? (N - thr + 7u) / 8u : kAllowNone;
        const int64_t after = (left - 1) >> 5;
        ti = make_int2(c.cells.ub[c.c0 + cl] >= thr ? cl : -1,
                       (left < 32 ? (int)left : 32) | (32 * t == r0 ? kTileFirst : 0) |
                           (left <= 32 ? kTileLast : 0) |
                           (int)(after < kLeftMax ? after : kLeftMax) << kLeftShift |
                           ((N + 31u) / 32u <= (unsigned)c.early ? kTileOwned : 0) | (int)(allow << kAllowShift));
    }
    c.tinfo[i] = ti;
}

template <int FAM>
__global__ void __launch_bounds__(256) k_prep(const __grid_constant__ Chunk c) {
    grid_start();
    using F = Fam<FAM>;
    static_assert(32 % (1 << F::K) == 0, "a cell's threads must lie in one warp");
    const int64_t gid = blockIdx.x * 256ll + threadIdx.x;
    const unsigned thr = prune_threshold(c.P, c.sc, c.prune);
    const int nc = chunk_cells(c);
    if (c.dyn && nc == 0) return;                    // the chain has stopped: the last step's scratch stays
    if (gid == 0) c.sc->n_uns = c.sc->ticket = 0u;   // this step's recheck queue and tile units
    if ((gid & ~31ll) < nc) {                        // uniform: a warp's cells
        const bool live = gid < nc && c.cells.ub[c.c0 + gid] >= thr;
        if (gid < nc) c.alive[gid] = live ? 1 : 0;
        // (a cell's records and tests count whether or not the count pass leaves it early)
        const unsigned n = live ? c.in_rcnt[c.in_c0 + gid] : 0u;
        const unsigned long long r = __reduce_add_sync(kFull, n & 0xffffu) +
                                     ((unsigned long long)__reduce_add_sync(kFull, n >> 16) << 16);
        if ((gid & 31) < 2 && r) atomicAdd((gid & 31) ? &c.sc->tests : &c.sc->records, (gid & 31) ? r << c.lns : r);
    }
    for (int64_t x = gid, nch = (int64_t)nc << c.lns; x < nch; x += gridDim.x * 256ll) {
        c.crec[x] = 0u;                              // the children's counters
        c.clb[x] = 0u;
        if (c.weighted) c.cub[x] = 0u;
        if (c.early) c.cfail[x] = 0u;
    }
    tile_info(c, gid, thr);
    if (c.geo64) {
        const int64_t cell = gid >> c.kf;
        if (cell < nc) {
            const int fs = (int)(gid & (c.nfs - 1));
            double d[F::NB];
            cell_change<FAM, false>(c, c.cells.key[c.c0 + cell], fs, d);
#pragma unroll
            for (int m = 0; m < F::NB; ++m) c.geo64[((size_t)cell * c.nfs + fs) * F::NB + m] = d[m];
        }
    }
    if constexpr (F::NBG > 0) {
        const int64_t cell = gid >> c.kg;
        const int r = (int)(gid & (c.ng - 1));
        if ((gid & ~31ll) >> c.kg >= nc) return;   // uniform: this warp only has tiles
        const bool in = cell < nc && c.cells.ub[c.c0 + cell] >= thr;
        float ga[F::NBG];
#pragma unroll
        for (int x = 0; x < F::NBG; ++x) ga[x] = 0.0f;
        if (in) {
            double d[F::NBG];
            geo_change<FAM, false>(c, c.cells.key[c.c0 + cell], r, d);
            float *gh = c.geo32 + (size_t)cell * c.gf + r, *gl = c.geo32lo + (size_t)cell * F::NBG * c.ng + r;
#pragma unroll
            for (int x = 0; x < F::NBG; ++x) {
                const float h = (float)d[x];
                gh[x * c.ng] = h;
                gl[x * c.ng] = (float)dsub(d[x], (double)h);
                ga[x] = __uint_as_float(__float_as_uint(fabsf(h)) + 1u);   // at least |d|
            }
        }
        for (int o = 1; o < c.ng; o <<= 1)
#pragma unroll
            for (int x = 0; x < F::NBG; ++x) ga[x] = fmaxf(ga[x], __shfl_xor_sync(kFull, ga[x], o));
        if (in && r == 0)
#pragma unroll
            for (int x = 0; x < F::NBG; ++x) c.geo32[(size_t)cell * c.gf + F::NBG * c.ng + x] = ga[x];
    }
}

__device__ __forceinline__ unsigned long long warp_max64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(kFull, v, o);
        v = y > v ? y : v;
    }
    return v;
}

// Block-wide exclusive scan of one 64-bit value per thread (blockDim = 256).
__device__ __forceinline__ unsigned long long block_excl_scan(unsigned long long v, unsigned long long *total) {
    __shared__ unsigned long long warp_tot[8];
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[w] = x;
    __syncthreads();
    if (w == 0) {
        unsigned long long t = lane < 8 ? warp_tot[lane] : 0ull;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            unsigned long long y = __shfl_up_sync(kFull, t, o);
            if (lane >= o) t += y;
        }
        if (lane < 8) warp_tot[lane] = t;   // inclusive warp prefix
    }
    __syncthreads();
    unsigned long long before = w ? warp_tot[w - 1] : 0ull;
    *total = warp_tot[7];
    __syncthreads();
    return before + x - v;
}

// Cells and records of the blocks before this one (v[0], v[1]) and of all nb (v[2], v[3]).
__device__ __forceinline__ void block_totals(const unsigned long long *cells, const unsigned long long *recs, int nb,
                                             unsigned long long *v) {
    __shared__ unsigned long long sum[8][4];
    v[0] = v[1] = v[2] = v[3] = 0ull;
    for (int i = threadIdx.x; i < nb; i += 256) {
        const unsigned long long x = cells[i], y = recs[i];
        if (i < (int)blockIdx.x) v[0] += x, v[1] += y;
        v[2] += x;
        v[3] += y;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(kFull, v[k], o);
        if ((threadIdx.x & 31) == 0) sum[threadIdx.x >> 5][k] = v[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[k] = 0ull;
        for (int w = 0; w < 8; ++w) v[k] += sum[w][k];
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// A5 best lower bound, pruning, allocation of surviving children, leaf argmax
// ---------------------------------------------------------------------------
__device__ __forceinline__ void trace_child(const Chunk &c, uint64_t key, unsigned ub, unsigned lb) {
    const unsigned long long t = atomicAdd(&c.sc->trace_n, 1ull);
    if (t >= c.trace.cap) return;
    c.trace.level[t] = c.lev.l + 1;
    c.trace.key[t] = key;
    c.trace.ub[t] = ub;
    c.trace.lb[t] = lb;
}

// Phase A: per child of the chunk -- trace, pruning decision, leaf argmax, and
// per-block totals of surviving children and their records.
__global__ void __launch_bounds__(256) k_child_mark(Chunk c, uint32_t *keepflag, uint32_t *recn,
                                                    unsigned long long *bs_cells, unsigned long long *bs_recs) {
    grid_start();
    const Problem &P = c.P;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    const int cl = idx >> c.lns, s = idx & (c.ns - 1);
    const int nc = chunk_cells(c);
    if (blockIdx.x * 256ll >= (int64_t)nc << c.lns) return;   // uniform: a chain's grid is sized by a bound
    const bool exists = cl < nc && c.alive[cl];
    unsigned ub = 0, lb = 0, nrec = 0;
    uint64_t key = 0;
    if (exists) {
        ub = c.cub[idx];
        if (c.lb) lb = c.clb[idx];
        nrec = c.crec[idx];
        key = child_key(P, c.cells.key[c.c0 + cl], c.lev.l, expand_bits(s, c.lev.split_mask));
        if (c.trace.cap) {
            trace_child(c, key, ub, lb);
        }
    }
    unsigned thr = prune_threshold(P, c.sc, c.prune);
    bool keep = exists && ub >= thr;
    if (c.lev.leaf_children) {
        if (keep) {
            unsigned long long kmask = (1ull << P.coord_bits) - 1ull;
            unsigned long long cand = ((unsigned long long)ub << P.coord_bits) | (~key & kmask);
            atomicMax(&c.sc->best_key, cand);
        }
        return;
    }
    // a child's records start at a multiple of 32 (whole tiles)
    const unsigned slots = keep ? (nrec + 31u) & ~31u : 0u;
    if (idx < nc << c.lns) {
        keepflag[idx] = keep ? 1u : 0u;
        recn[idx] = slots;
    }
    unsigned long long tc, tr;
    block_excl_scan(keep ? 1ull : 0ull, &tc);
    block_excl_scan((unsigned long long)slots, &tr);
    if (threadIdx.x == 0) {
        bs_cells[blockIdx.x] = tc;
        bs_recs[blockIdx.x] = tr;
    }
}

// Phase B: exclusive scan of the per-block totals (one block of 256 threads).
__global__ void __launch_bounds__(256) k_scan_sums(unsigned long long *a, unsigned long long *b, int nb, Scalars *sc) {
    grid_start();
    unsigned long long ca = 0, cb = 0;
    for (int base = 0; base < nb; base += 256) {
        int i = base + threadIdx.x;
        unsigned long long va = i < nb ? a[i] : 0ull, vb = i < nb ? b[i] : 0ull;
        unsigned long long ta, tb;
        unsigned long long ea = block_excl_scan(va, &ta);
        unsigned long long eb = block_excl_scan(vb, &tb);
        if (i < nb) {
            a[i] = ca + ea;
            b[i] = cb + eb;
        }
        ca += ta;
        cb += tb;
    }
    if (threadIdx.x == 0) {
        sc->n_cells = ca;
        sc->n_recs = cb;
    }
}

// What the step stores, to the host: it polls this instead of copying and synchronising
// (4 us instead of 15 us per step).
__device__ __forceinline__ void report(LevInfo *host, long long seq, unsigned long long cells, unsigned long long recs,
                                       bool overflow) {
    if (!host) return;
    volatile LevInfo *h = host;
    h->stored_cells = (long long)cells;
    h->stored_recs = (long long)recs;
    h->overflow = overflow;
    __threadfence_system();
    h->seq = seq;
}

// What a step stores: to the next level of a chain (it runs if there was room for it and
// it is not too large) and to the host.  Returns whether there was room.
__device__ __forceinline__ bool step_room(const Chunk &c, unsigned long long cells, unsigned long long recs) {
    return !c.dyn || ((int64_t)cells <= c.cap_cells && (int64_t)recs <= c.cap_recs);
}

__device__ __forceinline__ void step_result(const Chunk &c, unsigned long long cells, unsigned long long recs) {
    const bool room = step_room(c, cells, recs), runs = room && (int64_t)recs <= c.fit_recs;
    c.sc->n_cells = cells;
    c.sc->n_recs = recs;
    if (c.dyn) {
        c.dyn->overflow = !room;
        c.dyn[1].ncells = runs ? (long long)cells : 0ll;
        c.dyn[1].nrecs = runs ? (long long)recs : 0ll;
    }
    report(c.host, c.seq, cells, recs, !room);
}

// Lays out a kept child: cell index ci, records from rb.
__device__ __forceinline__ void place_child(const Chunk &c, int idx, unsigned long long ci, unsigned long long rb) {
    const int cl = idx >> c.lns, s = idx & (c.ns - 1);
    c.next_cells.key[ci] = child_key(c.P, c.cells.key[c.c0 + cl], c.lev.l, expand_bits(s, c.lev.split_mask));
    c.next_cells.rbeg[ci] = rb;
    c.next_cells.rcnt[ci] = c.crec[idx];
    c.next_cells.ub[ci] = c.cub[idx];
    c.next_cells.lb[ci] = c.lb ? c.clb[idx] : 0u;
    c.child_idx[idx] = (int32_t)ci;
    c.cbase[idx] = rb;
    c.alive[cl] = 3;                                 // the cell has something to write (every writer stores 3)
}

// Phases A to C of a small step in one block of 256 threads: 1024 children at a time,
// four consecutive ones per thread (all their loads in flight at once).  8 us instead of 3
// + 6.5 us; as the end of the tile scan it took longer than by itself.
__global__ void __launch_bounds__(256) k_children(const __grid_constant__ Chunk c) {
    grid_start();
    const Problem &P = c.P;
    const int nch = chunk_cells(c) << c.lns;
    if (nch == 0) return;                            // the chain has stopped
    const unsigned thr = prune_threshold(P, c.sc, c.prune);
    unsigned long long cand = 0ull, cells = 0ull, recs = 0ull;
    for (int base = 0; base < nch; base += 1024) {
        const int first = base + 4 * (int)threadIdx.x;
        unsigned ub[4], nrec[4];
        bool exists[4], keep[4];
        uint64_t key[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int idx = first + k < nch ? first + k : nch - 1, cl = idx >> c.lns;
            exists[k] = c.alive[cl] && first + k < nch;
            nrec[k] = c.crec[idx];
            ub[k] = c.weighted ? c.cub[idx] : nrec[k];
            key[k] = c.cells.key[c.c0 + cl];
        }
        unsigned long long v = 0ull;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            keep[k] = exists[k] && ub[k] >= thr;
            key[k] = child_key(P, key[k], c.lev.l, expand_bits((first + k) & (c.ns - 1), c.lev.split_mask));
            if (c.trace.cap && exists[k]) trace_child(c, key[k], ub[k], c.lb ? c.clb[first + k] : 0u);
            const unsigned long long leafv =
                ((unsigned long long)ub[k] << P.coord_bits) | (~key[k] & ((1ull << P.coord_bits) - 1ull));
            if (keep[k] && leafv > cand) cand = leafv;
            // a child's records start at a whole tile
            if (keep[k]) v += (1ull << 40) + ((nrec[k] + 31u) & ~31u);
        }
        if (c.lev.leaf_children) continue;
        unsigned long long total;
        v = block_excl_scan(v, &total);
        unsigned long long ci = c.next_c0 + cells + (v >> 40), rb = c.next_r0 + recs + (v & ((1ull << 40) - 1ull));
        cells += total >> 40;
        recs += total & ((1ull << 40) - 1ull);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (first + k >= nch) break;
            // without room the host lays the children out again; nothing is written past the end
            if (keep[k] && (!c.dyn || (int64_t)ci < c.cap_cells)) place_child(c, first + k, ci, rb);
            else c.cbase[first + k] = ~0ull;
            if (keep[k]) {
                ++ci;
                rb += (nrec[k] + 31u) & ~31u;
            }
        }
    }
    if (c.lev.leaf_children) {
        cand = warp_max64(cand);
        if ((threadIdx.x & 31) == 0 && cand) atomicMax(&c.sc->best_key, cand);
    } else if (threadIdx.x == 0) {
        step_result(c, cells, recs);
    }
}

// Phase C: surviving children get consecutive cell indices and record ranges in
// (parent, slot) order; recn holds the slots (record count rounded up to 32).  With few
// blocks every block adds up the totals before its own itself (scanned = 0) and phase B
// is left out.  In a chain the first block stores the next level's sizes; when they
// exceed its room nothing is written and the step waits for the host.
__global__ void __launch_bounds__(256) k_child_write(Chunk c, const uint32_t *keepflag, const uint32_t *recn,
                                                     const unsigned long long *bs_cells,
                                                     const unsigned long long *bs_recs, int scanned) {
    grid_start();
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    const int nch = chunk_cells(c) << c.lns, nb = (nch + 255) / 256;
    if ((int)blockIdx.x >= nb) return;                   // uniform
    unsigned long long c_before, r_before;
    if (scanned) {
        c_before = bs_cells[blockIdx.x];
        r_before = bs_recs[blockIdx.x];
        if (blockIdx.x == 0 && threadIdx.x == 0) report(c.host, c.seq, c.sc->n_cells, c.sc->n_recs, false);
    } else {
        unsigned long long v[4];
        block_totals(bs_cells, bs_recs, nb, v);
        c_before = v[0];
        r_before = v[1];
        if (blockIdx.x == 0 && threadIdx.x == 0) step_result(c, v[2], v[3]);
        if (!step_room(c, v[2], v[3])) return;           // uniform
    }
    const bool in = idx < nch;
    unsigned keep = in ? keepflag[idx] : 0u;
    unsigned nrec = in ? recn[idx] : 0u;
    unsigned long long tc, tr;
    unsigned long long ec = block_excl_scan(keep, &tc);
    unsigned long long er = block_excl_scan(nrec, &tr);
    if (!in) return;
    if (!keep) {
        c.cbase[idx] = ~0ull;
        return;
    }
    place_child(c, idx, c.next_c0 + c_before + ec, c.next_r0 + r_before + er);
}

// ---------------------------------------------------------------------------
// Beam selection (the search order; any count some leaf reaches is a valid lower
// bound, Sec. 3.3, so results do not depend on it).  A selection of a level's cells
// holds about `budget` record slots, in the cells with the largest UBs or (nk = 2) half
// of them there and half in those with the largest LBs.  Of the two the UB finds the
// best leaf's ancestor on the coarse levels of pose, ray, point-set and affine searches,
// the LB on the middle levels of planes, where almost every UB is alike; with more than
// three coordinates the LB half only opens cells that need not be (6DoF 13.1 against
// 9.2 ms).
//
// k_beam_hist: record slots per UB and LB bin (64 bins per octave) and the cells with
// the largest UB and LB; its last block finds the bin at which the slots of the bins above
// reach the budget, and the share of that bin's cells that still fits.  k_beam_mark:
// selected cells (the border bin's by a hash of their keys, so the choice depends on
// nothing but the cells) and block totals; k_scan_sums (with many blocks); k_beam_write:
// the selected cells in index order, their UB in the level set to 0 (no threshold is below
// 1, so they are found pruned later and no cell is tested twice).  Of few cells, the last
// block of k_beam_hist also takes those steps.  k_beam_gather: the selected cells'
// records, copied so that one contiguous chunk holds them (a warp per tile, the owning
// cell by binary search; the copy moves at most a few tens of MB).  A 3-DoF search of 1e6
// surfaces makes 28 selections: five kernels, a clear, a copy and a synchronisation for
// each took 1.2 ms in all, 0.9 ms now.
// ---------------------------------------------------------------------------

// 64 bins per octave: the exponent and six mantissa bits of a count as a float
__device__ __forceinline__ int beam_bin(unsigned v) {
    const int b = (int)((__float_as_uint((float)v) >> 17) - (127u << 6));
    return b < 0 ? 0 : (b >= kBeamBins ? kBeamBins - 1 : b);
}

__device__ __forceinline__ unsigned beam_hash(uint64_t key) {
    key = (key ^ (key >> 31)) * 0x9E3779B97F4A7C15ull;
    key = (key ^ (key >> 29)) * 0xff51afd7ed558ccdull;
    return (unsigned)(key >> 32);
}

// Adds a value to a kernel's ticket; whether this is its last block (all 256 threads).
__device__ __forceinline__ bool last_block(unsigned *ticket, unsigned blocks) {
    __shared__ bool s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(ticket, 1u) == blocks - 1u;
        if (s_last) *ticket = 0u;                    // for the next kernel
    }
    __syncthreads();
    if (s_last) __threadfence();
    return s_last;
}

__device__ __forceinline__ void beam_pick(BeamSel *sel, unsigned long long budget) {
    // thread t owns bins [8 t', 8 t' + 8), t' counted from the top, so a prefix over the
    // threads is the slots of all higher bins
    constexpr int PER = kBeamBins / 256;
    const int top = kBeamBins - 1 - (int)threadIdx.x * PER;
    if (threadIdx.x < 2) {
        sel->top[threadIdx.x] = __ldcg(&sel->best[threadIdx.x]);
        sel->best[threadIdx.x] = 0ull;
    }
    for (int k = 0; k < 2; ++k) {
        unsigned long long v[PER], sum = 0ull, total;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            v[i] = __ldcg(&sel->hist[k][top - i]);
            sel->hist[k][top - i] = 0ull;            // for the next selection
            sum += v[i];
        }
        unsigned long long above = block_excl_scan(sum, &total);
        if (total <= budget) {
            if (threadIdx.x == 0) {
                sel->border[k] = -1;
                sel->share[k] = 0u;
            }
            continue;
        }
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            if (above <= budget && above + v[i] > budget) {
                sel->border[k] = top - i;
                sel->share[k] = (unsigned)((double)(budget - above) / (double)v[i] * 4294967295.0);
            }
            above += v[i];
        }
    }
    __syncthreads();
}

__device__ __forceinline__ bool beam_selected(const CellView &cells, int64_t i, int64_t ncells, const BeamSel *sel,
                                              int nk, unsigned thr) {
    if (i >= ncells) i = ncells - 1, thr = 0xffffffffu;
    const unsigned ub = cells.ub[i];
    const unsigned v[2] = {ub, cells.lb[i]};
    const unsigned h = beam_hash(cells.key[i]);
    bool keep = false;
    if (ub < thr) return false;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if (k >= nk || !v[k]) continue;
        const int b = beam_bin(v[k]);
        keep |= b > sel->border[k] || (b == sel->border[k] && h < sel->share[k]) ||
                (unsigned)~(unsigned)sel->top[k] == (unsigned)i;
    }
    return keep;
}

// the selected cell i as cell o of the selection, its records from r
__device__ __forceinline__ void beam_place(const CellView &cells, int64_t i, const CellView &out, uint64_t *src_rbeg,
                                           unsigned long long o, unsigned long long r) {
    out.key[o] = cells.key[i];
    out.rbeg[o] = r;
    out.rcnt[o] = cells.rcnt[i];
    out.ub[o] = cells.ub[i];
    src_rbeg[o] = cells.rbeg[i];
    cells.ub[i] = 0u;
}

// up to kBeamSmall cells are selected by the last block
constexpr int kBeamSmall = 2048;

__global__ void __launch_bounds__(256) k_beam_hist(CellView cells, int64_t ncells, BeamSel *sel, int nk, Problem P,
                                                   const Scalars *sc, unsigned long long budget, CellView out,
                                                   uint64_t *src_rbeg, LevInfo *host, long long seq) {
    grid_start();
    __shared__ unsigned long long hist[2][kBeamBins];
    for (int i = threadIdx.x; i < 2 * kBeamBins; i += 256) hist[0][i] = 0ull;
    const unsigned thr = prune_threshold(P, sc, 1);
    __syncthreads();
    unsigned long long best[2] = {0ull, 0ull};
    for (int64_t i = blockIdx.x * 256ll + threadIdx.x; i < ncells; i += gridDim.x * 256ll) {
        const unsigned ub = cells.ub[i];
        if (ub < thr) continue;
        const unsigned v[2] = {ub, cells.lb[i]};
        const unsigned long long slots = (cells.rcnt[i] + 31u) & ~31u;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (k >= nk || !v[k]) continue;
            atomicAdd(&hist[k][beam_bin(v[k])], slots);
            const unsigned long long cand = ((unsigned long long)v[k] << 32) | (unsigned)~(unsigned)i;
            best[k] = cand > best[k] ? cand : best[k];
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        best[k] = warp_max64(best[k]);
        if ((threadIdx.x & 31) == 0 && best[k]) atomicMax(&sel->best[k], best[k]);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * kBeamBins; i += 256)
        if (hist[0][i]) atomicAdd(&sel->hist[0][i], hist[0][i]);
    if (!last_block(&sel->ticket, gridDim.x)) return;
    beam_pick(sel, budget);
    if (ncells > kBeamSmall) return;
    unsigned long long tc = 0ull, tr = 0ull;
    for (int base = 0; base < (int)ncells; base += 1024) {
        const int first = base + 4 * (int)threadIdx.x;
        bool keep[4];
        unsigned slots[4];
        unsigned long long x = 0ull, total;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            keep[k] = beam_selected(cells, first + k, ncells, sel, nk, thr);
            slots[k] = keep[k] ? (cells.rcnt[first + k] + 31u) & ~31u : 0u;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (keep[k]) x += (1ull << 40) + slots[k];
        x = block_excl_scan(x, &total);
        unsigned long long o = tc + (x >> 40), r = tr + (x & ((1ull << 40) - 1ull));
        tc += total >> 40;
        tr += total & ((1ull << 40) - 1ull);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (keep[k]) {
                beam_place(cells, first + k, out, src_rbeg, o++, r);
                r += slots[k];
            }
    }
    if (threadIdx.x == 0) report(host, seq, tc, tr, false);
}

__global__ void __launch_bounds__(256) k_beam_mark(CellView cells, int64_t ncells, const BeamSel *sel, int nk, Problem P,
                                                   const Scalars *sc, unsigned long long *bs_cells,
                                                   unsigned long long *bs_recs) {
    grid_start();
    const int64_t i = blockIdx.x * 256ll + threadIdx.x;
    const bool keep = beam_selected(cells, i, ncells, sel, nk, prune_threshold(P, sc, 1));
    unsigned long long tc, tr;
    block_excl_scan(keep ? 1ull : 0ull, &tc);
    block_excl_scan(keep ? (unsigned long long)((cells.rcnt[i] + 31u) & ~31u) : 0ull, &tr);
    if (threadIdx.x == 0) {
        bs_cells[blockIdx.x] = tc;
        bs_recs[blockIdx.x] = tr;
    }
}

__global__ void __launch_bounds__(256) k_beam_write(CellView cells, int64_t ncells, const BeamSel *sel, int nk, Problem P,
                                                    const Scalars *sc, const unsigned long long *bs_cells,
                                                    const unsigned long long *bs_recs, int scanned, CellView out,
                                                    uint64_t *src_rbeg, LevInfo *host, long long seq) {
    grid_start();
    unsigned long long c_before, r_before;
    if (scanned) {
        c_before = bs_cells[blockIdx.x];
        r_before = bs_recs[blockIdx.x];
        if (blockIdx.x == 0 && threadIdx.x == 0) report(host, seq, sc->n_cells, sc->n_recs, false);
    } else {
        unsigned long long v[4];
        block_totals(bs_cells, bs_recs, (int)gridDim.x, v);
        c_before = v[0];
        r_before = v[1];
        if (blockIdx.x == 0 && threadIdx.x == 0) report(host, seq, v[2], v[3], false);
    }
    const int64_t i = blockIdx.x * 256ll + threadIdx.x;
    const bool keep = beam_selected(cells, i, ncells, sel, nk, prune_threshold(P, sc, 1));
    unsigned long long tc, tr;
    const unsigned long long ec = block_excl_scan(keep ? 1ull : 0ull, &tc);
    const unsigned long long er =
        block_excl_scan(keep ? (unsigned long long)((cells.rcnt[i] + 31u) & ~31u) : 0ull, &tr);
    if (keep) beam_place(cells, i, out, src_rbeg, c_before + ec, r_before + er);
}

// nq: 16-byte words of one tile's records
__global__ void __launch_bounds__(256) k_beam_gather(RecView in, RecView out, CellView sel, const uint64_t *src_rbeg,
                                                     int64_t ncells, int64_t ntiles, int nq) {
    grid_start();
    const int64_t t = (blockIdx.x * 256ll + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (t >= ntiles) return;
    int64_t a = 0, b = ncells;                      // last cell whose first record is at or before the tile
    while (b - a > 1) {
        const int64_t m = (a + b) >> 1;
        if ((int64_t)(sel.rbeg[m] >> 5) <= t) a = m;
        else b = m;
    }
    const int64_t ts = (int64_t)(src_rbeg[a] >> 5) + (t - (int64_t)(sel.rbeg[a] >> 5));
    const uint4 *src = reinterpret_cast<const uint4 *>(in.rec) + ts * nq;
    uint4 *dst = reinterpret_cast<uint4 *>(out.rec) + t * nq;
    for (int i = lane; i < nq; i += 32) dst[i] = src[i];
    if (out.mult) out.mult[t * 32 + lane] = in.mult[ts * 32 + lane];
    if (lane == 0) out.tile_cell[t] = (uint32_t)a;
}

// ---------------------------------------------------------------------------
// Per-tile bookkeeping of the proximity test, so that the count and emit passes
// stream their inputs with bulk copies and never chase a pointer per tile.
// ---------------------------------------------------------------------------

// Counts and output positions from the ballots.  A warp takes 32 consecutive tiles,
// one per lane, and per child slot a segmented scan over them (segments = runs of one
// cell; UB-passing records in the low half of a word, LB-passing ones in the high
// half): a tile's records get consecutive places in the child, after those of the
// run's earlier tiles.  A run that is the whole cell owns the child's counters; any
// other run reserves its places with one atomic on them.  Partial LB sums are valid
// lower bounds, and each child's last addition returns its whole sum, so the best LB
// is raised here.  W: child slots at a time (2, 4 or 8); the atomics bound this
// kernel, so those of W slots are one request, a lane per slot.  Planes, 1e6 points: 77 ms
// with a request per slot, one after the other, 39 ms now.
template <int W>
__global__ void __launch_bounds__(256) k_tile_scan(const __grid_constant__ Chunk c) {
    grid_start();
    const int lane = threadIdx.x & 31;
    const int64_t nt = chunk_tiles(c);
    const int64_t t = (blockIdx.x * 8ll + (threadIdx.x >> 5)) * 32 + lane;
    if (t - lane >= nt) return;                                          // uniform
    const int2 ti = t < nt ? c.tinfo[t] : make_int2(-1, 0);
    const int cl = ti.x >= 0 && c.early && !c.alive[ti.x] ? -1 : ti.x;   // left by the count pass: no child survives
    const int prev = __shfl_up_sync(kFull, cl, 1);
    const unsigned heads = __ballot_sync(kFull, lane == 0 || prev != cl);
    const int next = __shfl_down_sync(kFull, cl, 1);
    const unsigned tails = __ballot_sync(kFull, lane == 31 || next != cl);
    const int head = 31 - __clz(heads & ((2u << lane) - 1u));          // this lane's segment head
    const int tail = __ffs(tails & ~((1u << lane) - 1u)) - 1;          // this lane's segment tail
    const int yh = __shfl_sync(kFull, ti.y, head), yt = __shfl_sync(kFull, ti.y, tail);   // by every lane
    const bool whole = (yh & kTileFirst) && (yt & kTileLast);
    const bool last = lane == tail && cl >= 0;
    const uint32_t *bp = c.ballot + (size_t)t * c.ns, *lp = c.lballot + (size_t)t * c.ns;
    // runs that are a part of their cell: the first and the last at most
    const unsigned partial = __ballot_sync(kFull, last && !whole);
    int partial_tail[2], partial_cell[2];
    partial_tail[0] = __ffs(partial) - 1;
    partial_tail[1] = __ffs(partial & (partial - 1u)) - 1;
#pragma unroll
    for (int k = 0; k < 2; ++k) partial_cell[k] = __shfl_sync(kFull, cl, partial_tail[k] & 31);
    unsigned best = 0;
#pragma unroll 1
    for (int s0 = 0; s0 < c.ns; s0 += W) {
        unsigned bw[W], lw[W], x[W], base[W];
#pragma unroll
        for (int q = 0; q < W; ++q) bw[q] = lw[q] = base[q] = 0u;
        if (cl >= 0) {
            load_row<W>(bp + s0, bw);
            if (c.lb) load_row<W>(lp + s0, lw);
        }
#pragma unroll
        for (int q = 0; q < W; ++q) {
            x[q] = (unsigned)__popc(bw[q]) | ((unsigned)__popc(lw[q]) << 16);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(kFull, x[q], o);
                if (lane - o >= head) x[q] += y;
            }
        }
        if (last && whole) {
            uint32_t *cr = c.crec + (size_t)cl * c.ns + s0, *cb = c.clb + (size_t)cl * c.ns + s0;
#pragma unroll
            for (int q = 0; q < W; ++q) {
                cr[q] = x[q] & 0xffffu;
                if (c.lb) cb[q] = x[q] >> 16;
                best = x[q] >> 16 > best ? x[q] >> 16 : best;
            }
        }
        // the first and the last run: lane q adds slot q's total, one request for all slots
        unsigned part[2] = {0u, 0u};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (partial_tail[k] < 0) continue;                          // uniform
            unsigned v = 0u;
#pragma unroll
            for (int q = 0; q < W; ++q) {
                const unsigned y = __shfl_sync(kFull, x[q], partial_tail[k]);
                if (lane == q) v = y;
            }
            const size_t i = (size_t)partial_cell[k] * c.ns + s0 + lane;
            if (v & 0xffffu) part[k] = atomicAdd(c.crec + i, v & 0xffffu);
            if (v >> 16) {
                const unsigned lb = (v >> 16) + atomicAdd(c.clb + i, v >> 16);
                best = lb > best ? lb : best;
            }
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (partial_tail[k] < 0) continue;                          // uniform
#pragma unroll
            for (int q = 0; q < W; ++q) {
                const unsigned y = __shfl_sync(kFull, part[k], q);
                if (tail == partial_tail[k]) base[q] = y;
            }
        }
        unsigned of[W];
#pragma unroll
        for (int q = 0; q < W; ++q)
            of[q] = base[q] + (x[q] & 0xffffu) - (unsigned)__popc(bw[q]);
        if (t < nt) store_row<W>(c.off + (size_t)t * c.ns + s0, of);
    }
    best = __reduce_max_sync(kFull, best);
    if (lane == 0 && best > *(volatile unsigned *)&c.sc->best_lb) atomicMax(&c.sc->best_lb, best);
}

// The same with multiplicities (grouping): a warp per tile.
__global__ void __launch_bounds__(256) k_tile_scan_weighted(const __grid_constant__ Chunk c) {
    grid_start();
    const int lane = threadIdx.x & 31;
    const int64_t nt = chunk_tiles(c);
    const int64_t t = blockIdx.x * 8ll + (threadIdx.x >> 5);
    if (t >= nt) return;                                                 // uniform
    const int2 ti = c.tinfo[t];
    if (ti.x < 0) return;                                                // uniform
    const uint32_t mult = lane < (ti.y & 63) ? c.in.mult[(c.t0 + t) * 32 + lane] : 0u;
    unsigned best = 0;
    for (int s = 0; s < c.ns; ++s) {
        const size_t i = (size_t)ti.x * c.ns + s;
        const unsigned b = c.ballot[(size_t)t * c.ns + s], l = c.lb ? c.lballot[(size_t)t * c.ns + s] : 0u;
        const unsigned ub = __reduce_add_sync(kFull, (b >> lane) & 1u ? mult : 0u);
        unsigned lb = __reduce_add_sync(kFull, (l >> lane) & 1u ? mult : 0u);
        if (lane == 0) {
            c.off[(size_t)t * c.ns + s] = b ? atomicAdd(c.crec + i, (unsigned)__popc(b)) : 0u;
            if (ub) atomicAdd(c.cub + i, ub);
            if (lb) lb += atomicAdd(c.clb + i, lb);
            best = lb > best ? lb : best;
        }
    }
    if (lane == 0 && best) atomicMax(&c.sc->best_lb, best);
}

// ---------------------------------------------------------------------------
// A7 replay of the original surfaces along one root-to-cell path
// ---------------------------------------------------------------------------
// path[0, lam): child slot and basis change of each step; then, for the replay's screen,
// path[lam].dpsi: the whole path's basis change; [lam + 1]: the root's basis; [lam + 2]: the
// whole shift of each coordinate; [lam + 3]: s_t of the root's level over that of the last.
template <int FAM>
__global__ void __launch_bounds__(64) k_path_geo(Problem P, const Level *levs, int lam, uint64_t key,
                                                 const Scalars *sc, PathStep *path) {
    grid_start();
    using F = Fam<FAM>;
    const int l = threadIdx.x;
    if (sc) key = ~sc->best_key & ((1ull << P.coord_bits) - 1ull);   // the best leaf
    if (l < lam) {
        const Level &lev = levs[l];
        int slot = 0;
        for (int j = 0; j < F::D; ++j)
            if (l < P.Lj[j]) slot |= (int)(cell_coord(P, key, l + 1, j) & 1) << j;
        double psi_par[F::NB], dpsi[F::NB];
        parent_psi<FAM>(P, lev, key, psi_par);
        child_dpsi<FAM>(P, lev, key, slot & ((1 << F::K) - 1), psi_par, dpsi);
        path[l].slot = slot;
#pragma unroll
        for (int m = 0; m < F::NB; ++m) path[l].dpsi[m] = dpsi[m];
    } else if (l == 63) {
        double c[F::D], psi[F::NB];
#pragma unroll
        for (int j = 0; j < F::D; ++j) c[j] = cell_center(P, levs[0].h, j, 0);
        F::basis(P, c, psi);
#pragma unroll
        for (int m = 0; m < F::NB; ++m) path[lam + 1].dpsi[m] = psi[m];
    }
    __syncthreads();
    if (l < F::NB) {
        double v = 0.0;
        for (int x = 0; x < lam; ++x) v = dadd(v, path[x].dpsi[l]);
        path[lam].dpsi[l] = v;
    } else if (l >= 16 && l < 16 + F::D) {
        double v = 0.0;
        for (int x = 0; x < lam; ++x) {
            const Level &lev = levs[x];
            const double h = lev.h1[l - 16];
            if ((lev.split_mask >> (l - 16)) & 1) v = dadd(v, (path[x].slot >> (l - 16)) & 1 ? h : -h);
        }
        path[lam + 2].dpsi[l - 16] = v;
    } else if (l >= 32 && l < 32 + F::LE) {
        path[lam + 3].dpsi[l - 32] = dmul(levs[0].s_t[l - 32], levs[lam - 1].inv_s_t[l - 32]);
    }
}

// Screen of the replay: whether a surface certainly fails the last step's test.  Its
// residual at the target cell's centre is taken from the root in one jump, without
// snapping: the steps' residual differs from it by at most the accumulated canonization
// error A.  The radius contains A once, so that no surface within reach is missed; a surface
// beyond reach can pass the steps' test by it once more, so the screen's limit is the radius
// plus A.  The essential parameters differ by at most one step of the last level (half of
// each grid they are snapped to on the way).  The FP64 rounding of either way is far below
// one snap step (fields below 2^30 steps), that of the FP32 radius and conversions below
// the 1e-4 added.
template <int FAM>
__device__ __forceinline__ bool replay_far(const Problem &P, const Level &lev, const PathStep *tail, const double *f,
                                           const double *t) {
    using F = Fam<FAM>;
    double fo[F::ND], sh[F::D], dpsi[F::NB];
#pragma unroll
    for (int m = 0; m < F::NB; ++m) dpsi[m] = tail[0].dpsi[m];
#pragma unroll
    for (int j = 0; j < F::D; ++j) sh[j] = tail[2].dpsi[j];
    F::residual64(f, t, dpsi, sh, fo);
    bool in = true, far = false;                     // in: the fields are in range (always, in a search)
    float qt[F::LE], R[F::ND];
#pragma unroll
    for (int m = 0; m < F::LE; ++m) {
        const float ratio = (float)tail[3].dpsi[m], x = fabsf((float)t[m] * (float)lev.inv_s_t[m]);
        in &= x < 1073741824.0f * ratio;
        qt[m] = x + 1.5f;
    }
    F::radius32(lev, qt, R);
#pragma unroll
    for (int j = 0; j < F::ND; ++j) {
        const float s = (float)P.inv_s_f[j];
        in &= fabsf((float)f[j] * s) < 1073741824.0f;
        far |= fabsf((float)fo[j] * s) > __fmaf_rn(__fmaf_rn((float)lev.A1[j], s, R[j]), 1.0001f, 2.0f);
    }
    return in && far;
}

// Which surfaces pass every test from the root to the target cell.  Nearly all fail, most
// of them at once: a block screens its surfaces first (30 FP64 instructions each) and only
// those that may pass go through the steps (50 FP64 instructions per step, the FP64 pipe's
// rate is the bound), collected so that warps are full.  1e6 surfaces of a 3-DoF pose, 10
// steps: 621 us with every surface through the steps until it fails, 120 us now.
// per: surfaces per block, a multiple of 32; at most 1024, fewer when the chip would be
// idle otherwise (the steps of 1024 surfaces on one SM take 40 us).
template <int FAM>
__global__ void __launch_bounds__(256) k_replay(Problem P, const Level *levs, const PathStep *path, int lam,
                                                const double *prm, int64_t n, int per, uint32_t *reach, Scalars *sc) {
    grid_start();
    using F = Fam<FAM>;
    constexpr int NS = 1024;
    __shared__ unsigned s_words[NS / 32], s_n, s_lb;
    __shared__ unsigned short s_list[NS];
    const int64_t base = (int64_t)blockIdx.x * per, left = n - base;
    const int share = left < per ? (int)left : per;
    const int lane = threadIdx.x & 31;
    const PathStep *tail = path + lam;
    if (threadIdx.x < NS / 32) s_words[threadIdx.x] = 0u;
    if (threadIdx.x == 0) s_n = s_lb = 0u;
    double c[F::D], psi[F::NB], f[F::ND], t[F::LE];
    if (lam > 0) {
#pragma unroll
        for (int j = 0; j < F::D; ++j) c[j] = cell_center(P, levs[0].h, j, 0);
#pragma unroll
        for (int m = 0; m < F::NB; ++m) psi[m] = tail[1].dpsi[m];
    }
    __syncthreads();
#pragma unroll 1
    for (int x0 = 0; x0 < share; x0 += 256) {
        const int x = x0 + threadIdx.x;
        bool maybe = x < share;
        if (maybe && lam > 0) {
            F::lift(prm, n, base + x, c, psi, f, t);
            maybe = !replay_far<FAM>(P, levs[lam - 1], tail, f, t);
        }
        const unsigned b = __ballot_sync(kFull, maybe);
        unsigned at = 0;
        if (lane == 0 && b) at = atomicAdd(&s_n, __popc(b));
        at = __shfl_sync(kFull, at, 0);
        if (maybe) s_list[at + __popc(b & ((1u << lane) - 1u))] = (unsigned short)x;
    }
    __syncthreads();
#pragma unroll 1
    for (unsigned q = threadIdx.x; q < s_n; q += 256) {
        const int x = s_list[q];
        bool reached = true, lbp = false;
        if (lam > 0) F::lift(prm, n, base + x, c, psi, f, t);
        for (int l = 0; l < lam; ++l) {
            const Level &lev = levs[l];
#pragma unroll
            for (int j = 0; j < F::ND; ++j) f[j] = dmul(rint(dmul(f[j], P.inv_s_f[j])), P.s_f[j]);
#pragma unroll
            for (int m = 0; m < F::LE; ++m) t[m] = dmul(rint(dmul(t[m], lev.inv_s_t[m])), lev.s_t[m]);
            double R[F::ND], fo[F::ND];
            radius64<FAM>(lev, t, R);
            int res = test64<FAM>(lev, f, t, R, path[l].dpsi, path[l].slot, fo);
            if (!(res & 1)) {
                reached = false;
                break;
            }
            if (l == lam - 1) lbp = (res >> 1) & 1;
#pragma unroll
            for (int j = 0; j < F::ND; ++j) f[j] = fo[j];
        }
        if (reached) atomicOr(&s_words[x >> 5], 1u << (x & 31));
        if (lbp) atomicAdd(&s_lb, 1u);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        static_assert(NS / 32 == 32, "a mask word per lane");
        const unsigned w = s_words[lane];
        if (reach && 32 * lane < share) reach[(base >> 5) + lane] = w;
        const unsigned total = __reduce_add_sync(kFull, (unsigned)__popc(w));
        if (lane == 0 && total) atomicAdd(&sc->replay_ub, (unsigned long long)total);
        if (lane == 0 && s_lb) atomicAdd(&sc->replay_lb, (unsigned long long)s_lb);
    }
}

// ---------------------------------------------------------------------------
// A3 grouping: merge records of a chunk with equal (cell, q_f, q_t) (the
// canonization's grouping, Sec. 3.2).  An open-addressing table of record
// indices: each record claims its home slot by atomicCAS of (its index + 1); a
// record that finds the slot taken compares its full key with the owner's
// (immutable) record and either adopts it or probes on.  Exact: different keys
// are never merged.  Canonical records are then laid out per cell (scan of
// per-cell counts) and their multiplicities summed with integer atomics, so the
// grouped records are deterministic up to their order inside a cell.
// ---------------------------------------------------------------------------
// A record slot of the chunk: its chunk-local cell, or -1 for the padding after a
// cell's last record.
__device__ __forceinline__ int slot_cell(const Chunk &c, int64_t r) {
    if (c.sc->err & kErrTimeout) return -1;          // an emit pass gave up: its tiles name no cells
    int64_t cell = (int64_t)c.in.tile_cell[r >> 5];
    int cl = (int)(cell - c.in_c0);
    return r < (int64_t)c.in_rbeg[cell] + (int64_t)c.in_rcnt[cell] ? cl : -1;
}

template <int NW>
__device__ __forceinline__ uint64_t key_hash(int cl, const uint32_t *w) {
    uint64_t h = 0x9E3779B97F4A7C15ull ^ (uint32_t)cl;
#pragma unroll
    for (int i = 0; i < NW; ++i) h = (h ^ w[i]) * 0xff51afd7ed558ccdull;
    return h ^ (h >> 29);
}

template <int FAM, bool Q16>
__global__ void k_group_insert(Chunk c, uint32_t *table, uint32_t tmask, uint32_t *owner, uint32_t *ccount) {
    constexpr int NW = rec_words(Fam<FAM>::NFP, Q16);
    const int64_t nr = (c.t1 - c.t0) * 32;
    int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (x >= nr) return;
    const int64_t r = c.t0 * 32 + x;
    const int cl = slot_cell(c, r);
    if (cl < 0) {
        owner[x] = 0xffffffffu;
        return;
    }
    uint32_t w[NW];
    load_words<NW>(c.in.rec, r, w);
    uint32_t slot = (uint32_t)key_hash<NW>(cl, w) & tmask;
    for (uint32_t probe = 0; probe <= tmask; ++probe) {
        uint32_t prev = atomicCAS(&table[slot], 0u, (uint32_t)(x + 1));
        if (prev == 0u) {                                   // new canonical record
            owner[x] = (uint32_t)x;
            atomicAdd(&ccount[cl], 1u);
            return;
        }
        const int64_t r2 = c.t0 * 32 + (int64_t)(prev - 1);
        bool same = slot_cell(c, r2) == cl;
        if (same) {
            uint32_t w2[NW];
            load_words<NW>(c.in.rec, r2, w2);
#pragma unroll
            for (int i = 0; i < NW; ++i) same &= w2[i] == w[i];
        }
        if (same) {
            owner[x] = prev - 1;
            return;
        }
        slot = (slot + 1) & tmask;
    }
    atomicOr(&c.sc->err, 4u);                               // table full (cannot happen at load <= 1/2)
    owner[x] = (uint32_t)x;
}

// exclusive scan of per-cell record counts rounded up to whole tiles (one block of
// 256 threads): start[i]; total[0] = slots used, total[1] = sum of cnt, total[2] =
// sum of in_cnt (the cells' record counts before grouping)
__global__ void __launch_bounds__(256) k_scan_slots(const uint32_t *cnt, const uint32_t *in_cnt, uint64_t *start,
                                                    int64_t n, unsigned long long *total) {
    unsigned long long carry = 0, recs = 0, recs_in = 0;
    for (int64_t base = 0; base < n; base += 256) {
        int64_t i = base + threadIdx.x;
        unsigned long long v = i < n ? (cnt[i] + 31u) & ~31u : 0u, t;
        unsigned long long e = block_excl_scan(v, &t);
        if (i < n) start[i] = carry + e;
        carry += t;
        if (i < n) {
            recs += cnt[i];
            recs_in += in_cnt[i];
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        recs += __shfl_xor_sync(0xffffffffu, recs, o);
        recs_in += __shfl_xor_sync(0xffffffffu, recs_in, o);
    }
    __shared__ unsigned long long s_r[8], s_ri[8];
    if ((threadIdx.x & 31) == 0) {
        s_r[threadIdx.x >> 5] = recs;
        s_ri[threadIdx.x >> 5] = recs_in;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long a = 0, b = 0;
        for (int w = 0; w < 8; ++w) a += s_r[w], b += s_ri[w];
        total[0] = carry;
        total[1] = a;
        total[2] = b;
    }
}

template <int FAM, bool Q16>
__global__ void k_group_place(Chunk c, const uint32_t *owner, const uint64_t *grbeg, uint32_t *ccur,
                              uint32_t *newpos, RecView out) {
    constexpr int NW = rec_words(Fam<FAM>::NFP, Q16);
    const int64_t nr = (c.t1 - c.t0) * 32;
    int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (x >= nr || owner[x] != (uint32_t)x) return;
    const int64_t r = c.t0 * 32 + x;
    const int cl = slot_cell(c, r);
    const uint64_t pos = grbeg[cl] + atomicAdd(&ccur[cl], 1u);
    newpos[x] = (uint32_t)pos;
    uint32_t w[NW];
    load_words<NW>(c.in.rec, r, w);
    store_words<NW>(out.rec, (int64_t)pos, w);
    out.mult[pos] = 0u;
    if ((pos & 31u) == 0) out.tile_cell[pos >> 5] = (uint32_t)cl;
}

__global__ void k_group_mult(Chunk c, const uint32_t *owner, const uint32_t *newpos, RecView out) {
    const int64_t nr = (c.t1 - c.t0) * 32;
    int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (x >= nr || owner[x] == 0xffffffffu) return;
    atomicAdd(&out.mult[newpos[owner[x]]], c.in.mult ? c.in.mult[c.t0 * 32 + x] : 1u);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static inline unsigned blocks_for(int64_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

#define GV_DISPATCH(fam, CALL)                                      \
    switch (fam) {                                                  \
    case FAM_LINE2D: { constexpr int FAMV = FAM_LINE2D; CALL; } break;           \
    case FAM_PLANE3D_SPH: { constexpr int FAMV = FAM_PLANE3D_SPH; CALL; } break; \
    case FAM_POSE3DOF: { constexpr int FAMV = FAM_POSE3DOF; CALL; } break;       \
    case FAM_RAYS3D: { constexpr int FAMV = FAM_RAYS3D; CALL; } break;           \
    case FAM_POSE6DOF: { constexpr int FAMV = FAM_POSE6DOF; CALL; } break;       \
    case FAM_POINTSET2D: { constexpr int FAMV = FAM_POINTSET2D; CALL; } break;   \
    case FAM_AFFINE4D: { constexpr int FAMV = FAM_AFFINE4D; CALL; } break;       \
    case FAM_RADIAL5DOF: { constexpr int FAMV = FAM_RADIAL5DOF; CALL; } break;   \
    default: break;                                                 \
    }

void launch_root_basis(const Problem &P, const Level &lev0, double *psi, cudaStream_t st) {
    GV_DISPATCH(P.fam, (k_root_basis<FAMV><<<1, 1, 0, st>>>(P, lev0, psi)));
}

void launch_lift(const Problem &P, const Level &lev0, const double *psi0, const double *prm, int64_t n, RecView out,
                 CellView root, Scalars *sc, cudaStream_t st) {
    if (n <= 0) return;
    const unsigned nb = blocks_for(n, 256), g = 4u * (unsigned)sm_count();
    GV_DISPATCH(P.fam, (launch(k_lift<FAMV>, nb < g ? nb : g, 256, 0, st, P, lev0, psi0, prm, n, out, root, sc)));
}

void launch_sincos_table(const Problem &P, int j, double2 *tab, cudaStream_t st) {
    const int64_t n = ((int64_t)2 << P.Lj[j]) - 1;
    k_sincos_table<<<blocks_for(n, 128), 128, 0, st>>>(P, j, tab, n);
}

int launch_prep(const Chunk &c, cudaStream_t st) {
    int n = 1;
    const int64_t geo = (int64_t)c.nc << (c.geo64 ? c.kf : c.kg);
    if (c.rot_ch) {                                  // rotation families only
        const unsigned g = blocks_for((int64_t)c.nc << c.kg, 256);
        if (c.P.fam == FAM_POSE6DOF) launch(k_rot_fill<FAM_POSE6DOF>, g, 256, 0, st, c);
        else launch(k_rot_fill<FAM_RADIAL5DOF>, g, 256, 0, st, c);
        n = 2;
    }
    const int64_t nt = c.t1 - c.t0 + 2, g = nt > geo ? nt : geo;
    GV_DISPATCH(c.P.fam, (launch(k_prep<FAMV>, blocks_for(g, 256), 256, 0, st, c)));
    return n;
}

int sm_count() {
    static const int sms = [] {
        int dev = 0, n = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        return n > 0 ? n : 1;
    }();
    return sms;
}

// Persistent grid: as many blocks as fit on the device at once (the kernel's
// occupancy at its shared memory), at most one per group.  The occupancy of each
// kernel is looked up once.
void launch_persistent(const void *kern, size_t smem, int64_t groups, const Chunk &c, cudaStream_t st) {
    static std::mutex mu;
    static std::map<std::pair<const void *, size_t>, int> occ;
    int per_sm = 0;
    {
        std::lock_guard<std::mutex> lock(mu);
        auto it = occ.find({kern, smem});
        if (it == occ.end()) {
            if (smem > 48 * 1024) cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 256, smem) != cudaSuccess || per_sm < 1)
                per_sm = 1;
            occ[{kern, smem}] = per_sm;
        } else {
            per_sm = it->second;
        }
    }
    int64_t g = (int64_t)sm_count() * per_sm;
    if (g > groups) g = groups;
    void *args[] = {(void *)&c};
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = launch_config((unsigned)g, 256, smem, st, &attr);
    cudaLaunchKernelExC(&cfg, kern, args);
}

void launch_tile_scan(const Chunk &c, cudaStream_t st) {
    const int64_t nt = c.t1 - c.t0;
    if (nt <= 0) return;
    if (c.in.mult) launch(k_tile_scan_weighted, blocks_for(nt, 8), 256, 0, st, c);
    else if (c.ns == 2) launch(k_tile_scan<2>, blocks_for(nt, 256), 256, 0, st, c);
    else if (c.ns == 4) launch(k_tile_scan<4>, blocks_for(nt, 256), 256, 0, st, c);
    else launch(k_tile_scan<8>, blocks_for(nt, 256), 256, 0, st, c);
}

__global__ void k_chain_start(LevInfo *info, long long cells, long long recs) {
    grid_start();
    info->ncells = cells;
    info->nrecs = recs;
    info->overflow = 0;
}

void launch_chain_start(LevInfo *info, int64_t cells, int64_t recs, cudaStream_t st) {
    launch(k_chain_start, 1, 1, 0, st, info, cells, recs);
}

// blocks up to which k_child_write adds up the block totals itself (each block reads all
// of them: 2 us saved by one launch less; at 4096 blocks it would cost more)
constexpr unsigned kSelfScan = 512;

int launch_child_alloc(const Chunk &c, bool small, uint32_t *keepflag, uint32_t *recn, unsigned long long *bsums,
                       cudaStream_t st) {
    const int64_t n = (int64_t)c.nc << c.lns;
    if (n <= 0) return 0;
    if (small) {
        launch(k_children, 1, 256, 0, st, c);
        return 1;
    }
    unsigned nb = blocks_for(n, 256);
    unsigned long long *ba = bsums, *bb = bsums + nb;
    launch(k_child_mark, nb, 256, 0, st, c, keepflag, recn, ba, bb);
    if (c.lev.leaf_children) return 1;
    if (!c.dyn && nb > kSelfScan) {
        launch(k_scan_sums, 1, 256, 0, st, ba, bb, (int)nb, c.sc);
        launch(k_child_write, nb, 256, 0, st, c, keepflag, recn, ba, bb, 1);
        return 3;
    }
    launch(k_child_write, nb, 256, 0, st, c, keepflag, recn, ba, bb, 0);
    return 2;
}

int launch_beam_select(const Problem &P, const CellView &cells, int64_t ncells, int64_t budget, int nk, BeamSel *sel,
                       unsigned long long *bsums, const CellView &out, uint64_t *src_rbeg, Scalars *sc, LevInfo *host,
                       long long seq, cudaStream_t st) {
    const unsigned nb = blocks_for(ncells, 256);
    unsigned long long *ba = bsums, *bb = bsums + nb;
    launch(k_beam_hist, nb < 1024u ? nb : 1024u, 256, 0, st, cells, ncells, sel, nk, P, sc, (unsigned long long)budget / nk,
           out, src_rbeg, host, seq);
    if (ncells <= kBeamSmall) return 1;
    launch(k_beam_mark, nb, 256, 0, st, cells, ncells, sel, nk, P, sc, ba, bb);
    const int scanned = nb > kSelfScan;
    if (scanned) launch(k_scan_sums, 1, 256, 0, st, ba, bb, (int)nb, sc);
    launch(k_beam_write, nb, 256, 0, st, cells, ncells, sel, nk, P, sc, ba, bb, scanned, out, src_rbeg, host, seq);
    return 3 + scanned;
}

void launch_beam_gather(const RecView &in, const RecView &out, const CellView &sel, const uint64_t *src_rbeg,
                        int64_t ncells, int64_t ntiles, int rec_bytes, cudaStream_t st) {
    if (ntiles > 0)
        launch(k_beam_gather, blocks_for(ntiles * 32, 256), 256, 0, st, in, out, sel, src_rbeg, ncells, ntiles,
                                                                    32 * rec_bytes / 16);
}

void launch_group(const Chunk &c, uint32_t *table, uint32_t tmask, uint32_t *owner, uint32_t *ccount,
                  uint32_t *ccur, uint32_t *newpos, uint64_t *grbeg, unsigned long long *total, RecView out,
                  cudaStream_t st) {
    const int64_t nr = (c.t1 - c.t0) * 32;
    if (nr <= 0) return;
    unsigned g = blocks_for(nr, 256);
    if (c.lev.q16) {
        GV_DISPATCH(c.P.fam, (k_group_insert<FAMV, true><<<g, 256, 0, st>>>(c, table, tmask, owner, ccount)));
    } else {
        GV_DISPATCH(c.P.fam, (k_group_insert<FAMV, false><<<g, 256, 0, st>>>(c, table, tmask, owner, ccount)));
    }
    k_scan_slots<<<1, 256, 0, st>>>(ccount, c.in_rcnt + c.in_c0, grbeg, c.nc, total);
    if (c.lev.q16) {
        GV_DISPATCH(c.P.fam, (k_group_place<FAMV, true><<<g, 256, 0, st>>>(c, owner, grbeg, ccur, newpos, out)));
    } else {
        GV_DISPATCH(c.P.fam, (k_group_place<FAMV, false><<<g, 256, 0, st>>>(c, owner, grbeg, ccur, newpos, out)));
    }
    k_group_mult<<<g, 256, 0, st>>>(c, owner, newpos, out);
}

void launch_path_geo(const Problem &P, const Level *levs_dev, int lam, uint64_t key, const Scalars *sc, PathStep *path,
                     cudaStream_t st) {
    if (lam <= 0) return;
    GV_DISPATCH(P.fam, (launch(k_path_geo<FAMV>, 1, 64, 0, st, P, levs_dev, lam, key, sc, path)));
}

void launch_replay(const Problem &P, const Level *levs_dev, const PathStep *path, int lam, const double *prm,
                   int64_t n, uint32_t *reach, Scalars *sc, cudaStream_t st) {
    if (n <= 0) return;
    const int64_t share = (n + 2 * sm_count() - 1) / (2 * sm_count());
    const int per = share >= 1024 ? 1024 : (int)((share + 31) & ~31);
    GV_DISPATCH(P.fam, (launch(k_replay<FAMV>, blocks_for(n, per), 256, 0, st, P, levs_dev, path, lam, prm, n, per,
                                                                            reach, sc)));
}

}  // namespace gv
