// gv_count.cu -- count pass of the proximity test (Algorithm 2's per-sub-box
// selection with the surface-box test of Sec. 3.2) for families with at most 8
// children: for every record of a chunk and every child of its cell, the UB test
// (|residual| <= eps + cell radius + Lipschitz term + accumulated canonization error)
// and, where lower bounds are wanted, the LB test (|residual| <= eps - accumulated
// error); per tile and child the ballot of passing lanes.  Counts and output positions
// come from the ballots (k_tile_scan); undecided records are queued for the FP64
// definition (k_recheck).
//
// The pass is bound by instruction issue (its records take a tenth of the DRAM rate), so
// it is built for few instructions per (tile, child): only children that exist are
// tested (a kernel per split mask); residuals, shifts and squared comparisons of two
// children go through the packed FP32 operations; a decision costs half a packed
// multiply-add, one compare and one ballot, and the band of a record is checked once,
// from the smallest |y^2 - R^2| of its children.  Records are read with plain coalesced
// loads one tile ahead, so nothing waits at a block barrier.
//
// Cells are left as soon as no child can reach the threshold (CellWatch).  Staging the
// ballots and the batches for that cost 10 to 15 % of a pass that leaves no cell (unrolled
// batches as much: their registers spill); planes of 1e6 points: 237 -> 193 ms of count
// passes (35 % of the records are not tested), of 1e4 points 7.7 -> 6.3.
#include "gv_tile.cuh"

namespace gv {

// KF: free coordinates that split, DM: dependent coordinates that split (bit mask).
// Warps take units of consecutive tiles (the cell's coefficients are spread from one register
// per lane only when the cell changes).  Loads run one tile ahead of the tests and tile
// information two: records and tile information are padded past their ends, so the loop has
// no boundary case.
template <int FAM, bool Q16, int KF, int DM, bool LB>
__global__ void __launch_bounds__(256, 4) k_count(const __grid_constant__ Chunk c) {
    grid_start();
    using F = Fam<FAM>;
    constexpr int ND = F::ND, LE = F::LE, NFS = 1 << KF, NS = NFS * dep_slots(DM), NP = (NFS + 1) / 2;
    constexpr int NW = rec_words(F::NFP, Q16), NG = F::NBG * NFS;
    static_assert(NG <= 32 && NS >= 2 && NS <= 8, "a cell's basis changes fit one register per lane");
    const int lane = threadIdx.x & 31;
    const Level &lev = c.lev;
    const int64_t nt = chunk_tiles(c);
    using W = CellWatch<1, LB>;
    __shared__ __align__(16) uint32_t s_watch[8][W::WORDS];          // whole 16 bytes per warp
    W watch;
    watch.s = s_watch[threadIdx.x >> 5];
    watch.run(make_int2(-1, -1));
    uint32_t *row = watch.s;
    constexpr int BT = 32 / NS;                                     // tiles of a batch of ballots
    if (nt == 0) return;                                            // the chain has stopped
    unsigned tt, tb;
    watch.split(c, (unsigned)nt, blockIdx.x * 8u + (threadIdx.x >> 5), lane, tt, tb);
    float hs[ND];
    f2 negL2[ND];
#pragma unroll
    for (int j = 0; j < ND; ++j) {
        hs[j] = lev.Hs[j];
        negL2[j] = f2_dup(-lev.Lc[j] * lev.Lc[j]);
    }
    const float *gp = c.geo32 + (lane < NG ? lane : 0);
    auto load_g = [&](int cell) {
        if constexpr (NG == 0) return 0.0f;
        else return gp[(unsigned)(cell < 0 ? 0 : cell) * (size_t)c.gf];
    };
    int run = -1;
    f2 G[ND][LE][NP];
#pragma unroll
    for (int j = 0; j < ND; ++j)
#pragma unroll
        for (int m = 0; m < LE; ++m)
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                G[j][m][p] = 0ull;
                if constexpr (NG == 0)                              // a linear basis: the same for every cell
                    if (F::uses(j, m))
                        G[j][m][p] = f2_make(coef32<FAM>(lev, j, m, lin_change<FAM>(c, F::cb(j, m), 2 * p, false)),
                                             coef32<FAM>(lev, j, m, lin_change<FAM>(c, F::cb(j, m), NFS > 1 ? 2 * p + 1 : 0, false)));
            }
    unsigned next;
    do {
        next = watch.next(c, lane);
        bool head = true;
        run = -1;
        while (tt < tb) {
            // the first tile of the unit, or after those skipped
            const uint32_t *rp = c.in.rec + ((c.t0 + tt) * 32 + lane) * NW;
            const int2 *tp = c.tinfo + tt;
            int2 ti, ti1 = tp[0], ti2 = tp[1];
            uint32_t w1[NW];
            load_words<NW>(rp, 0, w1);
            float g1 = load_g(ti1.x);
            if (head) {
                const unsigned skip = watch.begin(c, NS, ti1, tt, tb, lane);
                if (skip) {
                    tt += skip;
                    head = false;
                    continue;
                }
                head = false;
            }
            for (;;) {
                const int bt = tb - tt < BT ? (int)(tb - tt) : BT;
                int rs = 0;                                         // first row of the last run
#pragma unroll 1
                for (int b = 0; b < bt; ++b) {
                    ti = ti1;
                    const float g = g1;
                    uint32_t w[NW];
#pragma unroll
                    for (int i = 0; i < NW; ++i) w[i] = w1[i];
                    rp += 32 * NW;
                    ++tp;
                    load_words<NW>(rp, 0, w1);
                    ti1 = ti2;
                    g1 = load_g(ti1.x);
                    ti2 = tp[1];
                    if (ti.x < 0) continue;                         // uniform: the cell was pruned
                    if (ti.x != run) {                                          // uniform: a new cell
                        run = ti.x;
                        rs = b;
                        watch.run(ti);
                        if constexpr (NG > 0) {
                            float d[F::NBG ? F::NBG : 1][NFS];
#pragma unroll
                            for (int x = 0; x < F::NBG; ++x)
#pragma unroll
                                for (int f = 0; f < NFS; ++f) d[x][f] = __shfl_sync(kFull, g, x * NFS + f);
#pragma unroll
                            for (int j = 0; j < ND; ++j)
#pragma unroll
                                for (int m = 0; m < LE; ++m)
#pragma unroll
                                    for (int p = 0; p < NP; ++p)                // one free slot: the pair holds it twice
                                        if (F::uses(j, m))
                                            G[j][m][p] = f2_make(coef32<FAM>(lev, j, m, d[F::cb(j, m)][2 * p]),
                                                                 coef32<FAM>(lev, j, m, d[F::cb(j, m)][NFS > 1 ? 2 * p + 1 : 0]));
                        }
                    }
                    const int nvalid = ti.y & 63;
                    watch.cnt += (unsigned)nvalid;
                    float qf[ND], qt[LE], R[ND], near[ND], nearL[ND];
                    f2 negR2[ND], u[ND][NP];
#pragma unroll
                    for (int j = 0; j < ND; ++j) qf[j] = field_f<Q16>(w, j);
#pragma unroll
                    for (int m = 0; m < LE; ++m) qt[m] = field_f<Q16>(w, ND + m);
                    F::radius32(lev, qt, R);
                    // a lane without a record fails every test (its residual is out of reach)
                    if (lane >= nvalid) qf[0] = 1.0e15f;
#pragma unroll
                    for (int j = 0; j < ND; ++j) {
                        negR2[j] = f2_dup(-R[j] * R[j]);
                        near[j] = nearL[j] = 3.0e38f;
#pragma unroll
                        for (int p = 0; p < NP; ++p) u[j][p] = f2_dup(qf[j]);
                    }
#pragma unroll
                    for (int m = 0; m < LE; ++m) {
                        const f2 q2 = f2_dup(qt[m]);
#pragma unroll
                        for (int j = 0; j < ND; ++j)
#pragma unroll
                            for (int p = 0; p < NP; ++p)
                                if (F::uses(j, m)) u[j][p] = f2_fma(q2, G[j][m][p], u[j][p]);
                    }
                    unsigned bu[NS], bl[NS];
                    test_children<ND, NFS, DM, LB>(u, hs, negR2, negL2, near, nearL, bu, bl);
                    if (lane == 0) {
                        store_row<NS>(row + b * NS, bu);
                        if constexpr (LB) store_row<NS>(row + 32 + b * NS, bl);
                    }
                    const unsigned act = nvalid >= 32 ? kFull : (1u << nvalid) - 1u;
                    const unsigned unsb = __ballot_sync(kFull, undecided<FAM, LB>(lev, R, near, nearL)) & act;
                    if (unsb) {                                                 // rare: left to the definition
                        __syncwarp();                                           // lane 0's stores
                        if (lane < NS) {
                            row[b * NS + lane] &= ~unsb;
                            if constexpr (LB) row[32 + b * NS + lane] &= ~unsb;
                        }
                        watch.cnt -= (unsigned)__popc(unsb);
                        if (lane == 0) c.uns[atomicAdd(&c.sc->n_uns, 1u)] = make_uint2(tt + b, unsb);
                    }
                }
                __syncwarp();
                unsigned word = 0u;
                if (lane < bt * NS) {
                    const size_t at = (size_t)tt * NS + lane;
                    word = row[lane];
                    c.ballot[at] = word;
                    if constexpr (LB) c.lballot[at] = row[32 + lane];
                }
                __syncwarp();
                tt += (unsigned)bt;
                watch.add(NS, NS == 8 ? 3 : (NS == 4 ? 2 : 1), &word, rs, lane);
                const unsigned skip = watch.cnt > watch.lim || tt >= tb ? watch.look(c, NS, ti, tt, tb, lane) : 0u;
                if (skip) {
                    tt += skip;
                    break;
                }
                if (tt >= tb) break;
            }
        }
    } while (watch.unit(__shfl_sync(kFull, next, 0), (unsigned)nt, tt, tb));
    watch.report(c, NW, lane);
}

// a persistent grid: as many blocks as are resident (4 per SM), fewer when there are not
// two tiles per warp
template <int FAM, bool Q16, int KF, int DM>
static void launch_kd(const Chunk &c, cudaStream_t st) {
    if constexpr (KF <= Fam<FAM>::K && DM < (1 << Fam<FAM>::ND) && (KF || DM)) {
        const int64_t nt = c.t1 - c.t0;
        const int64_t want = (int64_t)sm_count() * 4, need = (nt + 15) / 16;
        const unsigned g = (unsigned)(want < need ? want : need);
        if (c.lb) launch(k_count<FAM, Q16, KF, DM, true>, g, 256, 0, st, c);
        else launch(k_count<FAM, Q16, KF, DM, false>, g, 256, 0, st, c);
    }
}

template <int FAM, bool Q16>
static void launch_fam(const Chunk &c, cudaStream_t st) {
    switch (c.kf * 4 + c.dm) {
    case 1: launch_kd<FAM, Q16, 0, 1>(c, st); break;
    case 2: launch_kd<FAM, Q16, 0, 2>(c, st); break;
    case 3: launch_kd<FAM, Q16, 0, 3>(c, st); break;
    case 4: launch_kd<FAM, Q16, 1, 0>(c, st); break;
    case 5: launch_kd<FAM, Q16, 1, 1>(c, st); break;
    case 6: launch_kd<FAM, Q16, 1, 2>(c, st); break;
    case 7: launch_kd<FAM, Q16, 1, 3>(c, st); break;
    case 8: launch_kd<FAM, Q16, 2, 0>(c, st); break;
    case 9: launch_kd<FAM, Q16, 2, 1>(c, st); break;
    default: break;
    }
}

void launch_count(const Chunk &c, cudaStream_t st) {
    if (c.t1 <= c.t0) return;
    if (c.precision == 0) return launch_count_exact(c, st);
    if (c.P.d > 3) return launch_count_wide(c, st);
#define GV_COUNT(FAMV)                                  \
    if (c.lev.q16) launch_fam<FAMV, true>(c, st);       \
    else launch_fam<FAMV, false>(c, st)
    switch (c.P.fam) {
    case FAM_LINE2D: GV_COUNT(FAM_LINE2D); break;
    case FAM_PLANE3D_SPH: GV_COUNT(FAM_PLANE3D_SPH); break;
    case FAM_POSE3DOF: GV_COUNT(FAM_POSE3DOF); break;
    case FAM_RAYS3D: GV_COUNT(FAM_RAYS3D); break;
    default: break;
    }
#undef GV_COUNT
    launch_recheck(c, st);
}

}  // namespace gv
