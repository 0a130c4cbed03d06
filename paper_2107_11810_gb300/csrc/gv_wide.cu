// gv_wide.cu -- the proximity test's count and emit passes for families whose
// cells split into up to 16, 32 or 64 children (d = 4, 5, 6: Algorithm 2's 2^d
// sub-boxes).  The same tests as gv_count.cu and gv_emit.cu (the surface-box test
// of Sec. 3.2 with the FP32 screen and FP64 recheck, and the snap of the child
// records for the next level), with a loop over groups of free slots: the screen's
// coefficients of the cell (the same for every lane of a warp) are staged in the
// warp's part of shared memory once per run of tiles of one cell, transposed so that
// one load serves the coefficients of a whole group.
//
// Warps of the count pass take units of consecutive tiles and leave cells early (CellWatch);
// those of the emit pass a contiguous range of tiles.  Both read their records with plain
// loads; there are no device-side waits.
#include "gv_tile.cuh"

namespace gv {

// The screen's coefficients of a cell, transposed: sg[(j * LE + m) * nfs + f], by all lanes
// of a warp; per (j, m) the largest magnitude at sg[ND * LE * nfs + j * LE + m].
template <int FAM, bool MAX>
__device__ __forceinline__ void stage_coefs(const Chunk &c, int cell, float *sg, int lane) {
    using F = Fam<FAM>;
    const float *geo = c.geo32 + (size_t)cell * c.gf;
    const int f = lane & (c.nfs - 1);
#pragma unroll
    for (int j = 0; j < F::ND; ++j)
#pragma unroll
        for (int m = 0; m < F::LE; ++m) {
            if (!F::uses(j, m)) continue;
            const int b = F::cb(j, m), x = j * F::LE + m;
            const float d = b < F::NBG ? geo[b * c.ng + (f & (c.ng - 1))] : lin_change<FAM>(c, b, f, false);
            if (lane < c.nfs) sg[x * c.nfs + f] = coef32<FAM>(c.lev, j, m, d);
            if constexpr (MAX) {
                const float g = b < F::NBG ? geo[F::NBG * c.ng + b] : fabsf(d);
                if (lane == 0) sg[F::ND * F::LE * c.nfs + x] = g * c.lev.gs[j][m];
            }
        }
}

// Blocks per SM that the registers have to leave room for: as many as the tests alone need
// (affine 4-space 40 registers), whatever the rare paths would like (56).
constexpr int wide_residents(int fam, bool lb) {
    return fam == FAM_AFFINE4D ? (lb ? 5 : 6) : (fam == FAM_POSE6DOF ? 2 : (lb ? 3 : 4));
}

// FG: free slots per group (4, or all of them when fewer split)
template <int FAM, bool Q16, int FG, int DM, bool LB>
__global__ void __launch_bounds__(256, wide_residents(FAM, LB)) k_count_wide(const __grid_constant__ Chunk c) {
    grid_start();
    using F = Fam<FAM>;
    constexpr int ND = F::ND, LE = F::LE, NDS = dep_slots(DM), NX = ND * LE;
    constexpr int NW = rec_words(F::NFP, Q16);
    constexpr int GMAX = (1 << F::K) * NX;
    const int lane = threadIdx.x & 31;
    __shared__ __align__(16) float s_g[8][GMAX];
    float *sg = s_g[threadIdx.x >> 5];                              // [j * LE + m][nfs]
    const int nfs = c.nfs;
    int run = -1;
    const int64_t nt = chunk_tiles(c);
    constexpr int V = (1 << F::D) > 32 ? 2 : 1, ROW = 32 * V;       // a batch: BT tiles' rows of ns ballots
    const int ns = c.ns, BT = ns < 32 ? 32 >> c.lns : 1;
    using W = CellWatch<V, LB>;
    __shared__ __align__(16) uint32_t s_watch[8][W::WORDS];          // whole 16 bytes per warp
    W watch;
    watch.s = s_watch[threadIdx.x >> 5];
    watch.run(make_int2(-1, -1));
    uint32_t *rows = watch.s;
    if (nt == 0) return;                                            // the chain has stopped
    unsigned tt, tb;
    watch.split(c, (unsigned)nt, blockIdx.x * 8u + (threadIdx.x >> 5), lane, tt, tb);
    const Level &lev = c.lev;
    float hs[ND];
    f2 negL2[ND];
#pragma unroll
    for (int j = 0; j < ND; ++j) {
        hs[j] = lev.Hs[j];
        negL2[j] = f2_dup(-lev.Lc[j] * lev.Lc[j]);
    }
    bool staged = false;
    unsigned next;
    do {
        next = watch.next(c, lane);
        bool head = true;
        run = -1;
        while (tt < tb) {
            int2 ti;
            if (head && c.early) {
                ti = c.tinfo[tt];
                const unsigned skip = watch.begin(c, ns, ti, tt, tb, lane);
                if (skip) {
                    tt += skip;
                    head = false;
                    continue;
                }
            }
            head = false;
            const int bt = tb - tt < (unsigned)BT ? (int)(tb - tt) : BT;
            int rs = 0;                                             // first row of the last run
#pragma unroll 1
            for (int b = 0; b < bt; ++b) {
                ti = c.tinfo[tt + b];
                const int cell = ti.x;
                if (cell < 0) continue;                                     // uniform: the cell was pruned
                uint32_t w[NW];
                load_words<NW>(c.in.rec, (c.t0 + (tt + b)) * 32 + lane, w);       // whole tiles are allocated
                if (cell != run) {                                          // uniform: a new cell
                    rs = b;
                    watch.run(ti);
                    if (F::NBG > 0 || !staged) {                            // linear bases: once
                        __syncwarp();                                       // the old cell's reads are done
                        stage_coefs<FAM, false>(c, cell, sg, lane);
                        __syncwarp();
                        staged = true;
                    }
                    run = cell;
                }
                const int nvalid = ti.y & 63;
                watch.cnt += (unsigned)nvalid;
                float qf[ND], qt[LE], R[ND], near[ND], nearL[ND];
                f2 negR2[ND];
#pragma unroll
                for (int j = 0; j < ND; ++j) qf[j] = field_f<Q16>(w, j);
#pragma unroll
                for (int m = 0; m < LE; ++m) qt[m] = field_f<Q16>(w, ND + m);
                F::radius32(lev, qt, R);
#pragma unroll
                for (int j = 0; j < ND; ++j) {
                    negR2[j] = f2_dup(-R[j] * R[j]);
                    near[j] = nearL[j] = 3.0e38f;
                }
                // a lane without a record fails every test (its residual is out of reach)
                if (lane >= nvalid) qf[0] = 1.0e15f;
                uint32_t *bp = rows + b * ns, *lp = rows + ROW + b * ns;
#pragma unroll 1
                for (int fs = 0; fs < nfs; fs += FG) {
                    f2 u[ND][(FG + 1) / 2];
#pragma unroll
                    for (int j = 0; j < ND; ++j) {
#pragma unroll
                        for (int p = 0; p < (FG + 1) / 2; ++p) u[j][p] = f2_dup(qf[j]);
#pragma unroll
                        for (int m = 0; m < LE; ++m) {
                            if (!F::uses(j, m)) continue;
                            const float *g = sg + (j * LE + m) * nfs + fs;
                            const f2 q2 = f2_dup(qt[m]);
                            if constexpr (FG == 4) {
                                const ulonglong2 g4 = *reinterpret_cast<const ulonglong2 *>(g);
                                u[j][0] = f2_fma(q2, g4.x, u[j][0]);
                                u[j][1] = f2_fma(q2, g4.y, u[j][1]);
                            } else if constexpr (FG == 2) {
                                u[j][0] = f2_fma(q2, *reinterpret_cast<const f2 *>(g), u[j][0]);
                            } else {
                                u[j][0] = f2_fma(q2, f2_dup(g[0]), u[j][0]);
                            }
                        }
                    }
                    unsigned bu[FG * NDS], bl[FG * NDS];
                    test_children<ND, FG, DM, LB>(u, hs, negR2, negL2, near, nearL, bu, bl);
                    if (lane == 0) {
#pragma unroll
                        for (int x = 0; x < NDS; ++x) {
                            uint32_t *b = bp + x * nfs + fs, *l = lp + x * nfs + fs;
                            if constexpr (FG == 4) {
                                *reinterpret_cast<uint4 *>(b) = make_uint4(bu[4 * x], bu[4 * x + 1], bu[4 * x + 2], bu[4 * x + 3]);
                                if constexpr (LB)
                                    *reinterpret_cast<uint4 *>(l) = make_uint4(bl[4 * x], bl[4 * x + 1], bl[4 * x + 2], bl[4 * x + 3]);
                            } else {
#pragma unroll
                                for (int f = 0; f < FG; ++f) {
                                    b[f] = bu[FG * x + f];
                                    if constexpr (LB) l[f] = bl[FG * x + f];
                                }
                            }
                        }
                    }
                }
                const unsigned act = nvalid >= 32 ? kFull : (1u << nvalid) - 1u;
                const unsigned unsb = __ballot_sync(kFull, undecided<FAM, LB>(lev, R, near, nearL)) & act;
                if (unsb) {                                                 // rare: left to the definition
                    __syncwarp();                                           // lane 0's stores
                    for (int s = lane; s < ns; s += 32) {
                        bp[s] &= ~unsb;
                        if constexpr (LB) lp[s] &= ~unsb;
                    }
                    watch.cnt -= (unsigned)__popc(unsb);
                    if (lane == 0) c.uns[atomicAdd(&c.sc->n_uns, 1u)] = make_uint2(tt + b, unsb);
                }
            }
            __syncwarp();
            unsigned word[V];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                word[v] = 0u;
                if (lane + 32 * v < bt * ns) {
                    word[v] = rows[lane + 32 * v];
                    c.ballot[(size_t)tt * ns + lane + 32 * v] = word[v];
                    if constexpr (LB) c.lballot[(size_t)tt * ns + lane + 32 * v] = rows[ROW + lane + 32 * v];
                }
            }
            __syncwarp();
            tt += (unsigned)bt;
            watch.add(ns, c.lns, word, rs, lane);
            if (watch.cnt > watch.lim || tt >= tb) tt += watch.look(c, ns, ti, tt, tb, lane);
        }
    } while (watch.unit(__shfl_sync(kFull, next, 0), (unsigned)nt, tt, tb));
    watch.report(c, NW, lane);
}

// The emit pass (see gv_emit.cu): slot rows of a tile (output address, passing lanes)
// staged by one lane per slot, then a loop over the free slots with the snaps of their
// dependent shifts (taken once per coordinate and shift) and one predicated store per
// child.
template <int FAM, bool QI16, bool QO16>
__global__ void __launch_bounds__(256) k_emit_wide(const __grid_constant__ Chunk c) {
    grid_start();
    using F = Fam<FAM>;
    constexpr int NDS = 1 << F::ND, ND = F::ND, LE = F::LE, NFP = F::NFP;
    static_assert(F::D <= 6 && ND <= 2, "at most 64 child slots, two dependent coordinates");
    constexpr int NWI = rec_words(NFP, QI16), NWO = rec_words(NFP, QO16);
    constexpr int GF = ((1 << F::K) + 1) * ND * LE;
    if (c.dyn && c.dyn->overflow) return;                           // the children were not laid out
    const int NS = c.ns, nfs = c.nfs;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the current cell's screen coefficients, staged once per run of tiles of the
    // cell in the warp's part of shared memory; the slot rows of the tile at hand
    __shared__ float s_g[8][GF];
    __shared__ uint4 s_rows[8][1 << F::D];
    float *G = s_g[warp];
    uint4 *s_row = s_rows[warp];
    int gcell = -1;
    const unsigned below = (1u << lane) - 1u, lanebit = 1u << lane;
    const int64_t nt = chunk_tiles(c);
    const int64_t nwarp = (int64_t)gridDim.x * 8, gw = (int64_t)blockIdx.x * 8 + warp;
    const int64_t ta = gw * nt / nwarp, tb = (gw + 1) * nt / nwarp;
    const Level &lev = c.lev;
    float hs[ND];
#pragma unroll
    for (int j = 0; j < ND; ++j) hs[j] = ((c.dm >> j) & 1) ? lev.Hs[j] : 0.0f;
    unsigned nrechk = 0, ndf = 0, bad = 0;

#pragma unroll 1
    for (int64_t tt = ta; tt < tb; ++tt) {
        const int cell = c.tinfo[tt].x;
        if (cell < 0) continue;                                     // uniform
        __syncwarp();                                               // the last tile's rows are read
        unsigned v[2] = {0u, 0u};                                   // child slots this tile writes
#pragma unroll
        for (int h = 0; h < (F::D > 5 ? 2 : 1); ++h) {
            const int s = lane + 32 * h;
            unsigned bal = 0;
            if (s < NS) {
                const unsigned long long base = c.cbase[(size_t)cell * NS + s];
                const unsigned long long p0 = base + c.off[(size_t)tt * NS + s];
                bal = base == ~0ull ? 0u : c.ballot[(size_t)tt * NS + s];
                const unsigned long long q = (p0 + 31) >> 5;
                if (bal && (q << 5) < p0 + (unsigned)__popc(bal))
                    c.out.tile_cell[q] = (uint32_t)c.child_idx[(size_t)cell * NS + s];
                const unsigned long long p = (unsigned long long)(c.out.rec + p0 * NWO);
                s_row[s] = make_uint4((unsigned)p, (unsigned)(p >> 32), bal, 0u);
            }
            v[h] = __ballot_sync(kFull, bal != 0u);
        }
        if (!(v[0] | v[1])) continue;                               // uniform: nothing to write
        const int64_t r = (c.t0 + tt) * 32 + lane;
        uint32_t w[NWI];
        load_words<NWI>(c.in.rec, r, w);
        if (F::NBG > 0 ? cell != gcell : gcell < 0) {               // uniform (linear bases: once)
            stage_coefs<FAM, true>(c, cell, G, lane);
            gcell = cell;
        }
        __syncwarp();
        // the child's essential parameters (re-snapped when the step doubles)
        uint32_t fb[NFP];
#pragma unroll
        for (int i = 0; i < NFP; ++i) fb[i] = 0u;
        float qf[ND], qt[LE];
#pragma unroll
        for (int j = 0; j < ND; ++j) qf[j] = field_f<QI16>(w, j);
#pragma unroll
        for (int m = 0; m < LE; ++m) {
            qt[m] = field_f<QI16>(w, ND + m);
            if constexpr (QO16) {
                // adding kMagic16 rounds to an integer, ties to even, biased by 2^15
                fb[ND + m] = __float_as_uint(__fmaf_rn(qt[m], lev.st_scale[m], kMagic16));
            } else {
                const int q = field_i<QI16>(w, ND + m);
                fb[ND + m] = (uint32_t)(lev.st_ratio_log2[m] ? resnap_half(q) : q);
            }
        }
        float es[ND], M[ND];                                        // a snap is certain within es of an integer
        {
            // every term a multiple of 2^ex and M below 2^(24 + ex): the FP32 residual, and
            // the definition's FP64 one, are exact, so a tie rounds to even in both
            const int ex = min(lev.g_exp, lev.hs_exp);
            const float tq = ex > -100 && c.precision == 1 ? __int_as_float((127 + 24 + ex) << 23) : 0.0f;
            magnitudes<FAM>(qf, qt, G + nfs * ND * LE, hs, M);
#pragma unroll
            for (int j = 0; j < ND; ++j) {
                // plain FP64 mode: no snap is certain
                es[j] = M[j] < tq ? 1.0f : __fmaf_rn(-kBandSnap, M[j], c.precision == 1 ? 0.5f : -1.0f);
            }
        }
        unsigned long long um = 0ull;                               // slots whose snap FP32 leaves undecided
#pragma unroll 1
        for (int f = 0; f < nfs; ++f) {
            unsigned any = 0;                                       // this free slot's children, bit ds
#pragma unroll
            for (int ds = 0; ds < NDS; ++ds) {
                if (ds & ~c.dm) continue;
                const int s = child_slot(f, ds, c.dm, c.kf);
                any |= ((s < 32 ? (v[0] >> s) : (v[1] >> (s - 32))) & 1u) << ds;
            }
            if (!any) continue;                                     // uniform
            float u[ND];
#pragma unroll
            for (int j = 0; j < ND; ++j) {
                u[j] = qf[j];
#pragma unroll
                for (int m = 0; m < LE; ++m)
                    if (F::uses(j, m)) u[j] = __fmaf_rn(qt[m], G[(j * LE + m) * nfs + f], u[j]);
            }
            uint32_t sv[ND][2];
            bool so[ND][2];
#pragma unroll
            for (int j = 0; j < ND; ++j)
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    // a coordinate that does not split has ds bit 0 and shift 0
                    const float y = k ? u[j] - hs[j] : u[j] + hs[j];
                    if constexpr (QO16) {
                        // |y| <= 32000: the record passed this level's UB test (finalize_levels)
                        const float t = y + kMagic16;
                        so[j][k] = fabsf(y - (t - kMagic16)) < es[j];
                        sv[j][k] = __float_as_uint(t);
                    } else {
                        const float t = y + kMagic;
                        so[j][k] = fabsf(y - (t - kMagic)) < es[j] && fabsf(y) < 4.0e6f;
                        sv[j][k] = (uint32_t)(__float_as_int(t) - 0x4B400000);
                    }
                }
#pragma unroll
            for (int ds = 0; ds < NDS; ++ds) {
                if (!((any >> ds) & 1)) continue;                   // uniform
                const int s = child_slot(f, ds, c.dm, c.kf);
                const uint4 rw = s_row[s];
                bool sure = true;
#pragma unroll
                for (int j = 0; j < ND; ++j) {
                    fb[j] = sv[j][(ds >> j) & 1];
                    sure &= so[j][(ds >> j) & 1];
                }
                uint32_t wo[NWO];
                pack<NFP, QO16>(fb, wo);
                store_words_if<NWO>(rw.z & lanebit, row_address(rw) + (unsigned)__popc(rw.z & below) * (NWO * 4u), wo);
                if ((rw.z & lanebit) && !sure) um |= 1ull << s;
            }
        }
        if (c.out.mult) {                                           // grouping: the records' multiplicities
            const uint32_t mult = c.in.mult[r];
            for (int s = 0; s < NS; ++s) {
                const uint4 rw = s_row[s];
                const unsigned long long i =
                    (row_address(rw) - (unsigned long long)c.out.rec) / (NWO * 4u) + (unsigned)__popc(rw.z & below);
                if (rw.z & lanebit) c.out.mult[i] = mult;
            }
        }
        if (um) {                                                   // rare
            const RecWords<NWI> rwords = rec_words_of<NWI>(w);
            for (unsigned long long m = um; m; m &= m - 1) {
                const int s = __ffsll((long long)m) - 1, f = s & (nfs - 1), x = s >> c.kf, ds = c.dm == 2 ? x << 1 : x;
                const uint4 rw = s_row[s];
                int3 q = make_int3(0, 0, 0);
                if (c.precision == 1) {                             // the double-float tier
                    q = snap_df_words<FAM, QI16>(&c, rwords, cell, f, ds, __fmaf_ru(kBandDF, M[0], kBandDFAbs),
                                                 __fmaf_ru(kBandDF, M[ND - 1], kBandDFAbs), QO16 ? 32767.0f : 1.0e9f);
                    ++ndf;
                }
                if (!q.z) {                                         // the FP64 definition
                    q = snap64_words<FAM, QI16>(&c, rwords, cell, f, ds);
                    bad |= (unsigned)(q.z != 0);
                    nrechk += c.precision == 1;
                }
                const int qn[2] = {q.x, q.y};
#pragma unroll
                for (int j = 0; j < ND; ++j) {
                    if constexpr (QO16) {
                        bad |= (unsigned)(qn[j] < -32768 || qn[j] > 32767) << 1;
                        fb[j] = (uint32_t)(qn[j] + 32768);
                    } else {
                        fb[j] = (uint32_t)qn[j];
                    }
                }
                uint32_t wo[NWO];
                pack<NFP, QO16>(fb, wo);
                store_words_if<NWO>(1u, row_address(rw) + (unsigned)__popc(rw.z & below) * (NWO * 4u), wo);
            }
        }
    }
    nrechk = __reduce_add_sync(kFull, nrechk);
    ndf = __reduce_add_sync(kFull, ndf);
    bad = __reduce_or_sync(kFull, bad);
    if (lane == 0) {
        if (nrechk) atomicAdd(&c.sc->rechecks, (unsigned long long)nrechk);
        if (ndf) atomicAdd(&c.sc->rechecks_df, (unsigned long long)ndf);
        if (bad) atomicOr(&c.sc->err, bad << 1);
    }
}

// a grid of 8-warp blocks: enough warps to fill the device, at most one per tile
static unsigned wide_blocks(int64_t nt) {
    const int64_t want = (int64_t)sm_count() * 8, need = (nt + 7) / 8;
    return (unsigned)(want < need ? want : need);
}

#define GV_DISPATCH_WIDE(fam, CALL)                                            \
    switch (fam) {                                                             \
    case FAM_POSE6DOF: { constexpr int FAMV = FAM_POSE6DOF; CALL; } break;     \
    case FAM_POINTSET2D: { constexpr int FAMV = FAM_POINTSET2D; CALL; } break; \
    case FAM_AFFINE4D: { constexpr int FAMV = FAM_AFFINE4D; CALL; } break;     \
    case FAM_RADIAL5DOF: { constexpr int FAMV = FAM_RADIAL5DOF; CALL; } break; \
    default: break;                                                            \
    }

template <int FAM, bool Q16, int FG, int DM>
static void launch_wide(const Chunk &c, cudaStream_t st) {
    if constexpr (DM < (1 << Fam<FAM>::ND) && (FG > 1 || DM)) {
        const unsigned g = wide_blocks(c.t1 - c.t0);
        if (c.early)                                    // resident warps only: they share the units
            launch_persistent(c.lb ? (const void *)k_count_wide<FAM, Q16, FG, DM, true>
                                   : (const void *)k_count_wide<FAM, Q16, FG, DM, false>,
                              0, g, c, st);
        else if (c.lb) launch(k_count_wide<FAM, Q16, FG, DM, true>, g, 256, 0, st, c);
        else launch(k_count_wide<FAM, Q16, FG, DM, false>, g, 256, 0, st, c);
    }
}

template <int FAM, bool Q16, int FG>
static void launch_wide_dm(const Chunk &c, cudaStream_t st) {
    if (c.dm == 0) launch_wide<FAM, Q16, FG, 0>(c, st);
    else if (c.dm == 1) launch_wide<FAM, Q16, FG, 1>(c, st);
    else if (c.dm == 2) launch_wide<FAM, Q16, FG, 2>(c, st);
    else launch_wide<FAM, Q16, FG, 3>(c, st);
}

template <int FAM, bool Q16>
static void launch_wide_fam(const Chunk &c, cudaStream_t st) {
    if (c.kf >= 2) launch_wide_dm<FAM, Q16, 4>(c, st);
    else if (c.kf == 1) launch_wide_dm<FAM, Q16, 2>(c, st);
    else launch_wide_dm<FAM, Q16, 1>(c, st);
}

void launch_count_wide(const Chunk &c, cudaStream_t st) {
    if (c.lev.q16) {
        GV_DISPATCH_WIDE(c.P.fam, (launch_wide_fam<FAMV, true>(c, st)));
    } else {
        GV_DISPATCH_WIDE(c.P.fam, (launch_wide_fam<FAMV, false>(c, st)));
    }
    launch_recheck(c, st);
}

bool launch_emit_wide(const Chunk &c, cudaStream_t st) {
    const int64_t nt = c.t1 - c.t0;
    if (nt <= 0) return true;
    const unsigned g = wide_blocks(nt);
    const int q = c.lev.q16, qn = c.lev.q16_next;
    bool known = false;
    GV_DISPATCH_WIDE(c.P.fam, (known = FAMV > 0));
    if (!known) return false;
    if (c.precision == 0 && (q || qn)) return false;    // plain FP64 mode keeps 32-bit records
    if (q && qn) {
        GV_DISPATCH_WIDE(c.P.fam, (launch(k_emit_wide<FAMV, true, true>, g, 256, 0, st, c)));
    } else if (!q && qn) {
        GV_DISPATCH_WIDE(c.P.fam, (launch(k_emit_wide<FAMV, false, true>, g, 256, 0, st, c)));
    } else if (!q && !qn) {
        GV_DISPATCH_WIDE(c.P.fam, (launch(k_emit_wide<FAMV, false, false>, g, 256, 0, st, c)));
    } else {
        return false;                                   // 16-bit to 32-bit: never chosen
    }
    return true;
}

}  // namespace gv
