// gv_emit.cu -- emit pass of the proximity test: every record of a chunk that
// passed the UB test of a surviving child (the ballots of the count pass) is
// written into that child's record range, with its free parameters snapped at the
// child's centre for the next level (canonization, Sec. 3.2: the residual at the
// child centre, rounded to the snap step; essential parameters re-snapped when
// their step doubles).
//
// Positions: every tile's first place in each child comes from k_tile_scan;
// inside a tile a lane's position is the number of passing lanes below it.
//
// The snap is taken in FP32 (in steps) when the value is at least the screen's
// band away from a rounding tie, or when the residual is exact in FP32 (every term
// a multiple of 2^e and the magnitudes below 2^(24+e): a tie then rounds to even as
// the definition's exact FP64 value does); else by a double-float recomputation
// when that is far enough from a tie; else in FP64 by the definition.
//
// The pass is bound by instruction issue, not by its stores: of a tile's 32 records
// about a sixth pass a given child of a plane cell.  So a child slot costs one 16-byte
// shared-memory load (its passing lanes and output address, staged by one lane per
// slot), the snap, and one predicated store, without a divergent branch; the lanes whose
// snap FP32 does not decide are put right afterwards.
#include "gv_tile.cuh"

namespace gv {

constexpr int kEmitTiles = 4;                        // tiles per warp and buffer
constexpr int kEmitUnit = 16;                        // consecutive tiles a warp takes at a time (kEmitTiles
                                                     // while that leaves under four units per warp)

// Shared memory of one block (8 warps): per warp two buffers of kEmitTiles tiles of
// records, ballots and positions, and the slot rows of the tile at hand (two, by turns).
template <int NW>
__host__ __device__ constexpr size_t emit_warp_bytes(int ns) {
    return 2 * (size_t)kEmitTiles * (32 * NW * 4 + ns * 8) + 2 * 16 * (size_t)ns;
}

// KF: free coordinates that split, DM: dependent coordinates that split (bit mask).
// Warps take units of kEmitUnit tiles by turns; the groups of kEmitTiles tiles of a unit
// with a cell that has surviving children stream through the warp's own two buffers
// (bulk copies completing on the warp's mbarriers), so warps never wait for each other,
// and neither reading nor the work falls to tiles that have nothing to write.
template <int FAM, bool QI16, bool QO16, int KF, int DM>
__global__ void __launch_bounds__(256, 3) k_emit(const __grid_constant__ Chunk c) {
    grid_start();
    using F = Fam<FAM>;
    constexpr int ND = F::ND, LE = F::LE, NFP = F::NFP, NFS = 1 << KF, NDS = dep_slots(DM), NS = NFS * NDS;
    constexpr int NWI = rec_words(NFP, QI16), NWO = rec_words(NFP, QO16), RW = 32 * NWI, NG = F::NBG * NFS;
    constexpr int GT = kEmitTiles, NP = (NFS + 1) / 2;
    // child slots of free slot 0 (those of free slot f: shifted left by f)
    constexpr unsigned kFsSlots = NDS == 4 ? 1u | 1u << NFS | 1u << 2 * NFS | 1u << 3 * NFS : (NDS == 2 ? 1u | 1u << NFS : 1u);
    static_assert(NG + F::NBG <= 32, "a cell's basis changes fit one register per lane");
    if (c.dyn && c.dyn->overflow) return;                           // the children were not laid out
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Level &lev = c.lev;
    extern __shared__ __align__(128) uint8_t s_dyn[];
    uint32_t *s_rec = reinterpret_cast<uint32_t *>(s_dyn + warp * emit_warp_bytes<NWI>(NS));   // [2][GT * RW]
    uint32_t *s_bal = s_rec + 2 * GT * RW;                                                  // [2][GT * NS]
    uint32_t *s_off = s_bal + 2 * GT * NS;                                                  // [2][GT * NS]
    uint4 *s_row = reinterpret_cast<uint4 *>(s_off + 2 * GT * NS);                          // [2][NS]
    __shared__ __align__(8) uint64_t s_bars[8][2];
    uint64_t *s_bar = s_bars[warp];

    const int nt = (int)chunk_tiles(c);
    const int nwarp = gridDim.x * 8, gw = blockIdx.x * 8 + warp;
    const int ut = nt > 4 * kEmitUnit * nwarp ? kEmitUnit : GT, nunits = (nt + ut - 1) / ut;
    if (lane == 0) {
        mbar_init(&s_bar[0], 1);
        mbar_init(&s_bar[1], 1);
        mbar_init_fence();
    }
    __syncwarp();

    // units of this warp: lane k < ut holds the cell of the unit's tile k (-1: nothing to
    // write); the next unit's are loaded, and the tile information of the one after it, so
    // no load waits for another
    int unit = gw, ucells, pcells, tcells;
    auto load_cells = [&](int u) {
        const int t = u * ut + lane;
        if (lane >= ut || u >= nunits || t >= nt) return -1;
        return c.tinfo[t].x;
    };
    auto live = [&](int cell) { return cell >= 0 && (c.alive[cell] & 2) ? cell : -1; };
    ucells = live(load_cells(unit));
    unsigned umask = __ballot_sync(kFull, ucells >= 0);             // the unit's tiles still to be taken
    pcells = live(load_cells(unit + nwarp));
    tcells = load_cells(unit + 2 * nwarp);
    // the next group with something to write: its first tile (-1: none is left), its cells
    auto next_group = [&](int &t0, int &cells) {
        while (!umask) {
            unit += nwarp;
            if (unit >= nunits) {
                t0 = -1;
                cells = -1;
                return;
            }
            ucells = pcells;
            umask = __ballot_sync(kFull, ucells >= 0);
            pcells = live(tcells);
            tcells = load_cells(unit + 2 * nwarp);
        }
        const int g = (__ffs(umask) - 1) / GT;
        umask &= ~(((1u << GT) - 1u) << (g * GT));
        t0 = unit * ut + g * GT;
        cells = __shfl_sync(kFull, ucells, g * GT + (lane & (GT - 1)));
    };
    // lane 0: copy number n (buffer n & 1)
    auto issue = [&](int n, int t0) {
        const int b = n & 1, ntl = t0 + GT < nt ? GT : nt - t0;
        // bulk copies take multiples of 16 bytes (the arrays are padded past the last tile)
        const unsigned rbytes = (unsigned)ntl * RW * 4, bbytes = ((unsigned)ntl * NS * 4 + 15u) & ~15u;
        mbar_expect_tx(&s_bar[b], rbytes + 2 * bbytes);
        bulk_load(s_rec + b * GT * RW, c.in.rec + (c.t0 + t0) * RW, rbytes, &s_bar[b]);
        bulk_load(s_bal + b * GT * NS, c.ballot + (size_t)t0 * NS, bbytes, &s_bar[b]);
        bulk_load(s_off + b * GT * NS, c.off + (size_t)t0 * NS, bbytes, &s_bar[b]);
    };
    // a cell's data, one word per lane: basis change, child's first slot and index
    float pg = 0.0f;
    unsigned long long pbase = ~0ull;
    int pidx = 0;
    auto prefetch = [&](int cell) {
        if (cell < 0) return;                                       // uniform
        if (lane < NG + F::NBG) pg = c.geo32[(size_t)cell * c.gf + lane];
        if (lane < NS) {
            pbase = c.cbase[(size_t)cell * NS + lane];
            pidx = c.child_idx[(size_t)cell * NS + lane];
        }
    };

    float hs[ND];
#pragma unroll
    for (int j = 0; j < ND; ++j) hs[j] = ((DM >> j) & 1) ? lev.Hs[j] : 0.0f;
    const unsigned below = (1u << lane) - 1u, lanebit = 1u << lane;
    int cur = -1, pcell = -1, row = 0;                              // the cell at hand, the prefetched one
    f2 G[ND][LE][NP];
    float Gmax[ND * LE];
    // every term a multiple of 2^ex and M below 2^(24 + ex): the FP32 residual, and the
    // definition's FP64 one, are exact, so a tie rounds to even in both
    const int ex = min(lev.g_exp, lev.hs_exp);
    const float tq = ex > -100 && c.precision == 1 ? __int_as_float((127 + 24 + ex) << 23) : 0.0f;
    const float es0 = c.precision == 1 ? 0.5f : -1.0f;              // plain FP64 mode: no snap is certain
    unsigned long long crec = 0;                                    // lane s: child s's first record, 0 when pruned
    uint32_t *ctile = nullptr;                                      // and its first tile -> cell entry
    int cidx = 0;
#pragma unroll
    for (int j = 0; j < ND; ++j)
#pragma unroll
        for (int x = 0; x < LE; ++x) {
            Gmax[j * LE + x] = 0.0f;
#pragma unroll
            for (int p = 0; p < NP; ++p) G[j][x][p] = 0ull;
            if constexpr (NG == 0) {                                // a linear basis: the same for every cell
                if (!F::uses(j, x)) continue;
#pragma unroll
                for (int p = 0; p < NP; ++p)
                    G[j][x][p] = f2_make(coef32<FAM>(lev, j, x, lin_change<FAM>(c, F::cb(j, x), 2 * p, false)),
                                         coef32<FAM>(lev, j, x, lin_change<FAM>(c, F::cb(j, x), NFS > 1 ? 2 * p + 1 : 0, false)));
                Gmax[j * LE + x] = fabsf(coef32<FAM>(lev, j, x, lin_change<FAM>(c, F::cb(j, x), 0, false)));
            }
        }
    unsigned nrechk = 0, ndf = 0, bad = 0;
    int t1, cells1, nfail = -1;                                     // copy that did not arrive
    next_group(t1, cells1);
    if (t1 >= 0 && lane == 0) issue(0, t1);
#pragma unroll 1
    for (int n = 0; t1 >= 0; ++n) {
        const int b = n & 1, t0 = t1, cells = cells1;
        next_group(t1, cells1);
        if (t1 >= 0 && lane == 0) issue(n + 1, t1);
        const unsigned gm = __ballot_sync(kFull, cells >= 0) & ((1u << GT) - 1u);
        if (pcell < 0) {                                            // the first group
            pcell = __shfl_sync(kFull, cells, __ffs(gm) - 1);
            prefetch(pcell);
        }
        const bool ok = mbar_wait(&s_bar[b], (unsigned)(n >> 1) & 1u, c.spin, &c.sc->err);
        if (!__all_sync(kFull, ok)) {
            nfail = n;
            break;
        }
#pragma unroll 1
        for (unsigned m = gm; m; m &= m - 1) {
            const int lt = __ffs(m) - 1, cl = __shfl_sync(kFull, cells, lt);
            if (cl != cur) {                                        // uniform: a new cell, prefetched
                cur = cl;
                crec = pbase == ~0ull ? 0ull : (unsigned long long)(c.out.rec + pbase * NWO);
                ctile = c.out.tile_cell + (pbase >> 5);
                cidx = pidx;
                if constexpr (NG > 0) {
                    float d[F::NBG ? F::NBG : 1][NFS + 1];          // the last: the largest magnitude
#pragma unroll
                    for (int x = 0; x < F::NBG; ++x) {
#pragma unroll
                        for (int f = 0; f < NFS; ++f) d[x][f] = __shfl_sync(kFull, pg, x * NFS + f);
                        d[x][NFS] = __shfl_sync(kFull, pg, NG + x);
                    }
#pragma unroll
                    for (int j = 0; j < ND; ++j)
#pragma unroll
                        for (int x = 0; x < LE; ++x) {
                            if (!F::uses(j, x)) continue;
#pragma unroll
                            for (int p = 0; p < NP; ++p)
                                G[j][x][p] = f2_make(coef32<FAM>(lev, j, x, d[F::cb(j, x)][2 * p]),
                                                     coef32<FAM>(lev, j, x, d[F::cb(j, x)][NFS > 1 ? 2 * p + 1 : 0]));
                            Gmax[j * LE + x] = d[F::cb(j, x)][NFS] * lev.gs[j][x];
                        }
                }
            }
            {
                // the cell of the next tile to be taken
                const unsigned rest = m & (m - 1);
                const unsigned gn = __ballot_sync(kFull, cells1 >= 0) & ((1u << GT) - 1u);
                const int a = __shfl_sync(kFull, cells, rest ? __ffs(rest) - 1 : 0);
                const int z = __shfl_sync(kFull, cells1, gn ? __ffs(gn) - 1 : 0);
                const int nx = rest ? a : z;
                if (nx >= 0 && nx != pcell) {                       // uniform
                    pcell = nx;
                    prefetch(nx);
                }
            }
            // slot rows: output address and passing lanes; the next level's tile -> cell
            // table for the one tile whose first slot this tile may fill
            row ^= NS;
            unsigned bal = 0;
            if (lane < NS) {
                const unsigned off = s_off[b * GT * NS + lt * NS + lane];
                bal = crec ? s_bal[b * GT * NS + lt * NS + lane] : 0u;
                const unsigned first = (off + 31u) & ~31u;
                if (first < off + (unsigned)__popc(bal)) ctile[first >> 5] = (uint32_t)cidx;
                const unsigned long long p = crec + off * (unsigned long long)(NWO * 4);
                s_row[row + lane] = make_uint4((unsigned)p, (unsigned)(p >> 32), bal, 0u);
            }
            const unsigned vmask = __ballot_sync(kFull, bal != 0u);  // child slots this tile writes
            __syncwarp();
            if (!vmask) continue;                                   // uniform: nothing to write
            uint32_t w[NWI];
            load_words<NWI>(s_rec + b * GT * RW + lt * RW, lane, w);
            // the child's essential parameters (re-snapped when the step doubles)
            uint32_t fb[NFP];
#pragma unroll
            for (int i = 0; i < NFP; ++i) fb[i] = 0u;
            float qf[ND], qt[LE];
#pragma unroll
            for (int j = 0; j < ND; ++j) qf[j] = field_f<QI16>(w, j);
#pragma unroll
            for (int x = 0; x < LE; ++x) {
                qt[x] = field_f<QI16>(w, ND + x);
                if constexpr (QO16) {
                    // adding kMagic16 rounds to an integer, ties to even, biased by 2^15
                    fb[ND + x] = __float_as_uint(__fmaf_rn(qt[x], lev.st_scale[x], kMagic16));
                } else {
                    const int q = field_i<QI16>(w, ND + x);
                    fb[ND + x] = (uint32_t)(lev.st_ratio_log2[x] ? resnap_half(q) : q);
                }
            }
            float es[ND], M[ND];                                    // a snap is certain within es of an integer
            magnitudes<FAM>(qf, qt, Gmax, hs, M);
#pragma unroll
            for (int j = 0; j < ND; ++j) es[j] = M[j] < tq ? 1.0f : __fmaf_rn(-kBandSnap, M[j], es0);
            unsigned um = 0;                                        // slots whose snap FP32 leaves undecided
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                constexpr unsigned kPair = NFS > 1 ? kFsSlots | kFsSlots << 1 : kFsSlots;
                if (!(vmask & (kPair << (2 * p)))) continue;        // uniform: no child of these free slots
                // snapped residuals of (free slots 2 p and 2 p + 1) x shift, or, with one free
                // slot, of the two shifts: y + kMagic(16) rounds to an integer, ties to even
                float sv[ND][2][2], er[ND][2][2];
#pragma unroll
                for (int j = 0; j < ND; ++j) {
                    f2 u = f2_dup(qf[j]);
#pragma unroll
                    for (int x = 0; x < LE; ++x)
                        if (F::uses(j, x)) u = f2_fma(f2_dup(qt[x]), G[j][x][p], u);
                    constexpr float kM = QO16 ? kMagic16 : kMagic;
                    const bool split = (DM >> j) & 1;
#pragma unroll
                    for (int v = 0; v < (NFS > 1 && split ? 2 : 1); ++v) {
                        f2 y = u;
                        if (split) y = f2_add(u, NFS > 1 ? f2_dup(v ? -hs[j] : hs[j]) : f2_make(hs[j], -hs[j]));
                        const f2 t = f2_add(y, f2_dup(kM));
                        // y - (t - kM), exact
                        const f2 e = f2_fma(f2_add(t, f2_dup(-kM)), f2_dup(-1.0f), y);
                        float a0, a1, b0, b1;
                        f2_get(t, a0, a1);
                        f2_get(e, b0, b1);
                        if constexpr (!QO16) {                      // 16-bit children: |y| <= 32000 (finalize_levels)
                            float y0, y1;
                            f2_get(y, y0, y1);
                            b0 = fabsf(y0) < 4.0e6f ? b0 : 1.0f;
                            b1 = fabsf(y1) < 4.0e6f ? b1 : 1.0f;
                        }
                        if (NFS > 1) {
                            sv[j][v][0] = a0; er[j][v][0] = b0;
                            sv[j][v][1] = a1; er[j][v][1] = b1;
                        } else {
                            sv[j][0][0] = a0; er[j][0][0] = b0;
                            sv[j][1][0] = a1; er[j][1][0] = b1;
                        }
                    }
                }
#pragma unroll
                for (int h = 0; h < (NFS > 1 ? 2 : 1); ++h) {
                    const int f = 2 * p + h;
                    if (NFS > 1 && !(vmask & (kFsSlots << f))) continue;   // uniform
#pragma unroll
                    for (int x = 0; x < NDS; ++x) {
                        const int s = x * NFS + f, ds = DM == 2 ? x << 1 : x;
                        const uint4 rw = s_row[row + s];            // no passing lane: nothing is stored
#pragma unroll
                        for (int j = 0; j < ND; ++j) {
                            const float t = sv[j][(ds >> j) & 1][h];
                            fb[j] = QO16 ? __float_as_uint(t) : (uint32_t)(__float_as_int(t) - 0x4B400000);
                        }
                        uint32_t wo[NWO];
                        pack<NFP, QO16>(fb, wo);
                        store_child<NWO, ND>(rw.z, lanebit, row_address(rw) + (unsigned)__popc(rw.z & below) * (NWO * 4u),
                                             wo, er[0][ds & 1][h], es[0], er[ND - 1][ND == 2 ? ds >> 1 : 0][h],
                                             es[ND - 1], um, 1u << s);
                    }
                }
            }
            if (c.out.mult) {                                       // grouping: the records' multiplicities
                const uint32_t mult = c.in.mult[(c.t0 + t0 + lt) * 32 + lane];
                for (int s = 0; s < NS; ++s) {
                    const uint4 rw = s_row[row + s];
                    const unsigned long long i =
                        (row_address(rw) - (unsigned long long)c.out.rec) / (NWO * 4u) + (unsigned)__popc(rw.z & below);
                    if (rw.z & lanebit) c.out.mult[i] = mult;
                }
            }
            if (um) {                                               // rare
                const RecWords<NWI> rwords = rec_words_of<NWI>(w);
                for (unsigned r = um; r; r &= r - 1) {
                    const int s = __ffs(r) - 1, f = s & (NFS - 1), x = s >> KF, ds = DM == 2 ? x << 1 : x;
                    const uint4 rw = s_row[row + s];
                    int3 q = make_int3(0, 0, 0);
                    if (c.precision == 1) {                         // the double-float tier
                        q = snap_df_words<FAM, QI16>(&c, rwords, cl, f, ds, __fmaf_ru(kBandDF, M[0], kBandDFAbs),
                                                     __fmaf_ru(kBandDF, M[ND - 1], kBandDFAbs), QO16 ? 32767.0f : 1.0e9f);
                        ++ndf;
                    }
                    if (!q.z) {                                     // the FP64 definition
                        q = snap64_words<FAM, QI16>(&c, rwords, cl, f, ds);
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
        __syncwarp();                                               // buffer b is free again
    }
    if (nfail >= 0 && lane == 0) {
        // the copies nfail and nfail + 1 (no later one was issued) may still be in flight:
        // wait for them, bounded, before the block's shared memory is released
        for (int n = nfail; n < nfail + (t1 >= 0 ? 2 : 1); ++n)
            if (!mbar_wait(&s_bar[n & 1], (unsigned)(n >> 1) & 1u, GV_SPIN_LIMIT, &c.sc->err)) break;
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

// The tiles whose records the emit pass is going to read, counted apart from it (on request;
// in k_emit_wide itself the count took 0.3 % of a search of affine 4-space): groups of
// kEmitTiles with a cell that has surviving children, or (wide) tiles with something to write.
__global__ void __launch_bounds__(256) k_emit_work(const __grid_constant__ Chunk c, int wide, int tile_bytes) {
    grid_start();
    const int64_t nt = chunk_tiles(c), t = blockIdx.x * 256ll + threadIdx.x;
    const int cell = t < nt ? c.tinfo[t].x : -1;
    bool read = cell >= 0 && (c.alive[cell] & 2);
    if (wide) {
        bool any = false;
        for (int s = 0; read && s < c.ns; ++s)
            any |= c.cbase[(size_t)cell * c.ns + s] != ~0ull && c.ballot[(size_t)t * c.ns + s];
        read &= any;
    } else {
        const unsigned b = __ballot_sync(kFull, read);
        read = t < nt && ((b >> (threadIdx.x & 31u & ~(kEmitTiles - 1u))) & ((1u << kEmitTiles) - 1u));
    }
    const unsigned n = (unsigned)__popc(__ballot_sync(kFull, read));
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(&c.sc->emit_bytes, (unsigned long long)n * (unsigned)tile_bytes);
}

void launch_emit_work(const Chunk &c, int rec_bytes, cudaStream_t st) {
    const int64_t nt = c.t1 - c.t0;
    if (nt > 0)
        launch(k_emit_work, (unsigned)((nt + 255) / 256), 256, 0, st, c, c.P.d > 3, 32 * rec_bytes + 4 * c.ns);
}

template <int FAM, bool QI, bool QO, int KF, int DM>
static void launch_kd(const Chunk &c, cudaStream_t st) {
    if constexpr (KF <= Fam<FAM>::K && DM < (1 << Fam<FAM>::ND) && (KF || DM)) {
        const int64_t ng = (c.t1 - c.t0 + kEmitTiles - 1) / kEmitTiles;
        launch_persistent((const void *)k_emit<FAM, QI, QO, KF, DM>,
                          8 * emit_warp_bytes<rec_words(Fam<FAM>::NFP, QI)>(c.ns), (ng + 7) / 8, c, st);
    }
}

template <int FAM, bool QI, bool QO>
static void launch_fam(const Chunk &c, cudaStream_t st) {
    switch (c.kf * 4 + c.dm) {
    case 1: launch_kd<FAM, QI, QO, 0, 1>(c, st); break;
    case 2: launch_kd<FAM, QI, QO, 0, 2>(c, st); break;
    case 3: launch_kd<FAM, QI, QO, 0, 3>(c, st); break;
    case 4: launch_kd<FAM, QI, QO, 1, 0>(c, st); break;
    case 5: launch_kd<FAM, QI, QO, 1, 1>(c, st); break;
    case 6: launch_kd<FAM, QI, QO, 1, 2>(c, st); break;
    case 7: launch_kd<FAM, QI, QO, 1, 3>(c, st); break;
    case 8: launch_kd<FAM, QI, QO, 2, 0>(c, st); break;
    case 9: launch_kd<FAM, QI, QO, 2, 1>(c, st); break;
    default: break;
    }
}

template <int FAM>
static bool launch_formats(const Chunk &c, cudaStream_t st) {
    const int q = c.lev.q16, qn = c.lev.q16_next;
    if (c.precision == 0 && (q || qn)) return false;    // plain FP64 mode keeps 32-bit records
    if (q && qn) launch_fam<FAM, true, true>(c, st);
    else if (!q && qn) launch_fam<FAM, false, true>(c, st);
    else if (!q && !qn) launch_fam<FAM, false, false>(c, st);
    else return false;                                  // 16-bit to 32-bit: never chosen
    return true;
}

bool launch_emit(const Chunk &c, cudaStream_t st) {
    if (c.t1 <= c.t0) return true;
    switch (c.P.fam) {
    case FAM_LINE2D: return launch_formats<FAM_LINE2D>(c, st);
    case FAM_PLANE3D_SPH: return launch_formats<FAM_PLANE3D_SPH>(c, st);
    case FAM_POSE3DOF: return launch_formats<FAM_POSE3DOF>(c, st);
    case FAM_RAYS3D: return launch_formats<FAM_RAYS3D>(c, st);
    default: return launch_emit_wide(c, st);
    }
}

}  // namespace gv
