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

// Shared memory of one block (8 warps): per warp two buffers of kEmitTiles tiles of
// records, ballots and positions, and the slot rows of the tile at hand (two, by turns).
template <int NW>
__host__ __device__ constexpr size_t emit_warp_bytes(int ns) {
    return 2 * (size_t)kEmitTiles * (32 * NW * 4 + ns * 8) + 2 * 16 * (size_t)ns;
}

// KF: free coordinates that split, DM: dependent coordinates that split (bit mask).
// Each warp takes a contiguous range of groups of kEmitTiles tiles and streams them
// through its own two buffers (bulk copies completing on the warp's mbarriers), so
// warps never wait for each other.
template <int FAM, bool QI16, bool QO16, int KF, int DM>
__global__ void __launch_bounds__(256, 4) k_emit(const __grid_constant__ Chunk c) {
    using F = Fam<FAM>;
    constexpr int ND = F::ND, LE = F::LE, NFP = F::NFP, NFS = 1 << KF, NDS = dep_slots(DM), NS = NFS * NDS;
    constexpr int NWI = rec_words(NFP, QI16), NWO = rec_words(NFP, QO16), RW = 32 * NWI, NG = NFS * ND * LE;
    constexpr int GT = kEmitTiles;
    static_assert(geo32_floats(NFS, ND, LE) <= 32, "a cell's coefficients fit one register per lane");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Level &lev = c.lev;
    extern __shared__ __align__(128) uint8_t s_dyn[];
    uint32_t *s_rec = reinterpret_cast<uint32_t *>(s_dyn + warp * emit_warp_bytes<NWI>(NS));   // [2][GT * RW]
    uint32_t *s_bal = s_rec + 2 * GT * RW;                                                  // [2][GT * NS]
    uint32_t *s_off = s_bal + 2 * GT * NS;                                                  // [2][GT * NS]
    uint4 *s_row = reinterpret_cast<uint4 *>(s_off + 2 * GT * NS);                          // [2][NS]
    __shared__ __align__(8) uint64_t s_bars[8][2];
    uint64_t *s_bar = s_bars[warp];

    const int64_t nt = c.t1 - c.t0, ng = (nt + GT - 1) / GT;
    const int64_t nwarp = (int64_t)gridDim.x * 8, gw = (int64_t)blockIdx.x * 8 + warp;
    const int64_t g0 = gw * ng / nwarp, g1 = (gw + 1) * ng / nwarp;
    if (lane == 0) {
        mbar_init(&s_bar[0], 1);
        mbar_init(&s_bar[1], 1);
        mbar_init_fence();
    }
    __syncwarp();
    auto issue = [&](int64_t g) {                                   // lane 0
        const int b = (int)((g - g0) & 1);
        const int64_t ta = g * GT;
        const int ntl = (int)((ta + GT < nt ? ta + GT : nt) - ta);
        // bulk copies take multiples of 16 bytes (the arrays are padded past the last tile)
        const unsigned rbytes = (unsigned)ntl * RW * 4, bbytes = ((unsigned)ntl * NS * 4 + 15u) & ~15u;
        mbar_expect_tx(&s_bar[b], rbytes + 2 * bbytes);
        bulk_load(s_rec + b * GT * RW, c.in.rec + (c.t0 + ta) * RW, rbytes, &s_bar[b]);
        bulk_load(s_bal + b * GT * NS, c.ballot + ta * NS, bbytes, &s_bar[b]);
        bulk_load(s_off + b * GT * NS, c.off + ta * NS, bbytes, &s_bar[b]);
    };
    // lane k: the cell of tile k of group g (-1: pruned, or past the end)
    auto load_cells = [&](int64_t g) {
        const int64_t t = g * GT + lane;
        return g < g1 && lane < GT && t < nt ? c.tinfo[t].x : -1;
    };
    // a cell's data, one word per lane: coefficient, child's first slot and index
    float pg = 0.0f;
    unsigned long long pbase = ~0ull;
    int pidx = 0;
    auto prefetch = [&](int cell) {
        const int x = cell < 0 ? 0 : cell;
        if (lane < c.gf) pg = __ldg(c.geo32 + (size_t)x * c.gf + lane);
        if (lane < NS) {
            pbase = c.cbase[(size_t)x * NS + lane];
            pidx = c.child_idx[(size_t)x * NS + lane];
        }
    };

    float hs[ND];
#pragma unroll
    for (int j = 0; j < ND; ++j) hs[j] = ((DM >> j) & 1) ? lev.Hs[j] : 0.0f;
    const unsigned below = (1u << lane) - 1u, lanebit = 1u << lane;
    int cur = -1, row = 0;
    float G[NG], Gmax[ND * LE], gexp = 0.0f;
    unsigned long long base = ~0ull;
    int cidx = 0;
#pragma unroll
    for (int i = 0; i < NG; ++i) G[i] = 0.0f;
#pragma unroll
    for (int i = 0; i < ND * LE; ++i) Gmax[i] = 0.0f;
    unsigned nrechk = 0, ndf = 0, bad = 0;
    int64_t gfail = -1;                                             // group whose copy did not arrive
    int cells1 = load_cells(g0);
    if (g0 < g1) {
        if (lane == 0) issue(g0);
        prefetch(__shfl_sync(kFull, cells1, 0));
    }
#pragma unroll 1
    for (int64_t g = g0; g < g1; ++g) {
        const int b = (int)((g - g0) & 1);
        if (lane == 0 && g + 1 < g1) issue(g + 1);
        const int cells = cells1;
        cells1 = load_cells(g + 1);
        const bool ok = mbar_wait(&s_bar[b], (unsigned)(((g - g0) >> 1) & 1), c.spin, &c.sc->err);
        if (!__all_sync(kFull, ok)) {
            gfail = g;
            break;
        }
#pragma unroll 1
        for (int lt = 0; lt < GT; ++lt) {
            const int cl = __shfl_sync(kFull, cells, lt);
            const float g_ = pg;
            const unsigned long long base_ = pbase;
            const int idx_ = pidx;
            {
                const int a = __shfl_sync(kFull, cells, (lt + 1) & (GT - 1)), n1 = __shfl_sync(kFull, cells1, 0);
                prefetch(lt + 1 < GT ? a : n1);
            }
            if (cl < 0) continue;                                   // uniform
            if (cl != cur) {                                        // uniform: a new cell
                cur = cl;
                base = base_;
                cidx = idx_;
#pragma unroll
                for (int i = 0; i < NG; ++i) G[i] = __shfl_sync(kFull, g_, i);
#pragma unroll
                for (int i = 0; i < ND * LE; ++i) Gmax[i] = __shfl_sync(kFull, g_, NG + i);
                gexp = __shfl_sync(kFull, g_, NG + ND * LE);
            }
            const int64_t tt = g * GT + lt;
            // slot rows: output address and passing lanes; the next level's tile -> cell
            // table for the one tile whose first slot this tile may fill
            row ^= NS;
            unsigned bal = 0;
            if (lane < NS) {
                const unsigned long long p0 = base + s_off[b * GT * NS + lt * NS + lane];
                bal = base == ~0ull ? 0u : s_bal[b * GT * NS + lt * NS + lane];
                const unsigned long long q = (p0 + 31) >> 5;
                if (bal && (q << 5) < p0 + (unsigned)__popc(bal)) c.out.tile_cell[q] = (uint32_t)cidx;
                const unsigned long long p = (unsigned long long)(c.out.rec + p0 * NWO);
                s_row[row + lane] = make_uint4((unsigned)p, (unsigned)(p >> 32), bal, 0u);
            }
            const unsigned vmask = __ballot_sync(kFull, bal != 0u);  // child slots this tile writes
            __syncwarp();
            if (!vmask) continue;                                   // uniform: nothing to write
            uint32_t w[NWI];
#pragma unroll
            for (int i = 0; i < NWI; ++i) w[i] = s_rec[b * GT * RW + lt * RW + lane * NWI + i];
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
                    float v = lev.st_ratio_log2[m] ? __fmaf_rn(qt[m], 0.5f, kMagic16) : qt[m] + kMagic16;
                    fb[ND + m] = __float_as_uint(v);
                } else {
                    const int q = field_i<QI16>(w, ND + m);
                    fb[ND + m] = (uint32_t)(lev.st_ratio_log2[m] ? resnap_half(q) : q);
                }
            }
            float es[ND], M[ND];                                    // a snap is certain within es of an integer
            {
                // every term a multiple of 2^ex and M below 2^(24 + ex): the FP32 residual, and
                // the definition's FP64 one, are exact, so a tie rounds to even in both
                const int ex = min(__float2int_rn(gexp), lev.hs_exp);
                const float tq = ex > -100 ? __int_as_float((127 + 24 + ex) << 23) : 0.0f;
                magnitudes<FAM>(qf, qt, Gmax, hs, M);
#pragma unroll
                for (int j = 0; j < ND; ++j) {
                    es[j] = M[j] < tq ? 1.0f : 0.5f - kBandSnap * M[j];
                    if (c.precision == 0) es[j] = -1.0f;            // plain FP64 mode: by the definition
                }
            }
            const uint32_t mult = c.out.mult ? c.in.mult[(c.t0 + tt) * 32 + lane] : 1u;
            unsigned um = 0;                                        // slots whose snap FP32 leaves undecided
#pragma unroll
            for (int f = 0; f < NFS; ++f) {
                float u[ND];
                partial32<FAM>(qf, qt, G, f, u);
                uint32_t sv[ND][2];
                bool so[ND][2];
#pragma unroll
                for (int j = 0; j < ND; ++j)
#pragma unroll
                    for (int v = 0; v < (((DM >> j) & 1) ? 2 : 1); ++v) {
                        const float y = ((DM >> j) & 1) ? (v ? u[j] - hs[j] : u[j] + hs[j]) : u[j];
                        if constexpr (QO16) {
                            // |y| <= 32000: the record passed this level's UB test (finalize_levels)
                            const float t = y + kMagic16;
                            so[j][v] = fabsf(y - (t - kMagic16)) < es[j];
                            sv[j][v] = __float_as_uint(t);
                        } else {
                            const float t = y + kMagic;
                            so[j][v] = fabsf(y - (t - kMagic)) < es[j] && fabsf(y) < 4.0e6f;
                            sv[j][v] = (uint32_t)(__float_as_int(t) - 0x4B400000);
                        }
                    }
#pragma unroll
                for (int x = 0; x < NDS; ++x) {
                    const int s = x * NFS + f, ds = DM == 2 ? x << 1 : x;
                    if (!((vmask >> s) & 1)) continue;              // uniform
                    const uint4 rw = s_row[row + s];
                    bool sure = true;
#pragma unroll
                    for (int j = 0; j < ND; ++j) {
                        fb[j] = sv[j][(ds >> j) & 1];
                        sure &= so[j][(ds >> j) & 1];
                    }
                    uint32_t wo[NWO];
                    pack<NFP, QO16>(fb, wo);
                    const unsigned k = (unsigned)__popc(rw.z & below);
                    uint32_t *op = reinterpret_cast<uint32_t *>(((unsigned long long)rw.y << 32) | rw.x);
                    if (rw.z & lanebit) {
                        store_words<NWO>(op, k, wo);
                        if (!sure) um |= 1u << s;
                        if (c.out.mult) c.out.mult[(op - c.out.rec) / NWO + k] = mult;
                    }
                }
            }
            if (um) {                                               // rare
                const RecWords rwords = rec_words_of<NWI>(w);
                for (unsigned m = um; m; m &= m - 1) {
                    const int s = __ffs(m) - 1, f = s & (NFS - 1), x = s >> KF, ds = DM == 2 ? x << 1 : x;
                    const uint4 rw = s_row[row + s];
                    int3 q = make_int3(0, 0, 0);
                    if (c.precision == 1) {                         // the double-float tier
                        q = snap_df_words<FAM, QI16>(&c.lev, rwords, c.geo32 + (size_t)cl * c.gf + f * ND * LE,
                                                     c.geo32lo + ((size_t)cl * NFS + f) * ND * LE, ds,
                                                     __fmaf_ru(kBandDF, M[0], kBandDFAbs),
                                                     __fmaf_ru(kBandDF, M[ND - 1], kBandDFAbs), QO16 ? 32767.0f : 1.0e9f);
                        ++ndf;
                    }
                    if (!q.z) {                                     // the FP64 definition
                        q = snap64_words<FAM, QI16>(&c.P, &c.lev, rwords,
                                                    c.geo64 + ((size_t)cl * NFS + f) * F::NB, ds, c.dm);
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
                    store_words<NWO>(reinterpret_cast<uint32_t *>(((unsigned long long)rw.y << 32) | rw.x),
                                     (unsigned)__popc(rw.z & below), wo);
                }
            }
        }
        __syncwarp();                                               // buffer b is free again
    }
    if (gfail >= 0 && lane == 0) {
        // the copies of groups gfail and gfail + 1 (no later one was issued) may still
        // be in flight: wait for them, bounded, before the block's shared memory is
        // released
        const int64_t ge = gfail + 2 < g1 ? gfail + 2 : g1;
        for (int64_t g = gfail; g < ge; ++g) {
            const int b = (int)((g - g0) & 1);
            if (!mbar_wait(&s_bar[b], (unsigned)(((g - g0) >> 1) & 1), GV_SPIN_LIMIT, &c.sc->err)) break;
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
