// gv_tile.cuh -- device code shared by the count and emit passes of the proximity
// test (the surface-box test of Sec. 3.2, "eps plus the cell radius", over every
// (canonical record, child cell) pair).
//
// A tile is 32 consecutive records of one cell, one record per lane of a warp; warps take
// runs of consecutive tiles (CellWatch in the count pass, units by turns in the emit pass),
// so that most of a run lies in one cell.
#pragma once
#include <type_traits>

#include "gv_kernels.h"

namespace gv {

constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------------------
// Bulk asynchronous copies (global -> shared) completing on an mbarrier: the emit
// pass streams its records through shared memory, two groups of tiles per warp in
// flight.  Every wait is bounded: after Chunk::spin unsuccessful polls the kernel
// records kErrTimeout and stops (the host maps it to VOTE_ETIMEOUT).
// ---------------------------------------------------------------------------
constexpr unsigned kErrTimeout = 0x100u;
#ifndef GV_SPIN_LIMIT
#define GV_SPIN_LIMIT (1u << 22)
#endif

__device__ __forceinline__ unsigned smem_u32(const void *p) {
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// make the initialised barriers visible to the asynchronous (bulk copy) proxy
__device__ __forceinline__ void mbar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// bytes: a multiple of 16; both addresses 16-byte aligned
__device__ __forceinline__ void bulk_load(void *dst, const void *src, unsigned bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for phase `parity` of a barrier; false (and the error bit set) if
// it did not complete within the limit.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity, unsigned limit, unsigned *err) {
    for (unsigned it = 0; it < limit; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    atomicOr(err, kErrTimeout);
    return false;
}

// 2^23 + 2^22: adding it to a float y with |y| < 2^22 rounds y to the nearest
// integer (ties to even) and leaves that integer in the low mantissa bits.
constexpr float kMagic = 12582912.0f;
// kMagic + 2^15: the same, with the integer biased by 2^15 (the 16-bit field format)
constexpr float kMagic16 = 12615680.0f;

template <int NW>
__device__ __forceinline__ void load_words(const uint32_t *base, int64_t r, uint32_t *w) {
    const uint32_t *p = base + r * NW;
    if constexpr (NW == 1) {
        w[0] = p[0];
    } else if constexpr (NW == 2) {
        uint2 v = *reinterpret_cast<const uint2 *>(p);
        w[0] = v.x; w[1] = v.y;
    } else {
        static_assert(NW % 4 == 0, "record words");
#pragma unroll
        for (int i = 0; i < NW; i += 4) {
            uint4 v = *reinterpret_cast<const uint4 *>(p + i);
            w[i] = v.x; w[i + 1] = v.y; w[i + 2] = v.z; w[i + 3] = v.w;
        }
    }
}

template <int NW>
__device__ __forceinline__ void store_words(uint32_t *base, int64_t r, const uint32_t *w) {
    uint32_t *p = base + r * NW;
    if constexpr (NW == 1) {
        p[0] = w[0];
    } else if constexpr (NW == 2) {
        *reinterpret_cast<uint2 *>(p) = make_uint2(w[0], w[1]);
    } else {
#pragma unroll
        for (int i = 0; i < NW; i += 4) *reinterpret_cast<uint4 *>(p + i) = make_uint4(w[i], w[i + 1], w[i + 2], w[i + 3]);
    }
}

// The emit pass's slot rows: (output address, passing lanes) of one child slot of a tile.
__device__ __forceinline__ unsigned long long row_address(const uint4 &rw) {
    return ((unsigned long long)rw.y << 32) | rw.x;
}

// A record's words to a global address, if this lane passes (bal & lanebit), and the slot's
// bit into um if it passes and its snap is not certain (|e0| >= es0 or |e1| >= es1; e1 is
// unused with one dependent coordinate): one predicate, one predicated store, no branch.
template <int NW, int ND>
__device__ __forceinline__ void store_child(unsigned bal, unsigned lanebit, unsigned long long p, const uint32_t *w,
                                            float e0, float es0, float e1, float es1, unsigned &um, unsigned bit) {
    static_assert(NW == 1 || NW == 2 || NW == 4, "records of at most four words");
    const float x0 = fabsf(e0), x1 = fabsf(e1);
#define GV_STORE_CHILD(ST, ...)                                                                                \
    if constexpr (ND == 1)                                                                                     \
        asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b32 t;\n\tand.b32 t, %1, %2;\n\tsetp.ne.u32 p, t, 0;\n\t" ST    \
                     "setp.ge.and.f32 q, %4, %5, p;\n\t@q or.b32 %0, %0, %6;\n\t}"                              \
                     : "+r"(um)                                                                                \
                     : "r"(bal), "r"(lanebit), "l"(p), "f"(x0), "f"(es0), "r"(bit), "f"(x1), "f"(es1), __VA_ARGS__ \
                     : "memory");                                                                              \
    else                                                                                                       \
        asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b32 t;\n\tand.b32 t, %1, %2;\n\tsetp.ne.u32 p, t, 0;\n\t" ST    \
                     "setp.ge.f32 q, %4, %5;\n\tsetp.ge.or.f32 q, %7, %8, q;\n\tand.pred q, q, p;\n\t"          \
                     "@q or.b32 %0, %0, %6;\n\t}"                                                              \
                     : "+r"(um)                                                                                \
                     : "r"(bal), "r"(lanebit), "l"(p), "f"(x0), "f"(es0), "r"(bit), "f"(x1), "f"(es1), __VA_ARGS__ \
                     : "memory")
    if constexpr (NW == 1) {
        GV_STORE_CHILD("@p st.global.u32 [%3], %9;\n\t", "r"(w[0]));
    } else if constexpr (NW == 2) {
        GV_STORE_CHILD("@p st.global.v2.u32 [%3], {%9, %10};\n\t", "r"(w[0]), "r"(w[1]));
    } else {
        GV_STORE_CHILD("@p st.global.v4.u32 [%3], {%9, %10, %11, %12};\n\t", "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]));
    }
#undef GV_STORE_CHILD
}

// one record's words to a global address where on != 0 (predicated stores, no branch)
template <int NW>
__device__ __forceinline__ void store_words_if(unsigned on, unsigned long long p, const uint32_t *w) {
    if constexpr (NW == 1) {
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.global.u32 [%1], %2;\n\t}" ::"r"(on), "l"(p),
                     "r"(w[0])
                     : "memory");
    } else if constexpr (NW == 2) {
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.global.v2.u32 [%1], {%2, %3};\n\t}" ::"r"(on),
                     "l"(p), "r"(w[0]), "r"(w[1])
                     : "memory");
    } else {
#pragma unroll
        for (int i = 0; i < NW; i += 4)
            asm volatile(
                "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.global.v4.u32 [%1], {%2, %3, %4, %5};\n\t}" ::"r"(on),
                "l"(p + 4u * i), "r"(w[i]), "r"(w[i + 1]), "r"(w[i + 2]), "r"(w[i + 3])
                : "memory");
    }
}

// Field i of a record as a float (exact: 16-bit fields always, 32-bit fields below 2^24).
template <bool Q16>
__device__ __forceinline__ float field_f(const uint32_t *w, int i) {
    if constexpr (Q16) {
        unsigned b = __byte_perm(w[i >> 1], 0x4B40u, (i & 1) ? 0x5432u : 0x5410u);
        return __int_as_float((int)b) - kMagic16;
    } else {
        return (float)(int32_t)w[i];
    }
}

template <bool Q16>
__device__ __forceinline__ int field_i(const uint32_t *w, int i) {
    if constexpr (Q16) return (int)((w[i >> 1] >> (16 * (i & 1))) & 0xffffu) - 32768;
    else return (int32_t)w[i];
}

// Pack NFP field values into record words.  fb[i]: for 16-bit records the low 16
// bits hold the biased field, for 32-bit records the field itself.
template <int NFP, bool Q16>
__device__ __forceinline__ void pack(const uint32_t *fb, uint32_t *w) {
    if constexpr (Q16) {
#pragma unroll
        for (int i = 0; i < NFP / 2; ++i) w[i] = __byte_perm(fb[2 * i], fb[2 * i + 1], 0x5410u);
    } else {
#pragma unroll
        for (int i = 0; i < NFP; ++i) w[i] = fb[i];
    }
}

// round half to even of q/2: re-snap of an essential parameter when its step doubles
__device__ __forceinline__ int32_t resnap_half(int32_t q) {
    int32_t k = q >> 1;
    return k + ((q & 1) & (k & 1));
}

// ---------------------------------------------------------------------------
// The count pass's way through a step's tiles, and cells it leaves early.
//
// A child whose records can no longer reach the threshold is pruned whatever the rest of
// its cell's records give, so a cell is left once that is certain of all its children: once
// each has more certain failures than the cell's allowance (records minus threshold).  A
// share (1 - threshold / N) / (1 - largest child / N) of a cell's N records settles that,
// and the levels that hold most records are those whose cells lie just above the
// threshold: of all records a search opens, planes of 1e4 points need 0.50, of 1e6 points
// 0.59, affine 4-space 0.36, point sets 0.66, radial 0.42; with whole batches and units
// 0.65, 0.70, 0.48, 0.79 and 0.64 are tested.  The surviving children's counts, and with
// them the search, are the same.  GB300, count passes and tile scans: planes of 1e6 points
// 275 -> 225 ms, of 1e4 points 9.9 -> 8.3, affine 25.8 -> 20.4, radial 6.1 -> 5.1 (steps of
// 2^23 records in the last two).
// ---------------------------------------------------------------------------

// Warps take units of consecutive tiles: the first tickets, one per warp, are the first
// units of equal parts of the step, the next ones the second units, and so on.  So few
// warps are in one cell at a time, and those that leave cells early take more tickets.
// Few tiles, or no early leaving: one unit per warp.
//
// Ballots are staged in shared memory, a batch of 32 / ns tiles at a time (one tile with 32 or
// more child slots), and stored from there by all lanes; a batch's words are also counted
// there, lane s of every ns for child slot s (and 32 + s).  Most of this work is a batch's, and
// little a tile's: the pass is bound by instruction issue.
template <int V, bool LB>
struct CellWatch {
    // a warp's shared memory: rows of a batch (with LB those of the lower bounds after them), the
    // step's units and their size, the tiles and records that it has left
    static constexpr int UNITS = LB ? 64 * V : 32 * V, SIZE = UNITS + 1, TILES = UNITS + 2, RECORDS = UNITS + 3,
                         WORDS = UNITS + 4;
    uint32_t *s;
    // the run of tiles at hand: its decided records, those of them that passed (per lane), both
    // since it began or since they were added up; more decided records than lim are looked at
    unsigned cnt, pass[V], lim;

    __device__ __forceinline__ static unsigned allowance(int2 ti) { return ((unsigned)ti.y >> kAllowShift) * 8u; }
    __device__ __forceinline__ static bool watched(int2 ti) { return (unsigned)ti.y >> kAllowShift != kAllowNone; }
    __device__ __forceinline__ static int after(int2 ti) { return (ti.y >> kLeftShift) & kLeftMax; }

    // The step's units of nt tiles, and this warp's first (its ticket is the warp's number):
    // tiles [tt, tb), none if tt >= tb.
    __device__ __forceinline__ void split(const Chunk &c, unsigned nt, unsigned warp, int lane, unsigned &tt,
                                          unsigned &tb) {
        const unsigned W = gridDim.x * 8u, per = (nt + W - 1u) / W;
        unsigned size = per, S = 1u;
        if (c.early && per >= 16u) {
            size = per >= 512u ? 64u : (per >= 256u ? 32u : (per >= 32u ? 16u : 8u));
            S = (per + size - 1u) / size;
        }
        if (lane == 0) {
            s[UNITS] = S;
            s[SIZE] = size;
            s[TILES] = s[RECORDS] = 0u;
        }
        const unsigned long long at = (unsigned long long)warp * S * size;
        tt = at < nt ? (unsigned)at : nt;
        tb = nt - tt < size ? nt : tt + size;
        __syncwarp();
    }
    // tiles of a later ticket's unit; false: there is none
    __device__ __forceinline__ bool unit(unsigned ticket, unsigned nt, unsigned &tt, unsigned &tb) const {
        const unsigned W = gridDim.x * 8u, S = s[UNITS], size = s[SIZE];
        if (S <= 1u || ticket / W >= S) return false;
        const unsigned long long at = ((unsigned long long)(ticket % W) * S + ticket / W) * size;
        tt = at < nt ? (unsigned)at : nt;
        tb = nt - tt < size ? nt : tt + size;
        return true;
    }
    // asks for the next ticket (lane 0 has it)
    __device__ __forceinline__ unsigned next(const Chunk &c, int lane) const {
        const unsigned W = gridDim.x * 8u;
        return s[UNITS] > 1u && lane == 0 ? W + atomicAdd(&c.sc->ticket, 1u) : 0xffffffffu;
    }

    // a run of tiles begins with tile ti
    __device__ __forceinline__ void run(int2 ti) {
        cnt = 0u;
#pragma unroll
        for (int v = 0; v < V; ++v) pass[v] = 0u;
        lim = !watched(ti) ? 0xffffffffu : ((ti.y & kTileOwned) ? allowance(ti) : 511u);
    }
    // lane 0: n tiles of ti's cell from tile tt on are left (none: ti is its last)
    __device__ __forceinline__ void leave(const Chunk &c, int2 ti, unsigned tt, unsigned n) {
        c.alive[ti.x] = 0;
        if (!c.work || n == 0u) return;
        const int64_t cell = c.in_c0 + ti.x;
        const int64_t rest = (int64_t)c.in_rbeg[cell] + c.in_rcnt[cell] - 32 * (c.t0 + tt);
        s[TILES] += n;
        s[RECORDS] += rest < 32ll * n ? (unsigned)rest : 32u * n;
    }
    // The warp is done: what it has left (nw: words of a record).
    __device__ __forceinline__ void report(const Chunk &c, int nw, int lane) const {
        if (!c.work || lane != 0 || s[TILES] == 0u) return;
        atomicAdd(&c.sc->left_tests, (unsigned long long)s[RECORDS] << c.lns);
        atomicAdd(&c.sc->left_bytes, (unsigned long long)s[TILES] * 4u * (unsigned)(32 * nw + c.ns));
    }
    // A unit [tt, tb) begins with tile ti: how many tiles of its cell are not this unit's (all, if
    // the cell is the warp's that has its first tile, or if others know that it can be left).
    __device__ __forceinline__ unsigned begin(const Chunk &c, int ns, int2 ti, unsigned tt, unsigned tb, int lane) {
        if (ti.x < 0 || (ti.y & kTileFirst)) return 0u;
        if (ti.y & kTileOwned) return 1u + after(ti);
        if (!watched(ti)) return 0u;
        const uint32_t *p = c.cfail + (size_t)ti.x * ns + (lane & (ns - 1));
        bool d = true;
#pragma unroll
        for (int v = 0; v < V; ++v)
            if (v == 0 || ns > 32) d &= __ldcg(p + 32 * v) > allowance(ti);
        if (!__all_sync(kFull, d)) return 0u;
        const unsigned n = 1u + after(ti);
        if (lane == 0) leave(c, ti, tt, n < tb - tt ? n : tb - tt);
        return n;
    }
    // A batch's ballots (word[v]: the lane's, 0 past its end) have been stored; its rows from
    // `first` on belong to the last run.
    __device__ __forceinline__ void add(int ns, int lns, const unsigned *word, int first, int lane) {
#pragma unroll
        for (int v = 0; v < V; ++v)
            if ((v == 0 || ns > 32) && lane >> lns >= first) pass[v] += (unsigned)__popc(word[v]);
    }
    // After the batch whose last tile ti is tile tt - 1, when cnt exceeds lim or the unit ends
    // (tb; a cell that is this warp's moves it): how many of the tiles from tt on need not be
    // counted.
    __device__ __forceinline__ unsigned look(const Chunk &c, int ns, int2 ti, unsigned tt, unsigned &tb, int lane) {
        if (ti.x < 0) return 0u;
        const unsigned rest = after(ti), allow = allowance(ti);
        const bool owned = ti.y & kTileOwned;
        if (owned && tt >= tb) tb = tt + rest;
        if (!watched(ti)) return 0u;
        bool d = true;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            if (v > 0 && ns <= 32) continue;
            unsigned f = pass[v];
            for (int o = ns; o < 32; o <<= 1) f += __shfl_xor_sync(kFull, f, o);
            f = cnt - f;
            if (!owned) {                                // others count the cell too: all failures are added up
                if (lane < ns) f += atomicAdd(c.cfail + (size_t)ti.x * ns + lane + 32 * v, f);
                f = __shfl_sync(kFull, f, lane & (ns - 1));             // modulo 32
                pass[v] = 0u;
            }
            d &= f > allow;
        }
        if (!owned) cnt = 0u;
        if (!__all_sync(kFull, d)) return 0u;
        if (lane == 0) leave(c, ti, tt, owned || rest < tb - tt ? rest : tb - tt);
        return rest;
    }
};

// ---------------------------------------------------------------------------
// Cell geometry: the changes of the basis values from a cell's centre to its children's.
// ---------------------------------------------------------------------------

// entry of a rotation table: the packed coordinates of a cell of the rotation
// coordinates 0..2 at level l
__device__ __forceinline__ int64_t rot_entry(const Problem &P, int l, const int64_t *ix) {
    return (((ix[0] << splits_at(P, l, 1)) | ix[1]) << splits_at(P, l, 2)) | ix[2];
}

// coordinates (of those the stored basis values depend on) of the cell itself or of the
// child of geometry slot r
template <int FAM>
__device__ __forceinline__ void geo_coords(const Chunk &c, uint64_t key, int r, bool child, int64_t *ix) {
    using F = Fam<FAM>;
    constexpr int NC = F::LINEAR_TAIL ? F::K - 1 : F::K;
    int bits = r;
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        ix[j] = cell_coord(c.P, key, c.lev.l, j);
        if (child && ((c.lev.split_mask >> j) & 1)) {
            ix[j] = 2 * ix[j] + (bits & 1);
            bits >>= 1;
        }
    }
}

// the stored basis values at a cell (level l: half-widths h) of these coordinates.  TAB: the
// tables hold them (else they are evaluated where there is no table).
template <int FAM, bool TAB>
__device__ __forceinline__ void geo_basis(const Chunk &c, int l, const double *h, const double *rot, const int64_t *ix,
                                          double *psi) {
    using F = Fam<FAM>;
    if constexpr (F::LINEAR_TAIL) {
        double R[9];
        if (TAB || rot) {
            const double *p = rot + 9 * rot_entry(c.P, l, ix);
#pragma unroll
            for (int m = 0; m < F::NBG; ++m) psi[m] = p[m];
            return;
        }
        double ph[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) ph[j] = cell_center(c.P, h, j, ix[j]);
        Fam<FAM_POSE6DOF>::rotation(c.P, ph, R);
#pragma unroll
        for (int m = 0; m < F::NBG; ++m) psi[m] = R[m];
    } else {
        constexpr int NC = F::K;
        double sn[2], cs[2];
        static_assert(FAM == FAM_PLANE3D_SPH || FAM == FAM_POSE3DOF, "angular coordinates");
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            if (TAB || c.sincos[j]) {
                const double2 v = c.sincos[j][(1ll << splits_at(c.P, l, j)) - 1 + ix[j]];
                sn[j] = v.x;
                cs[j] = v.y;
            } else {
                vsincos(cell_center(c.P, h, j, ix[j]), &sn[j], &cs[j]);
            }
        }
        if constexpr (FAM == FAM_PLANE3D_SPH) {     // as Fam::basis
            psi[0] = dmul(sn[0], cs[1]);
            psi[1] = dmul(sn[0], sn[1]);
            psi[2] = cs[0];
        } else {
            psi[0] = cs[0];
            psi[1] = sn[0];
        }
    }
}

// changes of the stored basis values for geometry slot r
template <int FAM, bool TAB>
__device__ __forceinline__ void geo_change(const Chunk &c, uint64_t key, int r, double *d) {
    using F = Fam<FAM>;
    int64_t ix[3];
    double par[F::NBG], ch[F::NBG];
    geo_coords<FAM>(c, key, r, false, ix);
    geo_basis<FAM, TAB>(c, c.lev.l, c.lev.h, c.rot_par, ix, par);
    geo_coords<FAM>(c, key, r, true, ix);
    geo_basis<FAM, TAB>(c, c.lev.l + 1, c.lev.h1, c.rot_ch, ix, ch);
#pragma unroll
    for (int m = 0; m < F::NBG; ++m) d[m] = dsub(ch[m], par[m]);
}

// changes of all basis values for free slot fs (the definition's)
template <int FAM, bool TAB>
__device__ __forceinline__ void cell_change(const Chunk &c, uint64_t key, int fs, double *d) {
    using F = Fam<FAM>;
    if constexpr (F::LINEAR_BASIS) {
        // psi is the free coordinates themselves: their changes are the exact child shifts
        int bits = fs;
#pragma unroll
        for (int m = 0; m < F::NB; ++m) {
            const bool split = (c.lev.split_mask >> m) & 1;
            d[m] = split ? ((bits & 1) ? c.lev.h1[m] : -c.lev.h1[m]) : 0.0;
            if (split) bits >>= 1;
        }
    } else {
        geo_change<FAM, TAB>(c, key, fs & (c.ng - 1), d);
        if constexpr (F::LINEAR_TAIL) {
            // the last basis value is the last free coordinate: its change is the exact shift
            constexpr int j = F::K - 1;
#pragma unroll
            for (int m = F::NBG; m < F::NB - 1; ++m) d[m] = 0.0;    // not used by the family
            d[F::NB - 1] = ((c.lev.split_mask >> j) & 1) ? ((fs >> c.kg) ? c.lev.h1[j] : -c.lev.h1[j]) : 0.0;
        }
    }
}

// the same of a chunk's cell, from its FP64 geometry where that is kept (plain FP64 mode,
// and where there are no tables: so the rare paths hold no evaluation)
template <int FAM>
__device__ __forceinline__ void chunk_change(const Chunk &c, int cell, int fs, double *d) {
    using F = Fam<FAM>;
    if (c.geo64) {
#pragma unroll
        for (int m = 0; m < F::NB; ++m) d[m] = c.geo64[((size_t)cell * c.nfs + fs) * F::NB + m];
    } else {
        cell_change<FAM, true>(c, c.cells.key[c.c0 + cell], fs, d);
    }
}

// FP32 change of basis value b for free slot f where it does not depend on the cell (a
// linear basis or tail coordinate), and what the rounding leaves
template <int FAM>
__device__ __forceinline__ float lin_change(const Chunk &c, int b, int f, bool low) {
    using F = Fam<FAM>;
    const int j = F::LINEAR_TAIL ? F::K - 1 : b;
    if (!((c.lev.split_mask >> j) & 1)) return 0.0f;
    const float h = low ? c.lev.h1f_lo[j] : c.lev.h1f[j];
    return (f >> __popc(c.lev.split_mask & ((1 << j) - 1))) & 1 ? h : -h;
}

// the screen's coefficient of t_m in residual j from the change of its basis value
template <int FAM>
__device__ __forceinline__ float coef32(const Level &lev, int j, int m, float d) {
    return (Fam<FAM>::cneg(j, m) ? -d : d) * lev.gs[j][m];
}

// ---------------------------------------------------------------------------
// Exact FP64 definition (the recheck of the screen, and the plain FP64 mode).
// ---------------------------------------------------------------------------

// UB radius R_j = ((eps_j + h1_j) + sum_i lam_ji h1_i) + A1_j, in this order.
template <int FAM>
__device__ __forceinline__ void radius64(const Level &lev, const double *t, double *R) {
    using F = Fam<FAM>;
    double lam[F::ND * F::K];
    F::lipschitz64(t, lam);
#pragma unroll
    for (int j = 0; j < F::ND; ++j) {
        double r = lev.Rbase[j];
#pragma unroll
        for (int i = 0; i < F::K; ++i) r = dadd(r, dmul(lam[j * F::K + i], lev.h1[i]));
        R[j] = dadd(r, lev.A1[j]);
    }
}

// shift of dependent coordinate j for the dependent bits ds of a child (dm: the
// dependent coordinates that split; bit j of ds is 0 where j does not)
template <int FAM>
__device__ __forceinline__ double dep_shift64(const Level &lev, int j, int ds, int dm) {
    constexpr int K = Fam<FAM>::K;
    return ((dm >> j) & 1) ? (((ds >> j) & 1) ? lev.h1[K + j] : -lev.h1[K + j]) : 0.0;
}

// the child slot of free slot f and dependent bits ds (a subset of dm, at most two bits)
__device__ __forceinline__ int child_slot(int f, int ds, int dm, int kf) { return f | ((dm == 2 ? ds >> 1 : ds) << kf); }

template <int FAM>
__device__ __forceinline__ void shifts64(const Level &lev, int s, double *sh) {
    using F = Fam<FAM>;
#pragma unroll
    for (int j = 0; j < F::D; ++j) {
        bool split = (lev.split_mask >> j) & 1;
        sh[j] = split ? (((s >> j) & 1) ? lev.h1[j] : -lev.h1[j]) : 0.0;
    }
}

// exact FP64 test of one (record, child): bit 0 UB pass, bit 1 LB pass; fo = the
// record's residual at the child centre
template <int FAM>
__device__ __forceinline__ int test64(const Level &lev, const double *f, const double *t, const double *R,
                                      const double *dpsi, int s, double *fo) {
    using F = Fam<FAM>;
    double sh[F::D];
    shifts64<FAM>(lev, s, sh);
    F::residual64(f, t, dpsi, sh, fo);
    int ub = 1, lb = 1;
#pragma unroll
    for (int j = 0; j < F::ND; ++j) {
        double a = fabs(fo[j]);
        ub &= a <= R[j];
        lb &= a <= lev.rlb[j];
    }
    return ub | (lb << 1);
}

// pass masks: one bit per child slot
template <int FAM>
using SlotMask = typename std::conditional<((1 << Fam<FAM>::D) > 32), unsigned long long, unsigned>::type;

// UB/LB pass masks of one record (integer fields) against the child slots of free slots
// [fs0, fs1), exactly
// as the definition evaluates them.
template <int FAM>
__device__ __forceinline__ void eval64(const Chunk &c, int cell, const int *qf, const int *qt, int fs0, int fs1,
                                       SlotMask<FAM> &ubm, SlotMask<FAM> &lbm) {
    using F = Fam<FAM>;
    const Problem &P = c.P;
    const Level &lev = c.lev;
    const int kf = c.kf, dm = c.dm;
    using Mask = SlotMask<FAM>;
    static_assert(F::ND <= 2, "two dependent coordinates at most");
    double f[F::ND], t[F::LE], R[F::ND];
#pragma unroll
    for (int j = 0; j < F::ND; ++j) f[j] = dmul((double)qf[j], P.s_f[j]);
#pragma unroll
    for (int m = 0; m < F::LE; ++m) t[m] = dmul((double)qt[m], lev.s_t[m]);
    radius64<FAM>(lev, t, R);
    ubm = 0;
    lbm = 0;
#pragma unroll 1
    for (int fs = fs0; fs < fs1; ++fs) {
        double pr[F::ND], d[F::NB];
        chunk_change<FAM>(c, cell, fs, d);
        F::partial64(f, t, d, pr);
#pragma unroll
        for (int ds = 0; ds < (1 << F::ND); ++ds) {
            if (ds & ~dm) continue;
            int ub = 1, lb = 1;
#pragma unroll
            for (int j = 0; j < F::ND; ++j) {
                double a = fabs(dsub(pr[j], dep_shift64<FAM>(lev, j, ds, dm)));
                ub &= a <= R[j];
                lb &= a <= lev.rlb[j];
            }
            const int s = child_slot(fs, ds, dm, kf);
            ubm |= (Mask)ub << s;
            lbm |= (Mask)lb << s;
        }
    }
}

// Record words passed by value to the out-of-line FP64 helpers below (so that the
// caller's arrays stay in registers).
template <int NW>
struct RecWords {
    uint32_t w[NW];
};

template <int NW>
__device__ __forceinline__ RecWords<NW> rec_words_of(const uint32_t *w) {
    RecWords<NW> r;
#pragma unroll
    for (int i = 0; i < NW; ++i) r.w[i] = w[i];
    return r;
}

// Exact FP64 snap of one record's free parameters at a child centre (free slot fs,
// dependent bits ds), out of line (the FP32 path needs it rarely): the snapped values
// (x, y: dependent coordinates 0 and 1) and z != 0 if a value leaves the representable
// range.
template <int FAM, bool Q16>
__device__ __noinline__ int3 snap64_words(const Chunk *c, RecWords<rec_words(Fam<FAM>::NFP, Q16)> rw, int cell, int fs, int ds) {
    using F = Fam<FAM>;
    static_assert(F::ND <= 2, "two dependent coordinates at most");
    const Problem *P = &c->P;
    const Level *lev = &c->lev;
    const int dm = c->dm;
    double f[F::ND], t[F::LE], pr[F::ND], g64[F::NB];
    chunk_change<FAM>(*c, cell, fs, g64);
#pragma unroll
    for (int j = 0; j < F::ND; ++j) f[j] = dmul((double)field_i<Q16>(rw.w, j), P->s_f[j]);
#pragma unroll
    for (int m = 0; m < F::LE; ++m) t[m] = dmul((double)field_i<Q16>(rw.w, F::ND + m), lev->s_t[m]);
    F::partial64(f, t, g64, pr);
    int bad = 0, qn[2] = {0, 0};
#pragma unroll
    for (int j = 0; j < F::ND; ++j) {
        double q = rint(dmul(dsub(pr[j], dep_shift64<FAM>(*lev, j, ds, dm)), P->inv_s_f[j]));
        bad |= !(fabs(q) < 1073741824.0);
        qn[j] = bad ? 0 : (int)q;
    }
    return make_int3(qn[0], qn[1], bad);
}

// ---------------------------------------------------------------------------
// Double-float tier.  An integer field as an unevaluated sum hi + lo of two FP32
// values (exact for |q| < 2^31: |q - hi| <= 2^6), and Knuth's two-sum.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void split_int(int q, float &hi, float &lo) {
    hi = __int2float_rn(q);
    lo = __int2float_rn(q - __float2int_rz(hi));
}

__device__ __forceinline__ float two_sum(float a, float b, float &err) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}

// The snap of one record's dependent coordinates at a child centre (free slot fs,
// dependent bits ds), from the residual q_f,j + sum_m q_t,m G64[j][m] -+ h1_j / s_f,j
// evaluated as a double-float (G64 = Gh + Gl, the slot's coefficients and their remainders):
// (x, y) the snapped values, z = 1 when both are decided (the value is more than
// bd_j away from a rounding tie and below lim in magnitude), else 0 (the FP64
// definition decides).  Out of line: the FP32 screen needs it rarely.
template <int FAM, bool Q16>
__device__ __noinline__ int3 snap_df_words(const Chunk *c, RecWords<rec_words(Fam<FAM>::NFP, Q16)> rw, int cell,
                                           int fs, int ds, float bd0, float bd1, float lim) {
    using F = Fam<FAM>;
    static_assert(F::ND <= 2, "two dependent coordinates at most");
    const Level *lev = &c->lev;
    const int r = fs & (c->ng - 1);
    int qn[2] = {0, 0}, ok = 1;
#pragma unroll
    for (int j = 0; j < F::ND; ++j) {
        float hi, lo;
        split_int(field_i<Q16>(rw.w, j), hi, lo);
#pragma unroll
        for (int m = 0; m < F::LE; ++m) {
            if (!F::uses(j, m)) continue;
            float th, tl;
            split_int(field_i<Q16>(rw.w, F::ND + m), th, tl);
            const int b = F::cb(j, m);
            float dh, dl;
            if (b < F::NBG) {
                dh = c->geo32[(size_t)cell * c->gf + b * c->ng + r];
                dl = c->geo32lo[((size_t)cell * F::NBG + b) * c->ng + r];
            } else {
                dh = lin_change<FAM>(*c, b, fs, false);
                dl = lin_change<FAM>(*c, b, fs, true);
            }
            const float gh = coef32<FAM>(*lev, j, m, dh), gl = coef32<FAM>(*lev, j, m, dl);
            const float p = __fmul_rn(th, gh);
            const float e = __fmaf_rn(th, gh, -p);                  // th gh = p + e exactly
            float err;
            hi = two_sum(hi, p, err);
            lo = __fadd_rn(lo, __fadd_rn(err, __fmaf_rn(tl, gl, __fmaf_rn(th, gl, __fmaf_rn(tl, gh, e)))));
        }
        if ((lev->split_mask >> (F::K + j)) & 1) {
            // the residual at the child centre: partial - h1 when the dependent bit is set
            const bool up = (ds >> j) & 1;
            const float h = up ? -lev->Hs[j] : lev->Hs[j], hl = up ? -lev->Hs_lo[j] : lev->Hs_lo[j];
            float err;
            hi = two_sum(hi, h, err);
            lo = __fadd_rn(lo, __fadd_rn(err, hl));
        }
        const float r = rintf(hi);                                  // hi - r is exact
        const float w = __fadd_rn(__fsub_rn(hi, r), lo);
        const float k = rintf(w);
        const float fr = __fsub_rn(w, k);
        ok &= (int)(fabsf(hi) < lim) & (int)(0.5f - fabsf(fr) > (j ? bd1 : bd0));
        qn[j] = ok ? __float2int_rn(r) + __float2int_rn(k) : 0;
    }
    return make_int3(qn[0], qn[1], ok);
}

// ---------------------------------------------------------------------------
// FP32 screen (in steps of s_f).
// ---------------------------------------------------------------------------

// The magnitudes the snap's band scales with (steps): M_j = |q_f,j| + |H_j| +
// sum_m |q_t,m| Gmax_jm, Gmax = the cell's largest |G| per (j, m).
template <int FAM>
__device__ __forceinline__ void magnitudes(const float *qf, const float *qt, const float *Gmax, const float *hs,
                                           float *M) {
    using F = Fam<FAM>;
#pragma unroll
    for (int j = 0; j < F::ND; ++j) {
        float v = fabsf(qf[j]) + hs[j];
#pragma unroll
        for (int m = 0; m < F::LE; ++m)
            if (F::uses(j, m)) v = __fmaf_ru(fabsf(qt[m]), Gmax[j * F::LE + m], v);
        M[j] = v;
    }
}

// Two FP32 values in one 64-bit register: the packed FP32 operations of sm_100+ (each
// half rounded as the scalar operation), two for one issue slot.
typedef unsigned long long f2;
__device__ __forceinline__ f2 f2_make(float x, float y) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ void f2_get(f2 v, float &x, float &y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v)); }
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// min(|a|, |b|, |c|)
__device__ __forceinline__ float min3_abs(float a, float b, float c) {
    float r;
    asm("min.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

__device__ __forceinline__ f2 f2_dup(float x) { return f2_make(x, x); }

// The screen's decisions on a pair of residuals y = (y0, y1) of one dependent coordinate
// against the squared radius: y^2 - R^2 < 0, by its sign; the smallest |y^2 - R^2| of the
// record goes into near, which leaves the record undecided when it falls below its band:
// one packed multiply-add, two compares and one minimum for two tests.
__device__ __forceinline__ void screen2(f2 y, f2 negr2, bool &p0, bool &p1, float &near) {
    float d0, d1;
    f2_get(f2_fma(y, y, negr2), d0, d1);
    p0 = d0 < 0.0f;
    p1 = d1 < 0.0f;
    near = min3_abs(near, d0, d1);
}

// number of dependent shifts (children per free slot) for the dependent split mask
__host__ __device__ constexpr int dep_slots(int dm) { return dm == 3 ? 4 : (dm ? 2 : 1); }

// Ballots of FG free slots (1, 2 or 4) times their dependent shifts: bu/bl[ds * FG + f].
// u[j][p]: residuals before the dependent shift, of free slots 2 p and 2 p + 1 (FG = 1:
// of the one slot, twice).  A child passes when every dependent coordinate passes, and
// the test of coordinate j depends only on its own shift, so with two coordinates the
// four children of a free slot take four tests, not eight: their ballots are combined.
template <int ND, int FG, int DM, bool LB>
__device__ __forceinline__ void test_children(const f2 (&u)[ND][(FG + 1) / 2], const float *hs, const f2 *negR2,
                                              const f2 *negL2, float *near, float *nearL, unsigned *bu,
                                              unsigned *bl) {
    constexpr int NDS = dep_slots(DM);
    unsigned au[ND][2][FG], al[ND][2][FG];
#pragma unroll
    for (int j = 0; j < ND; ++j) {
        const bool split = (DM >> j) & 1;
        if constexpr (FG >= 2) {
#pragma unroll
            for (int p = 0; p < FG; p += 2) {
#pragma unroll
                for (int v = 0; v < (split ? 2 : 1); ++v) {
                    f2 y = u[j][p / 2];
                    if (split) y = f2_add(y, f2_dup(v ? -hs[j] : hs[j]));
                    bool p0, p1;
                    screen2(y, negR2[j], p0, p1, near[j]);
                    au[j][v][p] = __ballot_sync(kFull, p0);
                    au[j][v][p + 1] = __ballot_sync(kFull, p1);
                    if constexpr (LB) {
                        screen2(y, negL2[j], p0, p1, nearL[j]);
                        al[j][v][p] = __ballot_sync(kFull, p0);
                        al[j][v][p + 1] = __ballot_sync(kFull, p1);
                    }
                }
            }
        } else {
            // the pair is the coordinate's two shifts (the same value twice without one)
            const f2 y = split ? f2_add(u[j][0], f2_make(hs[j], -hs[j])) : u[j][0];
            bool p0, p1;
            screen2(y, negR2[j], p0, p1, near[j]);
            au[j][0][0] = __ballot_sync(kFull, p0);
            if (split) au[j][1][0] = __ballot_sync(kFull, p1);
            if constexpr (LB) {
                screen2(y, negL2[j], p0, p1, nearL[j]);
                al[j][0][0] = __ballot_sync(kFull, p0);
                if (split) al[j][1][0] = __ballot_sync(kFull, p1);
            }
        }
    }
#pragma unroll
    for (int x = 0; x < NDS; ++x) {
        const int ds = DM == 2 ? x << 1 : x;                        // dependent bits of shift x
#pragma unroll
        for (int f = 0; f < FG; ++f) {
            unsigned b = au[0][ds & 1][f], l = LB ? al[0][ds & 1][f] : 0u;
            if constexpr (ND == 2) {
                b &= au[ND - 1][ds >> 1][f];
                if constexpr (LB) l &= al[ND - 1][ds >> 1][f];
            }
            bu[x * FG + f] = b;
            if constexpr (LB) bl[x * FG + f] = l;
        }
    }
}

// Whether the screen leaves a record undecided.  Its band is proportional to the radius
// (bandR, in finalize_levels): a residual is within bandR R of the radius only if
// |y^2 - R^2| < bandR (2 + bandR) R^2 = kappa R^2.
template <int FAM, bool LB>
__device__ __forceinline__ bool undecided(const Level &lev, const float *R, const float *near, const float *nearL) {
    using F = Fam<FAM>;
    bool u = false;
#pragma unroll
    for (int j = 0; j < F::ND; ++j) {
        u |= near[j] < R[j] * R[j] * lev.kappa[j];
        if constexpr (LB) {
            const float e = __fmaf_rn(lev.bandL[j], R[j], lev.bandL0[j]);
            u |= nearL[j] < e * (e + 2.0f * lev.Lc[j]);
        }
    }
    return u;
}

// a tile's row of N child slots (2, 4 or 8), aligned to its size
template <int N>
__device__ __forceinline__ void store_row(uint32_t *p, const unsigned *v) {
    if constexpr (N == 2) {
        *reinterpret_cast<uint2 *>(p) = make_uint2(v[0], v[1]);
    } else {
#pragma unroll
        for (int i = 0; i < N; i += 4) *reinterpret_cast<uint4 *>(p + i) = make_uint4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    }
}

template <int N>
__device__ __forceinline__ void load_row(const uint32_t *p, unsigned *v) {
    if constexpr (N == 2) {
        const uint2 x = *reinterpret_cast<const uint2 *>(p);
        v[0] = x.x; v[1] = x.y;
    } else {
#pragma unroll
        for (int i = 0; i < N; i += 4) {
            const uint4 x = *reinterpret_cast<const uint4 *>(p + i);
            v[i] = x.x; v[i + 1] = x.y; v[i + 2] = x.z; v[i + 3] = x.w;
        }
    }
}

}  // namespace gv
