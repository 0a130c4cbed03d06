// gv_exact.cu -- the proximity test by its FP64 definition: the records the FP32 screen
// left undecided, and every record in plain FP64 mode.
//
// The FP64 pipe of this part issues one lane per clock and SM, and a warp instruction
// occupies it for all 32 lanes whether they are active or not.  So the screen does not
// call the definition where it meets an undecided record (about one in 10^4): it queues
// the record, and k_recheck evaluates the queue with full warps.
#include "gv_tile.cuh"

namespace gv {

template <int FAM, bool Q16>
__device__ __forceinline__ void eval_record(const Chunk &c, int64_t r, int cell, int fs0, int fs1,
                                            SlotMask<FAM> &ubm, SlotMask<FAM> &lbm) {
    using F = Fam<FAM>;
    constexpr int NW = rec_words(F::NFP, Q16);
    uint32_t w[NW];
    load_words<NW>(c.in.rec, r, w);
    int qf[F::ND], qt[F::LE];
#pragma unroll
    for (int j = 0; j < F::ND; ++j) qf[j] = field_i<Q16>(w, j);
#pragma unroll
    for (int m = 0; m < F::LE; ++m) qt[m] = field_i<Q16>(w, F::ND + m);
    eval64<FAM>(c, cell, qf, qt, fs0, fs1, ubm, lbm);
}

// One queue entry (a tile and its undecided lanes, almost always one) per thread, or, of a
// short queue, one entry's children of one free slot: then the kernel's time is a single
// evaluation's (a chain of FP64 instructions, 40 clocks each: 8 children of a 3-DoF pose
// 5 us, 64 of a 6-DoF pose 70 us), and the work that the split repeats costs nothing: 6-DoF
// pose, 5000 matches: count and recheck 2.7 -> 1.1 ms.  The
// screen left the lanes' bits clear, so the passing ones are set here.
template <int FAM, bool Q16>
__global__ void __launch_bounds__(128) k_recheck(const __grid_constant__ Chunk c) {
    grid_start();
    if (chunk_tiles(c) == 0) return;                                // the chain has stopped: not its queue
    const unsigned nq = c.sc->n_uns;
    unsigned long long done = 0;
    const unsigned threads = gridDim.x * 128u, parts = nq * (unsigned)c.nfs <= threads ? (unsigned)c.nfs : 1u;
    for (unsigned x = blockIdx.x * 128u + threadIdx.x; x < nq * parts; x += threads) {
        const unsigned i = x / parts;
        const int fs0 = (int)(x - i * parts), fs1 = parts > 1u ? fs0 + 1 : c.nfs;
        const uint2 e = c.uns[i];
        const int cell = c.tinfo[e.x].x;
        for (unsigned m = e.y; m; m &= m - 1) {
            const int bit = __ffs(m) - 1;
            SlotMask<FAM> ubm, lbm;
            eval_record<FAM, Q16>(c, (c.t0 + e.x) * 32 + bit, cell, fs0, fs1, ubm, lbm);
            uint32_t *bp = c.ballot + (size_t)e.x * c.ns, *lp = c.lballot + (size_t)e.x * c.ns;
            for (SlotMask<FAM> x = ubm; x; x &= x - 1) atomicOr(bp + __ffsll((long long)x) - 1, 1u << bit);
            if (c.lb)
                for (SlotMask<FAM> x = lbm; x; x &= x - 1) atomicOr(lp + __ffsll((long long)x) - 1, 1u << bit);
            if (fs0 == 0) done += (unsigned)c.ns;
        }
    }
    if (done) atomicAdd(&c.sc->rechecks, done);
}

// Plain FP64 mode: a warp per tile, every record by the definition.
template <int FAM, bool Q16>
__global__ void __launch_bounds__(256) k_count_exact(const __grid_constant__ Chunk c) {
    grid_start();
    const int lane = threadIdx.x & 31;
    const int64_t nwarp = (int64_t)gridDim.x * 8, nt = chunk_tiles(c);
    for (int64_t tt = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); tt < nt; tt += nwarp) {
        const int2 ti = c.tinfo[tt];
        if (ti.x < 0) continue;                                     // uniform: the cell was pruned
        const int nvalid = ti.y & 63;
        SlotMask<FAM> ubm = 0, lbm = 0;
        if (lane < nvalid) eval_record<FAM, Q16>(c, (c.t0 + tt) * 32 + lane, ti.x, 0, c.nfs, ubm, lbm);
        uint32_t *bp = c.ballot + (size_t)tt * c.ns, *lp = c.lballot + (size_t)tt * c.ns;
        for (int s = 0; s < c.ns; ++s) {
            const unsigned bu = __ballot_sync(kFull, (ubm >> s) & 1), bl = __ballot_sync(kFull, (lbm >> s) & 1);
            if (lane == 0) {
                bp[s] = bu;
                if (c.lb) lp[s] = bl;
            }
        }
    }
}

#define GV_DISPATCH(fam, CALL)                                                   \
    switch (fam) {                                                               \
    case FAM_LINE2D: { constexpr int FAMV = FAM_LINE2D; CALL; } break;           \
    case FAM_PLANE3D_SPH: { constexpr int FAMV = FAM_PLANE3D_SPH; CALL; } break; \
    case FAM_POSE3DOF: { constexpr int FAMV = FAM_POSE3DOF; CALL; } break;       \
    case FAM_RAYS3D: { constexpr int FAMV = FAM_RAYS3D; CALL; } break;           \
    case FAM_POSE6DOF: { constexpr int FAMV = FAM_POSE6DOF; CALL; } break;       \
    case FAM_POINTSET2D: { constexpr int FAMV = FAM_POINTSET2D; CALL; } break;   \
    case FAM_AFFINE4D: { constexpr int FAMV = FAM_AFFINE4D; CALL; } break;       \
    case FAM_RADIAL5DOF: { constexpr int FAMV = FAM_RADIAL5DOF; CALL; } break;   \
    default: break;                                                              \
    }

void launch_recheck(const Chunk &c, cudaStream_t st) {
    const int64_t nt = c.t1 - c.t0;
    if (nt <= 0) return;
    // at most one entry per tile, nfs threads for each while the queue is short
    const int64_t need = (nt * c.nfs + 127) / 128;
    const unsigned g = (unsigned)(need < 608 ? need : 608);
    if (c.lev.q16) {
        GV_DISPATCH(c.P.fam, (launch(k_recheck<FAMV, true>, g, 128, 0, st, c)));
    } else {
        GV_DISPATCH(c.P.fam, (launch(k_recheck<FAMV, false>, g, 128, 0, st, c)));
    }
}

void launch_count_exact(const Chunk &c, cudaStream_t st) {
    const int64_t nt = c.t1 - c.t0;
    if (nt <= 0) return;
    const unsigned g = (unsigned)(nt < 8 * 152 * 8 ? (nt + 7) / 8 : 152 * 8);
    GV_DISPATCH(c.P.fam, (launch(k_count_exact<FAMV, false>, g, 256, 0, st, c)));   // 32-bit records in this mode
}

}  // namespace gv
