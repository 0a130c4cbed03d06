// gv_kernels.h -- launch interface between the host engine and the kernels.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "gv_device.cuh"

namespace gv {

// Records of one level.  A record is one canonical surface in one cell, packed as
// NFP fields [q_f (ND), q_t (LE), padding]: 16-bit fields biased by 2^15 (two per
// 32-bit word) on levels whose value bounds allow it, plain 32-bit fields
// otherwise.  The records of a cell start at a multiple of 32 (a tile); a tile's
// owning cell is tile_cell[tile].  mult (originals merged into a record) is NULL
// when every multiplicity is 1 (no grouping): it is then neither stored nor read.
struct RecView {
    uint32_t *rec;           // packed records
    uint32_t *mult;          // [records] or NULL
    uint32_t *tile_cell;     // [records / 32] cell index (as stored in the level's cell arrays)
};

// Cells of one level: packed leaf-aligned key, first record (a multiple of 32),
// record count, UB, LB.
struct CellView {
    uint64_t *key;
    uint64_t *rbeg;
    uint32_t *rcnt;
    uint32_t *ub;
    uint32_t *lb;
};

// Device-resident scalars of one solve.
struct Scalars {
    unsigned int best_lb;            // largest lower bound seen
    unsigned int n_uns;              // entries of the step's recheck queue
    unsigned long long best_key;     // (UB << coord_bits) | ~leaf key (max = best leaf)
    unsigned long long n_cells;      // cells written to the next level
    unsigned long long n_recs;       // record slots (32-aligned per cell) of the next level
    unsigned long long tests;        // (child, record) pairs decided
    unsigned long long records;      // records of the cells expanded
    unsigned long long rechecks;     // FP64 rechecks of the FP32 screen
    unsigned long long trace_n;      // trace entries
    unsigned long long replay_ub;    // replay: surfaces reaching the target cell
    unsigned long long replay_lb;    // replay: ... passing its lower-bound test
    unsigned int err;                // nonzero: input out of range
    unsigned int ticket;             // units of tiles handed out by the step's count pass
    unsigned int qmax[GV_MAXD + GV_MAXT];  // lift: largest |q_f,j|, |q_t,m| of the root records
    unsigned long long rechecks_df;  // snaps the double-float tier decided (FP32 screen undecided)
    // counted on request (Chunk::work):
    unsigned long long left_tests;   // tests not evaluated: of cells that the count pass left
    unsigned long long left_bytes;   // and the bytes it did not move for them
    unsigned long long emit_bytes;   // records and ballots of the tiles that the emit pass read
};

struct Trace {
    unsigned long long cap;
    int32_t *level;
    uint64_t *key;
    uint32_t *ub, *lb;
};

// Sizes of one level in a chain (levels expanded whole, one after the other, without the
// host): what its kernels expand, 0 once the chain has stopped; what the step before
// stored; whether its own step found no room in the next level.
struct LevInfo {
    long long ncells, nrecs;
    long long stored_cells, stored_recs;
    long long overflow;
    long long seq;           // the host's copy: written last, the number of the step
};

// Everything one expansion step (a chunk of cells of one level) needs.
//
// Children are numbered over the coordinates that still split at this level ("child
// slots"): slot = free bits | dependent bits << kf, each the bits of the level's
// split mask in coordinate order, so a cell has ns = 2^(splitting coordinates) slots
// and nothing is computed, stored or read for children that do not exist.
struct Chunk {
    Problem P;
    Level lev;
    CellView cells;          // cells of level l (key, ub: absolute index c0 + cl)
    int64_t c0;              // first cell of the chunk
    int nc;                  // number of cells in the chunk
    int ns, lns;             // child slots per cell, log2
    int nfs, kf;             // free slots (basis changes) per cell, log2
    int dm;                  // bit j: dependent coordinate j splits
    int gf;                  // floats of one cell's screen geometry
    RecView in;              // records of the chunk (tile_cell values: in_c0 + cl)
    const uint64_t *in_rbeg; // first record of chunk cell cl at in_rbeg[in_c0 + cl]
    const uint32_t *in_rcnt; // its record count
    int64_t in_c0;
    int64_t t0, t1;          // tile range of the chunk
    uint8_t *alive;          // [nc]   bit 0: cell still above the pruning threshold, and not left by the count
                             //        pass; bit 1: it has a surviving child
    // cell geometry: the changes of the cell-dependent basis values (Fam::NBG) from the
    // cell centre to the child centres, one per geometry slot (the free slots without a
    // linear tail coordinate's bit)
    int ng, kg;              // geometry slots, log2
    float *geo32;            // [nc][gf]: [NBG][ng] rounded to FP32, then [NBG] the largest magnitudes
    float *geo32lo;          // [nc][NBG][ng] what that rounding leaves, rounded to FP32
    double *geo64;           // [nc][nfs][NB] in plain FP64 mode and where a table is missing, else NULL
    const double2 *sincos[2];// (sin, cos) of every centre of angular coordinate 0, 1 (entry 2^e - 1 + i for
                             // cell i after e splits), or NULL
    double *rot_par, *rot_ch;// rotations (9 values) of every cell of the rotation coordinates at this level and
                             // the next, filled on demand, or NULL
    unsigned *rot_flag;      // bit per entry of rot_ch: filled
    uint32_t *crec, *clb;    // [nc][ns]  records (UB-passing) and LB sum per child
    uint32_t *cub;           // [nc][ns]  UB sum per child (= crec without multiplicities)
    int2 *tinfo;             // [t1 - t0 + 2] per tile: chunk-local cell (-1: pruned), valid lanes | kTileFirst |
                             //           kTileLast | tiles left << kLeftShift | allowance << kAllowShift
    uint32_t *ballot;        // [t1 - t0][ns] per tile and child: UB-passing lanes
    uint32_t *lballot;       // [t1 - t0][ns] the same for the LB test
    uint2 *uns;              // queue of (tile, lanes) the FP32 screen left undecided, sc->n_uns entries
    uint32_t *off;           // [t1 - t0][ns] per tile and child: its records' first place in the child
    unsigned long long *cbase; // [nc][ns] first record slot of the child (~0: pruned)
    int32_t *child_idx;      // [nc][ns] index of the child cell (where cbase is not ~0)
    CellView next_cells;     // cells of level l+1
    int64_t next_c0, next_r0;// its cells and record slots before this step (the step appends)
    RecView out;             // records of level l+1
    Scalars *sc;
    Trace trace;
    LevInfo *dyn;            // in a chain of levels: this level's sizes (the next level's follow), else NULL
    LevInfo *host;           // pinned: where the step reports what it stored, as step number seq
    long long seq;
    int64_t cap_cells, cap_recs, fit_recs;   // chain: room in the next level; what still is expanded whole
    int weighted;            // multiplicities: cub is an array of its own
    int prune;
    int precision;           // 0 = FP64, 1 = FP32 screen + FP64 recheck
    int lb;                  // lower bounds are wanted (lballot, clb)
    int work;                // count the work that is done and left out
    int early;               // the count pass leaves cells whose children all fall below the threshold; it
                             // takes cells of at most this many tiles (>= 1) whole, a warp each
    uint32_t *cfail;         // [nc][ns] early: records that certainly fail each child's UB test, of cells that
                             //          several warps count (child_idx's memory, which is written after)
    unsigned spin;           // polls of a bounded wait for a bulk copy before giving up
};
// The kernels of a step depend on one another and most are short: each is launched while
// the one before still runs (its blocks take free places on the SMs and wait), so a step
// of few records spends 3 us instead of 5 us per kernel.  Every kernel launched this way
// begins with grid_start() in all its threads: it returns when the kernel before has
// completed and its writes are visible.  Data of earlier kernels is read with plain loads
// only: the compiler may move read-only ones ahead of the wait.
__device__ __forceinline__ void grid_start() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

inline cudaLaunchConfig_t launch_config(unsigned blocks, unsigned threads, size_t smem, cudaStream_t st,
                                        cudaLaunchAttribute *attr) {
    attr->id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr->val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

template <class... P, class... A>
inline void launch(void (*kernel)(P...), unsigned blocks, unsigned threads, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = launch_config(blocks, threads, smem, st, &attr);
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// Sizes of a chunk: from the device in a chain of levels (the host's are then bounds).
__device__ __forceinline__ int64_t chunk_tiles(const Chunk &c) { return c.dyn ? c.dyn->nrecs >> 5 : c.t1 - c.t0; }
__device__ __forceinline__ int chunk_cells(const Chunk &c) { return c.dyn ? (int)c.dyn->ncells : c.nc; }
constexpr int kTileFirst = 64, kTileLast = 128;   // flags in tinfo.y: first / last tile of its cell
// the cell's tiles after it, at most kLeftMax (more are not skipped at once); kTileOwned: one
// warp of the count pass takes the whole cell; and how many of the
// cell's records may fail a child's UB test while the child can still reach the threshold, in
// eights rounded up (kAllowNone: the cell is counted in any case)
constexpr int kLeftShift = 8, kLeftMax = 127, kTileOwned = 1 << 15, kAllowShift = 16;
constexpr unsigned kAllowNone = 0xffffu;

constexpr int kNoExp = -1000;

// Selection of a level's cells with the largest UBs (index 0) and LBs (index 1)
// (k_beam_*); zeroed once, and every selection leaves it cleared for the next.
constexpr int kBeamBins = 2048;
struct BeamSel {
    unsigned long long hist[2][kBeamBins];  // record slots per bin
    unsigned long long best[2];      // (value << 32) | ~index of the cell with the largest value
    unsigned long long top[2];       // the same, of the finished histogram
    int border[2];                   // bins above are selected whole
    unsigned share[2];               // selected share of the border bin (2^32 = all)
    unsigned ticket;
};

// Path geometry for replaying surfaces along the root-to-cell path.
constexpr int kPathTail = 4; // entries after the steps (see k_path_geo)
struct PathStep {
    int slot;
    double dpsi[GV_MAXT];
};

// root records of the surfaces and the root cell
void launch_lift(const Problem &P, const Level &lev0, const double *psi0, const double *prm, int64_t n, RecView out,
                 CellView root, Scalars *sc, cudaStream_t st);
// psi [GV_MAXT]: basis of the root cell's centre
void launch_root_basis(const Problem &P, const Level &lev0, double *psi, cudaStream_t st);
// the (sin, cos) table of an angular coordinate (2^(splits + 1) - 1 entries)
void launch_sincos_table(const Problem &P, int j, double2 *tab, cudaStream_t st);
// cells (alive, geometry) and tiles (tinfo) of the chunk; returns the kernels launched
int launch_prep(const Chunk &c, cudaStream_t st);
// SMs of the device (read once)
int sm_count();
// launch a persistent kernel taking one Chunk: one block per resident slot on the
// device, at most `groups` blocks, 256 threads, smem bytes of dynamic shared memory
void launch_persistent(const void *kern, size_t smem, int64_t groups, const Chunk &c, cudaStream_t st);
// the ballots of every tile and child, by the FP32 screen (undecided records queued)
// or, in plain FP64 mode, by the definition
void launch_count(const Chunk &c, cudaStream_t st);
void launch_count_wide(const Chunk &c, cudaStream_t st);
// the definition: the queued records' bits are added to the ballots; every record
void launch_recheck(const Chunk &c, cudaStream_t st);
void launch_count_exact(const Chunk &c, cudaStream_t st);
// per child its counts, per tile and child its records' place in the child, best LB
void launch_tile_scan(const Chunk &c, cudaStream_t st);
bool launch_emit_wide(const Chunk &c, cudaStream_t st);
// adds the bytes of records and ballots that the emit pass will read to sc->emit_bytes
void launch_emit_work(const Chunk &c, int rec_bytes, cudaStream_t st);
// false if the level's record formats have no emit pass (never chosen by the engine)
bool launch_emit(const Chunk &c, cudaStream_t st);
// sizes of the level that a chain starts from, or goes on from
void launch_chain_start(LevInfo *info, int64_t cells, int64_t recs, cudaStream_t st);
// keepflag, recn: [nc * ns]; bsums: 2 * ceil(nc * ns / 256); returns the kernels launched
// (small: by one block)
int launch_child_alloc(const Chunk &c, bool small, uint32_t *keepflag, uint32_t *recn, unsigned long long *bsums,
                       cudaStream_t st);
// the cells of a level (whose sum of record slots exceeds budget) with the largest UBs (nk = 2: and LBs):
// out and src_rbeg receive them ([ncells] at most), host their number and slots; bsums:
// 2 * ceil(ncells / 256); returns the kernels launched; then their records
int launch_beam_select(const Problem &P, const CellView &cells, int64_t ncells, int64_t budget, int nk, BeamSel *sel,
                        unsigned long long *bsums, const CellView &out, uint64_t *src_rbeg, Scalars *sc,
                       LevInfo *host, long long seq, cudaStream_t st);
void launch_beam_gather(const RecView &in, const RecView &out, const CellView &sel, const uint64_t *src_rbeg,
                        int64_t ncells, int64_t ntiles, int rec_bytes, cudaStream_t st);
// the path to cell `key` at level lam, or to the best leaf of sc when sc is not NULL
void launch_path_geo(const Problem &P, const Level *levs_dev, int lam, uint64_t key, const Scalars *sc, PathStep *path,
                     cudaStream_t st);
void launch_replay(const Problem &P, const Level *levs_dev, const PathStep *path, int lam, const double *prm,
                   int64_t n, uint32_t *reach, Scalars *sc, cudaStream_t st);

// Grouping of a chunk's records (c.in, tiles [c.t0, c.t1), cells c.in_rbeg/in_rcnt)
// into out (cells indexed 0..nc-1 by chunk-local index): table [tmask + 1] zeroed;
// owner, newpos [32 (t1 - t0)]; ccount, ccur [nc] zeroed; grbeg [nc] receives the
// canonical records' first slots (32-aligned), ccount their counts; total[0] = slots
// used, total[1] = canonical records, total[2] = records that entered the grouping.
void launch_group(const Chunk &c, uint32_t *table, uint32_t tmask, uint32_t *owner, uint32_t *ccount,
                  uint32_t *ccur, uint32_t *newpos, uint64_t *grbeg, unsigned long long *total, RecView out,
                  cudaStream_t st);

// soft inlier score (gv_softscore.cu): forward writes out[0] = S; backward writes
// out[0..d) = grad_out * dS/dp and, if grad_prm, grad_out * dS/dparams [P][n].
// partial: softscore_partial_doubles() doubles of scratch.
void launch_softscore(int fam, bool bwd, const double *prm, int64_t n, const uint32_t *mask, const double *p,
                      const double *inv_tol2, int nd, const double *grad_out, double *grad_prm, double *partial,
                      double *out, cudaStream_t st);
int softscore_partial_doubles();
bool softscore_supported(int fam);

// words of one record of a family in the 16- or 32-bit format
__host__ __device__ constexpr int rec_words(int nfp, bool q16) { return q16 ? nfp / 2 : nfp; }

}  // namespace gv
