// gv_engine.cu -- host engine and C ABI of libvote (see include/vote.h).
//
// The engine drives Algorithm 2 (SurfaceConsensus) of arXiv 2107.11810 level by
// level on the GPU.  Each level keeps a stack of cells and of their records
// (canonical surfaces).  One expansion step takes a chunk of cells from the top of
// the deepest non-empty level, tests all their children (k_test count pass),
// raises the best lower bound, drops children below it (B&B pruning, Sec. 3.3),
// lays out the survivors and writes their records, snapped for the next level
// (emit pass, canonization of Sec. 3.2).  The order (search(), dive()) follows the
// cells with the largest bounds down to the leaves first, which raises the pruning
// bound to about its final value, then opens the rest level by level while the next
// level has room, else (and without dives) the deepest level first.  The result does
// not depend on it.
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <atomic>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "gv_kernels.h"
#include "gv_tile.cuh"
#include "vote.h"

using namespace gv;

static thread_local char g_err[512] = "";

static void set_err(const char *fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
}

#define CK(call)                                                                        \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess) {                                                        \
            set_err("%s failed: %s", #call, cudaGetErrorString(e_));                    \
            return VOTE_ECUDA;                                                          \
        }                                                                               \
    } while (0)

#define TRY(x)                                                                          \
    do {                                                                                \
        vote_status s_ = (x);                                                           \
        if (s_ != VOTE_OK) return s_;                                                   \
    } while (0)

struct DevBuf {
    void *p = nullptr;
    size_t bytes = 0;
};

struct LevelStore {
    DevBuf rec, mult, tile_cell;       // packed records (whole tiles), multiplicities, owning cell per tile
    DevBuf key, rbeg, rcnt, ub, lb;
    int64_t ncells = 0, nrecs = 0;     // nrecs: record slots in use (a multiple of 32)
};

struct vote_ctx {
    Problem P;
    Level lev[GV_MAXL];
    double h_leaf[GV_MAXD];
    int device = 0;
    cudaStream_t stream = 0;
    int precision = 1, prune = 1, group = 0;
    unsigned sched = 0;        // how the process wants its threads to wait (cudaDeviceSchedule*)
    int64_t chunk_records = 1 << 25;
    bool chunk_set = false;            // VOTE_OPT_CHUNK_RECORDS was given
    bool lean = false;                 // the solve at hand is repeated with less memory (solve_device)
    bool fault_hit = false;            // an allocation failed because the test hook asked for it
    uint32_t initial_lb = 0;
    int kernel_timing = 0;
    int count_work = 0;        // count what the passes leave out (with kernel timing, here or in the batch)
    int log = 0;               // VOTE_LOG=1: per-level counters on stderr after each solve;
                               // 2: also one line per expansion step
    unsigned spin_limit = GV_SPIN_LIMIT;   // VOTE_OPT_SPIN_LIMIT
    int batch_workers = 4;
    int dive = 2;              // dives along the cells with the largest bounds: 0 off, 1 or 2 on
    int family = 0;
    double eps_in[GV_MAXD] = {}, bounds_in[2 * GV_MAXD] = {};
    std::vector<vote_ctx *> workers;   // sub-contexts of vote_solve_batched
    static const int kEv = 24;
    cudaEvent_t ev[kEv] = {};
    int ev_n = 0;              // events recorded since the last collection
    int ev_cls[kEv] = {};      // kernel class of the interval ending at event i
    double kms[VOTE_K_CLASSES] = {};
    int64_t klaunch[VOTE_K_CLASSES] = {};
    double kbytes[VOTE_K_CLASSES] = {};
    int64_t lv_cells[GV_MAXL] = {}, lv_recs[GV_MAXL] = {};
    int64_t lv_gin[GV_MAXL] = {}, lv_gout[GV_MAXL] = {};  // records into / out of grouping
    int64_t trace_cap = 0;
    int64_t fault_alloc_at = 0, alloc_count = 0;
    LevelStore ls[GV_MAXL + 1];
    LevelStore beam;           // the selected cells of one level, during the dive
    DevBuf beam_sel, beam_src, linfo;
    LevInfo *h_info = nullptr; // pinned: the steps' reports, per level; the last for single steps
    long long steps = 0;       // numbers them
    DevBuf psi0;               // basis of the root cell's centre
    DevBuf sctab[2];           // (sin, cos) tables of the angular coordinates (launch_sincos_table)
    DevBuf rot[GV_MAXL + 1], rotflag[GV_MAXL + 1];   // rotation tables per level (k_rot_fill)
    DevBuf levs_dev, path, scal, alive, geo64, geo32, geo32lo, cnt, tinfo, ballot, lballot, uns, off, cbase, child_idx;
    DevBuf keepflag, recn, bsums;
    DevBuf tr_level, tr_key, tr_ub, tr_lb, surf_tmp, mask_tmp;
    DevBuf ss_partial, ss_io;  // soft score: block partials; point [d] + outputs [d] + grad_out [1]
    DevBuf g_table, g_owner, g_newpos, g_ccount, g_ccur, g_rbeg, g_rec, g_mult, g_tile;
    Scalars *h_sc = nullptr;   // pinned mirror of the device scalars
    uint64_t *h_tmp = nullptr; // pinned slot for single values
    // device slot for single values: 64 bytes after the scalars block
    void *h_tmp_dev() { return (char *)scal.p + ((sizeof(Scalars) + 63) / 64) * 64; }
    int64_t trace_written = 0;
    int64_t expanded = 0;      // record slots expanded in this solve
    int64_t evaluated = 0;     // tests that the solve evaluated (stats.tests without those of cells left early), -1: not counted
    bool trace_overflow = false;
    vote_stats stats;
};

// ---------------------------------------------------------------------------
// problem constants (the same definition as the paper-derived oracle, written
// independently: per-coordinate levels, power-of-two snap steps, accumulated
// canonization error)
// ---------------------------------------------------------------------------
static int family_shape(int fam, int d, int k, int *le, int *np) {
    switch (fam) {
    case VOTE_LINE2D: if (d != 2 || k != 1) return 1; *le = 1; *np = 2; return 0;
    case VOTE_PLANE3D_SPH: if (d != 3 || k != 2) return 1; *le = 3; *np = 3; return 0;
    case VOTE_POSE3DOF: if (d != 3 || k != 1) return 1; *le = 2; *np = 4; return 0;
    case VOTE_POSE6DOF: if (d != 6 || k != 4) return 1; *le = 11; *np = 5; return 0;
    case VOTE_RAYS3D: if (d != 3 || k != 1) return 1; *le = 2; *np = 4; return 0;
    case VOTE_POINTSET2D: if (d != 4 || k != 2) return 1; *le = 2; *np = 4; return 0;
    case VOTE_AFFINE4D: if (d != 4 || k != 3) return 1; *le = 3; *np = 4; return 0;
    case VOTE_RADIAL5DOF: if (d != 5 || k != 4) return 1; *le = 7; *np = 5; return 0;
    default: return 1;
    }
}

// bound on the change of each basis function across a cell of half-widths h
static void family_sigma(int fam, const double *h, double *sigma) {
    switch (fam) {
    case VOTE_LINE2D: sigma[0] = h[0]; break;
    case VOTE_PLANE3D_SPH:
        sigma[0] = h[0] + h[1];
        sigma[1] = h[0] + h[1];
        sigma[2] = h[0];
        break;
    case VOTE_POSE3DOF:
        sigma[0] = h[0];
        sigma[1] = h[0];
        break;
    case VOTE_RAYS3D:       // a and c multiply x
        sigma[0] = h[0];
        sigma[1] = h[0];
        break;
    case VOTE_AFFINE4D:     // x_i multiplies a_i
        sigma[0] = h[0];
        sigma[1] = h[1];
        sigma[2] = h[2];
        break;
    case VOTE_POINTSET2D:   // u, v multiply c in one equation and d in the other
        sigma[0] = h[0] > h[1] ? h[0] : h[1];
        sigma[1] = sigma[0];
        break;
    case VOTE_POSE6DOF: {
        // an entry of the rotation moves by at most |d phi|_2 <= sum of the phi
        // half-widths (its gradient has norm <= 1); z is linear
        const double hr = (h[0] + h[1]) + h[2];
        for (int m = 0; m < 9; ++m) sigma[m] = hr;
        sigma[9] = h[3];
        sigma[10] = h[3];
        break;
    }
    case VOTE_RADIAL5DOF: {
        // the six entries of rows r1, r2 (as for 6DoF); y is linear
        const double hr = (h[0] + h[1]) + h[2];
        for (int m = 0; m < 6; ++m) sigma[m] = hr;
        sigma[6] = h[3];
        break;
    }
    }
}

static double pow2_floor(double x, int *e_out) {
    int e;
    std::frexp(x, &e);
    if (e_out) *e_out = e - 1;
    return std::ldexp(1.0, e - 1);
}

// Linear bases: the largest e <= 0 with every coefficient h1_b s_t,m / s_f,j of the
// screen an FP32-exact multiple of 2^e; kNoExp when one is not, and for other bases.
template <int FAM>
static int linear_exp_fam(const Problem &, const Level &v) {
    using F = Fam<FAM>;
    if (!F::LINEAR_BASIS) return kNoExp;
    int e = 0;
    for (int j = 0; j < F::ND; ++j)
        for (int m = 0; m < F::LE; ++m) {
            const int b = F::cb(j, m);
            if (!F::uses(j, m) || !((v.split_mask >> b) & 1)) continue;
            const double g = v.h1[b] * v.gscale[j][m];
            if ((double)(float)g != g) return kNoExp;
            if (g != 0.0) e = std::min(e, lowbit_exp(g));
        }
    return e;
}
static int linear_exp(const Problem &P, const Level &v) {
    switch (P.fam) {
    case VOTE_LINE2D: return linear_exp_fam<FAM_LINE2D>(P, v);
    case VOTE_RAYS3D: return linear_exp_fam<FAM_RAYS3D>(P, v);
    case VOTE_POINTSET2D: return linear_exp_fam<FAM_POINTSET2D>(P, v);
    case VOTE_AFFINE4D: return linear_exp_fam<FAM_AFFINE4D>(P, v);
    default: return kNoExp;
    }
}

static vote_status problem_init(vote_ctx *c, int fam, int d, int k, const double *eps, const double *bounds) {
    int le, np;
    if (family_shape(fam, d, k, &le, &np)) {
        set_err("family %d does not take d=%d, k=%d", fam, d, k);
        return VOTE_EINVAL;
    }
    Problem &P = c->P;
    std::memset(&P, 0, sizeof(P));
    P.fam = fam; P.d = d; P.k = k; P.nd = d - k; P.le = le; P.np = np;
    P.inv_fact[0] = 1.0;
    for (int m = 1; m < 31; ++m) P.inv_fact[m] = P.inv_fact[m - 1] / (double)m;
    P.L = 0;
    for (int j = 0; j < d; ++j) {
        double lo = bounds[2 * j], hi = bounds[2 * j + 1];
        if (!(eps[j] > 0.0) || !std::isfinite(eps[j]) || !std::isfinite(lo) || !std::isfinite(hi) || !(hi > lo)) {
            set_err("coordinate %d: need finite eps > 0 and lo < hi", j);
            return VOTE_EINVAL;
        }
        P.lo[j] = lo;
        P.W[j] = hi - lo;
        P.eps[j] = eps[j];
        int Lj = 0;
        while (std::ldexp(P.W[j], -Lj) > eps[j]) ++Lj;
        if (Lj > 30) {
            set_err("coordinate %d needs %d levels (> 30)", j, Lj);
            return VOTE_EUNSUPPORTED;
        }
        P.Lj[j] = Lj;
        if (Lj > P.L) P.L = Lj;
    }
    if (P.L > GV_MAXL - 1) {
        set_err("too many levels");
        return VOTE_EUNSUPPORTED;
    }
    int bits = 0;
    for (int j = d - 1; j >= 0; --j) {
        P.coord_shift[j] = bits;
        bits += P.Lj[j];
    }
    P.coord_bits = bits;
    if (bits > 44) {       // the best leaf packs (UB << bits) | leaf key into 64 bits
        set_err("leaf key needs %d bits (> 44)", bits);
        return VOTE_EUNSUPPORTED;
    }
    double h[GV_MAXL + 1][GV_MAXD];
    for (int l = 0; l <= P.L; ++l)
        for (int j = 0; j < d; ++j) {
            int e = l < P.Lj[j] ? l : P.Lj[j];
            h[l][j] = std::ldexp(P.W[j], -(e + 1));
        }
    for (int j = 0; j < d; ++j) c->h_leaf[j] = h[P.L][j];
    if (P.L == 0) return VOTE_OK;
    double epsp_min = INFINITY;
    for (int j = 0; j < P.nd; ++j) {
        double epsp = P.eps[k + j] / (double)P.L;
        if (epsp < epsp_min) epsp_min = epsp;
        P.s_f[j] = pow2_floor(epsp / (double)(le + 1), nullptr);
        P.inv_s_f[j] = 1.0 / P.s_f[j];
    }
    double s_t[GV_MAXL + 1][GV_MAXT];
    int s_te[GV_MAXL + 1][GV_MAXT];
    double A[GV_MAXL + 1][GV_MAXD];
    for (int j = 0; j < P.nd; ++j) A[0][j] = 0.0;
    for (int l = 0; l < P.L; ++l) {
        double sigma[GV_MAXT];
        family_sigma(fam, h[l], sigma);
        for (int m = 0; m < le; ++m) s_t[l][m] = pow2_floor(epsp_min / ((double)(le + 1) * sigma[m]), &s_te[l][m]);
        for (int j = 0; j < P.nd; ++j) {
            double delta = P.s_f[j] * 0.5;
            for (int m = 0; m < le; ++m) delta = delta + (s_t[l][m] * 0.5) * sigma[m];
            delta = delta + std::ldexp(P.eps[k + j], -32);
            A[l + 1][j] = A[l][j] + delta;
        }
    }
    for (int l = 0; l < P.L; ++l) {
        Level &v = c->lev[l];
        std::memset(&v, 0, sizeof(v));
        v.l = l;
        v.leaf_children = (l + 1 == P.L);
        for (int j = 0; j < d; ++j) {
            if (l < P.Lj[j]) v.split_mask |= 1 << j;
            v.h[j] = h[l][j];
            v.h1[j] = h[l + 1][j];
        }
        for (int m = 0; m < le; ++m) {
            v.s_t[m] = s_t[l][m];
            v.inv_s_t[m] = std::ldexp(1.0, -s_te[l][m]);
            if (l + 1 < P.L) {
                int r = s_te[l + 1][m] - s_te[l][m];
                if (r < 0 || r > 1) {
                    set_err("internal: snap step ratio 2^%d at level %d", r, l);
                    return VOTE_EINTERNAL;
                }
                v.st_ratio_log2[m] = r;
                v.st_scale[m] = r ? 0.5f : 1.0f;
            }
        }
        for (int j = 0; j < P.nd; ++j) {
            v.Rbase[j] = P.eps[k + j] + h[l + 1][k + j];
            v.A1[j] = A[l + 1][j];
            v.rlb[j] = P.eps[k + j] - A[l + 1][j];
            // FP32 screen constants in steps of s_f,j (rounding is covered by its band)
            for (int m = 0; m < le; ++m) {
                v.gscale[j][m] = s_t[l][m] / P.s_f[j];
                v.gs[j][m] = (float)v.gscale[j][m];
            }
            v.Hs[j] = (float)(h[l + 1][k + j] / P.s_f[j]);
            v.Hs_lo[j] = (float)(h[l + 1][k + j] / P.s_f[j] - (double)v.Hs[j]);
            if (l < P.Lj[k + j]) {              // the dependent coordinate splits: its shift enters
                const double hs = h[l + 1][k + j] / P.s_f[j];
                if ((double)v.Hs[j] != hs) v.hs_exp = kNoExp;
                else if (v.hs_exp > kNoExp && hs != 0.0) v.hs_exp = std::min(v.hs_exp, lowbit_exp(hs));
            }
            v.rc0[j] = (float)((v.Rbase[j] + v.A1[j]) / P.s_f[j]);
            v.Lc[j] = (float)(v.rlb[j] / P.s_f[j]);
        }
        for (int j = 0; j < d; ++j) {
            v.h1f[j] = (float)v.h1[j];
            v.h1f_lo[j] = (float)(v.h1[j] - (double)v.h1f[j]);
        }
        v.g_exp = linear_exp(P, v);
        // Lipschitz term of the radius from the essential parameters in steps
        switch (fam) {
        case VOTE_LINE2D:        // |t| h1_m
            v.lam_c[0] = (float)(h[l + 1][0] * s_t[l][0] / P.s_f[0]);
            break;
        case VOTE_PLANE3D_SPH:   // |q| h1_theta + |q_xy| h1_phi; s_t,x = s_t,y
            v.lam_c[0] = (float)(h[l + 1][0] * s_t[l][0] / P.s_f[0]);
            v.lam_c[1] = (float)(h[l + 1][1] * s_t[l][0] / P.s_f[0]);
            v.rho2 = (float)((s_t[l][2] / s_t[l][0]) * (s_t[l][2] / s_t[l][0]));
            break;
        case VOTE_POSE3DOF:      // sqrt(a^2 + b^2) h1_yaw; s_t,a = s_t,b
            for (int j = 0; j < P.nd; ++j) v.lam_c[j] = (float)(h[l + 1][0] * s_t[l][0] / P.s_f[j]);
            break;
        case VOTE_RAYS3D:        // |a| h1_x and |c| h1_x
            v.lam_c[0] = (float)(h[l + 1][0] * s_t[l][0] / P.s_f[0]);
            v.lam_c[1] = (float)(h[l + 1][0] * s_t[l][1] / P.s_f[1]);
            break;
        case VOTE_AFFINE4D:      // sum_i |x_i| h1_i
            for (int m = 0; m < 3; ++m) v.lam_c[m] = (float)(h[l + 1][m] * s_t[l][m] / P.s_f[0]);
            break;
        case VOTE_POINTSET2D:    // a: |u| h1_c + |v| h1_d; b: |v| h1_c + |u| h1_d
            v.lam_c[0] = (float)(h[l + 1][0] * s_t[l][0] / P.s_f[0]);
            v.lam_c[1] = (float)(h[l + 1][1] * s_t[l][1] / P.s_f[0]);
            v.lam_c[2] = (float)(h[l + 1][0] * s_t[l][1] / P.s_f[1]);
            v.lam_c[3] = (float)(h[l + 1][1] * s_t[l][0] / P.s_f[1]);
            break;
        case VOTE_POSE6DOF: {    // (|xi w| + |w|) sum h1_phi + |xi| h1_z (and y with eta)
            const double hphi = (h[l + 1][0] + h[l + 1][1]) + h[l + 1][2];
            v.lam_c[0] = (float)(hphi * s_t[l][0] / P.s_f[0]);
            v.lam_c[1] = (float)(h[l + 1][3] * s_t[l][9] / P.s_f[0]);
            v.lam_c[2] = (float)(hphi * s_t[l][0] / P.s_f[1]);
            v.lam_c[3] = (float)(h[l + 1][3] * s_t[l][10] / P.s_f[1]);
            break;
        }
        case VOTE_RADIAL5DOF: {  // (|rho w| + |w|) sum h1_phi + |rho| h1_y
            const double hphi = (h[l + 1][0] + h[l + 1][1]) + h[l + 1][2];
            v.lam_c[0] = (float)(hphi * s_t[l][0] / P.s_f[0]);
            v.lam_c[1] = (float)(h[l + 1][3] * s_t[l][6] / P.s_f[0]);
            break;
        }
        }
        bool equal = true;
        if (fam == VOTE_PLANE3D_SPH || fam == VOTE_POSE3DOF) equal = s_t[l][0] == s_t[l][1];
        if (fam == VOTE_POSE6DOF)
            for (int m = 1; m < 9; ++m) equal &= s_t[l][m] == s_t[l][0];
        if (fam == VOTE_RADIAL5DOF)
            for (int m = 1; m < 6; ++m) equal &= s_t[l][m] == s_t[l][0];
        if (!equal) {
            set_err("internal: unequal essential steps at level %d", l);
            return VOTE_EINTERNAL;
        }
    }
    return VOTE_OK;
}

// Upper bounds on the Lipschitz factors Lambda_ji from bounds T_m on |t_m|.
static void lambda_max(int fam, const double *T, double *lam) {
    switch (fam) {
    case VOTE_LINE2D: lam[0] = T[0]; break;
    case VOTE_PLANE3D_SPH:
        lam[0] = std::sqrt(T[0] * T[0] + T[1] * T[1] + T[2] * T[2]);
        lam[1] = std::sqrt(T[0] * T[0] + T[1] * T[1]);
        break;
    case VOTE_POSE3DOF: lam[0] = lam[1] = std::sqrt(T[0] * T[0] + T[1] * T[1]); break;
    case VOTE_RAYS3D: lam[0] = T[0]; lam[1] = T[1]; break;
    case VOTE_POINTSET2D: lam[0] = T[0]; lam[1] = T[1]; lam[2] = T[1]; lam[3] = T[0]; break;
    case VOTE_AFFINE4D: lam[0] = T[0]; lam[1] = T[1]; lam[2] = T[2]; break;
    case VOTE_POSE6DOF: {
        const double nw = std::sqrt(T[0] * T[0] + T[1] * T[1] + T[2] * T[2]);
        const double nxw = std::sqrt(T[3] * T[3] + T[4] * T[4] + T[5] * T[5]);
        const double nyw = std::sqrt(T[6] * T[6] + T[7] * T[7] + T[8] * T[8]);
        lam[0] = lam[1] = lam[2] = nxw + nw;
        lam[3] = T[9];
        lam[4] = lam[5] = lam[6] = nyw + nw;
        lam[7] = T[10];
        break;
    }
    case VOTE_RADIAL5DOF: {
        const double nrw = std::sqrt(T[0] * T[0] + T[1] * T[1] + T[2] * T[2]);
        const double nw = std::sqrt(T[3] * T[3] + T[4] * T[4] + T[5] * T[5]);
        lam[0] = lam[1] = lam[2] = nrw + nw;
        lam[3] = T[6];
        break;
    }
    }
}

// Per-solve level constants, once the root records' largest |q| are known
// (qmax[j] for free, qmax[nd + m] for essential parameters): bounds on the records'
// fields at every level, and the record format of
// each level (16-bit fields where every bound stays below 32000; level 0, and
// every level in plain FP64 mode, 32-bit).  A level-l record (l >= 1) passed the
// UB test of level l-1, so |f| <= that radius; |q_t| only shrinks as steps double.
static void finalize_levels(vote_ctx *c, const unsigned *qmax) {
    const Problem &P = c->P;
    double rprev[GV_MAXD] = {};
    for (int l = 0; l < P.L; ++l) {
        Level &v = c->lev[l];
        double T[GV_MAXT], lam[GV_MAXD * GV_MAXD], qtb[GV_MAXT], sigma[GV_MAXT];
        family_sigma(P.fam, v.h, sigma);
        bool fits = c->precision == 1 && l >= 1;
        for (int m = 0; m < P.le; ++m) {
            double ratio = v.s_t[m] / c->lev[0].s_t[m];                 // a power of two >= 1
            qtb[m] = std::floor((double)qmax[P.nd + m] / ratio) + 1.0;
            T[m] = (qtb[m] + 1.0) * v.s_t[m];
            fits &= qtb[m] <= 32000.0;
        }
        lambda_max(P.fam, T, lam);
        for (int j = 0; j < P.nd; ++j) {
            double R = v.Rbase[j];
            for (int i = 0; i < P.k; ++i) R += lam[j * P.k + i] * v.h1[i];
            R = (R + v.A1[j]) * 1.001;
            double qfb = l == 0 ? (double)qmax[j] + 1.0 : std::ceil(rprev[j] / P.s_f[j]) + 1.0;
            // the screen's band (kBandTest (M + R), and M + Lc for the lower bound), as a
            // multiple of the record's radius: M <= mag R
            double mag = kMagPerRadius;
            if (l == 0) {
                double M = qfb + v.Hs[j];
                for (int m = 0; m < P.le; ++m) M += qtb[m] * v.gscale[j][m] * sigma[m];
                mag = M / v.rc0[j];
            }
            const double bandR = 1.01 * kBandTest * (mag + 1.0);
            v.kappa[j] = (float)(1.01 * bandR * (2.0 + bandR));
            v.bandL[j] = (float)(1.01 * kBandTest * mag);
            v.bandL0[j] = (float)(1.01 * kBandTest) * v.Lc[j];
            fits &= qfb <= 32000.0;
            rprev[j] = R;
        }
        v.q16 = fits ? 1 : 0;
    }
    // a level keeps 16-bit records only if every deeper level does (the bounds shrink
    // with depth, so this only guards the format sequence the emit pass supports)
    for (int l = P.L - 2; l >= 0; --l) c->lev[l].q16 &= c->lev[l + 1].q16;
    for (int l = 0; l < P.L; ++l) c->lev[l].q16_next = l + 1 < P.L ? c->lev[l + 1].q16 : 0;
}

// ---------------------------------------------------------------------------
// device memory
// ---------------------------------------------------------------------------
// keep: bytes of the old contents to preserve
static vote_status ensure(vote_ctx *c, DevBuf &b, size_t bytes, size_t keep = 0) {
    if (bytes <= b.bytes && b.p) return VOTE_OK;
    size_t want = bytes + bytes / 4 + 256;
    void *old = keep ? b.p : nullptr;
    if (old) want = std::max(want, 2 * b.bytes);     // appended to: few copies of the old contents
    if (b.p && !old) {
        CK(cudaFreeAsync(b.p, c->stream));
        b.p = nullptr;
        b.bytes = 0;
    }
    ++c->alloc_count;
    if (c->fault_alloc_at && c->alloc_count == c->fault_alloc_at) {
        set_err("injected allocation failure (allocation %lld)", (long long)c->alloc_count);
        c->fault_hit = true;
        return VOTE_ENOMEM;
    }
    cudaError_t e = cudaMallocAsync(&b.p, want, c->stream);
    if (e != cudaSuccess) {
        cudaGetLastError();
        b.p = old;
        set_err("device allocation of %zu bytes failed: %s", want, cudaGetErrorString(e));
        return VOTE_ENOMEM;
    }
    if (old) {
        CK(cudaMemcpyAsync(b.p, old, keep, cudaMemcpyDeviceToDevice, c->stream));
        CK(cudaFreeAsync(old, c->stream));
    }
    b.bytes = want;
    return VOTE_OK;
}

static void release(vote_ctx *c, DevBuf &b) {
    if (b.p) cudaFreeAsync(b.p, c->stream);
    b.p = nullptr;
    b.bytes = 0;
}

// Gives back what solves have grown: the levels, the beam, the steps' scratch, the rotations'
// and the grouping's tables, here and in the workers of batches (no solve of this context is
// running).
static void release_working(vote_ctx *c) {
    for (vote_ctx *w : c->workers) release_working(w);
    for (int l = 0; l <= GV_MAXL + 1; ++l) {
        LevelStore &s = l <= GV_MAXL ? c->ls[l] : c->beam;
        DevBuf *bufs[] = {&s.rec, &s.mult, &s.tile_cell, &s.key, &s.rbeg, &s.rcnt, &s.ub, &s.lb};
        for (DevBuf *b : bufs) release(c, *b);
        s.ncells = s.nrecs = 0;
        if (l <= GV_MAXL) release(c, c->rot[l]), release(c, c->rotflag[l]);
    }
    DevBuf *bufs[] = {&c->alive, &c->geo64, &c->geo32, &c->geo32lo, &c->cnt, &c->tinfo, &c->ballot, &c->lballot,
                      &c->uns, &c->off, &c->cbase, &c->child_idx, &c->keepflag, &c->recn, &c->bsums, &c->g_table,
                      &c->g_owner, &c->g_newpos, &c->g_ccount, &c->g_ccur, &c->g_rbeg, &c->g_rec, &c->g_mult,
                      &c->g_tile, &c->beam_src};
    for (DevBuf *b : bufs) release(c, *b);
    cudaStreamSynchronize(c->stream);                      // free for others
}

// record fields and basis values of a family, from its device definition
static int family_nfp(int fam) {
    switch (fam) {
    case VOTE_LINE2D: return Fam<FAM_LINE2D>::NFP;
    case VOTE_PLANE3D_SPH: return Fam<FAM_PLANE3D_SPH>::NFP;
    case VOTE_POSE3DOF: return Fam<FAM_POSE3DOF>::NFP;
    case VOTE_RAYS3D: return Fam<FAM_RAYS3D>::NFP;
    case VOTE_POINTSET2D: return Fam<FAM_POINTSET2D>::NFP;
    case VOTE_AFFINE4D: return Fam<FAM_AFFINE4D>::NFP;
    case VOTE_RADIAL5DOF: return Fam<FAM_RADIAL5DOF>::NFP;
    default: return Fam<FAM_POSE6DOF>::NFP;
    }
}
static int family_nb(int fam) {
    switch (fam) {
    case VOTE_LINE2D: return Fam<FAM_LINE2D>::NB;
    case VOTE_PLANE3D_SPH: return Fam<FAM_PLANE3D_SPH>::NB;
    case VOTE_POSE3DOF: return Fam<FAM_POSE3DOF>::NB;
    case VOTE_RAYS3D: return Fam<FAM_RAYS3D>::NB;
    case VOTE_POINTSET2D: return Fam<FAM_POINTSET2D>::NB;
    case VOTE_AFFINE4D: return Fam<FAM_AFFINE4D>::NB;
    case VOTE_RADIAL5DOF: return Fam<FAM_RADIAL5DOF>::NB;
    default: return Fam<FAM_POSE6DOF>::NB;
    }
}
// basis values whose changes depend on the cell
static int family_nbg(int fam) {
    switch (fam) {
    case VOTE_PLANE3D_SPH: return Fam<FAM_PLANE3D_SPH>::NBG;
    case VOTE_POSE3DOF: return Fam<FAM_POSE3DOF>::NBG;
    case VOTE_POSE6DOF: return Fam<FAM_POSE6DOF>::NBG;
    case VOTE_RADIAL5DOF: return Fam<FAM_RADIAL5DOF>::NBG;
    default: return 0;
    }
}
static bool family_rotation(int fam) { return fam == VOTE_POSE6DOF || fam == VOTE_RADIAL5DOF; }
static_assert((int)VOTE_LINE2D == FAM_LINE2D && (int)VOTE_PLANE3D_SPH == FAM_PLANE3D_SPH &&
                  (int)VOTE_POSE3DOF == FAM_POSE3DOF && (int)VOTE_POSE6DOF == FAM_POSE6DOF &&
                  (int)VOTE_RAYS3D == FAM_RAYS3D && (int)VOTE_POINTSET2D == FAM_POINTSET2D &&
                  (int)VOTE_AFFINE4D == FAM_AFFINE4D && (int)VOTE_RADIAL5DOF == FAM_RADIAL5DOF,
              "family numbers");

// bytes of one record of level l (its format is fixed per solve by finalize_levels)
static int rec_bytes_at(const vote_ctx *c, int l) {
    return 4 * rec_words(family_nfp(c->P.fam), l < c->P.L && c->lev[l].q16);
}

// Every array is checked against its own allocated size (ensure returns at once
// when it is large enough), so no separate capacity figure can drift from the
// allocations.  slots: record slots (a multiple of 32) in level l's format.  What the
// level holds (its ncells, nrecs) is preserved.
static vote_status ensure_level(vote_ctx *c, LevelStore &s, int l, size_t slots, size_t cells) {
    const size_t nr = (size_t)s.nrecs, nc = (size_t)s.ncells;
    if (slots > 0) {
        // one tile of padding: the count pass loads a tile ahead
        TRY(ensure(c, s.rec, (slots + 32) * rec_bytes_at(c, l), nr * rec_bytes_at(c, l)));
        if (c->group) TRY(ensure(c, s.mult, slots * 4, nr * 4));   // without grouping every mult is 1
        TRY(ensure(c, s.tile_cell, (slots / 32) * 4, (nr / 32) * 4));
    }
    if (cells > 0) {
        TRY(ensure(c, s.key, cells * 8, nc * 8));
        TRY(ensure(c, s.rbeg, cells * 8, nc * 8));
        TRY(ensure(c, s.rcnt, cells * 4, nc * 4));
        TRY(ensure(c, s.ub, cells * 4, nc * 4));
        TRY(ensure(c, s.lb, cells * 4, nc * 4));
    }
    return VOTE_OK;
}

static RecView rec_view(vote_ctx *c, const LevelStore &s) {
    RecView v;
    v.rec = (uint32_t *)s.rec.p;
    v.mult = c->group ? (uint32_t *)s.mult.p : nullptr;
    v.tile_cell = (uint32_t *)s.tile_cell.p;
    return v;
}

static CellView cell_view(const LevelStore &s) {
    CellView v;
    v.key = (uint64_t *)s.key.p;
    v.rbeg = (uint64_t *)s.rbeg.p;
    v.rcnt = (uint32_t *)s.rcnt.p;
    v.ub = (uint32_t *)s.ub.p;
    v.lb = (uint32_t *)s.lb.p;
    return v;
}

static Scalars *dsc(vote_ctx *c) { return (Scalars *)c->scal.p; }

static vote_status read_scalars(vote_ctx *c) {
    CK(cudaMemcpyAsync(c->h_sc, c->scal.p, sizeof(Scalars), cudaMemcpyDeviceToHost, c->stream));
    CK(cudaStreamSynchronize(c->stream));
    return VOTE_OK;
}

// ---------------------------------------------------------------------------
// kernel timing (CUDA events on the context's stream, read after the stream has
// passed them)
// ---------------------------------------------------------------------------
// Events are recorded in sequence; the interval ending at event i is charged to
// class ev_cls[i] (-1: not charged).  They are read once the stream has passed
// them (at the next synchronisation).
static void ev_mark(vote_ctx *c, int cls) {
    if (!c->kernel_timing || c->ev_n >= vote_ctx::kEv) return;
    cudaEventRecord(c->ev[c->ev_n], c->stream);
    c->ev_cls[c->ev_n] = cls;
    ++c->ev_n;
}

static void ev_collect(vote_ctx *c) {
    if (!c->kernel_timing) return;
    for (int i = 1; i < c->ev_n; ++i) {
        float ms;
        int cls = c->ev_cls[i];
        if (cls >= 0 && cudaEventElapsedTime(&ms, c->ev[i - 1], c->ev[i]) == cudaSuccess) {
            c->kms[cls] += ms;
            c->klaunch[cls] += 1;
        }
    }
    c->ev_n = 0;
}

// ---------------------------------------------------------------------------
// search
// ---------------------------------------------------------------------------

// rotation tables hold at most 2^kRotBits cells of the rotation coordinates per level
// (151 MB: seven levels of the 6DoF workload); deeper levels evaluate rotations directly
static const int kRotBits = 21;
// angular coordinates of at most this many splits have a (sin, cos) table (2 MB)
static const int kSincosBits = 16;

// Without dives the search goes depth first: the leaves below its first steps are then the
// only ones that raise the pruning bound.  Level by level as with dives, point sets (150 x
// 150, dives off) took 15.4 ms and 7.2 GB, 6.5 ms and 4.1 GB depth first.  So it does where
// memory is short: a level then holds what one step has left.
static bool depth_first(const vote_ctx *c) { return c->lean || !(c->dive && c->prune); }

// records of a step where memory is short
static int64_t lean_records(const vote_ctx *c) {
    return std::min(c->chunk_records, (int64_t)1 << (c->P.d >= 6 ? 21 : 23));
}

// Records of an expansion step.  Depth first every step starts from the bounds that the one
// before found, so with 16 and more children a default step is half as large: steps of 1 / 2
// / 4 times 2^23 records (6DoF 2^21), dives off, ms: point sets 4.8 / 6.5 / 9.8, radial 23 /
// 13 / 16, affine 4-space 88 / 75 / 68 and 178 / 146 / 130, 6DoF 37 / 34 / 39.
static int64_t step_records(const vote_ctx *c) {
    if (c->lean) return lean_records(c);
    return depth_first(c) && !c->chunk_set && c->P.d >= 4 ? c->chunk_records / 2 : c->chunk_records;
}

// records expanded with lower bounds outside dives
static int64_t lb_records(int d) { return d <= 3 ? (int64_t)1 << 28 : (int64_t)1 << 22; }

// Shape of a level's expansion steps.
struct StepDims {
    int kf, dm, lns, ns, nfs;  // child slots (see Chunk)
    int kg, ng, gf, NB, NBG;   // geometry slots, floats per cell, basis values
    bool rotation;
};

static StepDims step_dims(const vote_ctx *c, int l) {
    const Problem &P = c->P;
    const Level &lev = c->lev[l];
    StepDims s;
    s.kf = s.lns = 0;
    s.dm = lev.split_mask >> P.k;
    for (int j = 0; j < P.d; ++j) {
        const int split = (lev.split_mask >> j) & 1;
        s.lns += split;
        if (j < P.k) s.kf += split;
    }
    s.ns = 1 << s.lns;
    s.nfs = 1 << s.kf;
    s.NB = family_nb(P.fam);
    s.NBG = family_nbg(P.fam);
    s.rotation = family_rotation(P.fam);
    // geometry slots: the free slots, without the linear tail coordinate's bit
    s.kg = s.rotation ? s.kf - ((lev.split_mask >> (P.k - 1)) & 1) : s.kf;
    s.ng = 1 << s.kg;
    s.gf = s.NBG * s.ng + s.NBG;
    return s;
}

// Tables of a level's geometry; need64: the FP64 changes are stored per cell (plain FP64
// mode, or a table is missing).
static vote_status ensure_tables(vote_ctx *c, int l, const StepDims &s, bool *need64) {
    const Problem &P = c->P;
    *need64 = c->precision == 0;
    if (s.rotation) {
        for (int x = l; x <= l + 1; ++x) {       // this level's and the next level's rotations
            int bits = 0;
            for (int j = 0; j < 3; ++j) bits += std::min(x, P.Lj[j]);
            if (bits > kRotBits || c->rot[x].p) continue;
            const size_t flags = (((size_t)1 << bits) / 32 + 1) * 4;
            TRY(ensure(c, c->rotflag[x], flags));
            CK(cudaMemsetAsync(c->rotflag[x].p, 0, flags, c->stream));
            TRY(ensure(c, c->rot[x], (size_t)72 << bits));
        }
        *need64 |= !c->rot[l].p || !c->rot[l + 1].p;
    } else if (s.NBG) {
        for (int j = 0; j < P.k; ++j) *need64 |= !c->sctab[j].p;
    }
    return VOTE_OK;
}

// Scratch of a step of nc cells and nt tiles; fits: only whether all of it is there.
static vote_status ensure_scratch(vote_ctx *c, const StepDims &s, size_t nc, size_t nt, bool lb, bool need64,
                                  bool *fits = nullptr) {
    const size_t nch = nc * s.ns, ntp = nt > 0 ? nt : 1;
    auto need = [&](DevBuf &b, size_t bytes) {
        if (!fits) return ensure(c, b, bytes);
        if (!b.p || b.bytes < bytes) *fits = false;
        return VOTE_OK;
    };
    if (fits) *fits = true;
    TRY(need(c->alive, nc));
    if (s.NBG) {
        TRY(need(c->geo32, nc * s.gf * 4));
        TRY(need(c->geo32lo, nc * s.NBG * s.ng * 4));
    }
    if (need64) TRY(need(c->geo64, nc * s.nfs * s.NB * 8));
    TRY(need(c->cnt, nch * 4 * (c->group ? 3 : 2)));
    TRY(need(c->child_idx, nch * 4));
    TRY(need(c->cbase, nch * 8));
    TRY(need(c->keepflag, nch * 4));
    TRY(need(c->recn, nch * 4));
    TRY(need(c->bsums, ((nch + 255) / 256) * 16 + 16));
    TRY(need(c->tinfo, (ntp + 2) * 8));
    TRY(need(c->ballot, ntp * s.ns * 4 + 16));       // bulk copies round up to 16 bytes
    TRY(need(c->off, ntp * s.ns * 4 + 16));
    if (lb) TRY(need(c->lballot, ntp * s.ns * 4));
    if (c->precision == 1) TRY(need(c->uns, ntp * 8));
    return VOTE_OK;
}

// A step's chunk over nc cells and nt tiles from (c0, t0) of S, with the scratch's arrays.
static void fill_chunk(vote_ctx *c, int l, const LevelStore &S, const StepDims &s, int64_t c0, int64_t nc, int64_t t0,
                       int64_t nt, bool lb, bool need64, Chunk &ch) {
    const size_t nch = (size_t)nc * s.ns;
    std::memset(&ch, 0, sizeof(ch));
    ch.P = c->P;
    ch.lev = c->lev[l];
    ch.cells = cell_view(S);
    ch.c0 = c0;
    ch.nc = (int)nc;
    ch.ns = s.ns;
    ch.lns = s.lns;
    ch.nfs = s.nfs;
    ch.kf = s.kf;
    ch.dm = s.dm;
    ch.ng = s.ng;
    ch.kg = s.kg;
    ch.gf = s.gf;
    ch.in = rec_view(c, S);
    ch.in_rbeg = (const uint64_t *)S.rbeg.p;
    ch.in_rcnt = (const uint32_t *)S.rcnt.p;
    ch.in_c0 = c0;
    ch.t0 = t0;
    ch.t1 = t0 + nt;
    ch.alive = (uint8_t *)c->alive.p;
    ch.geo64 = need64 ? (double *)c->geo64.p : nullptr;
    for (int j = 0; j < 2; ++j) ch.sincos[j] = (const double2 *)c->sctab[j].p;
    if (s.rotation) {
        ch.rot_par = (double *)c->rot[l].p;
        ch.rot_ch = (double *)c->rot[l + 1].p;
        ch.rot_flag = (unsigned *)c->rotflag[l + 1].p;
    }
    ch.geo32 = (float *)c->geo32.p;
    ch.geo32lo = (float *)c->geo32lo.p;
    ch.crec = (uint32_t *)c->cnt.p;
    ch.clb = ch.crec + nch;
    ch.cub = c->group ? ch.crec + 2 * nch : ch.crec;
    ch.weighted = c->group;
    ch.child_idx = (int32_t *)c->child_idx.p;
    ch.cbase = (unsigned long long *)c->cbase.p;
    ch.sc = dsc(c);
    if (c->trace_cap > 0) {
        ch.trace.cap = (unsigned long long)c->trace_cap;
        ch.trace.level = (int32_t *)c->tr_level.p;
        ch.trace.key = (uint64_t *)c->tr_key.p;
        ch.trace.ub = (uint32_t *)c->tr_ub.p;
        ch.trace.lb = (uint32_t *)c->tr_lb.p;
    }
    ch.prune = c->prune;
    ch.precision = c->precision;
    ch.lb = lb;
    // a trace lists every child's counts; with multiplicities they are not the records'
    if (c->prune && c->precision == 1 && !c->group && c->trace_cap == 0) {
        const int64_t per = nt / (sm_count() * 32);         // tiles per warp, about
        ch.early = per >= 64 ? 64 : (per >= 32 ? 32 : (per >= 16 ? 16 : 1));
    }
    ch.work = c->count_work || c->log >= 2;
    ch.cfail = (uint32_t *)c->child_idx.p;
    ch.spin = c->spin_limit;
    ch.tinfo = (int2 *)c->tinfo.p;
    ch.ballot = (uint32_t *)c->ballot.p;
    ch.lballot = (uint32_t *)c->lballot.p;
    ch.uns = (uint2 *)c->uns.p;
    ch.off = (uint32_t *)c->off.p;
    if (!ch.lev.leaf_children) {
        ch.next_cells = cell_view(c->ls[l + 1]);
        ch.next_c0 = c->ls[l + 1].ncells;
        ch.next_r0 = c->ls[l + 1].nrecs;
        ch.out = rec_view(c, c->ls[l + 1]);
    }
}

// Waits until step number seq has reported into v (every step's report is its last but one
// or last kernel; the stream's state is looked at now and then, so a failed launch ends it).
// It waits as the process has chosen for the device (cudaSetDeviceFlags, read once per solve):
// blocked after polling for as long as the shortest steps take; or polling, with the core given
// up every microsecond or so from 100 us on unless spinning was asked for (a yield after every
// poll from 20 us on took 5 of 427 us on 10,000 lines).  A search that only polled took 442 ms of
// CPU time in 495 ms under cudaDeviceScheduleBlockingSync (planes, 1e6 points, eps 0.03).
static vote_status wait_report(vote_ctx *c, const LevInfo *v, long long seq) {
    auto reported = [&] { return __atomic_load_n(&v->seq, __ATOMIC_ACQUIRE) == seq; };
    const unsigned how = c->sched;
    for (unsigned i = how == cudaDeviceScheduleBlockingSync ? 0x4000u : 0x20000u; i > 0; --i)
        if (reported()) return VOTE_OK;
    if (how == cudaDeviceScheduleBlockingSync) {
        CK(cudaStreamSynchronize(c->stream));
    } else {
        for (unsigned i = 1; !reported(); ++i) {
            if (how != cudaDeviceScheduleSpin && !(i & 0x3ffu)) std::this_thread::yield();
            if (i & 0xffffu) continue;           // looking at the stream takes the lock that other threads launch under
            const cudaError_t e = cudaStreamQuery(c->stream);
            if (e == cudaErrorNotReady) {
                cudaGetLastError();
                continue;
            }
            CK(e);
            break;
        }
    }
    if (reported()) return VOTE_OK;
    set_err("internal: an expansion step ended without its report");
    return VOTE_EINTERNAL;
}

// Lower bounds cost a third of the count pass.  Leaves need none (their own counts are
// one).  Above them they prune before the first leaf is reached, and with d <= 3 they
// rank the cells of a dive; once lb_records() records are expanded, only dives take them.
// All steps / none / this rule, ms: planes of 1e4 points 38 / 98 / 34, of 1e6 points
// 810 / 741 / 744, 10,000 lines 0.67 / 0.96 / 0.67, affine 4-space 46 / 40 / 41.
static bool wants_lb(const vote_ctx *c, int l, bool beam) {
    return c->trace_cap > 0 || (!c->lev[l].leaf_children && (beam || c->expanded < lb_records(c->P.d)));
}

// Up to these children a kernel of one block lays them out; above, two kernels do.  The
// chain only knows a bound, mostly several times the real number.
static const int64_t kSmallStep = 2048, kSmallChain = 8192;

// Expand a chunk of level-l cells taken from the top of the level's stack, or, in the
// dive, all cells of the beam store (a selection of level l).
static vote_status expand_chunk(vote_ctx *c, int l, bool beam = false) {
    LevelStore &S = beam ? c->beam : c->ls[l];
    const Level &lev = c->lev[l];
    // chunk: cells [c0, c1) from the top of the stack, about step_records(c) records
    const int64_t c1 = S.ncells, r1 = S.nrecs;
    int64_t avg = S.nrecs / (S.ncells > 0 ? S.ncells : 1);
    const int64_t step = step_records(c);
    int64_t K = step / (avg > 0 ? avg : 1);
    if (K < 1) K = 1;
    if (K > (1 << 22)) K = 1 << 22;
    int64_t c0, r0;
    for (;;) {
        c0 = c1 - K > 0 ? c1 - K : 0;
        if (beam) c0 = 0;
        if (c0 == 0 && !c->kernel_timing && (beam || K == 1 || r1 <= 2 * step)) {
            r0 = 0;                                  // the level's first record: nothing to read back
            break;
        }
        CK(cudaMemcpyAsync(c->h_tmp, (uint64_t *)S.rbeg.p + c0, 8, cudaMemcpyDeviceToHost, c->stream));
        CK(cudaStreamSynchronize(c->stream));
        ev_collect(c);
        r0 = (int64_t)c->h_tmp[0];
        if (beam || r1 - r0 <= 2 * step || K == 1) break;
        K = K / 2;
    }
    nvtxRangePushA("expand_chunk");
    const int nc = (int)(c1 - c0);
    const StepDims dims = step_dims(c, l);
    const int ns = dims.ns;
    const size_t nch = (size_t)nc * ns;
    const int rb = rec_bytes_at(c, l);
    bool need64;
    TRY(ensure_tables(c, l, dims, &need64));
    if (!lev.leaf_children) TRY(ensure_level(c, c->ls[l + 1], l + 1, 0, (size_t)c->ls[l + 1].ncells + nch));
    const bool lb = wants_lb(c, l, beam), grouping = c->group && r1 - r0 > 32;
    c->expanded += r1 - r0;
    // canonical records need at most the slots of the originals plus one tile per cell
    const size_t gslots = (size_t)(r1 - r0) + 32 * (size_t)nc;
    TRY(ensure_scratch(c, dims, (size_t)nc, grouping ? gslots / 32 : (size_t)(r1 - r0) / 32, lb, need64));
    Chunk ch;
    fill_chunk(c, l, S, dims, c0, nc, r0 / 32, (r1 - r0) / 32, lb, need64, ch);

    if (grouping) {
        // canonization's grouping: merge records with equal (cell, q_f, q_t)
        const size_t nr = (size_t)(r1 - r0);
        size_t cap = 1;
        while (cap < nr * 2) cap <<= 1;
        TRY(ensure(c, c->g_table, cap * 4));
        TRY(ensure(c, c->g_owner, nr * 4));
        TRY(ensure(c, c->g_newpos, nr * 4));
        TRY(ensure(c, c->g_ccount, (size_t)nc * 4));
        TRY(ensure(c, c->g_ccur, (size_t)nc * 4));
        TRY(ensure(c, c->g_rbeg, (size_t)nc * 8));
        TRY(ensure(c, c->g_rec, (gslots + 32) * rb));       // one tile of padding, as for a level
        TRY(ensure(c, c->g_mult, gslots * 4));
        TRY(ensure(c, c->g_tile, (gslots / 32) * 4));
        CK(cudaMemsetAsync(c->g_table.p, 0, cap * 4, c->stream));
        CK(cudaMemsetAsync(c->g_ccount.p, 0, (size_t)nc * 4, c->stream));
        CK(cudaMemsetAsync(c->g_ccur.p, 0, (size_t)nc * 4, c->stream));
        RecView gv;
        gv.rec = (uint32_t *)c->g_rec.p;
        gv.mult = (uint32_t *)c->g_mult.p;
        gv.tile_cell = (uint32_t *)c->g_tile.p;
        ev_mark(c, -1);
        launch_group(ch, (uint32_t *)c->g_table.p, (uint32_t)(cap - 1), (uint32_t *)c->g_owner.p,
                     (uint32_t *)c->g_ccount.p, (uint32_t *)c->g_ccur.p, (uint32_t *)c->g_newpos.p,
                     (uint64_t *)c->g_rbeg.p, (unsigned long long *)c->h_tmp_dev(), gv, c->stream);
        ev_mark(c, VOTE_K_GROUP);
        CK(cudaGetLastError());
        CK(cudaMemcpyAsync(c->h_tmp, c->h_tmp_dev(), 24, cudaMemcpyDeviceToHost, c->stream));
        CK(cudaStreamSynchronize(c->stream));
        const int64_t gs = (int64_t)c->h_tmp[0];
        c->stats.launches += 4;
        c->kbytes[VOTE_K_GROUP] += (double)nr * (rb + 4) * 2;
        c->lv_gout[l] += (int64_t)c->h_tmp[1];
        c->lv_gin[l] += (int64_t)c->h_tmp[2];
        ch.in = gv;
        ch.in_rbeg = (const uint64_t *)c->g_rbeg.p;
        ch.in_rcnt = (const uint32_t *)c->g_ccount.p;
        ch.in_c0 = 0;
        ch.t0 = 0;
        ch.t1 = gs / 32;
    }
    const int64_t nt = ch.t1 - ch.t0;
    ch.host = c->h_info + GV_MAXL + 1;
    ch.seq = ++c->steps;
    ev_mark(c, -1);
    const int nprep = launch_prep(ch, c->stream);
    ev_mark(c, VOTE_K_CELL_GEO);
    launch_count(ch, c->stream);
    ev_mark(c, VOTE_K_TEST_COUNT);
    const bool small = !grouping && (int64_t)nch <= kSmallStep;
    launch_tile_scan(ch, c->stream);
    const int nchild = launch_child_alloc(ch, small, (uint32_t *)c->keepflag.p, (uint32_t *)c->recn.p,
                                                      (unsigned long long *)c->bsums.p, c->stream);
    ev_mark(c, VOTE_K_CHILDREN);
    // algorithmic bytes: the records of whole tiles read, the ballots written (those of the
    // tiles that the count pass leaves out, and what the emit pass reads: at the solve's end)
    c->kbytes[VOTE_K_TEST_COUNT] += (double)nt * 32 * rb + (double)nt * ns * 4;
    c->kbytes[VOTE_K_CELL_GEO] += (double)nc * (8 + 4);
    CK(cudaGetLastError());
    c->stats.chunks++;
    c->stats.launches += 2 + nprep + nchild + (c->precision == 1);
    c->stats.cells += nc;
    c->lv_cells[l] += nc;
    c->lv_recs[l] += nt * 32;
    S.ncells = c0;
    S.nrecs = r0;
    if (lev.leaf_children) {
        if (c->log >= 2) {
            const double left0 = (double)c->h_sc->left_bytes;
            TRY(read_scalars(c));
            std::fprintf(stderr, "[vote] step %lld level %d: %lld cells, %lld tiles, count %.0f B, leaves\n",
                         (long long)c->stats.chunks - 1, l, (long long)nc, (long long)nt,
                         (double)nt * 32 * rb + (double)nt * ns * 4 - ((double)c->h_sc->left_bytes - left0));
        }
        c->stats.leaves += (int64_t)nch;
        nvtxRangePop();
        return VOTE_OK;
    }
    TRY(wait_report(c, ch.host, ch.seq));
    LevelStore &N = c->ls[l + 1];
    int64_t new_cells = ch.host->stored_cells, new_slots = ch.host->stored_recs;
    if (new_slots > 0) {
        TRY(ensure_level(c, N, l + 1, (size_t)(N.nrecs + new_slots), 0));
        ch.out = rec_view(c, N);
        if (ch.work) {
            launch_emit_work(ch, rb, c->stream);
            c->stats.launches += 1;
        }
        ev_mark(c, -1);
        if (!launch_emit(ch, c->stream)) {
            set_err("internal: no emit pass for record formats %d -> %d", lev.q16, lev.q16_next);
            return VOTE_EINTERNAL;
        }
        c->stats.launches += 1;
        ev_mark(c, VOTE_K_TEST_EMIT);
        c->kbytes[VOTE_K_TEST_EMIT] += (double)new_slots * rec_bytes_at(c, l + 1);
    }
    CK(cudaGetLastError());
    if (c->log >= 2) {
        // the running counters (a synchronisation per step: logging only)
        const double left0 = (double)c->h_sc->left_bytes, read0 = (double)c->h_sc->emit_bytes;
        TRY(read_scalars(c));
        const double left = (double)c->h_sc->left_bytes - left0, read = (double)c->h_sc->emit_bytes - read0;
        std::fprintf(stderr, "[vote] step %lld level %d: %lld cells, %lld tiles, count %.0f B, emit %.0f B, "
                     "%lld child cells, %llu tests, %llu FP64 and %llu double-float rechecks so far\n",
                     (long long)c->stats.chunks - 1, l, (long long)nc, (long long)nt,
                     (double)nt * 32 * rb + (double)nt * ns * 4 - left, read + (double)new_slots * rec_bytes_at(c, l + 1),
                     (long long)new_cells, c->h_sc->tests, c->h_sc->rechecks, c->h_sc->rechecks_df);
    }
    N.ncells += new_cells;
    N.nrecs += new_slots;
    if (N.nrecs > c->stats.peak_records) c->stats.peak_records = N.nrecs;
    nvtxRangePop();
    return VOTE_OK;
}

static vote_status replay(vote_ctx *c, const double *surfaces, int64_t n, int lam, uint64_t key, uint32_t *reach,
                          int64_t *ub, int64_t *lb) {
    CK(cudaMemsetAsync(&dsc(c)->replay_ub, 0, 16, c->stream));
    ev_mark(c, -1);
    if (lam > 0)
        launch_path_geo(c->P, (const Level *)c->levs_dev.p, lam, key, nullptr, (PathStep *)c->path.p, c->stream);
    launch_replay(c->P, (const Level *)c->levs_dev.p, (const PathStep *)c->path.p, lam, surfaces, n, reach,
                  dsc(c), c->stream);
    c->stats.launches += lam > 0 ? 2 : 1;
    ev_mark(c, VOTE_K_REPLAY);
    CK(cudaGetLastError());
    TRY(read_scalars(c));
    ev_collect(c);
    c->kbytes[VOTE_K_REPLAY] += (double)n * (8 * c->P.np) + (double)((n + 31) / 32) * 4;
    *ub = (int64_t)c->h_sc->replay_ub;
    *lb = (int64_t)c->h_sc->replay_lb;
    return VOTE_OK;
}

// A dive takes max(kBeamRecords, level's records / beam_divisor(d)) records of a level.
// Measured (GB300, three instances per family, ms): 2^17, 2^19 and 2^20 records give
// 13.6, 12.5 and 13.9 on the batch of 24 3DoF problems (a larger beam opens more than
// it must) and 1.23, 0.70 and 0.70 on 10,000 lines (a smaller one takes more dependent
// steps than a level that is opened whole).  Divisors 4 / 8 / 16 / 32 / 64, mean of four
// instances, ms: point sets (300 x 300) 12.1 / 10.7 / 10.3 / 10.4 / 10.4, affine 4-space (1e4
// points) 33.1 / 28.5 / 27.2 / 26.4 / 26.1, radial 19.8 / 15.9 / 12.6 / 12.4 / 11.4, 6DoF 14.2 /
// 11.3 / 7.2 / 5.5 / 5.5, planes of 1e4 points 21.2 / 16.5 / 14.7 / 14.0 / 13.5, 3DoF of 1e6
// 4.8 / 4.4 / 4.4 / 4.4 / 4.4.  A smaller share can miss the best leaf's ancestor: with d = 4 it
// is 8 because point sets took 16 to 84 and 54 to 87 ms with 16 and 32 instead of 17 while the
// levels after the dive were opened in small steps, as they are where memory is short.
static const int64_t kBeamRecords = (int64_t)1 << 19;
static int64_t beam_divisor(int d) { return d == 4 ? 8 : (d > 4 ? 32 : 16); }

// records expanded into a level between two dives from it: a dive's cost (about a
// millisecond of dependent steps) stays below a few percent of theirs
static const int64_t kDiveEvery = (int64_t)1 << 28;

// A dive: from level l0 down to the leaves, expand on every level the cells with the
// largest UBs, with d <= 3 also those with the largest LBs (k_beam_*).  A level that fits is expanded whole.
static vote_status dive(vote_ctx *c, int l0) {
    for (int l = l0; l < c->P.L; ++l) {
        LevelStore &S = c->ls[l];
        if (S.ncells <= 0) return VOTE_OK;
        int64_t budget = std::max(kBeamRecords, S.nrecs / beam_divisor(c->P.d));
        if (budget > step_records(c)) budget = step_records(c);
        if (S.nrecs <= budget || S.ncells == 1) {
            TRY(expand_chunk(c, l));
            continue;
        }
        const int64_t m = S.ncells;
        c->beam.ncells = c->beam.nrecs = 0;
        TRY(ensure_level(c, c->beam, l, 0, (size_t)m));
        if (!c->beam_sel.p) {
            TRY(ensure(c, c->beam_sel, sizeof(BeamSel)));
            CK(cudaMemsetAsync(c->beam_sel.p, 0, sizeof(BeamSel), c->stream));   // every selection leaves it cleared
        }
        TRY(ensure(c, c->beam_src, (size_t)m * 8));
        TRY(ensure(c, c->bsums, (size_t)((m + 255) / 256) * 16 + 16));
        const LevInfo *v = c->h_info + GV_MAXL + 1;
        const long long seq = ++c->steps;
        c->stats.launches +=
            launch_beam_select(c->P, cell_view(S), m, budget, c->P.d <= 3 ? 2 : 1, (BeamSel *)c->beam_sel.p,
                               (unsigned long long *)c->bsums.p, cell_view(c->beam), (uint64_t *)c->beam_src.p, dsc(c),
                               c->h_info + GV_MAXL + 1, seq, c->stream);
        CK(cudaGetLastError());
        TRY(wait_report(c, v, seq));
        const int64_t nsel = v->stored_cells, rsel = v->stored_recs;
        if (nsel <= 0) {                 // no cell reaches the bound any more (it never falls)
            S.ncells = S.nrecs = 0;
            return VOTE_OK;
        }
        c->beam.ncells = nsel;
        TRY(ensure_level(c, c->beam, l, (size_t)rsel, 0));
        c->beam.nrecs = rsel;
        launch_beam_gather(rec_view(c, S), rec_view(c, c->beam), cell_view(c->beam), (const uint64_t *)c->beam_src.p,
                           nsel, rsel / 32, rec_bytes_at(c, l), c->stream);
        CK(cudaGetLastError());
        c->stats.launches += 1;
        TRY(expand_chunk(c, l, true));
    }
    return VOTE_OK;
}

// The chain: from the root, levels that hold at most kBeamRecords records are expanded
// whole, one after the other.  A level's sizes pass on to the next on the device, and the
// host queues each level's step while the one before runs, with grids and scratch sized
// by bounds from the level before that: without it every step of a few hundred surfaces
// waited 40 us for the host beside 20 us of kernels.  The chain ends at the leaves, at a
// level too large to expand whole (stored for the dives; the step queued for it finds no
// cells), or where nothing is left.  *replayed: the best leaf's mask was replayed into mask.
static vote_status chain(vote_ctx *c, const double *surfaces, int64_t n, uint32_t *mask, bool *replayed) {
    const Problem &P = c->P;
    const int L = P.L;
    *replayed = false;
    const int64_t slots0 = c->ls[0].nrecs, fit = std::min(kBeamRecords, step_records(c)) & ~(int64_t)31;
    if (slots0 > fit || c->group || c->kernel_timing || c->log >= 2) return VOTE_OK;
    TRY(ensure(c, c->linfo, sizeof(LevInfo) * (GV_MAXL + 1)));
    LevInfo *di = (LevInfo *)c->linfo.p;
    Chunk ch, last;                          // of the level at hand, of the one before
    int64_t cells = 1, recs = slots0;        // sizes of the level at hand, once known
    int64_t pcells = 0;                      // and of the one before
    StepDims dims, pdims;
    bool known = true;
    int launches = 0;
    for (int l = 0;;) {
        dims = step_dims(c, l);
        const bool lb = wants_lb(c, l, c->dive && c->prune);
        bool need64, fits;
        TRY(ensure_tables(c, l, dims, &need64));
        // every cell holds at least a tile, and at most as many as the root
        int64_t cb = cells, tb = recs / 32;
        const int64_t cmax = l ? std::min(pcells * pdims.ns, fit / 32) : 1;
        const bool small = cmax * dims.ns <= kSmallChain;
        if (!known) {
            cb = cmax;
            tb = std::min(cb * (slots0 / 32), fit / 32);
            // the step before may still need the scratch that would grow
            TRY(ensure_scratch(c, dims, (size_t)cb, (size_t)tb, lb, need64, &fits));
        }
        if (known || fits) {
            if (l + 1 < L) {
                // room for the next level: most levels need less; else see below
                const int64_t rc = std::min(cb * dims.ns, (int64_t)1 << 14);
                TRY(ensure_level(c, c->ls[l + 1], l + 1, (size_t)std::min(rc * slots0, (int64_t)1 << 17), (size_t)rc));
            }
            if (known) {
                TRY(ensure_scratch(c, dims, (size_t)cb, (size_t)tb, lb, need64));
                launch_chain_start(di + l, cells, recs, c->stream);
            }
            fill_chunk(c, l, c->ls[l], dims, 0, cb, 0, tb, lb, need64, ch);
            ch.dyn = di + l;
            ch.early = 0;                    // small steps: nothing to gain
            ch.host = c->h_info + l + 1;
            ch.seq = ++c->steps;
            ch.fit_recs = fit;
            if (l + 1 < L) {
                const LevelStore &N = c->ls[l + 1];
                ch.cap_cells = (int64_t)std::min(std::min(N.key.bytes, N.rbeg.bytes) / 8,
                                                 std::min(std::min(N.rcnt.bytes, N.ub.bytes), N.lb.bytes) / 4);
                ch.cap_recs = std::min((int64_t)(N.rec.bytes / rec_bytes_at(c, l + 1)) - 32,
                                       (int64_t)(N.tile_cell.bytes / 4) * 32);
            }
            const int nprep = launch_prep(ch, c->stream);
            launch_count(ch, c->stream);
            launch_tile_scan(ch, c->stream);
            const int nchild = launch_child_alloc(ch, small, (uint32_t *)c->keepflag.p, (uint32_t *)c->recn.p,
                                                              (unsigned long long *)c->bsums.p, c->stream);
            if (l + 1 < L && !launch_emit(ch, c->stream)) {
                set_err("internal: no emit pass for record formats %d -> %d", ch.lev.q16, ch.lev.q16_next);
                return VOTE_EINTERNAL;
            }
            CK(cudaGetLastError());
            launches = 2 + nprep + nchild + (c->precision == 1) + (l + 1 < L);
        }
        if (!known) {                        // what the step before stored
            const LevInfo *v = last.host;
            TRY(wait_report(c, v, last.seq));
            cells = v->stored_cells;
            recs = v->stored_recs;
            c->ls[l].ncells = cells;
            c->ls[l].nrecs = recs;
            if (recs > c->stats.peak_records) c->stats.peak_records = recs;
            if (v->overflow) {
                // its counts and ballots stand: make room, lay the children out, emit
                LevelStore &N = c->ls[l];
                N.ncells = N.nrecs = 0;
                TRY(ensure_level(c, N, l, (size_t)recs, (size_t)cells));
                last.nc = (int)pcells;
                last.t1 = c->ls[l - 1].nrecs / 32;
                last.dyn = nullptr;
                last.host = nullptr;
                last.trace.cap = 0;          // its children are in the trace
                last.next_cells = cell_view(N);
                last.out = rec_view(c, N);
                launch_child_alloc(last, false, (uint32_t *)c->keepflag.p, (uint32_t *)c->recn.p,
                                   (unsigned long long *)c->bsums.p, c->stream);
                launch_emit(last, c->stream);
                CK(cudaGetLastError());
                N.ncells = cells;
                N.nrecs = recs;
            }
            c->ls[l - 1].ncells = c->ls[l - 1].nrecs = 0;
            if (cells == 0 || recs > fit) return VOTE_OK;
            known = true;
            if (v->overflow || !fits) continue;      // no step is queued for this level yet
        }
        // the level's step is queued and its sizes are known
        c->stats.chunks++;
        c->stats.launches += launches;       // of the steps that ran: the same whatever was allocated before
        c->stats.cells += cells;
        c->lv_cells[l] += cells;
        c->lv_recs[l] += recs;
        c->expanded += recs;
        c->kbytes[VOTE_K_TEST_COUNT] += (double)recs * rec_bytes_at(c, l) + (double)recs / 32 * dims.ns * 4;
        if (++l == L) {
            c->ls[l - 1].ncells = c->ls[l - 1].nrecs = 0;
            c->stats.leaves += cells * dims.ns;
            break;
        }
        last = ch;
        pcells = cells;
        pdims = dims;
        known = false;
    }
    if (mask) {
        launch_path_geo(P, (const Level *)c->levs_dev.p, L, 0, dsc(c), (PathStep *)c->path.p, c->stream);
        launch_replay(P, (const Level *)c->levs_dev.p, (const PathStep *)c->path.p, L, surfaces, n, mask, dsc(c),
                      c->stream);
        CK(cudaGetLastError());
        c->stats.launches += 2;
        *replayed = true;
    }
    return VOTE_OK;
}

// The search.  The chain from the root; a dive from where it ends; then level by level, shallowest first, so that a
// level's bounds are raised by all of its cells before its children are opened, while
// the next level holds less than one step's records; when every level below is full,
// the deepest first, which bounds the memory (room for 4 steps: a first solve of planes
// with 1e6 points took 1564 ms instead of 1430 ms, more memory being mapped).  Without
// dives, and where memory is short: the deepest level first throughout (depth_first()).  Whenever
// a level has grown large, another dive starts from it: its own UBs and LBs point better
// than those of the levels above.  Measured against one root-to-leaf path of the largest
// UB for n >= 2^17 and the deepest level first: point sets 132 -> 17 ms, 6DoF 47 -> 13,
// radial 70 -> 22, affine 4-space 204 -> 55, planes of 1e4 points 110 -> 54, 3DoF with
// 1e6 matches 12.5 -> 7.9; with the final depth known from the start (VOTE_OPT_INITIAL_LB)
// they took 13.5, -, 19, 52, 47 and 4.4 ms.
static vote_status search(vote_ctx *c, const double *surfaces, int64_t n, uint32_t *mask, bool *replayed) {
    const int L = c->P.L;
    const bool dives = c->dive && c->prune;
    const int64_t full = depth_first(c) ? 0 : std::min(step_records(c), (int64_t)1 << 34);   // records of a full level
    int64_t since[GV_MAXL + 1];          // records expanded into the level since its last dive
    for (int l = 0; l <= L; ++l) since[l] = -1;
    TRY(chain(c, surfaces, n, mask, replayed));
    if (dives)
        for (int l = 0; l < L; ++l)
            if (c->ls[l].ncells > 0) {               // from where the chain ended
                TRY(dive(c, l));
                break;
            }
    for (;;) {
        int l = -1;
        for (int x = 0; x < L; ++x)
            if (c->ls[x].ncells > 0) {
                l = x;
                if (x + 1 == L || c->ls[x + 1].nrecs <= full) break;
            }
        if (l < 0) return VOTE_OK;
        const int64_t before = l + 1 < L ? c->ls[l + 1].nrecs : 0;
        TRY(expand_chunk(c, l));
        if (!dives || l + 1 >= L) continue;
        const int64_t grown = c->ls[l + 1].nrecs - before;
        if (since[l + 1] >= 0) since[l + 1] += grown;
        if (c->ls[l + 1].nrecs > 8 * kBeamRecords && (since[l + 1] < 0 || since[l + 1] > kDiveEvery)) {
            since[l + 1] = 0;
            TRY(dive(c, l + 1));
        }
    }
}

static vote_status solve_inner(vote_ctx *c, const double *surfaces, int64_t n, double *best_point,
                               int64_t *best_leaf, int64_t *depth, uint32_t *mask);

// Per-level counters of the last solve on stderr (VOTE_LOG=1).
static void log_solve(const vote_ctx *c, vote_status st) {
    const vote_stats &x = c->stats;
    std::fprintf(stderr, "[vote] family %d L %d status %d: %.3f s, %lld tests, %lld FP64 rechecks, %lld chunks, "
                 "%lld launches, peak %lld record slots\n", c->P.fam, c->P.L, (int)st, x.seconds,
                 (long long)x.tests, (long long)x.rechecks, (long long)x.chunks, (long long)x.launches,
                 (long long)x.peak_records);
    for (int l = 0; l < c->P.L; ++l) {
        std::fprintf(stderr, "[vote]   level %2d: %lld cells expanded, %lld record slots tested, records %s", l,
                     (long long)c->lv_cells[l], (long long)c->lv_recs[l], c->lev[l].q16 ? "16-bit" : "32-bit");
        if (c->lv_gin[l])
            std::fprintf(stderr, ", grouping %lld -> %lld records (%.4f merged)", (long long)c->lv_gin[l],
                         (long long)c->lv_gout[l], 1.0 - (double)c->lv_gout[l] / (double)c->lv_gin[l]);
        std::fprintf(stderr, "\n");
    }
}

// One solve.  When device memory runs out, what the solve holds is given back and, where no
// other solve of the same call holds memory (alone), it is repeated once depth first in small
// steps, which need the least.  Measured, as a rule and so: 6DoF +-30 deg 39 GB, 48 ms and 6 GB,
// 221 ms; planes of 1e6 points, eps 0.005, 106 GB, 13.0 s and 6 GB, 25.8 s; affine 4-space
// 10 GB, 25 ms and 3.5 GB, 31 ms.
static vote_status solve_device(vote_ctx *c, const double *surfaces, int64_t n, double *best_point,
                                int64_t *best_leaf, int64_t *depth, uint32_t *mask, bool alone = true) {
    nvtxRangePushA("vote_solve");
    c->fault_hit = false;
    vote_status st = solve_inner(c, surfaces, n, best_point, best_leaf, depth, mask);
    if (st != VOTE_OK) cudaStreamSynchronize(c->stream);   // steps in flight report into this context
    if (st == VOTE_ENOMEM && !c->fault_hit) {
        release_working(c);
        if (alone) {
            c->lean = true;
            st = solve_inner(c, surfaces, n, best_point, best_leaf, depth, mask);
            if (st != VOTE_OK) cudaStreamSynchronize(c->stream);
            c->lean = false;
        }
    }
    nvtxRangePop();
    if (c->log) log_solve(c, st);
    return st;
}

static vote_status solve_inner(vote_ctx *c, const double *surfaces, int64_t n, double *best_point,
                               int64_t *best_leaf, int64_t *depth, uint32_t *mask) {
    auto t0 = std::chrono::steady_clock::now();
    const Problem &P = c->P;
    std::memset(&c->stats, 0, sizeof(c->stats));
    for (int l = 0; l < GV_MAXL; ++l) c->lv_cells[l] = c->lv_recs[l] = c->lv_gin[l] = c->lv_gout[l] = 0;
    c->stats.levels = P.L;
    c->evaluated = c->count_work ? 0 : -1;
    if (n < 0 || !best_point || !depth || (n > 0 && !surfaces)) {
        set_err("invalid arguments");
        return VOTE_EINVAL;
    }
    if (n >= (int64_t)1 << 31 || (P.coord_bits > 0 && (uint64_t)n >= (1ull << (64 - P.coord_bits)))) {
        set_err("n = %lld too large", (long long)n);
        return VOTE_EUNSUPPORTED;
    }
    unsigned flags = 0;
    CK(cudaGetDeviceFlags(&flags));
    c->sched = flags & cudaDeviceScheduleMask;
    CK(cudaMemsetAsync(c->scal.p, 0, sizeof(Scalars), c->stream));
    if (c->initial_lb) CK(cudaMemcpyAsync(&dsc(c)->best_lb, &c->initial_lb, 4, cudaMemcpyHostToDevice, c->stream));
    for (int i = 0; i < VOTE_K_CLASSES; ++i) c->kms[i] = c->kbytes[i] = 0, c->klaunch[i] = 0;
    c->ev_n = 0;
    c->trace_written = 0;
    c->trace_overflow = false;
    c->expanded = 0;
    for (int l = 0; l <= P.L; ++l) c->ls[l].ncells = c->ls[l].nrecs = 0;
    uint64_t leafkey = 0;
    int64_t dep = 0;
    bool mask_done = false;
    if (n > 0 && P.L == 0) {
        dep = n;                                   // the domain is a leaf: every surface counts
    } else if (n > 0) {
        const int64_t slots0 = (n + 31) & ~(int64_t)31;
        TRY(ensure_level(c, c->ls[0], 0, (size_t)slots0, 1));
        ev_mark(c, -1);
        launch_lift(P, c->lev[0], (const double *)c->psi0.p, surfaces, n, rec_view(c, c->ls[0]), cell_view(c->ls[0]), dsc(c), c->stream);
        c->stats.launches += 1;
        ev_mark(c, VOTE_K_LIFT);
        CK(cudaGetLastError());
        c->ls[0].ncells = 1;
        c->ls[0].nrecs = slots0;
        TRY(read_scalars(c));
        ev_collect(c);
        c->kbytes[VOTE_K_LIFT] += (double)n * (8 * P.np + rec_bytes_at(c, 0) + (c->group ? 4 : 0));
        if (c->h_sc->err) {
            set_err("surface parameters are not finite or out of the representable range");
            return VOTE_EINVAL;
        }
        finalize_levels(c, c->h_sc->qmax);
        bool replayed = false;
        TRY(search(c, surfaces, n, mask, &replayed));
        TRY(read_scalars(c));
        ev_collect(c);
        if (c->h_sc->err & kErrTimeout) {
            set_err("a bounded device-side wait ran out (bulk copy not completed)");
            return VOTE_ETIMEOUT;
        }
        if (c->h_sc->err) {
            set_err("internal: residual out of range (err %u)", c->h_sc->err);
            return VOTE_EINTERNAL;
        }
        mask_done = replayed;
        unsigned long long bk = c->h_sc->best_key;
        if (bk) {
            dep = (int64_t)(bk >> P.coord_bits);
            leafkey = ~bk & ((1ull << P.coord_bits) - 1ull);
        }
        c->stats.tests = (int64_t)c->h_sc->tests;
        c->stats.records = (int64_t)c->h_sc->records;
        c->stats.rechecks = (int64_t)c->h_sc->rechecks;
        if (c->count_work) c->evaluated = (int64_t)(c->h_sc->tests - c->h_sc->left_tests);
        c->kbytes[VOTE_K_TEST_COUNT] -= (double)c->h_sc->left_bytes;
        c->kbytes[VOTE_K_TEST_EMIT] += (double)c->h_sc->emit_bytes;
        c->trace_written = (int64_t)c->h_sc->trace_n;
        if (c->trace_cap && c->trace_written > c->trace_cap) c->trace_overflow = true;
    }
    *depth = dep;
    for (int j = 0; j < P.d; ++j) {
        int64_t i = (int64_t)((leafkey >> P.coord_shift[j]) & ((1ull << P.Lj[j]) - 1ull));
        if (best_leaf) best_leaf[j] = i;
        best_point[j] = P.lo[j] + (double)(2 * i + 1) * c->h_leaf[j];
    }
    if (mask && n > 0) {
        if (dep > 0 && mask_done) {
            if ((int64_t)c->h_sc->replay_ub != dep) {
                set_err("internal: replayed inlier count %lld != depth %lld", (long long)c->h_sc->replay_ub, (long long)dep);
                return VOTE_EINTERNAL;
            }
        } else if (dep > 0) {
            int64_t ub = 0, lb = 0;
            TRY(replay(c, surfaces, n, P.L, leafkey, mask, &ub, &lb));
            if (ub != dep) {
                set_err("internal: replayed inlier count %lld != depth %lld", (long long)ub, (long long)dep);
                return VOTE_EINTERNAL;
            }
        } else {
            CK(cudaMemsetAsync(mask, 0, (size_t)((n + 31) / 32) * 4, c->stream));
        }
    }
    CK(cudaStreamSynchronize(c->stream));
    c->stats.seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    return VOTE_OK;
}

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------
extern "C" {

const char *vote_last_error(void) { return g_err; }

vote_status vote_create(int family, int d, int k, const double *eps, const double *bounds, vote_ctx **out) {
    if (!out || !eps || !bounds) {
        set_err("null argument");
        return VOTE_EINVAL;
    }
    *out = nullptr;
    vote_ctx *c = new (std::nothrow) vote_ctx();
    if (!c) {
        set_err("out of host memory");
        return VOTE_ENOMEM;
    }
    vote_status s = problem_init(c, family, d, k, eps, bounds);
    if (s != VOTE_OK) {
        delete c;
        return s;
    }
    // step size measured fastest on GB300 (1e6-surface workloads): planes keep almost
    // every cell above the bound, so larger steps only remove per-step overhead;
    // 3DoF prunes well and needs fine depth-first steps
    // a step's children can hold 2^d times its records: of a step of just this size, with
    // 16-bit fields, 9 GB (planes), 4 GB (16 children), 17 GB (radial camera, 6DoF).  A step
    // can be twice as large; what whole solves held is at solve_device().  The count pass needs tens of tiles per warp to share what it knows of a cell: steps of
    // 2^23, 2^24, 2^25, 2^26 records, affine 4-space 37.5, 33.3, 30.1, 30.3 ms, radial 9.6, 9.1,
    // 8.7, 8.4, point sets 7.6, 6.6, 6.4, 6.4; 2^21 to 2^24, 6DoF 6.0, 5.2, 4.7, 4.8.
    c->chunk_records = family == VOTE_PLANE3D_SPH ? (int64_t)1 << 27 : (d >= 6 ? (int64_t)1 << 23 : (int64_t)1 << 25);
    c->family = family;
    if (const char *lg = std::getenv("VOTE_LOG")) c->log = std::atoi(lg) > 0 ? std::atoi(lg) : 0;
    for (int j = 0; j < d; ++j) {
        c->eps_in[j] = eps[j];
        c->bounds_in[2 * j] = bounds[2 * j];
        c->bounds_in[2 * j + 1] = bounds[2 * j + 1];
    }
    cudaError_t e = cudaGetDevice(&c->device);
    if (e == cudaSuccess) e = cudaMallocHost((void **)&c->h_sc, sizeof(Scalars));
    if (e == cudaSuccess) e = cudaMallocHost((void **)&c->h_tmp, 64);
    if (e == cudaSuccess) e = cudaMallocHost((void **)&c->h_info, sizeof(LevInfo) * (GV_MAXL + 2));
    if (e == cudaSuccess) std::memset(c->h_info, 0, sizeof(LevInfo) * (GV_MAXL + 2));
    if (e != cudaSuccess) {
        set_err("CUDA unavailable: %s", cudaGetErrorString(e));
        delete c;
        return VOTE_ECUDA;
    }
    s = ensure(c, c->scal, ((sizeof(Scalars) + 63) / 64) * 64 + 64);
    if (s == VOTE_OK) s = ensure(c, c->levs_dev, sizeof(Level) * (c->P.L > 0 ? c->P.L : 1));
    if (s == VOTE_OK) s = ensure(c, c->path, sizeof(PathStep) * (c->P.L + kPathTail));
    if (s == VOTE_OK) s = ensure(c, c->psi0, sizeof(double) * GV_MAXT);
    if (s == VOTE_OK && c->P.L > 0) {
        launch_root_basis(c->P, c->lev[0], (double *)c->psi0.p, c->stream);
        const int nang = family == VOTE_PLANE3D_SPH ? 2 : (family == VOTE_POSE3DOF ? 1 : 0);
        for (int j = 0; j < nang && s == VOTE_OK; ++j)
            if (c->P.Lj[j] <= kSincosBits) {
                s = ensure(c, c->sctab[j], sizeof(double2) * (((size_t)2 << c->P.Lj[j]) - 1));
                if (s == VOTE_OK) launch_sincos_table(c->P, j, (double2 *)c->sctab[j].p, c->stream);
            }
        e = cudaMemcpyAsync(c->levs_dev.p, c->lev, sizeof(Level) * c->P.L, cudaMemcpyHostToDevice, c->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
        if (e != cudaSuccess) {
            set_err("upload of level constants failed: %s", cudaGetErrorString(e));
            s = VOTE_ECUDA;
        }
    }
    if (s != VOTE_OK) {
        vote_destroy(c);
        return s;
    }
    *out = c;
    return VOTE_OK;
}

vote_status vote_set_option(vote_ctx *c, int key, double v) {
    if (!c) { set_err("null context"); return VOTE_EINVAL; }
    switch (key) {
    case VOTE_OPT_PRECISION:
        if (v != 0 && v != 1) break;
        c->precision = (int)v;
        return VOTE_OK;
    case VOTE_OPT_PRUNE:
        if (v != 0 && v != 1) break;
        c->prune = (int)v;
        return VOTE_OK;
    case VOTE_OPT_CHUNK_RECORDS:
        if (!(v >= 1 && v <= 1e10)) break;
        c->chunk_records = (int64_t)v;
        c->chunk_set = true;
        return VOTE_OK;
    case VOTE_OPT_TRACE_CAP: {
        if (!(v >= 0 && v <= 1e9)) break;
        c->trace_cap = (int64_t)v;
        if (c->trace_cap > 0) {
            size_t m = (size_t)c->trace_cap;
            TRY(ensure(c, c->tr_level, m * 4));
            TRY(ensure(c, c->tr_key, m * 8));
            TRY(ensure(c, c->tr_ub, m * 4));
            TRY(ensure(c, c->tr_lb, m * 4));
        }
        return VOTE_OK;
    }
    case VOTE_OPT_GROUP:
        if (v != 0 && v != 1) break;
        c->group = (int)v;
        return VOTE_OK;
    case VOTE_OPT_FAULT_ALLOC_AT:
        if (!(v >= 0)) break;
        c->fault_alloc_at = (int64_t)v;
        c->alloc_count = 0;
        return VOTE_OK;
    case VOTE_OPT_INITIAL_LB:
        if (!(v >= 0 && v < 4294967295.0)) break;
        c->initial_lb = (uint32_t)v;
        return VOTE_OK;
    case VOTE_OPT_KERNEL_TIMING:
        if (v != 0 && v != 1) break;
        if (v == 1 && !c->ev[0])
            for (int i = 0; i < vote_ctx::kEv; ++i) CK(cudaEventCreate(&c->ev[i]));
        c->kernel_timing = c->count_work = (int)v;
        return VOTE_OK;
    case VOTE_OPT_BATCH_WORKERS:
        if (!(v >= 1 && v <= 32)) break;
        c->batch_workers = (int)v;
        return VOTE_OK;
    case VOTE_OPT_DIVE:
        if (v != 0 && v != 1 && v != 2) break;
        c->dive = (int)v;
        return VOTE_OK;
    case VOTE_OPT_SPIN_LIMIT:
        if (!(v >= 0 && v <= 4294967295.0)) break;
        c->spin_limit = (unsigned)v;
        return VOTE_OK;

    default:
        set_err("unknown option %d", key);
        return VOTE_EINVAL;
    }
    set_err("option %d: value %g out of range", key, v);
    return VOTE_EINVAL;
}

vote_status vote_set_stream(vote_ctx *c, void *stream) {
    if (!c) { set_err("null context"); return VOTE_EINVAL; }
    c->stream = (cudaStream_t)stream;
    return VOTE_OK;
}

vote_status vote_solve(vote_ctx *c, const double *surfaces, int64_t n, double *best_point, int64_t *best_leaf,
                       int64_t *depth, uint32_t *inlier_mask) {
    if (!c) { set_err("null context"); return VOTE_EINVAL; }
    return solve_device(c, surfaces, n, best_point, best_leaf, depth, inlier_mask);
}

vote_status vote_solve_host(vote_ctx *c, const double *surfaces, int64_t n, double *best_point, int64_t *best_leaf,
                            int64_t *depth, uint32_t *inlier_mask) {
    if (!c) { set_err("null context"); return VOTE_EINVAL; }
    if (n < 0 || (n > 0 && !surfaces)) { set_err("invalid arguments"); return VOTE_EINVAL; }
    size_t in_bytes = (size_t)n * c->P.np * 8, words = (size_t)(n + 31) / 32;
    TRY(ensure(c, c->surf_tmp, in_bytes > 0 ? in_bytes : 8));
    TRY(ensure(c, c->mask_tmp, words > 0 ? words * 4 : 4));
    if (n > 0) CK(cudaMemcpyAsync(c->surf_tmp.p, surfaces, in_bytes, cudaMemcpyHostToDevice, c->stream));
    TRY(solve_device(c, (const double *)c->surf_tmp.p, n, best_point, best_leaf, depth,
                     inlier_mask ? (uint32_t *)c->mask_tmp.p : nullptr));
    if (inlier_mask && words) {
        CK(cudaMemcpyAsync(inlier_mask, c->mask_tmp.p, words * 4, cudaMemcpyDeviceToHost, c->stream));
        CK(cudaStreamSynchronize(c->stream));
    }
    return VOTE_OK;
}

vote_status vote_solve_batched(vote_ctx *c, const double *surfaces, const int64_t *offsets, int B,
                               double *best_points, int64_t *best_leaves, int64_t *depths, uint32_t *masks,
                               double *latency_ms) {
    if (!c || !offsets || B < 0 || !best_points || !depths) { set_err("invalid arguments"); return VOTE_EINVAL; }
    std::memset(&c->stats, 0, sizeof(c->stats));     // this batch's counters, even when it is empty
    c->evaluated = c->count_work ? 0 : -1;
    if (offsets[0] != 0) { set_err("offsets[0] must be 0"); return VOTE_EINVAL; }
    for (int b = 0; b < B; ++b)
        if (offsets[b + 1] < offsets[b]) { set_err("offsets must be non-decreasing"); return VOTE_EINVAL; }
    if (B == 0) return VOTE_OK;
    if (offsets[B] > 0 && !surfaces) { set_err("null surfaces"); return VOTE_EINVAL; }
    const int d = c->P.d, np = c->P.np;
    int nw = c->batch_workers < B ? c->batch_workers : B;
    CK(cudaSetDevice(c->device));
    while ((int)c->workers.size() < nw) {     // sub-contexts with their own streams
        vote_ctx *w = nullptr;
        TRY(vote_create(c->family, d, c->P.k, c->eps_in, c->bounds_in, &w));
        cudaStream_t ws;
        cudaError_t e = cudaStreamCreateWithFlags(&ws, cudaStreamNonBlocking);
        if (e != cudaSuccess) { vote_destroy(w); set_err("stream creation failed"); return VOTE_ECUDA; }
        w->stream = ws;
        c->workers.push_back(w);
    }
    for (int i = 0; i < nw; ++i) {
        vote_ctx *w = c->workers[i];
        w->precision = c->precision;
        w->prune = c->prune;
        w->chunk_records = c->chunk_records;
        w->chunk_set = c->chunk_set;
        w->dive = c->dive;
        w->count_work = c->count_work;
        w->group = c->group;
        w->spin_limit = c->spin_limit;
        w->fault_alloc_at = 0;
    }
    std::vector<int64_t> wordoff(B + 1, 0);
    for (int b = 0; b < B; ++b) wordoff[b + 1] = wordoff[b] + (offsets[b + 1] - offsets[b] + 31) / 32;
    CK(cudaStreamSynchronize(c->stream));     // inputs written on the caller's stream are visible
    std::atomic<int> next(0);
    std::atomic<int> failed(0);
    std::vector<int> todo(B), again;          // problems of this turn; those that found no memory in it
    std::mutex again_mutex;
    again.reserve(B);
    for (int b = 0; b < B; ++b) todo[b] = b;
    bool alone = false;                       // this context's other solves hold no memory
    std::vector<vote_status> wst(nw, VOTE_OK);
    std::vector<std::string> wmsg(nw);
    std::vector<vote_stats> wsum((size_t)nw);   // per worker: totals over its problems
    std::vector<int64_t> wevaluated(nw, 0);
    for (auto &x : wsum) std::memset(&x, 0, sizeof(x));
    auto t0 = std::chrono::steady_clock::now();
    auto work = [&](int wi) {
        vote_ctx *w = c->workers[wi];
        cudaSetDevice(c->device);
        for (;;) {
            if (failed.load()) break;
            const int i = next.fetch_add(1);
            if (i >= (int)todo.size()) break;
            const int b = todo[i];
            int64_t n = offsets[b + 1] - offsets[b];
            vote_status st = solve_device(w, surfaces + np * offsets[b], n, best_points + (size_t)b * d,
                                          best_leaves ? best_leaves + (size_t)b * d : nullptr, depths + b,
                                          masks ? masks + wordoff[b] : nullptr, alone);
            if (st == VOTE_ENOMEM && !alone) {   // the other workers go on without this one
                std::lock_guard<std::mutex> lock(again_mutex);
                again.push_back(b);
                break;
            }
            if (st != VOTE_OK) {
                wst[wi] = st;
                wmsg[wi] = g_err;
                failed.store(1);
                break;
            }
            if (latency_ms)
                latency_ms[b] = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
            vote_stats &a = wsum[wi];
            const vote_stats &e = w->stats;
            a.levels = e.levels > a.levels ? e.levels : a.levels;
            a.cells += e.cells;
            a.records += e.records;
            a.tests += e.tests;
            wevaluated[wi] += w->evaluated;
            a.rechecks += e.rechecks;
            a.chunks += e.chunks;
            a.leaves += e.leaves;
            a.peak_records = e.peak_records > a.peak_records ? e.peak_records : a.peak_records;
            a.launches += e.launches;
        }
    };
    for (int k = nw;;) {
        std::vector<std::thread> th;
        for (int i = 1; i < k; ++i) th.emplace_back(work, i);
        work(0);
        for (auto &t : th) t.join();
        const int done = std::min(next.load(), (int)todo.size());
        again.insert(again.end(), todo.begin() + done, todo.end());
        if (again.empty() || failed.load()) break;
        // memory was short: what is left by half as many workers, at last by one, with what
        // this context's solves hold given back
        k = k / 2 > 1 ? k / 2 : 1;
        alone = k == 1;
        todo.swap(again);
        again.clear();
        next.store(0);
        release_working(c);
    }
    std::memset(&c->stats, 0, sizeof(c->stats));
    for (int i = 0; i < nw; ++i) {
        if (wst[i] != VOTE_OK) {
            set_err("%s", wmsg[i].c_str());
            return wst[i];
        }
    }
    for (int i = 0; i < nw; ++i) {                  // statistics of the whole batch
        const vote_stats &a = wsum[i];
        c->stats.levels = a.levels > c->stats.levels ? a.levels : c->stats.levels;
        c->stats.cells += a.cells;
        c->stats.records += a.records;
        c->stats.tests += a.tests;
        if (c->count_work) c->evaluated += wevaluated[i];
        c->stats.rechecks += a.rechecks;
        c->stats.chunks += a.chunks;
        c->stats.leaves += a.leaves;
        c->stats.peak_records = a.peak_records > c->stats.peak_records ? a.peak_records : c->stats.peak_records;
        c->stats.launches += a.launches;
    }
    c->stats.seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    return VOTE_OK;
}

vote_status vote_cell_counts(vote_ctx *c, const double *surfaces, int64_t n, int level, const int64_t *coords,
                             int64_t *ub, int64_t *lb, uint32_t *reach) {
    if (!c || !coords || !ub || !lb || n < 0 || (n > 0 && !surfaces)) { set_err("invalid arguments"); return VOTE_EINVAL; }
    const Problem &P = c->P;
    if (level < 0 || level > P.L) { set_err("level %d outside [0, %d]", level, P.L); return VOTE_EINVAL; }
    uint64_t key = 0;
    for (int j = 0; j < P.d; ++j) {
        int e = level < P.Lj[j] ? level : P.Lj[j];
        if (coords[j] < 0 || coords[j] >= ((int64_t)1 << e)) { set_err("coordinate %d out of range", j); return VOTE_EINVAL; }
        key |= (uint64_t)coords[j] << (P.coord_shift[j] + P.Lj[j] - e);
    }
    if (n == 0) { *ub = 0; *lb = 0; return VOTE_OK; }
    TRY(replay(c, surfaces, n, level, key, reach, ub, lb));
    return VOTE_OK;
}

static vote_status ss_prepare(vote_ctx *c, const double *tol, double *inv_tol2) {
    const Problem &P = c->P;
    if (!softscore_supported(P.fam)) {
        set_err("the soft score is not available for family %d", P.fam);
        return VOTE_EUNSUPPORTED;
    }
    for (int j = 0; j < P.nd; ++j) {
        double t = tol ? tol[j] : P.eps[P.k + j];
        if (!(t > 0.0) || !std::isfinite(t)) { set_err("tol must be finite and > 0"); return VOTE_EINVAL; }
        inv_tol2[j] = 1.0 / (t * t);
    }
    TRY(ensure(c, c->ss_partial, sizeof(double) * softscore_partial_doubles()));
    TRY(ensure(c, c->ss_io, sizeof(double) * (2 * GV_MAXD + 2)));
    return VOTE_OK;
}

vote_status vote_softscore_fwd(vote_ctx *c, const double *surfaces, int64_t n, const uint32_t *mask,
                               const double *point, const double *tol, double *score) {
    if (!c || n < 0 || (n > 0 && !surfaces) || !point || !score) { set_err("invalid arguments"); return VOTE_EINVAL; }
    double inv_tol2[GV_MAXD];
    TRY(ss_prepare(c, tol, inv_tol2));
    if (n == 0) { CK(cudaMemsetAsync(score, 0, sizeof(double), c->stream)); return VOTE_OK; }
    launch_softscore(c->P.fam, false, surfaces, n, mask, point, inv_tol2, c->P.nd, nullptr, nullptr,
                     (double *)c->ss_partial.p, score, c->stream);
    CK(cudaGetLastError());
    return VOTE_OK;
}

vote_status vote_softscore_bwd(vote_ctx *c, const double *surfaces, int64_t n, const uint32_t *mask,
                               const double *point, const double *tol, const double *grad_score,
                               double *grad_point, double *grad_surfaces) {
    if (!c || n < 0 || (n > 0 && !surfaces) || !point || !grad_score) { set_err("invalid arguments"); return VOTE_EINVAL; }
    double inv_tol2[GV_MAXD];
    TRY(ss_prepare(c, tol, inv_tol2));
    double *gp = grad_point ? grad_point : (double *)c->ss_io.p + GV_MAXD;
    if (n == 0) { CK(cudaMemsetAsync(gp, 0, sizeof(double) * c->P.d, c->stream)); return VOTE_OK; }
    launch_softscore(c->P.fam, true, surfaces, n, mask, point, inv_tol2, c->P.nd, grad_score, grad_surfaces,
                     (double *)c->ss_partial.p, gp, c->stream);
    CK(cudaGetLastError());
    return VOTE_OK;
}

vote_status vote_refine(vote_ctx *c, const double *surfaces, int64_t n, const uint32_t *mask, const double *cell_lo,
                        const double *cell_hi, const double *tol, int iters, double *point_inout,
                        double *score_out) {
    if (!c || n < 0 || (n > 0 && !surfaces) || !cell_lo || !cell_hi || !point_inout || iters < 0) {
        set_err("invalid arguments");
        return VOTE_EINVAL;
    }
    const int d = c->P.d;
    for (int j = 0; j < d; ++j)
        if (!(cell_hi[j] >= cell_lo[j])) { set_err("empty cell in coordinate %d", j); return VOTE_EINVAL; }
    double inv_tol2[GV_MAXD];
    TRY(ss_prepare(c, tol, inv_tol2));
    double *dio = (double *)c->ss_io.p;       // [0, d): point, [d, 2d): outputs, [2 MAXD]: 1.0
    double host[2 * GV_MAXD + 2];
    auto eval = [&](const double *pt, bool grad, double *res) -> vote_status {
        std::memcpy(host, pt, sizeof(double) * d);
        host[2 * GV_MAXD] = 1.0;
        CK(cudaMemcpyAsync(dio, host, sizeof(double) * d, cudaMemcpyHostToDevice, c->stream));
        CK(cudaMemcpyAsync(dio + 2 * GV_MAXD, host + 2 * GV_MAXD, sizeof(double), cudaMemcpyHostToDevice, c->stream));
        launch_softscore(c->P.fam, grad, surfaces, n, mask, dio, inv_tol2, c->P.nd, dio + 2 * GV_MAXD, nullptr,
                         (double *)c->ss_partial.p, dio + GV_MAXD, c->stream);
        CK(cudaGetLastError());
        CK(cudaMemcpyAsync(res, dio + GV_MAXD, sizeof(double) * (grad ? d : 1), cudaMemcpyDeviceToHost, c->stream));
        CK(cudaStreamSynchronize(c->stream));
        return VOTE_OK;
    };
    double p[GV_MAXD], q[GV_MAXD], g[GV_MAXD], D[GV_MAXD], S = 0.0, Sq = 0.0;
    for (int j = 0; j < d; ++j) {
        p[j] = std::fmin(std::fmax(point_inout[j], cell_lo[j]), cell_hi[j]);
        D[j] = (cell_hi[j] - cell_lo[j]) * (cell_hi[j] - cell_lo[j]);
    }
    if (n > 0) {
        TRY(eval(p, false, &S));
        for (int it = 0; it < iters; ++it) {
            TRY(eval(p, true, g));
            double gdg = 0.0;
            for (int j = 0; j < d; ++j) gdg += g[j] * g[j] * D[j];
            if (!(gdg > 0.0)) break;
            bool moved = false;
            for (double t = 1.0 / std::sqrt(gdg); t > 1e-14; t *= 0.5) {
                for (int j = 0; j < d; ++j) q[j] = std::fmin(std::fmax(p[j] + t * D[j] * g[j], cell_lo[j]), cell_hi[j]);
                TRY(eval(q, false, &Sq));
                if (Sq >= S + 1e-4 * t * gdg) {
                    std::memcpy(p, q, sizeof(double) * d);
                    S = Sq;
                    moved = true;
                    break;
                }
            }
            if (!moved) break;
        }
    }
    std::memcpy(point_inout, p, sizeof(double) * d);
    if (score_out) *score_out = S;
    return VOTE_OK;
}

vote_status vote_leaf_box(vote_ctx *c, const int64_t *leaf, double *lo, double *hi) {
    if (!c || !leaf || !lo || !hi) { set_err("invalid arguments"); return VOTE_EINVAL; }
    const Problem &P = c->P;
    for (int j = 0; j < P.d; ++j) {
        if (leaf[j] < 0 || leaf[j] >= ((int64_t)1 << P.Lj[j])) { set_err("leaf coordinate %d out of range", j); return VOTE_EINVAL; }
        double w = 2.0 * c->h_leaf[j];
        lo[j] = P.lo[j] + (double)leaf[j] * w;
        hi[j] = lo[j] + w;
    }
    return VOTE_OK;
}

vote_status vote_levels(vote_ctx *c, int *L, int *Lj) {
    if (!c || !L) { set_err("invalid arguments"); return VOTE_EINVAL; }
    *L = c->P.L;
    if (Lj) for (int j = 0; j < c->P.d; ++j) Lj[j] = c->P.Lj[j];
    return VOTE_OK;
}

vote_status vote_level_constants(int family, int d, int k, const double *eps, const double *bounds, int *L,
                                 int *Lj, double *s_f, double *s_t, double *A) {
    if (!eps || !bounds || !L) { set_err("invalid arguments"); return VOTE_EINVAL; }
    vote_ctx tmp;                        // host-side constants only (no device memory)
    TRY(problem_init(&tmp, family, d, k, eps, bounds));
    const Problem &P = tmp.P;
    *L = P.L;
    if (Lj) for (int j = 0; j < P.d; ++j) Lj[j] = P.Lj[j];
    if (s_f) for (int j = 0; j < P.nd; ++j) s_f[j] = P.s_f[j];
    for (int l = 0; l < P.L; ++l) {
        if (s_t) for (int m = 0; m < P.le; ++m) s_t[(size_t)l * P.le + m] = tmp.lev[l].s_t[m];
        if (A) for (int j = 0; j < P.nd; ++j) A[(size_t)l * P.nd + j] = tmp.lev[l].A1[j];
    }
    return VOTE_OK;
}

vote_status vote_get_trace(vote_ctx *c, int64_t cap, int32_t *level, int64_t *coords, int64_t *ub, int64_t *lb,
                           int64_t *count) {
    if (!c || !count || cap < 0) { set_err("invalid arguments"); return VOTE_EINVAL; }
    int64_t m = c->trace_written < c->trace_cap ? c->trace_written : c->trace_cap;
    if (m > cap) m = cap;
    *count = m;
    if (m > 0) {
        int32_t *lv = new int32_t[m];
        uint64_t *ky = new uint64_t[m];
        uint32_t *u = new uint32_t[m], *b = new uint32_t[m];
        cudaError_t e = cudaMemcpy(lv, c->tr_level.p, m * 4, cudaMemcpyDeviceToHost);
        if (e == cudaSuccess) e = cudaMemcpy(ky, c->tr_key.p, m * 8, cudaMemcpyDeviceToHost);
        if (e == cudaSuccess) e = cudaMemcpy(u, c->tr_ub.p, m * 4, cudaMemcpyDeviceToHost);
        if (e == cudaSuccess) e = cudaMemcpy(b, c->tr_lb.p, m * 4, cudaMemcpyDeviceToHost);
        if (e == cudaSuccess) {
            const Problem &P = c->P;
            for (int64_t i = 0; i < m; ++i) {
                if (level) level[i] = lv[i];
                if (ub) ub[i] = u[i];
                if (lb) lb[i] = b[i];
                if (coords)
                    for (int j = 0; j < P.d; ++j) {
                        int ex = lv[i] < P.Lj[j] ? lv[i] : P.Lj[j];
                        coords[i * P.d + j] = (int64_t)((ky[i] >> (P.coord_shift[j] + P.Lj[j] - ex)) & ((1ull << ex) - 1ull));
                    }
            }
        }
        delete[] lv; delete[] ky; delete[] u; delete[] b;
        if (e != cudaSuccess) { set_err("trace copy failed: %s", cudaGetErrorString(e)); return VOTE_ECUDA; }
    }
    if (c->trace_overflow) { set_err("trace overflowed (%lld entries)", (long long)c->trace_written); return VOTE_ECAPACITY; }
    return VOTE_OK;
}

vote_status vote_get_kernel_times(vote_ctx *c, double *ms, int64_t *launches, double *bytes) {
    if (!c) { set_err("null context"); return VOTE_EINVAL; }
    for (int i = 0; i < VOTE_K_CLASSES; ++i) {
        if (ms) ms[i] = c->kms[i];
        if (launches) launches[i] = c->klaunch[i];
        if (bytes) bytes[i] = c->kbytes[i];
    }
    return VOTE_OK;
}

vote_status vote_get_level_stats(vote_ctx *c, int64_t *cells, int64_t *records, int64_t *grouped_in,
                                 int64_t *grouped_out) {
    if (!c) { set_err("null context"); return VOTE_EINVAL; }
    for (int l = 0; l < c->P.L; ++l) {
        if (cells) cells[l] = c->lv_cells[l];
        if (records) records[l] = c->lv_recs[l];
        if (grouped_in) grouped_in[l] = c->lv_gin[l];
        if (grouped_out) grouped_out[l] = c->lv_gout[l];
    }
    return VOTE_OK;
}

vote_status vote_get_stats(vote_ctx *c, vote_stats *out) {
    if (!c || !out) { set_err("invalid arguments"); return VOTE_EINVAL; }
    *out = c->stats;
    return VOTE_OK;
}

vote_status vote_get_evaluated(vote_ctx *c, int64_t *tests) {
    if (!c || !tests) { set_err("invalid arguments"); return VOTE_EINVAL; }
    *tests = c->evaluated;
    return VOTE_OK;
}

void vote_destroy(vote_ctx *c) {
    if (!c) return;
    for (vote_ctx *w : c->workers) {
        cudaStream_t ws = w->stream;
        vote_destroy(w);
        if (ws) cudaStreamDestroy(ws);
    }
    c->workers.clear();
    release_working(c);
    DevBuf *bufs[] = {&c->levs_dev, &c->path, &c->scal, &c->tr_level, &c->tr_key, &c->tr_ub, &c->tr_lb, &c->surf_tmp,
                      &c->mask_tmp, &c->ss_partial, &c->ss_io, &c->beam_sel, &c->linfo};
    for (DevBuf *b : bufs) release(c, *b);
    for (DevBuf &b : c->sctab) release(c, b);
    release(c, c->psi0);
    cudaStreamSynchronize(c->stream);
    for (int i = 0; i < vote_ctx::kEv; ++i)
        if (c->ev[i]) cudaEventDestroy(c->ev[i]);
    if (c->h_sc) cudaFreeHost(c->h_sc);
    if (c->h_tmp) cudaFreeHost(c->h_tmp);
    if (c->h_info) cudaFreeHost(c->h_info);
    delete c;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Entry point without allocation (vote_cell_counts_noalloc).  Its scratch is this
// file-scope device array; host code must not use the symbol as an address (in
// host code it names a host-side stand-in), so the device address is looked up
// once per device with cudaGetSymbolAddress and passed to the kernels.
// ---------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_noalloc_scratch[VOTE_NOALLOC_SCRATCH_BYTES];

namespace {
constexpr size_t kNaLevels = 0;
constexpr size_t kNaPath = kNaLevels + sizeof(Level) * GV_MAXL;
constexpr size_t kNaScalars = (kNaPath + sizeof(PathStep) * (GV_MAXL + kPathTail) + 255) / 256 * 256;
constexpr size_t kNaEnd = kNaScalars + sizeof(Scalars);
static_assert(kNaEnd <= VOTE_NOALLOC_SCRATCH_BYTES, "no-alloc scratch too small");

constexpr int kNaMaxDevices = 64;
std::mutex g_na_mutex;
unsigned char *g_na_ptr[kNaMaxDevices] = {};
}  // namespace

static vote_status noalloc_scratch(unsigned char **out) {
    int dev = 0;
    CK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kNaMaxDevices) {
        set_err("device %d out of range", dev);
        return VOTE_EUNSUPPORTED;
    }
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (!g_na_ptr[dev]) {
        void *p = nullptr;
        CK(cudaGetSymbolAddress(&p, g_noalloc_scratch));   // once per device, this device current
        g_na_ptr[dev] = (unsigned char *)p;
    }
    *out = g_na_ptr[dev];
    return VOTE_OK;
}

extern "C" vote_status vote_cell_counts_noalloc(int family, int d, int k, const double *eps, const double *bounds,
                                                const double *surfaces, int64_t n, int level,
                                                const int64_t *coords, int64_t *ub, int64_t *lb, uint32_t *reach,
                                                void *cuda_stream) {
    if (!eps || !bounds || !coords || !ub || !lb || n < 0 || (n > 0 && !surfaces)) {
        set_err("invalid arguments");
        return VOTE_EINVAL;
    }
    vote_ctx tmp;                        // host-side constants only (no device memory)
    TRY(problem_init(&tmp, family, d, k, eps, bounds));
    const Problem &P = tmp.P;
    if (P.L > GV_MAXL - 1) {
        set_err("%d levels exceed the no-alloc scratch (%d)", P.L, GV_MAXL - 1);
        return VOTE_EUNSUPPORTED;
    }
    if (level < 0 || level > P.L) { set_err("level %d outside [0, %d]", level, P.L); return VOTE_EINVAL; }
    uint64_t key = 0;
    for (int j = 0; j < P.d; ++j) {
        int e = level < P.Lj[j] ? level : P.Lj[j];
        if (coords[j] < 0 || coords[j] >= ((int64_t)1 << e)) { set_err("coordinate %d out of range", j); return VOTE_EINVAL; }
        key |= (uint64_t)coords[j] << (P.coord_shift[j] + P.Lj[j] - e);
    }
    if (n == 0) { *ub = 0; *lb = 0; return VOTE_OK; }
    unsigned char *base = nullptr;
    TRY(noalloc_scratch(&base));
    cudaStream_t st = (cudaStream_t)cuda_stream;
    Level *levs = (Level *)(base + kNaLevels);
    PathStep *path = (PathStep *)(base + kNaPath);
    Scalars *sc = (Scalars *)(base + kNaScalars);
    if (P.L > 0) CK(cudaMemcpyAsync(levs, tmp.lev, sizeof(Level) * P.L, cudaMemcpyHostToDevice, st));
    CK(cudaMemsetAsync(sc, 0, sizeof(Scalars), st));        // the counters must start at zero
    if (level > 0) launch_path_geo(P, levs, level, key, nullptr, path, st);
    launch_replay(P, levs, path, level, surfaces, n, reach, sc, st);
    CK(cudaGetLastError());
    unsigned long long cnt[2] = {0, 0};
    CK(cudaMemcpyAsync(cnt, &sc->replay_ub, sizeof(cnt), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    *ub = (int64_t)cnt[0];
    *lb = (int64_t)cnt[1];
    return VOTE_OK;
}
