// gv_softscore.cu -- soft inlier score S(p) = sum_i w_i exp(-u_i^2 / 2),
// u_i^2 = sum_j (r_ij / tol_j)^2, r_ij the vertical residual of surface i at p in
// dependent coordinate j (Eq. 1 in global form), w_i = bit i of the inlier mask.
// Forward, backward (d S / d p and d S / d surface parameters, recomputing the
// residuals instead of storing them) and a projected gradient ascent that keeps p
// inside a cell.  This refines the voting result the way Sec. 4.2 suggests a
// "more accurate method" take over from the approximate pose.
//
// Reductions are deterministic: per-block partial sums in a fixed grid, every warp
// taking its surfaces in order, then one block adds the partials in a fixed tree.
//
// The FP64 pipe issues one lane per clock and SM, so a full evaluation (residuals,
// exp, derivatives: 60 to 200 FP64 instructions) of every surface bounds the pass.
// But exp(-u^2 / 2) is exactly 0 in FP64 from u = 38.61 on, and so are the surface's
// contributions.  Each warp first evaluates 32 residuals in FP32 with a bound on their
// error; surfaces certainly beyond that (or certainly masked out) contribute zeros, the
// others are queued and evaluated in FP64 by full warps.  What depends on the point
// alone is evaluated once per block.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

#include "gv_kernels.h"

namespace gv {

constexpr int kSsBlocks = 608;        // 4 per SM
constexpr int kSsThreads = 256;
// u beyond which exp(-u^2 / 2) underflows to 0 (sqrt(2 * 745.14) = 38.604), with a margin
constexpr float kSsFar = 38.7f;
// FP32 residuals: inputs truncated to FP32 (2^-23), at most three of them in a product,
// ten operations, constants rounded once: an error of at most 24 u m, u = 2^-24; taken as
constexpr float kSsErr = 64.0f * 5.9604645e-08f;

// Per family: what depends on the point alone (Pre: FP64, and FP32 copies), residuals
// r[j], d r / d p (dp[j][d]) and d r / d params (dq[j][P]) of a surface with parameters q,
// and its FP32 residuals with magnitudes m[j] their error scales with.
template <int FAM> struct SoftFam;

template <> struct SoftFam<FAM_LINE2D> {       // r = b - (y - x m)
    static constexpr int D = 2, ND = 1, NP = 2;
    struct Pre { float p[2]; };
    __device__ static void prep(const double *p, Pre &c) { c.p[0] = (float)p[0]; c.p[1] = (float)p[1]; }
    __device__ static void eval(const double *q, const double *p, const Pre &, double *r, double *dp, double *dq) {
        double x = q[0], y = q[1];
        r[0] = p[1] - (y - x * p[0]);
        dp[0] = x; dp[1] = 1.0;
        dq[0] = p[0]; dq[1] = -1.0;
    }
    __device__ static void resid32(const float *q, const Pre &c, float *r, float *m) {
        r[0] = c.p[1] - (q[1] - q[0] * c.p[0]);
        m[0] = fabsf(c.p[1]) + fabsf(q[1]) + fabsf(q[0] * c.p[0]);
    }
};

template <> struct SoftFam<FAM_PLANE3D_SPH> {  // r = d - q . n(theta, phi)
    static constexpr int D = 3, ND = 1, NP = 3;
    struct Pre { double st, ct, sp, cp; float n[3], d; };
    __device__ static void prep(const double *p, Pre &c) {
        sincos(p[0], &c.st, &c.ct);
        sincos(p[1], &c.sp, &c.cp);
        c.n[0] = (float)(c.st * c.cp); c.n[1] = (float)(c.st * c.sp); c.n[2] = (float)c.ct;
        c.d = (float)p[2];
    }
    __device__ static void eval(const double *q, const double *p, const Pre &c, double *r, double *dp, double *dq) {
        double qx = q[0], qy = q[1], qz = q[2];
        double nx = c.st * c.cp, ny = c.st * c.sp, nz = c.ct;
        r[0] = p[2] - (qx * nx + qy * ny + qz * nz);
        dp[0] = -(qx * c.ct * c.cp + qy * c.ct * c.sp - qz * c.st);
        dp[1] = -(-qx * c.st * c.sp + qy * c.st * c.cp);
        dp[2] = 1.0;
        dq[0] = -nx; dq[1] = -ny; dq[2] = -nz;
    }
    __device__ static void resid32(const float *q, const Pre &c, float *r, float *m) {
        r[0] = c.d - (q[0] * c.n[0] + q[1] * c.n[1] + q[2] * c.n[2]);
        m[0] = fabsf(c.d) + fabsf(q[0]) + fabsf(q[1]) + fabsf(q[2]);
    }
};

template <> struct SoftFam<FAM_POSE3DOF> {     // r_x = x - (w1 - (a c - b s)), r_y = y - (w2 - (a s + b c))
    static constexpr int D = 3, ND = 2, NP = 4;
    struct Pre { double s, c; float sf, cf, x, y; };
    __device__ static void prep(const double *p, Pre &e) {
        sincos(p[0], &e.s, &e.c);
        e.sf = (float)e.s; e.cf = (float)e.c; e.x = (float)p[1]; e.y = (float)p[2];
    }
    __device__ static void eval(const double *q, const double *p, const Pre &e, double *r, double *dp, double *dq) {
        double w1 = q[0], w2 = q[1], a = q[2], b = q[3], s = e.s, c = e.c;
        r[0] = p[1] - (w1 - (a * c - b * s));
        r[1] = p[2] - (w2 - (a * s + b * c));
        dp[0] = -a * s - b * c; dp[1] = 1.0; dp[2] = 0.0;
        dp[3] = a * c - b * s;  dp[4] = 0.0; dp[5] = 1.0;
        dq[0] = -1.0; dq[1] = 0.0; dq[2] = c; dq[3] = -s;
        dq[4] = 0.0; dq[5] = -1.0; dq[6] = s; dq[7] = c;
    }
    __device__ static void resid32(const float *q, const Pre &e, float *r, float *m) {
        const float ab = fabsf(q[2]) + fabsf(q[3]);
        r[0] = e.x - (q[0] - (q[2] * e.cf - q[3] * e.sf));
        r[1] = e.y - (q[1] - (q[2] * e.sf + q[3] * e.cf));
        m[0] = fabsf(e.x) + fabsf(q[0]) + ab;
        m[1] = fabsf(e.y) + fabsf(q[1]) + ab;
    }
};

// r_x = x - (xi (r3 . w + z) - r1 . w), r_y = y - (eta (r3 . w + z) - r2 . w) with
// R = R(phi) (Rodrigues); d(R w)/d phi_a = (J e_a) x (R w), J = I + B [phi]x +
// C [phi]x^2 the rotation's left Jacobian, B = (1 - cos th)/th^2, C = (th - sin th)/th^3.
template <> struct SoftFam<FAM_POSE6DOF> {
    static constexpr int D = 6, ND = 2, NP = 5;
    struct Pre { double Rm[9], u[9]; float R[9], t[3]; };   // u[3 a + .]: J e_a
    __device__ static void prep(const double *p, Pre &e) {
        const double f0 = p[0], f1 = p[1], f2 = p[2];
        const double th2 = f0 * f0 + f1 * f1 + f2 * f2;
        double A, B, C;
        if (th2 < 1e-8) {            // series: the closed forms lose accuracy near 0
            A = 1.0 - th2 / 6.0 + th2 * th2 / 120.0;
            B = 0.5 - th2 / 24.0 + th2 * th2 / 720.0;
            C = 1.0 / 6.0 - th2 / 120.0 + th2 * th2 / 5040.0;
        } else {
            const double th = sqrt(th2);
            double sn, cs;
            sincos(th, &sn, &cs);
            A = sn / th;
            B = (1.0 - cs) / th2;
            C = (th - sn) / (th2 * th);
        }
        // R = I + A K + B K^2, K = [phi]x, K^2 = phi phi^T - th2 I
        const double ph[3] = {f0, f1, f2};
        double *Rm = e.Rm;
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b) Rm[3 * a + b] = B * ph[a] * ph[b] + (a == b ? 1.0 - B * th2 : 0.0);
        Rm[1] -= A * f2; Rm[2] += A * f1;
        Rm[3] += A * f2; Rm[5] -= A * f0;
        Rm[6] -= A * f1; Rm[7] += A * f0;
        for (int a = 0; a < 3; ++a) {
            // u = J e_a = e_a + B (phi x e_a) + C (phi x (phi x e_a))
            double x[3] = {0.0, 0.0, 0.0};
            x[a] = 1.0;
            const double c1[3] = {ph[1] * x[2] - ph[2] * x[1], ph[2] * x[0] - ph[0] * x[2], ph[0] * x[1] - ph[1] * x[0]};
            const double c2[3] = {ph[1] * c1[2] - ph[2] * c1[1], ph[2] * c1[0] - ph[0] * c1[2],
                                  ph[0] * c1[1] - ph[1] * c1[0]};
            for (int b = 0; b < 3; ++b) e.u[3 * a + b] = x[b] + B * c1[b] + C * c2[b];
        }
        for (int i = 0; i < 9; ++i) e.R[i] = (float)Rm[i];
        for (int i = 0; i < 3; ++i) e.t[i] = (float)p[3 + i];
    }
    __device__ static void eval(const double *q, const double *p, const Pre &e, double *r, double *dp, double *dq) {
        const double w[3] = {q[0], q[1], q[2]};
        const double xi = q[3], eta = q[4];
        const double *Rm = e.Rm;
        double X[3];
        for (int a = 0; a < 3; ++a) X[a] = Rm[3 * a] * w[0] + Rm[3 * a + 1] * w[1] + Rm[3 * a + 2] * w[2];
        const double Dz = X[2] + p[3];
        r[0] = p[4] - (xi * Dz - X[0]);
        r[1] = p[5] - (eta * Dz - X[1]);
        for (int a = 0; a < 3; ++a) {
            const double *u = e.u + 3 * a;
            const double dX[3] = {u[1] * X[2] - u[2] * X[1], u[2] * X[0] - u[0] * X[2], u[0] * X[1] - u[1] * X[0]};
            dp[a] = -(xi * dX[2] - dX[0]);
            dp[D + a] = -(eta * dX[2] - dX[1]);
        }
        dp[3] = -xi; dp[4] = 1.0; dp[5] = 0.0;
        dp[D + 3] = -eta; dp[D + 4] = 0.0; dp[D + 5] = 1.0;
        for (int b = 0; b < 3; ++b) {
            dq[b] = -(xi * Rm[6 + b] - Rm[b]);
            dq[NP + b] = -(eta * Rm[6 + b] - Rm[3 + b]);
        }
        dq[3] = -Dz; dq[4] = 0.0;
        dq[NP + 3] = 0.0; dq[NP + 4] = -Dz;
    }
    __device__ static void resid32(const float *q, const Pre &e, float *r, float *m) {
        const float *R = e.R;
        const float x0 = R[0] * q[0] + R[1] * q[1] + R[2] * q[2], x1 = R[3] * q[0] + R[4] * q[1] + R[5] * q[2];
        const float dz = R[6] * q[0] + R[7] * q[1] + R[8] * q[2] + e.t[0];
        const float aw = fabsf(q[0]) + fabsf(q[1]) + fabsf(q[2]), az = aw + fabsf(e.t[0]);
        r[0] = e.t[1] - (q[3] * dz - x0);
        r[1] = e.t[2] - (q[4] * dz - x1);
        m[0] = fabsf(e.t[1]) + fabsf(q[3]) * az + aw;
        m[1] = fabsf(e.t[2]) + fabsf(q[4]) * az + aw;
    }
};

template <> struct SoftFam<FAM_RAYS3D> {       // r_y = y - (a x + b), r_z = z - (c x + d)
    static constexpr int D = 3, ND = 2, NP = 4;
    struct Pre { float p[3]; };
    __device__ static void prep(const double *p, Pre &c) {
        for (int i = 0; i < 3; ++i) c.p[i] = (float)p[i];
    }
    __device__ static void eval(const double *q, const double *p, const Pre &, double *r, double *dp, double *dq) {
        const double a = q[0], b = q[1], c = q[2], d = q[3];
        r[0] = p[1] - (a * p[0] + b);
        r[1] = p[2] - (c * p[0] + d);
        dp[0] = -a; dp[1] = 1.0; dp[2] = 0.0;
        dp[3] = -c; dp[4] = 0.0; dp[5] = 1.0;
        dq[0] = -p[0]; dq[1] = -1.0; dq[2] = 0.0; dq[3] = 0.0;
        dq[4] = 0.0; dq[5] = 0.0; dq[6] = -p[0]; dq[7] = -1.0;
    }
    __device__ static void resid32(const float *q, const Pre &c, float *r, float *m) {
        r[0] = c.p[1] - (q[0] * c.p[0] + q[1]);
        r[1] = c.p[2] - (q[2] * c.p[0] + q[3]);
        m[0] = fabsf(c.p[1]) + fabsf(q[0] * c.p[0]) + fabsf(q[1]);
        m[1] = fabsf(c.p[2]) + fabsf(q[2] * c.p[0]) + fabsf(q[3]);
    }
};

// r = b - (x4 - a . x)
template <> struct SoftFam<FAM_AFFINE4D> {
    static constexpr int D = 4, ND = 1, NP = 4;
    struct Pre { float p[4]; };
    __device__ static void prep(const double *p, Pre &c) {
        for (int i = 0; i < 4; ++i) c.p[i] = (float)p[i];
    }
    __device__ static void eval(const double *q, const double *p, const Pre &, double *r, double *dp, double *dq) {
        const double x1 = q[0], x2 = q[1], x3 = q[2], x4 = q[3];
        r[0] = p[3] - (x4 - ((p[0] * x1 + p[1] * x2) + p[2] * x3));
        dp[0] = x1; dp[1] = x2; dp[2] = x3; dp[3] = 1.0;
        dq[0] = p[0]; dq[1] = p[1]; dq[2] = p[2]; dq[3] = -1.0;
    }
    __device__ static void resid32(const float *q, const Pre &c, float *r, float *m) {
        const float a = c.p[0] * q[0], b = c.p[1] * q[1], d = c.p[2] * q[2];
        r[0] = c.p[3] - (q[3] - ((a + b) + d));
        m[0] = fabsf(c.p[3]) + fabsf(q[3]) + fabsf(a) + fabsf(b) + fabsf(d);
    }
};

// r_a = a - (p_x (q_x - c) + p_y (q_y - d)) / |p|^2, r_b = b - (p_y (q_x - c) - p_x (q_y - d)) / |p|^2
template <> struct SoftFam<FAM_POINTSET2D> {
    static constexpr int D = 4, ND = 2, NP = 4;
    struct Pre { float p[4]; };
    __device__ static void prep(const double *p, Pre &c) {
        for (int i = 0; i < 4; ++i) c.p[i] = (float)p[i];
    }
    __device__ static void eval(const double *q, const double *p, const Pre &, double *r, double *dp, double *dq) {
        const double px = q[0], py = q[1], qx = q[2], qy = q[3];
        const double N = px * px + py * py, ex = qx - p[0], ey = qy - p[1];
        const double A = px * ex + py * ey, B = py * ex - px * ey;
        r[0] = p[2] - A / N;
        r[1] = p[3] - B / N;
        dp[0] = px / N; dp[1] = py / N; dp[2] = 1.0; dp[3] = 0.0;
        dp[4] = py / N; dp[5] = -px / N; dp[6] = 0.0; dp[7] = 1.0;
        const double N2 = N * N;
        dq[0] = -(ex / N - A * 2.0 * px / N2);
        dq[1] = -(ey / N - A * 2.0 * py / N2);
        dq[2] = -(px / N);
        dq[3] = -(py / N);
        dq[4] = -(-ey / N - B * 2.0 * px / N2);
        dq[5] = -(ex / N - B * 2.0 * py / N2);
        dq[6] = -(py / N);
        dq[7] = -(-px / N);
    }
    __device__ static void resid32(const float *q, const Pre &c, float *r, float *m) {
        const float in = 1.0f / (q[0] * q[0] + q[1] * q[1]), ex = q[2] - c.p[0], ey = q[3] - c.p[1];
        const float ax = fabsf(q[2]) + fabsf(c.p[0]), ay = fabsf(q[3]) + fabsf(c.p[1]);
        const float px = fabsf(q[0]), py = fabsf(q[1]);
        r[0] = c.p[2] - (q[0] * ex + q[1] * ey) * in;
        r[1] = c.p[3] - (q[1] * ex - q[0] * ey) * in;
        m[0] = fabsf(c.p[2]) + (px * ax + py * ay) * in;
        m[1] = fabsf(c.p[3]) + (py * ax + px * ay) * in;
    }
};

struct SoftArgs {
    const double *prm;
    int64_t n;
    const uint32_t *mask;     // NULL: every weight 1
    const double *p;          // device [d]
    double inv_tol2[GV_MAXD]; // 1 / tol_j^2
    float far[GV_MAXD];       // |r_j| beyond which exp(-u^2 / 2) is 0
    const double *grad_out;   // device [1] (backward)
    double *grad_prm;         // device [P][n] or NULL (backward)
    double *partial;          // [kSsBlocks][1 + d]
};

__device__ __forceinline__ double block_sum(double v, double *sm) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sm[w] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < kSsThreads / 32; ++i) t += sm[i];
    return t;                 // valid in thread 0
}

// x truncated to FP32 (relative error below 2^-23) by moving its bits: an FP64 conversion
// would take the FP64 pipe.  ok is cleared when x is outside FP32's normal range and not 0.
__device__ __forceinline__ float trunc32(double x, bool &ok) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned e = (hi >> 20) & 0x7ffu;
    const unsigned b = (hi & 0x80000000u) | (((hi & 0x7fffffffu) - 0x38000000u) << 3) | (lo >> 29);
    const bool zero = !((hi & 0x7fffffffu) | lo);
    ok &= zero | (e - 897u <= 253u);
    return zero ? 0.0f : __uint_as_float(b);
}

template <int FAM, bool BWD>
__global__ void __launch_bounds__(kSsThreads, 4) k_softscore(SoftArgs a) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // k_softscore_final waits for this kernel
    using S = SoftFam<FAM>;
    __shared__ double sm[kSsThreads / 32];
    __shared__ typename S::Pre s_pre;
    __shared__ int64_t s_queue[kSsThreads / 32][64];
    double p[S::D];
#pragma unroll
    for (int j = 0; j < S::D; ++j) p[j] = a.p[j];
    if (threadIdx.x == 0) S::prep(p, s_pre);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    int64_t *queue = s_queue[threadIdx.x >> 5];
    const double g0 = BWD ? a.grad_out[0] : 0.0;
    // an infinite or NaN upstream gradient makes every contribution NaN: none is skipped
    const bool far_ok = !BWD || fabs(g0) <= 1.7976931348623157e308;
    float far[S::ND];
#pragma unroll
    for (int j = 0; j < S::ND; ++j) far[j] = a.far[j];
    double acc = 0.0, accp[S::D];
#pragma unroll
    for (int j = 0; j < S::D; ++j) accp[j] = 0.0;

    // the queue's first m surfaces, one per lane, in FP64
    auto take = [&](int m) {
        const int64_t i = lane < m ? queue[lane] : -1;
        if (i >= 0) {
            const double w = a.mask ? (double)((a.mask[i >> 5] >> (i & 31)) & 1u) : 1.0;
            double q[S::NP], r[S::ND], dp[S::ND * S::D], dq[S::ND * S::NP];
#pragma unroll
            for (int x = 0; x < S::NP; ++x) q[x] = a.prm[x * a.n + i];
            S::eval(q, p, s_pre, r, dp, dq);
            double u2 = 0.0;
#pragma unroll
            for (int j = 0; j < S::ND; ++j) u2 += r[j] * r[j] * a.inv_tol2[j];
            const double k = w * exp(-0.5 * u2);
            if (!BWD) {
                acc += k;
            } else {
                // dS_i / dr_j = -k r_j / tol_j^2
                double gq[S::NP];
#pragma unroll
                for (int x = 0; x < S::NP; ++x) gq[x] = 0.0;
#pragma unroll
                for (int j = 0; j < S::ND; ++j) {
                    const double dr = -g0 * k * r[j] * a.inv_tol2[j];
#pragma unroll
                    for (int x = 0; x < S::D; ++x) accp[x] += dr * dp[j * S::D + x];
#pragma unroll
                    for (int x = 0; x < S::NP; ++x) gq[x] += dr * dq[j * S::NP + x];
                }
                if (a.grad_prm)
#pragma unroll
                    for (int x = 0; x < S::NP; ++x) a.grad_prm[x * a.n + i] = gq[x];
            }
        }
    };

    const int64_t nwarp = (int64_t)gridDim.x * (kSsThreads / 32);
    const int64_t gw = (int64_t)blockIdx.x * (kSsThreads / 32) + (threadIdx.x >> 5), nb = (a.n + 31) / 32;
    int cnt = 0;                                     // queued surfaces (warp-uniform)
#pragma unroll 2
    for (int64_t g = gw; g < nb; g += nwarp) {
        const int64_t i = g * 32 + lane;
        const bool in = i < a.n;
        bool ok = in && far_ok, skip = false;
        float q[S::NP], r[S::ND], m[S::ND];
#pragma unroll
        for (int x = 0; x < S::NP; ++x) q[x] = trunc32(in ? a.prm[x * a.n + i] : 0.0, ok);
        S::resid32(q, s_pre, r, m);
        const bool off = a.mask && in && !((a.mask[g] >> lane) & 1u);
#pragma unroll
        for (int j = 0; j < S::ND; ++j) {
            skip |= fabsf(r[j]) - kSsErr * m[j] > far[j];
            ok &= m[j] < 1.0e30f;                    // finite (false for NaN): a zero weight then gives zeros
        }
        skip = ok && (skip || off);
        if constexpr (BWD) {
            if (skip && a.grad_prm)
#pragma unroll
                for (int x = 0; x < S::NP; ++x) a.grad_prm[x * a.n + i] = 0.0;
        }
        const unsigned want = __ballot_sync(0xffffffffu, in && !skip);
        if (in && !skip) queue[cnt + __popc(want & below)] = i;
        cnt += __popc(want);
        __syncwarp();
        if (cnt >= 32) {                             // uniform
            take(32);
            __syncwarp();
            const int64_t rest = lane < cnt - 32 ? queue[32 + lane] : 0;
            __syncwarp();
            if (lane < cnt - 32) queue[lane] = rest;
            cnt -= 32;
            __syncwarp();
        }
    }
    take(cnt);
    if (!BWD) {
        double t = block_sum(acc, sm);
        if (threadIdx.x == 0) a.partial[blockIdx.x] = t;
    } else {
#pragma unroll
        for (int q = 0; q < S::D; ++q) {
            double t = block_sum(accp[q], sm);
            if (threadIdx.x == 0) a.partial[blockIdx.x * S::D + q] = t;
        }
    }
}

// out[q] = sum over blocks of partial[b * width + q]: block q, a fixed tree (one thread
// adding 1024 partials one after the other took 30 us)
__global__ void __launch_bounds__(kSsThreads) k_softscore_final(const double *partial, int nb, int width, double *out) {
    grid_start();
    __shared__ double sm[kSsThreads / 32];
    double t = 0.0;
    for (int b = threadIdx.x; b < nb; b += kSsThreads) t += partial[b * width + blockIdx.x];
    t = block_sum(t, sm);
    if (threadIdx.x == 0) out[blockIdx.x] = t;
}

static int ss_blocks(int64_t n) {
    int64_t b = (n + kSsThreads - 1) / kSsThreads;
    return (int)(b < 1 ? 1 : (b > kSsBlocks ? kSsBlocks : b));
}

void launch_softscore(int fam, bool bwd, const double *prm, int64_t n, const uint32_t *mask, const double *p,
                      const double *inv_tol2, int nd, const double *grad_out, double *grad_prm, double *partial,
                      double *out, cudaStream_t st) {
    SoftArgs a;
    std::memset(&a, 0, sizeof(a));
    a.prm = prm; a.n = n; a.mask = mask; a.p = p; a.grad_out = grad_out; a.grad_prm = grad_prm;
    a.partial = partial;
    for (int j = 0; j < nd; ++j) {
        a.inv_tol2[j] = inv_tol2[j];
        const double far = kSsFar / std::sqrt(inv_tol2[j]);
        a.far[j] = far >= 1e-30 && far <= 1e30 ? (float)far : INFINITY;   // outside FP32's range: none is far
    }
    int nb = ss_blocks(n);
    int d = fam == FAM_LINE2D ? 2 : (fam == FAM_POSE6DOF ? 6 : ((fam == FAM_POINTSET2D || fam == FAM_AFFINE4D) ? 4 : 3));
    switch (fam) {
    case FAM_LINE2D:
        if (bwd) k_softscore<FAM_LINE2D, true><<<nb, kSsThreads, 0, st>>>(a);
        else k_softscore<FAM_LINE2D, false><<<nb, kSsThreads, 0, st>>>(a);
        break;
    case FAM_PLANE3D_SPH:
        if (bwd) k_softscore<FAM_PLANE3D_SPH, true><<<nb, kSsThreads, 0, st>>>(a);
        else k_softscore<FAM_PLANE3D_SPH, false><<<nb, kSsThreads, 0, st>>>(a);
        break;
    case FAM_POSE3DOF:
        if (bwd) k_softscore<FAM_POSE3DOF, true><<<nb, kSsThreads, 0, st>>>(a);
        else k_softscore<FAM_POSE3DOF, false><<<nb, kSsThreads, 0, st>>>(a);
        break;
    case FAM_AFFINE4D:
        if (bwd) k_softscore<FAM_AFFINE4D, true><<<nb, kSsThreads, 0, st>>>(a);
        else k_softscore<FAM_AFFINE4D, false><<<nb, kSsThreads, 0, st>>>(a);
        break;
    case FAM_POINTSET2D:
        if (bwd) k_softscore<FAM_POINTSET2D, true><<<nb, kSsThreads, 0, st>>>(a);
        else k_softscore<FAM_POINTSET2D, false><<<nb, kSsThreads, 0, st>>>(a);
        break;
    case FAM_RAYS3D:
        if (bwd) k_softscore<FAM_RAYS3D, true><<<nb, kSsThreads, 0, st>>>(a);
        else k_softscore<FAM_RAYS3D, false><<<nb, kSsThreads, 0, st>>>(a);
        break;
    case FAM_POSE6DOF:
        if (bwd) k_softscore<FAM_POSE6DOF, true><<<nb, kSsThreads, 0, st>>>(a);
        else k_softscore<FAM_POSE6DOF, false><<<nb, kSsThreads, 0, st>>>(a);
        break;
    }
    launch(k_softscore_final, bwd ? d : 1, kSsThreads, 0, st, partial, nb, bwd ? d : 1, out);
}

int softscore_partial_doubles() { return kSsBlocks * GV_MAXD; }

bool softscore_supported(int fam) {
    return fam == FAM_LINE2D || fam == FAM_PLANE3D_SPH || fam == FAM_POSE3DOF || fam == FAM_POSE6DOF ||
           fam == FAM_RAYS3D || fam == FAM_POINTSET2D || fam == FAM_AFFINE4D;
}

}  // namespace gv
