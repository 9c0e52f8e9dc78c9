// FP64 Lorenz-96 integrations of a few columns, the state split over many CTAs.
//
// What an outer iteration integrates is one state: the nonlinear trajectory, the gradient's
// adjoint, the product that scales the FP32 path, the quadratic cost.  GB300 issues one FP64
// warp instruction per 64 cycles and SM sub-partition, so a state held by one CTA (l96.cu) is
// bound by the FP64 issue of one SM of 152: 6.5 ms for the trajectory and 9 ms per product at
// n = 4096, T = 200.  Here a CTA holds B consecutive variables, one per thread, and advances
// them K whole RK4 steps by itself: a stage needs two variables on one side and one on the
// other, so a step needs 8 + 4, and the 12 K outermost threads recompute what the neighbouring
// CTAs own.  Nothing is exchanged inside a launch; the next launch reads the states that this
// one wrote.  The recomputation runs on SMs that would be idle (split_plan weighs the two).
// A state of at most 256 variables sits in one CTA that closes the ring and recomputes nothing.
// The stage coefficients of the next step are loaded before the current one is computed; stages
// exchange values through a double-buffered shared array, one barrier each.
//
// Bound: the serial chain of a stage.  One warp per sub-partition issues 5 FP64 instructions of
// 64 cycles, most of them dependent, behind a shared exchange and a barrier: 530 cycles per
// stage measured for the trajectory, 560 for the tangent linear.  n = 4096, T = 200 (128 CTAs of
// 128 threads, 8 steps a launch): trajectory 6540 -> 280 us, tangent linear 3900 -> 295 us, two
// adjoints in one pass 10100 -> 384 us; riot_outer_begin 24.57 -> 0.96 ms.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "internal.h"

namespace riot {

namespace {

// Place of one thread: its variable, the shared slots of the neighbours, whether it owns the
// variable.  hl: threads left of the owned ones (0 on a ring, where the CTA is the whole state).
struct Place {
    int i, l1, l2, r1, r2;
    bool own;
};

template <bool RING>
__device__ __forceinline__ Place place(int n, int U, int hl)
{
    Place p;
    const int q = threadIdx.x, B = blockDim.x;
    if (RING) {
        p.own = q < n;
        p.i = p.own ? q : 0;
        p.l1 = p.i >= 1 ? p.i - 1 : n - 1;
        p.l2 = p.i >= 2 ? p.i - 2 : p.i + n - 2;
        p.r1 = p.i + 1 < n ? p.i + 1 : 0;
        p.r2 = p.i + 2 < n ? p.i + 2 : p.i + 2 - n;
    } else {
        const int g = blockIdx.x * U + q - hl;
        p.own = q >= hl && q < hl + U && g < n;
        int i = g % n;
        p.i = i < 0 ? i + n : i;
        // threads at the ends read a neighbour that does not exist: their values are wrong from
        // the first stage on, and what depends on them never reaches an owned variable
        p.l1 = q >= 1 ? q - 1 : 0;
        p.l2 = q >= 2 ? q - 2 : 0;
        p.r1 = q + 1 < B ? q + 1 : B - 1;
        p.r2 = q + 2 < B ? q + 2 : B - 1;
    }
    return p;
}

__device__ __forceinline__ int wrap(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

struct NlSteps {
    ChunkGeom geom;
    int U, hl, t0, t1, last;
    double h, F;
    const double *in;    // state at t0
    double *traj;        // (T + 1) x n, may be null
    double *out;         // state at t1 when traj is null
    double2 *coef64;     // may be null
};

// RK4 steps t0 .. t1 - 1 of the nonlinear model, with the stage coefficients
// (X_{i-1}, X_{i+1} - X_{i-2}) of every stage state.
template <bool RING>
__global__ void __launch_bounds__(512) nl_steps_kernel(const NlSteps a)
{
    extern __shared__ double sm_nl[];
    const int n = a.geom.n, q = threadIdx.x, B = blockDim.x;
    const Place p = place<RING>(n, a.U, a.hl);
    const int slot = a.geom.slot(p.i);
    const double h = a.h, h2 = 0.5 * a.h, h6 = a.h / 6.0, F = a.F;
    cudaGridDependencySynchronize();
    double x = a.in[p.i];
    if (a.traj && a.t0 == 0 && p.own) a.traj[p.i] = x;
    int hb = 0;
    for (int t = a.t0; t < a.t1; ++t) {
        if (t == max(a.t0, a.t1 - 2)) cudaTriggerProgrammaticLaunchCompletion();
        double X = x, acc = 0.0;
#pragma unroll
        for (int st = 0; st < 4; ++st) {
            double *S = sm_nl + hb * B;
            hb ^= 1;
            S[q] = X;
            __syncthreads();
            const double ca = S[p.l1], cb = S[p.r1] - S[p.l2];
            if (a.coef64 && p.own) a.coef64[((size_t)t * 4 + st) * a.geom.Np + slot] = make_double2(ca, cb);
            const double f = fma(cb, ca, -X) + F;
            acc = (st == 0) ? f : fma(st == 3 ? 1.0 : 2.0, f, acc);
            if (st < 3) X = fma(st == 2 ? h : h2, f, x);
        }
        x = fma(h6, acc, x);
        if (a.traj && p.own) a.traj[(size_t)(t + 1) * n + p.i] = x;
    }
    if (!a.traj && p.own) a.out[p.i] = x;
}

constexpr int kMaxSteps = 48;   // steps of one launch

struct LinSteps {
    ChunkGeom geom;
    int U, hl, t0, t1, last;     // last: this launch ends the window
    double h;
    const double2 *coef;
    int row[kMaxSteps + 1];      // row of step t0 + i among the observed steps, -1 if none
    const double *wgt;           // tangent linear: weights of the rows (null: 1)
    const double *in;            // null: 0
    double *out;
    double *rows;                // [column][nrow][n]
    long long lds, ldr;          // columns of the states, of the rows
};

// A state's value at place o of its row: times its weight where there are weights, and 0 without an
// observation whatever the value (an infinity times zero would be NaN).
__device__ __forceinline__ double row_value(const double *wgt, size_t o, double x)
{
    if (!wgt) return x;
    const double w = wgt[o];
    return __double_as_longlong(w) == 0 ? 0.0 : w * x;
}

// Tangent-linear steps t0 .. t1 - 1; the (weighted) state of every observed step goes to its row.
template <bool RING>
__global__ void __launch_bounds__(512) tl_steps_kernel(const LinSteps a)
{
    extern __shared__ double sm_tl[];
    const int n = a.geom.n, Np = a.geom.Np, q = threadIdx.x, B = blockDim.x;
    const Place p = place<RING>(n, a.U, a.hl);
    const double2 *cf = a.coef + a.geom.slot(p.i);
    const double h = a.h, h2 = 0.5 * a.h, h6 = a.h / 6.0;
    double *rows = a.rows + (size_t)blockIdx.y * a.ldr;
    int hb = 0, row = a.row[0];
    double2 c[4], cn[4];
#pragma unroll
    for (int st = 0; st < 4; ++st)
        c[st] = cn[st] = a.t0 < a.t1 ? cf[((size_t)a.t0 * 4 + st) * Np] : make_double2(0.0, 0.0);
    cudaGridDependencySynchronize();
    double x = a.in[(size_t)blockIdx.y * a.lds + p.i];
    for (int t = a.t0; t < a.t1; ++t) {
        if (t == max(a.t0, a.t1 - 2)) cudaTriggerProgrammaticLaunchCompletion();
        if (row >= 0 && p.own) {
            const size_t o = (size_t)row * n + p.i;
            rows[o] = row_value(a.wgt, o, x);
        }
        if (t + 1 < a.t1) {
#pragma unroll
            for (int st = 0; st < 4; ++st) cn[st] = cf[((size_t)(t + 1) * 4 + st) * Np];
        }
        row = a.row[t + 1 - a.t0];
        double s = x, acc = 0.0;
#pragma unroll
        for (int st = 0; st < 4; ++st) {
            double *S = sm_tl + hb * B;
            hb ^= 1;
            S[q] = s;
            __syncthreads();
            const double k = fma(c[st].x, S[p.r1] - S[p.l2], fma(c[st].y, S[p.l1], -s));
            acc = (st == 0) ? k : fma(st == 3 ? 1.0 : 2.0, k, acc);
            if (st < 3) s = fma(st == 2 ? h : h2, k, x);
        }
        x = fma(h6, acc, x);
#pragma unroll
        for (int st = 0; st < 4; ++st) c[st] = cn[st];   // here, so that the loads have the whole step
    }
    if (!p.own) return;
    if (a.last) {
        if (row >= 0) {
            const size_t o = (size_t)row * n + p.i;
            rows[o] = row_value(a.wgt, o, x);
        }
    } else {
        a.out[(size_t)blockIdx.y * a.lds + p.i] = x;
    }
}

// Adjoint steps from state t1 down to t0; the row of every observed step is added before its
// step, and that of step 0 at the end.  With mu = (h / 6) lam the four stages of the adjoint are
// l4 = J4^T mu, 2 n3 = l3, n3 = J3^T (mu + (h / 2) l4), 2 n2 = l2, n2 = J2^T (mu + (h / 2) n3),
// l1 = J1^T (mu + h n2): eight operations per variable and step beside the tendencies.
template <bool RING>
__global__ void __launch_bounds__(512) ad_steps_kernel(const LinSteps a)
{
    extern __shared__ double sm_ad[];
    const int n = a.geom.n, Np = a.geom.Np, q = threadIdx.x, B = blockDim.x;
    const Place p = place<RING>(n, a.U, a.hl);
    // (J^T m)_i = a_{i-1} m_{i-1} - a_{i+2} m_{i+2} + b_{i+1} m_{i+1} - m_i
    const double2 *cl = a.coef + a.geom.slot(wrap(p.i - 1, n)), *cr1 = a.coef + a.geom.slot(wrap(p.i + 1, n)),
                  *cr2 = a.coef + a.geom.slot(wrap(p.i + 2, n));
    const double h = a.h, h2 = 0.5 * a.h, h6 = a.h / 6.0;
    const double *rows = a.rows + (size_t)blockIdx.y * a.ldr + p.i;
    int hb = 0, row = a.row[a.t1 - a.t0];
    double f = row >= 0 ? rows[(size_t)row * n] : 0.0, fn = 0.0;
    double c[4][3], cn[4][3];
#pragma unroll
    for (int st = 0; st < 4; ++st) {
        const size_t o = ((size_t)(a.t1 - 1) * 4 + st) * Np;
        c[st][0] = cn[st][0] = cl[o].x;
        c[st][1] = cn[st][1] = cr1[o].y;
        c[st][2] = cn[st][2] = cr2[o].x;
    }
    cudaGridDependencySynchronize();
    double lam = a.in ? a.in[(size_t)blockIdx.y * a.lds + p.i] : 0.0;
    for (int t = a.t1; t > a.t0; --t) {
        if (t == min(a.t1, a.t0 + 2)) cudaTriggerProgrammaticLaunchCompletion();
        if (row >= 0) lam += f;
        row = a.row[t - 1 - a.t0];
        if (row >= 0) fn = rows[(size_t)row * n];
        if (t - 1 > a.t0) {
#pragma unroll
            for (int st = 0; st < 4; ++st) {
                const size_t o = ((size_t)(t - 2) * 4 + st) * Np;
                cn[st][0] = cl[o].x;
                cn[st][1] = cr1[o].y;
                cn[st][2] = cr2[o].x;
            }
        }
        const double mu = h6 * lam;
        double m = mu;
#pragma unroll
        for (int st = 3; st >= 0; --st) {
            double *S = sm_ad + hb * B;
            hb ^= 1;
            S[q] = m;
            __syncthreads();
            const double k = fma(c[st][0], S[p.l1], fma(-c[st][2], S[p.r2], fma(c[st][1], S[p.r1], -m)));
            lam = (st == 0 || st == 3) ? lam + k : fma(2.0, k, lam);
            if (st > 0) m = fma(st == 1 ? h : h2, k, mu);
        }
#pragma unroll
        for (int st = 0; st < 4; ++st)
#pragma unroll
            for (int w = 0; w < 3; ++w) c[st][w] = cn[st][w];
        f = fn;
    }
    if (!p.own) return;
    // the row of a launch's last state is added by the next launch, or here at the end
    if (a.last && row >= 0) lam += f;
    a.out[(size_t)blockIdx.y * a.lds + p.i] = lam;
}

constexpr int kInnovCtas = kJoDoubles - 2;   // a partial sum each

// The sum of a value per thread of a CTA of 256, in a fixed order; thread 0 has it.
__device__ __forceinline__ double cta_sum(double s)
{
    __shared__ double ws[8];
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < 8; ++w) s += ws[w];
    return s;
}

// d = H(x) - y, 1/2 sum d^2 / sigma^2 added to jo[0], and R^-1 d added to the rows (zeroed before).
// The sum is the same bits every time: the CTAs' partial sums (jo[2] on) are added in order by the
// CTA that finishes last (counted in the bytes of jo[1], zero at launch).
__global__ void __launch_bounds__(256) innov_kernel(int p, int n, const int *obsrow, const int *rowstep, const int *oidx,
                                                    const double *traj, const double *y, const double *rinv, double *d,
                                                    double *rows, double *jo)
{
    __shared__ bool last;
    double s = 0.0;
    for (int o = blockIdx.x * blockDim.x + threadIdx.x; o < p; o += gridDim.x * blockDim.x) {
        const int r = obsrow[o], i = oidx[o];
        const double dd = traj[(size_t)rowstep[r] * n + i] - y[o], w = dd * rinv[o];
        d[o] = dd;
        if (rows) atomicAdd(&rows[(size_t)r * n + i], w);
        s = fma(0.5 * dd, w, s);
    }
    s = cta_sum(s);
    if (threadIdx.x == 0) {
        jo[2 + blockIdx.x] = s;
        __threadfence();
        last = atomicAdd((unsigned *)(jo + 1), 1u) + 1 == gridDim.x;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    s = cta_sum(threadIdx.x < gridDim.x ? __ldcg(jo + 2 + threadIdx.x) : 0.0);
    if (threadIdx.x == 0) jo[0] += s;
}

__global__ void rows_scatter_kernel(int p, int n, const int *obsrow, const int *oidx, const double *r, double *rows)
{
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o < p) atomicAdd(&rows[(size_t)obsrow[o] * n + oidx[o]], r[o]);
}

__global__ void rows_gather_kernel(int p, int n, const int *obsrow, const int *oidx, const double *rinv,
                                   const double *rows, double *r)
{
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o < p) r[o] = rinv[o] * rows[(size_t)obsrow[o] * n + oidx[o]];
}

// FP32 stage coefficients from the FP64 ones: float4 (j / 2) * Tp + t of a stage holds the pair
// of variables j, j + 1 of chunk t, as the FP32 Hessian kernel reads them.
__global__ void coef32_kernel(const double2 *c64, int E, int Tp, int Np, long long total, float4 *c32)
{
    const long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (id >= total) return;
    const int half = Np / 2;
    const long long stage = id / half;
    const int r = (int)(id - stage * half), jp = r / Tp, t = r - jp * Tp;
    const double2 *c = c64 + stage * Np + (size_t)t * E + 2 * jp;
    const double2 c0 = c[0], c1 = c[1];
    c32[id] = make_float4((float)c0.x, (float)c0.y, (float)c1.x, (float)c1.y);
}

inline unsigned blocks_for(size_t n, int t) { return (unsigned)((n + t - 1) / t); }

// Block size B and steps per launch K for `ncols` columns of n variables (K = 0: a ring).  Model:
// a step takes tau per warp of a sub-partition (5 FP64 instructions of 64 cycles per stage, the
// exchange and its barrier: 1.05 us measured for one warp, 0.85 each for more), a launch `gap`
// more.  More steps per launch recompute more, which costs nothing while SMs are idle: n = 4096
// takes 8 steps on 128 CTAs for one column and 6 on 148 for two.
struct SplitPlan {
    int B, K;
    double us;   // per step
};

constexpr double kTau = 0.85, kGap = 3.0;

SplitPlan split_plan(int n, int ncols)
{
    const int sms = num_sms();
    SplitPlan best = {0, 0, 1e300};
    if (n <= 256) {
        const int B = (n + 31) / 32 * 32;
        best = {B, 0, kTau * ((ncols + sms - 1) / sms) * ((B + 127) / 128)};
    }
    for (int B = 128; B <= 512; B *= 2)
        for (int K = 1; K <= kMaxSteps && B - 12 * K >= 16; ++K) {
            const int U = B - 12 * K;
            const long long ctas = (long long)((n + U - 1) / U) * ncols;
            const double us = kTau * (double)((ctas + sms - 1) / sms) * (B / 128) + kGap / K;
            if (us < best.us) best = {B, K, us};
        }
    return best;
}

// Launches of `ring` or `split` over steps [0, T) (up) or from state T down; set(args, first) fills
// the rest of the arguments, whose t0, t1 and last are set.  A launch after the first is queued
// as a programmatic dependent of the one before: its CTAs start in that one's last two steps,
// load their coefficients (written before the first launch) and wait for it to end before they
// touch a state or a row.
template <typename A, typename F>
cudaError_t for_steps(const SplitPlan &pl, int n, int T, bool up, int ncols, void (*ring)(A), void (*split)(A), A a,
                      cudaStream_t s, F set)
{
    const int K = pl.K ? pl.K : kMaxSteps;
    a.U = pl.K ? pl.B - 12 * pl.K : n;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(pl.K ? blocks_for(n, a.U) : 1, ncols);
    cfg.blockDim = dim3(pl.B);
    cfg.dynamicSmemBytes = 2 * pl.B * sizeof(double);
    cfg.stream = s;
    cfg.attrs = &attr;
    for (int b = 0; b < T; b += K) {
        const int e = b + K < T ? b + K : T;
        a.t0 = up ? b : T - e;
        a.t1 = up ? e : T - b;
        a.last = e == T;
        cfg.numAttrs = b > 0;
        set(a, b == 0);
        count_launch();
        const cudaError_t err = cudaLaunchKernelEx(&cfg, pl.K ? split : ring, a);
        if (err != cudaSuccess) return err;
    }
    return cudaSuccess;
}

cudaError_t rows_zero(const L96Dev &m, cudaStream_t s)
{
    return cudaMemsetAsync(m.sp.rows, 0, sizeof(double) * (size_t)m.sp.nrow * m.geom.n, s);
}

}  // namespace

// The nonlinear trajectory from x0 (traj, or only the final state into xT; x0 may lie in either)
// and its FP64 stage coefficients (may be null).
cudaError_t l96_nl_launch(const L96Dev &m, const double *x0, double *traj, double2 *coef64, double *xT, cudaStream_t s)
{
    const int n = m.geom.n, T = m.T;
    const SplitPlan pl = T > 0 ? split_plan(n, 1) : SplitPlan{0, 0, 0.0};
    // A launch's CTAs read the start while others write, so a start that overlaps what is written is
    // set aside (one that is row 0 itself is only written with its own values).  Without a
    // trajectory the states of successive launches alternate between xT and a temporary.
    const double *end = traj ? traj + (size_t)(T + 1) * n : xT + n;
    const bool clash = x0 != traj && x0 < end && (traj ? traj : xT) < x0 + n;
    const bool more = !traj && T > (pl.K > 0 ? pl.K : kMaxSteps);
    double *tmp = nullptr;
    cudaError_t e;
    if (clash || more) {
        if ((e = cudaMallocAsync((void **)&tmp, 2 * sizeof(double) * n, s)) != cudaSuccess) {
            cudaGetLastError();
            return e;
        }
        if (clash) {
            e = cudaMemcpyAsync(tmp + n, x0, sizeof(double) * n, cudaMemcpyDeviceToDevice, s);
            if (e != cudaSuccess) {
                cudaFreeAsync(tmp, s);
                return e;
            }
            x0 = tmp + n;
        }
    }
    const int K = pl.K > 0 ? pl.K : kMaxSteps, launches = (T + K - 1) / K;
    int at = 0;
    double *prev = nullptr;
    NlSteps a = {};
    a.geom = m.geom;
    a.hl = 8 * pl.K;
    a.h = m.dt;
    a.F = m.F;
    a.traj = traj;
    a.coef64 = coef64;
    if (T == 0) e = x0 == traj ? cudaSuccess : cudaMemcpyAsync(traj ? traj : xT, x0, sizeof(double) * n, cudaMemcpyDeviceToDevice, s);
    else e = for_steps(pl, n, T, true, 1, nl_steps_kernel<true>, nl_steps_kernel<false>, a, s, [&](NlSteps &b, bool first) {
        b.in = first ? x0 : traj ? traj + (size_t)b.t0 * n : prev;
        b.out = prev = ((launches - 1 - at++) & 1) ? tmp : xT;
    });
    if (tmp) {
        const cudaError_t e2 = cudaFreeAsync(tmp, s);
        if (e == cudaSuccess) e = e2;
    }
    return e;
}

cudaError_t l96_coef32(const L96Dev &m, const double2 *coef64, float2 *coef32, cudaStream_t s)
{
    const long long total = (long long)m.T * 4 * (m.geom.Np / 2);
    if (total == 0) return cudaSuccess;
    count_launch();
    coef32_kernel<<<blocks_for((size_t)total, 256), 256, 0, s>>>(coef64, m.geom.E, m.geom.Tp, m.geom.Np, total,
                                                                  (float4 *)coef32);
    return cudaGetLastError();
}

bool l96_split_better(const L96Dev &m, int ncols, double other_us)
{
    return ncols <= m.sp.cols && split_plan(m.geom.n, ncols).us < other_us;
}

static LinSteps lin_args(const L96Dev &m, const double2 *coef, double *rows)
{
    LinSteps a = {};
    a.geom = m.geom;
    a.h = m.dt;
    a.coef = coef;
    a.rows = rows;
    a.lds = m.geom.n;
    a.ldr = (long long)m.sp.nrow * m.geom.n;
    return a;
}

// Tangent-linear half: rows <- (R^-1) H M L W of `ncols` columns (with `weighted`, R^-1 in the
// form of the rows' weights)
static cudaError_t split_tl(const L96Dev &m, const double2 *coef, const double *W, int64_t ld, int ncols, bool weighted,
                            double *rows, cudaStream_t s)
{
    const int n = m.geom.n;
    const SplitWork &w = m.sp;
    SplitPlan pl = split_plan(n, ncols);
    cudaError_t e = bsqrt_launch(m, W, ld, w.a, n, 0, ncols, nullptr, s);
    if (e != cudaSuccess || w.nrow == 0) return e;
    LinSteps a = lin_args(m, coef, rows);
    a.wgt = weighted ? w.wgt : nullptr;
    a.hl = 8 * pl.K;
    double *src = w.a, *dst = w.b;
    if (w.last_step == 0) {   // only the initial state is observed: a launch without steps
        a.U = pl.K ? pl.B - 12 * pl.K : n;
        a.last = 1;
        a.in = src;
        const dim3 g(pl.K ? blocks_for(n, a.U) : 1, ncols);
        count_launch();
        if (pl.K == 0) tl_steps_kernel<true><<<g, pl.B, 2 * pl.B * sizeof(double), s>>>(a);
        else tl_steps_kernel<false><<<g, pl.B, 2 * pl.B * sizeof(double), s>>>(a);
        return cudaGetLastError();
    }
    return for_steps(pl, n, w.last_step, true, ncols, tl_steps_kernel<true>, tl_steps_kernel<false>, a, s,
                     [&](LinSteps &b, bool) {
                         std::copy(w.orow_h.begin() + b.t0, w.orow_h.begin() + b.t1 + 1, b.row);
                         b.in = src;
                         b.out = dst;
                         std::swap(src, dst);
                     });
}

// Adjoint half: *lam <- lambda_0 (n x ncols) from the rows
static cudaError_t split_ad(const L96Dev &m, const double2 *coef, int ncols, const double **lam, cudaStream_t s)
{
    const int n = m.geom.n;
    const SplitWork &w = m.sp;
    const SplitPlan pl = split_plan(n, ncols);
    *lam = w.a;
    if (w.nrow == 0) return cudaMemsetAsync(w.a, 0, sizeof(double) * (size_t)n * ncols, s);
    *lam = w.rows;   // nothing but the initial state observed: one row per column, lambda_0 itself
    if (w.last_step == 0) return cudaSuccess;
    LinSteps a = lin_args(m, coef, w.rows);
    a.hl = 4 * pl.K;
    double *src = w.a, *dst = w.b;
    const cudaError_t e = for_steps(pl, n, w.last_step, false, ncols, ad_steps_kernel<true>, ad_steps_kernel<false>, a, s,
                                    [&](LinSteps &b, bool first) {
                                        std::copy(w.orow_h.begin() + b.t0, w.orow_h.begin() + b.t1 + 1, b.row);
                                        b.in = first ? nullptr : src;
                                        b.out = dst;
                                        std::swap(src, dst);
                                    });
    *lam = src;
    return e;
}

cudaError_t l96_split_f64(const L96Dev &m, const double2 *coef, const double *W, double *Y, int64_t ld, int ncols,
                          int add_identity, double *r, int mode, cudaStream_t s)
{
    const SplitWork &w = m.sp;
    const int n = m.geom.n;
    if (ncols <= 0) return cudaSuccess;
    if (ncols > w.cols || (mode != 0 && ncols != 1)) return cudaErrorInvalidValue;
    cudaError_t e;
    const double *lam = nullptr;
    if (mode == 1) {
        if (m.p > 0) {
            if ((e = rows_zero(m, s)) != cudaSuccess) return e;
            count_launch();
            rows_scatter_kernel<<<blocks_for(m.p, 256), 256, 0, s>>>(m.p, n, w.obsrow, m.oidx, r, w.rows);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
    } else {
        if ((e = split_tl(m, coef, W, ld, ncols, mode == 0, w.rows, s)) != cudaSuccess) return e;
    }
    if (mode != 2) {
        if ((e = split_ad(m, coef, ncols, &lam, s)) != cudaSuccess) return e;
        return bsqrt_launch(m, lam, n, Y, ld, 1, ncols, mode == 0 && add_identity ? W : nullptr, s);
    }
    if (m.p == 0) return cudaSuccess;
    count_launch();
    rows_gather_kernel<<<blocks_for(m.p, 256), 256, 0, s>>>(m.p, n, w.obsrow, m.oidx, m.rinv64, w.rows, r);
    return cudaGetLastError();
}

cudaError_t l96_innov(const L96Dev &m, const double *traj, double *d, double *jo, bool rows, cudaStream_t s)
{
    if (m.p == 0) return cudaSuccess;
    cudaError_t e;
    if (rows && (e = rows_zero(m, s)) != cudaSuccess) return e;
    const unsigned grid = blocks_for(m.p, 256) < kInnovCtas ? blocks_for(m.p, 256) : kInnovCtas;
    count_launch();
    innov_kernel<<<grid, 256, 0, s>>>(m.p, m.geom.n, m.sp.obsrow, m.sp.rowstep, m.oidx, traj, m.y, m.rinv64, d,
                                      rows ? m.sp.rows : nullptr, jo);
    return cudaGetLastError();
}

// One adjoint pass serves the gradient (column 0, rows from l96_innov) and, with z, the product
// y = A z (column 1): two columns take 1.1 times the time of one, since one leaves SMs idle.
cudaError_t l96_split_gradient(const L96Dev &m, const double2 *coef, double *b, const double *z, double *y,
                               cudaStream_t s)
{
    const int n = m.geom.n;
    cudaError_t e;
    const double *lam = nullptr;
    if (z && (e = split_tl(m, coef, z, n, 1, true, m.sp.rows + (size_t)m.sp.nrow * n, s)) != cudaSuccess) return e;
    if ((e = split_ad(m, coef, z ? 2 : 1, &lam, s)) != cudaSuccess) return e;
    if ((e = bsqrt_launch(m, lam, n, b, n, 1, 1, nullptr, s)) != cudaSuccess || !z) return e;
    return bsqrt_launch(m, lam + n, n, y, n, 1, 1, nullptr, s);
}

}  // namespace riot
