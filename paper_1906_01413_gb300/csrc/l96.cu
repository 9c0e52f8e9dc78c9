// Lorenz-96 kernels of the RIOT inner loop on sm_103a.
//
// Model (Section 3.1): dx_i/dt = (x_{i+1} - x_{i-2}) x_{i-1} - x_i + F on a
// periodic ring, advanced by classical RK4.  The Hessian-vector product of
// Eq. 4, A w = L^T sum_t M_{0->t}^T H_t^T R^-1 H_t M_{0->t} L w, is one
// tangent-linear (TL) integration forward and one adjoint (AD) integration
// backward per sketch column (Algorithm 3, "do in parallel").
//
// Design (one GPU, probe-batched):
//  * A CTA owns P probes (sketch columns) x the whole state.  Thread t of a
//    probe keeps E consecutive variables of that probe in registers for the
//    whole window; the periodic stencil reaches across chunk boundaries
//    through a double-buffered shared-memory halo (3-4 words per thread per
//    RK4 stage, one barrier).
//  * The base trajectory enters as per-stage coefficients (a_i, b_i) =
//    (X_{i-1}, X_{i+1} - X_{i-2}) of every RK4 stage state X, written once per
//    outer iteration by the FP64 nonlinear kernel.  Then the TL tendency is
//    a_i (s_{i+1} - s_{i-2}) + b_i s_{i-1} - s_i and the AD tendency is the
//    gather p_{i-1} - p_{i+2} + q_{i+1} - m_i with p = a m, q = b m: both need
//    only per-element coefficients, loaded as 16-byte vectors from L2.
//  * Observations are gathered (TL) and scattered (AD) through a swizzled
//    shared copy of the state; the TL residuals R^-1 H dx wait in global
//    scratch for the AD pass of the same CTA.
//  * L (banded symmetric circulant times diag(sigma)) is applied in the
//    prologue and L^T in the epilogue of the same kernel, so one launch
//    computes the whole Hessian-vector product.
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace riot {

template <typename real> struct V2;
template <> struct V2<float> { using type = float2; };
template <> struct V2<double> { using type = double2; };

// one pad word every 8 words: conflict-free strided access to the state copy
__device__ __forceinline__ int sw(int x) { return x + (x >> 3); }

__host__ __device__ __forceinline__ int stage_pad(int Np) { return Np + (Np >> 3) + 2; }

bool choose_geom(int n, ChunkGeom *g)
{
    if (n < 16 || n > 8192) return false;
    const int cand[3] = {n > 4096 ? 16 : 8, 8, 4};
    for (int c = 0; c < 3; ++c) {
        int E = cand[c];
        int Tp = (n + E - 1) / E;
        int gg = Tp * E - n;
        if (Tp > 512) continue;
        if (gg <= Tp && E - 1 >= 3) {
            g->n = n; g->E = E; g->Tp = Tp; g->g = gg; g->Np = Tp * E;
            return true;
        }
    }
    return false;
}

// ---------------------------------------------------------------------------
// Halo exchanges.  H holds 2 buffers x 4 arrays x nthr words.
// ---------------------------------------------------------------------------
template <typename real, int E>
__device__ __forceinline__ void xchg_tl(const real (&s)[E], bool full, real *H, int nthr, int tid,
                                        int left, int right, int &hb, real &m2, real &m1, real &p1)
{
    real *Hb = H + hb * 4 * nthr;
    Hb[tid] = full ? s[E - 2] : s[E - 3];
    Hb[nthr + tid] = full ? s[E - 1] : s[E - 2];
    Hb[2 * nthr + tid] = s[0];
    __syncthreads();
    m2 = Hb[left];
    m1 = Hb[nthr + left];
    p1 = Hb[2 * nthr + right];
    hb ^= 1;
}

// TL tendency k = J(X) s with per-element coefficients (a, b) of stage X.
template <typename real, int E>
__device__ __forceinline__ void tl_tend(const real (&s)[E], real (&k)[E], const typename V2<real>::type *cf,
                                        bool full, real *H, int nthr, int tid, int left, int right, int &hb)
{
    real m2, m1, p1;
    xchg_tl<real, E>(s, full, H, nthr, tid, left, right, hb, m2, m1, p1);
#pragma unroll
    for (int j = 0; j < E; ++j) {
        typename V2<real>::type c = cf[j];
        real xm2 = (j == 0) ? m2 : (j == 1 ? m1 : s[j >= 2 ? j - 2 : 0]);
        real xm1 = (j == 0) ? m1 : s[j >= 1 ? j - 1 : 0];
        real xp1;
        if (j == E - 1) xp1 = p1;
        else if (j == E - 2) xp1 = full ? s[E - 1] : p1;
        else xp1 = s[j + 1 < E ? j + 1 : 0];
        k[j] = fma(c.x, xp1 - xm2, fma(c.y, xm1, -s[j]));
    }
    if (!full) k[E - 1] = real(0);
}

// AD tendency out = J(X)^T m: a_{j-1} m_{j-1} - a_{j+2} m_{j+2} + b_{j+1} m_{j+1} - m_j in three
// operations (the products a m, b m and their sums would be five); cl points at the left
// chunk's last coefficient pair, cr at the right chunk's first.
template <typename real, int E>
__device__ __forceinline__ void ad_tend(const real (&m)[E], real (&out)[E], const typename V2<real>::type *cf,
                                        const typename V2<real>::type *cl, const typename V2<real>::type *cr,
                                        bool full, real *H, int nthr, int tid, int left, int right, int &hb)
{
    real *Hb = H + hb * 4 * nthr;
    Hb[tid] = full ? m[E - 1] : m[E - 2];
    Hb[nthr + tid] = m[0];
    Hb[2 * nthr + tid] = m[1];
    real ca[E], cb[E];
#pragma unroll
    for (int j = 0; j < E; ++j) {
        typename V2<real>::type c = cf[j];
        ca[j] = c.x;
        cb[j] = c.y;
    }
    const real aL = cl->x, aR1 = cr[1].x;
    const typename V2<real>::type cR0 = cr[0];
    __syncthreads();
    const real mL = Hb[left], mR0 = Hb[nthr + right], mR1 = Hb[2 * nthr + right];
    hb ^= 1;
#pragma unroll
    for (int j = 0; j < E; ++j) {
        const real mm1 = (j == 0) ? mL : m[j >= 1 ? j - 1 : 0];
        const real am1 = (j == 0) ? aL : ca[j >= 1 ? j - 1 : 0];
        real mp1, bp1, mp2, ap2;
        if (j <= E - 2 && (full || j <= E - 3)) {
            mp1 = m[j + 1 < E ? j + 1 : 0];
            bp1 = cb[j + 1 < E ? j + 1 : 0];
        } else {
            mp1 = mR0;
            bp1 = cR0.y;
        }
        if (j <= E - 3 && (full || j <= E - 4)) {
            mp2 = m[j + 2 < E ? j + 2 : 0];
            ap2 = ca[j + 2 < E ? j + 2 : 0];
        } else if (full ? (j == E - 2) : (j == E - 3)) {
            mp2 = mR0;
            ap2 = cR0.x;
        } else {
            mp2 = mR1;
            ap2 = aR1;
        }
        out[j] = fma(am1, mm1, fma(-ap2, mp2, fma(bp1, mp1, -m[j])));
    }
    if (!full) out[E - 1] = real(0);
}

template <typename real>
struct HvpArgs {
    ChunkGeom geom;
    int T, P, p, hl, hh, ncols, add_identity, mode;
    real dt;
    const typename V2<real>::type *coef;
    const int *optr, *oslot;
    const real *rinv, *band, *sig, *W;
    real *Y, *r;
    long long ld;
};

// Banded circulant apply at own elements: out_j = pre_i * sum_d S_d u_{i+d}
template <typename real, int E>
__device__ __forceinline__ void band_apply(const real *st, const real *band, int hl, int hh, int n, int s0,
                                           int len, real (&out)[E])
{
#pragma unroll
    for (int j = 0; j < E; ++j) out[j] = real(0);
    for (int d = -hl; d <= hh; ++d) {
        real w = band[d + hl];
#pragma unroll
        for (int j = 0; j < E; ++j) {
            int ii = s0 + j + d;
            ii += (ii < 0) ? n : 0;
            ii -= (ii >= n) ? n : 0;
            if (j < len) out[j] += w * st[sw(ii)];
        }
    }
}

template <typename real, int E>
__global__ void __launch_bounds__(512) l96_hvp_kernel(const HvpArgs<real> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    real *H = reinterpret_cast<real *>(smem_raw);
    const int nthr = blockDim.x;
    const ChunkGeom &G = a.geom;
    const int Np = G.Np, n = G.n, Tp = G.Tp, P = a.P;
    const int SP = stage_pad(Np);
    real *state = H + 8 * nthr;

    const int tid = threadIdx.x;
    const int t = tid / P, pp = tid - (tid / P) * P;
    const int probe = blockIdx.x * P + pp;
    const bool active = probe < a.ncols;
    const int left = ((t == 0) ? Tp - 1 : t - 1) * P + pp;
    const int right = ((t == Tp - 1) ? 0 : t + 1) * P + pp;
    const int s0 = G.start(t);
    const int len = G.len(t);
    const bool full = (len == E);
    const int tl = (t == 0) ? Tp - 1 : t - 1, tr = (t == Tp - 1) ? 0 : t + 1, lenL = G.len(tl);
    real *st = state + pp * SP;
    int hb = 0;
    const real h = a.dt, h2 = real(0.5) * a.dt, h6 = a.dt / real(6);
    const size_t rbase = (size_t)(active ? probe : 0) * (size_t)a.p;

    real dx[E];
    if (a.mode != 1) {
        // ---- prologue: dx_0 = L w = diag(sigma) S w ----
        const real *w = a.W + (size_t)(active ? probe : 0) * a.ld;
        for (int i = t; i < n; i += Tp) st[sw(i)] = active ? w[i] : real(0);
        __syncthreads();
        band_apply<real, E>(st, a.band, a.hl, a.hh, n, s0, len, dx);
#pragma unroll
        for (int j = 0; j < E; ++j) dx[j] = (j < len) ? dx[j] * a.sig[s0 + (j < len ? j : 0)] : real(0);
        __syncthreads();

        // ---- TL forward ----
        for (int tt = 0;; ++tt) {
            const int o0 = a.optr[tt], o1 = a.optr[tt + 1];
            if (o0 < o1) {
#pragma unroll
                for (int j = 0; j < E; ++j) st[sw(t * E + j)] = dx[j];
                __syncthreads();
                if (active)
                    for (int o = o0 + t; o < o1; o += Tp) a.r[rbase + o] = a.rinv[o] * st[sw(a.oslot[o])];
                __syncthreads();
            }
            if (tt == a.T) break;
            const typename V2<real>::type *cf = a.coef + (size_t)tt * 4 * Np + t * E;
            real s[E], k[E], acc[E];
#pragma unroll
            for (int j = 0; j < E; ++j) s[j] = dx[j];
            tl_tend<real, E>(s, k, cf, full, H, nthr, tid, left, right, hb);
#pragma unroll
            for (int j = 0; j < E; ++j) { acc[j] = k[j]; s[j] = fma(h2, k[j], dx[j]); }
            tl_tend<real, E>(s, k, cf + Np, full, H, nthr, tid, left, right, hb);
#pragma unroll
            for (int j = 0; j < E; ++j) { acc[j] = fma(real(2), k[j], acc[j]); s[j] = fma(h2, k[j], dx[j]); }
            tl_tend<real, E>(s, k, cf + 2 * Np, full, H, nthr, tid, left, right, hb);
#pragma unroll
            for (int j = 0; j < E; ++j) { acc[j] = fma(real(2), k[j], acc[j]); s[j] = fma(h, k[j], dx[j]); }
            tl_tend<real, E>(s, k, cf + 3 * Np, full, H, nthr, tid, left, right, hb);
#pragma unroll
            for (int j = 0; j < E; ++j) { acc[j] += k[j]; dx[j] = fma(h6, acc[j], dx[j]); }
        }
        if (a.mode == 2) return;
    }

    // ---- AD backward ----
    real lam[E];
#pragma unroll
    for (int j = 0; j < E; ++j) lam[j] = real(0);
    for (int tt = a.T;; --tt) {
        const int o0 = a.optr[tt], o1 = a.optr[tt + 1];
        if (o0 < o1) {
#pragma unroll
            for (int j = 0; j < E; ++j) st[sw(t * E + j)] = lam[j];
            __syncthreads();
            if (active)
                for (int o = o0 + t; o < o1; o += Tp) atomicAdd(&st[sw(a.oslot[o])], a.r[rbase + o]);
            __syncthreads();
#pragma unroll
            for (int j = 0; j < E; ++j) lam[j] = (j < len) ? st[sw(t * E + j)] : real(0);
        }
        if (tt == 0) break;
        // lam_0 = lam + l4 + l3 + l2 + l1 with mu = (h / 6) lam, l4 = J4^T mu, l3 = 2 n3, n3 =
        // J3^T (mu + (h / 2) l4), l2 = 2 n2, n2 = J2^T (mu + (h / 2) n3), l1 = J1^T (mu + h n2)
        const typename V2<real>::type *cs = a.coef + (size_t)(tt - 1) * 4 * Np;
        const int oL = tl * E + lenL - 1, oR = tr * E;
        real mu[E], m[E], k[E];
#pragma unroll
        for (int j = 0; j < E; ++j) m[j] = mu[j] = h6 * lam[j];
#pragma unroll
        for (int st = 3; st >= 0; --st) {
            const typename V2<real>::type *c = cs + st * Np;
            ad_tend<real, E>(m, k, c + t * E, c + oL, c + oR, full, H, nthr, tid, left, right, hb);
#pragma unroll
            for (int j = 0; j < E; ++j) {
                lam[j] = (st == 0 || st == 3) ? lam[j] + k[j] : fma(real(2), k[j], lam[j]);
                if (st > 0) m[j] = fma(st == 1 ? h : h2, k[j], mu[j]);
            }
        }
    }

    // ---- epilogue: y = L^T lambda_0 = S diag(sigma) lambda_0 (+ w) ----
    __syncthreads();
#pragma unroll
    for (int j = 0; j < E; ++j)
        if (j < len) st[sw(s0 + j)] = a.sig[s0 + j] * lam[j];
    __syncthreads();
    real y[E];
    band_apply<real, E>(st, a.band, a.hl, a.hh, n, s0, len, y);
    if (active) {
        real *yo = a.Y + (size_t)probe * a.ld;
        const real *w = a.W ? a.W + (size_t)probe * a.ld : nullptr;
#pragma unroll
        for (int j = 0; j < E; ++j)
            if (j < len) yo[s0 + j] = y[j] + ((a.add_identity && w) ? w[s0 + j] : real(0));
    }
}

// Columns per CTA of the FP64 kernel and its modelled time per RK4 step.  The kernel is bound by
// FP64 issue, one warp instruction per 64 cycles and SM sub-partition, so what counts is the
// largest number of warps that a sub-partition gets: few columns per CTA spread over all SMs
// (128 columns of 1000 variables: 32 CTAs of four columns 3.5 ms, 128 CTAs of one 0.7 ms), more
// where a column alone leaves most of a warp's lanes idle.
double hvp_f64_plan(const ChunkGeom &g, int ncols, int *P_out)
{
    int Pmax = 512 / g.Tp;
    if (Pmax > ncols) Pmax = ncols;
    if (Pmax > 64) Pmax = 64;
    const int sms = num_sms();
    long long best = -1;
    for (int P = 1; P <= Pmax; ++P) {
        const long long ctas = (ncols + P - 1) / P, warps = (P * g.Tp + 31) / 32;
        const long long load = ((ctas + sms - 1) / sms * warps + 3) / 4;
        if (best < 0 || load < best) {
            best = load;
            *P_out = P;
        }
    }
    return 0.85 * (double)best * g.E;
}

template <typename real>
static cudaError_t hvp_launch(const L96Dev &m, const typename V2<real>::type *coef, const real *W, real *Y,
                              int64_t ld, int ncols, int add_identity, real *r, int mode,
                              const real *rinv, const real *band, const real *sig, cudaStream_t s)
{
    if (ncols <= 0) return cudaSuccess;
    HvpArgs<real> a;
    a.geom = m.geom;
    a.T = m.T;
    a.p = m.p;
    a.hl = m.band.hl;
    a.hh = m.band.hh;
    a.ncols = ncols;
    a.add_identity = add_identity;
    a.mode = mode;
    a.dt = (real)m.dt;
    a.coef = coef;
    a.optr = m.optr;
    a.oslot = m.oslot;
    a.rinv = rinv;
    a.band = band;
    a.sig = sig;
    a.W = W;
    a.Y = Y;
    a.r = r;
    a.ld = ld;
    const int Tp = m.geom.Tp;
    int P = 0;
    hvp_f64_plan(m.geom, ncols, &P);
    if (P < 1) return cudaErrorInvalidConfiguration;
    a.P = P;
    const int nthr = P * Tp;
    const size_t sm = sizeof(real) * (8 * (size_t)nthr + (size_t)P * stage_pad(m.geom.Np));
    const int grid = (ncols + P - 1) / P;
    static SmemLimit limit[3];
    auto launch = [&](auto kern, SmemLimit &lim) {
        const cudaError_t e = lim.raise((const void *)kern, sm);
        if (e != cudaSuccess) return e;
        count_launch();
        kern<<<grid, nthr, sm, s>>>(a);
        return cudaGetLastError();
    };
    switch (m.geom.E) {
    case 4: return launch(l96_hvp_kernel<real, 4>, limit[0]);
    case 8: return launch(l96_hvp_kernel<real, 8>, limit[1]);
    case 16: return launch(l96_hvp_kernel<real, 16>, limit[2]);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t l96_hvp_launch_f64(const L96Dev &m, const double2 *coef, const double *W, double *Y, int64_t ld,
                               int ncols, int add_identity, double *r, int mode, cudaStream_t s)
{
    return hvp_launch<double>(m, coef, W, Y, ld, ncols, add_identity, r, mode, m.rinv64, m.band64, m.sig64, s);
}

// ---------------------------------------------------------------------------
// Standalone L / L^T application in FP64 (outer-loop update, covariance, split integrations).
// A block of 64 threads forms 64 outputs of one column from a window of the column in shared
// memory (scaled there for L^T: one product per value instead of one per tap).
// ---------------------------------------------------------------------------
constexpr int kBsqrtBlock = 64;

__global__ void __launch_bounds__(kBsqrtBlock) bsqrt_kernel(int n, int hl, int hh, const double *band, const double *sig,
                                                            const double *in, long long ldi, double *out,
                                                            long long ldo, int transpose, const double *add)
{
    extern __shared__ double sm_band[];
    const int i0 = blockIdx.x * kBsqrtBlock, i = i0 + threadIdx.x;
    const double *x = in + (size_t)blockIdx.y * ldi;
    const int width = kBsqrtBlock + hl + hh;
    for (int w = threadIdx.x; w < width; w += kBsqrtBlock) {
        int ii = (i0 + w - hl) % n;
        ii += (ii < 0) ? n : 0;
        sm_band[w] = transpose ? sig[ii] * x[ii] : x[ii];
    }
    __syncthreads();
    if (i >= n) return;
    double acc = 0.0;
    for (int d = 0; d <= hl + hh; ++d) acc = fma(band[d], sm_band[threadIdx.x + d], acc);
    double y = transpose ? acc : sig[i] * acc;
    if (add) y += add[(size_t)blockIdx.y * ldo + i];
    out[(size_t)blockIdx.y * ldo + i] = y;
}

cudaError_t bsqrt_launch(const L96Dev &m, const double *in, int64_t ldi, double *out, int64_t ldo, int transpose,
                         int ncols, const double *add, cudaStream_t s)
{
    if (ncols <= 0) return cudaSuccess;
    const int n = m.geom.n;
    const size_t sm = sizeof(double) * (kBsqrtBlock + m.band.hl + m.band.hh);   // at most 64 + 8191 values
    static SmemLimit limit;
    cudaError_t e = limit.raise((const void *)bsqrt_kernel, sm);
    if (e != cudaSuccess) return e;
    for (int c0 = 0; c0 < ncols; c0 += 65535) {
        const dim3 grid((n + kBsqrtBlock - 1) / kBsqrtBlock, ncols - c0 < 65535 ? ncols - c0 : 65535);
        count_launch();
        bsqrt_kernel<<<grid, kBsqrtBlock, sm, s>>>(n, m.band.hl, m.band.hh, m.band64, m.sig64, in + (size_t)c0 * ldi, ldi,
                                                   out + (size_t)c0 * ldo, ldo, transpose,
                                                   add ? add + (size_t)c0 * ldo : nullptr);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace riot
