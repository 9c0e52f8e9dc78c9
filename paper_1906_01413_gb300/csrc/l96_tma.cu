// FP32 batched Lorenz-96 Hessian-vector kernel with TMA-streamed stage coefficients.
//
// Same mathematics as l96_hvp_kernel (Eq. 4 through one tangent-linear RK4
// integration forward and one adjoint integration backward per sketch
// column, Algorithm 3), arranged for sm_103a:
//  * The per-stage base coefficients (a, b) of a whole state (Np float2) are
//    streamed from global memory into a ring of S shared-memory stage
//    buffers by one thread with cp.async.bulk (the 1-D TMA copy), completion
//    tracked by an mbarrier per buffer.  The copy for stage u + S - 1 is
//    issued as soon as every thread has passed the barrier of stage u, so
//    global-memory latency is hidden behind S - 1 stages of arithmetic and
//    every coefficient is read once per CTA and shared by its P probes.
//  * P probes per CTA (512 threads for E <= 8) keep their state in
//    registers; halos cross chunk boundaries through shared memory, one CTA
//    barrier per stage.
//  * Every wait on an mbarrier is bounded; a wait that runs out raises a
//    flag in global memory (reported as RIOT_ETIMEOUT) and the CTA carries
//    on, so the kernel always finishes.
//
// Bound: instruction issue and the barrier of every stage (67 % of the issue slots of a busy
// SM; 157 instructions per warp and stage, 85 of them FP32).  What the stage's critical path
// does not do: no division by the run-time ring depth in the thread that feeds the ring (every
// warp waits for it at the barrier; 400 cycles a stage), no proxy fence before a refill
// (buffers are only read between copies; 150 cycles), no loads of coefficients behind the
// barrier (all warps at once: 40 cycles, and 350 more when they were held a stage ahead in a
// second set of registers).  n = 4096, T = 200, 512 columns: 2717 -> 1870 us; n = 1003, 77
// columns 807 -> 254 us; n = 40 200 -> 80 us; n = 8191, 192 columns 2495 -> 1778 us; the same
// products bit for bit.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "internal.h"

namespace riot {

namespace {

__device__ __forceinline__ int swz(int x) { return x + (x >> 3); }
__host__ __device__ __forceinline__ int stage_pad_t(int Np) { return Np + (Np >> 3) + 2; }

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

__device__ __forceinline__ void mbar_inval(uint32_t bar)
{
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait of at most `polls` polls (default kWaitPolls, about 2^20 polls,
// well under a second).  After one wait of the CTA has run out, later waits
// return at once: the results are then wrong, the flag says so (value 1),
// and the kernel still finishes promptly.
constexpr int kWaitPolls = 1 << 20;

__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity, int *err, volatile int *abort_flag,
                                                  int polls)
{
    for (int i = 0; i < polls; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if (i > 32) __nanosleep(64);
    }
    *abort_flag = 1;
    atomicMax(err, 1);
    return false;
}

struct TmaArgs {
    ChunkGeom geom;
    int T, P, S, p, hl, hh, ncols, add_identity, mode;
    int wait_polls;   // poll bound of each wait on a stage copy (kWaitPolls unless a test lowers it)
    float dt;
    const float2 *coef;
    const int *optr, *oslot;
    const float *rinv, *band, *sig, *W;
    float *Y, *r;
    long long ld;
    int *err;
};

// Ring of stage buffers fed by thread 0.  Stream position c = 0.. counts the
// stages this launch consumes; stage c of the stream is coefficient block
// blk(c) of the [T][4] array: forward for the tangent-linear pass, backward
// for the adjoint pass.  Thread 0 keeps `issued` (copies started) and
// `landed` (stages whose copy it has seen complete) so that after an abort it
// can still wait for every copy it started before the CTA exits.
template <typename Args>
struct Ring {
    const Args &a;
    float2 *buf;
    uint32_t buf0, bar0;
    int S, Np, total;
    int issued, landed;
    volatile int *abort_flag;
    bool aborted;   // a wait of this thread ran out (or one of an earlier item's)
    __device__ int blk(int c) const
    {
        const int T = a.T, u = ((a.mode == 1) ? 4 * T : 0) + c;
        return u < 4 * T ? u : 8 * T - 1 - u;
    }
    // Stage c into buffer `slot` (c mod S: kept by the caller, divisions by S would hold up the
    // barrier that everything waits at).
    __device__ void issue(int c, int slot)
    {
        const uint32_t bytes = (uint32_t)Np * 8u;
        const uint32_t bar = bar0 + 8u * slot;
        // the buffer's last readers have passed a CTA barrier; no proxy fence: within a body's run
        // ordinary accesses only read it (what came before is fenced at the run's start)
        mbar_expect_tx(bar, bytes);
        bulk_g2s(buf0 + (uint32_t)slot * bytes, a.coef + (size_t)blk(c) * Np, bytes, bar);
        issued = c + 1;
    }
    // Every thread: wait until stage c, in buffer `slot` with phase parity `phase`, has landed; its
    // reads of the buffer then need no barrier.
    __device__ void wait_ready(int c, int slot, int phase, int *err)
    {
        if (aborted) return;
        aborted = !mbar_wait_bounded(bar0 + 8u * slot, (uint32_t)phase, err, abort_flag, a.wait_polls);
        if (!aborted) landed = c + 1;
    }
    // Thread 0 only, behind the barrier of stage c: refill the buffer of stage c - 1 with stage
    // c - 1 + S.  Every thread has its coefficients of stage c - 1 by then: what it published before
    // the barrier depends on the neighbours' values of that stage, which it loaded after them, and
    // a warp's shared loads return in order.  Those of stage c may still be on their way.
    __device__ void refill(int c, int slot)
    {
        if (threadIdx.x == 0 && c > 0 && c - 1 + S < total && !aborted) issue(c - 1 + S, slot ? slot - 1 : S - 1);
    }
    __device__ const float4 *slot4(int slot) const { return reinterpret_cast<const float4 *>(buf + (size_t)slot * Np); }
    // After an abort: wait, with the full bound whatever the test limit, for every
    // copy this CTA started and has not seen land.  Each such stage sits in its own
    // buffer (a buffer is refilled only after its previous stage landed), so its
    // phase parity identifies it.  A copy still in flight after that raises the
    // flag to 2: it may land in shared memory the CTA no longer owns.
    __device__ void drain(int *err)
    {
        if (threadIdx.x != 0 || !aborted) return;
        for (int c = landed; c < issued; ++c) {
            bool done = false;
            for (int i = 0; i < kWaitPolls && !done; ++i) {
                done = mbar_try_wait(bar0 + 8u * (c % S), (uint32_t)((c / S) & 1));
                if (!done && i > 32) __nanosleep(64);
            }
            if (!done) atomicMax(err, 2);
        }
    }
};

// The PR probes of a thread as one shared-memory word (PR floats).
template <int PR>
struct Vec {
    float v[PR];
};
template <>
struct __align__(8) Vec<2> {
    float v[2];
};

// Stage coefficients of a thread's E variables in registers (shared by its PR probes), and for
// the adjoint those of the neighbours' variables it needs: a of the left chunk's last variable,
// (a, b) of the right chunk's first, a of its second.
template <int E>
struct Coefs {
    float a[E], b[E];
    float aL, aR0, bR0, aR1;
};

// Place of a thread's coefficients in a stage buffer (float4 pairs interleaved by thread).
struct CoefAt {
    int t, tr, Tp, offL, oddL;
};

template <int E, bool AD>
__device__ __forceinline__ void load_coefs(Coefs<E> &c, const float4 *s4, const CoefAt &at)
{
#pragma unroll
    for (int j2 = 0; j2 < E / 2; ++j2) {
        const float4 f = s4[j2 * at.Tp + at.t];
        c.a[2 * j2] = f.x;
        c.b[2 * j2] = f.y;
        c.a[2 * j2 + 1] = f.z;
        c.b[2 * j2 + 1] = f.w;
    }
    if (AD) {
        const float4 cl = s4[at.offL], cr = s4[at.tr];
        c.aL = at.oddL ? cl.z : cl.x;
        c.aR0 = cr.x;
        c.bR0 = cr.y;
        c.aR1 = cr.z;
    }
}

// Stream position c, its buffer c mod S and the parity of c / S.
struct StageAt {
    int c, slot, phase;
    __device__ __forceinline__ void advance(int S)
    {
        ++c;
        if (++slot == S) {
            slot = 0;
            phase ^= 1;
        }
    }
};

// One stage's inputs: the coefficients and the neighbours' edge values, exchanged around the
// stage's barrier.  The coefficients are loaded before it (while other warps still compute:
// behind it all warps' loads come at once), but behind it with 16 variables per thread, where
// shared memory holds two stages of the largest states and the next copy has to start first
// (n = 8191: 1.9 ms against 2.5).
template <int E, bool AD, int PR, typename Args>
__device__ __forceinline__ void stage_inputs(Coefs<E> &cc, const CoefAt &at, const Vec<PR> (&give)[3], Vec<PR> (&get)[3],
                                             Vec<PR> *H, int nthr, int tid, const int (&from)[3], int &hb,
                                             Ring<Args> &ring, const StageAt &sa, int *err)
{
    constexpr bool EARLY = E <= 8;
    Vec<PR> *Hb = H + hb * 3 * nthr;
#pragma unroll
    for (int i = 0; i < 3; ++i) Hb[i * nthr + tid] = give[i];
    if (EARLY) {
        ring.wait_ready(sa.c, sa.slot, sa.phase, err);
        load_coefs<E, AD>(cc, ring.slot4(sa.slot), at);
    }
    __syncthreads();
    ring.refill(sa.c, sa.slot);
    if (!EARLY) {
        ring.wait_ready(sa.c, sa.slot, sa.phase, err);
        load_coefs<E, AD>(cc, ring.slot4(sa.slot), at);
        asm volatile("" ::: "memory");   // in this order, as refill needs it
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) get[i] = Hb[i * nthr + from[i]];
    hb ^= 1;
}

// Tangent-linear tendency k = J(X) s of one probe.
template <int E>
__device__ __forceinline__ void tl_tend32(const float (&s)[E], float (&k)[E], const Coefs<E> &c, bool full, float m2,
                                          float m1, float p1)
{
#pragma unroll
    for (int j = 0; j < E; ++j) {
        const float xm2 = (j == 0) ? m2 : (j == 1 ? m1 : s[j >= 2 ? j - 2 : 0]);
        const float xm1 = (j == 0) ? m1 : s[j >= 1 ? j - 1 : 0];
        float xp1;
        if (j == E - 1) xp1 = p1;
        else if (j == E - 2) xp1 = full ? s[E - 1] : p1;
        else xp1 = s[j + 1 < E ? j + 1 : 0];
        k[j] = fmaf(c.a[j], xp1 - xm2, fmaf(c.b[j], xm1, -s[j]));
    }
    if (!full) k[E - 1] = 0.f;
}

// Adjoint tendency out = J(X)^T m of one probe:
// (J^T m)_j = a_{j-1} m_{j-1} - a_{j+2} m_{j+2} + b_{j+1} m_{j+1} - m_j, three FMAs
template <int E>
__device__ __forceinline__ void ad_tend32(const float (&m)[E], float (&out)[E], const Coefs<E> &c, bool full, float mL,
                                          float mR0, float mR1)
{
#pragma unroll
    for (int j = 0; j < E; ++j) {
        const float mm1 = (j == 0) ? mL : m[j >= 1 ? j - 1 : 0];
        const float am1 = (j == 0) ? c.aL : c.a[j >= 1 ? j - 1 : 0];
        float mp1, bp1;
        if (j <= E - 2 && (full || j <= E - 3)) {
            mp1 = m[j + 1 < E ? j + 1 : 0];
            bp1 = c.b[j + 1 < E ? j + 1 : 0];
        } else {
            mp1 = mR0;
            bp1 = c.bR0;
        }
        float mp2, ap2;
        if (j <= E - 3 && (full || j <= E - 4)) {
            mp2 = m[j + 2 < E ? j + 2 : 0];
            ap2 = c.a[j + 2 < E ? j + 2 : 0];
        } else if (full ? (j == E - 2) : (j == E - 3)) {
            mp2 = mR0;
            ap2 = c.aR0;
        } else {
            mp2 = mR1;
            ap2 = c.aR1;
        }
        out[j] = fmaf(am1, mm1, fmaf(-ap2, mp2, fmaf(bp1, mp1, -m[j])));
    }
    if (!full) out[E - 1] = 0.f;
}

// out_j = sum_d band_d st[s0 + j + d]: the E values that a tap multiplies are a window in
// registers that moves by one value per tap.
template <int E>
__device__ __forceinline__ void band_apply_t(const float *st, const float *band, int hl, int hh, int n, int s0,
                                             float (&out)[E])
{
    float x[E];
    int ii = s0 - hl;
    ii += (ii < 0) ? n : 0;
#pragma unroll
    for (int j = 0; j < E; ++j) {
        out[j] = 0.f;
        x[j] = st[swz(ii)];
        ii = (ii + 1 == n) ? 0 : ii + 1;
    }
    for (int d0 = 0; d0 <= hl + hh; d0 += E) {
#pragma unroll
        for (int u = 0; u < E; ++u) {
            if (d0 + u > hl + hh) break;
            const float w = band[d0 + u];
#pragma unroll
            for (int j = 0; j < E; ++j) out[j] = fmaf(w, x[(u + j) % E], out[j]);
            x[u] = st[swz(ii)];
            ii = (ii + 1 == n) ? 0 : ii + 1;
        }
    }
}

// One thread's first observation of a step (observation o0 + t), loaded a step ahead.
struct ObsAhead {
    int o0, o1, slot;
    float w;   // weight (tangent linear)
};

// A CTA holds P thread groups of Tp threads; group g owns probes
// blk * P * PR + g * PR + r, r < PR, and thread t of a group keeps chunk t of
// each of them in registers.  Threads from P * Tp up to blockDim.x (a
// persistent batch kernel runs windows of several sizes in one block shape)
// are idle: they follow the barriers and touch only their own halo slots.
// Args: TmaArgs, or volatile TmaArgs in shared memory (then nothing of it stays in registers).
template <int E, int PR, bool RAGGED, typename Args>
__device__ __forceinline__ void hvp_tma_body(const Args &a, int blk, unsigned char *smem_raw, int *abort_flag)
{
    ChunkGeom G;
    G.n = a.geom.n;
    G.E = E;
    G.Tp = a.geom.Tp;
    G.g = a.geom.g;
    G.Np = a.geom.Np;
    const int Np = G.Np, n = G.n, Tp = G.Tp, P = a.P, S = a.S;
    const int nthr = blockDim.x;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem_raw);
    float2 *ringbuf = reinterpret_cast<float2 *>(smem_raw + 128);
    Vec<PR> *H = reinterpret_cast<Vec<PR> *>(ringbuf + (size_t)S * Np);
    float *state = reinterpret_cast<float *>(H + 2 * 3 * nthr);
    const int SP = stage_pad_t(Np);

    const int tid = threadIdx.x;
    const bool live = tid < P * Tp;
    const int t = live ? tid / P : 0, g = live ? tid - (tid / P) * P : 0;
    const int probe0 = (blk * P + g) * PR;
    const int left = ((t == 0) ? Tp - 1 : t - 1) * P + g;
    const int right = ((t == Tp - 1) ? 0 : t + 1) * P + g;
    const int s0 = G.start(t);
    const int len = G.len(t);
    const bool full = !RAGGED || (len == E);   // RAGGED = false: every chunk has E variables
    const int tE = t * E;
    const int tl = (t == 0) ? Tp - 1 : t - 1, tr = (t == Tp - 1) ? 0 : t + 1;
    const int lenL = G.len(tl);
    const CoefAt at = {t, tr, Tp, ((lenL - 1) >> 1) * Tp + tl, (lenL - 1) & 1};
    int hb = 0;
    const float h = a.dt, h2 = 0.5f * a.dt, h6 = a.dt / 6.f, h3 = a.dt / 3.f;

    Ring<Args> ring = {a};
    ring.buf = ringbuf;
    ring.buf0 = smem_u32(ringbuf);
    ring.bar0 = smem_u32(bars);
    ring.S = S;
    ring.Np = Np;
    ring.total = ((a.mode == 2) ? 4 * a.T : 8 * a.T) - ((a.mode == 1) ? 4 * a.T : 0);
    ring.issued = 0;
    ring.landed = 0;
    ring.abort_flag = abort_flag;
    if (tid == 0) {
        for (int i = 0; i < S; ++i) mbar_init(ring.bar0 + 8u * i, 1);
        fence_mbar_init();
    }
    // a batch kernel's earlier item, whose ring had another size, may have written these bytes as
    // halo or state: order its ordinary accesses before the copies' writes
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    // behind the barrier: the flag is thread 0's store, and what the shared word held before it
    // (whatever an earlier kernel left) would end every wait of this thread at once
    ring.aborted = *ring.abort_flag;
    if (tid == 0) {
        for (int c = 0; c < S && c < ring.total; ++c) ring.issue(c, c);
    }
    StageAt sa = {0, 0, 0};
    Coefs<E> cc;

    float dx[PR][E];
    if (a.mode != 1) {
        ObsAhead ob = {a.optr[0], a.optr[1], 0, 0.f};
        if (live && ob.o0 + t < ob.o1) {
            ob.slot = a.oslot[ob.o0 + t];
            ob.w = a.rinv[ob.o0 + t];
        }
#pragma unroll
        for (int r = 0; r < PR; ++r) {
            const int probe = probe0 + r;
            const bool active = probe < a.ncols;
            float *st = state + (g * PR + r) * SP;
            const float *w = a.W + (size_t)(active ? probe : 0) * a.ld;
            if (live)
                for (int i = t; i < n; i += Tp) st[swz(i)] = active ? w[i] : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < PR; ++r) {
            float tmp[E];
            band_apply_t<E>(state + (g * PR + r) * SP, a.band, a.hl, a.hh, n, s0, tmp);
#pragma unroll
            for (int j = 0; j < E; ++j) dx[r][j] = (j < len) ? tmp[j] * a.sig[s0 + (j < len ? j : 0)] : 0.f;
        }
        __syncthreads();
        const int from[3] = {left, left, right};
        for (int tt = 0;; ++tt) {
            if (ob.o0 < ob.o1) {
                if (live)
#pragma unroll
                    for (int r = 0; r < PR; ++r) {
                        float *st = state + (g * PR + r) * SP;
#pragma unroll
                        for (int j = 0; j < E; ++j) st[swz(tE + j)] = dx[r][j];
                    }
                __syncthreads();
#pragma unroll
                for (int r = 0; r < PR; ++r) {
                    const int probe = probe0 + r;
                    if (live && probe < a.ncols) {
                        const float *st = state + (g * PR + r) * SP;
                        float *rr = a.r + (size_t)probe * (size_t)a.p;
                        if (ob.o0 + t < ob.o1) rr[ob.o0 + t] = ob.w * st[swz(ob.slot)];
                        for (int o = ob.o0 + t + Tp; o < ob.o1; o += Tp) rr[o] = a.rinv[o] * st[swz(a.oslot[o])];
                    }
                }
                __syncthreads();
            }
            if (tt == a.T) break;
            ob.o0 = ob.o1;
            ob.o1 = a.optr[tt + 2];
            float s[PR][E], acc[PR][E];
#pragma unroll
            for (int r = 0; r < PR; ++r)
#pragma unroll
                for (int j = 0; j < E; ++j) s[r][j] = dx[r][j];
#pragma unroll
            for (int st = 0; st < 4; ++st) {
                Vec<PR> give[3], get[3];
#pragma unroll
                for (int r = 0; r < PR; ++r) {
                    give[0].v[r] = full ? s[r][E - 2] : s[r][E - 3];
                    give[1].v[r] = full ? s[r][E - 1] : s[r][E - 2];
                    give[2].v[r] = s[r][0];
                }
                stage_inputs<E, false>(cc, at, give, get, H, nthr, tid, from, hb, ring, sa, a.err);
                if (st == 2 && live && ob.o0 + t < ob.o1) {   // the next step's observation, a step ahead
                    ob.slot = a.oslot[ob.o0 + t];
                    ob.w = a.rinv[ob.o0 + t];
                }
#pragma unroll
                for (int r = 0; r < PR; ++r) {
                    float k[E];
                    tl_tend32<E>(s[r], k, cc, full, get[0].v[r], get[1].v[r], get[2].v[r]);
#pragma unroll
                    for (int j = 0; j < E; ++j) {
                        acc[r][j] = (st == 0) ? k[j] : (st == 3) ? acc[r][j] + k[j] : fmaf(2.f, k[j], acc[r][j]);
                        if (st < 3) s[r][j] = fmaf(st == 2 ? h : h2, k[j], dx[r][j]);
                    }
                }
                sa.advance(S);
            }
#pragma unroll
            for (int r = 0; r < PR; ++r)
#pragma unroll
                for (int j = 0; j < E; ++j) dx[r][j] = fmaf(h6, acc[r][j], dx[r][j]);
        }
        if (a.mode == 2) {
            ring.drain(a.err);
            __syncthreads();
            if (tid == 0)
                for (int i = 0; i < S; ++i) mbar_inval(ring.bar0 + 8u * i);
            return;
        }
    }
    float lam[PR][E];
#pragma unroll
    for (int r = 0; r < PR; ++r)
#pragma unroll
        for (int j = 0; j < E; ++j) lam[r][j] = 0.f;
    ObsAhead ob = {a.optr[a.T], a.optr[a.T + 1], 0, 0.f};
    float ro[PR];
#pragma unroll
    for (int r = 0; r < PR; ++r) ro[r] = 0.f;
    auto obs_ahead = [&]() {
        if (live && ob.o0 + t < ob.o1) {
            ob.slot = a.oslot[ob.o0 + t];
#pragma unroll
            for (int r = 0; r < PR; ++r)
                if (probe0 + r < a.ncols) ro[r] = a.r[(size_t)(probe0 + r) * (size_t)a.p + ob.o0 + t];
        }
    };
    obs_ahead();
    const int from[3] = {left, right, right};
    for (int tt = a.T;; --tt) {
        if (ob.o0 < ob.o1) {
            if (live)
#pragma unroll
                for (int r = 0; r < PR; ++r) {
                    float *st = state + (g * PR + r) * SP;
#pragma unroll
                    for (int j = 0; j < E; ++j) st[swz(tE + j)] = lam[r][j];
                }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < PR; ++r) {
                const int probe = probe0 + r;
                if (live && probe < a.ncols) {
                    float *st = state + (g * PR + r) * SP;
                    const float *rr = a.r + (size_t)probe * (size_t)a.p;
                    if (ob.o0 + t < ob.o1) atomicAdd(&st[swz(ob.slot)], ro[r]);
                    for (int o = ob.o0 + t + Tp; o < ob.o1; o += Tp) atomicAdd(&st[swz(a.oslot[o])], rr[o]);
                }
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < PR; ++r) {
                const float *st = state + (g * PR + r) * SP;
#pragma unroll
                for (int j = 0; j < E; ++j) lam[r][j] = (j < len) ? st[swz(tE + j)] : 0.f;
            }
        }
        if (tt == 0) break;
        ob.o1 = ob.o0;
        ob.o0 = a.optr[tt - 1];
        // l4 = J4^T (h/6) lam, l3 = J3^T ((h/3) lam + h l4), l2 = J2^T ((h/3) lam + (h/2) l3), l1 =
        // J1^T ((h/6) lam + (h/2) l2), lam_0 = lam + l4 + l3 + l2 + l1
        float lx[PR][E], m[PR][E];
#pragma unroll
        for (int r = 0; r < PR; ++r)
#pragma unroll
            for (int j = 0; j < E; ++j) m[r][j] = h6 * lam[r][j];
#pragma unroll
        for (int st = 0; st < 4; ++st) {
            Vec<PR> give[3], get[3];
#pragma unroll
            for (int r = 0; r < PR; ++r) {
                give[0].v[r] = full ? m[r][E - 1] : m[r][E - 2];
                give[1].v[r] = m[r][0];
                give[2].v[r] = m[r][1];
            }
            stage_inputs<E, true>(cc, at, give, get, H, nthr, tid, from, hb, ring, sa, a.err);
            if (st == 2) obs_ahead();
#pragma unroll
            for (int r = 0; r < PR; ++r) {
                float k[E];
                ad_tend32<E>(m[r], k, cc, full, get[0].v[r], get[1].v[r], get[2].v[r]);
#pragma unroll
                for (int j = 0; j < E; ++j) {
                    lx[r][j] = (st == 0 ? lam[r][j] : lx[r][j]) + k[j];
                    if (st < 3) m[r][j] = fmaf(st == 2 ? h6 : h3, lam[r][j], (st == 0 ? h : h2) * k[j]);
                    else lam[r][j] = lx[r][j];
                }
            }
            sa.advance(S);
        }
    }

    ring.drain(a.err);
    __syncthreads();
    if (tid == 0)
        for (int i = 0; i < S; ++i) mbar_inval(ring.bar0 + 8u * i);
    if (live)
#pragma unroll
        for (int r = 0; r < PR; ++r) {
            float *st = state + (g * PR + r) * SP;
#pragma unroll
            for (int j = 0; j < E; ++j)
                if (j < len) st[swz(s0 + j)] = a.sig[s0 + j] * lam[r][j];
        }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < PR; ++r) {
        const int probe = probe0 + r;
        float y[E];
        band_apply_t<E>(state + (g * PR + r) * SP, a.band, a.hl, a.hh, n, s0, y);
        if (live && probe < a.ncols) {
            float *yo = a.Y + (size_t)probe * a.ld;
            const float *w = a.W ? a.W + (size_t)probe * a.ld : nullptr;
#pragma unroll
            for (int j = 0; j < E; ++j)
                if (j < len) yo[s0 + j] = y[j] + ((a.add_identity && w) ? w[s0 + j] : 0.f);
        }
    }
}

template <int E, int PR, int MAXT, bool RAGGED, int MINB = 1>
__global__ void __launch_bounds__(MAXT, MINB) l96_hvp_tma_kernel(const TmaArgs a)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ int abort_flag;
    if (threadIdx.x == 0) abort_flag = 0;
    hvp_tma_body<E, PR, RAGGED>(a, blockIdx.x, smem_raw, &abort_flag);
}

// Persistent kernel over a queue of (window, block) items of several
// Lorenz-96 windows: each CTA takes the next item until the queue is empty,
// so windows of different sizes share one launch.
struct BatchItem {
    int win, blk;
};

template <int MAXT>
__global__ void __launch_bounds__(MAXT, 1) l96_hvp_batch_kernel(const TmaArgs *args, const BatchItem *items, int nitems,
                                                                int *counter)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ int abort_flag, item_s;
    // the item's window; volatile, so that its fields are read where they are used: held in
    // registers beside the state they spill
    __shared__ volatile TmaArgs a;
    if (threadIdx.x == 0) abort_flag = 0;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) item_s = atomicAdd(counter, 1);
        __syncthreads();
        const int it = item_s;
        if (it >= nitems) break;
        const BatchItem bi = items[it];
        static_assert(sizeof(TmaArgs) % sizeof(int) == 0 && sizeof(TmaArgs) / sizeof(int) <= MAXT, "copied by words");
        if (threadIdx.x < sizeof(TmaArgs) / sizeof(int))
            reinterpret_cast<volatile int *>(&a)[threadIdx.x] = reinterpret_cast<const int *>(args + bi.win)[threadIdx.x];
        __syncthreads();
        const int E = a.geom.E;
        if (E == 4) hvp_tma_body<4, 2, true>(a, bi.blk, smem_raw, &abort_flag);
        else if (E == 8) hvp_tma_body<8, 2, true>(a, bi.blk, smem_raw, &abort_flag);
        else hvp_tma_body<16, 1, true>(a, bi.blk, smem_raw, &abort_flag);
    }
}


// Shared memory: barriers, S stage buffers, halo (2 buffers x 3 x PR x nthr),
// state copies of the P * PR probes.
size_t tma_smem_bytes(int Np, int nthr, int P, int S, int PR)
{
    return 128 + (size_t)S * Np * 8 + sizeof(float) * (6 * (size_t)PR * nthr + (size_t)P * PR * stage_pad_t(Np));
}

}  // namespace

// Probe groups P per CTA and ring depth S within the shared-memory budget; positive hints are
// taken when they fit.  Otherwise the shape with the least modelled time per stage: a wave of CTAs
// takes 350 cycles (exchange, barrier, latency) and 8 per variable and probe for each warp of a
// sub-partition, so a few columns spread over the SMs (77 columns of n = 1003: 77 CTAs of one
// column 254 us, ten of eight more than twice that) and many fill a CTA.  Returns that time, < 0 if nothing fits.
static double tma_plan(const ChunkGeom &g, int ncols, int PR, int maxthr, size_t smem_max, int P_hint, int S_hint,
                       int *P_out, int *S_out)
{
    const int groups_needed = (ncols + PR - 1) / PR, sms = num_sms();
    int Pmax = maxthr / g.Tp;
    if (Pmax > 64) Pmax = 64;
    if (Pmax > groups_needed) Pmax = groups_needed;
    if (P_hint > 0 || S_hint > 0) {
        const int P = (P_hint > 0 && P_hint <= Pmax) ? P_hint : Pmax;
        const int S = (S_hint >= 2 && S_hint <= 8) ? S_hint : 4;
        if (P >= 1 && tma_smem_bytes(g.Np, P * g.Tp, P, S, PR) <= smem_max) {
            *P_out = P;
            *S_out = S;
            return 0.0;
        }
    }
    double best = -1.0;
    for (int P = 1; P <= Pmax; ++P) {
        int S = 8;
        while (S > 2 && tma_smem_bytes(g.Np, P * g.Tp, P, S, PR) > smem_max) --S;
        const size_t sm = tma_smem_bytes(g.Np, P * g.Tp, P, S, PR);
        if (sm > smem_max) continue;
        const int warps = (P * g.Tp + 31) / 32, ctas = (groups_needed + P - 1) / P, per_sm = (ctas + sms - 1) / sms;
        int fit = maxthr / (32 * warps);   // CTAs an SM holds at a time
        if (fit > (int)(smem_max / sm)) fit = (int)(smem_max / sm);
        if (fit < 1) fit = 1;
        if (fit > per_sm) fit = per_sm;
        const double t = (double)((per_sm + fit - 1) / fit) * (350.0 + 8.0 * g.E * PR * ((fit * warps + 3) / 4));
        if (best < 0.0 || t < best) {
            best = t;
            *P_out = P;
            *S_out = S;
        }
    }
    return best;
}

template <int E, int PR, int MAXT, int MINB = 1>
static cudaError_t launch_tma(const TmaArgs &a, int grid, int nthr, size_t sm, cudaStream_t s)
{
    const bool ragged = a.geom.g != 0;
    auto kern = ragged ? l96_hvp_tma_kernel<E, PR, MAXT, true, MINB> : l96_hvp_tma_kernel<E, PR, MAXT, false, MINB>;
    static SmemLimit limit[2];
    const cudaError_t e = limit[ragged].raise((const void *)kern, sm);
    if (e != cudaSuccess) return e;
    count_launch();
    kern<<<grid, nthr, sm, s>>>(a);
    return cudaGetLastError();
}

cudaError_t l96_hvp_tma_launch(const L96Dev &m, const float2 *coef, const float *W, float *Y, int64_t ld, int ncols,
                               int add_identity, float *r, int mode, int *err, cudaStream_t s, int P_hint, int S_hint,
                               int wait_polls, bool two_per_sm)
{
    if (ncols <= 0) return cudaSuccess;
    int dev = 0, smem_optin = 0, smem_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    const int E = m.geom.E;
    // two probes per thread (registers) for E <= 8: 512-thread CTAs, one per SM; one where few
    // columns leave SMs idle otherwise (E = 8); two_per_sm (E = 8): one probe per thread in 64
    // registers, two CTAs per SM sharing its shared memory
    const bool pair = two_per_sm && E == 8;
    int PR = (E <= 8 && !pair) ? 2 : 1;
    const int maxthr = 512;
    const size_t smem_max = pair ? (size_t)smem_sm / 2 - 1024 : (size_t)smem_optin - 1024;
    int P = 1, S = 2;
    const double t = tma_plan(m.geom, ncols, PR, maxthr, smem_max, P_hint, S_hint, &P, &S);
    if (t < 0.0) return cudaErrorInvalidConfiguration;
    if (PR == 2 && E == 8 && t > 0.0) {
        int P1 = 1, S1 = 2;
        const double t1 = tma_plan(m.geom, ncols, 1, maxthr, smem_max, 0, 0, &P1, &S1);
        if (t1 >= 0.0 && t1 < t) {
            PR = 1;
            P = P1;
            S = S1;
        }
    }
    TmaArgs a;
    a.geom = m.geom;
    a.T = m.T;
    a.P = P;
    a.S = S;
    a.p = m.p;
    a.hl = m.band.hl;
    a.hh = m.band.hh;
    a.ncols = ncols;
    a.add_identity = add_identity;
    a.mode = mode;
    a.wait_polls = wait_polls >= 0 ? wait_polls : kWaitPolls;
    a.dt = (float)m.dt;
    a.coef = coef;
    a.optr = m.optr;
    a.oslot = m.oslot;
    a.rinv = m.rinv32;
    a.band = m.band32;
    a.sig = m.sig32;
    a.W = W;
    a.Y = Y;
    a.r = r;
    a.ld = ld;
    a.err = err;
    const int nthr = P * m.geom.Tp;
    const size_t sm = tma_smem_bytes(m.geom.Np, nthr, P, S, PR);
    const int per_cta = P * PR;
    const int grid = (ncols + per_cta - 1) / per_cta;
    switch (E) {
    case 4: return launch_tma<4, 2, 512>(a, grid, nthr, sm, s);
    case 8:
        if (pair) return launch_tma<8, 1, 512, 2>(a, grid, nthr, sm, s);
        return PR == 1 ? launch_tma<8, 1, 512>(a, grid, nthr, sm, s) : launch_tma<8, 2, 512>(a, grid, nthr, sm, s);
    case 16: return launch_tma<16, 1, 512>(a, grid, nthr, sm, s);
    default: return cudaErrorInvalidValue;
    }
}

// ---------------------------------------------------------------------------
// Batch of windows in one persistent launch
// ---------------------------------------------------------------------------
void hvp_batch_free(HvpBatchPlan *plan)
{
    if (!plan) return;
    cudaFree(plan->d_args);
    cudaFree(plan->d_items);
    cudaFree(plan->d_counter);
    plan->d_args = plan->d_items = nullptr;
    plan->d_counter = nullptr;
    plan->nitems = plan->nwin = 0;
}

cudaError_t hvp_batch_plan(const HvpBatchWindow *w, int nwin, int P_cap, int S_req, HvpBatchPlan *plan)
{
    constexpr int kThreads = 512;
    int dev = 0, smem_optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const size_t smax = (size_t)smem_optin - 1024;
    std::vector<TmaArgs> args(nwin);
    struct Cand {
        double cost;
        BatchItem it;
    };
    std::vector<Cand> items;
    size_t smem = 0;
    for (int i = 0; i < nwin; ++i) {
        const L96Dev &m = *w[i].m;
        const ChunkGeom &g = m.geom;
        const int PR = (g.E <= 8) ? 2 : 1;
        if (g.Tp > kThreads || w[i].ncols < 1) return cudaErrorInvalidConfiguration;
        int P = kThreads / g.Tp;
        if (P > 64) P = 64;
        if (P_cap > 0 && P > P_cap) P = P_cap;
        const int groups = (w[i].ncols + PR - 1) / PR;
        if (P > groups) P = groups;
        int S = (S_req >= 2 && S_req <= 8) ? S_req : 4;
        while (S > 2 && tma_smem_bytes(g.Np, kThreads, P, S, PR) > smax) --S;
        while (P > 1 && tma_smem_bytes(g.Np, kThreads, P, S, PR) > smax) --P;
        const size_t sm = tma_smem_bytes(g.Np, kThreads, P, S, PR);
        if (sm > smax) return cudaErrorInvalidConfiguration;
        if (sm > smem) smem = sm;
        TmaArgs &a = args[i];
        a.geom = g;
        a.T = m.T;
        a.P = P;
        a.S = S;
        a.p = m.p;
        a.hl = m.band.hl;
        a.hh = m.band.hh;
        a.ncols = w[i].ncols;
        a.add_identity = 0;
        a.mode = 0;
        a.wait_polls = kWaitPolls;
        a.dt = (float)m.dt;
        a.coef = w[i].coef;
        a.optr = m.optr;
        a.oslot = m.oslot;
        a.rinv = m.rinv32;
        a.band = m.band32;
        a.sig = m.sig32;
        a.W = w[i].W;
        a.Y = w[i].Y;
        a.r = w[i].r;
        a.ld = w[i].ld;
        a.err = w[i].err;
        const int nblk = (w[i].ncols + P * PR - 1) / (P * PR);
        // per-thread work of an item grows with T * E * PR: longest first
        const double cost = (double)m.T * g.E * PR;
        for (int b = 0; b < nblk; ++b) items.push_back({cost, {i, b}});
    }
    std::stable_sort(items.begin(), items.end(), [](const Cand &x, const Cand &y) { return x.cost > y.cost; });
    std::vector<BatchItem> its(items.size());
    for (size_t i = 0; i < items.size(); ++i) its[i] = items[i].it;
    hvp_batch_free(plan);
    cudaError_t e;
    if ((e = cudaMalloc(&plan->d_args, sizeof(TmaArgs) * nwin)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&plan->d_items, sizeof(BatchItem) * its.size())) != cudaSuccess) return e;
    if ((e = cudaMalloc(&plan->d_counter, sizeof(int))) != cudaSuccess) return e;
    if ((e = cudaMemcpy(plan->d_args, args.data(), sizeof(TmaArgs) * nwin, cudaMemcpyHostToDevice)) != cudaSuccess)
        return e;
    if ((e = cudaMemcpy(plan->d_items, its.data(), sizeof(BatchItem) * its.size(), cudaMemcpyHostToDevice)) !=
        cudaSuccess)
        return e;
    // a copy from pageable memory may still be in flight when cudaMemcpy returns, and the batch
    // kernel runs on streams that do not wait for the legacy stream: finish it here
    if ((e = cudaDeviceSynchronize()) != cudaSuccess) return e;
    static SmemLimit limit;
    if ((e = limit.raise((const void *)l96_hvp_batch_kernel<kThreads>, smem)) != cudaSuccess) return e;
    plan->nwin = nwin;
    plan->nitems = (int)its.size();
    plan->nthr = kThreads;
    plan->smem = smem;
    plan->grid = plan->nitems < num_sms() ? plan->nitems : num_sms();
    plan->P_cap = P_cap;
    plan->S = S_req;
    return cudaSuccess;
}

cudaError_t hvp_batch_launch(const HvpBatchPlan &plan, cudaStream_t s)
{
    if (plan.nitems == 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(plan.d_counter, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    count_launch();
    l96_hvp_batch_kernel<512><<<plan.grid, plan.nthr, plan.smem, s>>>(
        (const TmaArgs *)plan.d_args, (const BatchItem *)plan.d_items, plan.nitems, plan.d_counter);
    return cudaGetLastError();
}

}  // namespace riot
