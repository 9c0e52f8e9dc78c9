// Learned sketch proposal: a periodic 1-D conv-net maps snapshots of a
// Lorenz-96 background trajectory to m proposed sketch directions.  Forward
// (FP32, or BF16-rounded weights and activations with FP32 accumulation for
// inference), backward, the subspace loss and Adam, all as kernels here; the
// Gaussian sketch of Algorithm 3 stays the fallback (riot_rsvd_proposal).
//
// Layout: activations [B][C][n] (FP32), parameters one flat FP32 vector, per
// layer W[C_out][C_in][K] then b[C_out].  conv(x)[o][i] = b[o] +
// sum_c sum_d W[o][c][d] x[c][(i + d - h) mod n], h = K / 2.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>

#include "internal.h"

namespace riot {

namespace {

__device__ __forceinline__ float bf16r(float v) { return __bfloat162float(__float2bfloat16(v)); }

// Convolutions, forward and data gradient, as one tiled kernel.
//   forward: out[b][o][i] = act(bias[o] + sum_c sum_d W[o][c][d] in[b][c][(i + d - h) mod n])
//   data gradient (BWD): out[b][c][j] = (sum_o sum_d W[o][c][d] in[b][o][(j - d + h) mod n]) (1 - act^2)
// A CTA forms 64 output channels x 128 positions, a warp 8 channels, a lane 4 neighbouring
// positions of each: per input channel and tap 32 FMAs on 8 weights (two 16-byte broadcasts) and
// on a register window of the input row.  Input rows and weights pass through shared memory 8
// channels at a time.  Bound: FP32 FMA (33 of 78 TFLOP/s backward).  The sums run over input
// channels, then taps, as a plain loop's do.  n = 4096, batch 8, 8 - 64 - 64 - 64 - 128 channels, 5
// taps: forward 1.40 -> 0.27 ms, backward 1.20 -> 0.24 ms (one position per thread and every weight
// a global load -> this).
// NARROW: warps without output channels only load, and a last chunk ends with the input channels.
// For at most 32 output channels (half of the warps) or fewer than 8 inputs: forward of width 1
// at n = 4096, batch 8: 41 -> 27 us, of width 32 109 -> 96; of width 64, where nothing is saved, the run-time
// bound would cost 197 -> 214.
constexpr int kConvO = 64, kConvI = 128, kConvC = 8;

template <int K, bool TANH, bool BF16, bool BWD, bool NARROW>
__global__ void __launch_bounds__(256) conv_kernel(const float *in, int ci, const float *W, const float *bias,
                                                   const float *act, float *out, int co, int n)
{
    constexpr int h = K / 2, XW = kConvI + 8;
    __shared__ __align__(16) float xs[kConvC][XW];
    __shared__ __align__(16) float ws[kConvC][K][kConvO];
    const int tid = threadIdx.x, lane = tid & 31, og = (tid >> 5) * 8;
    const int i0 = blockIdx.x * kConvI, o0 = blockIdx.y * kConvO, b = blockIdx.z;
    float acc[8][4];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int o = o0 + og + q;
        float v = (!BWD && o < co) ? bias[o] : 0.f;
        if (BF16) v = bf16r(v);
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[q][p] = v;
    }
    const float *xb = in + (size_t)b * ci * n;
    for (int c0 = 0; c0 < ci; c0 += kConvC) {
        for (int t = tid; t < kConvC * (kConvI + K - 1); t += 256) {
            const int c = t / (kConvI + K - 1), x = t - c * (kConvI + K - 1);
            int j = (i0 + x - h) % n;
            j += (j < 0) ? n : 0;
            float v = (c0 + c < ci) ? xb[(size_t)(c0 + c) * n + j] : 0.f;
            if (BF16) v = bf16r(v);
            xs[c][x] = v;
        }
        for (int t = tid; t < kConvC * K * kConvO; t += 256) {
            int c, d, o;
            if (BWD) {   // W[c0 + c][o0 + o][d]: taps of one output channel are contiguous
                d = t % K;
                o = (t / K) % kConvO;
                c = t / (K * kConvO);
            } else {     // W[o0 + o][c0 + c][d]: taps of the chunk's channels are
                d = t % K;
                c = (t / K) % kConvC;
                o = t / (K * kConvC);
            }
            float v = 0.f;
            if (c0 + c < ci && o0 + o < co)
                v = W[(BWD ? (size_t)(c0 + c) * co + o0 + o : (size_t)(o0 + o) * ci + c0 + c) * K + d];
            if (BF16) v = bf16r(v);
            ws[c][d][o] = v;
        }
        __syncthreads();
        const int nc = !NARROW ? kConvC : o0 + og < co ? min(kConvC, ci - c0) : 0;
#pragma unroll 2
        for (int c = 0; c < nc; ++c) {
            constexpr int NX = (4 + K - 1 + 3) / 4;
            float x[4 * NX];
#pragma unroll
            for (int v = 0; v < NX; ++v) {
                const float4 f = *reinterpret_cast<const float4 *>(&xs[c][4 * lane + 4 * v]);
                x[4 * v] = f.x;
                x[4 * v + 1] = f.y;
                x[4 * v + 2] = f.z;
                x[4 * v + 3] = f.w;
            }
#pragma unroll
            for (int d = 0; d < K; ++d) {
                const float4 w0 = *reinterpret_cast<const float4 *>(&ws[c][d][og]);
                const float4 w1 = *reinterpret_cast<const float4 *>(&ws[c][d][og + 4]);
                const float w[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
#pragma unroll
                for (int q = 0; q < 8; ++q)
#pragma unroll
                    for (int p = 0; p < 4; ++p) acc[q][p] = fmaf(w[q], x[p + (BWD ? K - 1 - d : d)], acc[q][p]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int o = o0 + og + q;
        if (o >= co) continue;
        const size_t at = ((size_t)b * co + o) * n + i0 + 4 * lane;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            if (i0 + 4 * lane + p >= n) continue;
            float v = acc[q][p];
            if (BWD) {
                const float a = act[at + p];
                v *= 1.f - a * a;
            } else {
                if (TANH) v = tanhf(v);
                if (BF16) v = bf16r(v);
            }
            out[at + p] = v;
        }
    }
}

template <bool TANH, bool BF16, bool BWD>
cudaError_t conv(const float *in, int ci, const float *W, const float *bias, const float *act, float *out, int co, int n,
                 int K, int B, cudaStream_t s)
{
    const dim3 grid((n + kConvI - 1) / kConvI, (co + kConvO - 1) / kConvO, B);
    count_launch();
    const bool narrow = co <= kConvO / 2 || ci < kConvC;
    auto launch = [&](auto wide, auto small) { (narrow ? small : wide)<<<grid, 256, 0, s>>>(in, ci, W, bias, act, out, co, n); };
    if (K == 1) launch(conv_kernel<1, TANH, BF16, BWD, false>, conv_kernel<1, TANH, BF16, BWD, true>);
    else if (K == 3) launch(conv_kernel<3, TANH, BF16, BWD, false>, conv_kernel<3, TANH, BF16, BWD, true>);
    else if (K == 5) launch(conv_kernel<5, TANH, BF16, BWD, false>, conv_kernel<5, TANH, BF16, BWD, true>);
    else launch(conv_kernel<7, TANH, BF16, BWD, false>, conv_kernel<7, TANH, BF16, BWD, true>);
    return cudaGetLastError();
}

// Weight gradient: gW[o][c][d] = sum_b sum_i gout[b][o][i] in[b][c][(i + d - h) mod n], gb[o] =
// sum gout, to the accuracy of sums in 64 bits.  FP64 is 1/64 of the FP32 rate here, so each sum
// is a compensated FP32 one, the dot product in twice the working precision of Ogita, Rump and
// Oishi 2005 (Dot2): 10 FP32 operations a term, packed for two outputs, against 64 issue slots.  A
// warp owns 4 output channels x 1 input channel x K taps, lanes run over positions; 20 sums (K = 5)
// share 9 loads.  Slots' sums are then added in FP64.  A sum that is not finite (a product may
// leave the FP32 range) or so small that the rounding errors of its products may be below that
// range is formed again in FP64.
// Bound: the FP32 pipe (70 to 72 % active; unpacked operations were bound by issue at 77 %, 2.20 ms a
// training batch against 2.07), 16 warps an SM with the loads of 4 positions in flight (24 warps with
// 2: 2.23 ms).  n = 4096, batch 8, 8 - 64 - 64 - 64 - 128 channels: FP64 sums 12.2 ms, this 1.13 ms,
// the same gradient error (6.8e-7, that of the FP32 factors).  Fast2Sum without its ordering, 4 operations a term, took
// 0.93 ms and was off by 6 % where a lane's terms cancel to 2^-21.
constexpr int kGradO = 4;

// s + g x, what its product and its sum lose added to c.  Both losses are exact whatever the sizes of
// s and g x (products above 2^-102): where terms cancel, the sum is smaller than a term.
struct Two {
    float s, c;
};
__device__ __forceinline__ float sum2(float &s, float p)   // the loss of s += p
{
    const float t = __fadd_rn(s, p), z = __fsub_rn(t, s);
    const float lost = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));
    s = t;
    return lost;
}
// The same of two sums side by side, in packed instructions: s + g x, ng = -g.
using pair_t = unsigned long long;
struct Two2 {
    pair_t s, c;
};
__device__ __forceinline__ pair_t pk(float x, float y)
{
    pair_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 upk(pair_t p)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(p));
    return r;
}
__device__ __forceinline__ pair_t add_pair(pair_t a, pair_t b)
{
    pair_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ pair_t sub_pair(pair_t a, pair_t b)
{
    pair_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ void dot2(pair_t g, pair_t ng, pair_t x, Two2 &v)
{
    pair_t p, low;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(p) : "l"(g), "l"(x));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(low) : "l"(ng), "l"(x), "l"(p));   // what p has too much
    const pair_t t = add_pair(v.s, p), z = sub_pair(t, v.s);
    const pair_t lost = add_pair(sub_pair(v.s, sub_pair(t, z)), sub_pair(p, z));
    v.c = add_pair(v.c, sub_pair(lost, low));
    v.s = t;
}
__device__ __forceinline__ Two added(Two a, Two b)
{
    const float lost = sum2(a.s, b.s);
    return {a.s, __fadd_rn(__fadd_rn(a.c, b.c), lost)};
}
__device__ __forceinline__ double added(double a, double b) { return a + b; }
__device__ __forceinline__ double across(double v, int off) { return __shfl_xor_sync(0xffffffffu, v, off); }
__device__ __forceinline__ Two across(Two v, int off)
{
    return {__shfl_xor_sync(0xffffffffu, v.s, off), __shfl_xor_sync(0xffffffffu, v.c, off)};
}

// Sums over the lanes, lane j ending with sum j: each exchange halves the sums a lane carries.
template <int NV, typename T>
__device__ __forceinline__ T lane_sums(T (&v)[NV])
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const bool up = threadIdx.x & off;
#pragma unroll
        for (int j = 0; j < off && j < NV; ++j) {
            if (j + off < NV) {
                const T lo = v[j], hi = v[j + off < NV ? j + off : 0];
                v[j] = added(up ? hi : lo, across(up ? lo : hi, off));
            } else {
                v[j] = added(v[j], across(v[j], off));
            }
        }
    }
    return v[0];
}

// A warp's sum of fewer than 2^20 terms above this lost less than 2^-30 of itself to products whose
// rounding error is below the smallest FP32 number.
constexpr double kTinySum = 7.8886e-31;   // 2^-100

// What one warp adds up: positions lo, lo + 1, .. of the units (window, range) of its slot.
struct GradWork {
    const float *gout, *in;
    int co, ci, n, B, csplit, o0, c;
};

template <int K, typename F>
__device__ __forceinline__ void wgrad_sweep(const GradWork &a, F add)
{
    constexpr int h = K / 2, kGradU = K <= 5 ? 4 : 2;   // positions whose loads are in flight together
    const int lane = threadIdx.x & 31, n = a.n;
    const int len = ((n + a.csplit - 1) / a.csplit + 31) / 32 * 32;   // positions of a unit
    for (int u = blockIdx.z; u < a.B * a.csplit; u += gridDim.z) {
        const int b = u / a.csplit, lo = (u - b * a.csplit) * len, hi = min(n, lo + len);
        const float *x = a.in + ((size_t)b * a.ci + a.c) * n;
        const float *g = a.gout + ((size_t)b * a.co + a.o0) * n;
        for (int ib = lo; ib < hi; ib += 32 * kGradU) {
            // all loads of kGradU positions first; beyond the unit zeros
            float gv[kGradU][kGradO], xv[kGradU][K];
            const bool inside = ib >= h && ib + 32 * kGradU + h <= min(n, hi + h);   // no wrap, no end
#pragma unroll
            for (int t = 0; t < kGradU; ++t) {
                const int i = ib + 32 * t + lane;
                if (inside) {
#pragma unroll
                    for (int q = 0; q < kGradO; ++q) gv[t][q] = a.o0 + q < a.co ? g[(size_t)q * n + i] : 0.f;
#pragma unroll
                    for (int d = 0; d < K; ++d) xv[t][d] = x[i + d - h];
                } else {
#pragma unroll
                    for (int q = 0; q < kGradO; ++q) gv[t][q] = i < hi && a.o0 + q < a.co ? g[(size_t)q * n + i] : 0.f;
#pragma unroll
                    for (int d = 0; d < K; ++d) {
                        int j = i + d - h;
                        j += (j < 0) ? n : 0;
                        j -= (j >= n) ? n : 0;
                        xv[t][d] = i < hi ? x[j] : 0.f;
                    }
                }
            }
#pragma unroll
            for (int t = 0; t < kGradU; ++t) add(gv[t], xv[t]);
        }
    }
}

template <int K>
__global__ void __launch_bounds__(256, 2) conv_wgrad_kernel(const float *gout, int co, const float *in, int ci, int n,
                                                            int B, int csplit, double *part)
{
    constexpr int NV = kGradO * K;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int o0 = (blockIdx.x * 2 + (wp >> 2)) * kGradO, c = blockIdx.y * 4 + (wp & 3);
    if (o0 >= co || c >= ci) return;
    const GradWork a = {gout, in, co, ci, n, B, csplit, o0, c};
    const int q = lane / K, d = lane - q * K;
    const bool mine = lane < NV && o0 + q < co;
    double v = 0.0, vb[kGradO];   // sum `lane` of the weights, the sums of the biases
    for (bool again = false;; again = true) {
        if (!again) {
            Two u[NV], ub[kGradO];
            Two2 w[kGradO / 2][K];
#pragma unroll
            for (int r = 0; r < kGradO / 2; ++r)
#pragma unroll
                for (int j = 0; j < K; ++j) w[r][j] = {0, 0};
#pragma unroll
            for (int r = 0; r < kGradO; ++r) ub[r] = {0.f, 0.f};
            wgrad_sweep<K>(a, [&](const float(&g)[kGradO], const float(&x)[K]) {
#pragma unroll
                for (int r = 0; r < kGradO / 2; ++r) {
                    const pair_t gp = pk(g[2 * r], g[2 * r + 1]), ng = pk(-g[2 * r], -g[2 * r + 1]);
#pragma unroll
                    for (int j = 0; j < K; ++j) dot2(gp, ng, pk(x[j], x[j]), w[r][j]);
                }
                if (c == 0)
#pragma unroll
                    for (int r = 0; r < kGradO; ++r) ub[r].c = __fadd_rn(ub[r].c, sum2(ub[r].s, g[r]));
            });
#pragma unroll
            for (int r = 0; r < kGradO / 2; ++r)
#pragma unroll
                for (int j = 0; j < K; ++j) {
                    const float2 s2 = upk(w[r][j].s), c2 = upk(w[r][j].c);
                    u[2 * r * K + j] = {s2.x, c2.x};
                    u[(2 * r + 1) * K + j] = {s2.y, c2.y};
                }
            const Two t = lane_sums<NV>(u);
            v = (double)t.s + (double)t.c;
            if (c == 0)
#pragma unroll
                for (int r = 0; r < kGradO; ++r) {
                    for (int off = 16; off > 0; off >>= 1) ub[r] = added(ub[r], across(ub[r], off));
                    vb[r] = (double)ub[r].s + (double)ub[r].c;
                }
        } else {
            double u[NV];
#pragma unroll
            for (int j = 0; j < NV; ++j) u[j] = 0.0;
#pragma unroll
            for (int r = 0; r < kGradO; ++r) vb[r] = 0.0;
            wgrad_sweep<K>(a, [&](const float(&g)[kGradO], const float(&x)[K]) {
#pragma unroll
                for (int r = 0; r < kGradO; ++r) {
#pragma unroll
                    for (int j = 0; j < K; ++j) u[r * K + j] = fma((double)g[r], (double)x[j], u[r * K + j]);
                    vb[r] += g[r];
                }
            });
            v = lane_sums<NV>(u);
            if (c == 0)
#pragma unroll
                for (int r = 0; r < kGradO; ++r)
                    for (int off = 16; off > 0; off >>= 1) vb[r] += across(vb[r], off);
        }
        if (again) break;
        bool bad = mine && !isfinite(v);
        if (c == 0)
#pragma unroll
            for (int r = 0; r < kGradO; ++r) bad |= !isfinite(vb[r]);
        if (__any_sync(0xffffffffu, bad)) continue;
        if (!__any_sync(0xffffffffu, mine && fabs(v) < kTinySum)) break;
        // tiny sums of zeros are right: does one have factors?
        unsigned gs = 0, xs = 0;   // bit r: gradient of output r, bit 0: input
        wgrad_sweep<K>(a, [&](const float(&g)[kGradO], const float(&x)[K]) {
#pragma unroll
            for (int r = 0; r < kGradO; ++r) gs |= (g[r] != 0.f) << r;
#pragma unroll
            for (int j = 0; j < K; ++j) xs |= x[j] != 0.f;
        });
        gs = __reduce_or_sync(0xffffffffu, gs);
        xs = __reduce_or_sync(0xffffffffu, xs);
        if (!xs || !__any_sync(0xffffffffu, mine && fabs(v) < kTinySum && ((gs >> q) & 1))) break;
    }
    double *out = part + (size_t)blockIdx.z * ((size_t)co * ci * K + co);
    if (mine) out[((size_t)(o0 + q) * ci + c) * K + d] = v;
    if (c == 0)
#pragma unroll
        for (int r = 0; r < kGradO; ++r)
            if (lane == 0 && o0 + r < co) out[(size_t)co * ci * K + o0 + r] = vb[r];
}

__global__ void wgrad_sum_kernel(const double *part, int slots, size_t count, float *grad)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    double v = 0.0;
    for (int t = 0; t < slots; ++t) v += part[(size_t)t * count + i];
    grad[i] = (float)v;
}

// Partial sums of one layer's weight gradient: enough slots for about 8 warps per sub-partition.
int wgrad_slots(int co, int ci)
{
    const int warps = (co + kGradO - 1) / kGradO * ci;
    const int slots = (4864 + warps - 1) / warps;
    return slots < 8 ? 8 : slots > 64 ? 64 : slots;
}

cudaError_t conv_wgrad(const float *gout, int co, const float *in, int ci, int n, int K, int B, double *part, float *grad,
                       cudaStream_t s)
{
    int slots = wgrad_slots(co, ci);
    int csplit = (slots + B - 1) / B;   // units of a window
    if (csplit > (n + 127) / 128) csplit = (n + 127) / 128;
    if (slots > B * csplit) slots = B * csplit;
    const dim3 grid((co + 2 * kGradO - 1) / (2 * kGradO), (ci + 3) / 4, slots);
    count_launch();
    if (K == 1) conv_wgrad_kernel<1><<<grid, 256, 0, s>>>(gout, co, in, ci, n, B, csplit, part);
    else if (K == 3) conv_wgrad_kernel<3><<<grid, 256, 0, s>>>(gout, co, in, ci, n, B, csplit, part);
    else if (K == 5) conv_wgrad_kernel<5><<<grid, 256, 0, s>>>(gout, co, in, ci, n, B, csplit, part);
    else conv_wgrad_kernel<7><<<grid, 256, 0, s>>>(gout, co, in, ci, n, B, csplit, part);
    cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    const size_t count = (size_t)co * ci * K + co;   // weights then biases, as in the parameter vector
    count_launch();
    wgrad_sum_kernel<<<(unsigned)((count + 255) / 256), 256, 0, s>>>(part, slots, count, grad);
    return cudaGetLastError();
}

// out[0] += sum x^2 (double accumulation), for the loss normalisers
__global__ void sumsq_kernel(const float *x, size_t n, double *out)
{
    double s = 0.0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const double v = x[i];
        s += v * v;
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if ((threadIdx.x & 31) == 0 && s != 0.0) atomicAdd(out, s);
}

// The same for every window's R and X: sc[4 b] += ||R_b||^2, sc[4 b + 1] += ||X_b||^2
__global__ void sumsq2_kernel(const float *R, const float *X, size_t nm, double *sc)
{
    const float *x = (blockIdx.z ? X : R) + (size_t)blockIdx.y * nm;
    double s = 0.0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nm; i += (size_t)gridDim.x * blockDim.x) {
        const double v = x[i];
        s += v * v;
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if ((threadIdx.x & 31) == 0 && s != 0.0) atomicAdd(sc + 4 * blockIdx.y + blockIdx.z, s);
}

// FP32 products of the loss for all windows in one launch, 64 x 64 tiles of a column-major
// result, 4 x 4 outputs per thread.  Per window b, with X_b n x m and U_b n x r:
//   KIND 0: [U^T X; X^T X] ((r + m) x m), rows of the result from U, then X; the n terms of a sum
//           split over `splits` CTAs (partial results at part, added by inner_sum_kernel), since
//           a window has only a few tiles
//   KIND 1: R = X - U T (n x m), T = U^T X
//   KIND 2: gX = c1 R + c2 X + c3 X E (n x m; R is read from the place gX goes to), the loss
//           gradient with the window's scalars
// Launched window by window they took 6.0 ms at n = 4096, r = m = 128, batch 8 (4 CTAs for a 128
// x 128 product of 4096 terms), together 0.39 ms.
struct LossArgs {
    const float *U, *X, *T, *E;
    float *R, *part;
    const double *sc;
    int n, m, r, B, splits;
    double mu;
    int tld;      // leading dimension of T and of the inner products: r + m
};

template <int KIND>
__global__ void __launch_bounds__(256) loss_gemm_kernel(const LossArgs a)
{
    __shared__ __align__(16) float As[16][64];
    __shared__ __align__(16) float Bs[16][64];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int n = a.n, m = a.m, r = a.r, b = KIND == 0 ? blockIdx.z / a.splits : blockIdx.z;
    const int m0 = blockIdx.x * 64, n0 = blockIdx.y * 64;
    const float *X = a.X + (size_t)b * n * m, *U = a.U + (size_t)b * n * r;
    const float *T = KIND == 1 ? a.T + (size_t)b * a.tld * m : KIND == 2 ? a.E + (size_t)b * m * m : nullptr;
    const int K = KIND == 0 ? n : KIND == 1 ? r : m, rows = KIND == 0 ? r + m : n;
    const int chunk = KIND == 0 ? ((K + a.splits - 1) / a.splits + 15) / 16 * 16 : K;
    const int klo = KIND == 0 ? (int)(blockIdx.z % a.splits) * chunk : 0, khi = min(K, klo + chunk);
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    for (int k0 = klo; k0 < khi; k0 += 16) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int idx = tid + 256 * q;
            float va = 0.f, vb = 0.f;
            if (KIND == 0) {
                const int kk = idx & 15, i = idx >> 4, row = m0 + i;
                if (row < rows && k0 + kk < khi) va = row < r ? U[(size_t)row * n + k0 + kk] : X[(size_t)(row - r) * n + k0 + kk];
                if (n0 + i < m && k0 + kk < khi) vb = X[(size_t)(n0 + i) * n + k0 + kk];
                As[kk][i] = va;
                Bs[kk][i] = vb;
            } else {
                const int i = idx & 63, kk = idx >> 6;
                if (m0 + i < n && k0 + kk < K) va = (KIND == 1 ? U : X)[(size_t)(k0 + kk) * n + m0 + i];
                As[kk][i] = va;
                const int k2 = idx & 15, j = idx >> 4;
                if (n0 + j < m && k0 + k2 < K) vb = T[(size_t)(n0 + j) * (KIND == 1 ? a.tld : m) + k0 + k2];
                Bs[k2][j] = vb;
            }
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            const float4 a4 = *reinterpret_cast<const float4 *>(&As[kk][tx * 4]);
            const float4 b4 = *reinterpret_cast<const float4 *>(&Bs[kk][ty * 4]);
            const float av[4] = {a4.x, a4.y, a4.z, a4.w}, bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
        __syncthreads();
    }
    double c1 = 0, c2 = 0, c3 = 0;
    if (KIND == 2) {
        const double *sc = a.sc + 4 * b;
        const double bb = sc[1], L1 = sc[0] / bb, sn = bb / m;
        const double k2 = 4.0 / ((double)m * m * sn);
        c1 = 2.0 / bb / a.B;
        c2 = (-2.0 * L1 / bb - a.mu * k2 * sc[3] / m) / a.B;
        c3 = a.mu * k2 / a.B;
    }
    float *out = KIND == 0 ? a.part + (size_t)blockIdx.z * rows * m : a.R + (size_t)b * n * m;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int row = m0 + tx * 4 + i, col = n0 + ty * 4 + j;
            if (row >= rows || col >= m) continue;
            const size_t at = (size_t)col * rows + row;
            if (KIND == 0) out[at] = acc[i][j];
            if (KIND == 1) out[at] = X[at] - acc[i][j];
            if (KIND == 2) out[at] = (float)(c1 * out[at] + c2 * X[at] + c3 * acc[i][j]);
        }
}

// inner[b] = sum of the partial products of window b ((r + m) x m)
__global__ void inner_sum_kernel(const float *part, int splits, size_t count, float *inner)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x, b = blockIdx.y;
    if (i >= count) return;
    float v = 0.f;
    for (int t = 0; t < splits; ++t) v += part[(b * splits + t) * count + i];
    inner[b * count + i] = v;
}

// E = S - I with S = X^T X / s, s = ||X||^2 / m, and sc[2] += ||E||^2, sc[3] += tr(E S), per window
__global__ void __launch_bounds__(256) gram_to_e_kernel(const float *inner, int r, int m, double *scs, float *Es)
{
    const int b = blockIdx.y;
    double *sc = scs + 4 * b;
    const float *G = inner + (size_t)b * (r + m) * m;
    float *E = Es + (size_t)b * m * m;
    const double inv = m / sc[1];
    double e2 = 0.0, tr = 0.0;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < m * m; t += gridDim.x * blockDim.x) {
        const int i = t % m, j = t / m;
        const double S = (double)G[(size_t)j * (r + m) + r + i] * inv;
        const double e = S - (i == j ? 1.0 : 0.0);
        E[t] = (float)e;
        e2 += e * e;
        tr += e * S;
    }
    for (int off = 16; off > 0; off >>= 1) {
        e2 += __shfl_xor_sync(0xffffffffu, e2, off);
        tr += __shfl_xor_sync(0xffffffffu, tr, off);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(sc + 2, e2);
        atomicAdd(sc + 3, tr);
    }
}

// loss = mean over the windows of L1 + mu L2
__global__ void loss_sum_kernel(const double *sc, int m, int B, double mu, double *loss)
{
    double v = 0.0;
    for (int b = threadIdx.x; b < B; b += 32) v += (sc[4 * b] / sc[4 * b + 1] + mu * (sc[4 * b + 2] / ((double)m * m))) / B;
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if (threadIdx.x == 0) *loss = v;
}

// CTAs that share the n terms of the inner products: about two per SM, 8 at most
int inner_splits(int n, int m, int r, int B)
{
    const long long tiles = (long long)((r + m + 63) / 64) * ((m + 63) / 64) * B;
    long long sp = 304 / (tiles > 0 ? tiles : 1);
    if (sp > 8) sp = 8;
    if (sp > (n + 63) / 64) sp = (n + 63) / 64;
    return sp < 1 ? 1 : (int)sp;
}

__global__ void adam_kernel(float *p, const float *g, float *m, float *v, int64_t n, float lr, float b1, float b2,
                            float eps, float c1, float c2)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// x[c][i] = traj[floor(c T / C)][i] (FP32), and the mean / sum of squares into st[0..1]
__global__ void snapshot_kernel(const double *traj, int T, int64_t n, int C, float *x, double *st)
{
    double s = 0.0, s2 = 0.0;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * C; t += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(t / n);
        const int64_t i = t - (int64_t)c * n;
        const int step = (int)(((int64_t)c * T) / C);
        const double v = traj[(int64_t)step * n + i];
        x[t] = (float)v;
        s += v;
        s2 += v * v;
    }
    for (int off = 16; off > 0; off >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, off);
        s2 += __shfl_xor_sync(0xffffffffu, s2, off);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&st[0], s);
        atomicAdd(&st[1], s2);
    }
}

__global__ void standardise_kernel(const double *traj, int T, int64_t n, int C, float *x, const double *st)
{
    const double N = (double)n * C;
    const double mean = st[0] / N;
    const double var = st[1] / N - mean * mean;
    const double inv = var > 0.0 ? 1.0 / sqrt(var) : 1.0;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * C; t += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(t / n);
        const int64_t i = t - (int64_t)c * n;
        const int step = (int)(((int64_t)c * T) / C);
        x[t] = (float)((traj[(int64_t)step * n + i] - mean) * inv);
    }
}

inline unsigned blocks_for(size_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// ---------------------------------------------------------------------------
int64_t SketchNet::num_params() const
{
    int64_t tot = 0;
    for (int l = 0; l < depth; ++l) tot += (int64_t)chan[l + 1] * chan[l] * K + chan[l + 1];
    return tot;
}

int64_t SketchNet::w_offset(int l) const
{
    int64_t o = 0;
    for (int j = 0; j < l; ++j) o += (int64_t)chan[j + 1] * chan[j] * K + chan[j + 1];
    return o;
}

size_t sketchnet_gpart_doubles(const SketchNet &net)
{
    size_t most = 0;
    for (int l = 0; l < net.depth; ++l) {
        const size_t ci = net.chan[l], co = net.chan[l + 1], c = wgrad_slots((int)co, (int)ci) * (co * ci * net.K + co);
        if (c > most) most = c;
    }
    return most;
}

// inner products are split over CTAs only while tiles * splits <= 304
size_t sketchnet_part_floats() { return (size_t)304 * 64 * 64; }

// windows whose inner products are held at once (64 MB, at least one)
int sketchnet_group(int m, int r, int B)
{
    const size_t g = ((size_t)64 << 20) / (sizeof(float) * ((size_t)r + 2 * m) * m);
    return g < 1 ? 1 : g < (size_t)B ? (int)g : B;
}

cudaError_t sketchnet_forward(const SketchNet &net, const float *params, const float *x, int n, int B, float *Z,
                              bool bf16, float *acts, cudaStream_t s)
{
    // acts: (depth - 1) hidden layers of B * width * n floats, or nullptr to use ping-pong scratch
    const float *in = x;
    for (int l = 0; l < net.depth; ++l) {
        const int ci = net.chan[l], co = net.chan[l + 1];
        const float *W = params + net.w_offset(l);
        const float *bias = W + (size_t)co * ci * net.K;
        float *out = (l == net.depth - 1) ? Z : acts + (size_t)l * B * net.width * n;
        const bool tanh_act = l < net.depth - 1;
        const cudaError_t e =
            tanh_act ? (bf16 ? conv<true, true, false>(in, ci, W, bias, nullptr, out, co, n, net.K, B, s)
                             : conv<true, false, false>(in, ci, W, bias, nullptr, out, co, n, net.K, B, s))
                     : (bf16 ? conv<false, true, false>(in, ci, W, bias, nullptr, out, co, n, net.K, B, s)
                             : conv<false, false, false>(in, ci, W, bias, nullptr, out, co, n, net.K, B, s));
        if (e != cudaSuccess) return e;
        in = out;
    }
    return cudaSuccess;
}

cudaError_t sketchnet_loss_grad(const SketchNet &net, const float *params, const float *x, const float *U, int r,
                                int n, int B, double mu, float *grad, double *loss_dev, SketchWork &w,
                                cudaStream_t s)
{
    const int m = net.m;
    cudaError_t e;
    if ((e = sketchnet_forward(net, params, x, n, B, w.Z, false, w.acts, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(w.sc, 0, sizeof(double) * 4 * B, s)) != cudaSuccess) return e;
    const size_t nm = (size_t)n * m, inner = (size_t)(r + m) * m;
    LossArgs a;
    a.T = w.inner;        // U^T X in the first r rows of the inner products
    a.E = w.E;
    a.n = n;
    a.m = m;
    a.r = r;
    a.B = B;
    a.mu = mu;
    a.tld = r + m;
    const unsigned cols = (unsigned)((m + 63) / 64);
    for (int b0 = 0; b0 < B; b0 += w.group) {
        const int g = B - b0 < w.group ? B - b0 : w.group;
        a.U = U + (size_t)b0 * n * r;
        a.X = w.Z + (size_t)b0 * nm;   // per window n x m column-major: column j = direction j
        a.R = w.gZ + (size_t)b0 * nm;
        double *sc = w.sc + 4 * b0;
        a.sc = sc;
        a.splits = inner_splits(n, m, r, g);
        a.part = a.splits > 1 ? w.part : w.inner;
        count_launch();
        loss_gemm_kernel<0><<<dim3((r + m + 63) / 64, cols, g * a.splits), 256, 0, s>>>(a);
        if (a.splits > 1) {
            count_launch();
            inner_sum_kernel<<<dim3(blocks_for(inner, 256), g), 256, 0, s>>>(w.part, a.splits, inner, w.inner);
        }
        count_launch();
        loss_gemm_kernel<1><<<dim3((n + 63) / 64, cols, g), 256, 0, s>>>(a);
        count_launch();
        sumsq2_kernel<<<dim3(64, g, 2), 256, 0, s>>>(a.R, a.X, nm, sc);
        count_launch();
        gram_to_e_kernel<<<dim3(m * m > 4096 ? 16 : 1, g), 256, 0, s>>>(w.inner, r, m, sc, w.E);
        count_launch();
        loss_gemm_kernel<2><<<dim3((n + 63) / 64, cols, g), 256, 0, s>>>(a);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    count_launch();
    loss_sum_kernel<<<1, 32, 0, s>>>(w.sc, m, B, mu, loss_dev);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // backward through the layers; gZ (B x m x n) is dL/dZ in the activation layout
    const float *g = w.gZ;
    for (int l = net.depth - 1; l >= 0; --l) {
        const int ci = net.chan[l], co = net.chan[l + 1];
        const float *W = params + net.w_offset(l);
        float *gW = grad + net.w_offset(l);
        const float *in = (l == 0) ? x : w.acts + (size_t)(l - 1) * B * net.width * n;
        if ((e = conv_wgrad(g, co, in, ci, n, net.K, B, w.gpart, gW, s)) != cudaSuccess) return e;
        if (l > 0) {
            float *gin = (g == w.g0) ? w.g1 : w.g0;
            if ((e = conv<false, false, true>(g, co, W, nullptr, in, gin, ci, n, net.K, B, s)) != cudaSuccess) return e;
            g = gin;
        }
    }
    return cudaSuccess;
}

cudaError_t sketchnet_adam(const SketchNet &net, float *params, const float *grad, float *m1, float *m2, int t,
                           float lr, cudaStream_t s)
{
    const int64_t np = net.num_params();
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = (float)(1.0 - pow(0.9, t)), c2 = (float)(1.0 - pow(0.999, t));
    count_launch();
    adam_kernel<<<blocks_for(np, 256), 256, 0, s>>>(params, grad, m1, m2, np, lr, b1, b2, 1e-8f, c1, c2);
    return cudaGetLastError();
}

cudaError_t sketchnet_input(const double *traj, int T, int64_t n, int C, float *x, double *st, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(st, 0, 2 * sizeof(double), s);
    if (e != cudaSuccess) return e;
    const unsigned grid = blocks_for((size_t)n * C, 256) < 1024 ? blocks_for((size_t)n * C, 256) : 1024;
    count_launch();
    snapshot_kernel<<<grid, 256, 0, s>>>(traj, T, n, C, x, st);
    count_launch();
    standardise_kernel<<<grid, 256, 0, s>>>(traj, T, n, C, x, st);
    return cudaGetLastError();
}

cudaError_t sumsq(const float *x, size_t n, double *out, cudaStream_t s)
{
    count_launch();
    sumsq_kernel<<<64, 256, 0, s>>>(x, n, out);
    return cudaGetLastError();
}

}  // namespace riot
