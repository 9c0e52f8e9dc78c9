// Tracer transport of the surface-emission inversion (the setting of the
// paper's black-carbon experiments, Section 3.2, on a synthetic box model):
// batched RK4 tangent-linear and adjoint steppers, trilinear observation
// gather / scatter, and the separable exponential prior square root.
//
// The upwind advection of a column reduces to five coefficients (self and the four neighbours)
// computed from the face winds and scaled per level; the adjoint uses the transposed ones, so
// the same kernels step both directions.  For a linear autonomous system the RK4 step is
// c+ = P(hA) c + h Q(hA) s, and its adjoint gives the source adjoint h Q(hA^T) lam, added at
// level 0 of the emission blocks.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include "internal.h"

namespace riot {

namespace {

constexpr int kHalo = 4;

constexpr int kMaxNZ = 32;

// FP64 stepper: one launch per RK4 stage, one cell per thread.  The stages are the nested
// (Horner) form w_{s+1} = c + a_s (A w_s + s), a = h/4, h/3, h/2, h, w_0 = c, w_4 = c+ (equal to
// the classical stages for a linear autonomous tendency; see the FP32 stepper), ten FP64
// operations a cell.  Bound: FP64 issue, one warp instruction per 64 cycles and sub-partition,
// so nothing is computed twice (a step fused in one kernel computes 3.1 times the cells on the
// 16 x 2 tiles that fit) and every cell is a thread (4.6 us of issue per stage on 96 x 96 x 30);
// the re-read fields come from L2, the column coefficients from a table.  A launch is a
// programmatic dependent of the one before, so that its start overlaps that one's end.
// Measured: riot_outer_begin of 96 x 96 x 30 and 60 steps 16.86 -> 3.78 ms (134 -> 27 us a step).
struct StageArgs {
    double amp[kMaxNZ], ku[kMaxNZ], kl[kMaxNZ], nkd[kMaxNZ];
    const double *w, *c;
    double *out;
    long long pstride;    // cells per probe
    const double *cf;     // [5][ny][nx] self, east, west, north, south
    const double *src;    // surface source of this step's block (TL), per probe at sstride
    long long sstride;
    double *ebar;         // source adjoint of this step's block (last stage of AD), per probe at estride
    long long estride;
    int nx, ny, nz;
    double al;
};

constexpr int kStageBlock = 128;

__global__ void __launch_bounds__(kStageBlock) adv_stage_kernel(const __grid_constant__ StageArgs a)
{
    const int plane = a.nx * a.ny, col = blockIdx.x * kStageBlock + threadIdx.x, z = blockIdx.y;
    if (col >= plane) {
        cudaGridDependencySynchronize();
        return;
    }
    const int y = col / a.nx, x = col - y * a.nx;
    const int cE = x + 1 == a.nx ? col + 1 - a.nx : col + 1, cW = x == 0 ? col + a.nx - 1 : col - 1;
    const int cN = y + 1 == a.ny ? col : col + a.nx, cS = y == 0 ? col : col - a.nx;   // walls: coefficient 0
    double k[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) k[i] = a.cf[(size_t)i * plane + col];
    cudaGridDependencySynchronize();
    const size_t at = (size_t)blockIdx.z * a.pstride + (size_t)z * plane;
    const double *w = a.w + at;
    const double wo = w[col], up = z + 1 < a.nz ? w[plane + col] : 0.0, dn = z > 0 ? w[col - plane] : 0.0;
    const double wE = w[cE], wW = w[cW], wN = w[cN], wS = w[cS], c = a.c[at + col];
    cudaTriggerProgrammaticLaunchCompletion();
    double q = k[0] * wo;
    q = fma(k[1], wE, q);
    q = fma(k[2], wW, q);
    q = fma(k[3], wN, q);
    q = fma(k[4], wS, q);
    q *= a.amp[z];
    q = fma(a.ku[z], up, q);
    q = fma(a.kl[z], dn, q);
    q = fma(a.nkd[z], wo, q);
    if (z == 0) {
        if (a.src) q += a.src[(size_t)blockIdx.z * a.sstride + col];
        if (a.ebar) a.ebar[(size_t)blockIdx.z * a.estride + col] += a.al * wo;   // al = h in the last stage
    }
    a.out[at + col] = fma(a.al, q, c);
}

// Column coefficients of both directions: cf[0] tangent linear, cf[1] adjoint, [5][ny][nx] each.
__global__ void adv_coef_kernel(const double *u, const double *v, int nx, int ny, double rdx, double rdy, double *cf)
{
    const int plane = nx * ny, col = blockIdx.x * blockDim.x + threadIdx.x;
    if (col >= plane) return;
    const int x = col % nx;
    const double uL = u[col], uR = u[x + 1 == nx ? col + 1 - nx : col + 1], vS = v[col], vN = v[col + nx];
    const double uLp = fmax(uL, 0.0), uLm = fmin(uL, 0.0), uRp = fmax(uR, 0.0), uRm = fmin(uR, 0.0);
    const double vSp = fmax(vS, 0.0), vSm = fmin(vS, 0.0), vNp = fmax(vN, 0.0), vNm = fmin(vN, 0.0);
    const double c0 = (uLm - uRp) * rdx + (vSm - vNp) * rdy;
    const double tl[5] = {c0, -uRm * rdx, uLp * rdx, -vNm * rdy, vSp * rdy};
    const double ad[5] = {c0, uRp * rdx, -uLm * rdx, vNp * rdy, -vSm * rdy};
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        cf[(size_t)i * plane + col] = tl[i];
        cf[(size_t)(5 + i) * plane + col] = ad[i];
    }
}

// FP32 stepper: nested RK4 marching through the levels, packed FP32x2 arithmetic.  For the
// linear autonomous tendency f(w) = A w + s of one step, RK4 gives c+ = P(hA) c + h Q(hA) s,
// P and Q the Taylor polynomials of degree 4 and 3 of exp(z) and (exp(z) - 1) / z.  Nested
// (Horner), that is w_{s+1} = c + a_s (A w_s + s) for a = h/4, h/3, h/2, h from w_0 = c, w_4 being
// c+: the same four applications of A as the classical stages, with one state array besides
// c instead of two.  The adjoint P(hA^T) lam is the same recursion with A^T and no source;
// the input of its last stage is Q(hA^T) lam, so the source adjoint is h times its level 0.
//
// A CTA of NW warps owns a region of 64 columns in x by RW NW rows in y of one probe, of which
// the inner 56 x (RW NW - 8) are its tile; a warp holds RW rows, a lane two neighbouring columns
// of each as one register pair (every operation serves both).  Iteration k computes level k - 1 - s of
// stage s for all four stages: a stage needs its input one level up (computed earlier in the
// same iteration), one level down and at the four horizontal neighbours, so three levels per
// stage stay in registers and only one level per stage is published in shared memory (a warp's
// outer rows), by one barrier per iteration.  East and west neighbours come from the lane's own
// pair and two shuffles, a row's north and south neighbours from the warp's other rows.  The
// field's levels arrive by asynchronous copies three levels ahead; its level -1 holds the
// source, which enters level 0 as the neighbour below with coefficient 1.
//
// Bound: register ports and shared memory together.  A packed FMA of three different register
// pairs takes 3 cycles of its sub-partition (2 with one of them reused, hence the order of the
// operations over a warp's rows); the 10 packed operations of a pair and stage make 80 us of the
// 192 x 192 x 30, 32-column step with the halo's recomputation (64 x 36 regions, 76 % of the rows
// and 75 % of the columns owned), the shared-memory pipe 62 % of the time.  Measured: 262 -> 176
// us per step (column form -> this, ncu), 32 columns of 240 steps 132.8 -> 89.7 ms, with the same
// error.  Slower: 16 warps of two rows (97 ms), 8 of four (98 ms), scalar east and west products
// (mixed with packed ones they stall, 103 ms), barrier before the copies (97 ms).  Coefficients
// multiplied by a_s beforehand save nothing and round the balance of the vertical fluxes (error
// 2 to 5e-7).
constexpr int kZW = 64;             // columns of a region
constexpr int kZTX = kZW - 2 * kHalo;
constexpr int kZLevels = kMaxNZ + 6;

struct StepArgsZ {
    unsigned long long al[4];                                 // h/4, h/3, h/2, h, each twice
    float amp[kMaxNZ], ku[kMaxNZ], kl[kMaxNZ], nkd[kMaxNZ];   // 0 beyond nz
    const float *cin;
    float *cout;
    long long pstride;
    const float *src;
    long long sstride;
    float *ebar;
    long long estride;
    const float *u, *v;
    int nx, ny, nz;
    float h, rdx, rdy;
};

// Upwind coefficients of one column: self, east, west, north, south (0 outside the walls).
template <bool ADJ>
__device__ __forceinline__ void column_coefs(const StepArgsZ &a, int gx, int gy, float (&cf)[5])
{
#pragma unroll
    for (int i = 0; i < 5; ++i) cf[i] = 0.f;
    if (gy < 0 || gy >= a.ny) return;
    const size_t row = (size_t)gy * a.nx, col = row + gx;
    const float uL = a.u[col], uR = a.u[row + (gx + 1 == a.nx ? 0 : gx + 1)];
    const float vS = a.v[col], vN = a.v[col + a.nx];
    const float uLp = fmaxf(uL, 0.f), uLm = fminf(uL, 0.f);
    const float uRp = fmaxf(uR, 0.f), uRm = fminf(uR, 0.f);
    const float vSp = fmaxf(vS, 0.f), vSm = fminf(vS, 0.f);
    const float vNp = fmaxf(vN, 0.f), vNm = fminf(vN, 0.f);
    cf[0] = (uLm - uRp) * a.rdx + (vSm - vNp) * a.rdy;
    cf[1] = ADJ ? uRp * a.rdx : -uRm * a.rdx;
    cf[2] = ADJ ? -uLm * a.rdx : uLp * a.rdx;
    cf[3] = ADJ ? vNp * a.rdy : -vNm * a.rdy;
    cf[4] = ADJ ? -vSm * a.rdy : vSp * a.rdy;
}

// A pair of neighbouring columns in one 64-bit register.
using pair_t = unsigned long long;

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
__device__ __forceinline__ pair_t fma2(pair_t a, pair_t b, pair_t c)
{
    pair_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ pair_t mul2(pair_t a, pair_t b)
{
    pair_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// asynchronous copy of BYTES (4 or 8) to shared memory, zeros when !in
template <int BYTES>
__device__ __forceinline__ void copy_async(void *dst, const float *src, bool in)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int n = in ? BYTES : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(src), "n"(BYTES), "r"(n) : "memory");
}

constexpr int kZRing = 6;   // levels of the field in shared memory (the unrolling, so that slots are constants)
constexpr int kZAhead = 3;  // levels copied ahead of the iteration that reads them

// PAIR: nx is even and the fields are 8-byte aligned, so that a lane's two columns are one access.
template <int NW, int RW, bool ADJ, bool PAIR>
__global__ void __launch_bounds__(32 * NW) adv_step_z_kernel(const __grid_constant__ StepArgsZ a)
{
    constexpr int ROWS = RW * NW, TY = ROWS - 2 * kHalo;
    extern __shared__ __align__(16) unsigned char advz_smem[];
    // the field's levels (also the published input of stage 0): [kZRing][ROWS][32]; published
    // inputs of stages 1..3: [2][3][ROWS][32]; level coefficients, each twice (for both columns
    // of a pair): (amp, ku), (kl, nkd) of level z at z + 3, zeros below and from level nz on
    pair_t(*F)[ROWS][32] = reinterpret_cast<pair_t(*)[ROWS][32]>(advz_smem);
    pair_t(*S)[3][ROWS][32] = reinterpret_cast<pair_t(*)[3][ROWS][32]>(F + kZRing);
    ulonglong2(*LC)[2] = reinterpret_cast<ulonglong2(*)[2]>(S + 2);
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const int x0 = blockIdx.x * kZTX, y0 = blockIdx.y * TY;
    const int ix = 2 * lane - kHalo;
    int gx0 = (x0 + ix) % nx;
    if (gx0 < 0) gx0 += nx;
    const int gx1 = gx0 + 1 == nx ? 0 : gx0 + 1;
    const int plane = nx * ny;
    const float *cin = a.cin + (size_t)blockIdx.z * a.pstride;
    const int ry0 = RW * wp, sN = min(ry0 + RW, ROWS - 1), sS = max(ry0 - 1, 0);

    bool valid[RW], mine[RW];
    int row0[RW];
#pragma unroll
    for (int r = 0; r < RW; ++r) {
        const int gy = y0 - kHalo + ry0 + r;
        valid[r] = gy >= 0 && gy < ny;
        row0[r] = valid[r] ? gy * nx : 0;
        mine[r] = valid[r] && ry0 + r >= kHalo && ry0 + r < kHalo + TY && ix >= 0 && ix < kZTX && x0 + ix < nx;
    }
    // copy of level z (slot z mod kZRing); beyond the last level zeros, from an address in range
    auto fetch = [&](int z, int slot) {
        const float *lev = cin + (size_t)min(z, nz - 1) * plane;
        const bool top = z < nz;
#pragma unroll
        for (int r = 0; r < RW; ++r) {
            float *d = reinterpret_cast<float *>(&F[slot][ry0 + r][lane]);
            copy_async<PAIR ? 8 : 4>(d, lev + (row0[r] + gx0), valid[r] && top);
            if (!PAIR) copy_async<4>(d + 1, lev + (row0[r] + gx1), valid[r] && top);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int z = 0; z < kZAhead; ++z) fetch(z, z);
    for (int i = threadIdx.x; i < kZLevels; i += 32 * NW) {
        const int z = i - 3, zz = z >= 0 && z < nz ? z : 0;
        const float f = z >= 0 && z < nz ? 1.f : 0.f;
        const float am = f * a.amp[zz], u = f * a.ku[zz], l = z == 0 ? 1.f : f * a.kl[zz], d = f * a.nkd[zz];
        LC[i][0] = make_ulonglong2(pk(am, am), pk(u, u));
        LC[i][1] = make_ulonglong2(pk(l, l), pk(d, d));
    }
    pair_t C[RW][5];   // self, east, west, north, south
    float2 e0[RW];
#pragma unroll
    for (int r = 0; r < RW; ++r) {
        const int gy = y0 - kHalo + ry0 + r;
        float c0[5], c1[5];
        column_coefs<ADJ>(a, gx0, gy, c0);
        column_coefs<ADJ>(a, gx1, gy, c1);
#pragma unroll
        for (int i = 0; i < 5; ++i) C[r][i] = pk(c0[i], c1[i]);
        e0[r] = make_float2(0.f, 0.f);
    }

    // W[s][z mod 3][r]: input of stage s at level z; c3, c4: the field three and four levels back
    pair_t W[4][3][RW], c3[RW], c4[RW];
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int r = 0; r < RW; ++r) W[s][i][r] = 0;
    // the source enters level 0 of every stage as a level -1 that holds it, with coefficient 1
    // (kl of level 0, which has no neighbour below)
    if (!ADJ && a.src)
#pragma unroll
        for (int r = 0; r < RW; ++r)
            if (valid[r]) {
                const float *sp = a.src + (size_t)blockIdx.z * a.sstride + row0[r];
                W[0][2][r] = W[1][2][r] = pk(sp[gx0], sp[gx1]);
            }
    asm volatile("cp.async.wait_group %0;" ::"n"(kZAhead - 1) : "memory");
#pragma unroll
    for (int r = 0; r < RW; ++r) {
        c3[r] = c4[r] = 0;
        W[0][0][r] = F[0][ry0 + r][lane];
    }
    float *cout = a.cout + (size_t)blockIdx.z * a.pstride;

    for (int k0 = 1; k0 < nz + 4; k0 += 6) {
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            const int k = k0 + j;        // k = j + 1 (mod 6)
            if (k >= nz + 4) break;
            pair_t(*Sk)[ROWS][32] = S[(j + 1) & 1];
            // publish level k - 1 - s of the inputs of stages 1..3
#pragma unroll
            for (int s = 1; s < 4; ++s)
#pragma unroll
                for (int r = 0; r < RW; r += RW - 1) Sk[s - 1][ry0 + r][lane] = W[s][(j + 6 - s) % 3][r];
            fetch(k + kZAhead - 1, (j + kZAhead) % kZRing);
            asm volatile("cp.async.wait_group %0;" ::"n"(kZAhead - 1) : "memory");   // level k is here
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                c4[r] = c3[r];
                c3[r] = W[0][(j + 1) % 3][r];
                W[0][(j + 1) % 3][r] = F[(j + 1) % kZRing][ry0 + r][lane];
            }
            __syncthreads();
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const int z = k - 1 - s;
                const int im = (j + 6 - s) % 3, iu = (im + 1) % 3, id = (im + 2) % 3;
                const ulonglong2 l0 = LC[z + 3][0], l1 = LC[z + 3][1];
                const pair_t al = a.al[s];
                const pair_t(*P)[32] = s == 0 ? F[j] : Sk[s > 0 ? s - 1 : 0];   // level z of stage 0: k - 1 = j (mod 6)
                const pair_t nN = P[sN][lane], nS = P[sS][lane];
                float *lev = cout + (ptrdiff_t)z * plane;
                // operations with the same coefficient next to each other: a packed operation with
                // three different register pairs takes 3 cycles, with one of them kept 2
                pair_t q[RW];
#pragma unroll
                for (int r = 0; r < RW; ++r) {
                    const pair_t wo = W[s][im][r];
                    const float2 w = upk(wo);
                    const float wE = __shfl_down_sync(0xffffffffu, w.x, 1), wW = __shfl_up_sync(0xffffffffu, w.y, 1);
                    const pair_t N = r + 1 < RW ? W[s][im][r + 1 < RW ? r + 1 : 0] : nN;
                    const pair_t So = r > 0 ? W[s][im][r > 0 ? r - 1 : 0] : nS;
                    q[r] = mul2(C[r][0], wo);
                    q[r] = fma2(C[r][1], pk(w.y, wE), q[r]);
                    q[r] = fma2(C[r][2], pk(wW, w.x), q[r]);
                    q[r] = fma2(C[r][3], N, q[r]);
                    q[r] = fma2(C[r][4], So, q[r]);
                }
#pragma unroll
                for (int r = 0; r < RW; ++r) q[r] = mul2(l0.x, q[r]);
#pragma unroll
                for (int r = 0; r < RW; ++r) q[r] = fma2(l1.y, W[s][im][r], q[r]);
#pragma unroll
                for (int r = 0; r < RW; ++r) q[r] = fma2(l1.x, W[s][id][r], q[r]);
#pragma unroll
                for (int r = 0; r < RW; ++r) q[r] = fma2(l0.y, W[s][iu][r], q[r]);
#pragma unroll
                for (int r = 0; r < RW; ++r) {
                    const pair_t wo = W[s][im][r];
                    const pair_t wn = fma2(al, q[r], s < 2 ? W[0][im][r] : s == 2 ? c3[r] : c4[r]);
                    if (s < 3) {
                        W[s + 1][im][r] = wn;   // level z (mod 3 as im)
                    } else {
                        if (ADJ && j == 3 && k0 == 1) {   // z = 0
                            const float2 e = upk(wo);
                            e0[r] = e;
                        }
                        if (mine[r] && (j >= 3 || k0 > 1)) {   // 0 <= z < nz, as 4 <= k < nz + 4
                            float *o = lev + row0[r];
                            if (PAIR) {
                                *reinterpret_cast<pair_t *>(o + gx0) = wn;
                            } else {
                                const float2 t = upk(wn);
                                o[gx0] = t.x;
                                if (x0 + ix + 1 < nx) o[gx1] = t.y;
                            }
                        }
                    }
                }
            }
        }
    }
    if (ADJ && a.ebar)
#pragma unroll
        for (int r = 0; r < RW; ++r)
            if (mine[r]) {
                float *e = a.ebar + (size_t)blockIdx.z * a.estride + row0[r];
                e[gx0] += a.h * e0[r].x;
                if (PAIR || x0 + ix + 1 < nx) e[gx1] += a.h * e0[r].y;
            }
}

// FP32 stepper for few columns of the sketch: the recursion of adv_step_z_kernel with whole
// columns of levels in registers, four barriers per step on 32 x 8 tiles: four times the CTAs
// of the level-marching form, each done in a quarter of its time.  Levels are held in pairs (2p, 2p + 1) (padded with zero coefficients beyond nz) and
// combined by packed FP32x2 instructions, one instruction for two levels; the shared planes
// hold the pairs, so a horizontal neighbour fetch is one 64-bit load for two levels.  (Pairs
// (p, p + NZP), whose vertical neighbours are whole pairs, measured slower: the renamed
// stage inputs cost registers.)  A CTA owns a TX x TY tile of one
// probe plus a halo of 4 columns on each side, each stage on a region one column narrower.
struct StepArgsF2 {
    float2 amp2[16];   // (amp of level 2p, of level 2p + 1); 0 beyond nz
    float2 ku2[16];    // Kz / dz^2 on the face above each level of the pair
    float2 kl2[16];    // on the face below
    float2 nkd2[16];   // -(ku + kl)
    const float *cin;
    float *cout;
    long long pstride;
    const float *src;
    long long sstride;
    float *ebar;
    long long estride;
    const float *u, *v;
    int nx, ny, nz;
    float h, rdx, rdy;
};

// registers per thread that still fit one CTA of `threads` on an SM (registers go to warps in
// groups of four, in steps of 8 per thread)
constexpr int regs_for(int threads)
{
    return ((65536 / ((threads + 127) / 128 * 128)) / 8 * 8) > 255 ? 255 : (65536 / ((threads + 127) / 128 * 128)) / 8 * 8;
}

template <int NZP, int TX, int TY, bool ADJ>
__global__ void __maxnreg__(regs_for((TX + 2 * kHalo) * (TY + 2 * kHalo))) adv_step_f2_kernel(StepArgsF2 a)
{
    constexpr int RX = TX + 2 * kHalo, RY = TY + 2 * kHalo, PL = RX * RY;
    extern __shared__ __align__(16) unsigned char adv2_smem[];
    float2 *S0 = reinterpret_cast<float2 *>(adv2_smem);   // [2][NZP][RY][RX]
    const int tid = threadIdx.x;
    const int rx = tid % RX, ry = tid / RX;
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    int gx = (x0 - kHalo + rx) % nx;
    if (gx < 0) gx += nx;
    const int gy = y0 - kHalo + ry;
    const bool valid = gy >= 0 && gy < ny;
    const size_t plane = (size_t)nx * ny;
    const size_t col = valid ? (size_t)gy * nx + gx : 0;
    float c0 = 0.f, cE = 0.f, cW = 0.f, cN = 0.f, cS = 0.f;
    if (valid) {
        const float uL = a.u[col], uR = a.u[(size_t)gy * nx + (gx + 1 == nx ? 0 : gx + 1)];
        const float vS = a.v[col], vN = a.v[col + nx];
        const float uLp = fmaxf(uL, 0.f), uLm = fminf(uL, 0.f);
        const float uRp = fmaxf(uR, 0.f), uRm = fminf(uR, 0.f);
        const float vSp = fmaxf(vS, 0.f), vSm = fminf(vS, 0.f);
        const float vNp = fmaxf(vN, 0.f), vNm = fminf(vN, 0.f);
        c0 = (uLm - uRp) * a.rdx + (vSm - vNp) * a.rdy;
        if (!ADJ) {
            cE = -uRm * a.rdx;
            cW = uLp * a.rdx;
            cN = -vNm * a.rdy;
            cS = vSp * a.rdy;
        } else {
            cE = uRp * a.rdx;
            cW = -uLm * a.rdx;
            cN = vNp * a.rdy;
            cS = -vSm * a.rdy;
        }
    }
    const float2 C0 = make_float2(c0, c0), CE = make_float2(cE, cE), CW = make_float2(cW, cW);
    const float2 CN = make_float2(cN, cN), CS = make_float2(cS, cS);
    const size_t pb = (size_t)blockIdx.z * a.pstride;
    cudaGridDependencySynchronize();
    float2 c[NZP], w[NZP];
#pragma unroll
    for (int p = 0; p < NZP; ++p) {
        const int z0 = 2 * p, z1 = 2 * p + 1;
        c[p].x = (valid && z0 < nz) ? a.cin[pb + z0 * plane + col] : 0.f;
        c[p].y = (valid && z1 < nz) ? a.cin[pb + z1 * plane + col] : 0.f;
        w[p] = c[p];
    }
    float s0 = 0.f;
    if (!ADJ && valid && a.src) s0 = a.src[(size_t)blockIdx.z * a.sstride + col];
    float e0 = 0.f;
#pragma unroll
    for (int st = 0; st < 4; ++st) {
        float2 *S = S0 + (st & 1) * NZP * PL;
        // the stage input on the region of this stage grown by one column; rows beyond the
        // walls publish their zeros
        if (rx >= st && rx < RX - st && ry >= st && ry < RY - st) {
#pragma unroll
            for (int p = 0; p < NZP; ++p) S[p * PL + ry * RX + rx] = w[p];
        }
        if (ADJ && st == 3) e0 = w[0].x;
        if (st == 3) cudaTriggerProgrammaticLaunchCompletion();
        __syncthreads();
        if (valid && rx > st && rx < RX - st - 1 && ry > st && ry < RY - st - 1) {
            const float al = (st == 0) ? 0.25f * a.h : (st == 1) ? a.h / 3.f : (st == 2) ? 0.5f * a.h : a.h;
            const float2 AL = make_float2(al, al);
            float below = 0.f;   // the stage input of level 2p - 1
#pragma unroll
            for (int p = 0; p < NZP; ++p) {
                const float2 wo = w[p];
                const float2 *Sp = S + p * PL + ry * RX + rx;
                float2 hor = __fmul2_rn(C0, wo);
                hor = __ffma2_rn(CE, Sp[1], hor);
                hor = __ffma2_rn(CW, Sp[-1], hor);
                hor = __ffma2_rn(CN, Sp[RX], hor);
                hor = __ffma2_rn(CS, Sp[-RX], hor);
                const float2 up = make_float2(wo.y, (p + 1 < NZP) ? w[p + 1].x : 0.f);
                const float2 dn = make_float2(below, wo.x);
                float2 k = __fmul2_rn(a.amp2[p], hor);
                k = __ffma2_rn(a.ku2[p], up, k);
                k = __ffma2_rn(a.kl2[p], dn, k);
                k = __ffma2_rn(a.nkd2[p], wo, k);
                if (!ADJ && p == 0) k.x += s0;
                w[p] = __ffma2_rn(AL, k, c[p]);
                below = wo.y;
            }
        }
    }
    const int ix = rx - kHalo, iy = ry - kHalo;
    if (valid && ix >= 0 && ix < TX && iy >= 0 && iy < TY && x0 + ix < nx) {
#pragma unroll
        for (int p = 0; p < NZP; ++p) {
            const int z0 = 2 * p, z1 = 2 * p + 1;
            if (z0 < nz) a.cout[pb + z0 * plane + col] = w[p].x;
            if (z1 < nz) a.cout[pb + z1 * plane + col] = w[p].y;
        }
        if (ADJ && a.ebar) a.ebar[(size_t)blockIdx.z * a.estride + col] += a.h * e0;
    }
}

template <typename R>
__global__ void obs_gather_kernel(const R *c, long long pstride, int o0, int no, const int *cell, const R *w,
                                  const R *rinv, R *r, long long rstride)
{
    const int o = blockIdx.x * blockDim.x + threadIdx.x, oo = o0 + (o < no ? o : 0);
    R wq[8];
    int cq[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        wq[q] = w[8 * oo + q];
        cq[q] = cell[8 * oo + q];
    }
    const R ri = rinv[oo];
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
    if (o >= no) return;
    const R *cp = c + (size_t)blockIdx.y * pstride;
    R acc = R(0);
#pragma unroll
    for (int q = 0; q < 8; ++q) acc += wq[q] * cp[cq[q]];
    r[(size_t)blockIdx.y * rstride + oo] = ri * acc;
}

__global__ void obs_innov_kernel(const double *c, int o0, int no, const int *cell, const double *w,
                                 const double *y, const double *rinv, double *d, double *jo)
{
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    double j = 0.0;
    if (o < no) {
        const int oo = o0 + o;
        double acc = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) acc += w[8 * oo + q] * c[cell[8 * oo + q]];
        const double dd = acc - y[oo];
        d[oo] = dd;
        j = 0.5 * dd * dd * rinv[oo];
    }
    for (int off = 16; off > 0; off >>= 1) j += __shfl_down_sync(0xffffffffu, j, off);
    if ((threadIdx.x & 31) == 0 && j != 0.0) atomicAdd(jo, j);
}

template <typename R>
__global__ void obs_scatter_kernel(R *lam, long long pstride, int o0, int no, const int *cell, const R *w,
                                   const R *r, long long rstride)
{
    const int o = blockIdx.x * blockDim.x + threadIdx.x, oo = o0 + (o < no ? o : 0);
    R wq[8];
    int cq[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        wq[q] = w[8 * oo + q];
        cq[q] = cell[8 * oo + q];
    }
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
    if (o >= no) return;
    R *lp = lam + (size_t)blockIdx.y * pstride;
    const R rv = r[(size_t)blockIdx.y * rstride + oo];
#pragma unroll
    for (int q = 0; q < 8; ++q) atomicAdd(&lp[cq[q]], wq[q] * rv);
}

// Batched row-major GEMM C_f = alpha A_f B_f (M x K times K x N); the batch
// index f maps to offsets (f / inner) * so + (f % inner) * si per operand.
template <typename R>
struct BGArgs {
    const R *A;
    const R *B;
    R *C;
    int M, N, K, inner;
    long long lda, ldb, ldc;
    long long aso, asi, bso, bsi, cso, csi;
    R alpha;
};

template <typename R>
__global__ void __launch_bounds__(256) bgemm_kernel(BGArgs<R> g)
{
    __shared__ R As[16][64 + 1];
    __shared__ R Bs[16][64 + 4];
    const int f = blockIdx.z;
    const R *A = g.A + (f / g.inner) * g.aso + (f % g.inner) * g.asi;
    const R *B = g.B + (f / g.inner) * g.bso + (f % g.inner) * g.bsi;
    R *C = g.C + (f / g.inner) * g.cso + (f % g.inner) * g.csi;
    const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
    const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
    R acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = R(0);
    for (int k0 = 0; k0 < g.K; k0 += 16) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int idx = tid + 256 * i;
            const int mm = idx / 16, kk = idx % 16;
            As[kk][mm] = (m0 + mm < g.M && k0 + kk < g.K) ? A[(size_t)(m0 + mm) * g.lda + k0 + kk] : R(0);
            const int kb = idx / 64, nb = idx % 64;
            Bs[kb][nb] = (k0 + kb < g.K && n0 + nb < g.N) ? B[(size_t)(k0 + kb) * g.ldb + n0 + nb] : R(0);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            R av[4], bv[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) av[i] = As[kk][ty * 4 + i];
#pragma unroll
            for (int j = 0; j < 4; ++j) bv[j] = Bs[kk][tx * 4 + j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] += av[i] * bv[j];
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int mm = m0 + ty * 4 + i;
        if (mm >= g.M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int nn = n0 + tx * 4 + j;
            if (nn < g.N) C[(size_t)mm * g.ldc + nn] = g.alpha * acc[i][j];
        }
    }
}

// The same with one output per thread on 16 x 16 tiles, for few FP64 fields: a 64 x 64 tile is 95
// us of one SM's FP64 issue at K = 96 whatever the grid, a 16 x 16 tile 6 us.
__global__ void __launch_bounds__(256) bgemm16_kernel(BGArgs<double> g)
{
    __shared__ double As[16][17], Bs[16][17];
    const int f = blockIdx.z;
    const double *A = g.A + (f / g.inner) * g.aso + (f % g.inner) * g.asi;
    const double *B = g.B + (f / g.inner) * g.bso + (f % g.inner) * g.bsi;
    double *C = g.C + (f / g.inner) * g.cso + (f % g.inner) * g.csi;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int mm = blockIdx.y * 16 + ty, nn = blockIdx.x * 16 + tx;
    double acc = 0.0;
    for (int k0 = 0; k0 < g.K; k0 += 16) {
        As[ty][tx] = (mm < g.M && k0 + tx < g.K) ? A[(size_t)mm * g.lda + k0 + tx] : 0.0;
        Bs[ty][tx] = (k0 + ty < g.K && nn < g.N) ? B[(size_t)(k0 + ty) * g.ldb + nn] : 0.0;
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) acc = fma(As[ty][kk], Bs[kk][tx], acc);
        __syncthreads();
    }
    if (mm < g.M && nn < g.N) C[(size_t)mm * g.ldc + nn] = g.alpha * acc;
}

// out[j*ldo + i] = in[j*ldi + i] * s[i] (+ add[j*lda + i])
template <typename R>
__global__ void colscale_kernel(const R *in, long long ldi, const R *s, R *out, long long ldo, int n, int ncols)
{
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t total = (size_t)n * ncols;
    if (t >= total) return;
    const int j = (int)(t / n), i = (int)(t % n);
    out[(size_t)j * ldo + i] = in[(size_t)j * ldi + i] * s[i];
}

template <typename R>
__global__ void coladd_kernel(const R *in, long long ldi, R *out, long long ldo, int n, int ncols)
{
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t total = (size_t)n * ncols;
    if (t >= total) return;
    const int j = (int)(t / n), i = (int)(t % n);
    out[(size_t)j * ldo + i] += in[(size_t)j * ldi + i];
}

__global__ void emis_scale_kernel(const double *Eb, const double *x, double rdz, int n, double *Es64, float *Es32)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double e = Eb[i] * exp(x[i]) * rdz;
    Es64[i] = e;
    if (Es32) Es32[i] = (float)e;
}

inline unsigned blocks_for(size_t n, int t) { return (unsigned)((n + t - 1) / t); }

template <typename R>
struct Tab;
template <>
struct Tab<float> {
    static const float *w(const AdvDev &m) { return m.w32; }
    static const float *rinv(const AdvDev &m) { return m.rinv32; }
    static const float *Sx(const AdvDev &m) { return m.Sx32; }
    static const float *Sy(const AdvDev &m) { return m.Sy32; }
    static const float *Es(const AdvDev &m) { return m.Es32; }
};
template <>
struct Tab<double> {
    static const double *w(const AdvDev &m) { return m.w64; }
    static const double *rinv(const AdvDev &m) { return m.rinv64; }
    static const double *Sx(const AdvDev &m) { return m.Sx64; }
    static const double *Sy(const AdvDev &m) { return m.Sy64; }
    static const double *Es(const AdvDev &m) { return m.Es64; }
};

// Small grids spend their time between kernels: a step of 37 x 23 x 11 with 16 probes and its
// observation kernel took 12 us, 6.8 us since each starts during the one before (products of 48
// steps 1.14 -> 0.65 ms).
// Launch as a programmatic dependent of the kernel before it in the stream (which it waits for
// itself, by cudaGridDependencySynchronize, before it reads or writes what that one may touch).
template <typename... P, typename... A>
cudaError_t launch_after(void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, const A &...args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    count_launch();
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <int NW, int RW, bool ADJ, bool PAIR>
cudaError_t step_z_launch(const StepArgsZ &a, int P, cudaStream_t s)
{
    constexpr int TY = RW * NW - 2 * kHalo;
    const size_t smem = sizeof(pair_t) * (kZRing + 2 * 3) * RW * NW * 32 + sizeof(ulonglong2) * 2 * kZLevels;
    auto kern = adv_step_z_kernel<NW, RW, ADJ, PAIR>;
    static SmemLimit limit;
    const cudaError_t e = limit.raise((const void *)kern, smem);
    if (e != cudaSuccess) return e;
    dim3 grid((a.nx + kZTX - 1) / kZTX, (a.ny + TY - 1) / TY, P);
    kern<<<grid, 32 * NW, smem, s>>>(a);
    count_launch();
    return cudaGetLastError();
}

template <int NZP, int TX, int TY, bool ADJ>
cudaError_t step_f2_nz(const StepArgsF2 &a, int P, cudaStream_t s)
{
    constexpr int RX = TX + 2 * kHalo, RY = TY + 2 * kHalo;
    const size_t smem = sizeof(float2) * 2 * (size_t)NZP * RX * RY;
    auto kern = adv_step_f2_kernel<NZP, TX, TY, ADJ>;
    static SmemLimit limit;
    const cudaError_t e = limit.raise((const void *)kern, smem);
    if (e != cudaSuccess) return e;
    dim3 grid((a.nx + TX - 1) / TX, (a.ny + TY - 1) / TY, P);
    return launch_after(kern, grid, RX * RY, smem, s, a);
}


cudaError_t step_f32_cols(const AdvDev &m, const float *cin, float *cout, int P, const float *src, long long sstride,
                          float *ebar, long long estride, bool adj, cudaStream_t s)
{
    StepArgsF2 a;
    const int nzp = m.nz <= 8 ? 4 : m.nz <= 16 ? 8 : m.nz <= 30 ? 15 : 16;
    for (int p = 0; p < 16; ++p) {
        const int z0 = 2 * p, z1 = 2 * p + 1;
        auto kz = [&](int l) { return (l > 0 && l < m.nz) ? (float)(m.kz_h[l] / (m.dz * m.dz)) : 0.f; };
        a.amp2[p] = make_float2(z0 < m.nz ? (float)m.amp_h[z0] : 0.f, z1 < m.nz ? (float)m.amp_h[z1] : 0.f);
        a.ku2[p] = make_float2(kz(z0 + 1), kz(z1 + 1));
        a.kl2[p] = make_float2(kz(z0), kz(z1));
        a.nkd2[p] = make_float2(-(a.ku2[p].x + a.kl2[p].x), -(a.ku2[p].y + a.kl2[p].y));
    }
    a.cin = cin;
    a.cout = cout;
    a.pstride = m.ncells;
    a.src = src;
    a.sstride = sstride;
    a.ebar = ebar;
    a.estride = estride;
    a.u = m.u32;
    a.v = m.v32;
    a.nx = m.nx;
    a.ny = m.ny;
    a.nz = m.nz;
    a.h = (float)m.dt;
    a.rdx = (float)(1.0 / m.dx);
    a.rdy = (float)(1.0 / m.dy);
    if (nzp == 4) return adj ? step_f2_nz<4, 32, 8, true>(a, P, s) : step_f2_nz<4, 32, 8, false>(a, P, s);
    if (nzp == 8) return adj ? step_f2_nz<8, 32, 8, true>(a, P, s) : step_f2_nz<8, 32, 8, false>(a, P, s);
    if (nzp == 15) return adj ? step_f2_nz<15, 32, 8, true>(a, P, s) : step_f2_nz<15, 32, 8, false>(a, P, s);
    return adj ? step_f2_nz<16, 24, 8, true>(a, P, s) : step_f2_nz<16, 24, 8, false>(a, P, s);
}

constexpr int kZWarps = 12, kZRows = 3;   // 64 x 36 regions of 384 threads with 168 registers

// FP32 steps.  Both forms take whole waves of one CTA per SM; measured per wave on the 30-level
// grid 32 us for the level-marching form (0.92 us per level and 1 us) and 8.6 us for the
// column form (0.47 us per pair of levels and 1.5 us).  192 x 192 x 30, 32 columns: 6 waves,
// 176 us, against 31 waves, 262 us; one column of it 32 against 9 us.
cudaError_t step_f32(const AdvDev &m, const float *cin, float *cout, int P, const float *src, long long sstride,
                     float *ebar, long long estride, bool adj, cudaStream_t s)
{
    constexpr int TYZ = kZWarps * kZRows - 2 * kHalo;
    const int sms = num_sms(), nzp = m.nz <= 8 ? 4 : m.nz <= 16 ? 8 : m.nz <= 30 ? 15 : 16;
    auto waves = [&](int tx, int ty) {
        return (double)(((long long)((m.nx + tx - 1) / tx) * ((m.ny + ty - 1) / ty) * P + sms - 1) / sms);
    };
    if (waves(nzp == 16 ? 24 : 32, 8) * (1.5 + 0.47 * nzp) <= waves(kZTX, TYZ) * (1.0 + 0.92 * (m.nz + 4)))
        return step_f32_cols(m, cin, cout, P, src, sstride, ebar, estride, adj, s);
    StepArgsZ a;
    for (int z = 0; z < kMaxNZ; ++z) {
        auto kz = [&](int l) { return (l > 0 && l < m.nz) ? (float)(m.kz_h[l] / (m.dz * m.dz)) : 0.f; };
        a.amp[z] = z < m.nz ? (float)m.amp_h[z] : 0.f;
        a.ku[z] = kz(z + 1);
        a.kl[z] = kz(z);
        a.nkd[z] = -(a.ku[z] + a.kl[z]);
    }
    a.cin = cin;
    a.cout = cout;
    a.pstride = m.ncells;
    a.src = src;
    a.sstride = sstride;
    a.ebar = ebar;
    a.estride = estride;
    a.u = m.u32;
    a.v = m.v32;
    a.nx = m.nx;
    a.ny = m.ny;
    a.nz = m.nz;
    a.h = (float)m.dt;
    const float al[4] = {0.25f * a.h, a.h / 3.f, 0.5f * a.h, a.h};
    for (int i = 0; i < 4; ++i) {
        uint32_t w;
        memcpy(&w, &al[i], 4);
        a.al[i] = (unsigned long long)w << 32 | w;
    }
    a.rdx = (float)(1.0 / m.dx);
    a.rdy = (float)(1.0 / m.dy);
    const bool pair = m.nx % 2 == 0 && ((uintptr_t)cin | (uintptr_t)cout) % 8 == 0;
    if (pair) return adj ? step_z_launch<kZWarps, kZRows, true, true>(a, P, s) : step_z_launch<kZWarps, kZRows, false, true>(a, P, s);
    return adj ? step_z_launch<kZWarps, kZRows, true, false>(a, P, s) : step_z_launch<kZWarps, kZRows, false, false>(a, P, s);
}

// One step of P probes in FP64: cA -> cB, cX scratch of the same size.
cudaError_t step_f64(const AdvDev &m, const double *cA, double *cB, double *cX, int P, const double *src,
                     long long sstride, double *ebar, long long estride, bool adj, cudaStream_t s)
{
    StageArgs a;
    for (int l = 0; l < kMaxNZ; ++l) {
        auto kz = [&](int f) { return (f > 0 && f < m.nz) ? m.kz_h[f] / (m.dz * m.dz) : 0.0; };
        a.amp[l] = l < m.nz ? m.amp_h[l] : 0.0;
        a.ku[l] = kz(l + 1);
        a.kl[l] = kz(l);
        a.nkd[l] = -(a.ku[l] + a.kl[l]);
    }
    a.pstride = m.ncells;
    a.cf = m.cf64 + (adj ? (size_t)5 * m.nx * m.ny : 0);
    a.src = src;
    a.sstride = sstride;
    a.estride = estride;
    a.nx = m.nx;
    a.ny = m.ny;
    a.nz = m.nz;
    a.c = cA;
    const double al[4] = {0.25 * m.dt, m.dt / 3.0, 0.5 * m.dt, m.dt};
    const double *in[4] = {cA, cX, cB, cX};
    double *out[4] = {cX, cB, cX, cB};
    const dim3 grid((m.nx * m.ny + kStageBlock - 1) / kStageBlock, m.nz, P);
    for (int st = 0; st < 4; ++st) {
        a.w = in[st];
        a.out = out[st];
        a.al = al[st];
        a.ebar = adj && st == 3 ? ebar : nullptr;
        const cudaError_t e = launch_after(adv_stage_kernel, grid, kStageBlock, 0, s, a);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename R>
cudaError_t step(const AdvDev &m, const R *cin, R *cout, R *scratch, int P, const R *src, long long sstride, R *ebar,
                 long long estride, bool adj, cudaStream_t s)
{
    if constexpr (sizeof(R) == sizeof(float)) return step_f32(m, cin, cout, P, src, sstride, ebar, estride, adj, s);
    else return step_f64(m, cin, cout, scratch, P, src, sstride, ebar, estride, adj, s);
}

// The batch workspace as two fields of P probes (and the scratch field of FP64 steps).
template <typename R>
void batch_fields(const AdvDev &m, int P, R **cA, R **cB, R **cX)
{
    const size_t cells = (size_t)P * m.ncells;
    *cA = (R *)m.fields;
    *cB = *cA + cells;
    *cX = 3 * cells * sizeof(R) <= m.fields_bytes ? *cB + cells : (R *)m.c64X;   // FP64: c64X holds one probe
}

template <typename R>
cudaError_t gather(const AdvDev &m, const R *c, int P, int t, R *r, long long rstride, cudaStream_t s)
{
    const int o0 = m.optr_h[t], no = m.optr_h[t + 1] - o0;
    if (no <= 0) return cudaSuccess;
    dim3 grid(blocks_for(no, 128), P);
    return launch_after(obs_gather_kernel<R>, grid, 128, 0, s, c, (long long)m.ncells, o0, no, m.cell, Tab<R>::w(m),
                        Tab<R>::rinv(m), r, rstride);
}

template <typename R>
cudaError_t scatter(const AdvDev &m, R *lam, int P, int t, const R *r, long long rstride, cudaStream_t s)
{
    const int o0 = m.optr_h[t], no = m.optr_h[t + 1] - o0;
    if (no <= 0) return cudaSuccess;
    dim3 grid(blocks_for(no, 128), P);
    return launch_after(obs_scatter_kernel<R>, grid, 128, 0, s, lam, (long long)m.ncells, o0, no, m.cell, Tab<R>::w(m), r,
                        rstride);
}

template <typename R>
cudaError_t bgemm(const BGArgs<R> &g, int batch, cudaStream_t s)
{
    dim3 grid((g.N + 63) / 64, (g.M + 63) / 64, batch);
    if constexpr (sizeof(R) == sizeof(double)) {
        if ((long long)grid.x * grid.y * batch < 4 * num_sms()) {
            grid = dim3((g.N + 15) / 16, (g.M + 15) / 16, batch);
            bgemm16_kernel<<<grid, 256, 0, s>>>(g);
            count_launch();
            return cudaGetLastError();
        }
    }
    bgemm_kernel<R><<<grid, 256, 0, s>>>(g);
    count_launch();
    return cudaGetLastError();
}

// out (ncols columns at ldo) = sigma_b (S_y kron S_x) in (ncols columns at ldi),
// per emission block; tmp holds ncols * n reals.  S_x, S_y are symmetric, so
// this is also L^T.
template <typename R>
cudaError_t sep_apply(const AdvDev &m, const R *in, long long ldi, R *out, long long ldo, int ncols, R *tmp,
                      cudaStream_t s)
{
    const long long nyx = (long long)m.ny * m.nx;
    const int batch = ncols * m.nb;
    // tmp_f = F_f S_x   (ny x nx) (nx x nx)
    BGArgs<R> g1;
    g1.A = in;
    g1.B = Tab<R>::Sx(m);
    g1.C = tmp;
    g1.M = m.ny;
    g1.N = m.nx;
    g1.K = m.nx;
    g1.inner = m.nb;
    g1.lda = m.nx;
    g1.ldb = m.nx;
    g1.ldc = m.nx;
    g1.aso = ldi;
    g1.asi = nyx;
    g1.bso = 0;
    g1.bsi = 0;
    g1.cso = (long long)m.nb * nyx;
    g1.csi = nyx;
    g1.alpha = R(1);
    cudaError_t e = bgemm(g1, batch, s);
    if (e != cudaSuccess) return e;
    // out_f = sigma_b S_y tmp_f   (ny x ny) (ny x nx)
    BGArgs<R> g2;
    g2.A = Tab<R>::Sy(m);
    g2.B = tmp;
    g2.C = out;
    g2.M = m.ny;
    g2.N = m.nx;
    g2.K = m.ny;
    g2.inner = m.nb;
    g2.lda = m.ny;
    g2.ldb = m.nx;
    g2.ldc = m.nx;
    g2.aso = 0;
    g2.asi = 0;
    g2.bso = (long long)m.nb * nyx;
    g2.bsi = nyx;
    g2.cso = ldo;
    g2.csi = nyx;
    g2.alpha = (R)m.sigma_b;
    return bgemm(g2, batch, s);
}

template <typename R>
cudaError_t colscale(const R *in, long long ldi, const R *sc, R *out, long long ldo, int n, int ncols, cudaStream_t s)
{
    const size_t total = (size_t)n * ncols;
    if (!total) return cudaSuccess;
    colscale_kernel<R><<<blocks_for(total, 256), 256, 0, s>>>(in, ldi, sc, out, ldo, n, ncols);
    count_launch();
    return cudaGetLastError();
}

template <typename R>
cudaError_t hvp_batch(const AdvDev &m, const R *W, R *Y, long long ld, int P, int add_identity, R *r, cudaStream_t s)
{
    cudaError_t e;
    const long long n = m.n, nyx = (long long)m.ny * m.nx;
    R *cA, *cB, *cX, *src = (R *)m.src, *ebar = (R *)m.ebar, *tmp = (R *)m.tmp;
    const size_t cells = (size_t)P * m.ncells;
    batch_fields(m, P, &cA, &cB, &cX);
#define ADV_TRY(x)                          \
    do {                                    \
        if ((e = (x)) != cudaSuccess) return e; \
    } while (0)
    // source perturbation: E / dz * (L w)
    ADV_TRY(sep_apply<R>(m, W, ld, src, n, P, tmp, s));
    ADV_TRY(colscale<R>(src, n, Tab<R>::Es(m), src, n, (int)n, P, s));
    // tangent-linear window, residuals r = R^-1 H dc at the observation steps
    ADV_TRY(cudaMemsetAsync(cA, 0, cells * sizeof(R), s));
    for (int t = 0; t < m.T; ++t) {
        const int b = (int)(((long long)t * m.nb) / m.T);
        ADV_TRY(step<R>(m, cA, cB, cX, P, src + b * nyx, n, nullptr, 0, false, s));
        R *sw = cA;
        cA = cB;
        cB = sw;
        ADV_TRY(gather<R>(m, cA, P, t + 1, r, m.p, s));
    }
    // adjoint window
    ADV_TRY(cudaMemsetAsync(cA, 0, cells * sizeof(R), s));
    ADV_TRY(cudaMemsetAsync(ebar, 0, (size_t)P * n * sizeof(R), s));
    for (int t = m.T - 1; t >= 0; --t) {
        ADV_TRY(scatter<R>(m, cA, P, t + 1, r, m.p, s));
        const int b = (int)(((long long)t * m.nb) / m.T);
        ADV_TRY(step<R>(m, cA, cB, cX, P, nullptr, 0, ebar + b * nyx, n, true, s));
        R *sw = cA;
        cA = cB;
        cB = sw;
    }
    // Y = L^T (E / dz * ebar) (+ W)
    ADV_TRY(colscale<R>(ebar, n, Tab<R>::Es(m), ebar, n, (int)n, P, s));
    ADV_TRY(sep_apply<R>(m, ebar, n, Y, ld, P, tmp, s));
    if (add_identity) {
        const size_t total = (size_t)n * P;
        coladd_kernel<R><<<blocks_for(total, 256), 256, 0, s>>>(W, ld, Y, ld, (int)n, P);
        count_launch();
        ADV_TRY(cudaGetLastError());
    }
#undef ADV_TRY
    return cudaSuccess;
}

// The two halves of a product on P columns, for the observation-space dual of Algorithm 4:
// tangent linear r = R^-1 H' L w (ld ldw, r with stride p) and adjoint z = L^T H'^T f from an
// observation-space forcing f (stride p; z at ld ldz).
template <typename R>
cudaError_t tl_batch(const AdvDev &m, const R *W, long long ldw, int P, R *r, cudaStream_t s)
{
    cudaError_t e;
    const long long n = m.n, nyx = (long long)m.ny * m.nx;
    R *cA, *cB, *cX, *src = (R *)m.src, *tmp = (R *)m.tmp;
    const size_t cells = (size_t)P * m.ncells;
    batch_fields(m, P, &cA, &cB, &cX);
    if ((e = sep_apply<R>(m, W, ldw, src, n, P, tmp, s)) != cudaSuccess) return e;
    if ((e = colscale<R>(src, n, Tab<R>::Es(m), src, n, (int)n, P, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(cA, 0, cells * sizeof(R), s)) != cudaSuccess) return e;
    for (int t = 0; t < m.T; ++t) {
        const int b = (int)(((long long)t * m.nb) / m.T);
        if ((e = step<R>(m, cA, cB, cX, P, src + b * nyx, n, nullptr, 0, false, s)) != cudaSuccess) return e;
        R *sw = cA;
        cA = cB;
        cB = sw;
        if ((e = gather<R>(m, cA, P, t + 1, r, m.p, s)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename R>
cudaError_t ad_batch(const AdvDev &m, const R *f, int P, R *Z, long long ldz, cudaStream_t s)
{
    cudaError_t e;
    const long long n = m.n, nyx = (long long)m.ny * m.nx;
    R *cA, *cB, *cX, *ebar = (R *)m.ebar, *tmp = (R *)m.tmp;
    const size_t cells = (size_t)P * m.ncells;
    batch_fields(m, P, &cA, &cB, &cX);
    if ((e = cudaMemsetAsync(cA, 0, cells * sizeof(R), s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(ebar, 0, (size_t)P * n * sizeof(R), s)) != cudaSuccess) return e;
    for (int t = m.T - 1; t >= 0; --t) {
        if ((e = scatter<R>(m, cA, P, t + 1, f, m.p, s)) != cudaSuccess) return e;
        const int b = (int)(((long long)t * m.nb) / m.T);
        if ((e = step<R>(m, cA, cB, cX, P, nullptr, 0, ebar + b * nyx, n, true, s)) != cudaSuccess) return e;
        R *sw = cA;
        cA = cB;
        cB = sw;
    }
    if ((e = colscale<R>(ebar, n, Tab<R>::Es(m), ebar, n, (int)n, P, s)) != cudaSuccess) return e;
    return sep_apply<R>(m, ebar, n, Z, ldz, P, tmp, s);
}

}  // namespace

cudaError_t adv_coefs(const AdvDev &m, cudaStream_t s)
{
    count_launch();
    adv_coef_kernel<<<blocks_for((size_t)m.nx * m.ny, 256), 256, 0, s>>>(m.u64, m.v64, m.nx, m.ny, 1.0 / m.dx, 1.0 / m.dy,
                                                                          m.cf64);
    return cudaGetLastError();
}

cudaError_t adv_tl(const AdvDev &m, const double *W, int64_t ld, int ncols, double *r, cudaStream_t s)
{
    for (int c0 = 0; c0 < ncols; c0 += m.Pws64) {
        const int P = ncols - c0 < m.Pws64 ? ncols - c0 : m.Pws64;
        cudaError_t e = tl_batch<double>(m, W + (size_t)c0 * ld, ld, P, r + (size_t)c0 * m.p, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t adv_ad(const AdvDev &m, const double *f, int ncols, double *Z, int64_t ld, cudaStream_t s)
{
    for (int c0 = 0; c0 < ncols; c0 += m.Pws64) {
        const int P = ncols - c0 < m.Pws64 ? ncols - c0 : m.Pws64;
        cudaError_t e = ad_batch<double>(m, f + (size_t)c0 * m.p, P, Z + (size_t)c0 * ld, ld, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t adv_ad_obs(const AdvDev &m, const double *f, double *z, cudaStream_t s)
{
    cudaError_t e;
    const long long n = m.n, nyx = (long long)m.ny * m.nx;
    double *cA = m.c64A, *cB = m.c64B;
    if ((e = cudaMemsetAsync(cA, 0, (size_t)m.ncells * sizeof(double), s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(m.ebar64, 0, (size_t)n * sizeof(double), s)) != cudaSuccess) return e;
    for (int t = m.T - 1; t >= 0; --t) {
        if ((e = scatter<double>(m, cA, 1, t + 1, f, m.p, s)) != cudaSuccess) return e;
        const int bk = (int)(((long long)t * m.nb) / m.T);
        if ((e = step<double>(m, cA, cB, m.c64X, 1, nullptr, 0, m.ebar64 + bk * nyx, n, true, s)) != cudaSuccess) return e;
        double *sw = cA;
        cA = cB;
        cB = sw;
    }
    if ((e = colscale<double>(m.ebar64, n, m.Es64, m.ebar64, n, (int)n, 1, s)) != cudaSuccess) return e;
    return sep_apply<double>(m, m.ebar64, n, z, n, 1, m.tmp64, s);
}

cudaError_t adv_hvp(const AdvDev &m, bool fp64, const void *W, void *Y, int64_t ld, int ncols, int add_identity,
                    void *r, cudaStream_t s)
{
    for (int c0 = 0; c0 < ncols; c0 += m.Pmax) {
        const int P = ncols - c0 < m.Pmax ? ncols - c0 : m.Pmax;
        cudaError_t e;
        if (fp64)
            e = hvp_batch<double>(m, (const double *)W + (size_t)c0 * ld, (double *)Y + (size_t)c0 * ld, ld, P,
                                  add_identity, (double *)r, s);
        else
            e = hvp_batch<float>(m, (const float *)W + (size_t)c0 * ld, (float *)Y + (size_t)c0 * ld, ld, P,
                                 add_identity, (float *)r, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t adv_outer(const AdvDev &m, const double *x, double *d, double *jo, double *rd, double *b, cudaStream_t s)
{
    cudaError_t e;
    const long long n = m.n, nyx = (long long)m.ny * m.nx;
    emis_scale_kernel<<<blocks_for(n, 256), 256, 0, s>>>(m.Eb, x, 1.0 / m.dz, (int)n, m.Es64, m.Es32);
    count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    double *cA = m.c64A, *cB = m.c64B;
    // nonlinear window (the transport is linear in the tracer; the source is E(x) / dz)
    if ((e = cudaMemsetAsync(cA, 0, (size_t)m.ncells * sizeof(double), s)) != cudaSuccess) return e;
    for (int t = 0; t < m.T; ++t) {
        const int bk = (int)(((long long)t * m.nb) / m.T);
        if ((e = step<double>(m, cA, cB, m.c64X, 1, m.Es64 + bk * nyx, 0, nullptr, 0, false, s)) != cudaSuccess) return e;
        double *sw = cA;
        cA = cB;
        cB = sw;
        const int o0 = m.optr_h[t + 1], no = m.optr_h[t + 2] - o0;
        if (no > 0) {
            obs_innov_kernel<<<blocks_for(no, 128), 128, 0, s>>>(cA, o0, no, m.cell, m.w64, m.y, m.rinv64, d, jo);
            count_launch();
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
    }
    // gradient b = L^T (E / dz * ebar), ebar the source adjoint of R^-1 d
    if (m.p > 0) {
        if ((e = mul(m.p, d, m.rinv64, rd, s)) != cudaSuccess) return e;
    }
    if ((e = cudaMemsetAsync(cA, 0, (size_t)m.ncells * sizeof(double), s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(m.ebar64, 0, (size_t)n * sizeof(double), s)) != cudaSuccess) return e;
    for (int t = m.T - 1; t >= 0; --t) {
        if ((e = scatter<double>(m, cA, 1, t + 1, rd, m.p, s)) != cudaSuccess) return e;
        const int bk = (int)(((long long)t * m.nb) / m.T);
        if ((e = step<double>(m, cA, cB, m.c64X, 1, nullptr, 0, m.ebar64 + bk * nyx, n, true, s)) != cudaSuccess) return e;
        double *sw = cA;
        cA = cB;
        cB = sw;
    }
    if ((e = colscale<double>(m.ebar64, n, m.Es64, m.ebar64, n, (int)n, 1, s)) != cudaSuccess) return e;
    return sep_apply<double>(m, m.ebar64, n, b, n, 1, m.tmp64, s);
}

cudaError_t adv_tl_obs(const AdvDev &m, const double *w, double *r, cudaStream_t s)
{
    cudaError_t e;
    const long long n = m.n, nyx = (long long)m.ny * m.nx;
    double *cA = m.c64A, *cB = m.c64B, *src = m.ebar64;
    // source perturbation E / dz * (L w), then the tangent-linear window from zero
    if ((e = sep_apply<double>(m, w, n, src, n, 1, m.tmp64, s)) != cudaSuccess) return e;
    if ((e = colscale<double>(src, n, m.Es64, src, n, (int)n, 1, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(cA, 0, (size_t)m.ncells * sizeof(double), s)) != cudaSuccess) return e;
    for (int t = 0; t < m.T; ++t) {
        const int bk = (int)(((long long)t * m.nb) / m.T);
        if ((e = step<double>(m, cA, cB, m.c64X, 1, src + bk * nyx, n, nullptr, 0, false, s)) != cudaSuccess) return e;
        double *sw = cA;
        cA = cB;
        cB = sw;
        if ((e = gather<double>(m, cA, 1, t + 1, r, m.p, s)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t adv_bsqrt(const AdvDev &m, const double *in, double *out, int ncols, cudaStream_t s)
{
    for (int c0 = 0; c0 < ncols; c0 += m.Pmax64) {
        const int P = ncols - c0 < m.Pmax64 ? ncols - c0 : m.Pmax64;
        cudaError_t e = sep_apply<double>(m, in + (size_t)c0 * m.n, m.n, out + (size_t)c0 * m.n, m.n, P, m.tmp64, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// One column of the tracer forecast from x (FP64): the tracer field after
// steps steps, for building synthetic truths and tests.
cudaError_t adv_forecast(const AdvDev &m, const double *x, int steps, double *c_out, cudaStream_t s)
{
    cudaError_t e;
    const long long n = m.n, nyx = (long long)m.ny * m.nx;
    emis_scale_kernel<<<blocks_for(n, 256), 256, 0, s>>>(m.Eb, x, 1.0 / m.dz, (int)n, m.Es64, m.Es32);
    count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    double *cA = m.c64A, *cB = m.c64B;
    if ((e = cudaMemsetAsync(cA, 0, (size_t)m.ncells * sizeof(double), s)) != cudaSuccess) return e;
    for (int t = 0; t < steps; ++t) {
        const int bk = (int)(((long long)t * m.nb) / m.T);
        if ((e = step<double>(m, cA, cB, m.c64X, 1, m.Es64 + bk * nyx, 0, nullptr, 0, false, s)) != cudaSuccess) return e;
        double *sw = cA;
        cA = cB;
        cB = sw;
    }
    return cudaMemcpyAsync(c_out, cA, (size_t)m.ncells * sizeof(double), cudaMemcpyDeviceToDevice, s);
}

}  // namespace riot
