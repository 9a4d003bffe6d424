// rikfad_quadratic.cu -- batched BACD integration of R-iKFAD on many small
// dense quadratics f(X) = 1/2 vec(X)^T A vec(X) (the test problem of the
// paper's numerical validation of the gamma = 0 rates, Section 3.2 and Table
// tab:g0_slopes: A = B B^T / d + 0.8 I, d = m n, integrated to t = 1e7).
//
// Every system is tiny (m n <= 32) and its steps are strictly sequential, so
// the kernel maps one system to one aligned group of L lanes and packs
// 32 / L systems into a warp (L = MB NB clamped to [4, 32], where MB and NB
// are m and n rounded up to powers of two; both are template parameters).
// Lane a of a group owns element a = i n + j (row-major vec(X), as the
// oracle): its X_a, its momentum and row a of A in registers, plus its own
// copies of R_i, C_j and 1^T R.  The gradient A vec(X) reads X from shared
// memory with 128-bit broadcast loads and accumulates with paired float32
// FMAs (two round-to-nearest FMAs per instruction).  [P^(1)]^2 is written
// twice: row-major with row stride RS and column-major with column stride CS
// (NB and MB, plus 4 when that is a multiple of 8, so that consecutive rows
// or columns start in different 16-byte bank groups; padding stays zero).
// A row sum and a column sum are then a few 128-bit loads each, added in a
// fixed order with paired adds, so the lanes of one row (column) hold
// bit-identical R_i (C_j).  The total is added by every lane from shared memory
// (up to 16 lanes) or comes from an xor butterfly of shuffles; both leave
// identical bits in every lane.  One warp barrier per step (everything is
// exchanged together, double buffered); no global memory inside the step loop
// but the recorded energies.  Bound by the latency of the chain from [P^(1)]^2
// through the sums, the reciprocal and the exponential to the next kick, so a
// step is one straight run of code: the loads and FMAs of the next gradient are
// issued into that chain's gaps, and records and the end are looked at between
// runs of steps.  112 ns a step for 4 x 3 and 161 for 6 x 5 (193 and 224 with
// the gradient after the chain, a test for each step and a butterfly of four
// levels for 4 x 3).  Large batches take the kernel further down, with one lane
// per row or column.

// One step k follows the BACD sub-steps of the splitting table (Appendix A):
//   B  P^(B)_k = P_k - h A vec(X_k)
//   A  X_{k+1} = X_k + h P^(B)_k
//   C  P^(1)   = P^(B)_k exp(-h/2 xi~_k);  R, C <- e^{-alpha h}(R, C) + k (row, column sums of [P^(1)]^2)
//      P^(2)   = P^(1) exp(-h/2 xi~_{k+1})
//   D  P_{k+1} = P^(2) e^{-gamma h}
// 1^T R is filtered alongside, from the total of [P^(1)]^2 (equal to the sum
// of the filtered R_i up to rounding).
//
// Precision.  With gamma = 0 the friction decays like 1/t, and by t ~ 1e5
// one step's damping h/2 xi~ is ~1e-7: below half a float32 ulp of P, so a
// stored P (1 - 1e-7) rounds back to P and the damping is lost (the decay
// slopes bend from -1 to -0.7).  The kernel therefore never stores a damped
// momentum between steps: it carries P^(B)_{k-1} and the pending
// e1 = expm1(-h/2 xi~_{k-1}), and forms the next kick as
//   P^(B)_k = P^(B)_{k-1} + [P^(B)_{k-1} em - h g],
//   em = expm1(-h/2 xi~_{k-1} - h/2 xi~_k - gamma h)
//      = (1 + f) e2 + f,  f = (1 + e1)(1 + expm1(-gamma h)) - 1 = e1 e^{-gamma h} + expm1(-gamma h),
//   e2 = expm1(-h/2 xi~_k),
// in which the damping is part of a bracket about 50 times smaller than P,
// represented to its own float32 precision; the one rounding of the sum is
// unbiased.  e2 also gives this step's first half-damp, so one expm1 per
// step serves both.  P_k itself (for the energy and the output) is
// P^(B)_{k-1} + P^(B)_{k-1} em.  A launch starts from the stored P_k with
// nothing pending, so runs split at a launch boundary are bit-identical.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdint>
#include <string>

#include "rikfad.h"
#include "rikfad_records.hpp"

namespace rikfad {
int report_error(int code, const std::string &msg);
}

using namespace rikfad;

namespace {

constexpr int kQThreads = 128;                // 4 warps per block
constexpr int kQWarps = kQThreads / 32;
// Blocks per SM the registers are sized for (5: up to 102 registers).  A cap of
// 64 registers (8 blocks) measured slower in latency and in throughput.
#ifndef RIKFAD_QUAD_MIN_BLOCKS
#define RIKFAD_QUAD_MIN_BLOCKS 5
#endif
constexpr int kQMinBlocks = RIKFAD_QUAD_MIN_BLOCKS;
constexpr int64_t kQMaxDim = 32;
constexpr int64_t kQSchedulers = 608;         // warp schedulers of a GB300 (152 SMs)
constexpr int kQBufFloats = 128;             // per warp and parity, for each padded copy

struct QuadParams {
    int64_t batch;
    int m, n, d;
    const float *A;
    float *X, *P, *R, *C;
    const int64_t *record;
    int64_t nrecord;
    float *energy;
    int64_t k0, k1;                           // this launch runs steps k0 .. k1 - 1 and stops at k1
    float h, half_h, eg, oneg, decay, gain, eps;    // half_h = -h/2, eg = expm1(-gamma h), oneg = 1 + eg
};

// Two float32 lanes in one 64-bit register, and the paired add and FMA on
// them (PTX add/fma.rn.f32x2: two independent round-to-nearest operations).
__device__ __forceinline__ uint64_t pack2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// exp(z) - 1.  For |z| <= 1/16 the exponential series without its constant
// term, z (1 + z/2 (1 + z/3 (1 + z/4 (1 + z/5)))) written in Horner form with
// the coefficients 1/k!: the first omitted term, z^6/720, is below 1.3e-9 of
// the result.  Larger |z| use the library's expm1f.
__device__ __forceinline__ float expm1_series(float z)
{
    return z * fmaf(z, fmaf(z, fmaf(z, fmaf(z, 1.f / 120.f, 1.f / 24.f), 1.f / 6.f), 0.5f), 1.f);
}

__device__ __forceinline__ float expm1_small(float z)
{
    return fabsf(z) <= 0.0625f ? expm1_series(z) : expm1f(z);
}

// 1 / (1^T R + eps); 0 below the normal range (zero included, Theorem 3's
// convention), where the quotient can overflow: there R_i C_j / (1^T R) <= 1^T R
// is below any friction that a step can show, while an infinite factor turns the
// rows whose R_i is zero, and the lanes past the system's last row or column, into
// NaN.  The friction is formed as (R_i inv)(C_j h/2) for the same reason: R_i inv
// <= 1, whereas R_i C_j leaves the float32 range for factors beyond 1e+-19 (late in
// a damped run, or early in a diverging one).
__device__ __forceinline__ float inv_friction_denominator(float den)
{
    const float inv = __fdividef(1.f, den);
    return den < FLT_MIN ? 0.f : inv;
}

template <int MB, int NB>
struct QShape {
    static constexpr int L = MB * NB >= 32 ? 32 : (MB * NB < 4 ? 4 : MB * NB);   // lanes per system
    // Row stride of the row-major copy and column stride of the column-major
    // copy: an extent that is a multiple of 8 floats gets 4 more, so that
    // consecutive rows (columns) start in different 16-byte bank groups.
    static constexpr int RS = NB % 8 == 0 ? NB + 4 : NB;
    static constexpr int CS = MB % 8 == 0 ? MB + 4 : MB;
    static constexpr int BLK = ((MB * RS > NB * CS ? MB * RS : NB * CS) + 3) / 4 * 4;   // floats per system
    static_assert((32 / L) * BLK <= kQBufFloats, "padded blocks must fit the warp's buffer");
};

// Sum of K consecutive floats at p (16-byte aligned when K >= 4), in a fixed
// order: for K >= 4 the even- and odd-placed elements are summed as the two
// halves of paired adds (PTX add.rn.f32x2), then the two halves are added.
template <int K>
__device__ __forceinline__ float sum_run(const float *p)
{
    if constexpr (K >= 4) {
        const ulonglong2 *v = reinterpret_cast<const ulonglong2 *>(p);
        ulonglong2 w = v[0];
        uint64_t acc = add2(w.x, w.y);
#pragma unroll
        for (int q = 1; q < K / 4; ++q) {
            w = v[q];
            acc = add2(acc, w.x);
            acc = add2(acc, w.y);
        }
        float lo, hi;
        unpack2(acc, lo, hi);
        return lo + hi;
    } else {
        float s0 = 0.f;
#pragma unroll
        for (int q = 0; q < K; ++q)
            s0 += p[q];
        return s0;
    }
}

template <int MB, int NB>
__global__ void __launch_bounds__(kQThreads, kQMinBlocks) rikfad_quadratic_kernel(QuadParams q)
{
    constexpr int L = QShape<MB, NB>::L;
    constexpr int RS = QShape<MB, NB>::RS;
    constexpr int CS = QShape<MB, NB>::CS;
    constexpr int BLK = QShape<MB, NB>::BLK;
    __shared__ __align__(16) float xs[kQWarps][2][32];
    __shared__ __align__(16) float sq[kQWarps][2][32];           // [P^(1)]^2 in lane order (L <= 16)
    __shared__ __align__(16) float sr[kQWarps][2][kQBufFloats];  // row-major, row stride RS
    __shared__ __align__(16) float sc[kQWarps][2][kQBufFloats];  // column-major, column stride CS
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int a = lane & (L - 1);             // element within the system
    const int base = lane - a;                // first lane of the system's group
    const int pbase = (lane / L) * BLK;       // the system's padded blocks
    const int64_t sys = ((int64_t)blockIdx.x * kQWarps + warp) * (32 / L) + lane / L;
    const bool live = sys < q.batch;
    const int m = q.m, n = q.n, d = q.d;
    const bool elem = live && a < d;
    const int i = elem ? a / n : 0;
    const int j = elem ? a - i * n : 0;

    // Row a of A as packed pairs (A_a,2c, A_a,2c+1) for the paired FMAs below.
    uint64_t arow2[L / 2];
#pragma unroll
    for (int c = 0; c < L / 2; ++c) {
        const float lo = (elem && 2 * c < d) ? q.A[(sys * d + a) * d + 2 * c] : 0.f;
        const float hi = (elem && 2 * c + 1 < d) ? q.A[(sys * d + a) * d + 2 * c + 1] : 0.f;
        arow2[c] = pack2(lo, hi);
    }
    float x = elem ? q.X[sys * d + a] : 0.f;
    float pb = elem ? q.P[sys * d + a] : 0.f;   // P_k0 at the launch's first step, then P^(B)
    float Ri = 0.f, Cj = 0.f, S = 0.f;
    if (live) {
        Ri = q.R[sys * m + i];
        Cj = q.C[sys * n + j];
        for (int t = 0; t < m; ++t)
            S += q.R[sys * m + t];
    }
    // Damping owed at the next kick: em = e2 o + f, with f of the last half-damp
    // and o = 1 + f.  Nothing at the launch's first step,
    // which starts from P_k itself.
    float f = 0.f, o = 0.f;
    int cur = 0;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        xs[warp][u][lane] = 0.f;
#pragma unroll
        for (int v = 0; v < kQBufFloats; v += 32) {
            sr[warp][u][lane + v] = 0.f;
            sc[warp][u][lane + v] = 0.f;
        }
    }
    __syncwarp();
    xs[warp][0][lane] = x;
    __syncwarp();

    const int steps = (int)(q.k1 - q.k0);
    int64_t ri = q.nrecord > 0 ? first_record_at_or_after(q.record, q.nrecord, q.k0) : 0;
    int next = record_in_launch(q.record, q.nrecord, ri, q.k0, 0, steps);
    // The kick's bracket pb em - h g = e2 (pb o) + (pb f - h g): with the two
    // products formed before e2 is there, two operations of the chain fewer (6 x 5
    // 185 -> 164 ns a step, 2 x 2 102 -> 97; at 16 lanes 119 -> 122, not used).  It
    // rounds h g once more than the fused form; over 24 settings the error against
    // 64 bits is that of the fused form to 0.2% in the mean, 3% for single ones.
    constexpr bool kAhead = L != 16;
    float g, e2, pbo = 0.f, pre = 0.f;
    // g = A vec(X) of the published x (four partial sums over every fourth
    // column, as two pairs advanced by paired FMAs) and e2 = expm1(-h/2 xi~) of
    // the current factors, for the step to come: one straight run of two
    // independent chains, so that the loads and FMAs of g fill the latencies of
    // the factors' chain.
    auto prepare_step = [&]() {
        const ulonglong2 *xv = reinterpret_cast<const ulonglong2 *>(&xs[warp][cur][base]);
        uint64_t g01 = 0ull, g23 = 0ull;
#pragma unroll
        for (int b4 = 0; b4 < L / 4; ++b4) {
            const ulonglong2 v = xv[b4];
            g01 = fma2(arow2[2 * b4], v.x, g01);
            g23 = fma2(arow2[2 * b4 + 1], v.y, g23);
        }
        const float inv = inv_friction_denominator(S + q.eps);
        const float z = (Ri * inv) * (Cj * q.half_h);
        e2 = expm1_series(z);
        float g0, g1;
        unpack2(add2(g01, g23), g0, g1);
        g = g0 + g1;
        if constexpr (kAhead) {
            pbo = pb * o;
            pre = fmaf(pb, f, -q.h * g);
        }
        if (fabsf(z) > 0.0625f)
            e2 = expm1f(z);
    };
    prepare_step();
    for (int s = 0;;) {
        // One step is one straight run of code; records and the end are looked at
        // between runs of steps.
        const int stop = next >= 0 ? next : steps;
        for (; s < stop; ++s) {
            const float bracket = kAhead ? fmaf(e2, pbo, pre) : fmaf(-q.h, g, pb * fmaf(e2, o, f));
            pb = pb + bracket;                    // B (with the owed damping)
            x = fmaf(q.h, pb, x);                 // A
            const float p1 = fmaf(pb, e2, pb);    // C, first half
            const float p1sq = p1 * p1;
            f = fmaf(e2, q.oneg, q.eg);
            o = 1.f + f;
            xs[warp][cur ^ 1][lane] = x;
            if (L <= 16)
                sq[warp][cur][lane] = elem ? p1sq : 0.f;
            if (elem) {
                sr[warp][cur][pbase + i * RS + j] = p1sq;
                sc[warp][cur][pbase + j * CS + i] = p1sq;
            }
            __syncwarp();
            // Factor filter: row sum and column sum, in a fixed order.
            const float rs = sum_run<NB>(&sr[warp][cur][pbase + i * RS]);
            const float cs = sum_run<MB>(&sc[warp][cur][pbase + j * CS]);
            // Total of [P^(1)]^2 over the system.  Up to 16 lanes every lane adds
            // all of them in the same order (4 x 3: 166 -> 147 ns a step); at 32 an
            // xor butterfly (partners add the same two numbers, so every lane ends
            // with the same bits) is shorter than 8 loads and their sum.
            float tot;
            if (L <= 16) {
                tot = sum_run<L>(&sq[warp][cur][base]);
            } else {
                tot = elem ? p1sq : 0.f;
#pragma unroll
                for (int w = L / 2; w > 0; w >>= 1)
                    tot += __shfl_xor_sync(0xffffffffu, tot, w);
            }
            Ri = fmaf(q.gain, rs, q.decay * Ri);
            Cj = fmaf(q.gain, cs, q.decay * Cj);
            S = fmaf(q.gain, tot, q.decay * S);
            cur ^= 1;
            prepare_step();
        }
        while (s == next) {                   // energy of the state after k0 + s steps
            const float pk = fmaf(pb, fmaf(e2, o, f), pb);
            float e = 0.5f * x * g + 0.5f * pk * pk;
#pragma unroll
            for (int w = L / 2; w > 0; w >>= 1)
                e += __shfl_xor_sync(0xffffffffu, e, w);
            if (live && a == 0)
                q.energy[ri * q.batch + sys] = e;
            ++ri;
            next = record_in_launch(q.record, q.nrecord, ri, q.k0, s, steps);
        }
        if (s == steps)
            break;
    }
    if (elem) {
        q.X[sys * d + a] = x;
        q.P[sys * d + a] = fmaf(pb, fmaf(e2, o, f), pb);
        if (j == 0)
            q.R[sys * m + i] = Ri;
        if (i == 0)
            q.C[sys * n + j] = Cj;
    }
}

int q_fail(int code, const char *msg) { return rikfad::report_error(code, msg); }

template <int MB, int NB>
cudaError_t launch_all(QuadParams q, int64_t nsteps, int64_t per_launch, cudaStream_t s)
{
    constexpr int L = QShape<MB, NB>::L;
    const int64_t groups = (q.batch + (32 / L) - 1) / (32 / L);   // warps
    const int64_t blocks = (groups + kQWarps - 1) / kQWarps;
    for (int64_t k0 = 0;; k0 += per_launch) {
        q.k0 = k0;
        q.k1 = k0 + per_launch < nsteps ? k0 + per_launch : nsteps;
        rikfad_quadratic_kernel<MB, NB><<<(unsigned)blocks, kQThreads, 0, s>>>(q);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess || q.k1 == nsteps)
            return e;
    }
}

template <int MB>
cudaError_t dispatch_nb(int nb, QuadParams q, int64_t nsteps, int64_t per_launch, cudaStream_t s)
{
    switch (nb) {
    case 1: return launch_all<MB, 1>(q, nsteps, per_launch, s);
    case 2: return launch_all<MB, 2>(q, nsteps, per_launch, s);
    case 4:
        if constexpr (MB <= 16)
            return launch_all<MB, 4>(q, nsteps, per_launch, s);
        break;
    case 8:
        if constexpr (MB <= 8)
            return launch_all<MB, 8>(q, nsteps, per_launch, s);
        break;
    case 16:
        if constexpr (MB <= 4)
            return launch_all<MB, 16>(q, nsteps, per_launch, s);
        break;
    case 32:
        if constexpr (MB <= 2)
            return launch_all<MB, 32>(q, nsteps, per_launch, s);
        break;
    default: break;
    }
    return cudaErrorInvalidValue;
}

int pow2_ceil(int v)
{
    int p = 1;
    while (p < v)
        p <<= 1;
    return p;
}

// ---------------------------------------------------- large batches
//
// One lane per row (or per column, whichever are more), EPL = min(m, n)
// elements a lane: LN = max(m, n) rounded up to a power of two lanes a system,
// 32 / LN systems a warp.  Against one lane per element, the exchange of x, the
// sums, the reciprocal and the loop are shared by EPL times as many systems, the
// sum along a lane is local, and the one across lanes is a butterfly over LN
// lanes only (its total is the sum of the EPL results, so 1^T R needs no
// butterfly of its own).  EPL rows of A per lane are held in registers (160 of
// them for 6 x 5: 8 warps an SM).  Bound by the FP32 pipe (64% of its cycles for
// 6 x 5: 80 paired FMAs per lane and step, for 4 systems a warp, and ~30
// operations per element) and by latency between them; 70 warp instructions per
// 6 x 5 system and step against 119 with a lane per element.  65536 systems of
// 6 x 5: 7.4 -> 11.9 G system-steps/s.  With one row or column the lanes are the same
// in number, and what is saved is the exchange of the squares through shared memory.
template <int LN, int EPL>
struct QLanes {
    static constexpr int D = LN * EPL < 32 ? LN * EPL : 32;      // largest d (m n <= 32)
    static constexpr int DP = (D + 3) / 4 * 4;                   // columns of A held
    // Floats between the systems' copies of x: an odd number of 16-byte groups.
    static constexpr int XS = DP / 4 % 2 ? DP : DP + 4;
    static constexpr int SPW = 32 / LN;                          // systems per warp
    // Blocks per SM the registers are sized for.
    static constexpr int MB = EPL * DP >= 128 ? 2 : 3;
};

template <int LN, int EPL>
__global__ void __launch_bounds__(kQThreads, QLanes<LN, EPL>::MB) rikfad_quadratic_lanes_kernel(QuadParams q)
{
    using T = QLanes<LN, EPL>;
    constexpr int DP = T::DP, XS = T::XS, SPW = T::SPW;
    constexpr int kFlip = SPW * XS;
    __shared__ __align__(16) float xs[kQWarps][2][kFlip];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int l = lane & (LN - 1), grp = lane / LN;
    const int64_t sys = ((int64_t)blockIdx.x * kQWarps + warp) * SPW + grp;
    const int m = q.m, n = q.n, d = q.d;
    const bool cols = n > m;                     // lanes own columns
    const bool live = sys < q.batch && l < (cols ? n : m);
    // Element e of lane l; x is exchanged in the order l EPL + e.
    const int a0 = cols ? l : l * n, as = cols ? n : 1;

    uint64_t arow2[EPL][DP / 2];
    float x[EPL], pb[EPL], E[EPL], f[EPL];
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
        const float *A = q.A + (sys * d + a0 + e * as) * d;
#pragma unroll
        for (int c = 0; c < DP / 2; ++c) {
            float v[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int lb = (2 * c + u) / EPL, eb = (2 * c + u) % EPL;
                v[u] = live && lb * EPL + eb < d ? A[cols ? eb * n + lb : lb * n + eb] : 0.f;
            }
            arow2[e][c] = pack2(v[0], v[1]);
        }
        x[e] = live ? q.X[sys * d + a0 + e * as] : 0.f;
        pb[e] = live ? q.P[sys * d + a0 + e * as] : 0.f;
        f[e] = 0.f;         // damping owed at the next kick: em = e2 (o1 + f) + f (as in the kernel above)
        E[e] = 0.f;
    }
    float o1 = 0.f;                              // 1 after the launch's first step
    float F = 0.f, S = 0.f;                      // the lane's factor, 1^T R
    if (live) {
        const float *R = q.R + sys * m, *C = q.C + sys * n;
        F = cols ? C[l] : R[l];
#pragma unroll
        for (int e = 0; e < EPL; ++e)
            E[e] = cols ? R[e] : C[e];
        for (int t = 0; t < m; ++t)
            S += R[t];
    }
    for (int b = lane; b < 2 * kFlip; b += 32)
        xs[warp][0][b] = 0.f;
    __syncwarp();
    int cur = 0;
    auto publish = [&]() {
        float *to = &xs[warp][cur][grp * XS];
        if (live) {
            if constexpr (EPL == 4)
                *reinterpret_cast<float4 *>(to + 4 * l) = make_float4(x[0], x[1], x[2], x[3]);
            else if constexpr (EPL == 2)
                *reinterpret_cast<float2 *>(to + 2 * l) = make_float2(x[0], x[1]);
            else
            {
#pragma unroll
                for (int e = 0; e < EPL; ++e)
                    to[l * EPL + e] = x[e];
            }
        }
        __syncwarp();
    };
    publish();

    const int steps = (int)(q.k1 - q.k0);
    int64_t ri = q.nrecord > 0 ? first_record_at_or_after(q.record, q.nrecord, q.k0) : 0;
    int next = record_in_launch(q.record, q.nrecord, ri, q.k0, 0, steps);
    float g[EPL], e2[EPL];
    // g = A vec(X) of the published x and e2 = expm1(-h/2 xi~) of the current
    // factors, for the step to come.  One straight run of independent chains, so
    // that the FMAs of g fill the latencies of the factors' chain.
    auto prepare_step = [&]() {
        const float inv = inv_friction_denominator(S + q.eps);
        const float fh = (F * inv) * q.half_h;
        float zmax = 0.f;
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
            const float z = fh * E[e];
            zmax = fmaxf(zmax, fabsf(z));
            e2[e] = expm1_series(z);
        }
        uint64_t g01[EPL], g23[EPL];
#pragma unroll
        for (int e = 0; e < EPL; ++e)
            g01[e] = g23[e] = 0ull;
        const ulonglong2 *xv = reinterpret_cast<const ulonglong2 *>(&xs[warp][cur][grp * XS]);
#pragma unroll
        for (int b4 = 0; b4 < DP / 4; ++b4) {
            const ulonglong2 v = xv[b4];
#pragma unroll
            for (int e = 0; e < EPL; ++e) {
                g01[e] = fma2(arow2[e][2 * b4], v.x, g01[e]);
                g23[e] = fma2(arow2[e][2 * b4 + 1], v.y, g23[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
            float g0, g1;
            unpack2(add2(g01[e], g23[e]), g0, g1);
            g[e] = g0 + g1;
        }
        if (zmax > 0.0625f)
#pragma unroll
            for (int e = 0; e < EPL; ++e)
                e2[e] = expm1_small(fh * E[e]);
    };
    prepare_step();
    for (int s = 0;;) {
        // One step is one straight run of code; records and the end are looked at
        // between runs of steps.
        const int stop = next >= 0 ? next : steps;
        for (; s < stop; ++s) {
            float rs = 0.f, tot = 0.f, qe[EPL];
#pragma unroll
            for (int e = 0; e < EPL; ++e) {
                const float em = fmaf(e2[e], o1 + f[e], f[e]);
                pb[e] = pb[e] + fmaf(-q.h, g[e], pb[e] * em);   // B (with the owed damping)
                x[e] = fmaf(q.h, pb[e], x[e]);                  // A
                const float p1 = fmaf(pb[e], e2[e], pb[e]);     // C, first half
                qe[e] = p1 * p1;
                rs = e == 0 ? qe[0] : rs + qe[e];
                f[e] = fmaf(e2[e], q.oneg, q.eg);
            }
            o1 = 1.f;
            cur ^= 1;
            publish();
            // Factor filter: the lane's sum; the sums across lanes by an xor
            // butterfly (partners add the same two numbers, so every lane ends with
            // the same bits); their total.
#pragma unroll
            for (int w = LN / 2; w > 0; w >>= 1)
#pragma unroll
                for (int e = 0; e < EPL; ++e)
                    qe[e] += __shfl_xor_sync(0xffffffffu, qe[e], w);
#pragma unroll
            for (int e = 0; e < EPL; ++e) {
                E[e] = fmaf(q.gain, qe[e], q.decay * E[e]);
                tot = e == 0 ? qe[0] : tot + qe[e];
            }
            F = fmaf(q.gain, rs, q.decay * F);
            S = fmaf(q.gain, tot, q.decay * S);
            prepare_step();
        }
        while (s == next) {                   // energy of the state after k0 + s steps
            float en = 0.f;
#pragma unroll
            for (int e = 0; e < EPL; ++e) {
                const float pk = fmaf(pb[e], fmaf(e2[e], o1 + f[e], f[e]), pb[e]);
                en += 0.5f * x[e] * g[e] + 0.5f * pk * pk;
            }
#pragma unroll
            for (int w = LN / 2; w > 0; w >>= 1)
                en += __shfl_xor_sync(0xffffffffu, en, w);
            if (live && l == 0)
                q.energy[ri * q.batch + sys] = en;
            ++ri;
            next = record_in_launch(q.record, q.nrecord, ri, q.k0, s, steps);
        }
        if (s == steps)
            break;
    }
    if (live) {
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
            q.X[sys * d + a0 + e * as] = x[e];
            q.P[sys * d + a0 + e * as] = fmaf(pb[e], fmaf(e2[e], o1 + f[e], f[e]), pb[e]);
        }
        float *Fg = cols ? q.C + sys * n : q.R + sys * m;
        float *Eg = cols ? q.R + sys * m : q.C + sys * n;
        Fg[l] = F;
        if (l == 0)
#pragma unroll
            for (int e = 0; e < EPL; ++e)
                Eg[e] = E[e];
    }
}

template <int LN, int EPL>
cudaError_t launch_lanes(QuadParams q, int64_t nsteps, int64_t per_launch, cudaStream_t s)
{
    constexpr int64_t kSys = QLanes<LN, EPL>::SPW * kQWarps;     // systems per block
    const int64_t blocks = (q.batch + kSys - 1) / kSys;
    for (int64_t k0 = 0;; k0 += per_launch) {
        q.k0 = k0;
        q.k1 = k0 + per_launch < nsteps ? k0 + per_launch : nsteps;
        rikfad_quadratic_lanes_kernel<LN, EPL><<<(unsigned)blocks, kQThreads, 0, s>>>(q);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess || q.k1 == nsteps)
            return e;
    }
}

cudaError_t dispatch_lanes(QuadParams q, int64_t nsteps, int64_t per_launch, cudaStream_t s)
{
    const int big = q.m > q.n ? q.m : q.n, small = q.m > q.n ? q.n : q.m;
    switch (pow2_ceil(big) * 8 + small) {       // small <= 5: m n <= 32
#define RK_LANES(LN, EPL)         \
    case LN * 8 + EPL:            \
        return launch_lanes<LN, EPL>(q, nsteps, per_launch, s);
        RK_LANES(1, 1) RK_LANES(2, 1) RK_LANES(2, 2) RK_LANES(4, 1) RK_LANES(4, 2) RK_LANES(4, 3) RK_LANES(4, 4)
        RK_LANES(8, 1) RK_LANES(8, 2) RK_LANES(8, 3) RK_LANES(8, 4) RK_LANES(8, 5) RK_LANES(16, 1) RK_LANES(16, 2)
        RK_LANES(16, 3) RK_LANES(32, 1)
#undef RK_LANES
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

extern "C" RIKFAD_API int rikfad_quadratic_run(int64_t batch, int64_t m, int64_t n, const float *A,
                                               float *X, float *P, float *R, float *C, double step,
                                               const rikfad_hparams *hp, int64_t nsteps,
                                               const int64_t *record, int64_t nrecord, float *energy,
                                               void *stream)
{
    if (batch < 0 || batch > ((int64_t)1 << 24))
        return q_fail(RIKFAD_ERR_ARG, "batch must be in [0, 2^24]");
    if (m < 1 || n < 1 || m * n > kQMaxDim)
        return q_fail(RIKFAD_ERR_ARG, "need m >= 1, n >= 1 and m * n <= 32");
    if (nsteps < 0 || nrecord < 0)
        return q_fail(RIKFAD_ERR_ARG, "nsteps and nrecord must be >= 0");
    if (hp == nullptr)
        return q_fail(RIKFAD_ERR_ARG, "hp is NULL");
    if (!(std::isfinite(hp->alpha) && hp->alpha > 0) || !(hp->mu > 0) ||
        !(std::isfinite(hp->gamma) && hp->gamma >= 0) ||
        !(std::isfinite(hp->eps_stab) && hp->eps_stab >= 0))
        return q_fail(RIKFAD_ERR_ARG, "hyperparameters out of range");
    if (!(std::isfinite(step) && step > 0))
        return q_fail(RIKFAD_ERR_ARG, "step must be finite and > 0");
    if (batch > 0 && (A == nullptr || X == nullptr || P == nullptr || R == nullptr || C == nullptr))
        return q_fail(RIKFAD_ERR_ARG, "NULL state pointer");
    if (batch > 0 && nrecord > 0 && (record == nullptr || energy == nullptr))
        return q_fail(RIKFAD_ERR_ARG, "NULL record or energy pointer");
    if ((uintptr_t)A % 4 || (uintptr_t)X % 4 || (uintptr_t)P % 4 || (uintptr_t)R % 4 ||
        (uintptr_t)C % 4 || (uintptr_t)energy % 4 || (uintptr_t)record % 8)
        return q_fail(RIKFAD_ERR_ALIGN, "misaligned pointer");
    if (batch == 0)
        return RIKFAD_OK;

    QuadParams q{};
    q.batch = batch;
    q.m = (int)m;
    q.n = (int)n;
    q.d = (int)(m * n);
    q.A = A;
    q.X = X;
    q.P = P;
    q.R = R;
    q.C = C;
    q.record = nrecord > 0 ? record : nullptr;
    q.nrecord = nrecord;
    q.energy = energy;
    q.h = (float)step;
    q.half_h = (float)(-0.5 * step);
    q.eg = (float)std::expm1(-hp->gamma * step);
    q.oneg = (float)std::exp(-hp->gamma * step);
    q.decay = (float)std::exp(-hp->alpha * step);
    q.gain = std::isinf(hp->mu) ? 0.f : (float)(-std::expm1(-hp->alpha * step) / (hp->mu * hp->alpha));
    q.eps = (float)hp->eps_stab;

    // Launches of per_launch steps: 2^16, or the largest power of two that
    // keeps a launch within 2^31 system-steps (at least 128 for batch <=
    // 2^24), so that no launch runs for more than about a second.
    int64_t per_launch = (int64_t)1 << 16;
    while (per_launch > 128 && per_launch * batch > ((int64_t)1 << 31))
        per_launch >>= 1;

    const int mb = pow2_ceil((int)m), nb = pow2_ceil((int)n);   // mb nb <= 64 when m n <= 32
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e;
    // One lane per element (more lanes a system: the shorter step) while its
    // warps are few per scheduler, one lane per row or column (fewer
    // instructions a system) beyond; later where that leaves a fifth or more of
    // the elements' slots empty.  ns a step, elements / lanes, measured at 16
    // systems | just beyond the line, and throughput in G system-steps/s at 65536:
    //   6 x 5  161 / 271 | 255 / 275, 7.4 / 11.9     4 x 3  112 / 131 | 186 / 134, 20 / 57
    //   3 x 7  159 / 174 | 242 / 176, 8.4 / 22       2 x 2  95 / 91 | 140 / 116, 106 / 189
    //   10 x 3 158 / 222 | 280 / 307, 6.6 / 9.0      8 x 1  100 / 117 | 161 / 145, 50 / 66
    //   16 x 1 116 / 134 | 214 / 175, 18 / 28        32 x 1 161 / 160 | 276 / 221, 7.1 / 10.1
    // (6 x 5 and 10 x 3 at two warps per scheduler, where their line is three).  A
    // system's low bits so depend on the batch that it is run in.
    const int lanes = std::min(std::max(mb * nb, 4), 32);       // of the one-lane-per-element kernel
    const int64_t warps = (batch * lanes + 31) / 32;
    const int64_t slots = std::max(mb, nb) * std::min(m, n);    // of the one-lane-per-row kernel
    if (warps > (slots > 32 ? 3 : 2) * kQSchedulers) {
        e = dispatch_lanes(q, nsteps, per_launch, s);
    } else {
        switch (mb) {
        case 1: e = dispatch_nb<1>(nb, q, nsteps, per_launch, s); break;
        case 2: e = dispatch_nb<2>(nb, q, nsteps, per_launch, s); break;
        case 4: e = dispatch_nb<4>(nb, q, nsteps, per_launch, s); break;
        case 8: e = dispatch_nb<8>(nb, q, nsteps, per_launch, s); break;
        case 16: e = dispatch_nb<16>(nb, q, nsteps, per_launch, s); break;
        default: e = dispatch_nb<32>(nb, q, nsteps, per_launch, s); break;
        }
    }
    if (e != cudaSuccess)
        return q_fail(RIKFAD_ERR_CUDA, cudaGetErrorString(e));
    return RIKFAD_OK;
}
