// rikfad_diag_kernels.cuh -- kernels of the friction diagnostic: how far the
// rank-1 friction xi~ = R C^T / (1^T R + eps) built from shadow factors is
// from the full element-wise friction xi of the same trajectory, against the
// best rank-1 approximation (Eckart-Young: relative error
// sqrt(1 - sigma_1^2 / ||xi||_F^2)), and the stable rank ||xi||_F^2 /
// sigma_1^2 (the comparison of the paper's Section 4.4).
//
// sigma_1 comes from power iteration on xi^T xi, on the device, two kernels an
// iteration chained by programmatic dependent launch: the row kernel reads xi
// once from memory (u = xi v, then this block's share of xi^T u from the rows
// just read, still in L1 or L2 up to kDiagStageCols columns; the rows that all
// blocks of a wider one have in hand outgrow L2 from about 8000), the column
// kernel adds the blocks' shares, forms the next iterate and tests convergence.
// The first row kernel also takes the norms ||xi||^2 and ||xi - xi~||^2 from the
// same read.
//
// The iterate's length does not matter: sigma^2 = ||xi v||^2 / ||v||^2 is formed
// with the length of the float32 iterate itself, so no kernel waits for a norm
// over all columns, and a rounding of v enters the quotient at second order
// only.  What would enter at first order, the rounding of u = xi v, is kept
// below 1e-13 by compensated dot products (Ogita, Rump and Oishi, "Accurate sum
// and dot product", 2005, algorithm Dot2) in float32, about ten times the rate
// of float64 here.  So the quotient settles as soon as the iterate has
// converged: 2 to 4 iterations for GPT2-S layers, where a quotient from plain
// float32 sums wandered by ~1e-9 for 10 to 200 until two in a row agreed to
// 1e-10.
//
// Every reduction runs in a fixed order; float64 only adds per-row and
// per-block partial sums.  Bound by launch and L2 latency for a layer's 2 to 10
// MB, by the reads of xi for larger matrices.  Measured on GB300, six calls for the
// layers of a GPT2-S block: 3800 to 7400 us (by seed) with four kernels an
// iteration in a captured graph and the plain quotient, 325 us so; 8192 x 8192 (268
// MB) 453 us a call of 3 iterations, 4096 x 16384 647.
#pragma once
#include <algorithm>

#include "rikfad_kernels.cuh"

namespace rikfad {

constexpr int kDiagMaxBlocks = 456;      // row blocks: 3 per SM of a GB300
constexpr int kDiagStageCols = 4096;     // widest xi whose iterate and sums are staged in shared memory
constexpr int kDiagMaxColBlocks = 512;   // column blocks (each adds all of their sums of v^2)
constexpr int64_t kDiagMaxPartials = 1 << 24;   // floats of row-block partials (more only at 32 rows a block)
// Threads of the column kernel, whose warps share the partials of 32 columns:
// 1024 beyond 128 row blocks (768 x 768, 192 of them: 51 us a call against 59 with
// 256), else 256 (64 x 4096, 64 of them: 64 against 69 with 1024).
inline int diag_col_threads(int nblk) { return nblk > 128 ? 1024 : 256; }
constexpr int kDiagIters = 4;            // iterations enqueued before the host first looks

// State of one power iteration, in device memory, kept twice and used by turns:
// an iteration's kernels read one and its column kernel writes the other, so that
// no block of a launch reads what another block of it writes.  The record the host
// reads is a copy in mapped host memory.
struct DiagState {
    double sigma2;     // ||xi v||^2 / ||v||^2 of the current iterate
    double f2;         // ||xi||^2
    double e2;         // ||xi - xi~||^2
    int32_t it;        // iterations done
    int32_t done;      // converged, or max_iters reached, or xi^T xi v = 0
};

struct DiagParams {
    const float *xi;           // m x n, row-major, 16-byte aligned
    const float *R, *C;
    const float *spart;
    TensorDev td;
    float eps;
    int nblk;                  // blocks of the row kernel
    int wpr;                   // warps per row: 1, 2, 4 or 8
    int ncb;                   // blocks of the column kernel
    int64_t cpb;               // columns of each, a multiple of 32
    int parity;                // which half of v2part holds ||v||^2 of this iteration
    int last;                  // 1: write the host's record even if not done
    int max_iters;
    double tol;
    float *v;                  // iterate (written by the column kernel)
    float *wpart;              // nblk x n
    double *upart;             // nblk: sums of u_i^2
    double *npart;             // 2 x nblk: sums of xi^2 and (xi - xi~)^2
    double *v2part;            // 2 x ncb: sums of v_j^2
    DiagState *st;             // of this iteration
    DiagState *st_next;        // of the next
    DiagState *host;           // mapped host memory
};

// Warps per row: as many as give the row kernel a block per SM of a GB300.
inline int diag_warps_per_row(int64_t m)
{
    int wpr = 1;
    while (wpr < kWarps && m * wpr < 152 * kWarps)
        wpr *= 2;
    return wpr;
}

// Blocks of the row kernel.  Their partials stay within kDiagMaxPartials where
// that leaves at least a block per 32 rows.
inline int64_t diag_row_blocks(int64_t m, int64_t n)
{
    const int64_t rows = kWarps / diag_warps_per_row(m);
    const int64_t blocks = std::min<int64_t>(kDiagMaxBlocks, (m + rows - 1) / rows);
    return std::min(blocks, std::max(kDiagMaxPartials / n, (m + 31) / 32));
}

// Columns per block of the column kernel, a multiple of 32, and its blocks.
inline int64_t diag_cols_per_block(int64_t n)
{
    return (n + 32 * kDiagMaxColBlocks - 1) / (32 * kDiagMaxColBlocks) * 32;
}

inline int diag_col_blocks(int64_t n)
{
    return (int)((n + diag_cols_per_block(n) - 1) / diag_cols_per_block(n));
}

__device__ __forceinline__ double warp_sum_f64(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// s + e += a b, with the rounding errors of the product and of the sum in e.
__device__ __forceinline__ void dot2(float &s, float &e, float a, float b)
{
    const float p = __fmul_rn(a, b);
    const float pe = __fmaf_rn(a, b, -p);
    const float t = __fadd_rn(s, p);
    const float z = __fsub_rn(t, s);
    e += __fadd_rn(pe, __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z)));
    s = t;
}

// (s, e) += (s2, e2)
__device__ __forceinline__ void add2(float &s, float &e, float s2, float e2)
{
    const float t = __fadd_rn(s, s2);
    const float z = __fsub_rn(t, s);
    e = __fadd_rn(__fadd_rn(e, e2), __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(s2, z)));
    s = t;
}

// Row kernel.  A block takes a contiguous range of rows, kWarps / wpr at a
// time: wpr warps a row for u_i (columns interleaved between them), then every
// thread its own columns for the block's share of xi^T u.  FIRST: the iterate
// is C, scaled to at most unit length (all ones over sqrt(n) if C = 0), and the
// norms are taken too.  WIDTH: 16-byte loads where n is a multiple of 4 (xi of
// 4096 x 16384: 647 us a call with them, 926 without).
enum DiagWidth { kDiagScalar, kDiagVec, kDiagVecStaged };
template <bool FIRST, DiagWidth WIDTH>
__global__ void __launch_bounds__(kThreads, FIRST && WIDTH != kDiagScalar ? 2 : 3) rikfad_diag_rows_kernel(DiagParams d)
{
    constexpr bool VEC = WIDTH != kDiagScalar;
    extern __shared__ __align__(16) float dsm[];
    __shared__ float2 ue[kWarps], nf[kWarps];
    __shared__ float us[kWarps];
    __shared__ double dd[3][kWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t n = d.td.cols, m = d.td.rows;
    wait_for_predecessor();
    allow_successor_launch();
    if (!FIRST && d.st->done)
        return;
    const bool staged = VEC ? WIDTH == kDiagVecStaged : n <= kDiagStageCols;
    float *wacc = staged ? dsm + (n + 3) / 4 * 4 : d.wpart + (int64_t)blockIdx.x * n;
    const float *v = staged ? dsm : FIRST ? d.C : d.v;
    float inv = 0.f, vscale = 1.f, vbias = 0.f;
    if (FIRST) {
        inv = inv_denominator(row_total(d.spart, d.td), d.eps);
        float mx = 0.f;
        for (int64_t j = tid; j < n; j += kThreads)
            mx = fmaxf(mx, d.C[j]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0)
            us[warp] = mx;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kWarps; ++k)
            mx = fmaxf(mx, us[k]);
        __syncthreads();
        const float unit = rsqrtf((float)n);
        vscale = mx > 0.f ? unit / mx : 0.f;
        if (!isfinite(vscale) || vscale == 0.f) {   // C = 0, not finite, or too small to scale
            vscale = 0.f;
            vbias = unit;
        }
    }
    // v_j: as staged, or (FIRST, not staged) from C.
    auto first_v = [&](float c) { return vscale != 0.f ? __fmul_rn(c, vscale) : vbias; };
    if (staged) {
        for (int64_t j = tid; j < n; j += kThreads)
            dsm[j] = FIRST ? first_v(d.C[j]) : d.v[j];
    }
    if (VEC)
        for (int64_t j = tid; j < n / 4; j += kThreads)
            reinterpret_cast<float4 *>(wacc)[j] = make_float4(0.f, 0.f, 0.f, 0.f);
    else
        for (int64_t j = tid; j < n; j += kThreads)
            wacc[j] = 0.f;
    __syncthreads();
    auto v_at = [&](int64_t j) { return FIRST && !staged ? first_v(v[j]) : v[j]; };
    if (FIRST && blockIdx.x == 0) {     // a cleared state; ||v||^2 of the first iterate
        if (tid == 0)
            *d.st = DiagState{};
        double a = 0.0;
        for (int64_t j = tid; j < n; j += kThreads) {
            const double t = (double)v_at(j);
            a += t * t;
        }
        a = warp_sum_f64(a);
        if (lane == 0)
            dd[0][warp] = a;
        __syncthreads();
        for (int b = tid; b < d.ncb; b += kThreads) {
            double t = 0.0;
            if (b == 0)
                for (int k = 0; k < kWarps; ++k)
                    t += dd[0][k];
            d.v2part[b] = t;
        }
        __syncthreads();
    }

    const int wpr = d.wpr, rpb = kWarps / wpr;
    const int64_t r0 = m * blockIdx.x / d.nblk, r1 = m * (blockIdx.x + 1) / d.nblk;
    const int part = warp % wpr, sub = warp / wpr;
    double u2 = 0.0, n1 = 0.0, n2 = 0.0;        // thread k < rpb: its rows
    for (int64_t r = r0; r < r1; r += rpb) {
        const int64_t row = r + sub;
        float s = 0.f, e = 0.f, f1 = 0.f, f2 = 0.f;
        if (row < r1) {
            const float *x = d.xi + row * n;
            const float rhat = FIRST ? d.R[row] * inv : 0.f;
            if (VEC) {
                constexpr int kU = 4;
                const float4 *x4 = reinterpret_cast<const float4 *>(x);
                const float4 *v4 = reinterpret_cast<const float4 *>(v);
                const int n4 = (int)(n / 4), step = 32 * wpr;
                float4 sv = make_float4(0.f, 0.f, 0.f, 0.f), ev = sv, g1 = sv, g2 = sv;
                for (int q0 = part * 32 + lane; q0 < n4; q0 += step * kU) {
                    float4 xv[kU];
#pragma unroll
                    for (int k = 0; k < kU; ++k)
                        if (q0 + k * step < n4)
                            xv[k] = x4[q0 + k * step];
#pragma unroll
                    for (int k = 0; k < kU; ++k) {
                        const int q = q0 + k * step;
                        if (q < n4) {
                            const float4 b = FIRST && !staged ? make_float4(v_at(4 * q), v_at(4 * q + 1), v_at(4 * q + 2),
                                                                            v_at(4 * q + 3))
                                                              : v4[q];
                            dot2(sv.x, ev.x, xv[k].x, b.x);
                            dot2(sv.y, ev.y, xv[k].y, b.y);
                            dot2(sv.z, ev.z, xv[k].z, b.z);
                            dot2(sv.w, ev.w, xv[k].w, b.w);
                            if (FIRST) {
                                const float d0 = xv[k].x - rhat * d.C[4 * q];
                                const float d1 = xv[k].y - rhat * d.C[4 * q + 1];
                                const float d2 = xv[k].z - rhat * d.C[4 * q + 2];
                                const float d3 = xv[k].w - rhat * d.C[4 * q + 3];
                                g1.x = fmaf(xv[k].x, xv[k].x, g1.x);
                                g1.y = fmaf(xv[k].y, xv[k].y, g1.y);
                                g1.z = fmaf(xv[k].z, xv[k].z, g1.z);
                                g1.w = fmaf(xv[k].w, xv[k].w, g1.w);
                                g2.x = fmaf(d0, d0, g2.x);
                                g2.y = fmaf(d1, d1, g2.y);
                                g2.z = fmaf(d2, d2, g2.z);
                                g2.w = fmaf(d3, d3, g2.w);
                            }
                        }
                    }
                }
                s = sv.x;
                e = ev.x;
                add2(s, e, sv.y, ev.y);
                add2(s, e, sv.z, ev.z);
                add2(s, e, sv.w, ev.w);
                f1 = (g1.x + g1.y) + (g1.z + g1.w);
                f2 = (g2.x + g2.y) + (g2.z + g2.w);
            } else {
                constexpr int kU = 8;
                const int64_t step = 32 * wpr;
                for (int64_t j0 = part * 32 + lane; j0 < n; j0 += step * kU) {
                    float xv[kU], vv[kU];
#pragma unroll
                    for (int k = 0; k < kU; ++k)
                        if (j0 + k * step < n) {
                            xv[k] = x[j0 + k * step];
                            vv[k] = v_at(j0 + k * step);
                        }
#pragma unroll
                    for (int k = 0; k < kU; ++k)
                        if (j0 + k * step < n) {
                            dot2(s, e, xv[k], vv[k]);
                            if (FIRST) {
                                const float t = xv[k] - rhat * d.C[j0 + k * step];
                                f1 = fmaf(xv[k], xv[k], f1);
                                f2 = fmaf(t, t, f2);
                            }
                        }
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float s2 = __shfl_xor_sync(0xffffffffu, s, o);
            const float e2 = __shfl_xor_sync(0xffffffffu, e, o);
            add2(s, e, s2, e2);
        }
        if (FIRST) {
            f1 = warp_sum(f1);
            f2 = warp_sum(f2);
        }
        if (lane == 0) {
            ue[warp] = make_float2(s, e);
            if (FIRST)
                nf[warp] = make_float2(f1, f2);
        }
        __syncthreads();
        if (tid < rpb) {
            float us_ = ue[tid * wpr].x, ue_ = ue[tid * wpr].y;
            for (int k = 1; k < wpr; ++k)
                add2(us_, ue_, ue[tid * wpr + k].x, ue[tid * wpr + k].y);
            const double u = (double)us_ + (double)ue_;
            u2 += u * u;
            us[tid] = us_ + ue_;        // 0 for a row past the block's range
            if (FIRST)
                for (int k = 0; k < wpr; ++k) {
                    n1 += (double)nf[tid * wpr + k].x;
                    n2 += (double)nf[tid * wpr + k].y;
                }
        }
        __syncthreads();
        const int live = (int)(r1 - r < rpb ? r1 - r : rpb);
        const float *x = d.xi + r * n;
        if (VEC) {
            const int n4 = (int)(n / 4);
            float4 *w4 = reinterpret_cast<float4 *>(wacc);
            for (int q = tid; q < n4; q += kThreads) {
                float4 acc = w4[q];
                float4 xv[kWarps];
#pragma unroll
                for (int k = 0; k < kWarps; ++k)
                    if (k < live)
                        xv[k] = reinterpret_cast<const float4 *>(x)[(int64_t)k * n4 + q];
#pragma unroll
                for (int k = 0; k < kWarps; ++k)
                    if (k < live) {
                        acc.x = fmaf(xv[k].x, us[k], acc.x);
                        acc.y = fmaf(xv[k].y, us[k], acc.y);
                        acc.z = fmaf(xv[k].z, us[k], acc.z);
                        acc.w = fmaf(xv[k].w, us[k], acc.w);
                    }
                w4[q] = acc;
            }
        } else {
            for (int64_t j = tid; j < n; j += kThreads) {
                float acc = wacc[j];
                float xv[kWarps];
#pragma unroll
                for (int k = 0; k < kWarps; ++k)
                    if (k < live)
                        xv[k] = x[k * n + j];
#pragma unroll
                for (int k = 0; k < kWarps; ++k)
                    if (k < live)
                        acc = fmaf(xv[k], us[k], acc);
                wacc[j] = acc;
            }
        }
    }
    // The block's share of xi^T u (each thread the columns it owns), its sums.
    if (staged) {
        float *out = d.wpart + (int64_t)blockIdx.x * n;
        if (VEC)
            for (int64_t j = tid; j < n / 4; j += kThreads)
                reinterpret_cast<float4 *>(out)[j] = reinterpret_cast<const float4 *>(wacc)[j];
        else
            for (int64_t j = tid; j < n; j += kThreads)
                out[j] = wacc[j];
    }
    if (tid < kWarps) {
        dd[0][tid] = u2;
        dd[1][tid] = n1;
        dd[2][tid] = n2;
    }
    __syncthreads();
    if (tid < (FIRST ? 3 : 1)) {
        double t = 0.0;
        for (int k = 0; k < kWarps; ++k)
            t += dd[tid][k];
        if (tid == 0)
            d.upart[blockIdx.x] = t;
        else
            d.npart[2 * blockIdx.x + tid - 1] = t;
    }
}

template <bool FIRST>
auto diag_rows_kernel(int64_t n)
{
    return n % 4 != 0             ? rikfad_diag_rows_kernel<FIRST, kDiagScalar>
           : n <= kDiagStageCols ? rikfad_diag_rows_kernel<FIRST, kDiagVecStaged>
                                 : rikfad_diag_rows_kernel<FIRST, kDiagVec>;
}

// Column kernel: cpb columns a block, 32 at a time.  The next iterate v =
// (xi^T u) ||v||^2 / ||u||^2 (whose length stays near the last one's and equals
// it once converged): warp k of W adds the row blocks k, k + W, ... in order, then
// warp 0 the W warp sums; its squares go to the other half of v2part.
// Block 0 forms the quotient and tests convergence: |sigma^2 - previous| <= tol
// sigma^2 from the second iteration on, or max_iters, or nothing left to
// iterate on.  Once it is done, the launches that follow hand that on.
__global__ void __launch_bounds__(1024) rikfad_diag_cols_kernel(DiagParams d)
{
    constexpr int kU = 8;
    __shared__ float part[32][32];
    const int nwarps = blockDim.x >> 5;
    __shared__ double tot[4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n = d.td.cols;
    wait_for_predecessor();
    allow_successor_launch();
    if (d.st->done) {           // every block of the launch
        if (blockIdx.x == 0 && threadIdx.x == 0)
            d.st_next->done = 1;
        return;
    }
    const int it = d.st->it + 1;
    // Totals, each by one warp: ||u||^2, ||v||^2, and (block 0, first iteration) the norms.
    if (warp < 2 || (it == 1 && blockIdx.x == 0 && warp < 4)) {
        const double *src = warp == 0 ? d.upart : warp == 1 ? d.v2part + (int64_t)d.parity * d.ncb : d.npart + (warp - 2);
        const int cnt = warp == 1 ? d.ncb : d.nblk, stride = warp < 2 ? 1 : 2;
        double a = 0.0;
        for (int b = lane; b < cnt; b += 32)
            a += src[b * stride];
        a = warp_sum_f64(a);
        if (lane == 0)
            tot[warp] = a;
    }
    double q = 0.0;             // warp 0: squares of the next iterate
    for (int64_t c0 = 0; c0 < d.cpb; c0 += 32) {
        const int64_t j = (int64_t)blockIdx.x * d.cpb + c0 + lane;
        float acc = 0.f;
        if (j < n) {
            for (int g0 = warp; g0 < d.nblk; g0 += nwarps * kU) {
                float t[kU];
#pragma unroll
                for (int k = 0; k < kU; ++k) {
                    const int g = g0 + k * nwarps;
                    t[k] = g < d.nblk ? d.wpart[(int64_t)g * n + j] : 0.f;
                }
#pragma unroll
                for (int k = 0; k < kU; ++k)
                    acc += t[k];
            }
        }
        __syncthreads();        // warp 0 has read the last 32 columns' sums
        part[warp][lane] = acc;
        __syncthreads();
        if (warp == 0 && j < n) {
            float sum = 0.f;
#pragma unroll 8
            for (int k = 0; k < nwarps; ++k)
                sum += part[k][lane];
            const float vn = tot[0] > 0.0 ? (float)((double)sum * (tot[1] / tot[0])) : 0.f;
            d.v[j] = vn;
            q += (double)vn * (double)vn;
        }
    }
    if (warp != 0)
        return;
    q = warp_sum_f64(q);
    if (lane == 0)
        d.v2part[(int64_t)(d.parity ^ 1) * d.ncb + blockIdx.x] = q;
    if (blockIdx.x == 0 && lane == 0) {
        const double u2 = tot[0], v2 = tot[1];
        DiagState s = *d.st;
        const double prev = s.sigma2;
        if (it == 1) {
            s.f2 = tot[2];
            s.e2 = tot[3];
        }
        s.it = it;
        // An iterate that underflowed to zero leaves the last quotient.
        if (v2 > 0.0 && (u2 > 0.0 || it == 1))
            s.sigma2 = u2 / v2;
        s.done = !(u2 > 0.0) || it >= d.max_iters || (it > 1 && fabs(s.sigma2 - prev) <= d.tol * s.sigma2);
        *d.st_next = s;
        if (s.done || d.last)
            *d.host = s;
    }
}

}  // namespace rikfad
