// rikfad_kernels.cuh -- sm_103a kernels of the R-iKFAD optimiser step.
//
// The method (BACD splitting, Appendix A of the paper):
//   B  P^(B) = P_n - h G
//   A  X_{n+1} = X_n + h P^(B)
//   C  P^(1) = P^(B) exp(-(h/2) xi~_n),  xi~ = R C^T / (1^T R + eps)   (Eq. xi_def)
//      R_{n+1} = e^{-alpha h} R_n + k [P^(1)]^2 1_n,  k = (1 - e^{-alpha h})/(mu alpha)
//      C_{n+1} = e^{-alpha h} C_n + k ([P^(1)]^2)^T 1_m
//      P^(2) = P^(1) exp(-(h/2) xi~_{n+1})
//   D  P_{n+1} = P^(2) e^{-gamma h}
//
// Scheduling.  R_{n+1}, C_{n+1} are reductions over the whole matrix, so
// P^(2) cannot be formed in the same pass that produces P^(1).  The step
// kernel therefore stores P^(1) and the NEXT step applies the pending factor
// exp(-(h_prev/2) xi~_{n+1}) e^{-gamma h_prev} on the fly, with the factors
// that the finalise kernel of this step wrote.  Every element is read once
// and written once per step (grad, X, P read; X, P written).  When the step
// size does not change, the pending factor and this step's first half-damp
// are the same exponential and one exp2 serves both.
//
// Reductions are deterministic: a warp owns a row segment (row sums by a
// fixed shuffle tree), each lane owns fixed columns (column sums accumulate
// row by row in lane-private shared memory, then across warps in warp order,
// then across the blocks of a panel in slot order in the finalise kernel).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "rikfad_checks.cuh"
#include "rikfad_plan.hpp"

namespace rikfad {

// Non-finite guard.  A kernel that produces a non-finite factor, friction or
// denominator records the tensor: the lowest such index in device memory
// (atomicMin; INT32_MAX when there is none) and a flag in page-locked host
// memory that the host reads without waiting for the device.
struct Guard {
    int32_t *first;
    volatile int32_t *host;
};

__device__ __forceinline__ void report_nonfinite(const Guard &g, int tensor)
{
    atomicMin(g.first, tensor);
    *g.host = 1;
}

struct StepParams {
    const TensorDev *tensors;
    const PanelDev *panels;
    const PieceDev *pieces;
    const int32_t *block_piece;
    const TileGroupDev *groups;   // rikfad_elements_kernel
    float *const *xptr;        // ntensors device pointers
    const void *const *gptr;
    float *const *pptr;
    float *fac;                // R, C of matrices; friction of vectors
    float *rowpart;
    float *colpart;
    const float *spart;        // partial sums of R (denominators)
    float h;                   // step size
    float ex_cur;              // -(h/2) log2(e): exp(-(h/2) xi) = exp2(ex_cur xi)
    float ex_prev;             // -(h_prev/2) log2(e)
    float damp_prev;           // e^{-gamma h_prev}
    float damp_cur;            // e^{-gamma h} (vectors finish D inside the step)
    float decay;               // e^{-alpha h}
    float gain;                // (1 - e^{-alpha h})/(mu alpha)
    float eps;                 // eps_stab
    int band_width;            // WIDE: floats of a warp's column accumulators, columns of the widest band
    Guard guard;
    CheckBounds chk;           // read by checked builds only
};

// ---------------------------------------------------------------- helpers

// Programmatic dependent launch: the kernels of a step are launched so that
// they may start before their predecessor in the stream has finished; they
// run this wait before touching any data the predecessor may write, and let
// their own successor start launching early.
__device__ __forceinline__ void wait_for_predecessor()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ void allow_successor_launch()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ float warp_sum(float v)
{
    // Butterfly: float addition is commutative, so every lane ends with the
    // bitwise-same total.
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// 1^T R of a matrix from the finalise kernel's partial sums, in a fixed order
// (identical in every warp that computes it).
__device__ __forceinline__ float row_total(const float *spart, const TensorDev &td)
{
    const int lane = threadIdx.x & 31;
    float v = 0.f;
    for (int c = lane; c < td.spart_cnt; c += 32)
        v += spart[td.spart_off + c];
    return warp_sum(v);
}

// 1 / (1^T R + eps), with the friction set to zero when the denominator is
// zero (eps = 0 and R = 0; Theorem 3's convention).
__device__ __forceinline__ float inv_denominator(float s, float eps)
{
    const float den = s + eps;
    return den == 0.f ? 0.f : 1.f / den;
}

template <typename GT> struct Grad8;

template <> struct Grad8<float> {
    float v[8];
    __device__ __forceinline__ void load(const float *g)
    {
        const float4 a = __ldcs(reinterpret_cast<const float4 *>(g));
        const float4 b = __ldcs(reinterpret_cast<const float4 *>(g) + 1);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    }
    __device__ __forceinline__ float get(int e) const { return v[e]; }
};

template <> struct Grad8<__nv_bfloat16> {
    uint32_t w[4];
    __device__ __forceinline__ void load(const __nv_bfloat16 *g)
    {
        const uint4 a = __ldcs(reinterpret_cast<const uint4 *>(g));
        w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
    }
    // bf16 -> f32 is exact: the bf16 bits are the high half of the f32.
    __device__ __forceinline__ float get(int e) const
    {
        const uint32_t word = w[e >> 1];
        return __uint_as_float((e & 1) ? (word & 0xffff0000u) : (word << 16));
    }
};

__device__ __forceinline__ float grad_at(const float *g, int64_t i) { return __ldcs(g + i); }
__device__ __forceinline__ float grad_at(const __nv_bfloat16 *g, int64_t i)
{
    return __bfloat162float(__ushort_as_bfloat16(__ldcs(reinterpret_cast<const unsigned short *>(g + i))));
}

__device__ __forceinline__ void load8(const float *p, float (&v)[8])
{
    const float4 a = __ldcs(reinterpret_cast<const float4 *>(p));
    const float4 b = __ldcs(reinterpret_cast<const float4 *>(p) + 1);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

__device__ __forceinline__ void store8(float *p, const float (&v)[8])
{
    __stcs(reinterpret_cast<float4 *>(p), make_float4(v[0], v[1], v[2], v[3]));
    __stcs(reinterpret_cast<float4 *>(p) + 1, make_float4(v[4], v[5], v[6], v[7]));
}

// ------------------------------------------- one element, matrix rule
//
// p_hat is the stored P^(1) of the previous step.  Returns P^(1) of this step
// and updates x.  e_cur = exp(-(h/2) xi~_ij), e_prev = exp(-(h_prev/2) xi~_ij),
// both with the current factors (= R_{n}, C_{n} of this step).
__device__ __forceinline__ float matrix_element(float &x, float p_hat, float g, float e_cur,
                                                float e_prev, const StepParams &a)
{
    const float p_n = (p_hat * e_prev) * a.damp_prev;   // pending C half-damp, then D
    const float p_b = fmaf(-a.h, g, p_n);                 // B
    x = fmaf(a.h, p_b, x);                                // A
    return p_b * e_cur;                                   // C, first half-damp
}

// ------------------------------------------------- matrix piece, 8-wide

// 256-column chunks whose loads are issued together (registers: ~20 per chunk).
#ifndef RIKFAD_CHUNK_GROUP
#define RIKFAD_CHUNK_GROUP 1
#endif

// ACCUM: add each row's squares into the warp's column buffer (several rows
// per warp); otherwise store them (one row per warp, buffer not cleared).
// RPW rows per warp (1, 2, 4 or 8; panels of at most kPanelMax / RPW columns):
// each of the warp's RPW lane groups takes its own row, 256 / RPW columns per
// chunk, so a panel whose width is not a multiple of 256 still loads 256
// columns per warp and round trip; group h accumulates its columns at
// red[warp][h * kPanelMax / RPW + c].
template <typename GT, bool REUSE, bool ACCUM = true, int RPW = 1>
__device__ __forceinline__ void matrix_piece_vec(const StepParams &a, const PieceDev &pc,
                                                 const TensorDev &td, const PanelDev &pd,
                                                 const float *Cs, float *red, float inv,
                                                 const int stride = kPanelMax)
{
    constexpr int kRowLanes = 32 / RPW;                 // lanes per row
    constexpr int kRowChunk = kRowLanes * 8;            // columns per chunk of one row
    constexpr int kRowsPerWarp = RPW;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rl = lane & (kRowLanes - 1), half = lane / kRowLanes;   // lane group = row
    const int64_t n = td.cols;
    const int w = pd.width;
    const int nch = RPW > 1 ? (w + kRowChunk - 1) / kRowChunk : pd.nch;
    float *X = a.xptr[pc.tensor];
    const GT *G = static_cast<const GT *>(a.gptr[pc.tensor]);
    float *P = a.pptr[pc.tensor];
    const float *R = a.fac + td.fac_off;
    float *rowpart = a.rowpart + td.rowpart_off + (int64_t)(pc.panel - td.panel0) * td.rows;
    float *myred = red + warp * stride + half * (kPanelMax / RPW);

    for (int64_t r0 = pc.begin + kRowsPerWarp * warp; r0 < pc.end; r0 += kRowsPerWarp * kWarps) {
        const int64_t row = r0 + half;
        const bool live = RPW == 1 || row < pc.end;     // ragged piece: trailing lane groups idle
        const float rhat = live ? R[row] * inv : 0.f;
        const float a_cur = a.ex_cur * rhat;
        const float a_prev = REUSE ? a_cur : a.ex_prev * rhat;
        const int64_t base = row * n + pd.col0;

        // RIKFAD_CHUNK_GROUP chunks at a time: every load of the group is
        // issued before any arithmetic on it.
        float racc = 0.f;
#pragma unroll 1
        for (int g0 = 0; g0 < nch; g0 += RIKFAD_CHUNK_GROUP) {
            float xv[RIKFAD_CHUNK_GROUP][8], pv[RIKFAD_CHUNK_GROUP][8];
            Grad8<GT> gv[RIKFAD_CHUNK_GROUP];
#pragma unroll
            for (int k = 0; k < RIKFAD_CHUNK_GROUP; ++k) {
                const int c = (g0 + k) * kRowChunk + rl * 8;
                if (live && c < w) {
                    gv[k].load(G + base + c);
                    load8(X + base + c, xv[k]);
                    load8(P + base + c, pv[k]);
                }
            }
#pragma unroll
            for (int k = 0; k < RIKFAD_CHUNK_GROUP; ++k) {
                const int c = (g0 + k) * kRowChunk + rl * 8;
                if (live && c < w) {
                    const float4 c0 = *reinterpret_cast<const float4 *>(Cs + c);
                    const float4 c1 = *reinterpret_cast<const float4 *>(Cs + c + 4);
                    const float cv[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
                    float q[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const float e_cur = exp2f(a_cur * cv[e]);
                        const float e_prev = REUSE ? e_cur : exp2f(a_prev * cv[e]);
                        const float p1 = matrix_element(xv[k][e], pv[k][e], gv[k].get(e), e_cur,
                                                        e_prev, a);
                        pv[k][e] = p1;
                        q[e] = p1 * p1;
                        racc += q[e];
                    }
                    store8(X + base + c, xv[k]);
                    store8(P + base + c, pv[k]);
                    float4 *r4 = reinterpret_cast<float4 *>(myred + c);
                    if (ACCUM) {
                        float4 r0 = r4[0], r1 = r4[1];
                        r0.x += q[0]; r0.y += q[1]; r0.z += q[2]; r0.w += q[3];
                        r1.x += q[4]; r1.y += q[5]; r1.z += q[6]; r1.w += q[7];
                        r4[0] = r0;
                        r4[1] = r1;
                    } else {
                        r4[0] = make_float4(q[0], q[1], q[2], q[3]);
                        r4[1] = make_float4(q[4], q[5], q[6], q[7]);
                    }
                }
            }
        }
        if (RPW > 1) {
#pragma unroll
            for (int o = kRowLanes / 2; o > 0; o >>= 1)
                racc += __shfl_xor_sync(0xffffffffu, racc, o);
        } else {
            racc = warp_sum(racc);
        }
        if (live && rl == 0)
            rowpart[row] = racc;
    }
}

// --------------------------------------------------------- matrix band
//
// Whole rows of a band (pd spans it), one row per warp, in 256-column chunks; a
// last partial chunk of at most half a chunk is loaded together with the chunk
// before it, so that it costs no round trip of its own.
template <typename GT, bool REUSE>
__device__ __forceinline__ void matrix_band(const StepParams &a, const PieceDev &pc, const TensorDev &td,
                                            const PanelDev &pd, const float *Cs, float *red, float inv,
                                            const int stride)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n = td.cols;
    const int w = pd.width, tail = w % kChunk;
    const int w1 = tail <= kChunk / 2 ? w - tail - kChunk : w;      // columns before the joint pair
    float *X = a.xptr[pc.tensor];
    const GT *G = static_cast<const GT *>(a.gptr[pc.tensor]);
    float *P = a.pptr[pc.tensor];
    const float *R = a.fac + td.fac_off;
    float *rowpart = a.rowpart + td.rowpart_off + (int64_t)(pc.panel - td.panel0) * td.rows;
    float *myred = red + warp * stride;

    for (int64_t row = pc.begin + warp; row < pc.end; row += kWarps) {
        const float rhat = R[row] * inv;
        const float a_cur = a.ex_cur * rhat;
        const float a_prev = REUSE ? a_cur : a.ex_prev * rhat;
        const int64_t base = row * n + pd.col0;
        float racc = 0.f;
        auto update = [&](int c, float (&xv)[8], float (&pv)[8], const Grad8<GT> &gv) {
            const float4 c0 = *reinterpret_cast<const float4 *>(Cs + c);
            const float4 c1 = *reinterpret_cast<const float4 *>(Cs + c + 4);
            const float cv[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
            float q[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float e_cur = exp2f(a_cur * cv[e]);
                const float e_prev = REUSE ? e_cur : exp2f(a_prev * cv[e]);
                const float p1 = matrix_element(xv[e], pv[e], gv.get(e), e_cur, e_prev, a);
                pv[e] = p1;
                q[e] = p1 * p1;
                racc += q[e];
            }
            store8(X + base + c, xv);
            store8(P + base + c, pv);
            float4 *r4 = reinterpret_cast<float4 *>(myred + c);
            float4 s0 = r4[0], s1 = r4[1];
            s0.x += q[0]; s0.y += q[1]; s0.z += q[2]; s0.w += q[3];
            s1.x += q[4]; s1.y += q[5]; s1.z += q[6]; s1.w += q[7];
            r4[0] = s0;
            r4[1] = s1;
        };
        int c = lane * 8;
#pragma unroll 1
        for (; c < w1; c += kChunk) {
            Grad8<GT> gv;
            float xv[8], pv[8];
            gv.load(G + base + c);
            load8(X + base + c, xv);
            load8(P + base + c, pv);
            update(c, xv, pv, gv);
        }
        if (w1 < w) {
            const int t = c + kChunk;
            Grad8<GT> gv, gt;
            float xv[8], pv[8], xt[8], pt[8];
            gv.load(G + base + c);
            load8(X + base + c, xv);
            load8(P + base + c, pv);
            if (t < w) {
                gt.load(G + base + t);
                load8(X + base + t, xt);
                load8(P + base + t, pt);
            }
            update(c, xv, pv, gv);
            if (t < w)
                update(t, xt, pt, gt);
        }
        racc = warp_sum(racc);
        if (lane == 0)
            rowpart[row] = racc;
    }
}

// ----------------------------------------------- matrix piece, ragged
// For matrices whose rows are not 8-aligned (cols % 8 != 0): rows start at any
// element address, so lanes take single elements; a load instruction of a
// warp covers consecutive elements of a row.
//
// Bound by the bytes in flight: each lane issues its U loads of every array
// before any arithmetic (U = 8: 256 elements of each array per warp, as on the
// 8-wide path).  RPW rows per warp as there, so that a narrow panel fills the
// warp too: each of the RPW lane groups takes its own row.  Measured on a
// 10007 x 3001 matrix with fp32 gradients (600 MB a step, whole step): one load
// of each array in flight per lane 281 us, U = 4 144, U = 8 121 and, with
// streaming hints, 115 (5.2 TB/s); U = 16 was no faster (122 without hints).
template <typename GT, bool REUSE, bool ACCUM = true, int RPW = 1, int U = 8>
__device__ __forceinline__ void matrix_piece_ragged(const StepParams &a, const PieceDev &pc,
                                                    const TensorDev &td, const PanelDev &pd,
                                                    const float *Cs, float *red, float inv,
                                                    const int stride = kPanelMax)
{
    constexpr int kRowLanes = 32 / RPW;                 // lanes per row
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rl = lane & (kRowLanes - 1), half = lane / kRowLanes;   // lane group = row
    const int64_t n = td.cols;
    const int w = pd.width;
    float *X = a.xptr[pc.tensor];
    const GT *G = static_cast<const GT *>(a.gptr[pc.tensor]);
    float *P = a.pptr[pc.tensor];
    const float *R = a.fac + td.fac_off;
    float *rowpart = a.rowpart + td.rowpart_off + (int64_t)(pc.panel - td.panel0) * td.rows;
    float *myred = red + warp * stride + half * (kPanelMax / RPW);

    for (int64_t r0 = pc.begin + RPW * warp; r0 < pc.end; r0 += RPW * kWarps) {
        const int64_t row = r0 + half;
        const bool live = RPW == 1 || row < pc.end;     // ragged piece: trailing lane groups idle
        const float rhat = live ? R[row] * inv : 0.f;
        const float a_cur = a.ex_cur * rhat;
        const float a_prev = REUSE ? a_cur : a.ex_prev * rhat;
        const int64_t base = row * n + pd.col0 + rl;
        float *xr = X + base, *pr = P + base;
        const GT *gr = G + base;
        const int wl = live ? w : 0;
        float racc = 0.f;
#pragma unroll 1
        for (int c0 = rl; c0 < wl; c0 += kRowLanes * U) {
            float x[U], p[U], g[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (c0 + kRowLanes * u < w) {
                    g[u] = grad_at(gr, kRowLanes * u);
                    x[u] = __ldcs(xr + kRowLanes * u);
                    p[u] = __ldcs(pr + kRowLanes * u);
                }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int c = c0 + kRowLanes * u;
                if (c < w) {
                    const float cv = Cs[c];
                    const float e_cur = exp2f(a_cur * cv);
                    const float e_prev = REUSE ? e_cur : exp2f(a_prev * cv);
                    const float p1 = matrix_element(x[u], p[u], g[u], e_cur, e_prev, a);
                    __stcs(xr + kRowLanes * u, x[u]);
                    __stcs(pr + kRowLanes * u, p1);
                    const float q = p1 * p1;
                    racc += q;
                    if (ACCUM)
                        myred[c] += q;
                    else
                        myred[c] = q;
                }
            }
            xr += kRowLanes * U;
            pr += kRowLanes * U;
            gr += kRowLanes * U;
        }
#pragma unroll
        for (int o = kRowLanes / 2; o > 0; o >>= 1)
            racc += __shfl_xor_sync(0xffffffffu, racc, o);
        if (live && rl == 0)
            rowpart[row] = racc;
    }
}

// ------------------------------------------ element-wise rule (vectors)
//
// Element-wise iKFAD (Section 2, "Memory Complexity"): the friction xi of the
// element is local, so the whole step -- including the second half-damp and
// D -- completes here and P holds P_{n+1}.
__device__ __forceinline__ void vector_element(float &x, float &p, float &xi, float g,
                                               const StepParams &a)
{
    const float p_b = fmaf(-a.h, g, p);                       // B
    x = fmaf(a.h, p_b, x);                                    // A
    const float p1 = p_b * exp2f(a.ex_cur * xi);              // C, first half-damp
    xi = fmaf(a.gain, p1 * p1, a.decay * xi);                 // C, friction filter
    p = (p1 * exp2f(a.ex_cur * xi)) * a.damp_cur;             // C, second half-damp; D
}

template <typename GT>
__device__ __forceinline__ void vector_piece(const StepParams &a, const PieceDev &pc,
                                             const TensorDev &td)
{
    float *X = a.xptr[pc.tensor];
    const GT *G = static_cast<const GT *>(a.gptr[pc.tensor]);
    float *P = a.pptr[pc.tensor];
    float *XI = a.fac + td.fac_off;
    const int64_t b0 = pc.begin;                // multiple of 8 (planner)
    const int64_t nvec = (pc.end - b0) / 8;
    bool bad = false;
    for (int64_t v = threadIdx.x; v < nvec; v += kThreads) {
        const int64_t e0 = b0 + v * 8;
        Grad8<GT> g;
        g.load(G + e0);
        float x[8], p[8], xi[8];
        load8(X + e0, x);
        load8(P + e0, p);
        load8(XI + e0, xi);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            vector_element(x[e], p[e], xi[e], g.get(e), a);
            bad |= !isfinite(xi[e]);
        }
        store8(X + e0, x);
        store8(P + e0, p);
        store8(XI + e0, xi);
    }
    for (int64_t e = b0 + nvec * 8 + threadIdx.x; e < pc.end; e += kThreads) {
        float x = X[e], p = P[e], xi = XI[e];
        vector_element(x, p, xi, grad_at(G, e), a);
        bad |= !isfinite(xi);
        X[e] = x;
        P[e] = p;
        XI[e] = xi;
    }
    // The friction is d xi + k [P^(1)]^2: non-finite exactly when the
    // half-damped momentum (or the friction before) is.
    if (bad)
        report_nonfinite(a.guard, pc.tensor);
}

// ------------------------------ matrix with element-wise friction (full iKFAD)
//
// Full iKFAD on a matrix (Eqs. ikfad_1 to ikfad_3, the same expression as
// vector_element) with the squares of the half-damped momentum P^(1) also
// summed per row and per column, so the matrix's R, C follow R-iKFAD's factor
// filter as shadow factors of the same trajectory (the comparison of the
// paper's Section 4.4).  P holds P_{n+1}.
__device__ __forceinline__ float full_element(float &x, float &p, float &xi, float g,
                                              const StepParams &a)
{
    const float p_b = fmaf(-a.h, g, p);                       // B
    x = fmaf(a.h, p_b, x);                                    // A
    const float p1 = p_b * exp2f(a.ex_cur * xi);              // C, first half-damp
    xi = fmaf(a.gain, p1 * p1, a.decay * xi);                 // C, friction filter
    p = (p1 * exp2f(a.ex_cur * xi)) * a.damp_cur;             // C, second half-damp; D
    return p1 * p1;
}

//
// Rows per warp and loads in flight as matrix_piece_vec (VEC) and
// matrix_piece_ragged: one row per warp left most lanes of a narrow panel idle
// (bf16 gradients, share of the 6.8 TB/s floor: width 24 0.20 -> 0.76, 64 0.49 ->
// 0.88, 640 0.71 -> 0.87, 9000 0.39 -> 0.81).
template <typename GT, bool VEC, int RPW, int U = 8>
__device__ __forceinline__ void matrix_piece_full(const StepParams &a, const PieceDev &pc,
                                                  const TensorDev &td, const PanelDev &pd,
                                                  float *red)
{
    constexpr int kRowLanes = 32 / RPW;                 // lanes per row
    constexpr int kU = U;                               // ragged: elements per lane and pass
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rl = lane & (kRowLanes - 1), half = lane / kRowLanes;
    const int64_t n = td.cols;
    const int w = pd.width;
    float *X = a.xptr[pc.tensor];
    const GT *G = static_cast<const GT *>(a.gptr[pc.tensor]);
    float *P = a.pptr[pc.tensor];
    float *XI = a.fac + td.xi_off;
    float *rowpart = a.rowpart + td.rowpart_off + (int64_t)(pc.panel - td.panel0) * td.rows;
    float *myred = red + warp * kPanelMax + half * (kPanelMax / RPW);
    for (int64_t r0 = pc.begin + RPW * warp; r0 < pc.end; r0 += RPW * kWarps) {
        const int64_t row = r0 + half;
        const bool live = RPW == 1 || row < pc.end;
        const int64_t base = row * n + pd.col0;
        const int wl = live ? w : 0;
        float racc = 0.f;
        if (VEC) {
#pragma unroll 1
            for (int c = rl * 8; c < wl; c += kRowLanes * 8) {
                Grad8<GT> gv;
                gv.load(G + base + c);
                float x[8], p[8], xi[8];
                load8(X + base + c, x);
                load8(P + base + c, p);
                load8(XI + base + c, xi);
                float q[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    q[e] = full_element(x[e], p[e], xi[e], gv.get(e), a);
                    racc += q[e];
                }
                store8(X + base + c, x);
                store8(P + base + c, p);
                store8(XI + base + c, xi);
                float4 *r4 = reinterpret_cast<float4 *>(myred + c);
                float4 r0 = r4[0], r1 = r4[1];
                r0.x += q[0]; r0.y += q[1]; r0.z += q[2]; r0.w += q[3];
                r1.x += q[4]; r1.y += q[5]; r1.z += q[6]; r1.w += q[7];
                r4[0] = r0;
                r4[1] = r1;
            }
        } else {
#pragma unroll 1
            for (int c0 = rl; c0 < wl; c0 += kRowLanes * kU) {
                float x[kU], p[kU], xi[kU], g[kU];
#pragma unroll
                for (int u = 0; u < kU; ++u)
                    if (c0 + kRowLanes * u < w) {
                        const int64_t i = base + c0 + kRowLanes * u;
                        g[u] = grad_at(G, i);
                        x[u] = __ldcs(X + i);
                        p[u] = __ldcs(P + i);
                        xi[u] = __ldcs(XI + i);
                    }
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int c = c0 + kRowLanes * u;
                    if (c < w) {
                        const float q = full_element(x[u], p[u], xi[u], g[u], a);
                        __stcs(X + base + c, x[u]);
                        __stcs(P + base + c, p[u]);
                        __stcs(XI + base + c, xi[u]);
                        racc += q;
                        myred[c] += q;
                    }
                }
            }
        }
#pragma unroll
        for (int o = kRowLanes / 2; o > 0; o >>= 1)
            racc += __shfl_xor_sync(0xffffffffu, racc, o);
        if (live && rl == 0)
            rowpart[row] = racc;
    }
}

// ------------------------------------------------------ the step kernel

// Blocks per SM the register budget is sized for (2: 128 registers/thread).
#ifndef RIKFAD_STEP_MIN_BLOCKS
#define RIKFAD_STEP_MIN_BLOCKS 2
#endif

// out[c] = the piece's column sums: warp wi's lane group h holds its share at
// red[wi * stride + h * kPanelMax / RPW + c]; added warp by warp, groups in
// order.
template <int RPW>
__device__ __forceinline__ void column_partials(const float *red, float *out, int w, const int stride = kPanelMax)
{
    for (int c = threadIdx.x; c < w; c += kThreads) {
        float s = 0.f;
#pragma unroll
        for (int wi = 0; wi < kWarps; ++wi)
#pragma unroll
            for (int h = 0; h < RPW; ++h)
                s += red[wi * stride + h * (kPanelMax / RPW) + c];
        out[c] = s;
    }
}

// Rows per warp (RPW of the row loops).  An 8-wide panel that is not a whole
// number of 256-column chunks takes 8 rows per warp up to 32 columns, 4 up to 64
// and 2 up to kPanelMax / 2 columns; every other one takes 1.  A ragged panel
// takes as many as leave every lane its 8 elements: 8, 4, 2 up to 32, 64, 128.
// 40 M elements of width 24, bf16: 4 rows per warp 0.43 of the 6.8 TB/s floor, 8
// rows 0.64.
__host__ __device__ __forceinline__ int rows_per_warp(bool vec, int w)
{
    if (vec ? (w % kChunk == 0 || w > kPanelMax / 2) : w > kChunk / 2)
        return 1;
    return w <= kChunk / 8 ? 8 : w <= kChunk / 4 ? 4 : 2;
}

template <int N>
struct RowsPerWarp {
    static constexpr int value = N;
};

// SHADOW: the instantiation for handles whose matrices all keep element-wise
// friction with shadow factors (the R-iKFAD instantiations carry no code for
// it, nor it any for them).  RAGGED: how much of the list lies in matrices whose
// rows are not 8-aligned (RaggedKind).  The batched loops of kManyRagged take 126 to
// 128 registers, WIDE 118 to 122 and SHADOW 116, where the others take 103 to 109: two
// blocks of up to 112 leave an SM the 8192 registers of a finalise block, which can
// then wait beside them for the last one; beside the others it starts as they drain.
// WIDE: the instantiation for handles with bands, whose column accumulators lie
// in dynamic shared memory (40 M elements, bf16, panels / bands: width 1032 147 /
// 129 us, 1376 145 / 125, 1800 249 / 132, 2600 150 / 129, 9000 147 / 129; taking the
// rows' partial chunks 2 or 4 rows at a time after them instead: 130 to 143).
template <typename GT, bool REUSE, bool SHADOW = false, int RAGGED = kNoRagged, bool WIDE = false>
__global__ void __launch_bounds__(kThreads, RIKFAD_STEP_MIN_BLOCKS) rikfad_step_kernel(StepParams a)
{
    extern __shared__ __align__(16) float wide[];
    __shared__ __align__(16) float Cs_[WIDE ? 4 : kPanelMax];
    __shared__ __align__(16) float red_[WIDE ? 4 : kWarps * kPanelMax];
    float *red = WIDE ? wide : red_;
    const int stride = WIDE ? a.band_width : kPanelMax;
    float *Cs = WIDE ? wide + kWarps * stride : Cs_;
    const int b = blockIdx.x;
    if (!RK_DEV_CHECK(a.chk, b < a.chk.nblocks, kChkBlock))
        return;
    const int q0 = a.block_piece[b], q1 = a.block_piece[b + 1];
    wait_for_predecessor();
    allow_successor_launch();
    if (!block_ok(a.chk, b, q0, q1))
        return;
    for (int q = q0; q < q1; ++q) {
        const PieceDev pc = a.pieces[q];
        if (!piece_tensor_ok(a.chk, pc))
            continue;
        const TensorDev td = a.tensors[pc.tensor];
        if (pc.kind == kElements) {
            if (vector_piece_ok(a.chk, pc, td, a.xptr[pc.tensor], a.gptr[pc.tensor], a.pptr[pc.tensor],
                                true))
                vector_piece<GT>(a, pc, td);
            continue;
        }
        if (!piece_panel_ok(a.chk, pc, td))
            continue;
        if (WIDE && pc.band == 0)
            continue;                           // walked with an earlier panel
        PanelDev pd = a.panels[pc.panel];
        // Block-uniform: every thread evaluates the same checks on the same
        // entries, so a skipped piece is skipped by the whole block.
        if (!matrix_piece_ok(a.chk, pc, td, pd, a.xptr[pc.tensor], a.gptr[pc.tensor], a.pptr[pc.tensor],
                             true))
            continue;
        if (WIDE && pc.band > 1) {              // pd spans the band
            if (!band_ok(a.chk, pc, td, pd, a.pieces, q, q1, a.band_width))
                continue;
            pd.width = pd.slot_stride;
        }
        const int w = pd.width;
        // Stage this panel's C, clear the column accumulators.
        const float *C = a.fac + td.fac_off + td.rows + pd.col0;
        for (int c = threadIdx.x; c < w; c += kThreads)
            Cs[c] = C[c];
        if (WIDE) {
            for (int i = threadIdx.x; i < kWarps * stride / 4; i += kThreads)
                reinterpret_cast<float4 *>(red)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
            for (int i = threadIdx.x; i < kWarps * kPanelMax; i += kThreads)
                red[i] = 0.f;
        }
        const float inv = inv_denominator(row_total(a.spart, td), a.eps);
        __syncthreads();
        if (WIDE && pc.band > 1) {
            matrix_band<GT, REUSE>(a, pc, td, pd, Cs, red, inv, stride);
            __syncthreads();
            column_partials<1>(red, a.colpart + pc.colpart_off, w, stride);
            __syncthreads();
            continue;
        }
        if (RAGGED == kFewRagged && !td.vec) {  // one element per lane and load
            if (SHADOW)
                matrix_piece_full<GT, false, 1, 1>(a, pc, td, pd, red);
            else
                matrix_piece_ragged<GT, REUSE, true, 1, 1>(a, pc, td, pd, Cs, red, inv, stride);
            __syncthreads();
            column_partials<1>(red, a.colpart + pc.colpart_off, w, stride);
            __syncthreads();
            continue;
        }
        // The kManyRagged instantiations carry fewer row loops (1, 2 and 4 rows per
        // warp; with SHADOW 1, and 8 for ragged panels up to 64 columns): with more
        // of them the compiler spills inside the loops (40 M elements, bf16, width
        // 500: 182 us with all, 141 so; as functions of their own 197).
        constexpr bool kMany = RAGGED == kManyRagged;
        const int rpw = SHADOW && kMany ? (td.vec || w > 64 ? 1 : 8) : rows_per_warp(!kMany || td.vec, w);
        // One call of the piece's path for its rows per warp.
        auto piece = [&](auto n) {
            constexpr int N = decltype(n)::value;
            if (SHADOW) {
                if (!kMany || (N == 1 && td.vec))
                    matrix_piece_full<GT, true, N>(a, pc, td, pd, red);
                else
                    matrix_piece_full<GT, false, N>(a, pc, td, pd, red);
            } else if (!kMany || td.vec) {
                matrix_piece_vec<GT, REUSE, true, N>(a, pc, td, pd, Cs, red, inv, stride);
            } else {
                matrix_piece_ragged<GT, REUSE, true, N>(a, pc, td, pd, Cs, red, inv);
            }
            __syncthreads();
            // Column partial sums of this piece, warps (and their lane groups) added in order.
            column_partials<N>(red, a.colpart + pc.colpart_off, w, stride);
        };
        if (rpw == 1)
            piece(RowsPerWarp<1>());
        else if (SHADOW && kMany)
            piece(RowsPerWarp<8>());
        else if (rpw == 2)
            piece(RowsPerWarp<2>());
        else if (kMany || rpw == 4)
            piece(RowsPerWarp<4>());
        else
            piece(RowsPerWarp<8>());
        __syncthreads();
    }
}

// ------------------------------------------ the step of element-wise tensors
//
// A list without matrices (full-friction iKFAD, vectors alone) carries no sums
// between elements, so its step needs no shares: one tile of 8 elements per
// thread per block, in memory order.  Bound by HBM, 26 B an element with bf16
// gradients; many small blocks in order keep the DRAM accesses in a narrow
// window.  Full-friction iKFAD over GPT2-S: 457 us a step with bf16 gradients
// (3.24 GB, 7.1 TB/s) and 489 with fp32, against 509 and 546 from two persistent
// blocks per SM with a contiguous share each.  64 registers and 4 blocks per SM:
// 5 and 6 blocks spill (514 and 538 us).
template <typename GT>
__global__ void __launch_bounds__(kThreads, 4) rikfad_elements_kernel(StepParams a)
{
    if (!RK_DEV_CHECK(a.chk, (int)blockIdx.x / kTileGroup < a.chk.ngroups, kChkBlock))
        return;
    const TileGroupDev group = a.groups[blockIdx.x / kTileGroup];
    PieceDev pc{};
    pc.kind = kElements;
    pc.tensor = group.tensor;
    if (!piece_tensor_ok(a.chk, pc))
        return;
    const TensorDev td = a.tensors[pc.tensor];
    pc.begin = (group.first + blockIdx.x % kTileGroup) * kTileElems;
    pc.end = pc.begin + kTileElems < td.rows ? pc.begin + kTileElems : td.rows;
    if (pc.begin >= td.rows)
        return;
    wait_for_predecessor();
    allow_successor_launch();
    if (vector_piece_ok(a.chk, pc, td, a.xptr[pc.tensor], a.gptr[pc.tensor], a.pptr[pc.tensor], true))
        vector_piece<GT>(a, pc, td);
}

}  // namespace rikfad
