// rikfad_aux_kernels.cuh -- the kernels around the step kernel: the factor
// finalise (run after every step), the canonical-momentum pass (checkpoints,
// tests) and the denominator read-back.  Included by rikfad.cu only.
#pragma once
#include "rikfad_kernels.cuh"

namespace rikfad {

struct DenParams {
    const TensorDev *tensors;
    const float *spart;
    float *out;
    int ntensors;
    CheckBounds chk;           // read by checked builds only
};

struct CanonParams {
    const TensorDev *tensors;
    const PanelDev *panels;
    const TileGroupDev *groups;
    const float *const *src;
    float *const *dst;
    const float *fac;
    const float *spart;
    float ex_prev;
    float damp_prev;
    float eps;
    CheckBounds chk;           // read by checked builds only
};

struct FinParams {
    const TensorDev *tensors;
    const PanelDev *panels;
    const FinItemDev *items;
    const int64_t *slot_off;
    float *fac;
    const float *rowpart;
    const float *colpart;
    float *spart;
    float decay;
    float gain;
    int resum_only;            // 1: only recompute the partial sums of R
    Guard guard;
    CheckBounds chk;           // read by checked builds only
};

// Checks of one finalise item (checked builds): its tensor, rows or panel
// and slots, and the offsets they lead to.
__device__ __forceinline__ bool fin_item_ok(const FinParams &f, const FinItemDev &it, const TensorDev &td)
{
    (void)f; (void)it; (void)td;
    const CheckBounds &cb = f.chk;
    (void)cb;
    if (!RK_DEV_CHECK(cb, td.cols > 0 && td.fac_off >= 0 && td.fac_off + td.rows + td.cols <= cb.fac_floats,
                      kChkFactors))
        return false;
    if (it.kind == kFinRows)
        return RK_DEV_CHECK(cb, it.begin >= 0 && it.begin <= it.end && it.end <= td.rows, kChkRows) &&
               RK_DEV_CHECK(cb, it.chunk >= 0 && it.chunk < td.spart_cnt && td.spart_off >= 0 &&
                                    (int64_t)td.spart_off + td.spart_cnt <= cb.spart_floats, kChkSpart) &&
               RK_DEV_CHECK(cb, f.resum_only || (td.rowpart_off >= 0 &&
                                    td.rowpart_off + (int64_t)td.npanels * td.rows <= cb.rowpart_floats),
                            kChkRowpart);
    if (!RK_DEV_CHECK(cb, it.kind == kFinCols, kChkKind) ||
        !RK_DEV_CHECK(cb, it.panel >= td.panel0 && it.panel < td.panel0 + td.npanels && it.panel >= 0 &&
                              it.panel < cb.npanels, kChkPanel))
        return false;
    if (f.resum_only)
        return true;
    const PanelDev pd = f.panels[it.panel];
    const int ns = pd.nslots;
    (void)ns;                  // read by the checks only
    return RK_DEV_CHECK(cb, pd.tensor == it.tensor && pd.col0 >= 0 &&
                                (int64_t)pd.col0 + pd.width <= td.cols, kChkCols) &&
           RK_DEV_CHECK(cb, it.begin >= 0 && it.begin <= it.end && it.end <= pd.width, kChkCols) &&
           RK_DEV_CHECK(cb, pd.slot_begin >= 0 && ns >= 0 && pd.slot_end <= cb.nslots &&
                                (it.chunk != 0 || ns <= kFinSplitSlots), kChkColpart) &&
           RK_DEV_CHECK(cb, ns == 0 || (f.slot_off[pd.slot_begin] >= 0 &&
                                        f.slot_off[pd.slot_begin] + (int64_t)(ns - 1) * pd.slot_stride +
                                                pd.width <= cb.colpart_floats),
                        kChkColpart);
}


// ---------------------------------------------------- finalise kernel
//
// R_{n+1} = e^{-alpha h} R_n + k sum_panels rowpart,
// C_{n+1} = e^{-alpha h} C_n + k sum_slots colpart,
// and the partial sums of R_{n+1} that give 1^T R_{n+1}.
//
// A row item is kFinThreads rows, one thread per row.  A column item of a
// panel with few slots is up to 256 columns, one thread per column adding the
// slots in order; a panel with many slots (more than kFinSplitSlots) gets
// items of kFinColChunk (32) columns: warp w adds the slots slot_begin + w,
// + 8, ... for the 32 columns (coalesced 128-byte rows of the partials), then
// warp 0 adds the eight warp sums in order.
__global__ void __launch_bounds__(kFinThreads) rikfad_finalize_kernel(FinParams f)
{
    __shared__ float wsum[kFinThreads / 32];
    __shared__ float csum[kFinThreads / 32][32];
    if (!RK_DEV_CHECK(f.chk, (int)blockIdx.x < f.chk.nfin, kChkFinItem))
        return;
    const FinItemDev it = f.items[blockIdx.x];
    if (!RK_DEV_CHECK(f.chk, it.tensor >= 0 && it.tensor < f.chk.ntensors, kChkTensor))
        return;
    const TensorDev td = f.tensors[it.tensor];
    wait_for_predecessor();
    allow_successor_launch();
    if (!fin_item_ok(f, it, td))
        return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (it.kind == kFinRows) {
        const int64_t i = it.begin + threadIdx.x;
        float val = 0.f;
        if (i < it.end) {
            float *R = f.fac + td.fac_off;
            if (f.resum_only) {
                val = R[i];
            } else {
                float acc = 0.f;
                const float *rp = f.rowpart + td.rowpart_off + i;
#pragma unroll 4
                for (int k = 0; k < td.npanels; ++k)
                    acc += rp[(int64_t)k * td.rows];
                val = fmaf(f.gain, acc, f.decay * R[i]);
                R[i] = val;
            }
            if (!isfinite(val))
                report_nonfinite(f.guard, it.tensor);
        }
        val = warp_sum(val);
        if (lane == 0)
            wsum[warp] = val;
        __syncthreads();
        if (threadIdx.x < 32) {
            float v = threadIdx.x < kFinThreads / 32 ? wsum[threadIdx.x] : 0.f;
            v = warp_sum(v);
            if (threadIdx.x == 0) {
                f.spart[td.spart_off + it.chunk] = v;
                if (!isfinite(v))       // finite R whose sum overflows
                    report_nonfinite(f.guard, it.tensor);
            }
        }
    } else if (!f.resum_only && it.chunk == 0) {
        // A panel's partials are pd.slot_stride apart in colpart (the planner
        // checks this), so every slot's load is issued at once and
        // the sum is still taken in slot order.
        const PanelDev pd = f.panels[it.panel];
        const int64_t c = it.begin + threadIdx.x;
        if (c < it.end) {
            const int ns = pd.nslots;
            const float *cp = f.colpart + (ns > 0 ? f.slot_off[pd.slot_begin] : 0) + c;
            float v[kFinSplitSlots];
#pragma unroll
            for (int u = 0; u < kFinSplitSlots; ++u)
                v[u] = u < ns ? cp[(int64_t)u * pd.slot_stride] : 0.f;
            float acc = 0.f;
#pragma unroll
            for (int u = 0; u < kFinSplitSlots; ++u)
                if (u < ns)
                    acc += v[u];
            float *C = f.fac + td.fac_off + td.rows + pd.col0;
            const float cn = fmaf(f.gain, acc, f.decay * C[c]);
            C[c] = cn;
            if (!isfinite(cn))
                report_nonfinite(f.guard, it.tensor);
        }
    } else if (!f.resum_only) {
        const PanelDev pd = f.panels[it.panel];
        const int64_t c = it.begin + lane;
        float acc = 0.f;
        if (c < it.end) {
            const float *cp = f.colpart + f.slot_off[pd.slot_begin] + c;
#pragma unroll 4
            for (int s = warp; s < pd.nslots; s += kFinThreads / 32)
                acc += cp[(int64_t)s * pd.slot_stride];
        }
        csum[warp][lane] = acc;
        __syncthreads();
        if (warp == 0 && c < it.end) {
            float t = 0.f;
#pragma unroll
            for (int k = 0; k < kFinThreads / 32; ++k)
                t += csum[k][lane];
            float *C = f.fac + td.fac_off + td.rows + pd.col0;
            const float cn = fmaf(f.gain, t, f.decay * C[c]);
            C[c] = cn;
            if (!isfinite(cn))
                report_nonfinite(f.guard, it.tensor);
        }
    }
}

// ------------------------------------------- canonical momentum kernel
//
// dst = src exp(-(h_prev/2) xi~) e^{-gamma h_prev} for matrices (the same
// expression, in the same rounding order, as the start of the next step);
// vectors already hold P_{n+1} and are copied when dst != src.
//
// Bound by HBM (8 B an element).  No sums cross rows, so a block takes one tile
// of a panel's rows, in memory order; its first loads are issued before C is
// staged.  GPT2-S (1.0 GB): 147 us (6.8 TB/s), against 155 from two persistent
// blocks per SM with a contiguous share each, one row per warp.  A narrow
// matrix's tile is taken as a run of elements: 400000 x 64 in 37 us instead of
// 156, 1000000 x 8 in 16 instead of 287; 64-column panels beside wide ones gain
// from the order (eight layers of width 1600: 1394 -> 388 us).  A
// narrow ragged matrix's too (a warp a row left a block walking its tile of many
// rows alone: 300000 x 1 687 us, 600000 x 5 200; so 10 and 12), and a copy of
// element-wise friction's momentum (one load in flight per lane: 29296 x 1024 127
// us; so 39).
__device__ __forceinline__ void canonical_copy(const float *S, float *D, int64_t n)
{
    for (int64_t e = threadIdx.x; e < n; e += kThreads)
        D[e] = S[e];
}

// A panel's rows as a run of units (elements or float4), of which a thread takes
// every 256th from (i0, j0) on.
struct PanelWalk {
    int w, di, dj, i0, j0;
    __device__ __forceinline__ explicit PanelWalk(int width)
        : w(width), di(kThreads / width), dj(kThreads % width), i0((int)threadIdx.x / width), j0((int)threadIdx.x % width)
    {
    }
    __device__ __forceinline__ void next(int &i, int &j) const
    {
        i += di;
        j += dj;
        if (j >= w) {
            j -= w;
            ++i;
        }
    }
};

// Copy `rows` rows of w units, n units apart; a thread has kU loads in flight.
template <int kU, typename T>
__device__ __forceinline__ void canonical_copy_panel(const T *S, T *D, int64_t n, int w, int rows)
{
    const PanelWalk walk(w);
    const int cnt = rows * w;
    int i = walk.i0, j = walk.j0;
#pragma unroll 1
    for (int q0 = threadIdx.x; q0 < cnt; q0 += kThreads * kU) {
        T v[kU];
        int a = i, b = j;
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            if (q0 + kThreads * u < cnt)
                v[u] = __ldcs(S + a * n + b);
            walk.next(a, b);
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            if (q0 + kThreads * u < cnt)
                __stcs(D + i * n + j, v[u]);
            walk.next(i, j);
        }
    }
}

__global__ void __launch_bounds__(kThreads, 4) rikfad_canonical_kernel(CanonParams c)
{
    __shared__ float Cs[kPanelMax];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (!RK_DEV_CHECK(c.chk, (int)blockIdx.x / kTileGroup < c.chk.ngroups, kChkBlock))
        return;
    const TileGroupDev group = c.groups[blockIdx.x / kTileGroup];
    PieceDev pc{};
    pc.tensor = group.tensor;
    if (!piece_tensor_ok(c.chk, pc))
        return;
    const TensorDev td = c.tensors[pc.tensor];
    const uint32_t tile = (uint32_t)group.first + blockIdx.x % kTileGroup;      // the planner keeps it below 2^31
    const uint32_t np = td.npanels > 1 ? td.npanels : 1;
    pc.kind = td.cols == 0 ? kElements : kMatrixRows;
    pc.begin = (int64_t)(tile / np) * td.tile_rows;
    pc.end = pc.begin + td.tile_rows < td.rows ? pc.begin + td.tile_rows : td.rows;
    pc.panel = td.panel0 + (int)(tile % np);
    if (pc.begin >= td.rows)
        return;
    wait_for_predecessor();
    allow_successor_launch();
    const float *S = c.src[pc.tensor];
    float *D = c.dst[pc.tensor];
    if (pc.kind == kElements) {
        if (S != D && vector_piece_ok(c.chk, pc, td, D, nullptr, S, false))
            canonical_copy(S + pc.begin, D + pc.begin, pc.end - pc.begin);
        return;
    }
    if (!piece_panel_ok(c.chk, pc, td))
        return;
    const PanelDev pd = c.panels[pc.panel];
    if (!matrix_piece_ok(c.chk, pc, td, pd, D, nullptr, S, false))
        return;
    if (td.full) {      // element-wise friction: P already holds P_{n+1}
        const float *s0 = S + pc.begin * td.cols + pd.col0;
        float *d0 = D + pc.begin * td.cols + pd.col0;
        const int rows = (int)(pc.end - pc.begin);
        if (S != D && td.vec)
            canonical_copy_panel<4>(reinterpret_cast<const float4 *>(s0), reinterpret_cast<float4 *>(d0), td.cols / 4,
                                    pd.width / 4, rows);
        else if (S != D)
            canonical_copy_panel<8>(s0, d0, td.cols, pd.width, rows);
        return;
    }
    const float *C = c.fac + td.fac_off + td.rows + pd.col0;
    const float *R = c.fac + td.fac_off;
    // 16-byte aligned rows and panels: a whole panel row (at most kPanelMax /
    // 128 float4 per lane) is loaded before the first in-place store.
    constexpr int kV = kPanelMax / 128;
    const int w4 = pd.width / 4;
    float4 v[kV];
    auto load_row = [&](int64_t row) {
        const float4 *s4 = reinterpret_cast<const float4 *>(S + row * td.cols + pd.col0);
#pragma unroll
        for (int k = 0; k < kV; ++k)
            if (lane + 32 * k < w4)
                v[k] = __ldcs(s4 + lane + 32 * k);
    };
    // A narrow matrix (one panel): its tile is a run of elements, of which every
    // lane takes its share whatever the rows' width (run: single elements).
    const bool flat = td.vec && td.npanels == 1 && pd.width <= 128;
    const bool run = !td.vec && td.cols <= kRaggedRun;
    const int n4 = (int)(pc.end - pc.begin) * w4;       // flat: float4 of the tile
    const float4 *t4 = reinterpret_cast<const float4 *>(S + pc.begin * td.cols);
    auto load_flat = [&](int q0) {
#pragma unroll
        for (int k = 0; k < kV; ++k)
            if (q0 + 32 * k < n4)
                v[k] = __ldcs(t4 + q0 + 32 * k);
    };
    int64_t row = pc.begin + warp;
    float r = 0.f;
    if (flat) {
        load_flat(warp * 32 * kV + lane);
    } else if (!run && row < pc.end) {
        if (td.vec)
            load_row(row);
        r = R[row];
    }
    for (int j = threadIdx.x; j < pd.width; j += kThreads)
        Cs[j] = C[j];
    const float inv = inv_denominator(row_total(c.spart, td), c.eps);
    __syncthreads();
    if (flat) {
        float4 *d4 = reinterpret_cast<float4 *>(D + pc.begin * td.cols);
        for (int q0 = warp * 32 * kV + lane; q0 < n4; q0 += kThreads * kV) {
            if (q0 >= kThreads * kV)
                load_flat(q0);
#pragma unroll
            for (int k = 0; k < kV; ++k) {
                const unsigned q = q0 + 32 * k;
                if (q < (unsigned)n4) {
                    const unsigned i = q / (unsigned)w4, j = 4 * (q - i * w4);
                    const float a_prev = c.ex_prev * (R[pc.begin + i] * inv);
                    v[k].x = (v[k].x * exp2f(a_prev * Cs[j])) * c.damp_prev;
                    v[k].y = (v[k].y * exp2f(a_prev * Cs[j + 1])) * c.damp_prev;
                    v[k].z = (v[k].z * exp2f(a_prev * Cs[j + 2])) * c.damp_prev;
                    v[k].w = (v[k].w * exp2f(a_prev * Cs[j + 3])) * c.damp_prev;
                    __stcs(d4 + q, v[k]);
                }
            }
        }
        return;
    }
    if (run) {
        // A narrow ragged matrix: a run of elements too, of which a thread takes
        // every 256th, 8 of them loaded before the first in-place store.
        constexpr int kU = 8;
        const int cnt = (int)(pc.end - pc.begin) * pd.width;
        const float *s0 = S + pc.begin * td.cols;
        float *d0 = D + pc.begin * td.cols;
        const PanelWalk walk(pd.width);
        int i = walk.i0, j = walk.j0;
#pragma unroll 1
        for (int q0 = threadIdx.x; q0 < cnt; q0 += kThreads * kU) {
            float u8[kU], r8[kU];
            int a = i, b = j;
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                if (q0 + kThreads * u < cnt) {
                    u8[u] = __ldcs(s0 + q0 + kThreads * u);
                    r8[u] = R[pc.begin + a];
                }
                walk.next(a, b);
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                if (q0 + kThreads * u < cnt)
                    __stcs(d0 + q0 + kThreads * u, (u8[u] * exp2f((c.ex_prev * (r8[u] * inv)) * Cs[j])) * c.damp_prev);
                walk.next(i, j);
            }
        }
        return;
    }
    for (; row < pc.end; row += kWarps) {
        const int64_t base = row * td.cols + pd.col0;
        if (row >= pc.begin + kWarps) {
            if (td.vec)
                load_row(row);
            r = R[row];
        }
        const float a_prev = c.ex_prev * (r * inv);
        if (td.vec) {
            float4 *d4 = reinterpret_cast<float4 *>(D + base);
#pragma unroll
            for (int k = 0; k < kV; ++k) {
                const int j4 = lane + 32 * k;
                if (j4 < w4) {
                    const int j = 4 * j4;
                    v[k].x = (v[k].x * exp2f(a_prev * Cs[j])) * c.damp_prev;
                    v[k].y = (v[k].y * exp2f(a_prev * Cs[j + 1])) * c.damp_prev;
                    v[k].z = (v[k].z * exp2f(a_prev * Cs[j + 2])) * c.damp_prev;
                    v[k].w = (v[k].w * exp2f(a_prev * Cs[j + 3])) * c.damp_prev;
                    __stcs(d4 + j4, v[k]);
                }
            }
        } else {
            // Rows at any element address: 256 columns' loads before the first
            // in-place store (one load in flight per lane ran at a fraction of
            // the bandwidth, as in matrix_piece_ragged).
            constexpr int kU = 8;
#pragma unroll 1
            for (int j0 = lane; j0 < pd.width; j0 += 32 * kU) {
                float u8[kU];
#pragma unroll
                for (int u = 0; u < kU; ++u)
                    if (j0 + 32 * u < pd.width)
                        u8[u] = __ldcs(S + base + j0 + 32 * u);
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int j = j0 + 32 * u;
                    if (j < pd.width)
                        __stcs(D + base + j, (u8[u] * exp2f(a_prev * Cs[j])) * c.damp_prev);
                }
            }
        }
    }
}

// 1^T R of every matrix (0 for vectors), same summation order as the kernels.
// d.out may be page-locked host memory mapped into the device's address
// space (the enqueued read-back writes there directly).
__global__ void rikfad_denominators_kernel(DenParams d)
{
    wait_for_predecessor();
    allow_successor_launch();
    const int t = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    if (t >= d.ntensors)
        return;
    const TensorDev td = d.tensors[t];
    if (!RK_DEV_CHECK(d.chk, td.spart_off >= 0 && (int64_t)td.spart_off + td.spart_cnt <= d.chk.spart_floats,
                      kChkSpart))
        return;
    const float s = td.cols == 0 ? 0.f : row_total(d.spart, td);
    if ((threadIdx.x & 31) == 0)
        d.out[t] = s;
}

// A state image's header, stored from the kernel's argument.
struct HeaderParams {
    uint64_t *dst;
    uint64_t words[8];
};

__global__ void rikfad_header_kernel(HeaderParams p)
{
    wait_for_predecessor();
    allow_successor_launch();
    if (threadIdx.x < 8)
        p.dst[threadIdx.x] = p.words[threadIdx.x];
}

}  // namespace rikfad
