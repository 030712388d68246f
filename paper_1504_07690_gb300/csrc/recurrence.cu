// recurrence.cu - one step of the block Chebyshev three-term recurrence.
//
//   V_{k+1} = c (2 A~ V_k) - d V_{k-1}
//
// with (c, d) = (1/2, 0) for the first step (V_1 = A~ W) and (1, 1) after
// (Alg. 7, "V_p <- (2 - delta_l0) A~ V_c - V_m"; Section 2's map A~ =
// (2A - (a+b)I)/(b-a) is folded into the operator coefficients).
//
// Blocks are row-major, n rows x ld columns, ld a multiple of the 16-byte
// vector width.  The stencil kernel gives each output row to one warp whose
// lanes walk the row's 16-byte vectors (coalesced); the CSR kernel gives
// each thread one vector of one row.  Neighbour rows along the fastest grid
// axis are adjacent in memory and the rows one plane away are reused from L2
// by the warps working next to them.
#include <cuda_bf16.h>


#include "internal.h"
#include "sweep.cuh"

namespace ssm {

namespace {

template <typename T> struct Vec16;
template <> struct Vec16<float> { using type = float4; static constexpr int W = 4; };
template <> struct Vec16<double> { using type = double2; static constexpr int W = 2; };

__device__ __forceinline__ float4 vscale(float a, float4 x) { return make_float4(a * x.x, a * x.y, a * x.z, a * x.w); }
__device__ __forceinline__ double2 vscale(double a, double2 x) { return make_double2(a * x.x, a * x.y); }
__device__ __forceinline__ float4 vfma(float a, float4 x, float4 y) {
    return make_float4(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y), fmaf(a, x.z, y.z), fmaf(a, x.w, y.w));
}
__device__ __forceinline__ double2 vfma(double a, double2 x, double2 y) {
    return make_double2(fma(a, x.x, y.x), fma(a, x.y, y.y));
}
__device__ __forceinline__ float4 vadd(float4 x, float4 y) { return make_float4(x.x + y.x, x.y + y.y, x.z + y.z, x.w + y.w); }
__device__ __forceinline__ double2 vadd(double2 x, double2 y) { return make_double2(x.x + y.x, x.y + y.y); }
__device__ __forceinline__ float4 vzero(float) { return make_float4(0.f, 0.f, 0.f, 0.f); }
__device__ __forceinline__ double2 vzero(double) { return make_double2(0.0, 0.0); }

template <typename VT>
__device__ __forceinline__ VT ldg_stream(const VT* p) { return __ldg(p); }

// Split-bf16 panel of a float32 block for the tensor-core Gram (see
// gram_tc.cu): rows in panels of 32, columns in groups of 8 (G groups; columns past
// n_tot are zero), each (panel, part, group) a 512-byte run of four
// 8 x 16-byte core matrices (8 rows x 8 bf16 each) and a 16-byte pad (a
// 528-byte group stride); part 0 = hi = rn(v),
// part 1 = lo = rn(v - hi).  The CTA of 8 warps that writes 8 consecutive
// rows stages their hi/lo values in shared memory and writes whole 128-byte
// core matrices.
struct PanelOut {
    uint8_t* base;   // NULL: no panel output
    uint32_t G;      // column groups
};

// Shared-memory stage of one 32-row panel: [part][row 0..31][group, padded to
// G+1][16 B].  Consecutive columns of a row are adjacent (the split stores of
// consecutive threads do not conflict) and the one-chunk pad makes the 8
// rows read together by the flush fall in distinct banks.
__device__ __forceinline__ uint32_t stage_off(uint32_t G, uint32_t part, uint32_t row, uint32_t g) {
    return ((part * 32 + row) * (G + 1) + g) * 16;
}

// Write the staged panel as 512-byte runs (panel, part, group), 528 bytes
// apart (a 16-byte pad per group), in core-matrix order [kg][row8][16 B]
// (row = kg*8 + row8).
__device__ __forceinline__ void flush_panel(const uint8_t* stage, PanelOut po, uint32_t panel) {
    const uint32_t n16 = 2 * po.G * 32;  // 16-byte pieces: part x group x row
    for (uint32_t t = threadIdx.x; t < n16; t += blockDim.x) {
        const uint32_t row = t & 31, g = (t >> 5) % po.G, part = (t >> 5) / po.G;
        const uint4 v = *reinterpret_cast<const uint4*>(stage + stage_off(po.G, part, row, g));
        uint8_t* dst = po.base + (((size_t)panel * 2 + part) * po.G + g) * 528 + row * 16;
        *reinterpret_cast<uint4*>(dst) = v;
    }
}

// Split 4 consecutive columns of staged row `row` (0..31) of a panel stage.
__device__ __forceinline__ void stage_split4p(uint8_t* stage, int G, int row, int col0, float4 v) {
    __align__(8) __nv_bfloat16 h[4];
    __align__(8) __nv_bfloat16 l[4];
    const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        h[q] = __float2bfloat16_rn(x[q]);
        l[q] = __float2bfloat16_rn(x[q] - __bfloat162float(h[q]));
    }
    const uint32_t g = (uint32_t)col0 >> 3, half = ((uint32_t)col0 >> 2) & 1;
    *reinterpret_cast<uint2*>(stage + stage_off(G, 0, row, g) + half * 8) = *reinterpret_cast<const uint2*>(h);
    *reinterpret_cast<uint2*>(stage + stage_off(G, 1, row, g) + half * 8) = *reinterpret_cast<const uint2*>(l);
}

// Split 4 consecutive columns (col0 = 4 q) of row `row` (0..31) of panel `panel` and
// store the bf16 hi and lo parts straight into the panel layout (8 bytes each).
__device__ __forceinline__ void panel_store4(PanelOut po, uint32_t panel, uint32_t row, uint32_t col0, float4 v) {
    __align__(8) __nv_bfloat16 h[4];
    __align__(8) __nv_bfloat16 l[4];
    const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        h[q] = __float2bfloat16_rn(x[q]);
        l[q] = __float2bfloat16_rn(x[q] - __bfloat162float(h[q]));
    }
    const uint32_t g = col0 >> 3, half = (col0 >> 2) & 1;
    const size_t inner = (size_t)row * 16 + half * 8;
    uint8_t* hi = po.base + (((size_t)panel * 2) * po.G + g) * 528 + inner;
    uint8_t* lo = po.base + (((size_t)panel * 2 + 1) * po.G + g) * 528 + inner;
    *reinterpret_cast<uint2*>(hi) = *reinterpret_cast<const uint2*>(h);
    *reinterpret_cast<uint2*>(lo) = *reinterpret_cast<const uint2*>(l);
}
__device__ __forceinline__ void panel_store4(PanelOut, uint32_t, uint32_t, uint32_t, double2) {}

// Per-row neighbour table of a 32-row panel.
struct RowInfo {
    uint32_t nb[6];
    uint32_t has;  // bit a: neighbour a present; bit 31: row exists
};

// Operands of one (row, 16-byte chunk) item of a float32 stencil step: the centre
// value, the neighbour sums per axis, V_{k-1} and the folded diagonal.
struct ItemLoads {
    float4 x, s[3], vp;
    float dg;
    bool ok;
};

__device__ __forceinline__ void load_item(ItemLoads& L, const RowInfo& ri, uint32_t i, uint32_t cc, uint32_t nchunk,
                                          const float4* vc, const float4* vp, const float* diag2, bool need_vp) {
    L.ok = (ri.has >> 31) != 0;
    if (!L.ok) return;
    const size_t base = (size_t)i * nchunk;
    L.x = ldg_stream(vc + base + cc);
    L.dg = __ldg(diag2 + i);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const bool lo = (ri.has >> (2 * a)) & 1u, hi = (ri.has >> (2 * a + 1)) & 1u;
        float4 sacc = vzero(0.f);
        if (lo) sacc = vadd(sacc, ldg_stream(vc + (size_t)ri.nb[2 * a] * nchunk + cc));
        if (hi) sacc = vadd(sacc, ldg_stream(vc + (size_t)ri.nb[2 * a + 1] * nchunk + cc));
        L.s[a] = sacc;
    }
    L.vp = need_vp ? ldg_stream(vp + base + cc) : vzero(0.f);
}

// A CTA owns one 32-row panel at a time (grid-stride over panels): the first
// 32 threads tabulate the rows' neighbour rows, then all 256 threads walk the
// panel's (row, 16-byte chunk) items, so loads and stores are coalesced and
// every lane is busy; with PANEL each item's split-bf16 hi and lo parts go
// straight to their place in the panel (8-byte stores: no shared-memory stage
// and no barrier per panel, so more of these CTAs fit next to a Gram CTA).
template <bool PANEL>
__global__ void __launch_bounds__(256, 4)
stencil_step_kernel(const float* __restrict__ Vc, const float* __restrict__ Vp, float* __restrict__ Vn,
                    const float* __restrict__ diag2, StencilGeom g, float o0, float o1, float o2, float c, float d,
                    uint32_t nchunk, uint32_t n_rows, PanelOut po) {
    __shared__ RowInfo info[32];
    const uint32_t mdiv = ((1u << 20) + nchunk - 1) / nchunk;  // it / nchunk for it < 32 nchunk
    const float4* vc = reinterpret_cast<const float4*>(Vc);
    const float4* vp = reinterpret_cast<const float4*>(Vp);
    float4* vn = reinterpret_cast<float4*>(Vn);
    const uint32_t s1 = g.d2, s0 = g.d1 * g.d2;
    const float w[3] = {g.active[0] ? o0 : 0.f, g.active[1] ? o1 : 0.f, g.active[2] ? o2 : 0.f};
    const uint32_t n_pan = (n_rows + 31) / 32;
    const uint32_t items = 32 * nchunk;
    for (uint32_t pnl = blockIdx.x; pnl < n_pan; pnl += gridDim.x) {
        __syncthreads();  // info free
        if (threadIdx.x < 32) {
            const uint32_t i = pnl * 32 + threadIdx.x;
            RowInfo ri;
            ri.has = 0;
            if (i < n_rows) {
                ri.has = 1u << 31;
                const uint32_t i2 = i % g.d2, q = i / g.d2, i1 = q % g.d1, i0 = q / g.d1;
                const uint32_t co[3] = {i0, i1, i2}, ex[3] = {g.d0, g.d1, g.d2}, sd[3] = {s0, s1, 1u};
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const uint32_t cm = co[a], e = ex[a], st = sd[a];
                    const bool act = g.active[a] != 0;
                    if (act && (cm > 0 || g.per[a])) ri.has |= 1u << (2 * a);
                    if (act && (cm + 1 < e || g.per[a])) ri.has |= 1u << (2 * a + 1);
                    ri.nb[2 * a] = cm > 0 ? i - st : i + (e - 1) * st;
                    ri.nb[2 * a + 1] = cm + 1 < e ? i + st : i - (e - 1) * st;
                }
            }
            info[threadIdx.x] = ri;
        }
        __syncthreads();
        // two items per thread per pass, all their loads issued before either is used
        for (uint32_t it0 = threadIdx.x; it0 < items; it0 += 2 * blockDim.x) {
            ItemLoads L[2];
            uint32_t rr[2], cq[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const uint32_t it = it0 + u * blockDim.x;
                L[u].ok = false;
                rr[u] = 0;
                cq[u] = 0;
                if (it < items) {
                    rr[u] = (it * mdiv) >> 20;
                    cq[u] = it - rr[u] * nchunk;
                    load_item(L[u], info[rr[u]], pnl * 32 + rr[u], cq[u], nchunk, vc, vp, diag2, d != 0.f);
                }
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const uint32_t it = it0 + u * blockDim.x;
                if (it >= items) continue;
                float4 out = vzero(0.f);
                if (L[u].ok) {
                    float4 acc = vscale(L[u].dg, L[u].x);
#pragma unroll
                    for (int a = 0; a < 3; ++a) acc = vfma(w[a], L[u].s[a], acc);
                    out = vscale(c, acc);
                    if (d != 0.f) out = vfma(-d, L[u].vp, out);
                    vn[(size_t)(pnl * 32 + rr[u]) * nchunk + cq[u]] = out;
                }
                if constexpr (PANEL) panel_store4(po, pnl, rr[u], 4 * cq[u], out);
            }
        }
    }
}

// Float64 stencil step: one (row, 16-byte chunk) item a thread.  Two fmas a clock and SM
// bound it (6 float64 operations an element on a 2D grid), so what counts is that nothing
// else takes that pipe (the first step is a flag: comparing c and d would) and that enough
// warps are there to hide its latency; index arithmetic is free.  On 128 x 128 with 100
// columns 39 us a step in 32-row panels of 160-thread CTAs (3.4 CTAs an SM), 26 us here
// (17 us for the operations alone).
__global__ void __launch_bounds__(256)
stencil_flat_f64_kernel(const double2* __restrict__ vc, const double2* __restrict__ vp, double2* __restrict__ vn,
                        const double* __restrict__ diag2, StencilGeom g, double o0, double o1, double o2, double c,
                        double d, bool first, uint32_t nchunk, uint32_t n_rows) {
    const uint64_t u = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t i = (uint32_t)(u / nchunk), cc = (uint32_t)(u - (uint64_t)i * nchunk);
    if (u >= (uint64_t)n_rows * nchunk) return;
    const size_t at = (size_t)u;
    const double2 x = __ldg(vc + at);
    const double dg = __ldg(diag2 + i);
    double2 p = vzero(0.0);
    if (!first) p = __ldg(vp + at);
    const uint32_t i2 = i % g.d2, q = i / g.d2, i1 = q % g.d1, i0 = q / g.d1;
    const uint32_t co[3] = {i0, i1, i2}, ex[3] = {g.d0, g.d1, g.d2}, sd[3] = {g.d1 * g.d2, g.d2, 1u};
    double2 lo[3], hi[3];
    bool has_lo[3], has_hi[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {  // all loads before the first use
        const uint32_t cm = co[a], e = ex[a], st = sd[a];
        has_lo[a] = g.active[a] && (cm > 0 || g.per[a]);
        has_hi[a] = g.active[a] && (cm + 1 < e || g.per[a]);
        lo[a] = hi[a] = vzero(0.0);
        if (has_lo[a]) lo[a] = __ldg(vc + (size_t)(cm > 0 ? i - st : i + (e - 1) * st) * nchunk + cc);
        if (has_hi[a]) hi[a] = __ldg(vc + (size_t)(cm + 1 < e ? i + st : i - (e - 1) * st) * nchunk + cc);
    }
    const double w[3] = {o0, o1, o2};
    double2 acc = vscale(dg, x);
#pragma unroll
    for (int a = 0; a < 3; ++a)
        if (g.active[a]) {
            const double2 s = !has_hi[a] ? lo[a] : (has_lo[a] ? vadd(lo[a], hi[a]) : hi[a]);
            acc = vfma(w[a], s, acc);
        }
    vn[at] = first ? vscale(c, acc) : vfma(-d, p, acc);  // c = 1 after the first step
}

// Float32 stencil step on grids whose axis 0 is inactive (2D and 1D grids): a thread
// owns one 16-byte chunk of R consecutive rows of a 32-row panel and loads the centre
// rows row0-1 .. row0+R once; they are also the axis-2 neighbours of the group's rows
// wherever those are the adjacent rows (a wrapped neighbour is loaded where it is used).
// Against one (row, chunk) item a thread this issues 5 instead of 6 loads a row on a 2D
// grid, all of a group's loads before the first use.  The operations of
// stencil_step_kernel on the same grid, the inactive axis first, so the outputs are the
// same values (a zero may change sign).  Each CTA takes MARCH_UNITS consecutive (row
// group, chunk) units, K a thread.  One unit a thread: next to the Gram kernel on the
// other stream, short CTAs let the two interleave on the SMs (the mixed step on a 256^2
// grid: 62.0 ms against 62.8 with two units a thread, 65.2 with four, 69.2 with eight;
// four rows a thread 63.5, eight 74.1).
constexpr int MARCH_R = 2, MARCH_K = 1, MARCH_T = 256;
constexpr uint32_t MARCH_UNITS = (uint32_t)MARCH_T * MARCH_K;

template <bool PANEL>
__global__ void __launch_bounds__(MARCH_T)
stencil_march_kernel(const float* __restrict__ Vc, const float* __restrict__ Vp, float* __restrict__ Vn,
                     const float* __restrict__ diag2, StencilGeom g, float o1, float o2, float c, float d,
                     uint32_t nchunk, uint32_t n_rows, PanelOut po) {
    constexpr int R = MARCH_R;
    const float4* vc = reinterpret_cast<const float4*>(Vc);
    const float4* vp = reinterpret_cast<const float4*>(Vp);
    float4* vn = reinterpret_cast<float4*>(Vn);
    const uint32_t s1 = g.d2;
    const float w1 = g.active[1] ? o1 : 0.f, w2 = g.active[2] ? o2 : 0.f;
    const uint64_t units = (uint64_t)((n_rows + 31) / 32) * (32 / R) * nchunk;
    const bool need_vp = d != 0.f;
    const uint64_t u0 = (uint64_t)blockIdx.x * MARCH_UNITS + threadIdx.x;
    for (int k = 0; k < MARCH_K; ++k) {
        const uint64_t u = u0 + (uint64_t)k * MARCH_T;
        if (u >= units) break;
        const uint32_t grp = (uint32_t)(u / nchunk), cc = (uint32_t)(u - (uint64_t)grp * nchunk);
        const uint32_t row0 = grp * R;
        const uint32_t c2s = row0 % g.d2, c1s = (row0 / g.d2) % g.d1;
        float4 x[R + 2], a1[R][2], vpr[R];
        float dg[R];
        x[0] = (row0 >= 1 && c2s > 0 && g.active[2]) ? ldg_stream(vc + (size_t)(row0 - 1) * nchunk + cc) : vzero(0.f);
#pragma unroll
        for (int r = 0; r < R; ++r)
            x[r + 1] = row0 + r < n_rows ? ldg_stream(vc + (size_t)(row0 + r) * nchunk + cc) : vzero(0.f);
        {
            const uint32_t rl = row0 + R, cl = (c2s + R - 1) % g.d2;
            x[R + 1] = (rl < n_rows && cl + 1 < g.d2 && g.active[2]) ? ldg_stream(vc + (size_t)rl * nchunk + cc)
                                                                     : vzero(0.f);
        }
        uint32_t c2 = c2s, c1 = c1s;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const uint32_t i = row0 + r;
            a1[r][0] = a1[r][1] = vpr[r] = vzero(0.f);
            dg[r] = 0.f;
            if (i < n_rows) {
                if (g.active[1]) {
                    if (c1 > 0 || g.per[1])
                        a1[r][0] = ldg_stream(vc + (size_t)(c1 > 0 ? i - s1 : i + (g.d1 - 1) * s1) * nchunk + cc);
                    if (c1 + 1 < g.d1 || g.per[1])
                        a1[r][1] = ldg_stream(vc + (size_t)(c1 + 1 < g.d1 ? i + s1 : i - (g.d1 - 1) * s1) * nchunk + cc);
                }
                dg[r] = __ldg(diag2 + i);
                if (need_vp) vpr[r] = ldg_stream(vp + (size_t)i * nchunk + cc);
            }
            if (++c2 == g.d2) {
                c2 = 0;
                if (++c1 == g.d1) c1 = 0;
            }
        }
        c2 = c2s;
        c1 = c1s;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const uint32_t i = row0 + r;
            float4 out = vzero(0.f);
            if (i < n_rows) {
                // per axis (0 + lo) + hi, then dg x + w0 s0 + w1 s1 + w2 s2 as in the per-item kernel
                float4 s1v = vzero(0.f), s2v = vzero(0.f);
                if (g.active[1] && (c1 > 0 || g.per[1])) s1v = vadd(s1v, a1[r][0]);
                if (g.active[1] && (c1 + 1 < g.d1 || g.per[1])) s1v = vadd(s1v, a1[r][1]);
                if (g.active[2] && (c2 > 0 || g.per[2]))
                    s2v = vadd(s2v, c2 > 0 ? x[r] : ldg_stream(vc + (size_t)(i + (g.d2 - 1)) * nchunk + cc));
                if (g.active[2] && (c2 + 1 < g.d2 || g.per[2]))
                    s2v = vadd(s2v, c2 + 1 < g.d2 ? x[r + 2] : ldg_stream(vc + (size_t)(i - (g.d2 - 1)) * nchunk + cc));
                float4 acc = vscale(dg[r], x[r + 1]);
                acc = vfma(0.f, vzero(0.f), acc);
                acc = vfma(w1, s1v, acc);
                acc = vfma(w2, s2v, acc);
                out = vscale(c, acc);
                if (need_vp) out = vfma(-d, vpr[r], out);
                vn[(size_t)i * nchunk + cc] = out;
            }
            if constexpr (PANEL) panel_store4(po, i >> 5, i & 31, 4 * cc, out);
            if (++c2 == g.d2) {
                c2 = 0;
                if (++c1 == g.d1) c1 = 0;
            }
        }
    }
}

// Float32 stencil step on large 3D grids, by sweeps: a CTA owns an 8 x 8 tile of axes 1
// and 2 and SWEEP_C 16-byte column chunks, and sweeps a run of planes along axis 0.  A thread
// keeps its element of planes z - 1, z, z + 1 in registers; the plane's tile and its halo of
// 32 rows go through shared memory, so an element of V_k is read 1.5 times instead of once
// per neighbour, and the loads of plane z + 2, of the next halo and of V_{k-1} are in
// flight while plane z is computed.  Neighbours past an open edge are zeros in shared
// memory, which the sums pass unchanged; the operations and their order are those of
// stencil_step_kernel, so the outputs are the same values (a zero may change sign).
// What bounds it: memory.  On a 100^3 grid of 128 columns without panels 308 us and 3.6 GB
// between L2 and the SMs, against 328 us and 5.0 GB for the per-item kernel; with panels
// beside the Gram products a 64^3 grid of 256 columns takes 0.34 ms a step instead of 0.36.
// (A ring of asynchronous copies instead of the registers was slower there, 0.35 ms: the
// Gram CTA holds most of the shared memory; so were sweeps along axis 1 of 2D grids, 68-76
// ms a call against 61.6 ms on the 256^2 one.)  Four CTAs an SM, 64 registers a thread: with
// the 79 that the compiler takes for fewer a call on the 64^3 grid takes 71.3 ms instead of 63.7
// (256 columns, 128 of them hybrid, degree 300, 400 pencils).
using Tile3D = SweepTile<8, 8>;
constexpr uint32_t SWEEP_C = 4;

template <bool PANEL>
__global__ void __launch_bounds__(Tile3D::ROWS * SWEEP_C, 4)
stencil_sweep_kernel(const float* __restrict__ Vc, const float* __restrict__ Vp, float* __restrict__ Vn,
                     const float* __restrict__ diag2, StencilGeom g, float o0, float o1, float o2, float c, float d,
                     uint32_t nchunk, uint32_t ngrp, uint32_t nt2, uint32_t planes, PanelOut po) {
    using ST = Tile3D;
    constexpr uint32_t C = SWEEP_C, bufsz = ST::PLANE * C;
    __shared__ float4 sw[2 * bufsz];  // two staged planes
    const int d0 = (int)g.d0, d1 = (int)g.d1, d2 = (int)g.d2;
    const uint32_t grp = blockIdx.x % ngrp, tile = blockIdx.x / ngrp;
    const int b1 = (int)(tile / nt2) * ST::T1, b2 = (int)(tile % nt2) * ST::T2;
    const uint32_t cl = threadIdx.x % C, cc = grp * C + cl;
    const SweepRow<ST> R((int)(threadIdx.x / C));
    const int z0 = (int)(blockIdx.y * planes), z1 = min(z0 + (int)planes, d0);
    const bool col = cc < nchunk;
    const bool on1 = g.active[1] != 0, on2 = g.active[2] != 0;
    const float w1 = on1 ? o1 : 0.f, w2 = on2 ? o2 : 0.f;
    const bool need_vp = d != 0.f;
    const size_t pstride = (size_t)d1 * d2 * nchunk;
    const float4* vc = reinterpret_cast<const float4*>(Vc);
    // this thread's element (also one past an end of its axis, where it wraps) and, for
    // the first HALO rows of threads, one element of the halo
    const int p1 = b1 + R.r1, p2 = b2 + R.r2;
    const int m1 = axis_at(p1, d1, g.per[1] && on1), m2 = axis_at(p2, d2, g.per[2] && on2);
    const bool own = col && m1 >= 0 && m2 >= 0;
    const bool out_row = col && p1 < d1 && p2 < d2;
    const float4* vown = vc + (own ? ((size_t)m1 * d2 + m2) * nchunk + cc : 0);
    const int q1 = axis_at(b1 + R.h1, d1, g.per[1] && on1), q2 = axis_at(b2 + R.h2, d2, g.per[2] && on2);
    const bool hok = R.halo && col && q1 >= 0 && q2 >= 0 && (R.ax1 ? on1 : on2);
    const float4* vhal = vc + (hok ? ((size_t)q1 * d2 + q2) * nchunk + cc : 0);
    const uint32_t so = R.own_at() * C + cl, sh = R.halo_at() * C + cl;
    const float4 zero = vzero(0.f);
    auto plane = [&](int z, const float4* v, bool ok) {  // (z may be one past either end of axis 0)
        const int m = axis_at(z, d0, g.per[0] != 0);
        return ok && m >= 0 ? ldg_stream(v + (size_t)m * pstride) : zero;
    };
    const size_t orow = out_row ? (size_t)p1 * d2 + p2 : 0;
    const float4* vp = reinterpret_cast<const float4*>(Vp) + orow * nchunk + cc;
    const float* dgp = diag2 + orow;
    const uint32_t prow = (uint32_t)(d1 * d2);
    float4* vn = reinterpret_cast<float4*>(Vn) + orow * nchunk + cc;
    float4 xm = plane(z0 - 1, vown, own), xc = plane(z0, vown, own), xp = plane(z0 + 1, vown, own);
    float4 hc = plane(z0, vhal, hok), vpc = zero;
    float dg = 0.f;
    if (out_row) {
        if (need_vp) vpc = ldg_stream(vp + (size_t)z0 * pstride);
        dg = __ldg(dgp + (size_t)z0 * prow);
    }
    uint32_t buf = 0;
    for (int z = z0; z < z1; ++z, buf ^= 1) {
        // (two buffers: a thread here has passed the barrier of plane z - 1, which every
        // thread reached after its last read of plane z - 2's buffer)
        float4* S = sw + buf * bufsz;
        S[so] = xc;
        if (R.halo) S[sh] = hc;
        __syncthreads();
        // in flight during this plane: plane z + 2, the halo of plane z + 1, V_{k-1} of z + 1
        float4 xpp = zero, vpn = zero;
        float dgn = 0.f;
        if (z + 1 < z1) {
            xpp = plane(z + 2, vown, own);
            hc = plane(z + 1, vhal, hok);
            if (out_row) {
                if (need_vp) vpn = ldg_stream(vp + (size_t)(z + 1) * pstride);
                dgn = __ldg(dgp + (size_t)(z + 1) * prow);
            }
        }
        if (out_row) {
            const float4 s0 = vadd(vadd(zero, xm), xp);
            float4 s1 = zero, s2 = zero;
            if (on1) s1 = vadd(vadd(zero, S[so - ST::W2 * C]), S[so + ST::W2 * C]);
            if (on2) s2 = vadd(vadd(zero, S[so - C]), S[so + C]);
            float4 acc = vscale(dg, xc);
            acc = vfma(o0, s0, acc);
            acc = vfma(w1, s1, acc);
            acc = vfma(w2, s2, acc);
            float4 out = vscale(c, acc);
            if (need_vp) out = vfma(-d, vpc, out);
            vn[(size_t)z * pstride] = out;
            if constexpr (PANEL) {
                const uint32_t i = (uint32_t)((size_t)z * prow + orow);
                panel_store4(po, i >> 5, i & 31, 4 * cc, out);
            }
        }
        xm = xc;
        xc = xp;
        xp = xpp;
        vpc = vpn;
        dg = dgn;
    }
}

template <typename T, bool PANEL>
__global__ void __launch_bounds__(512)
csr_step_kernel(const T* __restrict__ Vc, const T* __restrict__ Vp, T* __restrict__ Vn,
                const int64_t* __restrict__ rowptr, const int32_t* __restrict__ colind,
                const T* __restrict__ val2, T beta, const T* __restrict__ beta_row, T c, T d, uint32_t nchunk,
                uint32_t n_rows, PanelOut po) {
    using VT = typename Vec16<T>::type;
    const VT* vc = reinterpret_cast<const VT*>(Vc);
    const VT* vp = reinterpret_cast<const VT*>(Vp);
    VT* vn = reinterpret_cast<VT*>(Vn);
    const uint32_t n_pan = (n_rows + 31) / 32;
    const uint32_t items = 32 * nchunk;
    for (uint32_t pnl = blockIdx.x; pnl < n_pan; pnl += gridDim.x) {
        for (uint32_t it = threadIdx.x; it < items; it += blockDim.x) {
            const uint32_t r = it / nchunk, cc = it - r * nchunk;
            const uint32_t i = pnl * 32 + r;
            VT out = vzero(T(0));
            if (i < n_rows) {
                const size_t base = (size_t)i * nchunk;
                VT acc = vscale(beta_row ? __ldg(beta_row + i) : beta, ldg_stream(vc + base + cc));
                const int64_t e1 = __ldg(rowptr + i + 1);
                for (int64_t e = __ldg(rowptr + i); e < e1; ++e) {
                    const uint32_t j = (uint32_t)__ldg(colind + e);
                    acc = vfma(__ldg(val2 + e), ldg_stream(vc + (size_t)j * nchunk + cc), acc);
                }
                out = vscale(c, acc);
                if (d != T(0)) out = vfma(-d, ldg_stream(vp + base + cc), out);
                vn[base + cc] = out;
            }
            if constexpr (PANEL) panel_store4(po, pnl, r, 4 * cc, out);
        }
    }
}

// Panels of an existing float32 block (the probe block V_0).
__global__ void __launch_bounds__(256)
panelize_kernel(const float* __restrict__ V, uint32_t nchunk, uint32_t n_rows, PanelOut po) {
    __shared__ __align__(16) uint8_t stage[2 * 32 * 33 * 16];
    const float4* v = reinterpret_cast<const float4*>(V);
    for (uint32_t t = threadIdx.x; t < 2 * 32 * 33; t += blockDim.x)
        reinterpret_cast<uint4*>(stage)[t] = make_uint4(0, 0, 0, 0);
    const uint32_t n_pan = (n_rows + 31) / 32;
    for (uint32_t pnl = blockIdx.x; pnl < n_pan; pnl += gridDim.x) {
        __syncthreads();
        for (uint32_t it = threadIdx.x; it < 32 * nchunk; it += blockDim.x) {
            const uint32_t r = it / nchunk, cc = it - r * nchunk;
            const uint32_t i = pnl * 32 + r;
            stage_split4p(stage, po.G, r, 4 * cc,
                          i < n_rows ? __ldg(v + (size_t)i * nchunk + cc) : make_float4(0.f, 0.f, 0.f, 0.f));
        }
        __syncthreads();
        flush_panel(stage, po, pnl);
    }
}

// One CTA per 32-row panel (grid-stride beyond 2^20 panels).
// Threads of a stencil-step CTA: the multiple of 32 up to 256 whose passes of two
// items a thread leave the fewest idle lanes over the 32 nchunk items of a panel
// (ties to the larger CTA).
int stencil_threads(uint32_t nchunk) {
    const uint32_t items = 32 * nchunk;
    int best = 256;
    uint32_t best_idle = ~0u;
    for (int t = 256; t >= 128; t -= 32) {
        const uint32_t per = 2u * (uint32_t)t, idle = (items + per - 1) / per * per - items;
        if (idle < best_idle) {
            best = t;
            best_idle = idle;
        }
    }
    return best;
}

int panel_grid(uint64_t n_rows) {
    uint64_t blocks = (n_rows + 31) / 32;
    if (blocks > (1u << 20)) blocks = 1u << 20;
    return blocks < 1 ? 1 : (int)blocks;
}

}  // namespace

// Launches the sweep kernel where it pays; false where it does not: tiles that do not fit
// the grid, blocks below 64 MiB, which the L2 holds (its neighbour reads then cost
// little, and a run's planes follow one another: 15 to 60 % slower on small grids), narrow
// rows, and small planes with ragged tiles.
//
// A CTA takes four chunks of a row, whole 32-byte sectors whatever the width:
// one chunk a CTA (all that divides 11, 13, 17, 31 evenly) costs 1.2 to 1.9 times the
// per-item kernel, three or five up to 1.1 times.  Recurrence and Gram of ten steps on a
// 128^3 grid, by tiles of four chunks and by items: 16.3 and 16.6 ms at 33 chunks, 25.2 and
// 26.8 at 51, 30.3 and 33.9 at 64; 14.4 and 14.4 at 29, 9.5 and 9.2 at 19, 5.1 and 4.8 at 9;
// without idle columns 9.3 and 9.4 at 20, 5.6 and 5.7 at 12, 4.6 and 4.5 at 8.
//
// Planes of 8 MiB outlast the caches between the uses of a row, and the sweep gains with
// tiles a quarter past the edges (60 x 250 x 250 of 128 columns: 26.1 and 29.9 ms; 128 x 121
// x 121 of 256: 28.1 and 29.2).  Smaller ones are read no more often by items, and where the
// step also writes panels every idle row shows (500 x 60 x 60 of 128: 12.9 and 12.4; 500 x 57 x
// 57: 12.0 and 11.2), so there the tiles have to fit to 1/32 (128^3 of 64 columns: 7.35 and
// 7.45; 64^3 of 256: 3.95 and 4.03).  Without panels a step of 100^3 of 128 takes 308 and 328 us.
static bool sweep_step(const StencilGeom& g, int64_t n, uint32_t nchunk, const float* Vc, const float* Vp, float* Vn,
                       const float* diag2, float o0, float o1, float o2, float c, float d, PanelOut po,
                       cudaStream_t s) {
    using ST = Tile3D;
    constexpr uint32_t C = SWEEP_C;
    if ((uint64_t)n * nchunk * 16 < (64ull << 20) || nchunk < (nchunk % C ? 24u : 12u)) return false;
    const uint64_t plane = (uint64_t)g.d1 * g.d2;
    const uint64_t tiled = (uint64_t)((g.d1 + ST::T1 - 1) / ST::T1) * ((g.d2 + ST::T2 - 1) / ST::T2) * ST::ROWS;
    if (po.base && plane * nchunk * 16 < (8ull << 20) && 32 * tiled > 33 * plane) return false;
    const uint32_t ngrp = (nchunk + C - 1) / C;
    // about sixteen 256-thread CTAs an SM over the launch (its last wave is then a small
    // part), at least eight planes a run
    const SweepRuns w = sweep_runs<ST>(g.d0, g.d1, g.d2, ngrp, (uint64_t)device_sms() * 16 * 256 / (ST::ROWS * C), 8);
    if (!w.nseg) return false;
    const dim3 grid(ngrp * w.nt1 * w.nt2, w.nseg);
    const auto kernel = po.base ? stencil_sweep_kernel<true> : stencil_sweep_kernel<false>;
    kernel<<<grid, ST::ROWS * C, 0, s>>>(Vc, Vp ? Vp : Vc, Vn, diag2, g, o0, o1, o2, c, d, nchunk, ngrp, w.nt2,
                                         w.planes, po);
    return true;
}

static cudaError_t stencil_step_f32(const Plan& P, const float* Vc, const float* Vp, float* Vn, const float* diag2,
                                    float o0, float o1, float o2, float c, float d, uint8_t* panel, cudaStream_t s) {
    const uint32_t nchunk = (uint32_t)(P.ld / Vec16<float>::W);
    const PanelOut po{panel, (uint32_t)P.panel_groups};
    {
        // Trailing axes of extent 1 (always inactive) change no row index: (d0, d1, 1) is
        // the grid (1, d0, d1).  With axis 0 then inactive (2D and 1D grids) the row-group
        // kernel runs, marching along the unit-stride axis (5 loads a row instead of 6).
        StencilGeom gn = P.geom;
        float w[3] = {o0, o1, o2};
        for (int sh = 0; sh < 2 && gn.d2 == 1; ++sh) {
            gn.d2 = gn.d1;
            gn.d1 = gn.d0;
            gn.d0 = 1;
            gn.per[2] = gn.per[1];
            gn.per[1] = gn.per[0];
            gn.per[0] = 0;
            gn.active[2] = gn.active[1];
            gn.active[1] = gn.active[0];
            gn.active[0] = 0;
            w[2] = w[1];
            w[1] = w[0];
            w[0] = 0.f;
        }
        if (!gn.active[0]) {
            const uint64_t units = (uint64_t)((P.n + 31) / 32) * (32 / MARCH_R) * nchunk;
            const int grid = (int)((units + MARCH_UNITS - 1) / MARCH_UNITS);
            if (panel)
                stencil_march_kernel<true><<<grid, MARCH_T, 0, s>>>(Vc, Vp ? Vp : Vc, Vn, diag2, gn, w[1], w[2], c, d,
                                                                     nchunk, (uint32_t)P.n, po);
            else
                stencil_march_kernel<false><<<grid, MARCH_T, 0, s>>>(Vc, Vp ? Vp : Vc, Vn, diag2, gn, w[1], w[2], c,
                                                                      d, nchunk, (uint32_t)P.n, po);
            return cudaGetLastError();
        }
        if (sweep_step(P.geom, P.n, nchunk, Vc, Vp, Vn, diag2, o0, o1, o2, c, d, po, s)) return cudaGetLastError();
    }
    const auto kernel = panel ? stencil_step_kernel<true> : stencil_step_kernel<false>;
    kernel<<<panel_grid(P.n), stencil_threads(nchunk), 0, s>>>(Vc, Vp ? Vp : Vc, Vn, diag2, P.geom, o0, o1, o2, c, d,
                                                               nchunk, (uint32_t)P.n, po);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t csr_step(const Plan& P, const T* Vc, const T* Vp, T* Vn, const T* val2, T beta,
                            const T* beta_row, T c, T d, uint8_t* panel, cudaStream_t s) {
    const uint32_t nchunk = (uint32_t)(P.ld / Vec16<T>::W);
    const PanelOut po{panel, (uint32_t)P.panel_groups};
    const int nt = P.csr_threads > 0 ? P.csr_threads : 256;
    if (panel)
        csr_step_kernel<T, true><<<panel_grid(P.n), nt, 0, s>>>(Vc, Vp ? Vp : Vc, Vn, P.d_rowptr, P.d_colind,
                                                                   val2, beta, beta_row, c, d, nchunk,
                                                                   (uint32_t)P.n, po);
    else
        csr_step_kernel<T, false><<<panel_grid(P.n), nt, 0, s>>>(Vc, Vp ? Vp : Vc, Vn, P.d_rowptr,
                                                                    P.d_colind, val2, beta, beta_row, c, d,
                                                                    nchunk, (uint32_t)P.n, po);
    return cudaGetLastError();
}

cudaError_t launch_stencil_step_f64(const Plan& P, const double* Vc, const double* Vp, double* Vn,
                                    double c, double d, cudaStream_t s) {
    if (d != 0.0 && c != 1.0) return cudaErrorInvalidValue;  // (1/2, 0) or (1, 1)
    const uint32_t nchunk = (uint32_t)(P.ld / 2);
    const uint64_t blocks = ((uint64_t)P.n * nchunk + 255) / 256;
    stencil_flat_f64_kernel<<<(unsigned)blocks, 256, 0, s>>>(
        (const double2*)Vc, (const double2*)(Vp ? Vp : Vc), (double2*)Vn, P.d_diag64, P.geom, P.off64[0], P.off64[1],
        P.off64[2], c, d, d == 0.0, nchunk, (uint32_t)P.n);
    return cudaGetLastError();
}
cudaError_t launch_stencil_step_f32(const Plan& P, const float* Vc, const float* Vp, float* Vn,
                                    float c, float d, uint8_t* panel, cudaStream_t s) {
    return stencil_step_f32(P, Vc, Vp, Vn, P.d_diag32, P.off32[0], P.off32[1], P.off32[2], c, d, panel, s);
}
cudaError_t launch_csr_step_f64(const Plan& P, const double* Vc, const double* Vp, double* Vn,
                                double c, double d, cudaStream_t s) {
    return csr_step<double>(P, Vc, Vp, Vn, P.d_val64, P.beta, P.d_beta_row64, c, d, nullptr, s);
}
cudaError_t launch_csr_step_f32(const Plan& P, const float* Vc, const float* Vp, float* Vn,
                                float c, float d, uint8_t* panel, cudaStream_t s) {
    return csr_step<float>(P, Vc, Vp, Vn, P.d_val32, (float)P.beta, P.d_beta_row32, c, d, panel, s);
}

cudaError_t launch_panelize(const Plan& P, const float* V, uint8_t* panel, cudaStream_t s) {
    const PanelOut po{panel, (uint32_t)P.panel_groups};
    panelize_kernel<<<panel_grid(P.n), 256, 0, s>>>(V, (uint32_t)(P.ld / 4), (uint32_t)P.n, po);
    return cudaGetLastError();
}

}  // namespace ssm
