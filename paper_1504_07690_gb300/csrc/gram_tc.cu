// gram_tc.cu - Gram products of the doubling identities on the 5th-generation
// tensor cores (tcgen05, accumulators in TMEM), split-bf16, mixed path.
//
// For a step that produced V_{k+1} (float32) from V_k the moments need
//   G^e = V_{k+1}^T V_{k+1}  (upper blocks; symmetric)  and  G^o = V_{k+1}^T V_k
// (see gram.cu for the identities).  Each float32 value v is split into
// bf16 hi = rn(v) and lo = rn(v - hi); the products hi.hi + hi.lo + lo.hi are
// accumulated in float32 in TMEM (the dropped lo.lo term is below 2^-16 of
// the product), so a Gram entry carries ~2^-17 relative error per term.
//
// Operands: the recurrence kernel writes every block it produces a second
// time as split-bf16 "panels" (recurrence.cu): 32-row panels, 8-column
// groups, hi and lo parts, each (panel, part, group) a 512-byte run of four
// 8 x 16-byte core matrices plus a 16-byte pad - exactly the MN-major,
// no-swizzle shared-memory operand layout of tcgen05 (K stride 128 B, MN
// stride 528 B).  This kernel
// therefore does no conversion: one thread streams panels into a shared-
// memory ring (stages of one to eight panels, as many as fit in 133 KB) with
// 1-D bulk TMA copies (cp.async.bulk, completion
// counted in bytes on an mbarrier), one thread issues M=128
// tcgen05.mma.kind::f16 into TMEM and releases each stage through
// tcgen05.commit (waiting threads are suspended on the mbarriers, not polling),
// and at the end all eight warps read the accumulators back
// with tcgen05.ld and write one float32 partial per slab; partials are
// reduced in slab order in float64.
//
// Work split: a CTA owns one slab of panels and one of the two products
// ("Ge" or "Go"); Go CTAs read two blocks, so their slabs are half as long.
// With a slab table and n_tot <= 128 a CTA may instead form both products of its
// slab ("both": Ge in TMEM columns 0.., Go next to it), reading every panel of
// V_{k+1} once instead of twice.
//
// TMEM: Ge uses ntp (+ ntp-128) columns, Go ntp (+ ntp) columns, ntp = n_tot
// rounded up to 16, n_tot <= 256; a CTA allocates all 512 columns and its
// shared-memory footprint keeps it alone on its SM (two or four CTAs with their parts of
// each share an SM where slabs are small and blocks narrow).  Every wait is bounded:
// on expiry the CTA sets bit 2 of the status word, waits once more (bounded)
// for its copies and MMAs, frees TMEM and returns.
#include <cuda_bf16.h>

#include <algorithm>

#include "internal.h"
#include "tcgen05.cuh"

namespace ssm {

namespace {

using namespace tc;

constexpr int KC = 32;                 // rows per panel (K of one pipeline stage)
constexpr int KG = KC / 8;             // 8-row core groups per panel
constexpr int STAGES = 16;             // barrier slots (most stages in flight)
constexpr int NTHREADS = 256;
constexpr int MAX_PS = 8;              // most panels in a stage
// A column group of a panel is 4 core matrices (512 B) plus a 16-byte pad:
// with a 528-byte group stride the M/N groups of an MMA operand start on
// rotating shared-memory banks instead of all on bank 0.
constexpr int GROUP_BYTES = KG * 128 + 16;
constexpr int PART_BYTES = 32 * GROUP_BYTES;  // one part of one stage: 32 column groups
constexpr int TMEM_COLS = 512;
// > half of an SM (one Gram CTA per SM, it owns all 512 TMEM columns) and small enough
// that two recurrence CTAs (34 KB each) share the SM with it: four one-source stages of
// 32 column groups.  Stages hold the panels' G groups only.
//
// A stage is PS consecutive panels (one contiguous run of the panel array, one bulk copy
// a source): as many, up to eight, as leave at least four stages in the ring.  The time
// of a narrow block is that of the two issuing threads, whose waits, copies and commits
// come once a stage: with one panel a stage and the tile table in local memory a panel of
// n_tot = 17 took them ~700 cycles (N = 2.08e6 rows: 478 us, 21 % of the DRAM rate; the
// KPM line of a 127 x 131 x 125 grid, degree 300: 79.0 ms a call, 46.7 ms with eight).
// Panels hold ceil(n_tot / 8) groups, not a multiple of two, which takes a quarter off
// their bytes there.
// Wide blocks keep one panel a stage, and the kernel alone is slower on them than with 128
// threads and a copy a part (65536 x 200: 38.5 us cold, 36.5 then), but the call is faster (400
// steps 14.1 ms, 14.6 then): held to 64 registers (four CTAs' worth, whatever the sharing) it
// leaves more of the SM to the recurrence CTAs beside it.  With 96 registers, which the compiler
// takes if it may, it is as slow alone and the call takes 14.4 ms.
constexpr int SMEM_BYTES = 4 * 2 * PART_BYTES + 1024;

struct TcArgs {
    const uint8_t* PX;  // panels of V_{k+1}
    const uint8_t* PY;  // panels of V_k (NULL: Ge only)
    int G;              // column groups of the panels
    int n_tot;
    int64_t n_panels;
    int n_e, n_o;       // slabs of the Ge and Go products
    int64_t pan_e, pan_o;  // panels per slab
    float* part_e;      // [n_e][n_tot][n_tot]
    float* part_o;      // [n_o][n_tot][n_tot]
    int* flag;
    const int2* slabs;  // NULL: uniform slabs; else panel range [x, y) of every CTA
    int both;           // every CTA forms Ge and Go of its slab (n_tot <= 128, PY given)
    uint32_t smem_bytes, tmem_cols;  // of a CTA
};

__global__ void __launch_bounds__(NTHREADS, 4) gram_tc_kernel(TcArgs P) {
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ uint64_t full[STAGES], empty[STAGES], done;
    __shared__ uint32_t tmem_slot;
    __shared__ int fail;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool both = P.both != 0;
    const bool cross = both || (int)blockIdx.x >= P.n_e;  // reads V_k's panels too
    const int slab = (cross && !both) ? (int)blockIdx.x - P.n_e : (int)blockIdx.x;
    const int64_t pan = (cross && !both) ? P.pan_o : P.pan_e;
    int64_t p0 = (int64_t)slab * pan;
    int64_t p1 = p0 + pan;
    if (P.slabs) {
        const int2 r = P.slabs[blockIdx.x];
        p0 = r.x;
        p1 = r.y;
    }
    if (p1 > P.n_panels) p1 = P.n_panels;
    const int nch = p1 > p0 ? (int)(p1 - p0) : 0;
    const int nsrc = cross ? 2 : 1;
    const int n_tot = P.n_tot, G = P.G;
    const int ntp = (n_tot + 15) / 16 * 16;  // N of an M = 128 MMA is a multiple of 16
    // a stage: nsrc sources x PS panels x (hi, lo) parts of G groups.  An M = 128 operand
    // reads 16 groups and an N operand ntp / 8 from its start: past the part's G groups
    // that is whatever follows (the next part, the next stage, or the room kept after the
    // ring), and only accumulator rows and columns >= n_tot, never stored, depend on it.
    const uint32_t part_bytes = (uint32_t)G * GROUP_BYTES;
    const uint32_t panel_bytes = 2 * part_bytes;
    const uint32_t over = (uint32_t)((G <= 16 ? 16 : 32) - G) * GROUP_BYTES;
    uint32_t PS = 1;
    while (PS < (uint32_t)MAX_PS && 4u * nsrc * 2 * PS * panel_bytes <= P.smem_bytes - over) PS *= 2;
    const uint32_t src_bytes = PS * panel_bytes;
    const uint32_t stage_bytes = (uint32_t)nsrc * src_bytes;
    int nstage = (int)((P.smem_bytes - over) / stage_bytes);
    if (nstage > STAGES) nstage = STAGES;
    if (nstage < 1) nstage = 1;
    const int nsg = (nch + (int)PS - 1) / (int)PS;  // stages of this slab
    float* out = (cross && !both) ? P.part_o + (size_t)slab * n_tot * n_tot : P.part_e + (size_t)slab * n_tot * n_tot;

    if (warp == 0) {
        tmem_alloc(&tmem_slot, P.tmem_cols);
    }
    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&done, 1);
        fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;

    // Two tiles at most: M block 0 (columns 0..127 of V_{k+1}) and M block 1 (128..255), or
    // with `both` Ge and Go of block 0.  A tile's second operand: V_{k+1}'s panels or V_k's
    // (y), from column group bg, N columns, accumulated in TMEM columns dc ...
    struct Tile {
        int ag, bg, n, dc, m0, n0;
        bool y;
        float* out;
    };
    Tile t0{0, 0, ntp, 0, 0, 0, cross, out}, t1{16, 0, 0, ntp, 128, 0, cross, out};
    if (both) {  // ntp <= 128: tile 0 = Ge, tile 1 = Go in the next ntp columns
        t0.y = false;
        t1 = Tile{0, 0, ntp, ntp, 0, 0, true, P.part_o + (size_t)slab * n_tot * n_tot};
    } else if (ntp > 128) {
        if (!cross) {  // upper blocks only
            t1.bg = 16;
            t1.n = ntp - 128;
            t1.n0 = 128;
        } else {
            t1.n = ntp;
        }
    }

    if (warp == 0) {
        if (lane == 0) {  // producer: bulk copies of runs of panels into the ring
            const uint8_t* px = P.PX + (size_t)p0 * panel_bytes;
            const uint8_t* py = P.PY + (size_t)p0 * panel_bytes;
            for (int c = 0; c < nsg; ++c) {
                const int s = c % nstage;
                if (c >= nstage && !mbar_wait_sleep(smem_u32(&empty[s]), ((c / nstage) - 1) & 1, nullptr)) {
                    atomicOr(&fail, 1);
                    break;
                }
                const uint32_t np = min(PS, (uint32_t)(nch - c * (int)PS)), bytes = np * panel_bytes;
                const uint32_t dst = smem_u32(smem + s * stage_bytes);
                mbar_expect_tx(&full[s], (uint32_t)nsrc * bytes);
                bulk_copy(dst, px + (size_t)c * src_bytes, bytes, &full[s]);
                if (nsrc == 2) bulk_copy(dst + src_bytes, py + (size_t)c * src_bytes, bytes, &full[s]);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {  // MMA issuer
            // descriptors of the first stage's first panel (the address field counts 16 bytes
            // and the shared memory ends below 2^18, so offsets are plain additions)
            const uint64_t base = smem_desc(smem_u32(smem), 128, GROUP_BYTES);
            const uint32_t part = part_bytes >> 4, panel = panel_bytes >> 4, grp = GROUP_BYTES >> 4;
            const uint32_t id0 = instr_desc(t0.n), id1 = instr_desc(t1.n);
            const uint32_t d0 = tmem + (uint32_t)t0.dc, d1 = tmem + (uint32_t)t1.dc;
            const uint32_t b0 = (t0.y ? src_bytes >> 4 : 0u) + (uint32_t)t0.bg * grp;
            const uint32_t b1 = (t1.y ? src_bytes >> 4 : 0u) + (uint32_t)t1.bg * grp, a1 = (uint32_t)t1.ag * grp;
            const bool two = t1.n > 0;
            uint32_t acc = 0;  // the first MMA into each accumulator overwrites it
            bool ok = true;
            auto issue = [&](uint32_t d, uint64_t a, uint64_t b, uint32_t id) {
#pragma unroll
                for (int kk = 0; kk < KC / 16; ++kk) {
                    const uint32_t o = 2 * kk * 128 / 16;
                    mma_bf16(d, a + o, b + o, id, kk == 0 ? acc : 1u);
                    mma_bf16(d, a + o, b + part + o, id, 1u);
                    mma_bf16(d, a + part + o, b + o, id, 1u);
                }
            };
            for (int c = 0; c < nsg; ++c) {
                const int s = c % nstage;
                if (!mbar_wait_sleep(smem_u32(&full[s]), (c / nstage) & 1, nullptr)) {
                    ok = false;
                    wait_copies(full, nstage, c, min(nsg, c + nstage));  // those before have landed
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t np = min(PS, (uint32_t)(nch - c * (int)PS));
                uint64_t x = base + (uint64_t)((uint32_t)s * (stage_bytes >> 4));
                for (uint32_t p = 0; p < np; ++p, x += panel) {
                    issue(d0, x, x + b0, id0);
                    if (two) issue(d1, x + a1, x + b1, id1);
                    acc = 1;
                }
                umma_commit(&empty[s]);
            }
            if (!ok) atomicOr(&fail, 1);
            if (acc)
                umma_commit(&done);  // arrives once every MMA issued above has completed
            else
                mbar_arrive(&done);
        }
        __syncwarp();
    }
    const bool dn = mbar_wait_sleep(smem_u32(&done), 0, nullptr);
    __syncthreads();
    const bool ok = dn && fail == 0;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok) {
        // each lane holds one accumulator row; 32 columns per TMEM round trip go out
        // through a per-warp 32 x 33 shared-memory tile (the stage ring is free now) as
        // coalesced 128-byte row stores; two warps share 32 rows (a warp reaches the TMEM
        // lanes of its number mod 4) and take every other run of columns
        float* tbuf = reinterpret_cast<float*>(smem) + (size_t)warp * 32 * 33;
        auto store = [&](const Tile& t) {
            const int q = warp & 3, mrow0 = t.m0 + 32 * q;
            if (mrow0 >= n_tot) return;
            for (int cc = 32 * (warp >> 2); cc < t.n; cc += 64) {
                float v[32];
                const int w = t.n - cc >= 32 ? 32 : 16;
                if (nch > 0) {
                    const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(t.dc + cc);
                    if (w == 32)
                        tmem_ld32(ta, v);
                    else
                        tmem_ld16(ta, v);
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = 0.f;
                }
#pragma unroll
                for (int j = 0; j < 32; ++j) tbuf[lane * 33 + j] = v[j];
                __syncwarp();
                const int col = t.n0 + cc + lane;
                if (lane < w && col < n_tot) {
                    const int nr = min(32, n_tot - mrow0);
                    for (int rr = 0; rr < nr; ++rr) t.out[(size_t)(mrow0 + rr) * n_tot + col] = tbuf[rr * 33 + lane];
                }
                __syncwarp();
            }
        };
        store(t0);
        if (t1.n > 0) store(t1);
    } else if (tid == 0) {
        atomicOr(P.flag, 2);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        tmem_dealloc(tmem, P.tmem_cols);
}

// Compensated (Neumaier) float32 sum: the slab partials are float32, and their
// sum in this form keeps float64-level accuracy with float32 operations only
// (float64 runs at 1/58 of the float32 rate on this part and was the bound of
// a plain float64 sum of ~150 partials per element and step).
struct Sum32 {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float t = s + x;
        c += fabsf(s) >= fabsf(x) ? (s - t) + x : (x - t) + s;
        s = t;
    }
    __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

// s.add(p[k nn + e]) for k = k0, k0 + 8, k0 + 16, ... < n, in that order; the loads of
// four slabs are issued before their adds (a zero added to a compensated sum leaves it
// unchanged, so the tail needs no separate loop).
__device__ __forceinline__ void sum_slabs(Sum32& s, const float* __restrict__ p, size_t nn, size_t e, int k0, int n) {
    for (int k = k0; k < n; k += 32) {
        const float v0 = p[(size_t)k * nn + e];
        const float v1 = k + 8 < n ? p[(size_t)(k + 8) * nn + e] : 0.f;
        const float v2 = k + 16 < n ? p[(size_t)(k + 16) * nn + e] : 0.f;
        const float v3 = k + 24 < n ? p[(size_t)(k + 24) * nn + e] : 0.f;
        s.add(v0);
        s.add(v1);
        s.add(v2);
        s.add(v3);
    }
}

// Slab sums (compensated float32 per warp, float64 across warps), coalesced: ge[e] = sum_s pe[s][lo][hi] (upper element of
// the pair), go[e] = sum_s po[s][e]; the symmetrisation of go reads it transposed
// from this small float64 buffer in a second pass.  A block covers 32
// consecutive elements; its 8 warps take every 8th slab and their partial
// sums are added in warp order, so the result is independent of timing.
__global__ void __launch_bounds__(256)
sum_tc_kernel(const float* __restrict__ pe, int n_e, const float* __restrict__ po, int n_o, int n_tot,
              double* __restrict__ ge, double* __restrict__ go) {
    __shared__ double se[8][32], so[8][32];
    const size_t nn = (size_t)n_tot * n_tot;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (size_t e0 = (size_t)blockIdx.x * 32; e0 < nn; e0 += (size_t)gridDim.x * 32) {
        const size_t e = e0 + lane;
        Sum32 a, b;
        if (e < nn) {
            const int i = (int)(e / n_tot), j = (int)(e - (size_t)i * n_tot);
            if (i <= j) sum_slabs(a, pe, nn, e, w, n_e);
            sum_slabs(b, po, nn, e, w, n_o);
        }
        se[w][lane] = a.value();
        so[w][lane] = b.value();
        __syncthreads();
        if (w == 0 && e < nn) {
            double a = 0.0, b = 0.0;
            for (int k = 0; k < 8; ++k) {
                a += se[k][lane];
                b += so[k][lane];
            }
            ge[e] = a;
            go[e] = b;
        }
        __syncthreads();
    }
}

// One launch for a whole ring batch: blockIdx.y selects the step.
__global__ void __launch_bounds__(256)
sum_tc_batch_kernel(const float* __restrict__ ring, size_t slot, int n_e, int n_o, int n_tot,
                    double* __restrict__ ge, double* __restrict__ go) {
    __shared__ double se[8][32], so[8][32];
    const size_t nn = (size_t)n_tot * n_tot;
    const float* pe = ring + (size_t)blockIdx.y * slot;
    const float* po = pe + (size_t)n_e * nn;
    double* gq = ge + (size_t)blockIdx.y * nn;
    double* oq = go + (size_t)blockIdx.y * nn;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (size_t e0 = (size_t)blockIdx.x * 32; e0 < nn; e0 += (size_t)gridDim.x * 32) {
        const size_t e = e0 + lane;
        Sum32 a, b;
        if (e < nn) {
            const int i = (int)(e / n_tot), j = (int)(e - (size_t)i * n_tot);
            if (i <= j) sum_slabs(a, pe, nn, e, w, n_e);
            sum_slabs(b, po, nn, e, w, n_o);
        }
        se[w][lane] = a.value();
        so[w][lane] = b.value();
        __syncthreads();
        if (w == 0 && e < nn) {
            double a = 0.0, b = 0.0;
            for (int k = 0; k < 8; ++k) {
                a += se[k][lane];
                b += so[k][lane];
            }
            gq[e] = a;
            oq[e] = b;
        }
        __syncthreads();
    }
}

__global__ void moments_tc_kernel(const double* __restrict__ ge, const double* __restrict__ go, int n_tot,
                                  double* __restrict__ X, int step) {
    const size_t nn = (size_t)n_tot * n_tot;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < nn; e += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / n_tot), j = (int)(e - (size_t)i * n_tot);
        const double gs = (i <= j) ? ge[e] : ge[(size_t)j * n_tot + i];
        const double gc = 0.5 * (go[e] + go[(size_t)j * n_tot + i]);
        if (step < 0) {
            X[e] = gs;
        } else if (step == 0) {
            X[nn + e] = gc;
            X[2 * nn + e] = 2.0 * gs - X[e];
        } else {
            X[(size_t)(2 * step + 1) * nn + e] = 2.0 * gc - X[nn + e];
            X[(size_t)(2 * step + 2) * nn + e] = 2.0 * gs - X[e];
        }
    }
}

__global__ void moments_tc_batch_kernel(const double* __restrict__ ge, const double* __restrict__ go, int n_tot,
                                        double* __restrict__ X, int k0) {
    const size_t nn = (size_t)n_tot * n_tot;
    const int q = blockIdx.y, step = k0 + q;
    const double* gq = ge + (size_t)q * nn;
    const double* oq = go + (size_t)q * nn;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < nn; e += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / n_tot), j = (int)(e - (size_t)i * n_tot);
        const double gs = (i <= j) ? gq[e] : gq[(size_t)j * n_tot + i];
        const double gc = 0.5 * (oq[e] + oq[(size_t)j * n_tot + i]);
        X[(size_t)(2 * step + 1) * nn + e] = 2.0 * gc - X[nn + e];
        X[(size_t)(2 * step + 2) * nn + e] = 2.0 * gs - X[e];
    }
}

// Batched plans: the blockIdx.y-th matrix b of `order` (NULL: b itself) sums its own slabs
// (Ge slabs [se[b], se[b+1]), Go slabs [so[b], so[b+1])), in the fixed order of sum_tc_kernel.
__global__ void __launch_bounds__(256)
sum_tc_seg_kernel(const float* __restrict__ pe, const float* __restrict__ po, const int* __restrict__ seg,
                  const int* __restrict__ order, int B, int n_tot, bool odd, double* __restrict__ ge, double* __restrict__ go) {
    __shared__ double se_[8][32], so_[8][32];
    const size_t nn = (size_t)n_tot * n_tot;
    const int b = order ? order[blockIdx.y] : (int)blockIdx.y;
    const int e0s = seg[b], e1s = seg[b + 1], o0s = seg[B + 1 + b], o1s = seg[B + 2 + b];
    double* gq = ge + (size_t)b * nn;
    double* oq = go + (size_t)b * nn;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (size_t e0 = (size_t)blockIdx.x * 32; e0 < nn; e0 += (size_t)gridDim.x * 32) {
        const size_t e = e0 + lane;
        Sum32 a, b;
        if (e < nn) {
            const int i = (int)(e / n_tot), j = (int)(e - (size_t)i * n_tot);
            if (i <= j) sum_slabs(a, pe, nn, e, e0s + w, e1s);
            if (odd) sum_slabs(b, po, nn, e, o0s + w, o1s);
        }
        se_[w][lane] = a.value();
        so_[w][lane] = b.value();
        __syncthreads();
        if (w == 0 && e < nn) {
            double a = 0.0, c = 0.0;
            for (int k = 0; k < 8; ++k) {
                a += se_[k][lane];
                c += so_[k][lane];
            }
            gq[e] = a;
            oq[e] = c;
        }
        __syncthreads();
    }
}

__global__ void moments_tc_seg_kernel(const double* __restrict__ ge, const double* __restrict__ go,
                                      const int* __restrict__ order, int n_tot, double* __restrict__ X, size_t xstride,
                                      int step) {
    const size_t nn = (size_t)n_tot * n_tot;
    const int b = order ? order[blockIdx.y] : (int)blockIdx.y;
    const double* gq = ge + (size_t)b * nn;
    const double* oq = go + (size_t)b * nn;
    double* Xb = X + (size_t)b * xstride;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < nn; e += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / n_tot), j = (int)(e - (size_t)i * n_tot);
        const double gs = (i <= j) ? gq[e] : gq[(size_t)j * n_tot + i];
        const double gc = 0.5 * (oq[e] + oq[(size_t)j * n_tot + i]);
        if (step < 0) {
            Xb[e] = gs;
        } else if (step == 0) {
            Xb[nn + e] = gc;
            Xb[2 * nn + e] = 2.0 * gs - Xb[e];
        } else {
            Xb[(size_t)(2 * step + 1) * nn + e] = 2.0 * gc - Xb[nn + e];
            Xb[(size_t)(2 * step + 2) * nn + e] = 2.0 * gs - Xb[e];
        }
    }
}

// The same sums and the moments of a step in one launch, for small matrices (the order's
// from n_many on): one thread an element pair (i, j), (j, i), the chains of sum_tc_kernel one
// after the other (an empty chain adds nothing).
__device__ __forceinline__ double chain_sum(const float* __restrict__ p, size_t nn, size_t e, int k0, int k1) {
    double s = 0.0;
    const int k8 = min(k1, k0 + 8);
#pragma unroll 1
    for (int k = k0; k < k8; ++k) {
        Sum32 a;
        sum_slabs(a, p, nn, e, k, k1);
        s += a.value();
    }
    return s;
}

__global__ void __launch_bounds__(256)
step_tc_seg_kernel(const float* __restrict__ pe, const float* __restrict__ po, const int* __restrict__ seg,
                   const int* __restrict__ order, int B, int n_tot, double* __restrict__ X, size_t xstride, int step) {
    const size_t nn = (size_t)n_tot * n_tot;
    const int b = order ? order[blockIdx.y] : (int)blockIdx.y;
    const int e0 = seg[b], e1 = seg[b + 1], o0 = seg[B + 1 + b], o1 = seg[B + 2 + b];
    double* Xb = X + (size_t)b * xstride;
    const unsigned npair = (unsigned)n_tot * (n_tot + 1) / 2;
    for (unsigned u = blockIdx.x * blockDim.x + threadIdx.x; u < npair; u += gridDim.x * blockDim.x) {
        // u -> (i, j), i <= j: row i of the upper triangle starts at i n_tot - i (i - 1) / 2
        const unsigned m = npair - 1 - u;  // counted from the end: t (t + 1) / 2 <= m
        unsigned t = (unsigned)((sqrtf(8.f * (float)m + 1.f) - 1.f) * 0.5f);
        while (t * (t + 1) / 2 > m) --t;
        while ((t + 1) * (t + 2) / 2 <= m) ++t;
        const unsigned i = n_tot - 1 - t, j = n_tot - 1 - (m - t * (t + 1) / 2);
        const size_t e = (size_t)i * n_tot + j, tr = (size_t)j * n_tot + i;
        const double gs = chain_sum(pe, nn, e, e0, e1);
        if (step < 0) {
            Xb[e] = Xb[tr] = gs;
            continue;
        }
        const double gc = 0.5 * (chain_sum(po, nn, e, o0, o1) + chain_sum(po, nn, tr, o0, o1));
        const double x0 = Xb[e];
        if (step == 0) {
            Xb[nn + e] = Xb[nn + tr] = gc;
            Xb[2 * nn + e] = Xb[2 * nn + tr] = 2.0 * gs - x0;
        } else {
            double* odd = Xb + (size_t)(2 * step + 1) * nn;
            double* even = Xb + (size_t)(2 * step + 2) * nn;
            odd[e] = odd[tr] = 2.0 * gc - Xb[nn + e];
            even[e] = even[tr] = 2.0 * gs - x0;
        }
    }
}

// Fused-step partials (fused_tc.cu): slab s holds accumulator rows 0..127 for
// s < nA and rows 128.. for s >= nA, so element (i, j) sums the slabs of its
// row range, in the fixed order of sum_tc_kernel.  blockIdx.y selects the step.
__global__ void __launch_bounds__(256)
sum_fused_kernel(const float* __restrict__ ring, size_t slot, int nA, int nF, int n_tot, double* __restrict__ ge,
                 double* __restrict__ go) {
    __shared__ double se[8][32], so[8][32];
    const size_t nn = (size_t)n_tot * n_tot;
    const float* pe = ring + (size_t)blockIdx.y * slot;
    const float* po = pe + (size_t)nF * nn;
    double* gq = ge + (size_t)blockIdx.y * nn;
    double* oq = go + (size_t)blockIdx.y * nn;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (size_t e0 = (size_t)blockIdx.x * 32; e0 < nn; e0 += (size_t)gridDim.x * 32) {
        const size_t e = e0 + lane;
        Sum32 a, b;
        if (e < nn) {
            const int i = (int)(e / n_tot), j = (int)(e - (size_t)i * n_tot);
            const int s0 = i < 128 ? 0 : nA, s1 = i < 128 ? nA : nF;
            if (i <= j) sum_slabs(a, pe, nn, e, s0 + w, s1);
            sum_slabs(b, po, nn, e, s0 + w, s1);
        }
        se[w][lane] = a.value();
        so[w][lane] = b.value();
        __syncthreads();
        if (w == 0 && e < nn) {
            double a = 0.0, b = 0.0;
            for (int k = 0; k < 8; ++k) {
                a += se[k][lane];
                b += so[k][lane];
            }
            gq[e] = a;
            oq[e] = b;
        }
        __syncthreads();
    }
}

}  // namespace

cudaError_t launch_reduce_fused(const float* ring, size_t slot, int nA, int nF, int n_tot, double* X, int k0,
                                int nk, double* ge, double* go, cudaStream_t s) {
    if (k0 == 0 && nk != 1) return cudaErrorInvalidValue;
    const int64_t nn = (int64_t)n_tot * n_tot;
    int64_t sb = (nn + 31) / 32;
    if (sb > 1024) sb = 1024;
    sum_fused_kernel<<<dim3((unsigned)sb, (unsigned)nk), 256, 0, s>>>(ring, slot, nA, nF, n_tot, ge, go);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const unsigned mb = (unsigned)((nn + 255) / 256 > 512 ? 512 : (nn + 255) / 256);
    if (k0 == 0)
        moments_tc_kernel<<<mb, 256, 0, s>>>(ge, go, n_tot, X, 0);
    else
        moments_tc_batch_kernel<<<dim3(mb, (unsigned)nk), 256, 0, s>>>(ge, go, n_tot, X, k0);
    return cudaGetLastError();
}

bool gram_tc_supported(int n_tot, int ld) { return n_tot >= 1 && n_tot <= 256 && (ld % 4) == 0; }

int gram_tc_groups(int n_tot) { return (n_tot + 7) / 8; }

void gram_tc_slabs(int64_t n_rows, int* n_e, int* n_o) {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // Go CTAs read two blocks: give them half the panels (a third of the SMs each way round)
    int e = sms / 3, o = sms - e;
    const int64_t cap = (n_rows + KC - 1) / KC;
    if (e > cap) e = (int)cap;
    if (o > cap) o = (int)cap;
    *n_e = e < 1 ? 1 : e;
    *n_o = o < 1 ? 1 : o;
}

size_t gram_tc_partial_floats(int n_e, int n_o, int n_tot) { return (size_t)(n_e + n_o) * n_tot * n_tot; }

cudaError_t launch_gram_tc(const uint8_t* PX, const uint8_t* PY, int n_tot, int64_t n_rows, int n_e, int n_o,
                           float* part, int* flag, cudaStream_t s, const int2* slabs, bool both) {
    if (both && (!slabs || n_o != n_e || n_tot > 128)) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(gram_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (e != cudaSuccess) return e;
    TcArgs a;
    a.PX = PX;
    a.PY = PY;
    a.G = gram_tc_groups(n_tot);
    a.n_tot = n_tot;
    a.n_panels = (n_rows + KC - 1) / KC;
    a.n_e = n_e;
    a.n_o = PY ? n_o : 0;
    a.pan_e = (a.n_panels + n_e - 1) / n_e;
    a.pan_o = (a.n_panels + n_o - 1) / n_o;
    a.part_e = part;
    a.part_o = part + (size_t)n_e * n_tot * n_tot;
    a.flag = flag;
    a.slabs = slabs;
    a.both = both && PY;
    // Narrow blocks in small slabs (batched plans): a CTA's life is its latencies, one after
    // the other (allocation, first copies, MMA chain, epilogue), so four share an SM (n_tot <=
    // 32; two up to 64, whose ring would be one stage), each with its part of the tensor memory
    // and of the shared memory.  1100 slabs of about 16 panels, the recurrence graph of 50
    // steps: n_tot = 32 10.1 ms with one, 8.8 with two, 8.1 with four; n_tot = 16 6.6, 5.3 and
    // 4.8; n_tot = 56 14.8 with two, 15.2 with four.
    const int ntp = (n_tot + 15) / 16 * 16, sms = device_sms();
    int share = 1;
    if (slabs && ntp <= 64 && n_e >= 2 * sms) share = ntp <= 32 && n_e >= 4 * sms ? 4 : 2;
    a.smem_bytes = SMEM_BYTES / share;
    a.tmem_cols = TMEM_COLS / share;
    gram_tc_kernel<<<a.both ? a.n_e : a.n_e + a.n_o, NTHREADS, a.smem_bytes, s>>>(a);
    return cudaGetLastError();
}

size_t gram_tc_partial_floats_total(int n_e, int n_o, int n_tot) {
    // float32 partials plus two float64 n_tot^2 sums (4 floats of room each)
    return gram_tc_partial_floats(n_e, n_o, n_tot) + (size_t)4 * n_tot * n_tot;
}

cudaError_t launch_reduce_tc(const float* part, int n_e, int n_o, int n_tot, double* X, int step, cudaStream_t s) {
    const int64_t nn = (int64_t)n_tot * n_tot;
    int64_t b = (nn + 255) / 256;
    if (b > (int64_t)device_sms() * 16) b = (int64_t)device_sms() * 16;
    if (b < 1) b = 1;
    const size_t pf = gram_tc_partial_floats(n_e, n_o, n_tot);
    // the float64 sums live after the float32 partials (8-byte aligned: pf is even)
    double* ge = reinterpret_cast<double*>(const_cast<float*>(part) + ((pf + 1) & ~(size_t)1));
    double* go = ge + nn;
    int64_t sb = (nn + 31) / 32;
    if (sb > (int64_t)device_sms() * 8) sb = (int64_t)device_sms() * 8;
    sum_tc_kernel<<<(int)sb, 256, 0, s>>>(part, n_e, part + (size_t)n_e * nn, step >= 0 ? n_o : 0, n_tot, ge, go);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    moments_tc_kernel<<<(int)b, 256, 0, s>>>(ge, go, n_tot, X, step);
    return cudaGetLastError();
}

// Steps k0 .. k0+nk-1 (k0 >= 1) whose partials sit in ring slots
// (k - k0) of `ring` (each slot [n_e + n_o][n_tot][n_tot] float32); ge/go
// scratch [nk][n_tot][n_tot] float64.
cudaError_t launch_reduce_tc_batch(const float* ring, int n_e, int n_o, int n_tot, double* X, int k0, int nk,
                                   double* ge, double* go, cudaStream_t s) {
    const int64_t nn = (int64_t)n_tot * n_tot;
    const size_t slot = gram_tc_partial_floats(n_e, n_o, n_tot);
    int64_t sb = (nn + 31) / 32;
    if (sb > 1024) sb = 1024;
    dim3 sgrid((unsigned)sb, (unsigned)nk);
    sum_tc_batch_kernel<<<sgrid, 256, 0, s>>>(ring, slot, n_e, n_o, n_tot, ge, go);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((nn + 255) / 256 > 512 ? 512 : (nn + 255) / 256), (unsigned)nk);
    moments_tc_batch_kernel<<<grid, 256, 0, s>>>(ge, go, n_tot, X, k0);
    return cudaGetLastError();
}

// Matrices of few slabs: a thread an element.  The eight warps an element of the other
// kernels spend the float64 pipe on converting and adding zeros there (1100 matrices of one
// slab, n_tot = 32: 125 us and 14 us for the moments, against 24 us); with more slabs they
// share the loads.  Each matrix goes by its own slabs: one of 200000 rows (550 slabs) beside
// 300 of 100, 30 steps: n_tot = 8 3.25 ms with a thread an element for all, 1.68 with eight
// warps for all, 1.77 so; 32: 7.0, 4.7 and 4.0; 64: 10.4, 11.0 and 7.4; 200: 39.8, 63.0 and
// 31.1.  1000 of 300 beside three of 100000: 32 7.4, 10.5 and 7.3.
cudaError_t launch_reduce_tc_seg(const float* part, int n_e, int n_tot, int B, const int* seg, int n_many, double* ge,
                                 double* go, double* X, size_t xstride, int step, cudaStream_t s) {
    const int64_t nn = (int64_t)n_tot * n_tot;
    const float* po = part + (size_t)n_e * nn;
    const int* order = n_many > 0 && n_many < B ? seg + 2 * (B + 1) : nullptr;  // (one kind only: any order)
    if (n_many < B) {
        int64_t pb = (nn / 2 + n_tot + 255) / 256;
        if (pb > 64) pb = 64;
        step_tc_seg_kernel<<<dim3((unsigned)pb, (unsigned)(B - n_many)), 256, 0, s>>>(
            part, po, seg, order ? order + n_many : nullptr, B, n_tot, X, xstride, step);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (n_many > 0) {
        // at most 64 CTAs a matrix, more where few matrices would leave SMs idle
        const int64_t cap = std::max<int64_t>(64, (int64_t)device_sms() * 8 / n_many);
        const int64_t sb = std::min((nn + 31) / 32, cap), mb = std::min((nn + 255) / 256, cap);
        sum_tc_seg_kernel<<<dim3((unsigned)sb, (unsigned)n_many), 256, 0, s>>>(part, po, seg, order, B, n_tot, step >= 0,
                                                                             ge, go);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        moments_tc_seg_kernel<<<dim3((unsigned)mb, (unsigned)n_many), 256, 0, s>>>(ge, go, order, n_tot, X, xstride, step);
    }
    return cudaGetLastError();
}

}  // namespace ssm
