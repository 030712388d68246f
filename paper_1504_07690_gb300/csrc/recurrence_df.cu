// recurrence_df.cu - the block three-term recurrence in float-pair arithmetic
// for the float64-accuracy tensor-core plans (SSM_FP64_TC).
//
//   V_{k+1} = c (2 A~ V_k) - d V_{k-1},   (c, d) = (1/2, 0) first, then (1, 1)
//
// (Alg. 7's loop, Section 2's map folded into the operator).  Every value is
// an unevaluated sum hi + lo of two float32 (|lo| <= 2^-24 |hi|, about 48
// significant bits), stored as two planes of the block (hi: N x ld floats,
// then lo: N x ld floats), and every operation is an error-free float32
// transformation (Knuth's two-sum, Dekker's fast two-sum, fma-based
// products), so the step runs on the float32 pipes (float64 runs at 1/58 of
// that rate here).  Each step also writes U_k = V_{k+1} + V_k, whose Gram
// product gives the odd moments, and the column maxima of |V_{k+1}| and |U_k|
// (bit patterns of |hi| (1 + 2^-22), an upper bound of |hi + lo|) into
// bucket blockIdx.x mod nbucket, for the column scales of the tensor-core
// Gram products (gram_oz.cu).
#include "internal.h"
#include "ozslice.cuh"

namespace ssm {

namespace {

using oz::pair32;
using oz::pair_add;
using oz::pair_fma;
using oz::pair_mul;
using oz::pair_of;
using oz::pair_sub;

struct F2 {
    float h, l;
};

// Two columns' float pairs, each operation on both at once (f32x2 instructions, rounded as
// the scalar ones): the step was bound by instruction issue (65 to 70 % active at 139 us a
// step of 65536 x 200), and this halves the arithmetic (101 us).
struct P2 {
    pair32 h, l;
};

__device__ __forceinline__ P2 two_sum(pair32 a, pair32 b) {
    const pair32 s = pair_add(a, b);
    const pair32 bb = pair_sub(s, a);
    return {s, pair_add(pair_sub(a, pair_sub(s, bb)), pair_sub(b, bb))};
}

__device__ __forceinline__ P2 two_diff(pair32 a, pair32 b) {  // two_sum(a, -b)
    const pair32 s = pair_sub(a, b);
    const pair32 bb = pair_sub(s, a);
    return {s, pair_sub(pair_sub(a, pair_sub(s, bb)), pair_add(b, bb))};
}

__device__ __forceinline__ P2 fast_two_sum(pair32 a, pair32 b) {
    const pair32 s = pair_add(a, b);
    return {s, pair_sub(b, pair_sub(s, a))};
}

__device__ __forceinline__ P2 df_renorm(P2 s, P2 t) {
    s.l = pair_add(s.l, t.h);
    s = fast_two_sum(s.h, s.l);
    s.l = pair_add(s.l, t.l);
    return fast_two_sum(s.h, s.l);
}

// (a.h + a.l) + (b.h + b.l), both parts summed error-free (about 2^-48 relative)
__device__ __forceinline__ P2 df_add(P2 a, P2 b) { return df_renorm(two_sum(a.h, b.h), two_sum(a.l, b.l)); }
__device__ __forceinline__ P2 df_sub(P2 a, P2 b) { return df_renorm(two_diff(a.h, b.h), two_diff(a.l, b.l)); }

// A coefficient for both columns: its parts, the negated leading one, and -0, an argument of
// the kernel: the rounded products below are fmas with it, since a multiply.rn of two
// columns is contracted into the addition after it (which then rounds once, and the error
// terms no longer belong to the sums: 2e-8 in the moments).
struct C2 {
    pair32 h, l, nh, nz;
    __device__ C2(F2 a, float nz0)
        : h(pair_of(a.h, a.h)), l(pair_of(a.l, a.l)), nh(pair_of(-a.h, -a.h)), nz(pair_of(nz0, nz0)) {}
};

__device__ __forceinline__ P2 df_mul(const C2& a, P2 b) {
    const pair32 p = pair_fma(a.h, b.h, a.nz);
    pair32 e = pair_fma(a.h, b.h, pair_fma(a.nh, b.h, a.nz));  // the product's rounding error
    e = pair_fma(a.h, b.l, e);
    e = pair_fma(a.l, b.h, e);
    return fast_two_sum(p, e);
}

struct DfBlock {
    const float* h;
    const float* l;
};

struct DfOut {
    float* vh;
    float* vl;
    float* uh;
    float* ul;
    unsigned long long* cmv;
    unsigned long long* cmu;
    uint32_t nbucket;
    float nz;  // -0
};

__device__ __forceinline__ unsigned long long bound_bits(float h) {
    // |hi + lo| <= |hi| (1 + 2^-24) < |hi| (1 + 2^-22), rounded up in float64
    return (unsigned long long)__double_as_longlong((double)fabsf(h) * (1.0 + 0x1.0p-22));
}

// A CTA of (nch, ty) threads takes up to DF_ROWS ty consecutive rows: thread (x, y) owns the
// 16-byte column chunk x (four columns, float4 loads and stores of each plane) of rows y,
// y + ty, ..., so no thread idles whatever the number of columns; it keeps the column
// maxima of its rows in registers, and the CTA combines them in shared memory before one
// atomicMax per column.
constexpr int DF_ROWS = 8, DF_THREADS = 256, DF_MAXCH = 64;

struct Q4 {  // four columns
    P2 v[2];
};

__device__ __forceinline__ P2 pair2(float h0, float h1, float l0, float l1) {
    return {pair_of(h0, h1), pair_of(l0, l1)};
}

__device__ __forceinline__ Q4 ld4(const DfBlock& b, size_t i4) {
    const float4 h = __ldg(reinterpret_cast<const float4*>(b.h) + i4);
    const float4 l = __ldg(reinterpret_cast<const float4*>(b.l) + i4);
    return {{pair2(h.x, h.y, l.x, l.y), pair2(h.z, h.w, l.z, l.w)}};
}

__device__ __forceinline__ float4 four(pair32 a, pair32 b) {
    float4 f;
    oz::pair_get(a, f.x, f.y);
    oz::pair_get(b, f.z, f.w);
    return f;
}

// Stores a block's four columns; returns the leading parts for the maxima.
__device__ __forceinline__ float4 st4(float* h, float* l, size_t i4, const Q4& a) {
    const float4 fh = four(a.v[0].h, a.v[1].h);
    reinterpret_cast<float4*>(h)[i4] = fh;
    reinterpret_cast<float4*>(l)[i4] = four(a.v[0].l, a.v[1].l);
    return fh;
}

__device__ __forceinline__ void track(float* m, float4 f) {
    m[0] = fmaxf(m[0], fabsf(f.x));
    m[1] = fmaxf(m[1], fabsf(f.y));
    m[2] = fmaxf(m[2], fabsf(f.z));
    m[3] = fmaxf(m[3], fabsf(f.w));
}

// v = c acc - d vp, u = v + x for four columns; running maxima of |v.h|, |u.h|
__device__ __forceinline__ void finish4(const Q4& acc, const Q4& x, const Q4& p, size_t i4, pair32 c, float d,
                                        const DfOut& out, float* mv, float* mu) {
    Q4 v, u;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        v.v[q] = {pair_mul(acc.v[q].h, c), pair_mul(acc.v[q].l, c)};  // c a power of two: exact
        if (d != 0.f) v.v[q] = df_sub(v.v[q], p.v[q]);
        u.v[q] = df_add(v.v[q], x.v[q]);
    }
    track(mv, st4(out.vh, out.vl, i4, v));
    track(mu, st4(out.uh, out.ul, i4, u));
}

__device__ __forceinline__ void flush_max(const float* mv, const float* mu, uint32_t n_cols, uint32_t ld,
                                          const DfOut& out) {
    __shared__ float smax[2][DF_THREADS * 4];  // [y][column]
    const uint32_t cols = 4 * blockDim.x, at = threadIdx.y * cols + 4 * threadIdx.x;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        smax[0][at + q] = mv[q];
        smax[1][at + q] = mu[q];
    }
    __syncthreads();
    const uint32_t t = threadIdx.y * blockDim.x + threadIdx.x, nt = blockDim.x * blockDim.y;
    const size_t b = (size_t)(blockIdx.x % out.nbucket) * ld;
    for (uint32_t col = t; col < n_cols; col += nt) {
        float a = 0.f, u = 0.f;
        for (uint32_t y = 0; y < blockDim.y; ++y) {
            a = fmaxf(a, smax[0][y * cols + col]);
            u = fmaxf(u, smax[1][y * cols + col]);
        }
        if (a > 0.f) atomicMax(out.cmv + b + col, bound_bits(a));
        if (u > 0.f) atomicMax(out.cmu + b + col, bound_bits(u));
    }
}

__global__ void __launch_bounds__(DF_THREADS)
stencil_step_df_kernel(DfBlock Vc, DfBlock Vp, const float* __restrict__ dgh, const float* __restrict__ dgl,
                       StencilGeom g, F2 o0, F2 o1, F2 o2, float c, float d, uint32_t ld, uint32_t n_cols,
                       uint32_t n_rows, DfOut out) {
    const uint32_t cx = threadIdx.x, nch = blockDim.x;
    const uint32_t s1 = g.d2, s0 = g.d1 * g.d2;
    const F2 o[3] = {o0, o1, o2};
    const pair32 c2 = pair_of(c, c);
    float mv[4] = {0.f, 0.f, 0.f, 0.f}, mu[4] = {0.f, 0.f, 0.f, 0.f};
    const uint32_t first = blockIdx.x * (DF_ROWS * blockDim.y) + threadIdx.y;
    for (uint32_t k = 0; k < DF_ROWS; ++k) {
        const uint32_t i = first + k * blockDim.y;
        if (i >= n_rows) break;
        const size_t i4 = (size_t)i * nch + cx;
        const Q4 x = ld4(Vc, i4);
        const C2 dg(F2{__ldg(dgh + i), __ldg(dgl + i)}, out.nz);
        const uint32_t i2 = i % g.d2, qq = i / g.d2, i1 = qq % g.d1, i0 = qq / g.d1;
        const uint32_t co[3] = {i0, i1, i2}, ex[3] = {g.d0, g.d1, g.d2}, sd[3] = {s0, s1, 1u};
        Q4 p{};
        if (d != 0.f) p = ld4(Vp, i4);
        Q4 acc;
#pragma unroll
        for (int q = 0; q < 2; ++q) acc.v[q] = df_mul(dg, x.v[q]);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (!g.active[a]) continue;
            const uint32_t cm = co[a], exa = ex[a], st = sd[a];
            const bool lo = cm > 0 || g.per[a], hi = cm + 1 < exa || g.per[a];
            Q4 nl{}, nh{};
            if (lo) nl = ld4(Vc, (size_t)(cm > 0 ? i - st : i + (exa - 1) * st) * nch + cx);
            if (hi) nh = ld4(Vc, (size_t)(cm + 1 < exa ? i + st : i - (exa - 1) * st) * nch + cx);
            const C2 w(o[a], out.nz);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                P2 sum{0, 0};
                if (lo) sum = nl.v[q];
                if (hi) sum = lo ? df_add(sum, nh.v[q]) : nh.v[q];
                acc.v[q] = df_add(acc.v[q], df_mul(w, sum));
            }
        }
        finish4(acc, x, p, i4, c2, d, out, mv, mu);
    }
    flush_max(mv, mu, n_cols, ld, out);
}

__global__ void __launch_bounds__(DF_THREADS)
csr_step_df_kernel(DfBlock Vc, DfBlock Vp, const int64_t* __restrict__ rowptr, const int32_t* __restrict__ colind,
                   const float* __restrict__ vh, const float* __restrict__ vl, F2 beta, float c, float d,
                   uint32_t ld, uint32_t n_cols, uint32_t n_rows, uint32_t per, DfOut out) {
    const uint32_t cx = threadIdx.x, nch = blockDim.x;
    const pair32 c2 = pair_of(c, c);
    float mv[4] = {0.f, 0.f, 0.f, 0.f}, mu[4] = {0.f, 0.f, 0.f, 0.f};
    const uint32_t first = blockIdx.x * (per * blockDim.y) + threadIdx.y;
    for (uint32_t k = 0; k < per; ++k) {
        const uint32_t i = first + k * blockDim.y;
        if (i >= n_rows) break;
        const size_t i4 = (size_t)i * nch + cx;
        const Q4 x = ld4(Vc, i4);
        Q4 p{};
        if (d != 0.f) p = ld4(Vp, i4);
        Q4 acc;
        const C2 b2(beta, out.nz);
#pragma unroll
        for (int q = 0; q < 2; ++q) acc.v[q] = df_mul(b2, x.v[q]);
        const int64_t e1 = __ldg(rowptr + i + 1);
        for (int64_t e = __ldg(rowptr + i); e < e1; ++e) {
            const uint32_t j = (uint32_t)__ldg(colind + e);
            const C2 a(F2{__ldg(vh + e), __ldg(vl + e)}, out.nz);
            const Q4 y = ld4(Vc, (size_t)j * nch + cx);
#pragma unroll
            for (int q = 0; q < 2; ++q) acc.v[q] = df_add(acc.v[q], df_mul(a, y.v[q]));
        }
        finish4(acc, x, p, i4, c2, d, out, mv, mu);
    }
    flush_max(mv, mu, n_cols, ld, out);
}

// float64 block (leading dimension ldsrc) -> float pairs (leading dimension ld,
// columns >= n_cols zero) and the column maxima of V_0.
__global__ void __launch_bounds__(256)
convert_in_df_kernel(const double* __restrict__ src, int64_t ldsrc, float* __restrict__ h, float* __restrict__ l,
                     uint32_t ld, uint32_t n_cols, uint32_t n_rows, unsigned long long* cm, uint32_t nbucket) {
    extern __shared__ unsigned long long df_cm3[];
    for (uint32_t q = threadIdx.x; q < ld; q += blockDim.x) df_cm3[q] = 0ull;
    __syncthreads();
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < (size_t)n_rows * ld;
         e += (size_t)gridDim.x * blockDim.x) {
        const uint32_t col = (uint32_t)(e % ld);
        const size_t i = e / ld;
        const double v = col < n_cols ? src[i * ldsrc + col] : 0.0;
        const float vh = (float)v;
        h[e] = vh;
        l[e] = (float)(v - (double)vh);
        if (col < n_cols) atomicMax(df_cm3 + col, bound_bits(vh));
    }
    __syncthreads();
    const size_t b = (size_t)(blockIdx.x % nbucket) * ld;
    for (uint32_t q = threadIdx.x; q < n_cols; q += blockDim.x)
        if (df_cm3[q]) atomicMax(cm + b + q, df_cm3[q]);
}

F2 split_f2(double v) {
    const float h = (float)v;
    return {h, (float)(v - (double)h)};
}

}  // namespace

cudaError_t launch_convert_in_df(const double* src, int64_t ldsrc, void* dst, int ld, int64_t n_rows, int n_cols,
                                 unsigned long long* cm, int nbucket, cudaStream_t s) {
    float* h = (float*)dst;
    float* l = h + (size_t)n_rows * ld;
    int64_t blocks = ((int64_t)n_rows * ld + 255) / 256;
    if (blocks > (int64_t)device_sms() * 16) blocks = (int64_t)device_sms() * 16;
    convert_in_df_kernel<<<(int)(blocks < 1 ? 1 : blocks), 256, (size_t)ld * 8, s>>>(
        src, ldsrc, h, l, (uint32_t)ld, (uint32_t)n_cols, (uint32_t)n_rows, cm, (uint32_t)nbucket);
    return cudaGetLastError();
}

cudaError_t launch_step_df(const Plan& P, const void* Vc, const void* Vp, void* Vn, void* Un, float c, float d,
                           unsigned long long* cmv, unsigned long long* cmu, int nbucket, cudaStream_t s) {
    const size_t plane = (size_t)P.n * P.ld;
    const DfBlock vc{(const float*)Vc, (const float*)Vc + plane};
    const DfBlock vp{Vp ? (const float*)Vp : vc.h, Vp ? (const float*)Vp + plane : vc.l};
    DfOut o{(float*)Vn, (float*)Vn + plane, (float*)Un, (float*)Un + plane, cmv, cmu, (uint32_t)nbucket, -0.f};
    if (P.ld > 4 * DF_MAXCH || (P.ld & 3)) return cudaErrorInvalidValue;  // a thread per 4 columns
    const uint32_t nch = (uint32_t)P.ld / 4;
    const dim3 nt(nch, DF_THREADS / nch);
    auto ctas = [&](uint32_t per) { return (unsigned)((P.n + per * nt.y - 1) / (per * nt.y)); };
    if (P.is_stencil) {
        const unsigned grid = ctas(DF_ROWS);
        stencil_step_df_kernel<<<grid, nt, 0, s>>>(
            vc, vp, P.d_diag32, P.d_diag32lo, P.geom, split_f2(P.off64[0]), split_f2(P.off64[1]),
            split_f2(P.off64[2]), c, d, (uint32_t)P.ld, (uint32_t)P.n_tot, (uint32_t)P.n, o);
    } else {
        // A CSR row is a serial chain of gathers, so a thread takes as many rows, up to
        // DF_ROWS, as leave two CTAs an SM.  Narrow blocks of eight rows a thread put few
        // CTAs on the chip: 30 steps of 30000 rows of 8 columns (30 CTAs) 5.2 ms, 1.7 with a
        // row a thread; 40 columns 4.1 and 2.1 with two rows; 300000 rows of one column 17.6
        // and 8.7.  Where eight rows leave enough, fewer cost the Gram products beside them
        // more than they gain (30011 rows of 160 columns, degree 200: 19.6 ms a call, 20.6 with
        // two rows; 300000 of 100: 32.6, 35.1 with one).
        uint32_t per = DF_ROWS;
        while (per > 1 && ctas(per) < 2u * (unsigned)device_sms()) per /= 2;
        csr_step_df_kernel<<<ctas(per), nt, 0, s>>>(vc, vp, P.d_rowptr, P.d_colind, P.d_val32, P.d_val32lo,
                                                    split_f2(P.beta), c, d, (uint32_t)P.ld, (uint32_t)P.n_tot,
                                                    (uint32_t)P.n, per, o);
    }
    return cudaGetLastError();
}

// Float pairs of a float64 array (the folded operator coefficients).
__global__ void split_df_kernel(const double* __restrict__ v, int64_t n, float* __restrict__ h, float* __restrict__ l) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const float vh = (float)v[e];
        h[e] = vh;
        l[e] = (float)(v[e] - (double)vh);
    }
}

cudaError_t launch_split_df(const double* v, int64_t n, float* h, float* l, cudaStream_t s) {
    int64_t blocks = (n + 255) / 256;
    if (blocks > (int64_t)device_sms() * 16) blocks = (int64_t)device_sms() * 16;
    split_df_kernel<<<(int)(blocks < 1 ? 1 : blocks), 256, 0, s>>>(v, n, h, l);
    return cudaGetLastError();
}

}  // namespace ssm
