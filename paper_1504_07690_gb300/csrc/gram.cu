// gram.cu - split-K Gram products of the doubling identities (CUDA-core path).
//
// For a step that produced V_{k+1} from V_k the moments X_{2k+2} and X_{2k+1}
// follow from G^e = V_{k+1}^T V_{k+1} and G^o = V_{k+1}^T V_k through
// T_{2j} = 2 T_j^2 - T_0 and T_{2j+1} = 2 T_{j+1} T_j - T_1 (the product rule
// T_p T_q = (T_{p+q} + T_{|p-q|})/2 used in Proposition 1's proof); the paper's
// own loop forms X_l = W^T V_l at every l (Alg. 7), which needs twice the
// recurrence steps.
//
// The row range is split into n_split slices; every CTA computes one square output tile
// over one slice and writes its partial sum in float64.  Only elements on or above the
// diagonal of the symmetric G^e are needed (16 x 16 pieces wholly below it are skipped).
// The partial sums are reduced in a fixed order by moments.cu, so results are bitwise
// reproducible.
#include "internal.h"

namespace ssm {

namespace {

constexpr int KT = 32;  // rows per staged slab

// Tile shapes.  A warp owns one 8 P x 4 Q piece of the tile, 8 x 4 lanes of P x Q outputs,
// and sums each output over the slice's rows in row order (one fma chain per output), so
// the shape changes no bit of the result.  Float64 runs at 2 fma a clock and SM here: the
// kernel is bound by the fma pipe (97 % busy), and what counts is that no warp multiplies
// padding and that the chains are spread over the SMs.
//   Broad: 64 x 64 tiles of eight 32 x 16 warp pieces, float32 only: there shared memory is
//     the bound, and 16 outputs from 8 loads a lane take less of it than 8 from 6.
//   Wide: 32 x 32 tiles of four 16 x 16 warp pieces.  Pieces past n_tot or below the
//     diagonal idle.  The Gram pair of two 65536 x 200 float64 blocks: 8.05 ms, 13.7 ms
//     with 64 x 64 tiles computed whole (1.77 times the useful products; 6.3 ms is the
//     pipe's floor for these alone).
//   Mid: one warp a 16 x 16 tile, for problems with few tiles and slices.
//   Small: 8 x 8 tiles of two warps, one output a lane, for the smallest: an fma holds its
//     warp for 65 to 73 cycles whatever the others do, so a lane's second output would double
//     the chain of a slice (1024 rows x 40 columns in two slices of 512 rows: 545 us in
//     64 x 64 tiles, on four SMs; 43 us with two outputs a lane, 28 us with one, launch
//     included).
// ST: staged slabs (more than two did not help the small tiles).  Staged with 16-byte
// copies where rows are whole 16-byte units: 7.2 ms a call of the 32 x 32 grid, 40 probes,
// degree 200, against 7.7 with 8-byte ones (both with two outputs a lane).
struct BroadTile { static constexpr int P = 4, Q = 4, WR = 2, WC = 4, ST = 2; };
struct WideTile { static constexpr int P = 2, Q = 4, WR = 2, WC = 2, ST = 2; };
struct MidTile { static constexpr int P = 2, Q = 4, WR = 1, WC = 1, ST = 2; };
struct SmallTile { static constexpr int P = 1, Q = 1, WR = 1, WC = 2, ST = 2; };

template <typename S>
constexpr int tile_dim() {
    static_assert(8 * S::P * S::WR == 4 * S::Q * S::WC, "square tiles");
    return 8 * S::P * S::WR;
}

// 16 aligned bytes, of which the first `bytes` are read and the others zero.
__device__ __forceinline__ void async_vec(void* dst, const void* src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(bytes)
                 : "memory");
}

template <typename T>
__device__ __forceinline__ void async_elem(T* dst, const T* src, bool ok) {
    // ok = false: nothing is read and the element is zero
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "n"((int)sizeof(T)), "r"(ok ? (int)sizeof(T) : 0)
                 : "memory");
}

// Tile u of the nt1 x nt1 tiles of G^o (which = 1), then the upper ones of G^e.
__device__ __forceinline__ void tile_of_index(int u, int nt1, int n_sym, int& which, int& ti, int& tj) {
    const int n_all = nt1 * nt1;
    const bool odd = (int)gridDim.x > n_sym;
    if (odd && u < n_all) {
        which = 1;
        ti = u / nt1;
        tj = u - ti * nt1;
        return;
    }
    which = 0;
    int r = odd ? u - n_all : u;
    ti = 0;
    while (r >= nt1 - ti) {
        r -= nt1 - ti;
        ++ti;
    }
    tj = ti + r;
}

template <typename T, typename Acc, typename S>
__global__ void __launch_bounds__(32 * S::WR * S::WC)
gram_kernel(const T* __restrict__ A, const T* __restrict__ B, int ld, int n_tot, int64_t n_rows,
            int64_t rows_per_split, double* __restrict__ part, int nt1, int n_sym, bool vec) {
    constexpr int NT = 32 * S::WR * S::WC, TD = tile_dim<S>(), P = S::P, Q = S::Q, PR = 8 * P, PC = 4 * Q;
    __shared__ __align__(16) T Ls[S::ST][KT][TD];
    __shared__ __align__(16) T Rs[S::ST][KT][TD];
    int which, ti, tj;
    tile_of_index((int)blockIdx.x, nt1, n_sym, which, ti, tj);
    const T* L = A;
    const T* R = which == 0 ? A : B;
    const int64_t r0 = (int64_t)blockIdx.y * rows_per_split;
    int64_t r1 = r0 + rows_per_split;
    if (r1 > n_rows) r1 = n_rows;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cl0 = ti * TD, cr0 = tj * TD;
    const int pr = (warp / S::WC) * PR, pc = (warp % S::WC) * PC;  // the warp's piece of the tile
    const bool on = cl0 + pr < n_tot && cr0 + pc < n_tot && (which == 1 || cr0 + pc + PC > cl0 + pr);
    const int ri = pr + (lane >> 2) * P, ci = pc + (lane & 3) * Q;
    Acc acc[P][Q];
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
        for (int q = 0; q < Q; ++q) acc[p][q] = Acc(0);
    // 16-byte copies (vec: rows of aligned 16-byte units): a thread keeps one unit column of
    // both tiles and steps over the rows
    constexpr int VE = 16 / (int)sizeof(T), VC = TD / VE, VR = NT / VC;
    const int vr = (int)threadIdx.x / VC, vc = ((int)threadIdx.x % VC) * VE;
    const int vl = max(0, min(VE, n_tot - cl0 - vc)) * (int)sizeof(T);  // bytes of the unit in the row
    const int vq = max(0, min(VE, n_tot - cr0 - vc)) * (int)sizeof(T);
    const T* Lv = L + (vl ? cl0 + vc : 0);
    const T* Rv = R + (vq ? cr0 + vc : 0);
    auto stage = [&](int buf, int64_t r) {  // rows r .. r + KT - 1 (an empty group past the slice)
        if (vec) {
            if (r < r1) {
                const size_t o = (size_t)(r + vr) * ld;
#pragma unroll
                for (int q = 0; q < KT / VR; ++q) {
                    const bool in = r + vr + q * VR < r1;
                    const size_t at = in ? o + (size_t)q * VR * ld : 0;
                    async_vec(&Ls[buf][vr + q * VR][vc], Lv + at, in ? vl : 0);
                    async_vec(&Rs[buf][vr + q * VR][vc], Rv + at, in ? vq : 0);
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            return;
        }
        for (int e = threadIdx.x; e < KT * TD && r < r1; e += NT) {
            const int rr = e / TD, cc = e - rr * TD;
            const int64_t row = r + rr;
            const bool okr = row < r1;
            const int cl = cl0 + cc, cr = cr0 + cc;
            const bool okl = okr && cl < n_tot, okc = okr && cr < n_tot;
            async_elem(&Ls[buf][rr][cc], okl ? L + row * ld + cl : L, okl);
            async_elem(&Rs[buf][rr][cc], okc ? R + row * ld + cr : R, okc);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int q = 0; q + 1 < S::ST; ++q) stage(q, r0 + q * KT);
    int buf = 0;
    for (int64_t r = r0; r < r1; r += KT) {
        stage(buf == 0 ? S::ST - 1 : buf - 1, r + (S::ST - 1) * KT);
        asm volatile("cp.async.wait_group %0;" ::"n"(S::ST - 1) : "memory");
        __syncthreads();
        if (on) {
#pragma unroll 8
            for (int rr = 0; rr < KT; ++rr) {
                T a[P], b[Q];
#pragma unroll
                for (int p = 0; p < P; ++p) a[p] = Ls[buf][rr][ri + p];
#pragma unroll
                for (int q = 0; q < Q; ++q) b[q] = Rs[buf][rr][ci + q];
#pragma unroll
                for (int p = 0; p < P; ++p)
#pragma unroll
                    for (int q = 0; q < Q; ++q) acc[p][q] = fma(Acc(a[p]), Acc(b[q]), acc[p][q]);
            }
        }
        __syncthreads();
        if (++buf == S::ST) buf = 0;
    }
    if (!on) return;
    double* out = part + ((size_t)blockIdx.y * 2 + which) * (size_t)n_tot * n_tot;
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const int i = cl0 + ri + p;
        if (i >= n_tot) continue;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int j = cr0 + ci + q;
            if (j < n_tot) out[(size_t)i * n_tot + j] = (double)acc[p][q];
        }
    }
}

template <typename T, typename Acc, typename S>
cudaError_t gram_launch(const T* A, const T* B, int ld, int n_tot, int64_t n_rows, int n_split, int64_t rps,
                        double* part, cudaStream_t s) {
    const int nt1 = (n_tot + tile_dim<S>() - 1) / tile_dim<S>();
    const int n_sym = nt1 * (nt1 + 1) / 2;
    dim3 grid((unsigned)(n_sym + (B ? nt1 * nt1 : 0)), (unsigned)n_split);
    const bool vec = ld % (16 / (int)sizeof(T)) == 0 && ((uintptr_t)A & 15) == 0 && ((uintptr_t)B & 15) == 0;
    gram_kernel<T, Acc, S><<<grid, 32 * S::WR * S::WC, 0, s>>>(A, B, ld, n_tot, n_rows, rps, part, nt1, n_sym, vec);
    return cudaGetLastError();
}

template <typename S>
int64_t gram_ctas(int n_tot, bool odd, int n_split) {
    const int64_t t = (n_tot + tile_dim<S>() - 1) / tile_dim<S>();
    return (t * (t + 1) / 2 + (odd ? t * t : 0)) * n_split;
}

// The widest float64 tile that still gives every SM a CTA (a chain of 512 rows or more per output
// runs either way; with fewer CTAs than SMs the pipes of the others would idle).
template <typename T, typename Acc>
cudaError_t gram(const T* A, const T* B, int ld, int n_tot, int64_t n_rows, int n_split, double* part,
                 cudaStream_t s) {
    int64_t rps = (n_rows + n_split - 1) / n_split;
    rps = (rps + KT - 1) / KT * KT;
    const int sms = device_sms();
    if constexpr (sizeof(T) == 4) {
        // 64-wide tiles with three CTAs or more an SM and at most 1/7 wider padding (16384 rows
        // of 700 columns, 20 steps: Gram 12.3 ms, 18.1 in 32-wide tiles; 4096 of 512 1.93 and
        // 2.52; 65536 of 200 6.63 and 7.17; but 4096 of 257, 320 CTAs, 1.14 and 0.98, 16384 of
        // 160, padded to 192, 1.28 and 1.17)
        const int broad = (n_tot + 63) / 64 * 64, wide = (n_tot + 31) / 32 * 32;
        if (gram_ctas<BroadTile>(n_tot, B != nullptr, n_split) >= 3 * sms && 7 * broad <= 8 * wide)
            return gram_launch<T, Acc, BroadTile>(A, B, ld, n_tot, n_rows, n_split, rps, part, s);
    }
    if (gram_ctas<WideTile>(n_tot, B != nullptr, n_split) >= sms)
        return gram_launch<T, Acc, WideTile>(A, B, ld, n_tot, n_rows, n_split, rps, part, s);
    if (gram_ctas<MidTile>(n_tot, B != nullptr, n_split) >= sms)
        return gram_launch<T, Acc, MidTile>(A, B, ld, n_tot, n_rows, n_split, rps, part, s);
    return gram_launch<T, Acc, SmallTile>(A, B, ld, n_tot, n_rows, n_split, rps, part, s);
}

__global__ void reduce_gram_pair_kernel(const double* __restrict__ part, int n_split, int n, double* __restrict__ gaa,
                                        double* __restrict__ gab) {
    const size_t nn = (size_t)n * n;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < nn; e += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / n), j = (int)(e - (size_t)i * n);
        const int lo = i < j ? i : j, hi = i < j ? j : i;
        double a = 0.0, b = 0.0;
        for (int s = 0; s < n_split; ++s) {
            const double* ps = part + (size_t)s * 2 * nn;
            a += ps[(size_t)lo * n + hi];
            if (gab) b += ps[nn + e];
        }
        gaa[e] = a;
        if (gab) gab[e] = b;
    }
}

}  // namespace

cudaError_t launch_reduce_gram_pair(const double* part, int n_split, int n, double* gaa, double* gab, cudaStream_t s) {
    int64_t b = ((int64_t)n * n + 255) / 256;
    if (b > (int64_t)device_sms() * 16) b = (int64_t)device_sms() * 16;
    if (b < 1) b = 1;
    reduce_gram_pair_kernel<<<(int)b, 256, 0, s>>>(part, n_split, n, gaa, gab);
    return cudaGetLastError();
}

int gram_split_count(int64_t n_rows, int n_tot) {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // slices for about four 64 x 64 tiles an SM (the summation order follows from it)
    const int nt1 = (n_tot + 63) / 64;
    const int tiles = nt1 * (nt1 + 1) / 2 + nt1 * nt1;
    int64_t want = (4LL * sms + tiles - 1) / tiles;
    int64_t cap = (n_rows + 511) / 512;
    if (want > cap) want = cap;
    if (want < 1) want = 1;
    if (want > 4096) want = 4096;
    return (int)want;
}

cudaError_t launch_gram_f64(const double* A, const double* B, int ld, int n_tot, int64_t n_rows,
                            int n_split, double* part, cudaStream_t s) {
    return gram<double, double>(A, B, ld, n_tot, n_rows, n_split, part, s);
}

cudaError_t launch_gram_f32(const float* A, const float* B, int ld, int n_tot, int64_t n_rows,
                            int n_split, double* part, cudaStream_t s) {
    return gram<float, float>(A, B, ld, n_tot, n_rows, n_split, part, s);
}

}  // namespace ssm
