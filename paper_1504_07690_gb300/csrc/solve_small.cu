// solve_small.cu - points of n_v <= 32 without hybrid columns, one warp each: the three exact tests and the
// sum of the route that keeps everything with every eigenvalue inside the filter (as in
// solve_kernel), which settle most points.  Lane i holds row i of a matrix in registers;
// a Cholesky is n right-looking steps of shuffles and fmas without a barrier, where the
// CTA-per-point kernel spends a step's time in barriers and one-warp sections.  The points
// that need more go into the list `pend` (pend[0]: their number) for solve_kernel; their
// order does not matter to the results.  17600 points of n_v = 32 (1100 graphs, 16 points
// each; 4300 are left): solve 19.0 -> 11.2 ms.
#include <float.h>

#include "solve_launch.h"

namespace ssm {

namespace {

constexpr int SM_N = SOLVE_SMALL_N, SM_WARPS = 4, SM_PITCH = SM_N + 1;
constexpr size_t SM_BYTES = (size_t)SM_WARPS * 2 * SM_N * SM_PITCH * sizeof(double);

// Cholesky of the n x n matrix whose row `lane` is a[0..lane]: a becomes the row of L.
// False (on every lane) at the first pivot that is not positive.
__device__ __forceinline__ bool warp_cholesky(double (&a)[SM_N], int n, int lane) {
    bool ok = true;
#pragma unroll
    for (int k = 0; k < SM_N; ++k) {
        if (k < n && ok) {
            const double piv = __shfl_sync(0xffffffffu, a[k], k);
            ok = piv > 0.0;
            const double r0 = rsqrt(piv);
            const double rr = r0 * fma(-0.5 * piv * r0, r0, 1.5);  // one Newton step
            const double lik = (lane == k ? piv : a[k]) * rr;
            a[k] = lik;
#pragma unroll
            for (int j = k + 1; j < SM_N; ++j)
                if (j < n) {
                    const double ljk = __shfl_sync(0xffffffffu, lik, j);
                    if (lane >= j) a[j] = fma(-lik, ljk, a[j]);
                }
        }
    }
    return ok;
}

__global__ void __launch_bounds__(32 * SM_WARPS)
solve_small_kernel(const double* __restrict__ Kfull, const double* __restrict__ KZ, int64_t n_t, int n, double tau,
                   double xlo, double xhi, const double* __restrict__ mu, int ldmu, int K, double floor_scale,
                   double* __restrict__ dos, int32_t* __restrict__ rank, const double* __restrict__ floor_pt,
                   int32_t* __restrict__ pend) {
    extern __shared__ __align__(16) double dyn[];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    double* tw = dyn + (size_t)wp * 2 * SM_N * SM_PITCH;  // K_W, then L (column SM_N: 1 / its diagonal)
    double* tz = tw + SM_N * SM_PITCH;                    // K_Z, then L1
    const int64_t it = (int64_t)blockIdx.x * SM_WARPS + wp;
    if (it >= n_t) return;
    const double* Kt = Kfull + (size_t)it * n * n;
    const double* Zk = KZ + (size_t)it * n * n;
    for (int e = lane; e < n * n; e += 32) {
        const int i = e / n, j = e - i * n;
        tw[i * SM_PITCH + j] = Kt[e];
        tz[i * SM_PITCH + j] = Zk[e];
    }
    double fs = 0.0;
    if (floor_scale > 0.0 || floor_pt)
        for (int l = lane; l <= K; l += 32) fs = fma((double)(l + 1), fabs(mu[it * ldmu + l]), fs);
    for (int o = 16; o > 0; o >>= 1) fs += __shfl_xor_sync(0xffffffffu, fs, o);
    const double floor_t = (floor_pt ? floor_pt[3 * it] : floor_scale) * fs;
    const double xl = floor_pt ? floor_pt[3 * it + 1] : xlo, xh = floor_pt ? floor_pt[3 * it + 2] : xhi;
    __syncwarp();
    // row `lane` of the symmetrised matrices; g = the largest absolute column sum of K_W
    const bool row = lane < n;
    auto kw = [&](int j) { return 0.5 * (tw[lane * SM_PITCH + j] + tw[j * SM_PITCH + lane]); };
    auto kz = [&](int j) { return 0.5 * (tz[lane * SM_PITCH + j] + tz[j * SM_PITCH + lane]); };
    double g = 0.0, dmax = -DBL_MAX;
    if (row) {
        for (int j = 0; j < n; ++j) g += fabs(kw(j));
        dmax = tw[lane * SM_PITCH + lane];
    }
    for (int o = 16; o > 0; o >>= 1) {
        g = fmax(g, __shfl_xor_sync(0xffffffffu, g, o));
        dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    }
    double phi = 0.0;
    int r = 0;
    bool done = g < floor_t || g <= 0.0;  // nothing kept
    bool hard = false;
    const double thr = fmax(tau * g, floor_t);
    // the Choleskys in order: 0 K_W - thr I (everything kept?), 1 K_Z - xl K_W, 2 xh K_W - K_Z
    // (every eigenvalue inside?), 3 K_W; 4 floor I - K_W after a failed 0 (nothing kept?)
    for (int ph = 0; !done && !hard;) {
        double a[SM_N];
#pragma unroll
        for (int j = 0; j < SM_N; ++j) {
            a[j] = 0.0;
            if (row && j < n && j <= lane) {
                const double w = kw(j);
                a[j] = ph == 0   ? (j == lane ? w - thr : w)
                       : ph == 1 ? fma(-xl, w, kz(j))
                       : ph == 2 ? fma(xh, w, -kz(j))
                       : ph == 3 ? w
                                 : (j == lane ? floor_t - w : -w);
            }
        }
        const bool pos = warp_cholesky(a, n, lane);
        if (ph == 0) {
            if (pos) ph = 2;
            else if (dmax < floor_t) ph = 4;
            else hard = true;
        } else if (ph == 2) {
            ph = 1;
            hard = !pos;
        } else if (ph == 1) {
            hard = !pos;
            if (pos) {  // L1 takes K_Z's tile, upper half zero (K_Z is not read again)
                __syncwarp();
#pragma unroll
                for (int j = 0; j < SM_N; ++j)
                    if (row && j < n) tz[lane * SM_PITCH + j] = j <= lane ? a[j] : 0.0;
                ph = 3;
            }
        } else if (ph == 4) {
            done = pos;
            hard = !pos;
        } else {
            hard = !pos;
            if (pos) {  // sum = ||L^-1 L1||_F^2 + xl n, column `lane` of L^-1 L1 a forward substitution
                __syncwarp();
#pragma unroll
                for (int j = 0; j < SM_N; ++j)
                    if (row && j < n && j <= lane) {
                        tw[lane * SM_PITCH + j] = a[j];
                        if (j == lane) tw[lane * SM_PITCH + SM_N] = 1.0 / a[j];
                    }
                __syncwarp();
                double x[SM_N], f = 0.0;
#pragma unroll
                for (int i = 0; i < SM_N; ++i) {
                    x[i] = 0.0;
                    if (i < n) {
                        double s = row ? tz[i * SM_PITCH + lane] : 0.0;
#pragma unroll
                        for (int k = 0; k < i; ++k) s = fma(-tw[i * SM_PITCH + k], x[k], s);
                        x[i] = s * tw[i * SM_PITCH + SM_N];
                        f = fma(x[i], x[i], f);
                    }
                }
                for (int o = 16; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
                phi = fma(xl, (double)n, f);
                r = n;
                done = true;
            }
        }
    }
    if (lane == 0) {
        if (done) {
            dos[it] = phi;
            if (rank) rank[2 * it] = rank[2 * it + 1] = r;
        } else {
            pend[1 + atomicAdd(pend, 1)] = (int32_t)it;
        }
    }
}

}  // namespace

cudaError_t launch_solve_small(const double* Kfull, const double* KZ, int64_t n_t, int n_v, double tau, double xlo,
                               double xhi, const double* mu, int ldmu, int K, double floor_scale, double* dos,
                               int32_t* rank, const double* floor_pt, int32_t* pend, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(pend, 0, sizeof(int32_t), s);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(solve_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SM_BYTES);
    if (e != cudaSuccess) return e;
    solve_small_kernel<<<(unsigned)((n_t + SM_WARPS - 1) / SM_WARPS), 32 * SM_WARPS, SM_BYTES, s>>>(
        Kfull, KZ, n_t, n_v, tau, xlo, xhi, mu, ldmu, K, floor_scale, dos, rank, floor_pt, pend);
    return cudaGetLastError();
}

}  // namespace ssm
