// solve.cu - launches of the per-sweep-point solve (solve_body.cuh): the kernel of points
// without hybrid columns, workspaces and the schedule.
#include "solve_body.cuh"
#include "solve_launch.h"

namespace ssm {

namespace {

// Threads per CTA: one per row of the per-point matrices up to 256 (smaller
// problems, e.g. n_v = 64 in batched plans, get small CTAs and more of them
// per SM).
int solve_threads(int n_v) { return n_v <= 128 ? 128 : NT; }

// ... but a call of few points lasts as long as its slowest ones, and a float64 fma holds
// its warp for 65 cycles of which the pipe is busy 16: eight warps a point, for points with
// hybrid columns up to four an SM (400 points of n_v = 128, n_vh = 128: 12.4 ms against 18.3;
// 600 of n_v = 100: 7.5 against 8.6, 900: no gain), without up to two (20 points of n_v = 100:
// 5.1 against 6.4; where every point keeps a part of its directions 300 take 7.4 against 7.8,
// 450 9.3 against 9.1).  The step-by-step route of float64 plans keeps its sums' order.
int solve_threads(int n_v, int n_vh, bool hyb, int64_t n_call) {
    const int per_sm = hyb ? (n_v > 32 ? 4 : 0) : (n_vh == 0 && n_v > 64 ? 2 : 0);
    return n_call <= (int64_t)per_sm * device_sms() ? NT : solve_threads(n_v);
}

// CTAs with a private workspace: 4 x (256 / threads) per SM to overlap the
// serial QL chains, fewer when their workspaces would exceed 2 GiB in total.
int workspace_ctas(int n_v, bool hyb) {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const size_t per = workspace_doubles(n_v, hyb) * sizeof(double);
    size_t cap = ((size_t)2 << 30) / per;
    size_t g = (size_t)4 * sms * (NT / solve_threads(n_v));
    if (g > cap) g = cap;
    return g < 1 ? 1 : (int)g;
}

size_t solve_smem(int n) {
    return (size_t)(7 * n + NT / 32 + (2 * n + 16 + 1) / 2 + 3 * 32 * 33) * sizeof(double);
}

}  // namespace

size_t solve_workspace_bytes(int n_v, bool hyb) {
    return (size_t)workspace_ctas(n_v, hyb) * workspace_doubles(n_v, hyb) * sizeof(double);
}

// Schedule of the next solve launch from the routes of the previous one (its kept
// ranks): CTA b runs on SM b mod S of the first wave (b < S k, k CTAs per SM), so the
// points that kept part of the directions (the longest, bound by float64 issue) take
// blocks 0.. and their SMs' other slots go to points that kept nothing (the shortest)
// or stay empty, as far as free slots allow; every other point fills the rest in order.
// One CTA (the placement by one thread, in shared memory); perm has S k entries.
__global__ void solve_schedule_kernel(const int32_t* __restrict__ rank_prev, int64_t n_t, int n, int S, int k,
                                      int32_t* __restrict__ perm_out) {
    extern __shared__ int32_t sched[];  // perm (S k), then the route class of each point
    const int64_t slots = (int64_t)S * k;
    int32_t* perm = sched;
    int32_t* cl = sched + slots;  // 0 nothing kept, 1 part, 2 everything
    for (int64_t i = threadIdx.x; i < n_t; i += blockDim.x) {
        const int r = rank_prev[2 * i];
        cl[i] = r <= 0 ? 0 : (r >= n ? 2 : 1);
    }
    for (int64_t b = threadIdx.x; b < slots; b += blockDim.x) perm[b] = -2;  // unassigned
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t free_slots = slots - n_t;
        int np = 0;
        int64_t ce = 0;  // cursor over the points that kept nothing
        for (int64_t i = 0; i < n_t && np < S; ++i)
            if (cl[i] == 1) perm[np++] = (int32_t)i;
        for (int s = 0; s < np; ++s)
            for (int j = 1; j < k; ++j) {
                while (ce < n_t && cl[ce] != 0) ++ce;
                if (ce < n_t) {
                    perm[s + (int64_t)j * S] = (int32_t)ce++;
                } else if (free_slots > 0) {
                    perm[s + (int64_t)j * S] = -1;
                    --free_slots;
                }
            }
        // the rest in order: points not placed yet into the unassigned slots
        int64_t b = 0;
        int placed_part = 0;
        for (int64_t i = 0; i < n_t; ++i) {
            const int c = cl[i];
            if (c == 1 && placed_part < np) {
                ++placed_part;
                continue;
            }
            if (c == 0 && i < ce) continue;  // placed next to a part point (cursor passed it)
            while (b < slots && perm[b] != -2) ++b;
            if (b >= slots) break;  // cannot happen: holes never exceed the free slots
            perm[b++] = (int32_t)i;
        }
    }
    __syncthreads();
    for (int64_t b = threadIdx.x; b < slots; b += blockDim.x) perm_out[b] = perm[b] == -2 ? -1 : perm[b];
}

cudaError_t launch_solve(const double* Kfull, const double* KZ, int64_t n_t, int64_t n_call, int n_v, int n_vh,
                         double tau, double xlo, double xhi, const double* mu, int ldmu, int K, double floor_scale,
                         void* work, double* dos, int32_t* rank, int* flag, cudaStream_t s, const double* floor_pt,
                         const int32_t* perm, bool pinv, bool hyb, int32_t* pend) {
    if (n_t <= 0) return cudaSuccess;
    if (n_v > MAXN) return cudaErrorInvalidValue;
    const size_t smem = solve_smem(n_v);
    const SolveKernel kernel = hyb ? solve_kernel_hyb() : solve_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int64_t grid = workspace_ctas(n_v, hyb), n_slot = n_t;
    if (perm) {
        n_slot = solve_slots(n_v, hyb, n_call);
        if (n_slot < n_t || n_slot > grid) return cudaErrorInvalidValue;
    }
    if (grid > n_slot) grid = n_slot;
    // small points without hybrid columns: a warp each; what is left goes on
    const int32_t* n_dev = nullptr;
    if (pend && solve_uses_small(n_call, n_v, n_vh, pinv)) {
        e = launch_solve_small(Kfull, KZ, n_t, n_v, tau, xlo, xhi, mu, ldmu, K, floor_scale, dos, rank, floor_pt, pend,
                               s);
        if (e != cudaSuccess) return e;
        n_dev = pend;
        perm = pend + 1;
    }
    kernel<<<(int)grid, solve_threads(n_v, n_vh, hyb, n_call), smem, s>>>(Kfull, KZ, n_t, n_v, n_vh, tau, xlo, xhi, mu,
                                                                          ldmu, K, floor_scale, (double*)work, dos,
                                                                          rank, flag, floor_pt, perm, n_slot, pinv,
                                                                          n_dev);
    return cudaGetLastError();
}

// A warp a point when the points fill the device with warps; fewer take one wave of CTAs
// either way, and a warp's serial chain is the longer one (n_v = 32: 1.06 against 1.31 ms
// at 73 points, 1.19 against 1.34 at 600, 1.79 against 1.44 at 1200; n_v = 16: 0.42
// against 0.55, 0.60 against 0.59, 0.72 against 0.65).
bool solve_uses_small(int64_t n_call, int n_v, int n_vh, bool pinv) {
    return n_v <= SOLVE_SMALL_N && n_vh == 0 && !pinv && n_call >= (int64_t)8 * device_sms();
}

int64_t solve_slots(int n_v, bool hyb, int64_t n_t) {
    int dev = 0, sms = 0, k = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const size_t smem = solve_smem(n_v);
    const SolveKernel kernel = hyb ? solve_kernel_hyb() : solve_kernel<false>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, kernel, solve_threads(n_v, hyb ? 1 : 0, hyb, n_t), smem) != cudaSuccess)
        return 0;
    const int64_t slots = (int64_t)sms * k;
    return slots <= workspace_ctas(n_v, hyb) ? slots : 0;
}

cudaError_t launch_solve_schedule(const int32_t* rank_prev, int64_t n_t, int n_v, bool hyb, int32_t* perm,
                                  cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t slots = solve_slots(n_v, hyb, n_t);
    if (slots < n_t || slots <= 0) return cudaErrorInvalidValue;
    const size_t smem = (size_t)(slots + n_t) * sizeof(int32_t);
    if (smem > 48 * 1024) return cudaErrorInvalidValue;
    solve_schedule_kernel<<<1, 256, smem, s>>>(rank_prev, n_t, n_v, sms, (int)(slots / sms), perm);
    return cudaGetLastError();
}

}  // namespace ssm
