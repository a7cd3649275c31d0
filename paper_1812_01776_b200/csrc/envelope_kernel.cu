// Traffic envelope of the bound trace (Section 5): for each window length, the
// largest number of arrivals inside any window of that length.  A maximising
// window can be moved right until it starts at an arrival, so the answer is the
// maximum over j of end(j) - j, end(j) being the first arrival at or after
// a_j + window.
//
// What bounds it: the binary searches for end(j) in the L2-resident trace (their
// latency, and a sector of L2 per step), so most of them are not made.  end()
// never decreases, so for neighbouring starts j .. k - 1 the counts are at most
// end(k) - j.  A CTA searches every 256th start of its stretch, all windows side
// by side; these counts also are lower bounds of the answer, which the CTAs share
// as they go.  Only where 256 starts could still beat the best count known so
// far, a warp looks closer: start m can only be better than B if arrival m + B still
// lies in its window, one coalesced load and a compare, and only a start that passes
// is searched.  10^6 arrivals, 12 windows: the whole call 361 -> 46 us (before:
// 12 x 10^6 searches in two launches).
#include "il_internal.h"

namespace il {

namespace {
constexpr int kEnvThreads = 256;
constexpr int kEnvGroups = 4;                    // groups of 256 starts per CTA
constexpr int kEnvGroup = 256;
constexpr int kMaxWindows = 64;
}

struct EnvParams {
    const int64_t *arrival;
    int32_t n;
    int32_t n_windows;
    int64_t window[kMaxWindows];
    int *out;                  // [n_windows], zero on entry
    int *status;               // checked build: where an index out of range is recorded
};

// Arrival i (checked build: recorded and 0 where there is none)
__device__ __forceinline__ int64_t arrival_at(const EnvParams &p, int64_t i)
{
    return IL_IN_RANGE(i, p.n, p.status) ? __ldg(p.arrival + i) : 0;
}

// First index in [lo, hi] whose arrival is `window` or more after a (hi if there is none before it).
__device__ __forceinline__ int first_at(const EnvParams &p, int lo, int hi, int64_t a, int64_t window)
{
    while (lo < hi) {
        const int mid = lo + (hi - lo) / 2;
        if (arrival_at(p, mid) - a < window) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// The best count of a window in shared memory as it is now: the warps of the CTA raise it with atomicMax while others look.
__device__ __forceinline__ int best_now(const int *best)
{
    int v;
    asm volatile("ld.relaxed.cta.shared.s32 %0, [%1];" : "=r"(v) : "r"((unsigned)__cvta_generic_to_shared(best)) : "memory");
    return v;
}

__global__ void __launch_bounds__(kEnvThreads) envelope_kernel(const __grid_constant__ EnvParams p)
{
    __shared__ int end[kMaxWindows][kEnvGroups + 1];
    __shared__ int best[kMaxWindows];
    const int j0 = blockIdx.x * (kEnvGroups * kEnvGroup);
    const int W = p.n_windows;
    for (int w = threadIdx.x; w < W; w += kEnvThreads) best[w] = 0;
    __syncthreads();
    for (int k = threadIdx.x; k < W * (kEnvGroups + 1); k += kEnvThreads) {
        const int w = k / (kEnvGroups + 1), g = k - w * (kEnvGroups + 1);
        const int64_t j = (int64_t)j0 + g * kEnvGroup;
        int e = p.n;
        if (j < p.n) {
            e = first_at(p, (int)j, p.n, arrival_at(p, j), p.window[w]);
            atomicMax(&best[w], e - (int)j);
        }
        end[w][g] = e;
    }
    __syncthreads();
    for (int w = threadIdx.x; w < W; w += kEnvThreads) best[w] = max(best[w], atomicMax(&p.out[w], best[w]));
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int k = threadIdx.x >> 5; k < W * kEnvGroups; k += kEnvThreads / 32) {
        const int w = k / kEnvGroups, g = k - w * kEnvGroups;
        const int64_t j = (int64_t)j0 + g * kEnvGroup;
        // read once and shared by the warp: its lanes have to take the same way to the reduction below
        const int known = __shfl_sync(0xffffffffu, best_now(&best[w]), 0);
        if (j >= p.n || end[w][g + 1] - (int)j <= known) continue;       // none of these 256 can be better
        int count = 0;
#pragma unroll
        for (int i = 0; i < kEnvGroup; i += 32) {
            const int64_t m = j + i + lane;
            if (m + known >= p.n) continue;
            const int64_t a = arrival_at(p, m);
            if (arrival_at(p, m + known) - a < p.window[w])
                count = max(count, first_at(p, (int)m + known + 1, end[w][g + 1], a, p.window[w]) - (int)m);
        }
        count = __reduce_max_sync(0xffffffffu, count);
        if (lane == 0 && count > known) atomicMax(&best[w], max(count, atomicMax(&p.out[w], count)));
    }
}

cudaError_t launch_envelope(const int64_t *d_arrival, int n, const int64_t *h_windows, int n_windows,
                            int *d_out, int *d_status, cudaStream_t stream)
{
    EnvParams p;
    p.arrival = d_arrival; p.n = n; p.n_windows = n_windows; p.out = d_out; p.status = d_status;
    for (int w = 0; w < n_windows; w++) p.window[w] = h_windows[w];
    const int64_t per_cta = kEnvGroups * kEnvGroup;
    envelope_kernel<<<(int)((n + per_cta - 1) / per_cta), kEnvThreads, 0, stream>>>(p);
    return cudaGetLastError();
}

int envelope_max_windows() { return kMaxWindows; }

}  // namespace il
