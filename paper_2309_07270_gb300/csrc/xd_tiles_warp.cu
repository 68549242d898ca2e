// The warp-per-extension kernel: small batches, and the extensions that
// outgrew a first tier.
#include <algorithm>

#include "xd_launch.h"
#include "xd_warp16.cuh"

namespace xd {

// A warp per task: tasks list[0 .. *n_ptr), or all tasks of the job without
// a list, by a counter; tasks too wide for 512 slots go to out.  Without a
// list: tasks that outgrew 128 slots are noted in over, and with n_bad the
// pairs are validated as validate_kernel does.  ANY as in extend_warp: its code
// costs the others registers (137 and 165) and 200 pairs of 2-4 kb reads 8 us
// of 443.
template <bool ANY>
__global__ void __launch_bounds__(kWarpThreads)
warp_kernel(Job *jp, const Job value, bool by_value, const uint32_t *list, const uint32_t *n_ptr, uint32_t *counter,
            int from, uint32_t *n_bad, Spill over, Spill out)
{
    const Job J = by_value ? value : *jp;
    if (by_value && blockIdx.x == 0 && threadIdx.x == 0) *jp = value;  // for the next launch
    const int lane = threadIdx.x & 31;
    const uint32_t n = list ? *n_ptr : (uint32_t)(2 * J.n_pairs);
    for (;;) {
        uint32_t k = 0;
        if (lane == 0) k = atomicAdd(counter, 1u);
        k = __shfl_sync(FULL, k, 0);
        if (k >= n) break;
        const uint32_t task = list ? list[k] : k;
        const Ext e = decode(J, task);
        if (n_bad && e.side == 0 && lane == 0) write_status(J, e.pair, e.ok, n_bad);
        if (!e.ok) continue;
        int32_t sc, bi, bj;
        const int st = extend_warp<ANY>(e, J.sc, from, lane, sc, bi, bj);
        if (lane == 0) {
            if (!list && st) over.list[atomicAdd(over.count, 1u)] = task;
            if (st < 0) hand_on_wide(out, task, e.m);
            else write_result(J, e, sc, bi, bj);
        }
        __syncwarp();
    }
}

bool warp_packed(const Scoring &sc) { return warp16_ok<2>(sc); }

cudaError_t launch_warp(uint64_t n_tasks, int sm_count, Job *jp, const Job *value, const uint32_t *list,
                        const uint32_t *n_ptr, uint32_t *counter, int from, uint32_t *n_bad,
                        Spill over, Spill out, cudaStream_t s)
{
    // a warp per task, in blocks of one warp while there are few (every
    // scheduler gets one before any gets two), at most what fits the SMs
    const int threads = n_tasks <= (uint64_t)sm_count * 4 ? 32 : kWarpThreads;
    const uint64_t warps = threads / 32, cap = (uint64_t)sm_count * 16 / warps;
    const uint64_t blocks = std::min<uint64_t>((n_tasks + warps - 1) / warps, cap);
    if (!blocks) return cudaSuccess;
    (void)cudaGetLastError();
    // a list's scoring is in device memory, and a captured launch serves them all
    const Scoring sc = value ? effective(value->sc) : Scoring{};
    const bool any = !value || (packed16_ok(sc) && !warp_packed(sc));
    const auto kernel = any ? warp_kernel<true> : warp_kernel<false>;
    kernel<<<(unsigned)blocks, threads, 0, s>>>(jp, value ? *value : Job{}, value != nullptr, list,
                                                n_ptr, counter, from, n_bad, over, out);
    return cudaGetLastError();
}

}  // namespace xd
