// Packed 16-bit band tiles (two window slots per register): 4x8, 2x16 and
// 1x32 (width 32, narrow bands such as x = 15), 4x16, 8x8 and 2x32 (width 64),
// 8x16, 16x8, 4x32 and 2x64 (width 128).  Lanes of 32 and 64 slots spread each
// diagonal's per-lane bookkeeping over more cells; 1x64 lost to 2x32 (50.6
// against 45.0 ms, 29x, x = 50: twice the events per warp, half the warps).
#include "xd_launch.h"
#include "xd_serve_kernels.cuh"
#include "xd_warp16.cuh"

namespace xd {

// The single-extension part of a group tier's kernel (WarpRole): first the
// n_long longest tasks of the order, then the tier's overflow, with wait
// until the tier is done or none came for kRoleIdleNs (the warp then joins
// the tier), else what there is now.  Entries of the overflow list start as
// kNoTask and appear right after their position was reserved, so the wait
// for one is short; it is bounded all the same.  (A compare-and-swap on the
// number taken claims safely too, but loses to every other claim: 1,824
// warps on one word and 154,000 entries took 230 ms instead of 25.)
constexpr unsigned long long kRoleIdleNs = 300000;
constexpr int kEntryTries = 1 << 20;

static __device__ __noinline__ void run_warp_role(const Job *jp, const uint32_t *order, Spill spill,
                                           WarpRole role, uint32_t n_long, int width, bool wait,
                                           uint32_t first_warps)
{
    const Job J = *jp;
    const int lane = threadIdx.x & 31;
    bool longest = n_long > 0;
    unsigned long long idle = 0;
    int busy = 0;  // turns in a row without a right, though entries were left
    for (;;) {
        enum { kAgain = 0, kTask = 1, kLeave = 2 };
        int act = kAgain;
        uint32_t task = kNoTask;
        if (lane == 0) {
            if (longest) {
                const uint32_t k = atomicAdd(role.long_ctr, 1u);
                if (k < n_long) {
                    task = order[k];
                    act = kTask;
                } else {
                    longest = false;
                }
            }
            if (act == kAgain) {
                // done before count: what the last warp handed on is seen
                const uint32_t done = *(volatile uint32_t *)role.done;
                __threadfence();
                DeviceMem mem;
                uint32_t t = 0;
                Claim claim = Claim::kBusy;
                for (int tries = 0; tries < 4 && claim == Claim::kBusy; ++tries)
                    claim = claim_entry(mem, ClaimWords{spill.count, role.ready, role.taken}, &t);
                if (claim == Claim::kGot) {
                    for (int spin = 0; spin < kEntryTries && task == kNoTask; ++spin) {
                        task = *(volatile uint32_t *)&spill.list[t];
                        if (task == kNoTask) __nanosleep(32);
                    }
                    if (task == kNoTask) *role.err = 1u;
                    act = kTask;
                    busy = 0;
                } else if (claim == Claim::kEmpty) {
                    busy = 0;
                    if (!wait || done >= first_warps) {
                        act = kLeave;
                    } else {
                        unsigned long long now;
                        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                        if (idle == 0) idle = now;
                        if (now - idle > kRoleIdleNs) act = kLeave;
                        else __nanosleep(1000);
                    }
                } else if (++busy > kEntryTries) {
                    *role.err = 1u;  // a reserved entry was never written
                    act = kLeave;
                } else {
                    __nanosleep(200 + 37 * (blockIdx.x & 31));  // lost every race
                }
            }
        }
        act = __shfl_sync(FULL, act, 0);
        if (act == kLeave) return;
        if (act == kAgain) continue;
        idle = 0;
        task = __shfl_sync(FULL, task, 0);
        const bool whole = __shfl_sync(FULL, (int)longest, 0) != 0;
        if (task == kNoTask) continue;
        const Ext e = decode(J, task);
        if (!e.ok) continue;
        int32_t sc, bi, bj;
        // (with ANY the group loop of the calling kernel is compiled worse: 29x,
        // x = 15, 22.4 and 23.9 ms)
        const int st = extend_warp<false>(e, J.sc, whole ? 0 : width, lane, sc, bi, bj);
        if (lane == 0) {
            if (whole && st) {
                const uint32_t k = atomicAdd(role.grown, 1u);
                if (role.grown_end) *(role.grown_end - 1 - k) = task;
            }
            if (st < 0) hand_on_wide(role.wide, task, e.m);
            else write_result(J, e, sc, bi, bj);
        }
        __syncwarp();
    }
}

// Batched form of the packed kernel (same task source as lockstep_kernel).
// With a WarpRole the first blocks give their warps to single extensions
// first: a launch ends with its longest extension, and one that outgrew the
// window would start over only after the launch.  Every warp that runs out of
// tasks takes overflow too, so none is left when the kernel ends (short
// overflow, which can be plentiful, goes to `brief`, the tasks of a second,
// wider group tier: a warp each costs it four times as much).
// Blocks of 128 threads.  The registers are capped for 3 blocks per SM with 32
// or 64 slots per lane, 4 with 16 and 5 with fewer: more warps at fewer
// registers measured slower (29x, x = 50, first tier: 2x32 at 3, 4 and 5
// blocks 45.8, 46.0 and 48.8 ms; 4x16 at 4, 5 and 6 blocks 52.0, 54.2 and 57.7).
template <int C2>
__host__ __device__ constexpr int packed_min_blocks() { return C2 >= 16 ? 3 : C2 == 8 ? 4 : 5; }
template <int L, int C2>
__global__ void __launch_bounds__(kPackedThreads, packed_min_blocks<C2>())
lockstep16_kernel(const Job *jp, const uint32_t *order, const uint32_t *n_tasks_ptr,
                  uint32_t *counter, Spill spill, Spill brief, uint32_t one, WarpRole role)
{
    constexpr int W = L * 2 * C2;
    const uint32_t n_tasks = *n_tasks_ptr;
    if (role.n_long) {
        const uint32_t mine = *role.n_blocks;
        const bool all = n_tasks <= role.few;
        if (all || blockIdx.x < mine)
            run_warp_role(jp, order, spill, role, all ? n_tasks : *role.n_long, all ? W / 2 : W,
                          !all, (gridDim.x - mine) * (kPackedThreads / 32));
        if (all) return;
    }
    BatchSrc src{jp, order, n_tasks, counter, spill, brief, role.ready};
    lockstep16_loop<L, C2>(src, jp->packed, jp->n_words, one);
    if (role.n_long) {
        __syncwarp();
        if ((threadIdx.x & 31) == 0 && blockIdx.x >= *role.n_blocks) {
            __threadfence();  // this warp's overflow entries before its count
            atomicAdd(role.done, 1u);
        }
        run_warp_role(jp, order, spill, role, 0, W, false, 0);
    }
}

template <int L, int C2>
static cudaError_t abs_impl(int grid, const Job *jp, const uint32_t *order, const uint32_t *n,
                            uint32_t *ctr, Spill sp, cudaStream_t s)
{
    (void)cudaGetLastError();
    lockstep16_abs_kernel<L, C2><<<grid, kPackedThreads, 0, s>>>(jp, order, n, ctr, sp, 1u);
    return cudaGetLastError();
}

template <int L, int C2>
static cudaError_t packed_impl(int grid, const Job *jp, const uint32_t *order, const uint32_t *n,
                               uint32_t *ctr, Spill sp, Spill brief, WarpRole role,
                               cudaStream_t s)
{
    (void)cudaGetLastError();
    lockstep16_kernel<L, C2><<<grid, kPackedThreads, 0, s>>>(jp, order, n, ctr, sp, brief, 1u, role);
    return cudaGetLastError();
}

template <class K>
static int occupancy_impl(K kernel)
{
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, kPackedThreads, 0);
    return b;
}

template <int L, int C2>
static int packed_occupancy_impl()
{
    return occupancy_impl(lockstep16_kernel<L, C2>);
}

cudaError_t launch_persistent_packed(Tile t, int grid, const Job *jp, const uint32_t *order,
                                     const uint32_t *n, uint32_t *ctr, Spill sp, Spill brief,
                                     WarpRole role, cudaStream_t s, bool *handled)
{
    *handled = true;
    if (t.packed) {
        if (t.absolute && t.c == 32) {
            if (t.lanes == 2) return abs_impl<2, 16>(grid, jp, order, n, ctr, sp, s);
            if (t.lanes == 4) return abs_impl<4, 16>(grid, jp, order, n, ctr, sp, s);
        }
        if (t.lanes == 4 && t.c == 8) return packed_impl<4, 4>(grid, jp, order, n, ctr, sp, brief, role, s);
        if (t.lanes == 2 && t.c == 16) return packed_impl<2, 8>(grid, jp, order, n, ctr, sp, brief, role, s);
        if (t.lanes == 4 && t.c == 16) return packed_impl<4, 8>(grid, jp, order, n, ctr, sp, brief, role, s);
        if (t.lanes == 8 && t.c == 8) return packed_impl<8, 4>(grid, jp, order, n, ctr, sp, brief, role, s);
        if (t.lanes == 8 && t.c == 16) return packed_impl<8, 8>(grid, jp, order, n, ctr, sp, brief, role, s);
        if (t.lanes == 16 && t.c == 8) return packed_impl<16, 4>(grid, jp, order, n, ctr, sp, brief, role, s);
        if (t.lanes == 2 && t.c == 32) return packed_impl<2, 16>(grid, jp, order, n, ctr, sp, brief, role, s);
        if (t.lanes == 4 && t.c == 32) return packed_impl<4, 16>(grid, jp, order, n, ctr, sp, brief, role, s);
        if (t.lanes == 1 && t.c == 32) return packed_impl<1, 16>(grid, jp, order, n, ctr, sp, brief, role, s);
        if (t.lanes == 2 && t.c == 64) return packed_impl<2, 32>(grid, jp, order, n, ctr, sp, brief, role, s);
    }
    *handled = false;
    return cudaSuccess;
}

int occupancy_packed(Tile t)
{
    if (!t.packed) return -1;
    if (t.absolute && t.c == 32) {
        if (t.lanes == 2) return occupancy_impl(lockstep16_abs_kernel<2, 16>);
        if (t.lanes == 4) return occupancy_impl(lockstep16_abs_kernel<4, 16>);
    }
    if (t.lanes == 4 && t.c == 8) return packed_occupancy_impl<4, 4>();
    if (t.lanes == 2 && t.c == 16) return packed_occupancy_impl<2, 8>();
    if (t.lanes == 4 && t.c == 16) return packed_occupancy_impl<4, 8>();
    if (t.lanes == 8 && t.c == 8) return packed_occupancy_impl<8, 4>();
    if (t.lanes == 8 && t.c == 16) return packed_occupancy_impl<8, 8>();
    if (t.lanes == 16 && t.c == 8) return packed_occupancy_impl<16, 4>();
    if (t.lanes == 2 && t.c == 32) return packed_occupancy_impl<2, 16>();
    if (t.lanes == 4 && t.c == 32) return packed_occupancy_impl<4, 16>();
    if (t.lanes == 1 && t.c == 32) return packed_occupancy_impl<1, 16>();
    if (t.lanes == 2 && t.c == 64) return packed_occupancy_impl<2, 32>();
    return -1;
}

bool packed_scoring_ok(const Scoring &sc) { return packed16_ok(sc); }

bool packed_tile_ok(Tile t, const Scoring &sc)
{
    if (!t.packed) return false;
    if (t.c == 64) return relative_ok<64>(sc);
    if (t.c == 32) return t.lanes == 1 ? relative_ok<32>(sc) : packed32_ok(sc);
    return packed16_ok(sc);
}

// Lanes of 32 slots hold x + match <= 1022 (packed32_ok) in the absolute
// frame; the relative one needs x + 2 match + 2|gap| < 1024 there.
Tile in_frame(Tile t, const Scoring &sc)
{
    t.absolute = t.packed && t.c == 32 && t.lanes > 1 && !relative_ok<32>(sc);
    return t;
}

Tile usable_tile(Tile t, const Scoring &sc)
{
    if (!t.packed || packed_tile_ok(t, sc)) return in_frame(t, sc);
    // the 16-slot tile of the same width, or its 32-bit twin
    const Tile h{t.width() / 16, 16, true};
    if (t.c >= 32 && packed16_ok(sc)) return h;
    if (t.width() < 64) return Tile{4, 16, false};  // no 32-bit tile this narrow
    if (t.c >= 32) return Tile{h.lanes, 16, false};
    return Tile{t.lanes, t.c, false};
}

bool has_warp_role(Tile t) { return t.packed && !t.absolute; }

// What the price of a cut between single warps and groups (bin_scan_kernel)
// takes from the tile: diagonals per ns of a full first tier (3,500 window
// slots per ns; 5,000 at its best) and the ns per diagonal of one of its extensions.
void tile_rates(Tile t, float *rate, float *group_ns)
{
    *rate = 3500.f / (float)t.width();
    *group_ns = 40.f + 9.f * (float)t.c;
}

int persistent_block_threads(Tile t) { return t.packed ? kPackedThreads : 256; }

template <int L1, int C2a, int L2, int C2>
static cudaError_t serve16_impl(int grid, const ServeArgs &a, const uint32_t *pk, int64_t nw,
                                cudaStream_t s)
{
    (void)cudaGetLastError();
    serve16_kernel<L1, C2a, L2, C2><<<grid, 256, 0, s>>>(a, pk, nw);
    return cudaGetLastError();
}

template <int L1, int C2a, int L2, int C2>
static int serve16_occupancy_impl()
{
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, serve16_kernel<L1, C2a, L2, C2>, 256, 0);
    return b;
}

// The ring warps' tile: 2x32 as it is (75 requests of 1,000 to 20,000 pairs of
// 29x reads, x = 50: 163 ms, and 172 ms with 4x16), other lanes of 32 and
// more slots as the 16-slot tile of their width.
static Tile serve_tile(Tile t)
{
    if (t.c <= 16 || (t.lanes == 2 && t.c == 32)) return t;
    return Tile{t.width() / 16, 16, true};
}

// Second tier as for the 32-bit tiles: 16x8 after a 64-slot first tier,
// 32x16 after a 128-slot one.
cudaError_t launch_serve_packed(Tile t, int grid, const ServeArgs &a, const uint32_t *pk,
                                int64_t nw, cudaStream_t s, bool *handled)
{
    *handled = true;
    if (t.packed) {
        t = serve_tile(t);
        if (t.lanes == 2 && t.c == 32) return serve16_impl<2, 16, 16, 8>(grid, a, pk, nw, s);
        if (t.lanes == 4 && t.c == 16) return serve16_impl<4, 8, 16, 8>(grid, a, pk, nw, s);
        if (t.lanes == 8 && t.c == 8) return serve16_impl<8, 4, 16, 8>(grid, a, pk, nw, s);
        if (t.lanes == 8 && t.c == 16) return serve16_impl<8, 8, 32, 16>(grid, a, pk, nw, s);
        if (t.lanes == 16 && t.c == 8) return serve16_impl<16, 4, 32, 16>(grid, a, pk, nw, s);
    }
    *handled = false;
    return cudaSuccess;
}

int serve_occupancy_packed(Tile t)
{
    if (!t.packed) return -1;
    t = serve_tile(t);
    if (t.lanes == 2 && t.c == 32) return serve16_occupancy_impl<2, 16, 16, 8>();
    if (t.lanes == 4 && t.c == 16) return serve16_occupancy_impl<4, 8, 16, 8>();
    if (t.lanes == 8 && t.c == 8) return serve16_occupancy_impl<8, 4, 16, 8>();
    if (t.lanes == 8 && t.c == 16) return serve16_occupancy_impl<8, 8, 32, 16>();
    if (t.lanes == 16 && t.c == 8) return serve16_occupancy_impl<16, 4, 32, 16>();
    return -1;
}

}  // namespace xd
