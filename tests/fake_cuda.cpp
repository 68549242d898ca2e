// A CUDA runtime of host memory, and launchers that run no kernel, under the
// library's host code (paper_2309_07270_gb300/csrc/xd_api.cu, compiled with
// it), for tests of what the host does when an allocation fails, an event
// is late or a kernel reports an error (test infrastructure).  Streams are
// synchronous; a captured graph replays its launches.
#include <cuda_runtime.h>
#include <stdint.h>

static inline uint32_t atomicAdd(uint32_t *p, uint32_t v) { const uint32_t o = *p; *p += v; return o; }
static inline uint32_t atomicMax(uint32_t *p, uint32_t v) { const uint32_t o = *p; if (v > o) *p = v; return o; }

#include "../paper_2309_07270_gb300/csrc/xd_api.cu"

#include <atomic>
#include <functional>

// ------------------------------------------------------------ the test's side
namespace fake {
struct Event { std::chrono::steady_clock::time_point at; };
struct Graph { std::vector<std::function<void()>> run; };
std::map<void *, size_t> device_mem;
size_t device_used = 0, device_size = (size_t)-1, pool_reserved = 0, seed_tables = 0;
int graphs = 0, last_longest = -1, bad_scratch = 0;
int lose_entries = 0;                        // the next first tiers lose an entry
std::atomic<int> late_us{0}, polling{0}, polling_max{0};
Graph *capture = nullptr;
uint32_t *ctrs = nullptr;
cudaError_t launched(std::function<void()> f)
{
    if (capture) capture->run.push_back(f);
    else f();
    return cudaSuccess;
}
}  // namespace fake

extern "C" {
int xdrop_align_static(const uint32_t *, uint64_t, const uint64_t *, const uint32_t *, uint32_t,
                       const xdrop_pair *, size_t, const xdrop_scoring *, uint32_t, xdrop_result *,
                       void *) { return XDROP_ECUDA; }
const char *xdrop_static_last_error(void) { return ""; }
void fake_device_size(size_t bytes) { fake::device_size = bytes; }
size_t fake_device_used(void) { return fake::device_used + fake::pool_reserved; }
void fake_pool_reserved(size_t bytes) { fake::pool_reserved = bytes; }
void fake_seed_tables(size_t bytes) { fake::seed_tables = bytes; }
void fake_lose_entries(int n) { fake::lose_entries = n; }
void fake_late_us(int us) { fake::late_us = us; }
int fake_polling_max(void) { return fake::polling_max.exchange(0); }
int fake_bad_scratch(void) { return fake::bad_scratch; }
int fake_graphs(void) { return fake::graphs; }
int fake_last_longest(void) { return fake::last_longest; }

// ------------------------------------------------------------ the runtime
cudaError_t cudaMalloc(void **p, size_t n)
{
    if (n > fake::device_size || fake::device_used + fake::pool_reserved > fake::device_size - n)
        return cudaErrorMemoryAllocation;
    *p = calloc(1, n ? n : 1);
    fake::device_mem[*p] = n;
    fake::device_used += n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    auto it = fake::device_mem.find(p);
    if (!p || it == fake::device_mem.end()) return p ? cudaErrorInvalidValue : cudaSuccess;
    fake::device_used -= it->second;
    fake::device_mem.erase(it);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    return fake::launched([=] { memcpy(d, s, n); });
}
cudaError_t cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t)
{
    return fake::launched([=] { memset(d, v, n); });
}
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 4; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "fake error"; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { free((void *)s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t) new fake::Event(); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete (fake::Event *)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t)
{
    ((fake::Event *)e)->at = std::chrono::steady_clock::now() + std::chrono::microseconds(fake::late_us);
    return cudaSuccess;
}
cudaError_t cudaEventRecordWithFlags(cudaEvent_t e, cudaStream_t s, unsigned) { return cudaEventRecord(e, s); }
cudaError_t cudaEventQuery(cudaEvent_t e)
{
    const int now = ++fake::polling;
    for (int m = fake::polling_max; now > m && !fake::polling_max.compare_exchange_weak(m, now);) {}
    std::this_thread::sleep_for(std::chrono::microseconds(20));
    --fake::polling;
    return std::chrono::steady_clock::now() < ((fake::Event *)e)->at ? cudaErrorNotReady : cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e)
{
    std::this_thread::sleep_until(((fake::Event *)e)->at);
    return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { fake::capture = new fake::Graph(); return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g)
{
    *g = (cudaGraph_t)fake::capture;
    fake::capture = nullptr;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long)
{
    *x = (cudaGraphExec_t) new fake::Graph(*(fake::Graph *)g);
    ++fake::graphs;
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t)
{
    for (auto &f : ((fake::Graph *)x)->run) f();
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete (fake::Graph *)g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { delete (fake::Graph *)x; return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) { *p = (cudaMemPool_t)malloc(1); return cudaSuccess; }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t p) { free((void *)p); fake::pool_reserved = 0; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *v)
{
    *(uint64_t *)v = fake::pool_reserved;
    return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t keep)
{
    fake::pool_reserved = std::min(fake::pool_reserved, keep);
    return cudaSuccess;
}
}  // extern "C"

// ------------------------------------------------------------ the launchers
namespace xd {
bool packed_scoring_ok(const Scoring &) { return true; }
bool packed_tile_ok(Tile, const Scoring &) { return true; }
bool warp_packed(const Scoring &) { return true; }
Tile in_frame(Tile t, const Scoring &) { return t; }
Tile usable_tile(Tile t, const Scoring &) { return t; }
bool has_warp_role(Tile t) { return t.packed; }
int persistent_block_threads(Tile) { return 128; }
int persistent_blocks_per_sm(Tile) { return 3; }
cudaError_t launch_persistent(Tile, int, const Job *, const uint32_t *, const uint32_t *, uint32_t *,
                              Spill, Spill, WarpRole role, cudaStream_t)
{
    return fake::launched([=] {
        if (role.err && fake::lose_entries > 0 && !fake::capture) {
            --fake::lose_entries;
            *role.err = 1;
        }
    });
}
cudaError_t launch_warp(uint64_t, int, Job *jp, const Job *value, const uint32_t *, const uint32_t *,
                        uint32_t *, int, uint32_t *, Spill, Spill, cudaStream_t)
{
    if (value) *jp = *value;
    return cudaSuccess;
}
cudaError_t launch_wide(bool, int grid, const Job *, Spill, int32_t *scratch, int64_t per, uint32_t *, cudaStream_t)
{
    return fake::launched([=] {  // a scratch that is not there, or too small for the slices
        auto it = fake::device_mem.find(scratch);
        fake::bad_scratch += it == fake::device_mem.end() || it->second < (size_t)per * 4 * grid;
    });
}
cudaError_t launch_window(Tile, bool, const Job *, uint32_t, uint32_t, Spill, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_validate(const Job *, uint64_t, uint32_t *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_binning(const Job *, int, uint32_t *, uint32_t *, uint32_t *, uint32_t *, uint32_t *,
                           Tile, int, WarpRole, bool longest, cudaStream_t)
{
    return fake::launched([=] { fake::last_longest = longest; });
}
cudaError_t launch_length_hist(const Job *, int, uint32_t *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_sample_pairs(const Pair *, uint64_t, uint32_t, uint32_t, Pair *, uint64_t, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_plain_setup(uint64_t, uint64_t, uint32_t *, uint32_t *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_revcomp(const uint32_t *, int64_t, const uint64_t *, const uint32_t *, uint32_t, uint32_t *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_best_seeds(const Pair *, const int32_t *, uint64_t, int32_t, uint32_t *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_accept(const Pair *, const int32_t *, const uint32_t *, uint32_t, uint64_t, int32_t, int32_t, uint32_t, uint32_t, uint8_t *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_max_len(const uint32_t *len, uint32_t n, uint32_t *out, cudaStream_t)
{
    for (uint32_t k = 0; k < n; ++k) *out = std::max(*out, len[k]);
    return cudaSuccess;
}
// its tables: as much as the test sets aside
int find_candidates(cudaStream_t, cudaMemPool_t, int, size_t, const uint32_t *, const uint64_t *,
                    const uint32_t *, uint32_t, const uint32_t *, uint32_t, uint32_t, uint32_t,
                    uint32_t, uint32_t, std::vector<Pair> &, std::vector<uint32_t> &, SeedStats &,
                    std::string &err)
{
    if (fake::device_used + std::max(fake::seed_tables, fake::pool_reserved) > fake::device_size) {
        err = "out of memory";
        return XDROP_ENOMEM;
    }
    fake::pool_reserved = std::max(fake::seed_tables, fake::pool_reserved);
    return XDROP_OK;
}
Server *server_create(int, int, size_t, Tile, const ResidentReads &, const uint32_t *, int32_t *,
                      int64_t, int, uint64_t, std::string &) { return nullptr; }
int server_submit(Server *, const xdrop_pair *, size_t, const Scoring &, xdrop_result *, uint64_t *, std::string &) { return XDROP_ECUDA; }
int server_sync(Server *, uint64_t, int64_t, std::string &) { return XDROP_ECUDA; }
ServerStats server_stats(Server *) { return ServerStats{}; }
void server_set_idle_ns(Server *, uint64_t) {}
void server_destroy(Server *) {}
}  // namespace xd
