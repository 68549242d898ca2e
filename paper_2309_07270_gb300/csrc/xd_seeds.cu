// Seed discovery on the device: reliable k-mers and candidate read pairs
// (the per-element steps and the readings are in xd_seeds.cuh).
//
// Front steps, shared by both products, on one stream, tables in HBM:
//   1. kmer_kernel: one thread per k-mer occurrence computes its canonical
//      code (3 word loads, a 2-bit-group reversal), its read (binary search
//      of the per-read occurrence offsets) and its strand (one warp ballot
//      per 32 occurrences);
//   2. a stable radix sort of (code, occurrence id) over the code's 2k bits:
//      each k-mer's occurrences become one run, in read and position order;
//   3. the runs of length >= 2 (run-length encoding).
// Then A * A^T, A the read-by-reliable-k-mer matrix, one of two ways:
//   sort-based (XDROP_SEEDS_SORT): count_kernel and emit_kernel write one
//      entry per (read pair, shared reliable k-mer); a radix sort by pair, a
//      gather and a reduce-by-key with xs::CandMerge give one candidate per
//      pair;
//   row-wise (default): A's columns and the place of every occurrence in
//      them (column_kernel), then row_kernel, one block per read a, accumulates
//      a's partners b > a in a shared-memory hash table (count + 64-bit
//      minimum seed key per partner, shared-memory atomics) in one pass,
//      staging up to 256 partners per read (a second pass rewrites the rare
//      reads with more); a radix sort of the few candidates orders them.  No per-entry
//      table exists.  A read with more partners than the table holds makes
//      the call take the sort-based product instead (same result).
// The sorts, run-length encoding, scans and reduce-by-key are CUB library
// primitives; everything else is the kernels here.
#include <cuda_runtime.h>

#include <cub/device/device_radix_sort.cuh>
#include <cub/device/device_reduce.cuh>
#include <cub/device/device_run_length_encode.cuh>
#include <cub/device/device_scan.cuh>

#include <algorithm>
#include <string>
#include <vector>

#include "../../include/xdrop.h"
#include "xd_launch.h"
#include "xd_seeds.cuh"

namespace xd {

namespace {

constexpr int kThreads = 256;
constexpr uint64_t kMaxItems = (1ull << 31) - 1;  // CUB item counts are int

// ---------------------------------------------------------------- front

__global__ void __launch_bounds__(kThreads)
kmer_kernel(const uint32_t *__restrict__ packed, const uint64_t *__restrict__ read_off,
            const uint64_t *__restrict__ occ_off, uint32_t n_reads, uint64_t n_occ, uint32_t k,
            uint32_t stride, uint64_t *__restrict__ keys, uint32_t *__restrict__ occ,
            uint32_t *__restrict__ occ_rd, uint32_t *__restrict__ fwd_bits)
{
    const uint32_t lane = threadIdx.x & 31;
    // base is a multiple of 32 and the same for all lanes of a warp, so the
    // loop and the ballot are warp-uniform
    for (uint64_t base = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x - lane; base < n_occ;
         base += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t q = base + lane;
        bool fwd = false;
        if (q < n_occ) {
            uint32_t r;
            keys[q] = xs::occurrence(packed, read_off, occ_off, n_reads, k, stride, q, &r, &fwd);
            occ[q] = (uint32_t)q;
            occ_rd[q] = r;
        }
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, fwd);
        if (lane == 0) fwd_bits[base >> 5] = m;
    }
}

// ---------------------------------------------------- sort-based product

__global__ void __launch_bounds__(kThreads)
count_kernel(const uint32_t *__restrict__ occ, const uint32_t *__restrict__ occ_rd,
             const int *__restrict__ run_off, const int *__restrict__ run_len, int n_runs,
             uint32_t lo, uint32_t hi, uint64_t *__restrict__ npairs)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_runs; i += gridDim.x * blockDim.x)
        npairs[i] = xs::run_pairs(occ, occ_rd, (uint64_t)run_off[i], (uint32_t)run_len[i], lo, hi);
}

__global__ void __launch_bounds__(kThreads)
emit_kernel(const uint64_t *__restrict__ codes, const uint32_t *__restrict__ occ,
            const uint32_t *__restrict__ occ_rd, const uint32_t *__restrict__ fwd_bits,
            const uint64_t *__restrict__ occ_off, const uint32_t *__restrict__ read_len,
            const int *__restrict__ run_off, const int *__restrict__ run_len,
            const uint64_t *__restrict__ pair_end, int n_runs, uint32_t k, uint32_t stride,
            uint32_t nb, uint64_t *__restrict__ keys, xs::Cand *__restrict__ ent,
            uint32_t *__restrict__ idx)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_runs; i += gridDim.x * blockDim.x) {
        const uint64_t e0 = i ? pair_end[i - 1] : 0;
        if (pair_end[i] == e0) continue;
        const uint64_t s = (uint64_t)run_off[i];
        xs::run_emit(occ, occ_rd, fwd_bits, occ_off, read_len, codes[s], s, (uint32_t)run_len[i],
                     k, stride, nb, e0, keys, ent, idx);
    }
}

__global__ void __launch_bounds__(kThreads)
gather_kernel(const xs::Cand *__restrict__ ent, const uint32_t *__restrict__ idx, uint64_t n,
              xs::Cand *__restrict__ out)
{
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x)
        out[i] = ent[idx[i]];
}

__global__ void __launch_bounds__(kThreads)
out_kernel(const uint64_t *__restrict__ keys, const xs::Cand *__restrict__ agg, int n,
           uint32_t nb, uint32_t k, Pair *__restrict__ pairs, uint32_t *__restrict__ shared)
{
    const uint64_t mask = nb >= 32 ? 0xFFFFFFFFull : (1ull << nb) - 1;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const xs::Cand c = agg[i];
        Pair p;
        p.a = (uint32_t)(keys[i] >> nb);
        p.b = (uint32_t)(keys[i] & mask) | (c.rc ? xs::kPairRC : 0u);
        p.seed_a = c.pa;
        p.seed_b = c.sb;
        p.seed_len = k;
        pairs[i] = p;
        shared[i] = c.shared;
    }
}

// ------------------------------------------------------ row-wise product

// The columns of A (reliable runs) and where their members stand.  A warp
// takes 32 runs, reserves room for their entries with one atomic (columns
// may stand in any order, and the entries that are no read's first leave
// holes after a column), then writes one column after the other, a lane per
// entry: member words in read order, the last one marked kLast, and for the
// member's occurrence q, row_of[q] = the member's index.  Rows need no table
// of their own: row a is the occurrences of read a, in order of position.
// Bound by the gathers of occ_rd and occ_off: 0.60 ms at 1 Mb and 29x, where
// a thread per run, a scan and a scatter of the rows took 1.51.
constexpr unsigned long long kLast = 1ull << 63;  // read ids are below 2^31
constexpr uint32_t kNone = 0xFFFFFFFFu;

__global__ void __launch_bounds__(kThreads)
column_kernel(const uint32_t *__restrict__ occ, const uint32_t *__restrict__ occ_rd,
              const uint32_t *__restrict__ fwd_bits, const uint64_t *__restrict__ occ_off,
              const int *__restrict__ run_off, const int *__restrict__ run_len, int n_runs,
              uint32_t lo, uint32_t hi, uint32_t stride, uint64_t *__restrict__ members,
              uint32_t *__restrict__ row_of, uint32_t *__restrict__ cursor,
              unsigned long long *__restrict__ nonzeros)
{
    const uint32_t lane = threadIdx.x & 31;
    const int warps = (int)((gridDim.x * blockDim.x) >> 5);
    uint32_t nnz = 0;
    for (int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); w * 32ll < n_runs; w += warps) {
        const int i = w * 32 + (int)lane;
        uint32_t cnt = 0, off = 0;
        if (i < n_runs) {
            cnt = (uint32_t)run_len[i];
            off = (uint32_t)run_off[i];
            if (cnt < lo || cnt > hi) cnt = 0;
        }
        uint32_t sum = cnt;  // inclusive scan over the warp's runs
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, sum, d);
            if (lane >= (uint32_t)d) sum += v;
        }
        uint32_t base = 0;
        if (lane == 31 && sum) base = atomicAdd(cursor, sum);
        base = __shfl_sync(0xFFFFFFFFu, base, 31) + sum - cnt;
        for (unsigned todo = __ballot_sync(0xFFFFFFFFu, cnt != 0); todo; todo &= todo - 1) {
            const int r = __ffs((int)todo) - 1;
            const uint32_t s0 = __shfl_sync(0xFFFFFFFFu, off, r), n = __shfl_sync(0xFFFFFFFFu, cnt, r);
            const uint32_t c0 = __shfl_sync(0xFFFFFFFFu, base, r);
            uint32_t u = 0, before = kNone;  // members so far, read of the last entry
            for (uint32_t e0 = 0; e0 < n; e0 += 32) {
                const bool in = e0 + lane < n;
                const uint32_t q = in ? occ[s0 + e0 + lane] : 0u;
                const uint32_t rd = in ? occ_rd[q] : kNone;
                uint32_t prev = __shfl_up_sync(0xFFFFFFFFu, rd, 1);
                if (lane == 0) prev = before;
                const bool first = in && rd != prev;  // its read's first occurrence
                const unsigned m = __ballot_sync(0xFFFFFFFFu, first);
                if (first) {
                    const uint32_t j = c0 + u + __popc(m & ((1u << lane) - 1u));
                    members[j] = xs::member_word(rd, (uint32_t)((q - occ_off[rd]) * stride),
                                                 xs::fwd_bit(fwd_bits, q));
                    row_of[q] = j;
                }
                u += (uint32_t)__popc(m);
                before = __shfl_sync(0xFFFFFFFFu, rd, 31);
            }
            __syncwarp();
            if (lane == 0) {
                members[c0 + u - 1] |= kLast;
                nnz += u;
            }
        }
    }
    if (lane == 0 && nnz) atomicAdd(nonzeros, (unsigned long long)nnz);
}

// Partners of a read kept in its staging area by the first pass; a read
// with more goes through the second pass.
constexpr uint32_t kStage = 256;

// Per-read staging of the first pass: partner id, 64-bit best seed and
// shared count of up to kStage partners of every read.
struct Stage {
    uint32_t *key;
    unsigned long long *best;
    uint32_t *cnt;
};

// One block per read a: the partners b > a of a in a shared-memory table.
// The members behind a's own in a column are exactly those (columns are in
// read order), so half of the column is never read.  A warp takes 32
// positions of a, then a half warp per reliable one walks its column from
// behind a's member to the one marked kLast, a lane per member.  Positions
// come in increasing order, so the first term of a partner almost always
// holds its smallest position and the 64-bit minimum is skipped after it (a
// stale read of it can only be too large, which costs one atomic).  1 Mb
// genome at 29x, 182.8 M terms: 1.28 ms, issue and the columns' loads
// (1.6 GB of DRAM); with a warp per whole column and three atomics a term
// 4.85.  A block lasts as long as its read, so long reads take 1,024 threads
// (that genome's pipeline at 256, 512 and 1,024: 4.9, 4.5, 4.5 ms; 12 reads of
// 100-200 kb 4.7, 2.6, 1.6), and fills and empties its table, so short ones take
// 256 (60,000 of 100-150 bases: 3.0, 3.4, 4.8 ms; 40,000 of 300: 2.7, 2.8, 3.7;
// 5,000 of 1 kb: 0.98, 0.95, 1.02).
//
// WRITE = false (first pass, block a = read a): cand_cnt[a] = number of
// partners (0 and the overflow flag when the table is full); up to kStage
// partners go to a's staging area, a read with more is listed in big.
// WRITE = true (second pass, block i = read big[i]): the partners' records
// at cand_end[a-1] ..., in table order.
constexpr int kRowThreads = 1024, kShortRowThreads = 256;
constexpr uint64_t kShortMean = 1024, kShortLongest = 32768;  // positions a read, of short reads
constexpr int kCols = 2;          // columns in flight per half warp
template <bool WRITE>
__global__ void __launch_bounds__(kRowThreads)
row_kernel(const uint64_t *__restrict__ occ_off, const uint32_t *__restrict__ row_of,
           const uint64_t *__restrict__ members, const uint32_t *__restrict__ read_len,
           uint32_t k, uint32_t stride, uint32_t nb, uint64_t n_occ,
           uint64_t *__restrict__ cand_cnt, const uint64_t *__restrict__ cand_end,
           uint32_t *__restrict__ overflow, Stage stage,
           uint32_t *__restrict__ big, uint32_t *__restrict__ n_big,
           uint64_t *__restrict__ rkey, unsigned long long *__restrict__ rbest,
           uint32_t *__restrict__ rshared, uint32_t *__restrict__ ridx)
{
    constexpr uint32_t kSlots = 1u << xs::kTableLg;
    __shared__ uint32_t tkey[kSlots], tcnt[kSlots];
    __shared__ unsigned long long tbest[kSlots];
    __shared__ uint32_t ovf, cursor;
    const uint32_t a = WRITE ? big[blockIdx.x] : blockIdx.x;
    const uint64_t q0 = occ_off[a], q1 = occ_off[a + 1];
    if (q0 == q1) {  // a holds no k-mer
        if (!WRITE && threadIdx.x == 0) cand_cnt[a] = 0;
        return;
    }
    for (uint32_t h = threadIdx.x; h < kSlots; h += blockDim.x) {
        tkey[h] = xs::kEmpty;
        tcnt[h] = 0;
        tbest[h] = ~0ull;
    }
    if (threadIdx.x == 0) {
        ovf = 0;
        cursor = 0;
    }
    __syncthreads();
    const xs::RowTable t{tkey, tcnt, tbest, xs::kTableLg};
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const uint32_t half = lane >> 4, hl = lane & 15;
    for (uint64_t b0 = q0 + 32 * warp; b0 < q1; b0 += 32 * n_warps) {
        // a vote: other warps set the flag at any time, and the collectives
        // below need all lanes of this one
        if (__any_sync(0xFFFFFFFFu, *(volatile uint32_t *)&ovf)) break;
        const uint64_t q = b0 + lane;
        uint32_t own = q < q1 ? row_of[q] : kNone;
        uint64_t word = 0;
        if (own != kNone) {
            word = members[own];
            if (word & kLast) own = kNone;  // no read behind a in the column
        }
        const uint32_t pw = (uint32_t)word;  // position << 1 | forward
        unsigned todo = __ballot_sync(0xFFFFFFFFu, own != kNone);
        while (todo) {  // kCols positions per half warp at a time: their loads overlap
            uint32_t j[kCols], p[kCols];
            uint64_t m[kCols];
            bool more[kCols];
#pragma unroll
            for (int c = 0; c < kCols; ++c) {
                const int s0 = todo ? __ffs((int)todo) - 1 : -1;
                todo &= todo - 1;
                const int s1 = todo ? __ffs((int)todo) - 1 : -1;
                todo &= todo - 1;
                const int src = half ? s1 : s0;
                j[c] = __shfl_sync(0xFFFFFFFFu, own, src < 0 ? 0 : src) + 1 + hl;
                p[c] = __shfl_sync(0xFFFFFFFFu, pw, src < 0 ? 0 : src);
                more[c] = src >= 0;
                m[c] = more[c] && j[c] < n_occ ? members[j[c]] : 0ull;
            }
#pragma unroll
            for (int c = 0; c < kCols; ++c) {
                while (__any_sync(0xFFFFFFFFu, more[c])) {
                    const unsigned ends =
                        (__ballot_sync(0xFFFFFFFFu, more[c] && (m[c] & kLast)) >> (16 * half)) & 0xFFFFu;
                    // members up to the marked one; what follows is another column's
                    const bool in = more[c] && (!ends || hl <= (uint32_t)__ffs((int)ends) - 1u);
                    if (in && !xs::row_term(t, a, p[c] >> 1, (p[c] & 1u) != 0, m[c] & ~kLast, read_len, k))
                        ovf = 1;
                    more[c] = more[c] && !ends;
                    j[c] += 16;
                    m[c] = more[c] && j[c] < n_occ ? members[j[c]] : 0ull;
                }
            }
        }
    }
    __syncthreads();
    if (ovf) {
        if (!WRITE && threadIdx.x == 0) {
            cand_cnt[a] = 0;
            atomicOr(overflow, 1u);
        }
        return;
    }
    if (!WRITE) {
        uint32_t n = 0;
        for (uint32_t h = threadIdx.x; h < kSlots; h += blockDim.x) n += tkey[h] != xs::kEmpty;
        n = __reduce_add_sync(0xFFFFFFFFu, n);
        if (lane == 0) atomicAdd(&cursor, n);
        __syncthreads();
        const uint32_t total = cursor;
        if (threadIdx.x == 0) {
            cand_cnt[a] = total;
            if (total > kStage) big[atomicAdd(n_big, 1u)] = a;
        }
        if (total > kStage) return;  // the second pass writes this read
        __syncthreads();
        if (threadIdx.x == 0) cursor = 0;
        __syncthreads();
        const uint64_t base = (uint64_t)a * kStage;
        for (uint32_t h = threadIdx.x; h < kSlots; h += blockDim.x) {
            if (tkey[h] == xs::kEmpty) continue;
            const uint64_t i = base + atomicAdd(&cursor, 1u);
            stage.key[i] = tkey[h];
            stage.best[i] = tbest[h];
            stage.cnt[i] = tcnt[h];
        }
    } else {
        const uint64_t base = a ? cand_end[a - 1] : 0;
        for (uint32_t h = threadIdx.x; h < kSlots; h += blockDim.x) {
            if (tkey[h] == xs::kEmpty) continue;
            const uint64_t i = base + atomicAdd(&cursor, 1u);
            rkey[i] = ((uint64_t)a << nb) | tkey[h];
            rbest[i] = tbest[h];
            rshared[i] = tcnt[h];
            ridx[i] = (uint32_t)i;
        }
    }
}

// The staged partners of every read with at most kStage of them, to their
// records at cand_end[a-1] ...; a warp per read.
__global__ void __launch_bounds__(kThreads)
stage_out_kernel(const uint64_t *__restrict__ cand_cnt, const uint64_t *__restrict__ cand_end,
                 Stage stage, uint32_t n_reads, uint32_t nb, uint64_t *__restrict__ rkey,
                 unsigned long long *__restrict__ rbest, uint32_t *__restrict__ rshared,
                 uint32_t *__restrict__ ridx)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t a = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; a < n_reads;
         a += warps) {
        const uint64_t n = cand_cnt[a];
        if (n == 0 || n > kStage) continue;
        const uint64_t base = a ? cand_end[a - 1] : 0;
        for (uint32_t j = lane; j < n; j += 32) {
            const uint64_t s = a * kStage + j, i = base + j;
            rkey[i] = (a << nb) | stage.key[s];
            rbest[i] = stage.best[s];
            rshared[i] = stage.cnt[s];
            ridx[i] = (uint32_t)i;
        }
    }
}

__global__ void __launch_bounds__(kThreads)
row_out_kernel(const uint64_t *__restrict__ keys, const uint32_t *__restrict__ idx,
               const unsigned long long *__restrict__ best, const uint32_t *__restrict__ cnt,
               int n, uint32_t nb, uint32_t k, Pair *__restrict__ pairs,
               uint32_t *__restrict__ shared)
{
    const uint64_t mask = nb >= 32 ? 0xFFFFFFFFull : (1ull << nb) - 1;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const uint32_t j = idx[i];
        const uint64_t b = best[j];
        Pair p;
        p.a = (uint32_t)(keys[i] >> nb);
        p.b = (uint32_t)(keys[i] & mask) | ((b & 1u) ? xs::kPairRC : 0u);
        p.seed_a = (uint32_t)(b >> 32);
        p.seed_b = (uint32_t)(b & 0xFFFFFFFFu) >> 1;
        p.seed_len = k;
        pairs[i] = p;
        shared[i] = cnt[j];
    }
}

// ------------------------------------------------------------------ host

int grid_for(uint64_t n, int sm_count)
{
    const uint64_t blocks = (n + kThreads - 1) / kThreads;
    const uint64_t cap = (uint64_t)sm_count * 8;
    return (int)std::max<uint64_t>(1, std::min(blocks, cap));
}

// Stream-ordered device allocations of one call, released together.
struct Arena {
    cudaStream_t s;
    cudaMemPool_t pool;
    size_t budget, used = 0;
    std::vector<void *> held;
    int rc = XDROP_OK;
    std::string err;
    Arena(cudaStream_t st, cudaMemPool_t p, size_t b) : s(st), pool(p), budget(b) {}
    ~Arena()
    {
        for (void *p : held) cudaFreeAsync(p, s);
    }
    template <class T>
    bool get(T *&p, uint64_t count)
    {
        size_t bytes = std::max<size_t>((size_t)count * sizeof(T), 16);
        if (budget && used + bytes > budget) {
            err = "seed discovery tables exceed the device memory budget";
            rc = XDROP_ENOMEM;
            return false;
        }
        void *q = nullptr;
        const cudaError_t e = cudaMallocFromPoolAsync(&q, bytes, pool, s);
        if (e != cudaSuccess) {
            err = std::string("cudaMallocFromPoolAsync: ") + cudaGetErrorString(e);
            rc = e == cudaErrorMemoryAllocation ? XDROP_ENOMEM : XDROP_ECUDA;
            return false;
        }
        held.push_back(q);
        used += bytes;
        p = (T *)q;
        return true;
    }
    int cuda(cudaError_t e, const char *what)
    {
        if (e == cudaSuccess) return XDROP_OK;
        err = std::string(what) + ": " + cudaGetErrorString(e);
        return rc = XDROP_ECUDA;
    }
};

#define XS_GET(ptr, count) \
    if (!ar.get(ptr, (count))) return ar.rc
#define XS_CK(call)                                         \
    do {                                                    \
        if (ar.cuda((call), #call) != XDROP_OK) return ar.rc; \
    } while (0)

// Input and front-step tables shared by both products.
struct Front {
    const uint32_t *packed, *read_len;
    const uint64_t *read_off;
    uint32_t n_reads, k, stride, lo, hi, nb;
    int sm_count;
    uint64_t n_occ = 0, longest = 0;  // positions of all reads, of the longest
    uint64_t *occ_off = nullptr;
    const uint64_t *codes = nullptr;
    const uint32_t *occ = nullptr;
    uint64_t *spare8 = nullptr;  // the sort's other buffers: n_occ words of 8
    uint32_t *spare4 = nullptr;  // and of 4 bytes, free after it
    uint32_t *occ_rd = nullptr, *fwd_bits = nullptr;
    int *run_off = nullptr, *run_len = nullptr;
    int n_runs = 0;
};

template <class T>
int read_back(Arena &ar, T *h, const T *d)
{
    XS_CK(cudaMemcpyAsync(h, d, sizeof(T), cudaMemcpyDeviceToHost, ar.s));
    XS_CK(cudaStreamSynchronize(ar.s));
    return XDROP_OK;
}

int front(Arena &ar, Front &f, const std::vector<uint64_t> &occ_off)
{
    const int n = (int)f.n_occ;
    uint64_t *keys0, *keys1;
    uint32_t *occ0, *occ1;
    XS_GET(f.occ_off, f.n_reads + 1);
    XS_GET(keys0, f.n_occ);
    XS_GET(keys1, f.n_occ);
    XS_GET(occ0, f.n_occ);
    XS_GET(occ1, f.n_occ);
    XS_GET(f.occ_rd, f.n_occ);
    XS_GET(f.fwd_bits, (f.n_occ + 31) / 32);
    XS_CK(cudaMemcpyAsync(f.occ_off, occ_off.data(), (f.n_reads + 1) * sizeof(uint64_t),
                          cudaMemcpyHostToDevice, ar.s));
    kmer_kernel<<<grid_for(f.n_occ, f.sm_count), kThreads, 0, ar.s>>>(
        f.packed, f.read_off, f.occ_off, f.n_reads, f.n_occ, f.k, f.stride, keys0, occ0, f.occ_rd,
        f.fwd_bits);
    XS_CK(cudaGetLastError());
    // occurrences grouped by k-mer, stable: read, then position order
    cub::DoubleBuffer<uint64_t> dk(keys0, keys1);
    cub::DoubleBuffer<uint32_t> dv(occ0, occ1);
    char *tmp;
    size_t tmp_bytes = 0;
    XS_CK(cub::DeviceRadixSort::SortPairs(nullptr, tmp_bytes, dk, dv, n, 0, (int)(2 * f.k), ar.s));
    XS_GET(tmp, tmp_bytes);
    XS_CK(cub::DeviceRadixSort::SortPairs(tmp, tmp_bytes, dk, dv, n, 0, (int)(2 * f.k), ar.s));
    f.codes = dk.Current();
    f.occ = dv.Current();
    f.spare8 = dk.Alternate();
    f.spare4 = dv.Alternate();
    // runs of length >= 2 (a k-mer seen once pairs no reads)
    int *d_nruns;
    XS_GET(f.run_off, f.n_occ / 2 + 1);
    XS_GET(f.run_len, f.n_occ / 2 + 1);
    XS_GET(d_nruns, 1);
    size_t rle_bytes = 0;
    char *rle_tmp;
    XS_CK(cub::DeviceRunLengthEncode::NonTrivialRuns(nullptr, rle_bytes, f.codes, f.run_off,
                                                     f.run_len, d_nruns, n, ar.s));
    XS_GET(rle_tmp, rle_bytes);
    XS_CK(cub::DeviceRunLengthEncode::NonTrivialRuns(rle_tmp, rle_bytes, f.codes, f.run_off,
                                                     f.run_len, d_nruns, n, ar.s));
    return read_back(ar, &f.n_runs, d_nruns);
}

int copy_out(Arena &ar, const Pair *d_pairs, const uint32_t *d_shared, int n_cand,
             std::vector<Pair> &out_pairs, std::vector<uint32_t> &out_shared)
{
    out_pairs.resize(n_cand);
    out_shared.resize(n_cand);
    XS_CK(cudaMemcpyAsync(out_pairs.data(), d_pairs, (size_t)n_cand * sizeof(Pair),
                          cudaMemcpyDeviceToHost, ar.s));
    XS_CK(cudaMemcpyAsync(out_shared.data(), d_shared, (size_t)n_cand * 4, cudaMemcpyDeviceToHost,
                          ar.s));
    return XDROP_OK;
}

int sort_product(Arena &ar, const Front &f, std::vector<Pair> &out_pairs,
                 std::vector<uint32_t> &out_shared)
{
    const int n_runs = f.n_runs;
    // pairs per reliable run and their output slots
    uint64_t *npairs, *pair_end;
    XS_GET(npairs, n_runs);
    XS_GET(pair_end, n_runs);
    count_kernel<<<grid_for(n_runs, f.sm_count), kThreads, 0, ar.s>>>(
        f.occ, f.occ_rd, f.run_off, f.run_len, n_runs, f.lo, f.hi, npairs);
    XS_CK(cudaGetLastError());
    size_t scan_bytes = 0;
    char *scan_tmp;
    XS_CK(cub::DeviceScan::InclusiveSum(nullptr, scan_bytes, npairs, pair_end, n_runs, ar.s));
    XS_GET(scan_tmp, scan_bytes);
    XS_CK(cub::DeviceScan::InclusiveSum(scan_tmp, scan_bytes, npairs, pair_end, n_runs, ar.s));
    uint64_t n_ent = 0;
    if (int rc = read_back(ar, &n_ent, pair_end + (n_runs - 1))) return rc;
    if (n_ent == 0) return XDROP_OK;
    if (n_ent > kMaxItems) {
        ar.err = "more than 2^31 - 1 shared-k-mer entries; narrow the frequency window";
        return ar.rc = XDROP_ENOMEM;
    }
    // one entry per (read pair, shared reliable k-mer)
    uint64_t *ek0, *ek1;
    uint32_t *ei0, *ei1;
    xs::Cand *ent, *ent_sorted;
    XS_GET(ek0, n_ent);
    XS_GET(ek1, n_ent);
    XS_GET(ei0, n_ent);
    XS_GET(ei1, n_ent);
    XS_GET(ent, n_ent);
    XS_GET(ent_sorted, n_ent);
    emit_kernel<<<grid_for(n_runs, f.sm_count), kThreads, 0, ar.s>>>(
        f.codes, f.occ, f.occ_rd, f.fwd_bits, f.occ_off, f.read_len, f.run_off, f.run_len, pair_end,
        n_runs, f.k, f.stride, f.nb, ek0, ent, ei0);
    XS_CK(cudaGetLastError());
    // entries grouped by read pair, reduced to one candidate each
    const int ne = (int)n_ent;
    cub::DoubleBuffer<uint64_t> ek(ek0, ek1);
    cub::DoubleBuffer<uint32_t> ei(ei0, ei1);
    size_t sort_bytes = 0;
    char *sort_tmp;
    XS_CK(cub::DeviceRadixSort::SortPairs(nullptr, sort_bytes, ek, ei, ne, 0, (int)(2 * f.nb), ar.s));
    XS_GET(sort_tmp, sort_bytes);
    XS_CK(cub::DeviceRadixSort::SortPairs(sort_tmp, sort_bytes, ek, ei, ne, 0, (int)(2 * f.nb), ar.s));
    gather_kernel<<<grid_for(n_ent, f.sm_count), kThreads, 0, ar.s>>>(ent, ei.Current(), n_ent,
                                                                      ent_sorted);
    XS_CK(cudaGetLastError());
    uint64_t *uniq;
    xs::Cand *agg;
    int *d_ncand;
    XS_GET(uniq, n_ent);
    XS_GET(agg, n_ent);
    XS_GET(d_ncand, 1);
    size_t red_bytes = 0;
    char *red_tmp;
    XS_CK(cub::DeviceReduce::ReduceByKey(nullptr, red_bytes, ek.Current(), uniq, ent_sorted, agg,
                                         d_ncand, xs::CandMerge(), ne, ar.s));
    XS_GET(red_tmp, red_bytes);
    XS_CK(cub::DeviceReduce::ReduceByKey(red_tmp, red_bytes, ek.Current(), uniq, ent_sorted, agg,
                                         d_ncand, xs::CandMerge(), ne, ar.s));
    int n_cand = 0;
    if (int rc = read_back(ar, &n_cand, d_ncand)) return rc;
    if (n_cand <= 0) return XDROP_OK;
    Pair *d_pairs;
    uint32_t *d_shared;
    XS_GET(d_pairs, n_cand);
    XS_GET(d_shared, n_cand);
    out_kernel<<<grid_for(n_cand, f.sm_count), kThreads, 0, ar.s>>>(uniq, agg, n_cand, f.nb, f.k,
                                                                     d_pairs, d_shared);
    XS_CK(cudaGetLastError());
    return copy_out(ar, d_pairs, d_shared, n_cand, out_pairs, out_shared);
}

// *done = false when some read's table overflowed (nothing written).
int row_product(Arena &ar, const Front &f, std::vector<Pair> &out_pairs,
                std::vector<uint32_t> &out_shared, bool *done, uint64_t *nonzeros)
{
    *done = false;
    const int n_runs = f.n_runs, n_reads = (int)f.n_reads;
    // columns and row entries, in the buffers the sort no longer needs (a
    // column has at most as many members as its run has occurrences)
    uint64_t *members = f.spare8;
    uint32_t *row_of = f.spare4;
    struct Counts {
        unsigned long long nonzeros;
        uint32_t cursor, pad;
    } *counts, h_counts{};
    XS_GET(counts, 1);
    XS_CK(cudaMemsetAsync(counts, 0, sizeof(Counts), ar.s));
    XS_CK(cudaMemsetAsync(row_of, 0xFF, f.n_occ * sizeof(uint32_t), ar.s));
    column_kernel<<<grid_for(n_runs, f.sm_count), kThreads, 0, ar.s>>>(
        f.occ, f.occ_rd, f.fwd_bits, f.occ_off, f.run_off, f.run_len, n_runs, f.lo, f.hi, f.stride,
        members, row_of, &counts->cursor, &counts->nonzeros);
    XS_CK(cudaGetLastError());
    // each read's partners in one pass: counted, and staged when there are
    // at most kStage of them; reads with more are recomputed and written
    // by a second pass over those reads alone
    uint64_t *cand_cnt, *cand_end;
    uint32_t *flags, *big;  // flags[0]: table overflow, flags[1]: reads listed in big
    Stage stage;
    const uint64_t n_stage = (uint64_t)n_reads * kStage;
    if (!(ar.get(cand_cnt, n_reads) && ar.get(cand_end, n_reads) && ar.get(flags, 2) &&
          ar.get(big, n_reads) && ar.get(stage.key, n_stage) && ar.get(stage.best, n_stage) &&
          ar.get(stage.cnt, n_stage))) {
        // without a reliable k-mer there is nothing to accumulate (asked only
        // here: the answer costs a round trip)
        const int rc = ar.rc;
        if (rc != XDROP_ENOMEM) return rc;
        if (read_back(ar, &h_counts, counts)) return ar.rc;
        if (h_counts.nonzeros) return rc;
        ar.rc = XDROP_OK;
        *done = true;
        return XDROP_OK;
    }
    XS_CK(cudaMemsetAsync(flags, 0, 8, ar.s));
    const int threads = f.n_occ <= kShortMean * f.n_reads && f.longest <= kShortLongest
                            ? kShortRowThreads : kRowThreads;
    row_kernel<false><<<n_reads, threads, 0, ar.s>>>(
        f.occ_off, row_of, members, f.read_len, f.k, f.stride, f.nb, f.n_occ, cand_cnt, nullptr, flags,
        stage, big, flags + 1, nullptr, nullptr, nullptr, nullptr);
    XS_CK(cudaGetLastError());
    size_t bytes = 0;
    char *tmp;
    XS_CK(cub::DeviceScan::InclusiveSum(nullptr, bytes, cand_cnt, cand_end, n_reads, ar.s));
    XS_GET(tmp, bytes);
    XS_CK(cub::DeviceScan::InclusiveSum(tmp, bytes, cand_cnt, cand_end, n_reads, ar.s));
    uint32_t hflags[2] = {0, 0};
    uint64_t n_cand = 0;
    XS_CK(cudaMemcpyAsync(hflags, flags, 8, cudaMemcpyDeviceToHost, ar.s));
    XS_CK(cudaMemcpyAsync(&h_counts, counts, sizeof(Counts), cudaMemcpyDeviceToHost, ar.s));
    if (int rc = read_back(ar, &n_cand, cand_end + (n_reads - 1))) return rc;
    *nonzeros = h_counts.nonzeros;
    const uint32_t ovf = hflags[0], n_big = hflags[1];
    if (ovf) return XDROP_OK;  // not done: the sort-based product takes over
    *done = true;
    if (n_cand == 0) return XDROP_OK;
    if (n_cand > kMaxItems) {
        ar.err = "more than 2^31 - 1 candidate pairs";
        return ar.rc = XDROP_ENOMEM;
    }
    uint64_t *rk0, *rk1;
    uint32_t *ri0, *ri1, *rshared;
    unsigned long long *rbest;
    XS_GET(rk0, n_cand);
    XS_GET(rk1, n_cand);
    XS_GET(ri0, n_cand);
    XS_GET(ri1, n_cand);
    XS_GET(rbest, n_cand);
    XS_GET(rshared, n_cand);
    stage_out_kernel<<<grid_for((uint64_t)n_reads * 32, f.sm_count), kThreads, 0, ar.s>>>(
        cand_cnt, cand_end, stage, (uint32_t)n_reads, f.nb, rk0, rbest, rshared, ri0);
    XS_CK(cudaGetLastError());
    if (n_big) {
        row_kernel<true><<<n_big, threads, 0, ar.s>>>(
            f.occ_off, row_of, members, f.read_len, f.k, f.stride, f.nb, f.n_occ, nullptr, cand_end,
            nullptr, stage, big, nullptr, rk0, rbest, rshared, ri0);
        XS_CK(cudaGetLastError());
    }
    // candidates in (a, b) order
    const int nc = (int)n_cand;
    cub::DoubleBuffer<uint64_t> rk(rk0, rk1);
    cub::DoubleBuffer<uint32_t> ri(ri0, ri1);
    bytes = 0;
    XS_CK(cub::DeviceRadixSort::SortPairs(nullptr, bytes, rk, ri, nc, 0, (int)(2 * f.nb), ar.s));
    XS_GET(tmp, bytes);
    XS_CK(cub::DeviceRadixSort::SortPairs(tmp, bytes, rk, ri, nc, 0, (int)(2 * f.nb), ar.s));
    Pair *d_pairs;
    uint32_t *d_shared;
    XS_GET(d_pairs, n_cand);
    XS_GET(d_shared, n_cand);
    row_out_kernel<<<grid_for(n_cand, f.sm_count), kThreads, 0, ar.s>>>(
        rk.Current(), ri.Current(), rbest, rshared, nc, f.nb, f.k, d_pairs, d_shared);
    XS_CK(cudaGetLastError());
    return copy_out(ar, d_pairs, d_shared, nc, out_pairs, out_shared);
}

}  // namespace

int find_candidates(cudaStream_t st, cudaMemPool_t pool, int sm_count, size_t budget, const uint32_t *packed,
                    const uint64_t *read_off, const uint32_t *read_len, uint32_t n_reads,
                    const uint32_t *h_len, uint32_t k, uint32_t stride, uint32_t lo, uint32_t hi,
                    uint32_t flags, std::vector<Pair> &out_pairs,
                    std::vector<uint32_t> &out_shared, SeedStats &stats, std::string &err)
{
    out_pairs.clear();
    out_shared.clear();
    stats = SeedStats{};
    std::vector<uint64_t> occ_off(n_reads + 1, 0);
    for (uint32_t r = 0; r < n_reads; ++r)
        occ_off[r + 1] = occ_off[r] + (h_len[r] >= k ? (h_len[r] - k) / stride + 1 : 0);
    stats.occurrences = occ_off[n_reads];
    if (stats.occurrences < 2) return XDROP_OK;
    if (stats.occurrences > kMaxItems) {
        err = "more than 2^31 - 1 k-mer occurrences; raise the stride";
        return XDROP_ENOMEM;
    }
    cudaEvent_t ev[2] = {nullptr, nullptr};
    if (cudaEventCreate(&ev[0]) != cudaSuccess || cudaEventCreate(&ev[1]) != cudaSuccess) {
        for (cudaEvent_t e : ev)
            if (e) cudaEventDestroy(e);
        err = "cudaEventCreate failed";
        return XDROP_ECUDA;
    }
    int rc = XDROP_OK;
    {
        Arena ar(st, pool, budget);
        Front f;
        f.packed = packed;
        f.read_len = read_len;
        f.read_off = read_off;
        f.n_reads = n_reads;
        f.k = k;
        f.stride = stride;
        f.lo = lo;
        f.hi = hi;
        f.nb = xs::id_bits(n_reads);
        f.sm_count = sm_count;
        f.n_occ = stats.occurrences;
        for (uint32_t r = 0; r < n_reads; ++r)
            f.longest = std::max(f.longest, occ_off[r + 1] - occ_off[r]);
        rc = ar.cuda(cudaEventRecord(ev[0], st), "cudaEventRecord");
        if (!rc) rc = front(ar, f, occ_off);
        stats.runs = rc ? 0 : (uint64_t)std::max(f.n_runs, 0);
        bool done = rc != XDROP_OK || f.n_runs <= 0;
        const bool rows_ok = n_reads < kMaxItems;  // one block per read
        if (!done && !(flags & XDROP_SEEDS_SORT) && rows_ok) {
            rc = row_product(ar, f, out_pairs, out_shared, &done, &stats.nonzeros);
            if (done && !rc) stats.product = XDROP_SEEDS_ROWWISE;
        }
        if (!done && !rc) {
            rc = sort_product(ar, f, out_pairs, out_shared);
            if (!rc) stats.product = XDROP_SEEDS_SORT;
        }
        if (!rc) rc = ar.cuda(cudaEventRecord(ev[1], st), "cudaEventRecord");
        if (!rc) rc = ar.cuda(cudaStreamSynchronize(st), "cudaStreamSynchronize");
        if (!rc) {
            float ms = 0.f;
            rc = ar.cuda(cudaEventElapsedTime(&ms, ev[0], ev[1]), "cudaEventElapsedTime");
            stats.ms = ms;
        }
        if (rc) err = ar.err;
    }
    cudaEventDestroy(ev[0]);
    cudaEventDestroy(ev[1]);
    if (rc) {
        out_pairs.clear();
        out_shared.clear();
        return rc;
    }
    stats.candidates = out_pairs.size();
    return XDROP_OK;
}

#undef XS_GET
#undef XS_CK

}  // namespace xd
