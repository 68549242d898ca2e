// Types and host/device helpers shared by the kernels and the host
// runtime (no kernels here).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace xd {

// Pruned cell.  Every threshold T - x is >= -x > -2^25 > NEG, and any
// live or pruned value times 16 plus 15 still fits in int32 (the packed
// best-cell key of the lockstep kernels).
constexpr int32_t NEG = -(1 << 26);
constexpr uint32_t FULL = 0xffffffffu;

struct Pair {
    uint32_t a, b, seed_a, seed_b, seed_len;
};

struct Scoring {
    int32_t match, mismatch, gap, x;
};

// Everything a kernel needs to decode and write one task.  Task t is the
// left (t even) or right (t odd) extension of pair t/2.
// Top bit of a pair's b: align against the reverse complement of read b
// (XDROP_PAIR_RC).  The library stores the reverse complement of every
// read after the reads themselves, rc_off bases further on, and an RC pair
// reads its b there; the band kernels never see the flag.
constexpr uint32_t kPairRC = 0x80000000u;

struct Job {
    const uint32_t *packed;  // the reads, then (rc_off > 0) their reverse complements
    int64_t n_words;         // words of the whole buffer
    int64_t rc_off;          // bases from a read to its reverse complement; 0 = none stored
    const uint64_t *read_off;
    const uint32_t *read_len;
    uint32_t n_reads;
    const Pair *pairs;
    uint64_t n_pairs;
    Scoring sc;
    int32_t *out;    // 7 int32 per pair (xdrop_result)
    int64_t *cells;  // per task cell count (counting launches only)
    // Serving requests only: finished / spilled task counters, the list of
    // spilled task ids, and the tag written to the host when all finished.
    uint32_t *ctr;
    uint32_t *spill_list;
    uint32_t tag;
};

// Length bins: four an octave of min(m, n), the last one for 2^28 and more.
constexpr int NBINS = 128;

__host__ __device__ inline int length_bin(uint32_t w)
{
    if (w < 4) return (int)w;
    int lg = 0;
    for (uint32_t v = w; v > 1; v >>= 1) ++lg;
    return 4 * lg + (int)((w >> (lg - 2)) & 3u);
}

// Diagonals of the longest extension of a bin (about).
__host__ __device__ inline double bin_diagonals(int b)
{
    if (b < 8) return 2.0 * (b < 4 ? b : 3);
    return 2.0 * (double)((uint64_t)(5 + b % 4) << (b / 4 - 2));
}

// Overflow hand-off between tiers.
struct Spill {
    uint32_t *list;   // task ids
    uint32_t *count;  // number of ids in list
    uint32_t *longest = nullptr;  // unbounded tier: the largest m of them
};

// Device words of a batched launch whose first blocks give a warp to single
// extensions (xd_tiles_packed.cu): the longest tasks of the order, then the
// first tier's overflow while the first tier still runs.
struct WarpRole {
    uint32_t *n_long;    // tasks at the head of the order for single warps
    uint32_t *n_blocks;  // blocks that start with them
    uint32_t *long_ctr;  // next of those tasks
    uint32_t *ready;     // overflow entries written and not claimed (xd_claim.cuh)
    uint32_t *taken;     // overflow entries taken
    uint32_t *done;      // first-tier warps that found no more tasks
    uint32_t *grown;     // longest tasks that outgrew a warp's first window
    uint32_t *grown_end; // their ids, stored downwards from here (null: not noted)
    uint32_t *err;       // set when an overflow entry never appeared
    Spill wide;          // tasks for the unbounded tier
    uint32_t few;        // up to this many tasks all go to single warps
};
constexpr int32_t kBriefDiagonals = 2048;  // overflow up to this long goes to a second group tier
constexpr uint32_t kNoTask = 0xFFFFFFFFu;  // overflow entry not written yet

// One base stream c_k (k >= 1): c_k is base s0 + dir*(k-1) of the packed
// buffer.
struct Seq {
    const uint32_t *pk;
    int64_t nw;
    int64_t s0;
    int dir;
};

struct Ext {
    Seq A, B;
    int32_t m, n;
    uint32_t pair;
    int side;       // 0 left, 1 right
    uint32_t sa, sb, L;
    bool ok;
};

// ---------------------------------------------------------------------------
// Limits (also enforced on the host for host submits).
// ---------------------------------------------------------------------------
constexpr int64_t LEN_LIMIT = (int64_t)1 << 28;    // read length
constexpr int64_t SCORE_LIMIT = (int64_t)1 << 25;  // |score| * (len_a + len_b), and x

__host__ __device__ inline int32_t max_abs_score(const Scoring &s)
{
    int32_t a = s.match < 0 ? -s.match : s.match;
    int32_t b = s.mismatch < 0 ? -s.mismatch : s.mismatch;
    int32_t c = s.gap < 0 ? -s.gap : s.gap;
    int32_t m = a > b ? a : b;
    return m > c ? m : c;
}

// The scoring with a mismatch worth no less than two gaps: the same scores,
// positions and live cells.  If H(i-1,j-1) + 2 gap reaches the threshold of
// diagonal d, then H(i-1,j-1) + gap, larger, reaches the one of d-1, which is
// no larger: cell (i-1,j), inside the rectangle like (i,j), is live with at
// least that value and offers (i,j) at least H(i-1,j-1) + 2 gap.  So a
// mismatch below two gaps never decides a live cell, and raising it to two
// gaps offers nothing that is not offered already.
__host__ __device__ inline Scoring effective(Scoring s)
{
    if (s.mismatch < 2 * s.gap) s.mismatch = 2 * s.gap;
    return s;
}

// n_words: words of the reads themselves (without reverse complements);
// rc_ok: whether a pair may ask for the reverse strand of b.
__host__ __device__ inline bool pair_ok(const Pair &p, uint32_t n_reads,
                                        const uint32_t *read_len,
                                        const uint64_t *read_off,
                                        int64_t n_words, const Scoring &s, bool rc_ok)
{
    const uint32_t b = p.b & ~kPairRC;
    if ((p.b & kPairRC) && !rc_ok) return false;
    if (p.a >= n_reads || b >= n_reads) return false;
    uint64_t la = read_len[p.a], lb = read_len[b];
    if ((int64_t)la >= LEN_LIMIT || (int64_t)lb >= LEN_LIMIT) return false;
    if ((uint64_t)p.seed_a + p.seed_len > la) return false;
    if ((uint64_t)p.seed_b + p.seed_len > lb) return false;
    if ((int64_t)(la + lb) * max_abs_score(s) >= SCORE_LIMIT) return false;
    uint64_t oa = read_off[p.a], ob = read_off[b];
    if ((oa & 15) || (ob & 15)) return false;
    if ((int64_t)((oa + la + 15) / 16) > n_words) return false;
    if ((int64_t)((ob + lb + 15) / 16) > n_words) return false;
    return true;
}

__host__ __device__ inline bool job_pair_ok(const Job &J, const Pair &p)
{
    return pair_ok(p, J.n_reads, J.read_len, J.read_off, J.rc_off ? J.rc_off / 16 : J.n_words,
                   J.sc, J.rc_off > 0);
}

__device__ __forceinline__ Ext decode(const Job &J, uint32_t task)
{
    Ext e;
    e.pair = task >> 1;
    e.side = (int)(task & 1u);
    Pair p = J.pairs[e.pair];
    e.ok = job_pair_ok(J, p);
    e.sa = p.seed_a;
    e.sb = p.seed_b;
    e.L = p.seed_len;
    e.A.pk = e.B.pk = J.packed;
    e.A.nw = e.B.nw = J.n_words;
    e.m = e.n = 0;
    e.A.s0 = e.B.s0 = 0;
    e.A.dir = e.B.dir = 1;
    if (!e.ok) return e;
    const uint32_t b = p.b & ~kPairRC;
    int64_t oa = (int64_t)J.read_off[p.a];
    int64_t ob = (int64_t)J.read_off[b] + ((p.b & kPairRC) ? J.rc_off : 0);
    int64_t la = J.read_len[p.a], lb = J.read_len[b];
    if (e.side) {  // right: c_k = X[seed + L + k - 1]
        e.m = (int32_t)(la - p.seed_a - p.seed_len);
        e.n = (int32_t)(lb - p.seed_b - p.seed_len);
        e.A.s0 = oa + p.seed_a + p.seed_len;
        e.B.s0 = ob + p.seed_b + p.seed_len;
        e.A.dir = e.B.dir = 1;
    } else {       // left: c_k = X[seed - k]
        e.m = (int32_t)p.seed_a;
        e.n = (int32_t)p.seed_b;
        e.A.s0 = oa + (int64_t)p.seed_a - 1;
        e.B.s0 = ob + (int64_t)p.seed_b - 1;
        e.A.dir = e.B.dir = -1;
    }
    return e;
}

__device__ __forceinline__ void write_result(const Job &J, const Ext &e,
                                             int32_t score, int32_t bi,
                                             int32_t bj)
{
    int32_t *o = J.out + (size_t)e.pair * 7;
    if (e.side) {
        o[3] = score;
        o[4] = (int32_t)(e.sa + e.L) + bi;
        o[5] = (int32_t)(e.sb + e.L) + bj;
    } else {
        o[0] = score;
        o[1] = (int32_t)e.sa - bi;
        o[2] = (int32_t)e.sb - bj;
    }
}

// Hands a task on to the unbounded tier (one thread).
__device__ __forceinline__ void hand_on_wide(const Spill &wide, uint32_t task, int32_t m)
{
    if (wide.longest) atomicMax(wide.longest, (uint32_t)m);
    wide.list[atomicAdd(wide.count, 1u)] = task;
}

// Status of a pair of a device submit: zero scores for a pair that fails
// the limits.
__device__ __forceinline__ void write_status(const Job &J, uint64_t pair, bool ok, uint32_t *n_bad)
{
    int32_t *o = J.out + pair * 7;
    if (!ok) {
        for (int k = 0; k < 6; ++k) o[k] = 0;
        atomicAdd(n_bad, 1u);
    }
    o[6] = ok ? 0 : 1;
}

}  // namespace xd
