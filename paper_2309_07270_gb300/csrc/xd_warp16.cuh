// One extension per warp, tuned for the latency of a diagonal.
//
// A batch ends with its longest extension, small batches (and the extensions
// that outgrow a narrower first tier) are nothing but a few long chains of
// anti-diagonals, and there the time of one diagonal counts, not the cells
// per second.  This is the packed tile of xd_lockstep16.cuh in its relative
// frame with 32 lanes of 4 slots (window 128), rearranged for one extension:
//   - Match flags for 8 pairs of diagonals at once.  A slot keeps its
//     diagonal offset, so its bases on successive pairs are successive bases
//     of both reads: one XOR of two 16-base words compares a slot with 8
//     pairs' bases (xd_lockstep16.cuh compares a diagonal's slots instead).
//     Bases past the read ends are cleared from the flags there, so
//     no diagonal is special near the rectangle's ends.
//   - Four pairs of diagonals between two looks at anything else.  Cells move
//     by at most one slot per pair, so while the end lanes (4 or 8 slots each) are
//     dead before the block, nothing can leave the window in it.  One ballot
//     of the live lanes then says whether the extension is over (the last two
//     diagonals are dead), and whether, and by how many whole lanes, the
//     window must move: a move is one shuffle per register.
//   - One key for the whole warp: KS = W and the window slot (7 or 8 bits) in
//     each half, so the maximum over the warp of the larger half needs no lane
//     bits, and the bits below it need no clearing.
// The chain of a diagonal is then: maximum of r over the warp (a redux), the
// rise of T, the threshold step, the prune of the next diagonal; and beside
// it the shuffle of the end register.  Because the keys are taken before the
// prune (dp16r), two diagonals' chains overlap.
//
// Measured, one extension per warp scheduler: a diagonal takes 57 ns (200 pairs
// of 2-4 kb reads: 0.41 ms of kernels, 0.44 ms a call) against 81 ns for the
// same window in lockstep16_loop's order and about 200 ns before (1.59 ms a
// call on the 16x8 tile).  As the tier behind a 2x32 first tier (29x, x = 50,
// 3,582 extensions) it takes 2.5 ms where the 32-bit window of 128 slots took 8.2.
#pragma once
#include <stdint.h>

#include "xd_lockstep16.cuh"

namespace xd {

// Scorings of the warp tile of R registers per lane (window W = 64 R): values
// stay below 2^15 in units of W, and a pruned half cannot sink past the
// signed range within a block (8 diagonals, and two steps at once).
template <int R>
__host__ __device__ inline bool warp16_ok(const Scoring &sc)
{
    constexpr int W = 64 * R;
    return packed16_ok(sc) && (sc.match - sc.gap) * W <= 12 * 128 &&
           (sc.x + 2 * sc.match - 2 * sc.gap + 1) * W <= 0x8000;
}

namespace p16 {

// State of one warp's extension between blocks (everything but E and O is
// the same in every lane).
template <int R>
struct Warp16 {
    uint32_t E[R], O[R];   // even and odd diagonals: slots t (low half) and t + R
    uint32_t dA, dB;       // threshold steps d-2 -> d-1 and d-1 -> d, both halves
    int32_t sA, sB, T;
    int32_t bkey, bi0, bd; // best cell: warp maximum, window base i, diagonal
};

template <int R>
struct Warp16Const {
    uint32_t k[4], c[4], mi2;  // substitution of pair p of a block (RelSubst)
    uint32_t idx[R];           // window slot part of the keys
    uint32_t ngp;
    int32_t ng, x;
    bool first, last;          // this lane is the first, the last of the warp
};

template <int R, bool ODD, bool ADD>
__device__ __forceinline__ void warp16_diag(Warp16<R> &s, const Warp16Const<R> &q,
                                            const uint32_t (&G)[R], int p, int32_t d, int32_t i0)
{
    constexpr uint32_t KS = 64 * R;
    constexpr int VS = 16 + (R == 2 ? 7 : 8);  // value shift of the maximum
    uint32_t(&V)[R] = ODD ? s.O : s.E;
    const uint32_t(&P)[R] = ODD ? s.E : s.O;
    uint32_t U[R];
#pragma unroll
    for (int t = 0; t < R; ++t) U[t] = P[t] + s.dA;
    uint32_t edge = ODD ? __shfl_down_sync(FULL, U[0], 1) : __shfl_up_sync(FULL, U[R - 1], 1);
    if (ODD ? q.last : q.first) edge = kDead2;
    const uint32_t nstep = 0x00010000u - (s.dA + s.dB);
    uint32_t key[R];
#pragma unroll
    for (int t = 0; t < R; ++t) {
        const uint32_t sh = ODD ? (t + 1 < R ? U[t + 1] : prmt(U[0], edge, 0x5432))
                                : (t > 0 ? U[t - 1] : prmt(edge, U[R - 1], 0x5432));
        const uint32_t w = (G[t] & (0x00010001u << (2 * p + 1))) | q.c[p];
        uint32_t cand = w * q.k[p] + V[t];
        if (ADD) cand += q.mi2;
        const uint32_t r = __vimax3_s16x2(cand, U[t], sh);
        V[t] = __viaddmin_u16x2(r, nstep, kDead2);
        key[t] = r + q.idx[t];
    }
    const uint32_t kk = tree_max2s<R>(key);
    // the larger half on top; what lies below it never decides (one slot per key)
    const int32_t M = __reduce_max_sync(FULL, max((int32_t)kk, (int32_t)(kk << 16)));
    const int32_t rise = max((M >> VS) - (s.sA + s.sB) - q.x, 0);
    s.dA = s.dB;
    s.dB = (uint32_t)rise * (KS * 0x10001u) + q.ngp;
    s.sA = s.sB;
    s.sB = rise + q.ng;
    s.T += rise;
    if (rise > 0) {
        s.bkey = M;
        s.bi0 = i0;
        s.bd = d;
    }
}

// Four pairs of diagonals after the even diagonal d, window base i0 there.
template <int R, bool ADD>
__device__ __forceinline__ void warp16_block(Warp16<R> &s, const Warp16Const<R> &q,
                                             const uint32_t (&Go)[R], const uint32_t (&Ge)[R],
                                             int32_t d, int32_t i0)
{
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        warp16_diag<R, true, ADD>(s, q, Go, p, d + 2 * p + 1, i0 + p + 1);
        warp16_diag<R, false, ADD>(s, q, Ge, p, d + 2 * p + 2, i0 + p + 1);
    }
}

}  // namespace p16

// Extends one task with the whole warp (all arguments warp-uniform, the
// scoring passes warp16_ok<R>).  Returns 0 when done, 1 when the band outgrew
// the window.
template <int R>
__device__ __forceinline__ int extend_warp16(const Ext &e, const Scoring sc, int lane,
                                             int32_t &best, int32_t &best_i, int32_t &best_j)
{
    using namespace p16;
    constexpr int S = 2 * R, W = 32 * S;
    constexpr uint32_t KS = W;
    static_assert(S == 4 || S == 8, "a lane's slots and 8 pairs fit a 16-base word");
    const int32_t m = e.m, n = e.n, mn = m + n;
    const int dir = e.A.dir;
    const uint32_t *pk = e.A.pk;
    const int32_t last = (int32_t)e.A.nw - 1;
    const int32_t aw0 = (int32_t)(e.A.s0 >> 4), ab0 = (int32_t)(e.A.s0 & 15);
    const int32_t bw0 = (int32_t)(e.B.s0 >> 4), bb0 = (int32_t)(e.B.s0 & 15);

    Warp16Const<R> q;
    q.ng = -sc.gap;
    q.x = sc.x;
    q.ngp = (uint32_t)q.ng * (KS * 0x10001u);
    q.first = lane == 0;
    q.last = lane == 31;
    const int32_t mm = sc.mismatch + 2 * q.ng, bonus = sc.match - sc.mismatch;
    const bool folds = subst_folds(sc);
    q.mi2 = folds ? 0u : pack2(mm * (int32_t)KS);
    const uint32_t c = folds ? (uint32_t)(2 * mm / bonus) * 0x10001u : 0u;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        q.k[p] = (uint32_t)bonus * KS >> (1 + 2 * p);
        q.c[p] = c << (2 * p);
    }
#pragma unroll
    for (int t = 0; t < R; ++t)
        q.idx[t] = (uint32_t)(W - 1 - S * lane - t) | ((uint32_t)(W - 1 - S * lane - t - R) << 16);

    Warp16<R> s;
    // origin (H = 0, x above the threshold) at window slot W/2
#pragma unroll
    for (int t = 0; t < R; ++t) s.E[t] = s.O[t] = kDead2;
    if (lane == 16) s.E[0] = (uint32_t)sc.x * KS | (kDead2 & 0xFFFF0000u);
    s.dA = s.dB = q.ngp;
    s.sA = s.sB = q.ng;
    s.T = 0;
    s.bkey = s.bi0 = s.bd = 0;
    int32_t d = 0, i0 = -(W / 2), j0 = W / 2;  // window slot 0 on the even diagonal d
    uint32_t ra0 = 0, ra1 = 0, rb0 = 0, rb1 = 0;  // raw words of the next flags
    bool ready = false, second = false;
    uint32_t Go[R], Ge[R];

    auto raw = [&](int32_t ia, int32_t jb) {
        const int32_t wa = aw0 + ((ab0 + (dir > 0 ? ia : -ia - 15)) >> 4);
        const int32_t wb = bw0 + ((bb0 + (dir > 0 ? jb - S : S - 15 - jb)) >> 4);
        ra0 = __ldg(pk + min(max(wa, 0), last));
        ra1 = __ldg(pk + min(max(wa + 1, 0), last));
        rb0 = __ldg(pk + min(max(wb, 0), last));
        rb1 = __ldg(pk + min(max(wb + 1, 0), last));
    };
    for (;;) {
        const int32_t il = i0 + S * lane, jl = j0 - S * lane;
        // a window slot can leave the rectangle within the next 8 pairs
        const bool ends = i0 + W + 8 > m || j0 + 9 > n;
        if (!second) {
            // flags of the next 8 pairs: field u of A is a[il + 1 + u], of B
            // b[jl - (S-1) + u]; slot t meets a[il+1+t+u], b[jl-t+u] on odd
            // diagonals and b[jl+1-t+u] on even ones
            if (!ready) raw(il, jl);
            const uint32_t sa = 2u * (uint32_t)((ab0 + (dir > 0 ? il : -il - 15)) & 15);
            const uint32_t sb = 2u * (uint32_t)((bb0 + (dir > 0 ? jl - S : S - 15 - jl)) & 15);
            uint32_t A = __funnelshift_r(ra0, ra1, sa), B = __funnelshift_r(rb0, rb1, sb);
            if (dir < 0) {
                A = rev16(A);
                B = rev16(B);
            }
            uint32_t fo[S], fe[S];
#pragma unroll
            for (int t = 0; t < S; ++t) {
                const uint32_t xo = (A >> (2 * t)) ^ (B >> (2 * (S - 1 - t)));
                const uint32_t xe = (A >> (2 * t)) ^ (B >> (2 * (S - t)));
                fo[t] = ~(xo | (xo << 1));
                fe[t] = ~(xe | (xe << 1));
                if (ends) {  // no match outside the rectangle (xd_lockstep16.cuh)
                    const int32_t ua = m - il - 1 - t, ub = n - jl + t;
                    fo[t] &= flag_range(0, min(ua, ub));
                    fe[t] &= flag_range(0, min(ua, ub - 1));
                }
            }
#pragma unroll
            for (int t = 0; t < R; ++t) {
                Go[t] = prmt(fo[t], fo[t + R], 0x5410);
                Ge[t] = prmt(fe[t], fe[t + R], 0x5410);
            }
            raw(il + 8, jl + 8);
            ready = true;
        } else {
#pragma unroll
            for (int t = 0; t < R; ++t) {
                Go[t] >>= 8;
                Ge[t] >>= 8;
            }
        }
        if (folds) warp16_block<R, false>(s, q, Go, Ge, d, i0);
        else warp16_block<R, true>(s, q, Go, Ge, d, i0);
        d += 8;
        i0 += 4;
        j0 += 4;
        second = !second;
        if (ends) {  // end what lives outside the rectangle
            const int32_t lo = jl + 4 - n, hi = m - il - 4;
#pragma unroll
            for (int t = 0; t < R; ++t) {
                s.E[t] = keep_range<R>(s.E[t], t, lo, hi);
                s.O[t] = keep_range<R>(s.O[t], t, lo - 1, hi);
            }
        }
        uint32_t dead = s.E[0] & s.O[0];
#pragma unroll
        for (int t = 1; t < R; ++t) dead &= s.E[t] & s.O[t];
        const unsigned live = __ballot_sync(FULL, (~dead & 0x80008000u) != 0u);
        if (live == 0u || d >= mn) break;
#pragma unroll
        for (int t = 0; t < R; ++t) {  // lift the pruned slots back up
            s.E[t] = __vmaxs2(s.E[t], kDead2);
            s.O[t] = __vmaxs2(s.O[t], kDead2);
        }
        if (live & 0x80000001u) {
            // move the window by whole lanes, the free ones shared between its ends
            const int lo = __ffs((int)live) - 1, hi = __clz((int)live);
            if (lo + hi < 2) return 1;
            const int by = (lo - hi) / 2, src = lane + by;
            const bool in = src >= 0 && src < 32;
#pragma unroll
            for (int t = 0; t < R; ++t) {
                const uint32_t ve = __shfl_sync(FULL, s.E[t], src & 31);
                const uint32_t vo = __shfl_sync(FULL, s.O[t], src & 31);
                s.E[t] = in ? ve : kDead2;
                s.O[t] = in ? vo : kDead2;
            }
            i0 += S * by;
            j0 -= S * by;
            ready = second = false;
        }
    }
    best = s.T;
    best_i = best_j = 0;
    if (s.bd > 0) {
        best_i = s.bi0 + (W - 1 - ((s.bkey >> 16) & (W - 1)));
        best_j = s.bd - best_i;
    }
    return 0;
}

// Words of the longest buffer for extend_warp: extend_warp16 counts words in
// 32 bits, and an extension's last loads lie up to 2^21 words and a window
// behind its first base.
constexpr int64_t kWarp16Words = INT32_MAX - (1 << 22);

// Task source of lockstep16_loop for one extension and the whole warp.
struct OneSrc {
    static constexpr bool kCanAbort = false;
    static constexpr int kWaitPairs = 1;
    const Ext &e;
    const Scoring &s;
    bool fresh = true;
    int32_t status = 1, best = 0, bi = 0, bj = 0;  // lane 0
    __device__ __forceinline__ int fetch_warp(unsigned, int, int, unsigned, bool, uint32_t &,
                                              const Job *&)
    {
        const bool first = fresh;
        fresh = false;
        return first ? 1 : -1;
    }
    __device__ __forceinline__ void idle() {}
    __device__ __forceinline__ bool aborted() const { return false; }
    __device__ __forceinline__ Ext open(const Job *, uint32_t, Scoring &sc)
    {
        sc = s;
        return e;
    }
    __device__ __forceinline__ void retire(const Job *, uint32_t, bool overflow, int32_t T, int32_t i,
                                           int32_t j)
    {
        status = overflow;
        best = T;
        bi = i;
        bj = j;
    }
};

// extend_warp16<2>'s window for the packed scorings beyond warp16_ok: the group
// loop on 32 lanes of 4 slots, whose keys take 16 units where a window's take
// 128 (81 ns a diagonal; the 32-bit window about 200).  Out of line and on
// copies, for the callers' registers.
struct WarpResult { int32_t status, best, bi, bj; };
static __device__ __noinline__ WarpResult extend_lockstep16(const Ext &e, const Scoring &sc)
{
    OneSrc src{e, sc};
    uint32_t one;
    asm volatile("mov.u32 %0, 1;" : "=r"(one));
    lockstep16_loop<32, 2>(src, e.A.pk, e.A.nw, one);
    return WarpResult{__shfl_sync(FULL, src.status, 0), __shfl_sync(FULL, src.best, 0),
                      __shfl_sync(FULL, src.bi, 0), __shfl_sync(FULL, src.bj, 0)};
}

// Extends one task with the whole warp on windows of 128 slots (packed if the
// scoring fits, else 32-bit), 256 (packed scorings only) and 512 slots
// (32-bit), from the first that is wider than `from` slots.  Returns how many
// of them the band outgrew, or -1 for all.  With ANY every 16-bit scoring takes
// packed cells in the first, else only those of warp16_ok.
template <bool ANY>
__device__ __forceinline__ int extend_warp(const Ext &e, const Scoring &s, int from, int lane,
                                           int32_t &best, int32_t &bi, int32_t &bj)
{
    const Scoring sc = effective(s);
    int64_t cells;
    int grown = 0;
    if (from < 128) {
        int st;
        if (warp16_ok<2>(sc)) {
            st = extend_warp16<2>(e, sc, lane, best, bi, bj);
        } else if (ANY && packed16_ok(sc)) {
            const Ext ec = e;
            const Scoring scc = sc;
            const WarpResult r = extend_lockstep16(ec, scc);
            st = r.status;
            best = r.best;
            bi = r.bi;
            bj = r.bj;
        } else {
            st = extend_window<32, 4, false>(e, sc, lane, 0, best, bi, bj, cells);
        }
        if (!st) return 0;
        ++grown;
    }
    if (warp16_ok<4>(sc)) {
        if (!extend_warp16<4>(e, sc, lane, best, bi, bj)) return grown;
        ++grown;
    }
    return extend_window<32, 16, false>(e, sc, lane, 0, best, bi, bj, cells) ? -1 : grown;
}

constexpr int kWarpThreads = 128;  // per block of a kernel that runs it

}  // namespace xd
