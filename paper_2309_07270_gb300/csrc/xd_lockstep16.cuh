// Packed 16-bit lockstep band kernel: two window slots per 32-bit register.
//
// Same extension, same reading of the X-drop recurrence and the same
// results as lockstep_loop (xd_device.cuh); only the arithmetic changes.
// It is exact whenever the scoring passes packed16_ok():
//   match - gap <= 128, mismatch >= -128, mismatch + 2|gap| >= 0,
//   x + match <= 1536,
// and, for lanes of 32 and 64 slots, relative_ok().
//
// What bounds it: integer issue.  Byte permutes, logic, minima, maxima and
// DPX instructions issue on the ALU pipe and multiply-adds on the FMA pipe,
// two cycles each per warp, so the count of instructions per register and
// their split over the two pipes decide the time, and the bookkeeping of a
// diagonal (base windows, lane and group maximum, T, events), which is per
// lane: lanes of more slots spread it over more cells (29x, first tier: x = 50
// 4x16 51.6 ms, 2x32 45.0, 1x64 50.6; x = 100 4x32 88.6, 2x64 84.9; x = 15 2x16
// 25.7, 1x32 23.0).  Rare events cost as a group's event stops the whole warp:
// shifts by an eighth of the window instead of one slot, on registers moved
// directly and with bases loaded once for both directions, took 1x64 from
// 90 to 50 ms and 2x32 from 50.2 to 46.0.
//
// Relative frame.  A live cell of anti-diagonal d is kept as its height
// above the diagonal's X-drop threshold,
//   v = KS * (H - (T_{d-1} - x)) >= 0        (KS = 16, 32 or 64, see Key),
// and a pruned one as a negative half, kDead = -2^14 or below.  In the
// normalised score H + d*|gap| the threshold grows by step(d) = |gap| + the
// rise of T on diagonal d, gap predecessors enter unchanged and diagonal
// ones with s' = s + 2|gap| >= 0.  So, in the frame of d-2,
//   r = max3(V + s', U_t + step(d-2), U_t+-1 + step(d-2)),
// V the slot's value two diagonals ago and U diagonal d-1, and
//   v = min_unsigned(r - step(d-2) - step(d-1), kDead)
// moves r into the frame of d and prunes it in one DPX instruction: a live
// result is >= 0 and stays, a result below the threshold wraps above kDead
// as an unsigned half and becomes kDead.  No threshold, mask or rebase per
// cell.  Per register: a LOP3, a three-way maximum, the add-minimum and half
// a key maximum on the ALU pipe; the substitution, the step and the key on
// the FMA pipe: 6.5 instructions, 3.5 of them ALU (the absolute frame of
// xd_lockstep16_abs.cuh takes 8.5 and 4.5).  Measured on 304,178 pairs of 29x
// reads, first tier: x = 50 (2x32) 64.3 ms in the absolute frame, 50.2 ms in
// this one; x = 100 (4x32) 122.8 and 94.8 ms; x = 15 (2x16) 35.3 and 31.3 ms.
//   Ranges.  Every half formed from a live one is at most KS * (x + 2 match +
// 2|gap|) + KS - 1 < 2^15 (relative_ok).  A pruned half sinks by at most one
// step per diagonal; every lift_period pairs the pruned halves are lifted
// back to kDead, before one can wrap.  s' and steps add less than 2^14 to a
// half, so a pruned half never reaches 0 by them either, and the plain
// 32-bit adds never carry from the low half (it stays below 2^16 when
// pruned and below 2^15 when live).
//   Substitution.  One XOR of the 2-bit base windows gives a flag per slot
// (bit 2s+1).  A shift shared by two or three registers brings register
// t's two flags to bits p and p+16, p = 1, 3 or 5; one LOP3 keeps them and
// adds a constant c, and w * k + V adds the match bonus and, through c, the
// mismatch score s'(mismatch) = k c / KS (subst_folds; other scorings take
// one more add).
//   Chain.  The keys are taken from r, before the prune, so the maximum of a
// diagonal does not wait for the maximum of the one before it.
//   Rectangle ends.  Cells with i > m or j > n are not masked; their match
// flags are cleared instead.  Without matches no such cell exceeds T, and none
// leads back inside, so scores, positions and the two-dead-diagonal end
// are those of the cells inside.  They can only keep a finished extension
// running, so every 16 pairs they are pruned explicitly.  (Per-register
// masks take 5 more instructions per register, on a quarter of the pairs.)
//   Key.  r + (S-1-slot) per half, compared signed, KS = 2^(slot bits): for
// live cells it orders by value and then by lowest slot.  Across lanes the
// key becomes value * 2^(SB+5) + (31 - lane) * 2^SB + slot bits, so one group
// maximum gives the largest value and, among equal ones, the lowest window
// slot: the first cell in order of increasing i on the diagonal.
//
// Layout.  Lane g of a group of L lanes holds the window slots g*S .. g*S+S-1
// (S = 2*C2 slots).  Register t holds slot t in its low half and slot t+C2
// in its high half, so the neighbour slot s+1 (s-1) of every slot in
// register t sits in register t+1 (t-1) at the same half; only the end
// registers need a byte permute and, between lanes, one shuffle.
//
// Window edges.  The edges are tested once per pair of diagonals, after the
// even one: no live cell of diagonals d+1, d+2 can leave the window unless
// E's top slot (diagonal d) or O's top slot (d-1) is live, or E's bottom slot
// is.  The window can then shift up by k slots if E's k+1 bottom slots and
// O's k bottom slots are dead, or down by k if the k+1 top slots of E and of
// O are dead; it shifts by NSH slots (an eighth of the window, at most a
// quarter lane) if it can, since a band that drifts by chance comes back to
// such an edge far less often than to one shifted by one slot, else by one
// slot; otherwise the band has outgrown the window and the task goes to a
// wider tier.
#pragma once
#include <stdint.h>

#include <type_traits>

#include "xd_device.cuh"
#include "xd_lockstep16_abs.cuh"

namespace xd {

namespace p16 {

constexpr uint32_t kDead2 = 0xC000C000u;  // a pruned slot, both halves

__device__ __forceinline__ bool rel_live_lo(uint32_t v) { return (v & 0x8000u) == 0u; }
__device__ __forceinline__ bool rel_live_hi(uint32_t v) { return (int32_t)v >= 0; }

template <int N>
__device__ __forceinline__ uint32_t tree_max2s(const uint32_t (&k)[N])
{
    if constexpr (N == 1) {
        return k[0];
    } else if constexpr (N == 2) {
        return __vmaxs2(k[0], k[1]);
    } else {
        constexpr int M = (N + 2) / 3;
        uint32_t r[M];
#pragma unroll
        for (int i = 0; i < M; ++i) {
            if (3 * i + 2 < N) r[i] = __vimax3_s16x2(k[3 * i], k[3 * i + 1], k[3 * i + 2]);
            else if (3 * i + 1 < N) r[i] = __vmaxs2(k[3 * i], k[3 * i + 1]);
            else r[i] = k[3 * i];
        }
        return tree_max2s<M>(r);
    }
}

// Match-bit positions.  A lane's shifted flag word puts register t's two
// flags at bits pos and pos + 16.  With KS >= 32 one shift serves three
// registers (positions 1, 3, 5), else two (1, 3).
template <int C2>
__host__ __device__ constexpr int rel_group() { return C2 >= 16 ? 3 : 2; }
template <int C2>
__host__ __device__ constexpr int rel_pos(int t) { return 1 + 2 * ((t % 8) % rel_group<C2>()); }

// The flag bits of slots lo .. hi of a 16-slot flag word.
__device__ __forceinline__ uint32_t flag_range(int32_t lo, int32_t hi)
{
    uint32_t below, upto;
    asm("shl.b32 %0, 0xFFFFFFFF, %1;" : "=r"(below) : "r"(2 * min(max(lo, 0), 16)));
    asm("shl.b32 %0, 0xFFFFFFFF, %1;" : "=r"(upto) : "r"(2 * min(max(hi + 1, 0), 16)));
    return below & ~upto;
}

// Slots of register t outside lo .. hi, to the pruned value.
template <int C2>
__device__ __forceinline__ uint32_t keep_range(uint32_t v, int t, int32_t lo, int32_t hi)
{
    const uint32_t l = (t >= lo && t <= hi) ? 0x0000FFFFu : 0u;
    const uint32_t h = (t + C2 >= lo && t + C2 <= hi) ? 0xFFFF0000u : 0u;
    return (v & (l | h)) | (kDead2 & ~(l | h));
}

// N words of 16 bases each from consecutive base positions, word k starting
// 16 * step * k bases (step = 1 or -1) after base pos of word w0 of the packed
// buffer, its 16 fields in reverse order with rev.  One code path for
// both directions (groups of one warp differ in theirs) in 32-bit
// arithmetic; words outside the buffer are clamped (ld_word).
template <int N>
__device__ __forceinline__ void load_words(const uint32_t *pk, int32_t last, int32_t w0,
                                           int32_t pos, int step, bool rev, uint32_t (&out)[N])
{
    const int32_t w = w0 + (pos >> 4) + (step < 0 ? 1 : 0);
    const uint32_t sh = 2u * (uint32_t)(pos & 15);
    uint32_t r[N + 1];
#pragma unroll
    for (int k = 0; k <= N; ++k) r[k] = __ldg(pk + min(max(w + step * k, 0), last));
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const uint32_t v = __funnelshift_r(step > 0 ? r[k] : r[k + 1], step > 0 ? r[k + 1] : r[k], sh);
        out[k] = rev ? rev16(v) : v;
    }
}

// V moved by K slots towards lane 0 (UP: slot s takes slot s + K) or away
// from it, where mine; the slots that enter come from the neighbouring lane,
// pruned beyond the group.  Every lane of the warp takes part.
template <int L, int C2, int K, bool UP>
__device__ __forceinline__ void shift_slots(uint32_t (&V)[C2], bool mine, bool edge_lane)
{
    static_assert(K < C2, "shift within a register's reach");
    uint32_t in[K];
#pragma unroll
    for (int q = 0; q < K; ++q) {
        in[q] = kDead2;
        if constexpr (L > 1) {
            in[q] = UP ? __shfl_down_sync(FULL, V[q], 1, L) : __shfl_up_sync(FULL, V[C2 - 1 - q], 1, L);
            if (edge_lane) in[q] = kDead2;
        }
    }
    if (!mine) return;
    uint32_t e[K];  // the registers whose slots cross a half
#pragma unroll
    for (int q = 0; q < K; ++q)
        e[q] = UP ? prmt(V[q], in[q], 0x5432) : prmt(in[q], V[C2 - 1 - q], 0x5432);
    if (UP) {
#pragma unroll
        for (int t = 0; t < C2 - K; ++t) V[t] = V[t + K];
#pragma unroll
        for (int q = 0; q < K; ++q) V[C2 - K + q] = e[q];
    } else {
#pragma unroll
        for (int t = C2 - 1; t >= K; --t) V[t] = V[t - K];
#pragma unroll
        for (int q = 0; q < K; ++q) V[K - 1 - q] = e[q];
    }
}

// Per-group constants of the substitution: k[q] multiplies a flag at bit
// 1 + 2q into the match bonus, c[q] (both halves) the mismatch score when
// the scoring allows it (else 0, and mi2 is added).
struct RelSubst {
    uint32_t k[3], c[3];
    uint32_t mi2;
};

// One anti-diagonal for one lane.  V: diagonal d-2 (in its own frame),
// overwritten with d; U: diagonal d-1 plus the threshold step from d-2 to
// d-1, so both predecessors are in the frame of d-2.  edge: the neighbouring
// lane's end register of U.  eq[w]: bit 2s+1 set iff the bases of slot
// 16w + s match.  nstep: minus the threshold step from d-2 to d, per half.
// Returns the largest keys of the low and of the high halves, in the frame
// of d-2 and before the prune: they do not wait for the threshold of d, which
// the previous diagonal's maximum decides, so the two diagonals' chains
// overlap.
template <int C2, int NW, bool ODD, bool ADD>
__device__ __forceinline__ uint32_t dp16r(uint32_t (&V)[C2], const uint32_t (&U)[C2],
                                          uint32_t edge, const uint32_t (&eq)[NW],
                                          const RelSubst &sb, uint32_t nstep, uint32_t one)
{
    constexpr int G = rel_group<C2>();
    constexpr int NS = (8 + G - 1) / G;  // shifts per flag word of 8 registers
    constexpr int NE = C2 >= 16 ? C2 / 8 : 1;
    // registers 8h .. 8h+7: slot t's flag at 2(t-8h)+1, slot t+C2's 16 bits on
    uint32_t es[NE][NS];
#pragma unroll
    for (int h = 0; h < NE; ++h) {
        uint32_t e;
        if constexpr (C2 == 2) e = (eq[0] & 0xFu) | (eq[0] << 12);
        else if constexpr (C2 == 4) e = prmt(eq[0], eq[0], 0x2100);
        else if constexpr (C2 == 8) e = eq[0];
        else e = prmt(eq[h / 2], eq[NW / 2 + h / 2], (h & 1) ? 0x7632 : 0x5410);
#pragma unroll
        for (int q = 0; q < NS; ++q) es[h][q] = e >> (2 * G * q);
    }
    uint32_t key[C2];
#pragma unroll
    for (int t = 0; t < C2; ++t) {
        uint32_t sh;
        if (ODD) sh = (t + 1 < C2) ? U[t + 1] : prmt(U[0], edge, 0x5432);
        else sh = (t > 0) ? U[t - 1] : prmt(edge, U[C2 - 1], 0x5432);
        const int q = (t % 8) % G;
        const uint32_t w = (es[t / 8][(t % 8) / G] & (0x00010001u << rel_pos<C2>(t))) | sb.c[q];
        uint32_t cand = fma_add(w, sb.k[q], V[t]);
        if (ADD) cand = fma_add(cand, one, sb.mi2);
        const uint32_t r = __vimax3_s16x2(cand, U[t], sh);
        // r - threshold step: a live cell stays >= 0; below the threshold it
        // wraps to an unsigned value above kDead, which the minimum replaces
        V[t] = __viaddmin_u16x2(r, nstep, kDead2);
        key[t] = fma_add(r, one, idx2<C2>(t));
    }
    return tree_max2s<C2>(key);
}

}  // namespace p16

// The relative frame on lanes of S slots: every value a step forms from a
// live one, at most x + 2 match + 2|gap| in units of KS, stays below 2^15.
// Lanes of up to 16 slots hold every scoring of packed16_ok.  With KS = 64
// the steps are kept below 2^12, so that pruned slots sink slowly enough.
template <int S>
__host__ __device__ inline bool relative_ok(const Scoring &sc)
{
    return packed16_ok(sc) &&
           (sc.x + 2 * sc.match - 2 * sc.gap + 1) * p16::key_scale<S>() <= 0x8000 &&
           (S < 64 || sc.match - sc.gap <= 64);
}

// Whether the mismatch score can ride on the flag word (RelSubst::c): c =
// 2 mm / bonus at flag bit 1 (mm = mismatch + 2|gap|, bonus = match -
// mismatch) must be whole, leave the flag bit free and fit its half.
__host__ __device__ inline bool subst_folds(const Scoring &sc)
{
    const int32_t mm = sc.mismatch - 2 * sc.gap, bonus = sc.match - sc.mismatch;
    const int32_t c = 2 * mm / bonus;
    return c * bonus == 2 * mm && !(c & 2) && c < 0x800;
}

// Pairs of diagonals after which pruned slots must be lifted back to the
// pruned value: one may sink by the threshold's growth, at most match +
// |gap|, on every diagonal, and by two such steps at once, and has 2^14 of
// room.
template <int S>
__host__ __device__ inline int32_t lift_period(const Scoring &sc)
{
    const int32_t step = (sc.match - sc.gap) * p16::key_scale<S>();
    const int32_t p = ((1 << 14) / step - 2) / 2;
    return p < 1 ? 1 : p;
}

// one: 1 (see fma_add).
template <int L, int C2, class Src>
__device__ __forceinline__ void lockstep16_loop(Src &src, const uint32_t *pk, int64_t nw,
                                                uint32_t one)
{
    using namespace p16;
    constexpr int S = 2 * C2;  // slots per lane
    constexpr int W = L * S;
    constexpr int NW = S > 16 ? S / 16 : 1;      // base-window words per read
    constexpr int SB = slot_bits<S>();           // slot bits of a key
    constexpr int VS = L == 1 ? SB : SB + 5;     // value shift of a group key
    constexpr uint32_t SMASK = (1u << SB) - 1u;
    constexpr uint32_t KS = (uint32_t)key_scale<S>();
    // slots of a long window shift
    constexpr int NSH = S / 4 < 2 ? 1 : S / 4 < W / 8 ? S / 4 : W / 8;
    constexpr int32_t kForever = 1 << 20;
    using T0 = std::integral_constant<bool, false>;
    using T1 = std::integral_constant<bool, true>;
    static_assert(S <= 64 && 32 % L == 0 && (C2 == 2 || C2 == 4 || C2 == 8 || C2 % 16 == 0),
                  "packed tile shape");
    const int lane = threadIdx.x & 31;
    const int glane = lane % L;
    const int gbase = lane - glane;
    const unsigned gm = group_mask<L>(gbase);
    const bool bot_lane = glane == 0, top_lane = glane == L - 1;
    // per-lane constants: factors and addends that prune the edge beyond
    // the group
    const uint32_t keep_up = top_lane ? 0u : 1u, keep_dn = bot_lane ? 0u : 1u;
    const uint32_t edge_up = top_lane ? kDead2 : 0u, edge_dn = bot_lane ? kDead2 : 0u;

    // Per-group task state (uniform within a group).
    bool active = false, exhausted = false;
    uint32_t task = 0;
    const Job *gj = nullptr;
    Scoring sc{1, -1, -1, 0};
    int32_t aw0 = 0, bw0 = 0, ab0 = 0, bb0 = 0;  // word and base in it of both streams' first base
    int dir = 1;
    int32_t mn = 0, m = 0, n = 0, d = 0, i0 = 0, j0 = 0, T = 0;
    int32_t bkey = 0, bi0 = 0, bd = 0;  // best cell: group key, this lane's i0, diagonal
    RelSubst rs = {{0, 0, 0}, {0, 0, 0}, 0};
    uint32_t dA = 0, dB = 0;            // threshold steps d-2 -> d-1, d-1 -> d
    int32_t sA = 0, sB = 0;             // the same steps in units of the score
    int32_t ng = 0;                     // |gap|
    uint32_t ngp = 0;                   // |gap| * KS in both halves
    int32_t lift = kForever;            // lift_period of the group's scoring
    bool add_mi = false;                // the group's scoring needs rs.mi2 added
    // event masks, 0 while the group waits: the half of this lane's end
    // slots the edge test reads, and the sign bit for the end test
    uint32_t tmask = 0, bmask = 0, amask = 0;
    int32_t ptop = 0;                   // best value of the last even diagonal
    uint32_t finw = 0;                  // nonzero: two dead diagonals in a row
    uint32_t E[C2], O[C2];
#pragma unroll
    for (int t = 0; t < C2; ++t) { E[t] = kDead2; O[t] = kDead2; }
    uint32_t Aw[NW], Bw[NW], LA = 0, LB = 0;  // base windows, lookahead words
#pragma unroll
    for (int k = 0; k < NW; ++k) { Aw[k] = 0; Bw[k] = 0; }
    // Warp-uniform countdowns, in pairs of diagonals.
    int la_n = 16;             // the lookahead words still cover
    int32_t budget = 0;        // known to stay inside every rectangle
    int32_t lift_n = kForever; // until pruned slots must be lifted
    int32_t ctr = 0, ctr0 = 0; // until the next event that is due anyway, and its start
    const int32_t lane_bits = (31 - glane) << SB;

    auto retire = [&](bool overflow) {
        int32_t bi = 0, bj = 0;
        if (bd > 0) {
            const int32_t slot = S - 1 - (int)(bkey & SMASK);
            bi = L == 1 ? bi0 + slot : (bi0 - glane * S) + (31 - ((bkey >> SB) & 31)) * S + slot;
            bj = bd - bi;
        }
        if (glane == 0) src.retire(gj, task, overflow, T, bi, bj);
        active = false;
        tmask = bmask = amask = 0;
        add_mi = false;
        lift = kForever;
    };

    // Diagonal pairs until a cell of this group's window can leave the
    // rectangle: each pair moves the top slot's i and the bottom slot's j
    // up by one (window shifts recompute it).
    auto refresh_budget = [&]() {
        const int32_t mg = min(m - (i0 - glane * S + W - 1), n - (j0 + glane * S));
        budget = __reduce_min_sync(FULL, active ? mg : INT32_MAX);
    };

    // The base windows of this lane's slots at the current i0, j0: slot s
    // holds a[i0 + s] and b[j0 - s]; the lookahead words the next 16 bases.
    const int32_t last = (int32_t)nw - 1;
    auto load_ahead = [&]() {
        uint32_t v[1];
        const int32_t ia = i0 + 16 * NW;
        load_words<1>(pk, last, aw0, ab0 + (dir > 0 ? ia - 1 : -ia - 14), 1, dir < 0, v);
        LA = v[0];
        load_words<1>(pk, last, bw0, bb0 + (dir > 0 ? j0 : -j0 - 15), 1, dir > 0, v);
        LB = v[0];
    };
    auto load_windows = [&]() {
        uint32_t v[NW + 1];
        load_words<NW + 1>(pk, last, aw0, ab0 + (dir > 0 ? i0 - 1 : -i0 - 14), dir, dir < 0, v);
#pragma unroll
        for (int k = 0; k < NW; ++k) Aw[k] = v[k];
        LA = v[NW];
        load_words<NW + 1>(pk, last, bw0, bb0 + (dir > 0 ? j0 : -j0 - 15), -dir, dir > 0, v);
        LB = v[0];
#pragma unroll
        for (int k = 0; k < NW; ++k) Bw[k] = v[k + 1];
    };

    // One anti-diagonal and the bookkeeping that cannot wait for the end of
    // the pair: T and the best cell.  Returns the best value above the
    // threshold (negative iff every cell of the diagonal was pruned).
    auto diag = [&](auto odd_tag, auto masked_tag, auto add_tag) -> int32_t {
        constexpr bool ODD = decltype(odd_tag)::value;
        constexpr bool MASKED = decltype(masked_tag)::value;
        constexpr bool ADD = decltype(add_tag)::value;
        ++d;
        if (ODD) {
            ++i0;
#pragma unroll
            for (int k = 0; k < NW; ++k)
                Aw[k] = __funnelshift_r(Aw[k], k + 1 < NW ? Aw[k + 1] : LA, 2);
            LA >>= 2;
        } else {
            ++j0;
#pragma unroll
            for (int k = NW - 1; k > 0; --k) Bw[k] = __funnelshift_l(Bw[k - 1], Bw[k], 2);
            Bw[0] = __funnelshift_l(LB, Bw[0], 2);
            LB <<= 2;
        }
        uint32_t eq[NW];
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            const uint32_t xx = Aw[k] ^ Bw[k];
            eq[k] = ~(xx | (xx << 1));
            if (MASKED) eq[k] &= flag_range(j0 - n - 16 * k, m - i0 - 16 * k);
        }
        const uint32_t nstep = 0x00010000u - (dA + dB);  // both halves of dA and dB are equal
        uint32_t U[C2];
#pragma unroll
        for (int t = 0; t < C2; ++t) U[t] = fma_add(ODD ? E[t] : O[t], one, dA);
        uint32_t kk;
        if (ODD) {
            uint32_t edge = kDead2;
            if constexpr (L > 1)
                edge = fma_add(__shfl_down_sync(FULL, U[0], 1, L), keep_up, edge_up);
            kk = dp16r<C2, NW, true, ADD>(O, U, edge, eq, rs, nstep, one);
        } else {
            uint32_t edge = kDead2;
            if constexpr (L > 1)
                edge = fma_add(__shfl_up_sync(FULL, U[C2 - 1], 1, L), keep_dn, edge_dn);
            kk = dp16r<C2, NW, false, ADD>(E, U, edge, eq, rs, nstep, one);
        }
        int32_t mkey = max((int32_t)kk >> 16, (int32_t)(kk << 16) >> 16);
        // with key = 2^SB v + i: 32 key - 31 i = 2^VS v + i (multiply-adds)
        if constexpr (L > 1)
            mkey = lockstep_group_max<L>((int32_t)fma_add(
                (uint32_t)mkey, one << 5,
                fma_add((uint32_t)mkey & SMASK, 0u - 31u, (uint32_t)lane_bits)));
        // the best value above the diagonal's threshold, and above T
        const int32_t top = (mkey >> VS) - (sA + sB);
        const int32_t rise = max(top - sc.x, 0);
        dA = dB;
        dB = (uint32_t)rise * (KS * 0x10001u) + ngp;
        sA = sB;
        sB = rise + ng;
        T += rise;
        if (rise > 0) {  // decoded at retire
            bkey = mkey;
            bi0 = i0;
            bd = d;
        }
        return top;
    };

    // One pair of anti-diagonals (odd, then even).  Returns the warp-wide
    // "something to do" vote: a window edge went live, a task ended, or the
    // countdown ran out.
    auto pair = [&](auto masked_tag, auto add_tag) -> bool {
        constexpr bool MASKED = decltype(masked_tag)::value;
        const int32_t top_o = diag(std::true_type{}, masked_tag, add_tag);
        const int32_t top_e = diag(std::false_type{}, masked_tag, add_tag);
        // sign bits: the odd diagonal is dead, and so is the even one before or after it
        finw = (uint32_t)top_o & (uint32_t)(ptop | top_e) & amask;
        if (MASKED && d >= mn) finw = amask;
        ptop = top_e;
        // window edges: this group's bottom lane tests E's bottom slot, its
        // top lane the top slots of E and O
        const uint32_t ew = (~(E[C2 - 1] & O[C2 - 1]) & tmask) | (~E[0] & bmask);
        --ctr;
        return __any_sync(FULL, (ew | finw) != 0u) || ctr == 0;
    };

    // The work behind an event, after the even diagonal of a pair.  Returns
    // true when the loop must go back to the task switch (a group waits for
    // a task, no group is left running, the masking-free budget no longer
    // covers a pair, or, masked, it covers one again).
    auto handle = [&](const bool masked) -> bool {
        la_n -= ctr0 - ctr;
        bool fin = finw != 0u, ovf = false;
        const bool go = active && !fin;
        const bool need_dn_l = bot_lane && rel_live_lo(E[0]);
        const bool need_up_l = top_lane && (rel_live_hi(E[C2 - 1]) || rel_live_hi(O[C2 - 1]));
        if (__any_sync(FULL, go && (need_dn_l || need_up_l))) {
            // dead slots at both ends of this lane: k + 1 of E (and of O at
            // the top, k at the bottom), for k = 1 and k = NSH
            uint32_t lo1 = E[0] & E[1] & O[0], hi1 = E[C2 - 1] & O[C2 - 1] & E[C2 - 2] & O[C2 - 2];
            uint32_t los = lo1, his = hi1;
#pragma unroll
            for (int k = 1; k < NSH; ++k) {
                los &= E[k + 1] & O[k];
                his &= E[C2 - 2 - k] & O[C2 - 2 - k];
            }
            // bit 0: the lane's edge is live; 1, 2: one slot, NSH slots are free
            int bot = (rel_live_lo(E[0]) ? 1 : 0) | (rel_live_lo(lo1) ? 0 : 2) |
                      (rel_live_lo(los) ? 0 : 4);
            int top = (need_up_l ? 1 : 0) | (rel_live_hi(hi1) ? 0 : 2) | (rel_live_hi(his) ? 0 : 4);
            if constexpr (L > 1) {  // every lane takes part in every shuffle
                bot = __shfl_sync(FULL, bot, 0, L);
                top = __shfl_sync(FULL, top, L - 1, L);
            }
            const bool nu = go && (top & 1), nd = go && !(top & 1) && (bot & 1);
            const int room = nu ? bot : top;  // of the opposite edge
            ovf = (nu || nd) && !(room & 2);
            const int by = (nu || nd) && !ovf ? ((room & 4) ? NSH : 1) : 0;
            auto shift = [&](auto k_tag, auto up_tag) {  // groups that move by k slots
                constexpr int K = decltype(k_tag)::value;
                constexpr bool UP = decltype(up_tag)::value;
                const bool mine = by == K && (UP ? nu : nd);
                if (!__any_sync(FULL, mine)) return;
                shift_slots<L, C2, K, UP>(E, mine, UP ? top_lane : bot_lane);
                shift_slots<L, C2, K, UP>(O, mine, UP ? top_lane : bot_lane);
                if (mine) {
                    i0 += UP ? K : -K;
                    j0 -= UP ? K : -K;
                }
            };
            if constexpr (NSH > 1) {
                shift(std::integral_constant<int, NSH>{}, T1{});
                shift(std::integral_constant<int, NSH>{}, T0{});
            }
            shift(std::integral_constant<int, 1>{}, T1{});
            shift(std::integral_constant<int, 1>{}, T0{});
            if (by > 0) load_windows();
            fin = fin || ovf;
        }
        if (fin) retire(ovf);
        const bool refill = la_n == 0;
        if (refill) {
            load_ahead();
            la_n = 16;
            if (masked) {  // end what lives outside the rectangle
                const int32_t lo = j0 - n, hi = m - i0;
#pragma unroll
                for (int t = 0; t < C2; ++t) {
                    E[t] = keep_range<C2>(E[t], t, lo, hi);
                    O[t] = keep_range<C2>(O[t], t, lo - 1, hi);  // one diagonal earlier
                }
            }
            lift_n -= 16;
            if (lift_n < 16) {  // before the next refill: lift the pruned slots
#pragma unroll
                for (int t = 0; t < C2; ++t) {
                    E[t] = __vmaxs2(E[t], kDead2);
                    O[t] = __vmaxs2(O[t], kDead2);
                }
                lift_n = __reduce_min_sync(FULL, lift);
                la_n = min(16, lift_n);
            }
        }
        if constexpr (Src::kCanAbort) {
            if (__any_sync(FULL, src.aborted())) return true;
        }
        if (__any_sync(FULL, !active && !exhausted) || !__any_sync(FULL, active)) return true;
        // Masked pairs are dearer: look every 16 of them (with the refill)
        // whether the unmasked copy is safe again.
        if (!masked || refill) {
            refresh_budget();
            if (masked ? budget >= 1 : budget < 1) return true;
        }
        ctr0 = ctr = masked ? la_n : min(la_n, budget);
        return false;
    };

    for (;;) {
        // A serving kernel can be told to leave at once (teardown).
        if constexpr (Src::kCanAbort) {
            if (__any_sync(FULL, src.aborted())) break;
        }
        // ---------------- task switches (top of an odd diagonal) ----------------
        const bool need = !active && !exhausted;
        const unsigned needm = __ballot_sync(FULL, need && glane == 0);
        if (needm) {
            const int r = src.fetch_warp(needm, lane, gbase, gm, need, task, gj);
            if (need) {
                if (r < 0) {
                    exhausted = true;
                } else if (r > 0) {
                    const Ext e = src.open(gj, task, sc);
                    if (e.ok && !relative_ok<S>(sc)) {
                        // A scoring 16-bit cells cannot hold exactly (a serving
                        // request's own): hand the task to the next, 32-bit tier.
                        if (glane == 0) src.retire(gj, task, true, 0, 0, 0);
                    } else if (e.ok) {
                        aw0 = (int32_t)(e.A.s0 >> 4);
                        ab0 = (int32_t)(e.A.s0 & 15);
                        bw0 = (int32_t)(e.B.s0 >> 4);
                        bb0 = (int32_t)(e.B.s0 & 15);
                        dir = e.A.dir;
                        m = e.m;
                        n = e.n;
                        mn = m + n;
                        ng = -sc.gap;
                        const int32_t mm = sc.mismatch + 2 * ng;
                        const int32_t bonus = sc.match - sc.mismatch;
                        const bool folds = subst_folds(sc);
                        add_mi = !folds;
                        rs.mi2 = folds ? 0u : pack2(mm * (int32_t)KS);
                        const uint32_t c = folds ? (uint32_t)(2 * mm / bonus) * 0x10001u : 0u;
#pragma unroll
                        for (int q = 0; q < 3; ++q) {
                            rs.k[q] = (uint32_t)bonus * KS >> (1 + 2 * q);
                            rs.c[q] = c << (2 * q);
                        }
                        ngp = (uint32_t)ng * (KS * 0x10001u);
                        dA = dB = ngp;
                        sA = sB = ng;
                        lift = lift_period<S>(sc);
                        // origin (H = 0, x above the threshold) at window slot W/2
#pragma unroll
                        for (int t = 0; t < C2; ++t) {
                            const int slo = glane * S + t, shi = slo + C2;
                            const uint32_t orig = (uint32_t)sc.x * KS, dead = kDead2 & 0xFFFFu;
                            E[t] = (slo == W / 2 ? orig : dead) |
                                   ((shi == W / 2 ? orig : dead) << 16);
                            O[t] = kDead2;
                        }
                        i0 = -(W / 2) + glane * S;
                        j0 = (W / 2) - glane * S;
                        load_windows();
                        d = 0;
                        T = 0;
                        bd = 0;
                        ptop = 0;
                        active = true;
                        tmask = top_lane ? 0x80000000u : 0u;
                        bmask = bot_lane ? 0x00008000u : 0u;
                        amask = 0x80000000u;
                    }
                }
            }
        }
        if (__all_sync(FULL, exhausted && !active)) break;
        if (!__any_sync(FULL, active)) {
            src.idle();
            continue;
        }
        refresh_budget();
        lift_n = min(lift_n, __reduce_min_sync(FULL, lift));
        la_n = min(la_n, lift_n);
        // a group that still waits for a task asks again after kWaitPairs pairs
        const bool waits = __any_sync(FULL, !active && !exhausted);
        const int32_t most = budget >= 1 ? min(la_n, budget) : la_n;
        if constexpr (Src::kWaitPairs == 1) ctr0 = ctr = waits ? 1 : most;
        else ctr0 = ctr = waits ? min(most, Src::kWaitPairs) : most;
        if (budget < 1) {
            for (;;) {
                if (pair(T1{}, T1{}) && handle(true)) break;
            }
        } else if (__any_sync(FULL, add_mi)) {
            for (;;) {
                if (pair(T0{}, T1{}) && handle(false)) break;
            }
        } else {
            for (;;) {  // no cell of any window can leave its rectangle
                if (pair(T0{}, T0{}) && handle(false)) break;
            }
        }
    }
}

}  // namespace xd
