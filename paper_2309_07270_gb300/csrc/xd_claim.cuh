// Claims on a list that some threads append to while others take from it.
//
// Taking an entry by an add on the number taken, after a look at how many
// there are, can go past the end: between the look and the add any number of
// other threads may take entries.  So the right to an entry is drawn from a
// count of written entries (ready): who brings it down from above 0 has one,
// who does not puts it back.  As many positions are handed out as rights, so
// every position is below the number of entries reserved.  A thread that
// reads taken, then count, and finds no more entries than were taken knows
// that each of them has an owner.
#pragma once
#include <stdint.h>

#if defined(__CUDACC__)
#define XC_HD __device__ __forceinline__
#else
#define XC_HD inline
#endif

namespace xd {

// Device words, 0 at the start.
struct ClaimWords {
    uint32_t *count;  // entries reserved
    uint32_t *ready;  // entries written, less the rights drawn (signed)
    uint32_t *taken;  // positions handed out
};

// A producer reserves position add(count, 1), writes the entry, then:
template <class Mem>
XC_HD void entry_written(Mem &m, const ClaimWords &w)
{
    m.fence();
    m.add(w.ready, 1u);
}

enum class Claim { kGot, kBusy, kEmpty };

// kGot: *pos is the caller's (its entry may be a moment away: the producer of
// another one may have been first to count it); kBusy: ask again.
template <class Mem>
XC_HD Claim claim_entry(Mem &m, const ClaimWords &w, uint32_t *pos)
{
    const uint32_t taken = m.load(w.taken);
    if (taken >= m.load(w.count)) return Claim::kEmpty;
    if ((int32_t)m.load(w.ready) <= 0) return Claim::kBusy;
    if ((int32_t)m.add(w.ready, 0xFFFFFFFFu) <= 0) {
        m.add(w.ready, 1u);
        return Claim::kBusy;
    }
    *pos = m.add(w.taken, 1u);
    return Claim::kGot;
}

}  // namespace xd
