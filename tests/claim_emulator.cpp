// CPU run of the claims of paper_2309_07270_gb300/csrc/xd_claim.cuh (the
// functions the kernels call) under a scheduler that lets one thread at a
// time do one memory operation, chosen at random, and holds single threads
// up for long stretches (test infrastructure).
#include <stdint.h>

#include <condition_variable>
#include <mutex>
#include <random>
#include <thread>
#include <vector>

#include "../paper_2309_07270_gb300/csrc/xd_claim.cuh"

namespace {

struct Scheduler {
    std::mutex mu;
    std::condition_variable cv;
    std::mt19937 rng;
    int n, left, turn = -1, waiting = 0;
    std::vector<char> alive, ready;
    std::vector<int> held;  // operations of others before this thread may go on
    explicit Scheduler(int threads, uint32_t seed)
        : rng(seed), n(threads), left(threads), alive(threads, 1), ready(threads, 0), held(threads, 0)
    {
    }
    void pick()  // every living thread waits: choose the next
    {
        std::vector<int> free;
        for (int k = 0; k < n; ++k) {
            if (!alive[k]) continue;
            if (held[k] > 0) --held[k];
            else free.push_back(k);
        }
        if (free.empty())
            for (int k = 0; k < n; ++k)
                if (alive[k]) free.push_back(k);
        turn = free[rng() % free.size()];
        if (rng() % 16 == 0) held[turn] = (int)(rng() % 400);  // held up after this operation
        cv.notify_all();
    }
    void step(int me)
    {
        std::unique_lock<std::mutex> lk(mu);
        ready[me] = 1;
        if (turn == me) turn = -1;
        if (++waiting == left) pick();
        cv.wait(lk, [&] { return turn == me; });
        --waiting;
        ready[me] = 0;
    }
    void leave(int me)
    {
        std::lock_guard<std::mutex> lk(mu);
        alive[me] = 0;
        --left;
        turn = -1;
        if (left && waiting == left) pick();
    }
};

struct HostMem {
    Scheduler *s;
    int me;
    uint32_t load(const uint32_t *p)
    {
        s->step(me);
        return *p;
    }
    uint32_t add(uint32_t *p, uint32_t v)
    {
        s->step(me);
        const uint32_t old = *p;
        *p = old + v;
        return old;
    }
    void fence() {}
};

}  // namespace

// Every thread appends `each` entries and takes entries between and after, as
// a warp of the first tier does, until it finds none left.  Returns 0, or 1 if
// a position at or past the number of entries was handed out, 2 if one was
// handed out twice, 3 if entries were left without an owner.
extern "C" int emulate_claims(int threads, int each, uint32_t seed)
{
    Scheduler s(threads, seed);
    uint32_t count = 0, ready = 0, taken = 0;
    std::vector<int> owners((size_t)threads * each + threads, 0);
    int past = 0, twice = 0;
    std::vector<std::thread> th;
    for (int k = 0; k < threads; ++k)
        th.emplace_back([&, k] {
            HostMem m{&s, k};
            const xd::ClaimWords w{&count, &ready, &taken};
            auto take = [&] {
                uint32_t pos = 0;
                const xd::Claim c = xd::claim_entry(m, w, &pos);
                if (c == xd::Claim::kGot) {
                    if (pos >= count) past = 1;
                    if (pos < owners.size() && owners[pos]++) twice = 1;
                }
                return c;
            };
            for (int e = 0; e < each; ++e) {
                m.add(&count, 1u);
                s.step(k);  // the entry itself
                xd::entry_written(m, w);
                if (e % 3 == k % 3) take();
            }
            while (take() != xd::Claim::kEmpty) {
            }
            s.leave(k);
        });
    for (auto &t : th) t.join();
    if (past) return 1;
    if (twice) return 2;
    return taken == count && ready == 0 && count == (uint32_t)threads * (uint32_t)each ? 0 : 3;
}
