// A model of the one-launch brick scheduler (csrc/fmm_march.cu): the work
// words, the ready queue, the waiting ring, raises and scans, with the warps as
// state machines that take turns at random, one atomic operation a turn, and
// now and then stay away for long.  Lanes that put entries into a ring go on
// independently of each other.  The model ends when the scheduler says that the
// launch is done (exit 0), when no warp can move (stalled, exit 2), or when a
// chunk of a scan is taken twice, an entry is lost or work is left (exit 3).
//
//   scheduler_model bricks waiting warps levels release seeds ring_slots any_raise keep
//
// waiting: bricks that wait at the start, their work spread over `levels`
// strides; release: strides a raise goes up; ring_slots: slots of the waiting
// ring (0: the library's); any_raise: 1 takes a claim without a look at its raise;
// keep: 1 leaves the entry of a scanning warp's own ticket where it is.
#include "fmm_ring.h"

#include <algorithm>
#include <climits>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

namespace {

using u64 = unsigned long long;
constexpr int kNone = INT_MAX;
enum { kActive = 1, kWaiting = 2 };

struct Put {
    bool ring;   // the waiting ring, else the queue
    u64 pos;
    int b;
};
struct Level {
    u64 base = 0, end = 0;
    int chunk = 32;
    u64 chunks = 0;
    int bound = 0;
};
enum State { POLL, CLAIM, ACCEPT, READ, DECIDE, COUNT, PUTS, SCANNED, TAKE, MARCH, FLAG, COUNT2, PUTS2, STOP };
struct Warp {
    State st = POLL;
    long long ticket = -1;
    u64 claim = 0;
    int ch = 0, ep = 0, i = 0, kept = kNone;
    std::vector<int> got;                      // bricks of the 32 ring entries (-1: none)
    std::vector<int> act;
    std::vector<Put> puts;
    size_t at = 0;
    int brick = -1, held = -1;
    std::vector<std::pair<int, int>> flags;    // brick, work
    long away = 0;
};

struct Model {
    int n, nw;
    u64 cap_w, cap_q;
    int stride, budget;
    bool any_raise = false, keep = false;
    std::mt19937_64 rng;
    std::vector<int> key, fl;
    std::vector<u64> queue, ring;
    u64 q_head = 0, q_tail = 0, w_tail = 0, w_head = 0, scan_word = 0;
    int pending = 0, scan_done = 0, scan_min = 0, raise_lock = 0;
    Level level[2];
    std::vector<Warp> w;
    std::vector<char> seen;   // chunks of the current scan that were taken
    const char *bad = nullptr;

    int rnd(int k) { return (int)(rng() % (u64)k); }
    static u64 entry(u64 pos, int b) { return ((pos & 0xffffffffull) << 32) | (u64)(b + 1); }

    bool try_put(const Put &p)
    {
        u64 &s = p.ring ? ring[p.pos % cap_w] : queue[p.pos % cap_q];
        if (s)
            return false;
        s = entry(p.pos, p.b);
        return true;
    }
    // Lanes put their entries one by one, in any order; true when one moved.
    bool puts(Warp &x, State next)
    {
        if (x.puts.empty()) {
            x.st = next;
            return true;
        }
        const size_t o = (size_t)rnd((int)x.puts.size());
        for (size_t k = 0; k < x.puts.size(); ++k) {
            const size_t j = (o + k) % x.puts.size();
            if (try_put(x.puts[j])) {
                x.puts.erase(x.puts.begin() + (long)j);
                return true;
            }
        }
        // a scanning warp that waits for a queue slot takes its own ticket's
        // entry out
        if (!keep && x.ticket >= 0 && x.held < 0) {
            u64 &s = queue[(u64)x.ticket % cap_q];
            if (s && (s >> 32) == ((u64)x.ticket & 0xffffffffull)) {
                x.held = (int)(s & 0xffffffffull) - 1;
                s = 0;
                return true;
            }
        }
        return false;
    }
    bool try_raise()
    {
        const int ep = (int)(scan_word >> 32);
        const Level &lv = level[ep & 1];
        if (scan_done < (int)(unsigned)lv.chunks || w_tail == w_head || raise_lock != ep)
            return false;
        Level &nl = level[(ep + 1) & 1];
        nl.base = w_head;
        nl.end = w_tail;
        nl.bound = std::max(lv.bound, scan_min == kNone ? lv.bound : scan_min) + stride;
        const unsigned count = (unsigned)(nl.end - nl.base);
        nl.chunk = (((int)((count + nw - 1) / nw)) + 31) & ~31;
        const unsigned nchunks = (count + (unsigned)nl.chunk - 1) / (unsigned)nl.chunk;
        nl.chunks = fmmgb::chunk_word((unsigned)(ep + 1), nchunks);
        w_head = nl.end;
        scan_done = 0;
        scan_min = kNone;
        seen.assign(nchunks, 0);
        raise_lock = ep + 1;
        scan_word = (u64)(ep + 1) << 32;
        return true;
    }
    bool poll(Warp &x)
    {
        if (x.ticket < 0)
            x.ticket = (long long)q_head++;
        u64 &s = queue[(u64)x.ticket % cap_q];
        if (s && (s >> 32) == ((u64)x.ticket & 0xffffffffull)) {
            x.brick = (int)(s & 0xffffffffull) - 1;
            s = 0;
            x.ticket = -1;
            x.st = TAKE;
            return true;
        }
        const int ep = (int)(scan_word >> 32);
        if (fmmgb::claimed_chunk(scan_word, level[ep & 1].chunks) >= 0) {
            x.st = CLAIM;
            return true;
        }
        if (pending < nw && try_raise())
            return true;
        if (pending == 0 && scan_done >= (int)(unsigned)level[ep & 1].chunks && w_tail == w_head && raise_lock == ep) {
            x.st = STOP;
            return true;
        }
        return false;
    }
    bool read(Warp &x)
    {
        const Level &lv = level[x.ep & 1];
        bool moved = false;
        for (int l = 0; l < 32; ++l) {
            const u64 pos = lv.base + (u64)x.ch * (u64)lv.chunk + (u64)(x.i + l);
            if (pos >= lv.end || x.got[(size_t)l] != -2)
                continue;
            u64 &s = ring[pos % cap_w];
            if (s && (s >> 32) == (pos & 0xffffffffull)) {
                x.got[(size_t)l] = (int)(s & 0xffffffffull) - 1;
                s = 0;
                moved = true;
                break;
            }
        }
        for (int l = 0; l < 32; ++l)
            if (x.got[(size_t)l] == -2 && lv.base + (u64)x.ch * (u64)lv.chunk + (u64)(x.i + l) < lv.end)
                return moved;
        x.st = DECIDE;
        x.at = 0;
        x.act.assign(32, 0);
        return true;
    }
    bool step(Warp &x)
    {
        switch (x.st) {
        case POLL:
            return poll(x);
        case CLAIM:
            x.claim = scan_word++;
            x.st = ACCEPT;
            if (rnd(8) == 0)
                x.away = rnd(40 * n);
            return true;
        case ACCEPT: {
            x.ep = (int)(x.claim >> 32);
            x.st = POLL;
            const u64 chunks = level[x.ep & 1].chunks;
            x.ch = fmmgb::claimed_chunk(any_raise ? ((chunks >> 32) << 32) | (unsigned)x.claim : x.claim, chunks);
            if (x.ch >= 0) {
                if ((u64)x.ch >= seen.size() || seen[(size_t)x.ch]++)
                    bad = "a chunk was taken twice";
                x.i = 0;
                x.kept = kNone;
                x.got.assign(32, -2);
                x.st = READ;
            }
            return true;
        }
        case READ:
            return read(x);
        case DECIDE: {   // one lane's compare-and-swap a turn
            const int b = x.got[x.at];
            if (b >= 0) {
                const int bound = level[x.ep & 1].bound;
                if (!(fl[(size_t)b] & kActive) && key[(size_t)b] != kNone && key[(size_t)b] > bound) {
                    x.act[x.at] = 2;
                    x.kept = std::min(x.kept, key[(size_t)b]);
                } else {
                    if (!(fl[(size_t)b] & kActive) && key[(size_t)b] != kNone) {
                        x.act[x.at] = 1;
                        fl[(size_t)b] |= kActive;
                    }
                    fl[(size_t)b] &= ~kWaiting;
                }
            }
            if (++x.at == 32)
                x.st = COUNT;
            return true;
        }
        case COUNT:
            x.puts.clear();
            for (int l = 0; l < 32; ++l) {
                if (x.act[(size_t)l] == 1) {
                    ++pending;
                    x.puts.push_back({false, q_tail++, x.got[(size_t)l]});
                } else if (x.act[(size_t)l] == 2)
                    x.puts.push_back({true, w_tail++, x.got[(size_t)l]});
            }
            x.st = PUTS;
            return true;
        case PUTS:
            if (!x.puts.empty())
                return puts(x, PUTS);
            x.i += 32;
            x.got.assign(32, -2);
            x.st = x.i < level[x.ep & 1].chunk ? READ : SCANNED;
            return true;
        case SCANNED:
            scan_min = std::min(scan_min, x.kept);
            ++scan_done;
            x.st = POLL;
            if (x.held >= 0) {
                x.brick = x.held;
                x.held = -1;
                x.ticket = -1;
                x.st = TAKE;
            }
            return true;
        case TAKE:
            key[(size_t)x.brick] = kNone;
            x.st = MARCH;
            return true;
        case MARCH: {
            x.flags.clear();
            const int bound = level[(scan_word >> 32) & 1].bound;
            for (int k = rnd(7); k > 0 && budget > 0; --k, --budget)
                x.flags.push_back({rnd(n), bound + rnd(3 * stride + 1) - stride});
            x.flags.push_back({x.brick, kNone});   // the end of the march comes with the flags
            x.puts.clear();
            x.act.clear();
            x.at = 0;
            x.st = FLAG;
            return true;
        }
        case FLAG: {   // one lane's compare-and-swap a turn
            const int b = x.flags[x.at].first, bound = level[(scan_word >> 32) & 1].bound;
            const bool own = x.at + 1 == x.flags.size();
            int k = std::min(key[(size_t)b], own ? kNone : x.flags[x.at].second), a = 0;
            if (own)
                fl[(size_t)b] &= ~kActive;
            if (!(fl[(size_t)b] & kActive) && k != kNone) {
                if (k <= bound) {
                    fl[(size_t)b] |= kActive;
                    a = 1;
                } else if (!(fl[(size_t)b] & kWaiting)) {
                    fl[(size_t)b] |= kWaiting;
                    a = 2;
                }
            }
            key[(size_t)b] = k;
            x.act.push_back(a);
            if (++x.at == x.flags.size())
                x.st = COUNT2;
            return true;
        }
        case COUNT2: {
            int q = 0;
            for (size_t l = 0; l < x.flags.size(); ++l) {
                if (x.act[l] == 1) {
                    ++q;
                    x.puts.push_back({false, q_tail++, x.flags[l].first});
                } else if (x.act[l] == 2)
                    x.puts.push_back({true, w_tail++, x.flags[l].first});
            }
            pending += q - 1;
            x.st = PUTS2;
            return true;
        }
        case PUTS2:
            return puts(x, POLL);
        case STOP:
            return false;
        }
        return false;
    }
    int run()
    {
        for (long long quiet = 0;;) {
            bool all = true;
            for (Warp &x : w)
                all = all && x.st == STOP;
            if (all)
                break;
            Warp &x = w[(size_t)rnd(nw)];
            if (x.away > 0) {
                --x.away;
                continue;
            }
            if (rnd(400) == 0)
                x.away = rnd(200);
            if (step(x))
                quiet = 0;
            else if (++quiet > 64ll * nw) {
                quiet = 0;
                bool any = false;
                for (Warp &y : w) {
                    y.away = 0;
                    any = step(y) || any;
                }
                if (!any)
                    return 2;
            }
            if (bad)
                return 3;
        }
        for (int b = 0; b < n; ++b)
            if (key[(size_t)b] != kNone || fl[(size_t)b]) {
                bad = "work was left";
                return 3;
            }
        return 0;
    }
};

}  // namespace

int main(int argc, char **argv)
{
    if (argc != 10)
        return 1;
    const int n = atoi(argv[1]), waiting = atoi(argv[2]), warps = atoi(argv[3]), levels = atoi(argv[4]),
              release = atoi(argv[5]), seeds = atoi(argv[6]);
    const unsigned long long slots = strtoull(argv[7], nullptr, 10);
    int worst = 0, stalled = 0;
    for (int s = 0; s < seeds; ++s) {
        Model m;
        m.n = n;
        m.nw = warps;
        m.cap_q = (unsigned long long)n;
        m.cap_w = slots ? slots : fmmgb::waiting_slots(n);
        m.any_raise = atoi(argv[8]) != 0;
        m.keep = atoi(argv[9]) != 0;
        m.stride = release;
        m.budget = 4 * n;
        m.rng.seed((unsigned long long)s + 1);
        m.key.assign((size_t)n, kNone);
        m.fl.assign((size_t)n, 0);
        m.queue.assign((size_t)m.cap_q, 0);
        m.ring.assign((size_t)m.cap_w, 0);
        m.w.resize((size_t)warps);
        for (int b = 0; b < waiting; ++b) {
            m.key[(size_t)b] = 1 + m.rnd(levels);
            m.fl[(size_t)b] = kWaiting;
            m.ring[m.w_tail] = Model::entry(m.w_tail, b);
            ++m.w_tail;
        }
        const int r = m.run();
        stalled += r == 2;
        worst = std::max(worst, r);
        if (m.bad)
            printf("seed %d: %s\n", s, m.bad);
    }
    printf("%d of %d stalled\n", stalled, seeds);
    return worst;
}
