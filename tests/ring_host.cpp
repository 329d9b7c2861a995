// The ring of bsd_ring.cuh on the host: candidate groups as coroutines, one atomic
// step at a time in a seeded order, with groups that stand still for long and a
// clock that jumps, so that groups leave.  Every item drawn must have been pushed
// and not drawn before; every shot must end.  Returns 0, or a code for what failed.
#include <ucontext.h>

#include <cstdlib>
#include <vector>

#include "bsd_ring.cuh"

namespace {

struct Rng {
    uint64_t s;
    uint32_t below(uint32_t n)
    {
        s ^= s >> 12; s ^= s << 25; s ^= s >> 27;
        return (uint32_t)((s * 2685821657736338717ull) >> 33) % n;
    }
};

constexpr size_t kStack = 32 * 1024;
struct Fiber {
    ucontext_t ctx;
    std::vector<char> stack;
    bool done = true;
    long asleep = 0;               // steps it stands still
    int group = 0, lane = 0;       // lane > 0: pushes for its group's selection
    std::vector<uint32_t> push;
};

struct Sim {
    Rng rng;
    int groups, entries, width, shots, rounds;
    ucontext_t main;
    std::vector<Fiber> fibers;     // [groups][1 + kLanes]
    Fiber* cur = nullptr;
    std::vector<uint32_t> ring;
    uint32_t head = 0, tail = 0, mask = 0, left = 0, next = 0;
    std::vector<int> pending, round;
    std::vector<std::vector<char>> out;     // items pushed and not drawn
    unsigned long long clock = 1;
    int jumps = 0, bad = 0;
    long marks = 0;
};
Sim* S;
constexpr int kLanes = 3;

void yield() { swapcontext(&S->cur->ctx, &S->main); }

struct HostRing {
    static uint32_t add(uint32_t* p, uint32_t v) { yield(); const uint32_t o = *p; *p += v; return o; }
    static uint32_t cas(uint32_t* p, uint32_t want, uint32_t v)
    {
        yield();
        const uint32_t o = *p;
        if (o == want) {
            *p = v;
            S->marks += v == bsd::kRingLeft;
        }
        return o;
    }
    static uint32_t and_(uint32_t* p, uint32_t v) { yield(); const uint32_t o = *p; *p &= v; return o; }
    static uint32_t load(const uint32_t* p) { yield(); return *p; }
    static void pause() { yield(); }
    static unsigned long long now() { return S->clock; }
};

void run_lane()
{
    Fiber& f = *S->cur;
    for (uint32_t it : f.push) bsd::ring_push_pair<HostRing>(S->ring.data(), &S->tail, S->mask, it);
    f.push.clear();
    f.done = true;
    yield();
}

void start(Fiber& f, void (*fn)())
{
    f.done = false;
    f.stack.resize(kStack);
    getcontext(&f.ctx);
    f.ctx.uc_stack.ss_sp = f.stack.data();
    f.ctx.uc_stack.ss_size = kStack;
    f.ctx.uc_link = &S->main;
    makecontext(&f.ctx, fn, 0);
}

// the lanes of a group push side by side, the group goes on when all have
void push_all(const std::vector<uint32_t>& items)
{
    Fiber& f = *S->cur;
    Fiber* lanes = &S->fibers[(size_t)f.group * (1 + kLanes) + 1];
    for (size_t k = 0; k < items.size(); ++k) lanes[k % kLanes].push.push_back(items[k]);
    for (int l = 0; l < kLanes; ++l)
        if (!lanes[l].push.empty()) start(lanes[l], run_lane);
    for (int l = 0; l < kLanes; ++l)
        while (!lanes[l].done) yield();
}

void run_group()
{
    Sim& s = *S;
    for (;;) {
        const uint32_t ticket = HostRing::add(&s.head, 1u);
        const uint32_t it = bsd::ring_draw<HostRing>(s.ring.data(), s.mask, &s.left, ticket);
        if (it == bsd::kRingEmpty) break;
        const int a = bsd::ring_entry(it), c = bsd::ring_child(it);
        if (it == bsd::kRingLeft || a >= s.entries || c >= 2 * s.width) { s.bad = 1; break; }
        if (!s.out[a][c]) { s.bad = 2; break; }
        s.out[a][c] = 0;
        for (uint32_t k = s.rng.below(s.rng.below(4) ? 12 : 1500); k > 0; --k) yield();   // the child's BP
        if (--s.pending[a] > 0) continue;
        std::vector<uint32_t> items;
        auto put = [&](int n) {
            s.pending[a] = n;
            for (int k = 0; k < n; ++k) s.out[a][k] = 1;
            for (int k = 0; k < n; k += 2) items.push_back(bsd::ring_item(a, k));        // (a path's two children)
        };
        if (s.round[a] < s.rounds && s.rng.below(8) != 0) {
            ++s.round[a];
            put(2 * (1 + (int)s.rng.below((uint32_t)s.width)));
            push_all(items);
        } else {
            if ((int)s.next < s.shots) {
                ++s.next;
                s.round[a] = 1;
                put(2);
                push_all(items);
            }
            HostRing::add(&s.left, (uint32_t)-1);
        }
    }
    S->cur->done = true;
    yield();
}

}  // namespace

// stalls: one in this many steps puts the running fiber to sleep for up to `sleep`
// steps; jumps: how often the clock passes the groups' idle limit
extern "C" int ring_host(uint64_t seed, int groups, int entries, int width, int shots, int rounds, int stalls, int sleep,
                         int jumps, long max_steps, long* left_marks)
{
    Sim s;
    S = &s;
    s.rng.s = seed * 0x9e3779b97f4a7c15ull + 1;
    s.groups = groups; s.entries = entries; s.width = width; s.shots = shots; s.rounds = rounds;
    uint32_t slots = 4;
    while (slots < 2u * (uint32_t)entries * (uint32_t)width) slots *= 2;
    if ((uint32_t)groups > slots) groups = (int)slots;                         // the others leave at once
    s.mask = slots - 1;
    s.ring.assign(slots, bsd::kRingEmpty);
    s.pending.assign(entries, 2);
    s.round.assign(entries, 1);
    s.out.assign(entries, std::vector<char>(2 * (size_t)width, 0));
    const int cnt = entries < shots ? entries : shots;
    for (int q = 0; q < 2 * cnt; ++q) { s.ring[q] = bsd::ring_item(q / 2, q & 1); s.out[q / 2][q & 1] = 1; }
    s.tail = 2u * (uint32_t)cnt;
    s.left = (uint32_t)shots;
    s.next = (uint32_t)cnt;
    s.fibers.resize((size_t)groups * (1 + kLanes));
    for (size_t q = 0; q < s.fibers.size(); ++q) {
        s.fibers[q].group = (int)(q / (1 + kLanes));
        s.fibers[q].lane = (int)(q % (1 + kLanes));
        if (s.fibers[q].lane == 0) start(s.fibers[q], run_group);
    }
    for (long step = 0; step < max_steps && !s.bad; ++step) {
        std::vector<int> live;
        bool running = false;
        for (size_t q = 0; q < s.fibers.size(); ++q) {
            Fiber& f = s.fibers[q];
            if (f.done) continue;
            running = true;
            if (f.asleep > 0) --f.asleep; else live.push_back((int)q);
        }
        if (!running) break;
        if (s.jumps < jumps && s.rng.below(300) == 0) { s.clock += bsd::kIdleNs + 2; ++s.jumps; }
        if (live.empty()) continue;
        s.cur = &s.fibers[(size_t)live[s.rng.below((uint32_t)live.size())]];
        swapcontext(&s.main, &s.cur->ctx);
        if (stalls > 0 && s.rng.below((uint32_t)stalls) == 0) s.cur->asleep = (long)s.rng.below((uint32_t)sleep);
    }
    if (left_marks) *left_marks = s.marks;
    if (s.bad) return s.bad;
    return s.left == 0 ? 0 : 3;                                                // a shot was left behind
}
