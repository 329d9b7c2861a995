// bsd_ring.cuh -- the ring of beam items: how candidate groups pass children on.
//
// Written over a policy Ops (atomics, a relaxed load, a pause, a clock), so that
// the host can run the same code in any interleaving; the kernels use GpuRing
// (bsd_kernels.cu).
//
// A group draws a ticket (one add to the head) and waits at the ticket's slot; a
// pusher takes the next ticket of the tail and puts its item there.  An item is
// whatever comes first at a slot: tickets of several laps may wait at one slot
// while a pusher is between its two steps, and items are interchangeable.  What
// must hold is the count: every ticket drawn is matched by one push, or cancelled
// by one mark.
//   * A group that has waited kIdleNs leaves: it puts the mark kRingLeft into its
//     empty slot.  The pusher that meets the mark takes it away and pushes its
//     item at another ticket.  A group of a later lap that meets the mark leaves it
//     (atomicAnd takes an item and keeps a mark).
//   * A pusher never puts an item over another one: it waits for the slot's group.
//     That group only has to take the item, since no group holds a ticket while it
//     selects or pushes (an item undrawn has a group: at most as many items are
//     undrawn as the ring has slots, so the ticket one lap before the pusher's has
//     been drawn).  A group that held a ticket while it pushed would make the
//     pusher wait for it; one that put its item over the other and pushed that
//     again would leave one group at the slot waiting for ever.
// No item is lost and no wait is unbounded.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define BSD_RING_FN __host__ __device__ __forceinline__
#define BSD_RING_DEV __device__ __forceinline__
#else
#define BSD_RING_FN inline
#define BSD_RING_DEV inline
#endif

namespace bsd {

// an item of the ring: child c (< 2w <= 128) of window entry a (< 2^20), never
// one of the two marks
constexpr uint32_t kRingEmpty = 0u;
constexpr uint32_t kRingLeft = 0x80000000u;   // the group that held this slot's ticket has left
BSD_RING_FN uint32_t ring_item(int a, int c) { return (((uint32_t)a << 7) | (uint32_t)c) + 1u; }
BSD_RING_FN int ring_entry(uint32_t it) { return (int)((it - 1u) >> 7); }
BSD_RING_FN int ring_child(uint32_t it) { return (int)((it - 1u) & 127u); }
BSD_RING_FN bool ring_has_item(uint32_t v) { return (v & ~kRingLeft) != 0u; }

constexpr unsigned long long kIdleNs = 1000ull * 1000 * 1000;
constexpr unsigned long long kStuckNs = 16ull * kIdleNs;   // past any wait that can come about

// an item whose ticket's slot holds `old`, not kRingEmpty
template <class Ops>
BSD_RING_DEV void ring_settle(uint32_t* ring, uint32_t* tail, uint32_t mask, uint32_t* slot, uint32_t item, uint32_t old)
{
    unsigned long long t0 = 0ull;
    for (;;) {
        uint32_t want = old == kRingLeft ? kRingLeft : kRingEmpty;
        if (ring_has_item(old)) {                              // its group is about to take it
            Ops::pause();
            const unsigned long long t = Ops::now();
            if (t0 == 0ull) t0 = t;
            else if (t - t0 > kStuckNs) want = old;
        }
        old = Ops::cas(slot, want, want == kRingLeft ? kRingEmpty : item);
        if (old != want) continue;
        if (want == kRingEmpty) return;
        if (want != kRingLeft) item = want;                    // (past kStuckNs: pushed in its place)
        slot = ring + (Ops::add(tail, 1u) & mask);
        t0 = 0ull;
        old = Ops::cas(slot, kRingEmpty, item);
        if (old == kRingEmpty) return;
    }
}

// push item and item + 1, the two children of a path: two tickets in one step, both
// slots tried before either is waited for
template <class Ops>
BSD_RING_DEV void ring_push_pair(uint32_t* ring, uint32_t* tail, uint32_t mask, uint32_t item)
{
    const uint32_t t = Ops::add(tail, 2u);
    uint32_t* const s0 = ring + (t & mask);
    uint32_t* const s1 = ring + ((t + 1u) & mask);
    const uint32_t o0 = Ops::cas(s0, kRingEmpty, item), o1 = Ops::cas(s1, kRingEmpty, item + 1u);
    if (o0 != kRingEmpty) ring_settle<Ops>(ring, tail, mask, s0, item, o0);
    if (o1 != kRingEmpty) ring_settle<Ops>(ring, tail, mask, s1, item + 1u, o1);
}

// the item of a ticket, or kRingEmpty when every shot has ended (*left = 0) or
// none came for kIdleNs
template <class Ops>
BSD_RING_DEV uint32_t ring_draw(uint32_t* ring, uint32_t mask, const uint32_t* left, uint32_t ticket)
{
    uint32_t* const slot = ring + (ticket & mask);
    uint32_t it = Ops::and_(slot, kRingLeft);
    unsigned long long t0 = 0ull;
    for (unsigned spins = 0; !ring_has_item(it); ++spins) {
        if ((spins & 3u) == 0u && Ops::load(left) == 0u) return kRingEmpty;
        if (spins >= 4u) Ops::pause();
        if ((spins & 63u) == 0u) {
            const unsigned long long t = Ops::now();
            if (t0 == 0ull) t0 = t;
            else if (t - t0 > kIdleNs && (Ops::cas(slot, kRingEmpty, kRingLeft) == kRingEmpty || t - t0 > kStuckNs))
                return kRingEmpty;
        }
        it = Ops::load(slot);
        if (ring_has_item(it)) it = Ops::and_(slot, kRingLeft);
    }
    return it;
}

}  // namespace bsd
