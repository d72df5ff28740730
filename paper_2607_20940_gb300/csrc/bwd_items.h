// Bookkeeping of the persistent bf16 backward's items (attn_bwd_tc.cu), free of
// CUDA so that the host can run it too.
#pragma once

#include <stdint.h>
#include <string.h>

#include "../../include/msf.h"

#ifdef __CUDACC__
#define MSF_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define MSF_HOST_DEVICE inline
#endif

namespace msf {

// The barrier that says that a CTA's k-th item is done, and the parity of its
// phase there. A parity wait can tell a phase only from the one before it, and
// item k - 1 may be done by the time the producer, about to load item k, asks for
// item k - 2: on one barrier "both done" would look like "neither done". With a
// barrier per item parity, item k is the next to complete on the one asked, and
// it has not been loaded yet.
constexpr int kDoneBars = 2;
MSF_HOST_DEVICE int done_bar(int k) { return k & 1; }
MSF_HOST_DEVICE uint32_t done_parity(int k) { return (uint32_t)((k >> 1) & 1); }

// The items of every CTA: CTA c takes item[first[c]], ..., item[first[c + 1] - 1].
constexpr int kMaxOrderCtas = 160, kMaxOrderItems = 2048;
struct BwdOrder {
    int on;  // 0: rounds of alternating direction
    uint16_t first[kMaxOrderCtas + 1];
    uint16_t item[kMaxOrderItems];
};
// Equal items of a launch.
struct ItemClass {
    int kind, group, count;
    int blocks;  // MMA blocks of 128x128xD: 3 per K/V tile of a dq item, 4 per query tile of a dK/dV item
    int ns;      // what an item takes, as measured
    int base;    // its first item
};

// Gives every item, longest first, to the CTA that would be free first, where
// that ends the launch at least a hundredth and a microsecond earlier than the
// rounds of alternating direction: those keep neighbouring tiles of a head and
// items of one kind together, and are near enough once a CTA has a dozen items.
// New loads of a class only grow, so two sorted queues hold the CTAs and an item
// costs the host a few nanoseconds. Forward and backward, rounds / placed: a fine
// and a coarse state of 40 x 36 tokens, 16 heads x 128, 278.6 / 238.0 us (576
// items); 46 x 26, three frames a state, 3 heads x 64, 239.7 / 220.0. (8 x 39 of four
// streams, 480 items, and the 480p layer, 1044, stay below the line.)
inline void place_items(BwdOrder& o, const ItemClass* cl, int n, int total, int ctas) {
    o.on = 0;
    if (total <= ctas || total > kMaxOrderItems || ctas > kMaxOrderCtas) return;
    struct Cta {
        long long load;
        int c;
    };
    Cta old[kMaxOrderCtas], grown[kMaxOrderItems], rest[kMaxOrderCtas];
    long long rounds[kMaxOrderCtas];
    uint8_t cta_of[kMaxOrderItems];  // by item
    uint16_t taken[kMaxOrderItems];  // items, longest first
    for (int c = 0; c < ctas; ++c) {
        old[c] = {0, c};
        rounds[c] = 0;
    }
    int by_ns[2 * MSF_MAX_GROUPS];
    for (int k = 0; k < n; ++k) {
        int at = k;
        for (; at > 0 && cl[by_ns[at - 1]].ns < cl[k].ns; --at) by_ns[at] = by_ns[at - 1];
        by_ns[at] = k;
        for (int x = 0; x < cl[k].count; ++x) {
            const int r = (cl[k].base + x) / ctas, c = (cl[k].base + x) % ctas;
            rounds[r & 1 ? ctas - 1 - c : c] += cl[k].ns;
        }
    }
    memset(o.first, 0, sizeof(o.first));
    int done = 0;
    for (int k = 0; k < n; ++k) {
        const ItemClass& ic = cl[by_ns[k]];
        int i = 0, head = 0, tail = 0;
        auto lightest = [&] {
            return head == tail || (i < ctas && old[i].load <= grown[head].load) ? old[i++] : grown[head++];
        };
        for (int x = 0; x < ic.count; ++x) {
            Cta t = lightest();
            t.load += ic.ns;
            grown[tail++] = t;
            cta_of[ic.base + x] = (uint8_t)t.c;
            taken[done++] = (uint16_t)(ic.base + x);
            ++o.first[t.c + 1];
        }
        for (int m = 0; m < ctas; ++m) rest[m] = lightest();
        memcpy(old, rest, sizeof(old));
    }
    long long end = 0;
    for (int c = 0; c < ctas; ++c) end = rounds[c] > end ? rounds[c] : end;
    const long long gain = end - old[ctas - 1].load;
    if (gain < 1000 || 100 * gain < end) return;
    o.on = 1;
    for (int c = 0; c < ctas; ++c) o.first[c + 1] = (uint16_t)(o.first[c + 1] + o.first[c]);
    uint16_t at[kMaxOrderCtas];
    memcpy(at, o.first, sizeof(at));
    for (int x = 0; x < total; ++x) o.item[at[cta_of[taken[x]]]++] = taken[x];
}

}  // namespace msf
