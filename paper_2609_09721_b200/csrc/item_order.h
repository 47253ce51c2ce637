// The order in which the persistent CTAs of the fused forward take the items (query tile, head) of a packed batch.
//
// CTAs walk the item table in turn: a round of it has a place for every CTA, every other round in reverse.  With the items one after the
// other, heaviest first, a CTA that starts with one far heavier than the rest still gets as many others as its neighbours.  Handed out as
// CTAs become free, as the hardware does with one CTA per item, they would not.  So where that is unbalanced each item goes to the CTA that has
// the least so far, and the rounds that a CTA has nothing in are left empty.
//
// Measured, us, one CTA per item / one after the other / in this order: 2 heads, not causal, 3000 tokens and 60 sequences of up to 500
// 39.6 / 47.1 / 40.0; 4 heads, 6000 and 60 of up to 500 111 / 122 / 106; 2 heads, causal, 12000 and 30 of up to 1500 99.7 / 112.6 / 96.5; one
// head, not causal, 6000 and 30 of up to 1500 53.9 / 61.6 / 54.4.
#pragma once

#include <stdint.h>

#include <algorithm>
#include <vector>

namespace efq {

struct ItemRun { int32_t tiles, count; };      // items one after the other that walk as many KV tiles each

constexpr int kItemCost = 3;                   // what an item costs beside its tiles, in tiles
// Up to this many items (16 for each of 148 CTAs) it is tried: with more, the last ones are small against a CTA's total.
constexpr int64_t kOrderMaxItems = 16 * 148;
// Items for which ordering has to save a tile: they take the host some 0.5 us, a tile 0.7 to 1.3
constexpr int64_t kOrderItemsPerTile = 64;
// Places of the item table for n items, in order or not.  More items never take fewer: a workspace that is large enough for a batch
// stays so for a smaller one, though that may be ordered and the larger one not.
constexpr int64_t order_places(int64_t n_items) { return n_items + 2 * std::min(n_items, kOrderMaxItems); }

// Place of a CTA's item number k
constexpr int64_t place_in_turn(int64_t k, int64_t cta, int64_t ctas) { return k * ctas + (k & 1 ? ctas - 1 - cta : cta); }

// Fills places[0 .. result) with the items of the table, -1 in an empty place, if items one after the other would leave a CTA with 2 %
// more than need be, and enough more to be worth it; else, or if that takes more than order_places(), returns 0.  places has room
// for order_places() of them.
inline int64_t order_items(const std::vector<ItemRun>& runs, int64_t n_items, int ctas, int32_t* places)
{
    if (ctas <= 0 || n_items <= ctas || n_items > kOrderMaxItems) return 0;
    std::vector<int32_t> work(3 * static_cast<size_t>(ctas), 0);
    int32_t* const load = work.data();
    int64_t total = 0;
    int32_t heaviest = 0;
    int at = 0;
    bool reverse = false;
    for (const ItemRun& r : runs) {
        const int32_t cost = r.tiles + kItemCost;
        heaviest = std::max(heaviest, cost);
        total += int64_t{r.count} * cost;
        if (total > INT32_MAX) return 0;
        for (int32_t left = r.count; left > 0;) {            // round by round
            const int m = std::min(left, ctas - at), first = reverse ? ctas - at - m : at;
            for (int c = first; c < first + m; ++c) load[c] += cost;
            left -= m;
            at += m;
            if (at == ctas) { at = 0; reverse = !reverse; }
        }
    }
    const int64_t least = std::max<int64_t>(heaviest, (total + ctas - 1) / ctas), excess = *std::max_element(load, load + ctas) - least;
    if (excess * 50 <= least || excess * kOrderItemsPerTile <= n_items) return 0;

    // CTAs in buckets by what they have, the buckets in a ring that holds the heaviest item (in coarser steps from 1024 tiles on)
    int shift = 0;
    while (heaviest >> shift >= 1024) ++shift;
    const int ring = std::max(1, heaviest >> shift) + 1;
    std::vector<int32_t> bucket(ring, -1);
    int32_t *const below = work.data() + ctas, *const taken = below + ctas;
    for (int c = ctas - 1; c >= 0; --c) { below[c] = bucket[0]; bucket[0] = c; }
    const int64_t room = order_places(n_items);
    std::fill(places, places + room, -1);
    int64_t used = 0;
    int32_t item = 0;
    at = 0;
    for (const ItemRun& r : runs) {
        const int cost = std::max(1, (r.tiles + kItemCost) >> shift);
        for (int32_t k = 0; k < r.count; ++k, ++item) {
            while (bucket[at] < 0) at = at + 1 == ring ? 0 : at + 1;
            const int32_t c = bucket[at], to = at + cost < ring ? at + cost : at + cost - ring;
            bucket[at] = below[c];
            below[c] = bucket[to]; bucket[to] = c;
            const int64_t place = place_in_turn(taken[c]++, c, ctas);
            if (place >= room) return 0;
            places[place] = item;
            used = std::max(used, place + 1);
        }
    }
    return used;
}

}  // namespace efq
