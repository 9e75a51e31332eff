// Which tiles of a batch can be brought by bulk copies of whole 16-byte granules (plain
// arithmetic on addresses, also for the host tests).
#pragma once
#include <stdint.h>

namespace kron {

// X starts at address x0; instance p spans xspan elements of es bytes from x0 + p ldxp es,
// and a tile is P of them.  A copy takes every granule that holds a byte of its tile, so
// the first tiles (head) and the last ones (tail) may reach bytes that are not X's; there the
// elements outside whole granules are loaded one by one.  One tile each as a rule, a second
// one where the first or last tile is shorter than a granule.  copies = 0 where there are
// more, which strides of a few bytes bring about.
struct SpanEdges {
    int head, tail, copies;
};
inline SpanEdges span_edges(uintptr_t x0, int64_t batch, int64_t P, int64_t ldxp, int64_t xspan, int es) {
    const int64_t ntiles = (batch + P - 1) / P;
    const uintptr_t x1 = x0 + (uintptr_t)(((batch - 1) * ldxp + xspan) * es);
    auto before = [&](int64_t t) { return ((x0 + (uintptr_t)(t * P * ldxp * es)) & ~(uintptr_t)15) < x0; };
    auto beyond = [&](int64_t t) {
        const int64_t last = (t + 1) * P < batch ? (t + 1) * P - 1 : batch - 1;
        return ((x0 + (uintptr_t)((last * ldxp + xspan) * es) + 15) & ~(uintptr_t)15) > x1;
    };
    SpanEdges e{0, 0, 1};
    while (e.tail < 2 && e.tail < ntiles && beyond(ntiles - 1 - e.tail)) ++e.tail;
    while (e.head < 2 && e.head < ntiles - e.tail && before(e.head)) ++e.head;
    if (e.head + e.tail < ntiles && (before(e.head) || beyond(ntiles - 1 - e.tail))) e.copies = 0;
    return e;
}

}  // namespace kron
