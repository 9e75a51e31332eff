// Which calls of general layout the scalar fiber body serves faster than the span body
// (plain arithmetic, also for the host tests).
//
// Figures: time of the span body over the scalar one's, device time on one GB300; "large"
// is 2^25 elements.  E is the number of elements of the larger of X and Y.
#pragma once
#include <stdint.h>

namespace kron {

struct SpanCall {
    int D, es, N;            // kind, bytes per element, largest extent
    int64_t nx, ny, batch;   // elements of one operand and of one result; instances
    bool square;             // every extent N
    bool up_one;             // every mode of Y one longer than X's
    bool beta;               // beta != 0
    bool x_packed;           // square, packed, aligned X: the scalar body copies it in bulk
    bool y_packed;           // packed Y, aligned or not
    bool y_aligned;          // ... on 16 bytes
    int yvec;                // elements per store of the scalar body
    int row_bytes;           // column stride of Y
};

inline bool scalar_body_faster(const SpanCall& c) {
    const int64_t E = c.batch * (c.nx > c.ny ? c.nx : c.ny);
    if (c.N == 1) return true;                             // 1.05-1.25
    // 3-D, old values of Y in rows of a few elements (n = 5: 1.09, 6: 1.03; 7: 0.86)
    if (c.D == 3 && c.beta && c.N <= 6) return true;
    if (c.x_packed && c.y_aligned) return false;           // odd n of 16-bit storage: 0.3-1.0
    // Calls of a few instances are all latency, which the bulk copy's way through the ring
    // adds to (1 to 16 instances: 1.05-1.5 up to here, 0.4-1.0 beyond), n = 2 the longest
    // (1.07-1.2).
    if (E <= (c.N == 2 ? 65536 : 512)) return true;
    // 16-bit storage without an instantiation of its own.
    if (c.es == 2 && !c.square) {
        // 3-D up to 10 nodes needs this many elements to pay (6 -> 10 at 2^17: 1.4, 5 -> 9 1.4; at
        // 2^20 0.6-1.0; 2-D n = 3, 4: 1.05-1.15), 5 -> 6 never does (large 1.07).
        if (E <= 2048) return true;                        // (2-D 13 -> 11, 4 instances: 1.25)
        if (c.D == 3 && (c.N == 6 || (c.N <= 10 && E < (1 << 20)))) return true;
        if (c.D == 2 && c.N <= 4 && E <= (1 << 17)) return true;
        // With old values, to larger results (3-D 9 -> 10: 1.13, 13 -> 14: 1.13, 10 -> 14: 1.06,
        // 6 -> 7: 1.28; 2-D 2 -> 3: 1.11, 5 -> 6: 1.24; 9 -> 10: 0.90; to smaller ones 0.5-0.9)
        if (c.beta && c.ny > c.nx) {
            if (c.D == 3 ? c.N % 2 == 0 || c.up_one : c.up_one && c.N <= 8) return true;
        }
    }
    // Operands that the scalar body copies in bulk too: what is left is how Y is written.
    if (c.x_packed && c.beta) {
        // Old values, large: FP32 2-D n = 5: 1.5, 9: 1.2-1.3, 11: packed Y 1.03, padded 0.86-0.98,
        // 12: 0.7-0.9, 13: 1.0-1.1; 3-D n = 7: 1.3-1.7, 12: 1.0-1.7, 14: 1.25, 15: packed 1.07-1.16,
        // padded 0.9, 16: 0.8-1.0; 16-bit 2-D n = 5-8: 0.95-1.4, 9: packed 1.06-1.24, padded
        // 0.7-0.9, 12: 0.6-1.04, 10, 14, 16 with vector stores 1.07-1.28, without 0.5-0.95; 3-D
        // n = 5: 1.3-1.4, 13: 1.1-1.3, 16: 0.5-1.0.  100 instances: all n 1.0-1.5.
        if (c.D == 3) return c.N <= (c.y_packed ? 15 : 14) || E < (1 << 19);
        if (c.es == 4)
            return (c.N >= 3 && c.N <= 9) || (c.y_packed && (c.N <= 11 || c.N == 13) && c.N >= 3) || E < (1 << 17);
        return (c.N >= 5 && c.N <= 8) || (c.y_packed && c.N == 9) ||
               (c.yvec >= 2 && (c.N == 10 || c.N >= 14)) || E < (1 << 19);
    }
    if (c.x_packed && !c.y_packed) {
        // Y with gaps.  3-D n = 5: 1.0-1.4, n = 8: 0.75-1.06, n = 9-13 in FP32 1.0-1.15 (11: 0.9-1.0),
        // even n with vector stores 1.1-1.5 (odd stores 0.5-1.0); 2-D n = 5, 6 in rows of less than
        // a sector 1.04-1.24 (longer rows 0.8-1.06), 16-byte stores at n = 12, 16 1.04-1.16.
        if (c.N <= 8 && E < (1 << 17)) return true;
        if (c.D == 3)
            return (c.N >= 3 && c.N <= 7) || (c.yvec >= 2 && c.N >= 10 && c.N < 16) ||
                   (c.es == 4 && c.N >= 9 && c.N <= 13 && c.N != 11);
        return ((c.N == 5 || c.N == 6) && c.row_bytes < 32) || (c.es == 4 && c.yvec == 4 && c.N >= 12);
    }
    // Packed results off a 16-byte boundary: 0.4-1.0, but 3-D n = 12 with vector stores 1.07-1.28.
    return c.x_packed && c.D == 3 && c.N == 12 && c.yvec >= 2;
}

// Whether the span body is asked at all: every general layout, and packed calls of odd n
// with 16-bit storage and beta = 0, unless a tile or a depth is set for them (those are the
// scalar body's).
inline bool span_body_asked(bool y_aligned, int N, bool half, bool beta, bool tile_set) {
    return !y_aligned || (N % 2 == 1 && half && !beta && !tile_set);
}

}  // namespace kron
