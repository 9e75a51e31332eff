// CUDA-core kernels for general layouts: rectangular components, padded or
// transposed operands, results with gaps (FP32 arithmetic; FP32 or 16-bit storage).
//
// A general layout is still a run of memory per tile: the span from the first
// element of a tile's first operand to the last element of its last one, padding
// included, arrives as ONE bulk copy (TMA) into a ring of buffers and is addressed
// in shared memory with the caller's own strides.  A copy takes whole 16-byte granules; the
// tiles at either end of X, where such a granule would hold bytes that are not X's, go to
// CTAs of their own that load the elements there one by one (a test for them inside the tile
// loop cost every shape 5-20%).  Padding inside a span costs little: DRAM delivers whole 32-byte
// sectors anyway.  (The fiber kernel this
// replaces loads each element with its own division and bounds test, with nothing
// in flight behind the arithmetic; spans mostly made of gaps are left to it.)
//
// The contractions run on the exact extents: a stage reads fibers of xe elements
// (compile-time bound NI, the longest) and walks the output rows in packed pairs
// (fma.rn.f32x2 with the coefficient pair (M[2r, l], M[2r+1, l]) from the parameter
// bank), four rows at a time up to the mode's own extent, so an 8 -> 12 product
// spends no work on padding it to 12 x 12.  A thread takes two fibers at a time:
// every coefficient read feeds two packed FMAs.
//
// On chip there is a ring of operand slots and one exchange buffer E per CTA:
//
//   2-D   stage 1: fibers along the stored rows l of X, contracted over the stored
//                  columns: W(l, o) at o + KP l of E
//         stage 2: fibers o, contracted over l.  For op(X) = X the first product is
//                  with M2 and the second gives Y's columns; for op(X) = X^T the
//                  first is with M1 and the second gives Y's rows, so the transposed
//                  operand is read along its stored rows just the same.
//   3-D   stage A (mode 3)  T(i, j, k) at k + KP i + JS j of E
//         stage B (mode 2)  U(i, j, k) in place: a fiber's outputs over its inputs
//         stage C (mode 1)  Y(i, j, k)
//
// Pairs (STS.64) go out KP = 2 mod 4 words apart and every fiber is read with
// consecutive lanes on consecutive words, or (stage C) JS = 2 mod 32 words apart.
// The results are staged in the slot their operands came in (dead by then).  Packed
// Y with beta = 0 leaves as one bulk copy per tile; any other Y is written by the
// whole CTA in row chunks of up to 16 bytes, where beta and the rounding to the
// storage type are applied, so old values of Y are read in whole sectors too.  A
// slot is refilled once its results have left, one tile later.
//
// Measured against the fiber kernel on one GB300 (device time per call): 3-D 8 -> 12,
// 100,003 instances: 713 -> 182 us (4.9 TB/s, 32 TFLOP/s; HBM floor 132 us); 2-D n = 16
// row-major (op(X) = X^T) in rows of 20, 2^18 instances: 390 -> 197 us (padding included
// the call moves 671 MB, and the half-written sectors of Y are read back: about 120 us);
// the same without padding: 94 us; bf16 n = 15: 576 -> 207 us in 2-D and 600 -> 340 us in
// 3-D (120 M elements).  What bounds it now: shared memory (63% of its peak at 8 -> 12)
// and the barriers between the stages; instantiating the extents took 8 -> 12 from 90 to
// 70 us at a third of that batch (index arithmetic), two fibers per thread and the larger
// tile from 78 to 70.  Two slots and about four CTAs per SM measured best (three to six
// tried; one slot 10-15% slower in 2-D).
#pragma once

#include <string.h>

#include <algorithm>

#include "kron_pair.cuh"
#include "kron_span_copy.h"
#include "kron_span_rule.h"

namespace kron {

constexpr int kSpanThreads = 128;
constexpr int kSpanRing = 2;

// f / d for f d < 2^32 (mul = ceil(2^32 / d); d = 1 has no 32-bit multiplier).
struct FastDiv {
    unsigned d, mul;
    __device__ __forceinline__ unsigned div(unsigned f) const { return d == 1 ? f : __umulhi(f, mul); }
};
inline FastDiv fast_div(unsigned d) {
    return FastDiv{d, d == 1 ? 0u : (unsigned)((0x100000000ull + d - 1) / d)};
}

struct SpanArgs {
    f2 m[3][8 * kMaxN];           // stage s: rows (2r, 2r+1) of column l at r + 8 l, zero-padded
    const void* X;
    void* Y;
    int64_t ldxp, ldyp;           // elements
    int ntiles, last;             // tiles; instances of the last one
    int xs_col, xs_plane;         // strides of the contracted / plane index of X (elements)
    int xspan;                    // elements spanned by one operand
    int head, tail;               // first / last tiles whose copies would reach outside X
    int ce[3];                    // contracted extent of each stage
    int oe[3];                    // output extent of each stage
    int kp, js;                   // strides of the exchange buffer
    int eq;                       // its words per instance
    FastDiv fib[3];               // fibers per instance of each stage
    FastDiv in[3];                // fastest fiber index of each stage
    // Y
    int ye1, ny;                  // rows and elements of one result
    int sf, so;                   // staged: fiber f, output o at sf f + so o
    int sq;                       // staged: instance stride
    int srow;                     // staged: row stride (copy by the CTA)
    FastDiv chunks;               // chunks per row
    FastDiv rows, cols;           // rows per result; columns per plane (3-D)
    int ldy, ldy2, ldyp32;
    int nk;                       // planes per result
    int dc, dj, dk, dq;           // kSpanThreads chunks in mixed radix (chunk, row, plane, instance)
    int P;
    int slot_bytes;
    int vec;                      // elements per chunk (4, 2, 1)
    int bulk;                     // packed Y, beta = 0: bulk stores
    int beta_zero, alpha_one;
    float alpha, beta;
    unsigned* err;
};

// Row length of the first stage's outputs: even, 2 mod 4, room for the padding row.
__host__ __device__ constexpr int span_kp(int rows) {
    return rows + (rows & 1) + ((rows + (rows & 1)) % 4 == 2 ? 0 : 2);
}

// Extents and exchange-buffer strides: compile-time constants when every mode maps NI
// elements to NO (the kernel's instantiations for NO > 0), else from the arguments.
template <int NI, int NO, int D>
struct SpanShape {
    static constexpr bool fixed = NO > 0;
    static constexpr int KP = span_kp(NO);
    static constexpr int JS = stride_mod32(KP * NI, 2);
    static constexpr int EQ = D == 2 ? stride_mod32(KP * NI, (NO + 1) / 2 * 2 % 32) : JS * (NI > NO ? NI : NO);
    const SpanArgs& a;
    __device__ __forceinline__ int rows(int s) const { return fixed ? NO : a.oe[s]; }
    __device__ __forceinline__ int kp() const { return fixed ? KP : a.kp; }
    __device__ __forceinline__ int js() const { return fixed ? JS : a.js; }
    __device__ __forceinline__ int eq() const { return fixed ? EQ : a.eq; }
    // fibers per instance of stage s, and the quotient by it
    static constexpr int fib_of(int s) {
        return D == 2 ? (s == 0 ? NI : NO) : (s == 0 ? NI * NI : s == 1 ? NI * NO : NO * NO);
    }
    __device__ __forceinline__ int fib(int s) const { return fixed ? fib_of(s) : (int)a.fib[s].d; }
    __device__ __forceinline__ int div_fib(int s, int f) const {
        return fixed ? f / (fixed ? fib_of(s) : 1) : (int)a.fib[s].div(f);
    }
    // extent of the fastest fiber index of stage s (3-D), and the quotient by it
    static constexpr int in_of(int s) { return s == 0 ? NI : NO; }
    __device__ __forceinline__ int in(int s) const { return fixed ? in_of(s) : (int)a.in[s].d; }
    __device__ __forceinline__ int div_in(int s, int r) const {
        return fixed ? r / (fixed ? in_of(s) : 1) : (int)a.in[s].div(r);
    }
};

// y = M x for NF fibers, four output rows per step: out(v, o, y01, y23) takes rows
// o..o+3 of fiber v.
template <int NI, int NF, typename Out>
__device__ __forceinline__ void span_contract(const f2* __restrict__ M, const float (&x)[NF][NI], int rows, Out out) {
#pragma unroll
    for (int c = 0; c < kMaxN / 4; ++c) {
        if (4 * c >= rows) break;
        f2 y0[NF], y1[NF];
#pragma unroll
        for (int v = 0; v < NF; ++v) {
            const f2 xx = f2_pack(x[v][0], x[v][0]);
            y0[v] = fmul2(M[2 * c], xx);
            y1[v] = fmul2(M[2 * c + 1], xx);
        }
#pragma unroll
        for (int l = 1; l < NI; ++l) {
#pragma unroll
            for (int v = 0; v < NF; ++v) {
                const f2 xx = f2_pack(x[v][l], x[v][l]);
                y0[v] = ffma2(M[2 * c + 8 * l], xx, y0[v]);
                if (4 * c + 2 < rows) y1[v] = ffma2(M[2 * c + 1 + 8 * l], xx, y1[v]);
            }
        }
#pragma unroll
        for (int v = 0; v < NF; ++v) out(v, 4 * c, y0[v], y1[v]);
    }
}

// Two fibers per thread and step, except with runtime extents above 8: there two of them
// do not fit in the 128 registers that four CTAs per SM leave a thread (NI = 16: up to 1168
// bytes of spill stores and 2496 of loads; one fiber: none, and calls of that body take
// 0.43-1.0 of the time; NI = 4 and 8 have room for two, and one is up to 1.2x slower).
template <int NI, int NO>
constexpr bool span_two() { return NO > 0 || NI <= 8; }

// One stage over F fibers.  in(f, x) reads fiber f and returns where its outputs go;
// out(dst, o, y01, y23) writes rows o..o+3.
template <int NI, int NO, typename In, typename Out>
__device__ __forceinline__ void span_stage_run(const f2* M, int F, int rows, In in, Out out) {
    if constexpr (!span_two<NI, NO>()) {
        for (int f = threadIdx.x; f < F; f += kSpanThreads) {
            float x[1][NI];
            auto* d0 = in(f, x[0]);
            span_contract<NI, 1>(M, x, rows, [&](int, int o, f2 y0, f2 y1) { out(d0, o, y0, y1); });
        }
        return;
    }
    for (int f = threadIdx.x; f < F; f += 2 * kSpanThreads) {
        if (f + kSpanThreads < F) {
            float x[2][NI];
            auto* d0 = in(f, x[0]);
            auto* d1 = in(f + kSpanThreads, x[1]);
            span_contract<NI, 2>(M, x, rows, [&](int v, int o, f2 y0, f2 y1) { out(v ? d1 : d0, o, y0, y1); });
        } else {
            float x[1][NI];
            auto* d0 = in(f, x[0]);
            span_contract<NI, 1>(M, x, rows, [&](int, int o, f2 y0, f2 y1) { out(d0, o, y0, y1); });
        }
    }
}

// A fiber of ce <= NI elements, `stride` apart (EXACT: ce = NI).
template <int NI, bool EXACT, typename S>
__device__ __forceinline__ void span_load(const S* p, int stride, int ce, float (&x)[NI]) {
#pragma unroll
    for (int l = 0; l < NI; ++l) x[l] = (EXACT || l < ce) ? load_cvt<float, S>(p[stride * l]) : 0.f;
}

// Output rows o..o+3 of the first stage: adjacent pairs (KP has room for an even
// number of outputs).
__device__ __forceinline__ void span_put(float* dst, int o, int rows, f2 y0, f2 y1) {
    *reinterpret_cast<f2*>(dst + o) = y0;
    if (o + 2 < rows) *reinterpret_cast<f2*>(dst + o + 2) = y1;
}

// Output rows o..o+3 at stride so, one by one.
template <typename T>
__device__ __forceinline__ void span_put_strided(T* dst, int so, int o, int rows, f2 y0, f2 y1) {
    dst[so * o] = store_cvt<T, float>(f2_lo(y0));
    if (o + 1 < rows) dst[so * (o + 1)] = store_cvt<T, float>(f2_hi(y0));
    if (o + 2 < rows) dst[so * (o + 2)] = store_cvt<T, float>(f2_lo(y1));
    if (o + 3 < rows) dst[so * (o + 3)] = store_cvt<T, float>(f2_hi(y1));
}

// The last stage of a tile: exchange buffer -> staging (element type T), alpha applied.
// MODE: 0 = adjacent outputs as aligned pairs, 1 = adjacent outputs one by one, 2 = at
// stride so.
template <int NI, int NO, int D, int MODE, typename T>
__device__ __forceinline__ void span_last(const SpanArgs& a, int F, const float* e, T* stage) {
    constexpr int L = D - 1;
    const SpanShape<NI, NO, D> sh{a};
    const f2 al = f2_pack(a.alpha, a.alpha);
    const int so = MODE == 2 ? a.so : 1, rows = sh.rows(L);
    const bool alpha_one = a.alpha_one;
    span_stage_run<NI, NO>(
        a.m[L], F, rows,
        [&](int f, float (&x)[NI]) {
            const int q = sh.div_fib(L, f), r = f - q * sh.fib(L);
            const float* p = e + q * sh.eq();
            if constexpr (D == 2) {
                p += r;
            } else {
                const int k = sh.div_in(L, r), j = r - k * sh.in(L);
                p += k + sh.js() * j;
            }
            span_load<NI, (NO > 0), float>(p, sh.kp(), a.ce[L], x);
            return stage + q * a.sq + a.sf * r;
        },
        [&](T* dst, int o, f2 y0, f2 y1) {
            if (!alpha_one) {
                y0 = fmul2(y0, al);
                y1 = fmul2(y1, al);
            }
            if constexpr (MODE == 0 && sizeof(T) == 4) {
                span_put(reinterpret_cast<float*>(dst), o, rows, y0, y1);
            } else if constexpr (MODE == 0) {
                *reinterpret_cast<unsigned*>(dst + o) = pack16<T>(y0);
                if (o + 2 < rows) *reinterpret_cast<unsigned*>(dst + o + 2) = pack16<T>(y1);
            } else {
                span_put_strided<T>(dst, so, o, rows, y0, y1);
            }
        });
}

template <int NI, int NO, int D, typename T>
__device__ __forceinline__ void span_last_any(const SpanArgs& a, int F, const float* e, T* stage) {
    const SpanShape<NI, NO, D> sh{a};
    // Pairs: even rows (then every stride is even) and an aligned start.
    if (a.so != 1) {
        span_last<NI, NO, D, 2, T>(a, F, e, stage);
    } else if ((sh.rows(D - 1) & 1) == 0 && ((uintptr_t)stage & (2 * sizeof(T) - 1)) == 0) {
        span_last<NI, NO, D, 0, T>(a, F, e, stage);
    } else {
        span_last<NI, NO, D, 1, T>(a, F, e, stage);
    }
}

// V contiguous elements of Y.
template <typename S, int V> struct SpanChunk { alignas(V * sizeof(S)) S v[V]; };
template <typename S, int V>
__device__ __forceinline__ void span_read(SpanChunk<S, V>& c, const S* src) {
    if constexpr (V * sizeof(S) == 16) *reinterpret_cast<uint4*>(c.v) = *reinterpret_cast<const uint4*>(src);
    else if constexpr (V * sizeof(S) == 8) *reinterpret_cast<uint2*>(c.v) = *reinterpret_cast<const uint2*>(src);
    else if constexpr (V * sizeof(S) == 4) *reinterpret_cast<unsigned*>(c.v) = *reinterpret_cast<const unsigned*>(src);
    else c.v[0] = src[0];
}
// Staged values, old values of Y (beta != 0), rounding, store.
template <typename S, int V>
__device__ __forceinline__ void span_write(const SpanArgs& a, S* dst, const float* src, const SpanChunk<S, V>& old) {
    alignas(16) float v[V];
    if constexpr (V == 4) *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(src);
    else if constexpr (V == 2) *reinterpret_cast<float2*>(v) = *reinterpret_cast<const float2*>(src);
    else v[0] = src[0];
    S o[V];
#pragma unroll
    for (int e = 0; e < V; ++e) {
        if (!a.beta_zero) v[e] = fmaf(a.beta, load_cvt<float, S>(old.v[e]), v[e]);
        o[e] = store_cvt<S, float>(v[e]);
    }
    if constexpr (V * sizeof(S) >= 4)
        store_chunks<V * (int)sizeof(S), S, V>(dst, o);
    else
        dst[0] = o[0];
}

// Staged FP32 results of a tile to a Y with gaps, or with beta != 0: row chunks of V
// elements, consecutive threads on consecutive chunks.  The chunk's place (c, row j,
// plane k, instance q) advances by kSpanThreads chunks per step in mixed radix, so no
// step divides.
template <typename S, int D, int V>
__device__ __forceinline__ void span_copy_out(const SpanArgs& a, int64_t inst0, int cnt, const float* stage) {
    S* Y = static_cast<S*>(a.Y) + inst0 * a.ldyp;
    const int ch = (int)a.chunks.d, nj = (int)a.cols.d, nk = D == 3 ? a.nk : 1;
    const int total = cnt * (int)a.rows.d * ch;
    int row = (int)a.chunks.div(threadIdx.x);
    int c = threadIdx.x - row * ch;
    int q = (int)a.rows.div(row), j = row - q * (int)a.rows.d, k = 0;
    if constexpr (D == 3) {
        k = (int)a.cols.div(j);
        j -= k * nj;
    }
    const int ldy = a.ldy, ldy2 = a.ldy2, ldyp = a.ldyp32;
    // Groups of U chunks: all their old values are requested before the first store.
    constexpr int U = 4;
    for (int e = threadIdx.x; e < total; e += U * kSpanThreads) {
        int off[U], so[U];
        SpanChunk<S, V> old[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            off[u] = V * c + j * ldy + (D == 3 ? k * ldy2 : 0) + q * ldyp;
            so[u] = V * c + (j + (D == 3 ? k * nj : 0)) * a.srow + q * a.sq;
            c += a.dc;
            j += a.dj;
            if (c >= ch) { c -= ch; ++j; }
            q += a.dq;
            if constexpr (D == 3) {
                k += a.dk;
                if (j >= nj) { j -= nj; ++k; }
                if (k >= nk) { k -= nk; ++q; }
            } else {
                if (j >= nj) { j -= nj; ++q; }
            }
        }
        if (!a.beta_zero) {
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (e + u * kSpanThreads < total) span_read<S, V>(old[u], Y + off[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (e + u * kSpanThreads < total) span_write<S, V>(a, Y + off[u], stage + so[u], old[u]);
    }
}

// Bulk copy of the 16-byte granules that hold tile `tile`'s operand span; the first
// element sits at the span's own phase in the buffer.
template <typename S>
__device__ __forceinline__ void span_issue(const SpanArgs& a, unsigned char* dst, uint64_t* bar, int tile,
                                           uint64_t pol) {
    const int64_t inst0 = (int64_t)tile * a.P;
    const int cnt = tile == a.ntiles - 1 ? a.last : a.P;
    const uintptr_t b0 = (uintptr_t)(static_cast<const S*>(a.X) + inst0 * a.ldxp);
    const uintptr_t b1 = b0 + ((cnt - 1) * a.ldxp + a.xspan) * sizeof(S);
    const uintptr_t a0 = b0 & ~(uintptr_t)15;
    const unsigned bytes = (unsigned)(((b1 + 15) & ~(uintptr_t)15) - a0);
    mbar_arrive_expect_tx(bar, bytes);
    bulk_g2s(dst, (const void*)a0, bytes, bar, pol);
}

// As span_issue, for the whole CTA: the copy takes the granules that lie inside the span,
// the threads load the elements before and after them.  The caller's barrier follows.
template <typename S>
__device__ __forceinline__ void span_issue_inside(const SpanArgs& a, unsigned char* dst, uint64_t* bar, int tile,
                                                  uint64_t pol) {
    const int64_t inst0 = (int64_t)tile * a.P;
    const int cnt = tile == a.ntiles - 1 ? a.last : a.P;
    const uintptr_t b0 = (uintptr_t)(static_cast<const S*>(a.X) + inst0 * a.ldxp);
    const uintptr_t b1 = b0 + ((cnt - 1) * a.ldxp + a.xspan) * sizeof(S);
    const uintptr_t from = (b0 + 15) & ~(uintptr_t)15, to = b1 & ~(uintptr_t)15;
    unsigned char* buf = dst - (b0 & ~(uintptr_t)15);   // + address
    if (threadIdx.x == 0) {
        const unsigned bytes = to > from ? (unsigned)(to - from) : 0u;
        mbar_arrive_expect_tx(bar, bytes);
        if (bytes) bulk_g2s(buf + from, (const void*)from, bytes, bar, pol);
    }
    const uintptr_t head = b0 + threadIdx.x * sizeof(S), tail = (to > from ? to : from) + threadIdx.x * sizeof(S);
    if (head < from && head < b1) *reinterpret_cast<S*>(buf + head) = *reinterpret_cast<const S*>(head);
    if (tail < b1) *reinterpret_cast<S*>(buf + tail) = *reinterpret_cast<const S*>(tail);
}

template <typename S, int NI, int NO, int D>
__global__ void __launch_bounds__(kSpanThreads, 4) span_kernel(const __grid_constant__ SpanArgs a) {
    const SpanShape<NI, NO, D> sh{a};
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    unsigned char* slots = smem + 128;
    float* e = reinterpret_cast<float*>(slots + kSpanRing * a.slot_bytes);
    const int tid = threadIdx.x;
    // The last CTAs of the grid take the tiles at the ends of X whose copies would reach
    // outside, one each; the others walk the tiles between them.
    const int walkers = (int)gridDim.x - a.head - a.tail;
    const int grid = walkers > 0 ? walkers : 1;   // step of the walk
    int first = a.head + (int)blockIdx.x, end = a.ntiles - a.tail;
    const bool edge = (int)blockIdx.x >= walkers;
    if (edge) {
        first = (int)blockIdx.x - walkers;
        if (first >= a.head) first += end - a.head;
        end = first + 1;
    }
    uint64_t pol = 0;
    if (tid == 0) {
        for (int s = 0; s < kSpanRing; ++s) mbar_init(&full[s], 1);
        fence_barrier_init();
        pol = l2_evict_first_policy();
        for (int s = 0; s < kSpanRing; ++s) {
            const int t = first + s * grid;
            if (t < end && !edge) span_issue<S>(a, slots + s * a.slot_bytes, &full[s], t, pol);
        }
    }
    if (edge) span_issue_inside<S>(a, slots, full, first, pol);
    __syncthreads();

    int it = 0;
    for (int tile = first; tile < end; tile += grid, ++it) {
        const int s = it % kSpanRing;
        const int64_t inst0 = (int64_t)tile * a.P;
        const int cnt = tile == a.ntiles - 1 ? a.last : a.P;
        unsigned char* slot = slots + s * a.slot_bytes;
        const S* xt = reinterpret_cast<const S*>(
            slot + ((uintptr_t)(static_cast<const S*>(a.X) + inst0 * a.ldxp) & 15u));
        const bool ok = mbar_wait_bounded(&full[s], (unsigned)(it / kSpanRing) & 1u, a.err);

        // ---- first contraction: operand span -> e -------------------------------------
        {
            const int rows = sh.rows(0), ldxq = (int)a.ldxp, col = a.xs_col;
            span_stage_run<NI, NO>(
                a.m[0], cnt * sh.fib(0), rows,
                [&](int f, float (&x)[NI]) {
                    const int q = sh.div_fib(0, f), r = f - q * sh.fib(0);
                    const S* p = xt + q * ldxq;
                    float* dst = e + q * sh.eq();
                    if constexpr (D == 2) {
                        p += r;
                        dst += sh.kp() * r;
                    } else {
                        const int j = sh.div_in(0, r), i = r - j * sh.in(0);
                        p += i + col * j;
                        dst += sh.kp() * i + sh.js() * j;
                    }
                    span_load<NI, (NO > 0), S>(p, D == 2 ? col : a.xs_plane, a.ce[0], x);
                    return dst;
                },
                [&](float* dst, int o, f2 y0, f2 y1) { span_put(dst, o, rows, y0, y1); });
        }
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {   // let in-flight copies land before the CTA exits
                for (int j = it; j < it + kSpanRing - (it > 0); ++j)
                    if (tile + (j - it) * grid < end)
                        mbar_wait_bounded(&full[j % kSpanRing], (unsigned)(j / kSpanRing) & 1u, a.err);
                bulk_wait_all();
            }
            return;
        }
        // The previous tile's slot: its results have left, the next operands come in.
        if (tid == 0 && it > 0) {
            const int next = tile + (kSpanRing - 1) * grid;
            if (next < end) {
                const int p = (it - 1) % kSpanRing;
                bulk_wait_read();
                fence_proxy_async_smem();
                span_issue<S>(a, slots + p * a.slot_bytes, &full[p], next, pol);
            }
        }
        // ---- 3-D second contraction, in place -----------------------------------------
        if constexpr (D == 3) {
            const int rows = sh.rows(1), js = sh.js();
            span_stage_run<NI, NO>(
                a.m[1], cnt * sh.fib(1), rows,
                [&](int f, float (&x)[NI]) {
                    const int q = sh.div_fib(1, f), r = f - q * sh.fib(1);
                    const int i = sh.div_in(1, r), k = r - i * sh.in(1);
                    float* p = e + q * sh.eq() + k + sh.kp() * i;
                    span_load<NI, (NO > 0), float>(p, js, a.ce[1], x);
                    return p;
                },
                [&](float* dst, int o, f2 y0, f2 y1) { span_put_strided<float>(dst, js, o, rows, y0, y1); });
            __syncthreads();
        }
        // ---- last contraction -> staging in the operand slot --------------------------
        const int F = cnt * sh.fib(D - 1);
        // Packed Y: the tile's run may start anywhere, so it is staged at its own phase;
        // the 16-byte-aligned middle leaves as one bulk copy, the ends by plain stores.
        S* yt = static_cast<S*>(a.Y) + inst0 * a.ny;
        const unsigned ph = a.bulk ? (unsigned)((uintptr_t)yt & 15u) : 0u;
        if constexpr (sizeof(S) == 4) {
            span_last_any<NI, NO, D, float>(a, F, e, reinterpret_cast<float*>(slot + ph));
        } else {
            if (a.bulk) span_last_any<NI, NO, D, S>(a, F, e, reinterpret_cast<S*>(slot + ph));
            else span_last_any<NI, NO, D, float>(a, F, e, reinterpret_cast<float*>(slot));
        }
        if (a.bulk) {
            const S* stage = reinterpret_cast<const S*>(slot + ph);
            fence_proxy_async_smem();
            __syncthreads();
            const unsigned total = (unsigned)(cnt * a.ny) * (unsigned)sizeof(S);
            const unsigned head = min(total, (16u - ph) & 15u), mid = (total - head) & ~15u;
            if (tid == 0) {
                if (mid)
                    bulk_s2g_hint(reinterpret_cast<unsigned char*>(yt) + head,
                                  reinterpret_cast<const unsigned char*>(stage) + head, mid, pol);
                bulk_commit();
            }
            const int nh = (int)(head / sizeof(S)), t0 = (int)((head + mid) / sizeof(S));
            if (tid < nh) yt[tid] = stage[tid];
            if (t0 + tid < (int)(total / sizeof(S))) yt[t0 + tid] = stage[t0 + tid];
        } else {
            const float* stage = reinterpret_cast<const float*>(slot);
            __syncthreads();
            if (a.vec == 4) span_copy_out<S, D, 4>(a, inst0, cnt, stage);
            else if (a.vec == 2) span_copy_out<S, D, 2>(a, inst0, cnt, stage);
            else span_copy_out<S, D, 1>(a, inst0, cnt, stage);
        }
    }
    if (tid == 0) bulk_wait_all();
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
template <typename S, int NI, int NO, int D>
kron_status launch_span_n(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st) {
    const DeviceInfo& dev = device_info();
    auto kern = span_kernel<S, NI, NO, D>;
    if (!ensure_smem_optin((const void*)kern, smem)) return KRON_ERR_CUDA;
    const int64_t ntiles = a.ntiles, edges = a.head + a.tail;
    int64_t grid = d.grid;
    if (grid <= 0) {
        int per_sm = 0;
        if (!resident_ctas(&per_sm, (const void*)kern, kSpanThreads, smem))
            return KRON_ERR_CUDA;
        grid = (int64_t)(per_sm < 1 ? 1 : per_sm) * dev.sms;
    }
    // (one CTA for each tile that is loaded element by element, at least one for the rest)
    grid = std::max<int64_t>(edges + (ntiles > edges), std::min<int64_t>(grid, ntiles));
    kern<<<(unsigned)grid, kSpanThreads, smem, st>>>(a);
    return cudaPeekAtLastError() == cudaSuccess ? KRON_OK : KRON_ERR_CUDA;
}

// Instantiations NI -> NO with |NI - NO| <= W (interpolation and its transpose), one
// translation unit per group G of four NI.  The range is a trade against build time: the
// 248 FP32 ones compile for about 320 CPU seconds, the 32 square ones of each 16-bit type
// for 135, and a shape outside runs the body with run-time extents (8 -> 12 at a third of the
// batch: 90 instead of 70 us).
template <typename S, int D, int NI, int W, int NO>
kron_status launch_span_no(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st) {
    if constexpr (NO > kMaxN || NO > NI + W) {
        return KRON_ERR_NOT_SUPPORTED;
    } else {
        if (a.oe[0] == NO) return launch_span_n<S, NI, NO, D>(d, a, smem, st);
        return launch_span_no<S, D, NI, W, NO + 1>(d, a, smem, st);
    }
}
template <typename S, int D, int G>
kron_status launch_span_group(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st) {
    constexpr int W = sizeof(S) == 4 ? 4 : 0;   // 16-bit storage: square shapes only
    constexpr int N0 = 4 * G + 1;
    switch (a.ce[0] - N0) {
        case 0: return launch_span_no<S, D, N0, W, (N0 > W ? N0 - W : 1)>(d, a, smem, st);
        case 1: return launch_span_no<S, D, N0 + 1, W, (N0 + 1 > W ? N0 + 1 - W : 1)>(d, a, smem, st);
        case 2: return launch_span_no<S, D, N0 + 2, W, (N0 + 2 > W ? N0 + 2 - W : 1)>(d, a, smem, st);
        case 3: return launch_span_no<S, D, N0 + 3, W, (N0 + 3 > W ? N0 + 3 - W : 1)>(d, a, smem, st);
    }
    return KRON_ERR_NOT_SUPPORTED;
}
// Defined by the translation units.
template <typename S, int D, int G>
kron_status span_group(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st);

template <typename S, int D>
kron_status launch_span_fixed(const KronDesc& d, const SpanArgs& a, size_t smem, cudaStream_t st) {
    switch ((a.ce[0] - 1) / 4) {
        case 0: return span_group<S, D, 0>(d, a, smem, st);
        case 1: return span_group<S, D, 1>(d, a, smem, st);
        case 2: return span_group<S, D, 2>(d, a, smem, st);
        default: return span_group<S, D, 3>(d, a, smem, st);
    }
}

template <typename S, int D>
kron_status launch_span(const KronDesc& d, cudaStream_t st) {
    const DeviceInfo& dev = device_info();
    if (dev.sms <= 0) return KRON_ERR_CUDA;
    const int es = (int)sizeof(S);
    // Extents of X and Y per mode of the stored arrays.
    const int x1 = d.transx ? d.xe[1] : d.xe[0], x2 = d.transx ? d.xe[0] : d.xe[1], x3 = d.xe[2];
    const int64_t xspan = (int64_t)d.ldx * (x2 - 1) + x1 + (D == 3 ? (int64_t)d.ldx2 * (x3 - 1) : 0);
    const int64_t useful = (int64_t)x1 * x2 * x3;
    // A span that is mostly gaps is read element by element instead (fiber kernel).
    if (xspan > 2 * useful || (d.batch > 1 && d.ldxp > 2 * useful)) return KRON_ERR_NOT_SUPPORTED;
    const bool square = x1 == d.N && x2 == d.N && (D == 2 || x3 == d.N) && d.ye[0] == d.N && d.ye[1] == d.N &&
                        (D == 2 || d.ye[2] == d.N);
    const bool cubic = x1 == x2 && d.ye[0] == d.ye[1] && (D == 2 || (x1 == x3 && d.ye[0] == d.ye[2]));
    SpanCall call;
    call.D = D;
    call.es = es;
    call.N = d.N;
    call.nx = useful;
    call.ny = (int64_t)d.ye[0] * d.ye[1] * d.ye[2];
    call.batch = d.batch;
    call.square = square;
    call.up_one = d.ye[0] == d.xe[0] + 1 && d.ye[1] == d.xe[1] + 1 && (D == 2 || d.ye[2] == d.xe[2] + 1);
    call.beta = d.beta != 0.0;
    call.x_packed = d.contiguous;
    call.y_packed = d.ldy == d.ye[0] && (D == 2 || d.ldy2 == d.ye[0] * d.ye[1]) && (d.batch == 1 || d.ldyp == call.ny);
    call.y_aligned = d.ycontig;
    call.yvec = d.yvec / es;
    call.row_bytes = (int)std::min<int64_t>(INT32_MAX, (int64_t)d.ldy * es);
    if (scalar_body_faster(call)) return KRON_ERR_NOT_SUPPORTED;
    // Offsets of a tile (at most 256 instances) in Y are kept in 32 bits.
    if (d.ldyp >= (int64_t)INT32_MAX / 256) return KRON_ERR_NOT_SUPPORTED;
    SpanArgs a;
    const int y1 = d.ye[0], y2 = d.ye[1], y3 = d.ye[2];
    // Stage order, extents and matrices.
    const double* mats[3];
    if (D == 2) {
        const bool t = d.transx;
        mats[0] = t ? d.m1 : d.m2;
        mats[1] = t ? d.m2 : d.m1;
        mats[2] = nullptr;
        a.ce[0] = x2; a.oe[0] = t ? y1 : y2;
        a.ce[1] = x1; a.oe[1] = t ? y2 : y1;
        a.kp = span_kp(a.oe[0]);
        a.fib[0] = fast_div(x1);
        a.fib[1] = fast_div(a.oe[0]);
        // instances of one warp on different banks: as many words apart as fibers (mod 32)
        a.eq = stride_mod32(a.kp * x1, (a.oe[0] + 1) / 2 * 2 % 32);
    } else {
        mats[0] = d.m3; mats[1] = d.m2; mats[2] = d.m1;
        a.ce[0] = x3; a.oe[0] = y3;
        a.ce[1] = x2; a.oe[1] = y2;
        a.ce[2] = x1; a.oe[2] = y1;
        a.kp = span_kp(y3);
        a.js = stride_mod32(a.kp * x1, 2);
        a.eq = a.js * std::max(x2, y2);
        a.fib[0] = fast_div(x1 * x2); a.in[0] = fast_div(x1);
        a.fib[1] = fast_div(x1 * y3); a.in[1] = fast_div(y3);
        a.fib[2] = fast_div(y2 * y3); a.in[2] = fast_div(y2);
    }
    memset(a.m, 0, sizeof(a.m));
    for (int s = 0; s < D; ++s)
        for (int l = 0; l < a.ce[s]; ++l) {
            float col[kMaxN];   // an odd last row is paired with the zero after it
            for (int r = 0; r < a.oe[s]; ++r) col[r] = (float)mats[s][r + d.N * l];
            memcpy(&a.m[s][8 * l], col, a.oe[s] * sizeof(float));
        }
    a.X = d.X;
    a.Y = d.Y;
    a.ldxp = d.ldxp;
    a.ldyp = d.ldyp;
    a.xs_col = d.ldx;
    a.xs_plane = d.ldx2;
    a.xspan = (int)xspan;
    a.ye1 = y1;
    a.ny = y1 * y2 * y3;
    a.alpha = (float)d.alpha;
    a.beta = (float)d.beta;
    a.beta_zero = d.beta == 0.0;
    a.alpha_one = d.alpha == 1.0;
    a.ldy = d.ldy;
    a.ldy2 = D == 3 ? d.ldy2 : 0;
    a.ldyp32 = d.batch > 1 ? (int)d.ldyp : 0;
    a.err = device_error_word();
    if (!a.err) return KRON_ERR_CUDA;

    // Instances per tile: about two fibers per thread in the stage with the fewest.
    // (A tuned tile belongs to the contiguous bodies and is not used here.)
    int P = std::max(1, 2 * kSpanThreads / (int)std::min(a.fib[0].d, std::min(a.fib[1].d, D == 3 ? a.fib[2].d : 256u)));
    const bool packed = d.beta == 0.0 && call.y_packed;
    // Chunks of a row of Y: up to 16 bytes, every row of every instance aligned to it.
    a.vec = 1;
    for (int v = 4; v >= 2; v /= 2) {
        const int b = v * es;
        if (y1 % v == 0 && ((uintptr_t)d.Y) % b == 0 && ((int64_t)d.ldy * es) % b == 0 &&
            (D == 2 || ((int64_t)d.ldy2 * es) % b == 0) && (d.batch == 1 || (d.ldyp * es) % b == 0)) {
            a.vec = v;
            break;
        }
    }
    auto smem_of = [&](int p) {
        // staged rows: packed, or padded like the other stage outputs
        a.bulk = packed;
        // (16-byte chunks are read from rows an odd number of chunks apart)
        a.srow = a.bulk ? y1 : a.vec == 4 ? (y1 % 8 == 4 ? y1 : y1 + 4) : span_kp(y1);
        a.sq = a.srow * y2 * y3;
        if (D == 2 && d.transx) { a.sf = 1; a.so = a.srow; }
        else { a.sf = a.srow; a.so = 1; }
        const size_t xb = ((size_t)(p - 1) * d.ldxp + xspan) * es + 32;
        const size_t yb = (size_t)p * a.sq * (a.bulk ? es : 4) + 16;
        a.slot_bytes = (int)round_up(std::max(xb, yb), 128);
        return 128 + (size_t)kSpanRing * a.slot_bytes + (size_t)p * a.eq * 4;
    };
    // Four CTAs per SM when the tile allows it.
    const size_t want = dev.smem_per_sm / 4 - 1024;
    P = (int)std::min<int64_t>(P, d.batch);
    if (smem_of(P) > want) {
        const size_t per = kSpanRing * std::max<size_t>(d.ldxp * es, a.sq * (a.bulk ? es : 4)) + a.eq * 4;
        P = std::max(1, std::min(P, (int)(want / per)));
        while (P > 1 && smem_of(P) > want) --P;
    }
    size_t smem = smem_of(P);
    while (smem > dev.smem_per_block_optin && P > 1) smem = smem_of(--P);
    if (smem > dev.smem_per_block_optin) return KRON_ERR_NOT_SUPPORTED;
    a.P = P;
    const int64_t ntiles = (d.batch + P - 1) / P;
    if (ntiles > (1 << 30)) return KRON_ERR_NOT_SUPPORTED;   // tiles are counted in 32 bits
    a.ntiles = (int)ntiles;
    a.last = (int)(d.batch - (ntiles - 1) * P);
    const SpanEdges ed = span_edges((uintptr_t)d.X, d.batch, P, d.batch > 1 ? d.ldxp : 0, xspan, es);
    if (!ed.copies) return KRON_ERR_NOT_SUPPORTED;
    a.head = ed.head;
    a.tail = ed.tail;
    {
        const int ch = y1 / a.vec;
        a.dc = kSpanThreads % ch;
        a.dj = kSpanThreads / ch % y2;
        a.dk = kSpanThreads / ch / y2 % y3;
        a.dq = kSpanThreads / ch / y2 / y3;
        a.nk = y3;
    }
    a.chunks = fast_div(y1 / a.vec);
    a.rows = fast_div(y2 * y3);
    a.cols = fast_div(y2);
    // Instantiations for every mode NI -> NO, else runtime extents up to NI = 4, 8, 12, 16.
    kron_status r = KRON_ERR_NOT_SUPPORTED;
    if (cubic) r = launch_span_fixed<S, D>(d, a, smem, st);
    if (r != KRON_ERR_NOT_SUPPORTED) return r;
    const int ni = std::max(std::max(a.ce[0], a.ce[1]), D == 3 ? a.ce[2] : 1);
    if (ni <= 4) return launch_span_n<S, 4, 0, D>(d, a, smem, st);
    if (ni <= 8) return launch_span_n<S, 8, 0, D>(d, a, smem, st);
    if (ni <= 12) return launch_span_n<S, 12, 0, D>(d, a, smem, st);
    return launch_span_n<S, 16, 0, D>(d, a, smem, st);
}

}  // namespace kron
