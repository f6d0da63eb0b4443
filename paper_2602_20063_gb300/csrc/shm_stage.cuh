// Shared-memory staging of one glyph's table for the per-glyph segment kernels (forward query,
// reverse pass): one thread issues cp.async.bulk copies completing on an mbarrier, every thread
// waits on it with a time limit.
//
// Work split: the segments are cut into `units` of equal cost along the path that runs through the
// glyphs in order, paying `w` for every glyph (its table copy) and 1 for every query.  A unit is a CTA's
// whole work: it starts and ends anywhere inside a glyph, so a few long segments spread over every SM
// and uneven ones balance (one CTA per glyph left 37 glyphs of 60,000 queries on 37 of 304 CTAs).  w is
// the copy's cost in queries at memory bandwidth, table bytes / 40 B of directions and outputs (a quarter of
// it where there are one to four units a glyph, path_weight).
#pragma once
#include "shm_internal.h"

namespace shm {
namespace stage {

constexpr uint64_t WAIT_NS = 1000000000ull;   // 1 s
constexpr uint64_t DRAIN_NS = 100000000ull;   // 100 ms
constexpr uint32_t BULK_PIECE = 32768;        // bytes per cp.async.bulk
constexpr int TABLE_OFFSET = 128;             // mbarriers first, tables 128-byte aligned
constexpr int QUERY_BYTES = 40;               // direction and outputs of one query
constexpr int UNIT_MIN = 1024;                // queries a unit should have before another CTA pays for a copy

__device__ __forceinline__ uint64_t gtimer()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ bool bar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity, uint64_t limit)
{
    if (bar_try_wait(bar, parity)) return true;
    const uint64_t t0 = gtimer();
    while (!bar_try_wait(bar, parity))
        if (gtimer() - t0 > limit) return false;
    return true;
}

// Thread 0 of the CTA: initialise the barrier (once per kernel).
__device__ __forceinline__ void init(uint32_t bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Thread 0: `bar` completes when `bytes` have arrived.  Earlier generic-proxy accesses of the destination
// are ordered before the copies that follow.
__device__ __forceinline__ void expect(uint32_t bar, uint32_t bytes)
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// Thread 0: copy `bytes` (a multiple of 16; 16-byte aligned addresses) into shared memory, counted on `bar`.
__device__ __forceinline__ void copy(uint32_t bar, uint32_t dst, const void* src, uint32_t bytes)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// Thread 0: copy `bytes` (a multiple of 16, 16-byte aligned source) into shared memory at dst,
// completing on `bar`.
__device__ __forceinline__ void issue(uint32_t bar, uint32_t dst, const unsigned char* src, uint32_t bytes)
{
    expect(bar, bytes);
    for (uint32_t off = 0; off < bytes; off += BULK_PIECE) copy(bar, dst + off, src + off, min(BULK_PIECE, bytes - off));
}

// Position on the path: query q of glyph g (g = G: past the last one).
struct Pos {
    int g;
    int64_t q;
};

// Part [a, b) of glyph g's queries; b <= a: no part left.
struct Part {
    int g;
    int64_t a, b;
};

__device__ __forceinline__ int64_t seg_at(const int64_t* seg, int64_t Q, int g)
{
    return min(max(__ldg(seg + g), (int64_t)0), Q);
}

// The path and its cut into `units` (see above), the same on every CTA and on the host.
struct Path {
    const int64_t* seg;
    int G;
    int64_t Q;
    int64_t w;       // cost of a glyph
    uint32_t units;
    uint64_t inv;    // 2^64 / units, rounded up: x / units = umulhi(x, inv) for x units < 2^64

    Path(const int64_t* seg_, int G_, int64_t Q_, int64_t w_, int64_t units_)
        : seg(seg_), G(G_), Q(Q_), w(w_), units((uint32_t)units_), inv(UINT64_MAX / (uint64_t)units_ + 1) {}

    // Start of unit u on the path (a whole warp calls it): u units of cost.  The first 32 probes surround the
    // glyph that even segments would put there and wait for nothing, so that a near miss costs one memory round trip,
    // together with the ends' that the cost needs; otherwise 32 probes per round, two or three dependent round trips.
    __device__ __forceinline__ Pos at(uint32_t u) const
    {
        const int lane = threadIdx.x & 31;
        const int guess = units > 1 ? (int)__umul64hi((uint64_t)u * (uint32_t)G, inv) : (u ? G : 0);
        const int base = max(0, min(guess - 15, G - 31)), near = base + lane;
        int64_t v = near <= G ? seg_at(seg, Q, near) : INT64_MAX / 2;
        const int64_t lo = seg_at(seg, Q, 0);
        const uint64_t total = seg_at(seg, Q, G) - lo + w * G;
        int64_t D = (int64_t)total;  // cost of the path up to unit u
        if (u < units) {
            const uint64_t per = units > 1 ? __umul64hi(total, inv) : total;
            D = (int64_t)(per * u + (u ? __umul64hi((total - per * units) * u, inv) : 0));
        }
        // the largest g in [0, G] with cost(g) = seg[g] - seg[0] + w g <= D, and seg[g]
        unsigned m = __ballot_sync(0xffffffffu, near <= G && v - lo + w * near <= D);
        int k = 31 - __clz((int)(m | 1u));
        int g = base + k;
        int64_t s = __shfl_sync(0xffffffffu, v, k);
        if (!(m & 1u) || (k == 31 && g < G)) {
            g = 0;
            s = lo;
            for (int n = G + 1; n > 1;) {
                const int step = (n + 31) / 32, at = lane * step;
                v = at < n ? seg_at(seg, Q, g + at) : INT64_MAX / 2;
                m = __ballot_sync(0xffffffffu, at < n && v - lo + w * (g + at) <= D);
                k = 31 - __clz((int)(m | 1u));
                s = __shfl_sync(0xffffffffu, v, k);
                g += k * step;
                n = min(step, n - k * step);
            }
        }
        return Pos{g, min(Q, s + max((int64_t)0, D - (s - lo + w * g) - w))};
    }

    // This CTA's unit: start and end positions through shared memory (every thread calls it).
    __device__ __forceinline__ void unit(Pos* sh, Pos& start, Pos& end) const
    {
        const int warp = threadIdx.x >> 5;
        if (warp < 2) {
            const Pos p = at(blockIdx.x + warp);
            if ((threadIdx.x & 31) == 0) sh[warp] = p;
        }
        __syncthreads();
        start = sh[0];
        end = sh[1];
    }
};

// The first non-empty part of glyph g or a later one, up to the end position.
__device__ __forceinline__ Part next_part(const int64_t* seg, int G, int64_t Q, int g, const Pos& start, const Pos& end)
{
    for (; g <= end.g && g < G; ++g) {
        int64_t a = seg_at(seg, Q, g), b = max(seg_at(seg, Q, g + 1), a);
        if (g == start.g) a = max(a, start.q);
        if (g == end.g) b = min(b, end.q);
        if (a < b) return Part{g, a, b};
    }
    return Part{G, 0, 0};
}

// Host: units for Q queries over G glyphs, at most `cap` (the CTAs that run at once); just under one
// glyph each becomes one glyph each, which leaves even segments uncut.
inline int64_t units_for(int64_t Q, int64_t G, int64_t w, int64_t cap)
{
    const int64_t n = (Q + w * G) / (UNIT_MIN + (w < UNIT_MIN ? w : UNIT_MIN)) + 1;
    const int64_t m = n < cap ? n : cap;
    return m > G && m - G <= m / 32 ? G : m;
}

// Host: cost of a glyph on the path.  With up to four units a glyph most units start inside one and pay a copy of
// their own, so that glyphs are cut nearly by queries alone (152 even glyphs of 4,096, N = 32 f32: 16.4 -> 12.4 us); a
// quarter is left so that runs of tiny glyphs do not pile up in one unit.  More units, or tables below 40 KB, keep
// the whole cost, which spares slivers of glyphs (152 uneven glyphs, N = 13: 12.4 against 14.4 us; 37 of N = 32 f16,
// 60,000 queries each: 28.9 against 29.2).
inline int64_t path_weight(int64_t w, int64_t G, int64_t units) { return units > G && units < 4 * G && w >= 1024 ? w / 4 : w; }

template <int DT>
__device__ __forceinline__ float4 rec(const unsigned char* table, int r)
{
    if (DT == SHM_F32) return reinterpret_cast<const float4*>(table)[r];
    const uint2 v = reinterpret_cast<const uint2*>(table)[r];
    return DT == SHM_F16 ? h4_to_f4(v) : b4_to_f4(v);
}

// The 2x2 footprint of cell (i, j) on face f from a staged texel table of padded width P.
template <int DT>
__device__ __forceinline__ Corners corners(const unsigned char* table, int P, int f, int i, int j)
{
    const int r = (f * P + j) * P + i;
    Corners c;
    c.c00 = rec<DT>(table, r);
    c.c10 = rec<DT>(table, r + 1);
    c.c01 = rec<DT>(table, r + P);
    c.c11 = rec<DT>(table, r + P + 1);
    return c;
}

}  // namespace stage
}  // namespace shm
