// How a launch's units are shared out over its CTAs: the host's plan and the range arithmetic that the kernels do with it.  Plain C++
// beside CUDA, so that a host program can go through every CTA of a plan.
#pragma once
#include <algorithm>
#include <cstdint>

#include "fq_internal.h"

#ifdef __CUDACC__
#define FQ_HD __host__ __device__ __forceinline__
#else
#define FQ_HD inline
#endif

namespace fq {

// Division by a number that the host knows: n / d = upper half of n * (floor(2^64 / d) + 1), exact for every 32-bit n; d = 1 has
// no such factor (0).  The compiler's division is a chain of some forty instructions, and up to ten of them stood between a CTA's last
// unit and its last sum: 14336 x 4096 at 16 rows 17.8 us, so 17.1; 4096 x 4096 at 16 8.6 and 8.3; 4096 x 28672 at 8 24.7 and 24.3.
struct Divisor {
    uint32_t lo, hi;
    FQ_HD static Divisor of(uint32_t d) {
        const uint64_t m = d > 1 ? ~0ull / d + 1 : 0;         // (a power of two: ~0 / d + 1 = 2^64 / d exactly)
        return {(uint32_t)m, (uint32_t)(m >> 32)};
    }
    FQ_HD uint32_t operator()(uint32_t n) const {
        const uint32_t quotient = (uint32_t)(((uint64_t)hi * n + (((uint64_t)lo * n) >> 32)) >> 32);
        return (lo | hi) ? quotient : n;
    }
};
// How NT x KT units are shared out (see split_units): q units and one more for the first r CTAs, or `split` CTAs to a tile.
struct Shares {
    uint32_t q, r;
    uint32_t split;   // 0 = units dealt out as one contiguous range per CTA (stream-K);
                      // c > 0 = every column tile belongs to c CTAs, CTA b takes part b mod c of tile b / c
    Divisor by_q, by_q1, by_split, by_kt;
    // which CTA owns unit u, and the first unit of CTA c, of contiguous ranges
    FQ_HD uint32_t cta_of_unit(uint32_t u) const {
        const uint32_t big = r * (q + 1);
        return u < big ? by_q1(u) : r + by_q(u - big);
    }
    FQ_HD uint32_t unit_begin_of(uint32_t c) const { return c * q + (c < r ? c : r); }
    // the units [begin, end) of CTA c
    FQ_HD void range(uint32_t c, uint32_t KT, uint32_t& begin, uint32_t& end) const {
        if (split) {
            // tile-aligned: no CTA works on two tiles, so none settles two split tiles one after the other
            const uint32_t tile = by_split(c), part = c - tile * split;
            begin = tile * KT + by_split(part * KT);
            end = tile * KT + by_split((part + 1) * KT);
        } else {
            begin = unit_begin_of(c);
            end = begin + q + (c < r ? 1u : 0u);
        }
    }
    // the first and the last CTA that have units of tile tn
    FQ_HD void owners(uint32_t tn, uint32_t KT, uint32_t& first, uint32_t& last) const {
        first = split ? tn * split : cta_of_unit(tn * KT);
        last = split ? first + split - 1 : cta_of_unit(tn * KT + KT - 1);
    }
    // which of its two partial slots CTA c uses for its part of tile tn: the second if its range begins before the tile
    FQ_HD uint32_t slot_of(uint32_t c, uint32_t tn, uint32_t KT) const { return split || unit_begin_of(c) >= tn * KT ? 0u : 1u; }
};

// How the NT x KT units of a launch are shared out over persistent CTAs: split = 0, one contiguous range each; else a tile-aligned
// split, every column tile to `split` CTAs, when that costs at most `slack` more units per CTA: then no CTA has to settle two
// split tiles in a row.  us, ranges / tiles: two units more in the streaming kernel 8192 x 8192 at one row 14.7 / 13.6, at eight 16.5 / 16.1,
// but seven more 28672 x 8192 33.9 / 36.0; in the tcgen05 kernel three or four more at 64 rows and groups of 128 5120 x 5120 16.2 / 14.8, 11008 x 4096 20.7 /
// 19.4, 14336 x 4096 23.6 / 22.7, 8192 x 8192 24.3 / 23.9, six more 13824 x 5120 25.9 / 26.7; otherwise one, at 32 rows three more 14336 x
// 4096 18.6 / 19.0, at 128 33.6 / 34.1, with groups of 64 at 24 19.2 / 20.3.
struct Split {
    uint32_t grid, split, units_per_cta;
};
inline Split split_units(uint32_t NT, uint32_t KT, uint32_t sms, uint32_t slack) {
    const uint32_t grid = std::min<uint32_t>({sms, kMaxCtas, NT * KT}), units_per_cta = (NT * KT + grid - 1) / grid;
    const uint32_t c = std::min<uint32_t>(grid / NT, KT);
    if (c >= 2 && (KT + c - 1) / c <= units_per_cta + slack) return {NT * c, c, (KT + c - 1) / c};
    return {grid, 0, units_per_cta};
}
inline Shares shares_of(const Split& sp, uint32_t NT, uint32_t KT) {
    const uint32_t q = NT * KT / sp.grid, r = NT * KT % sp.grid;
    return {q, r, sp.split, Divisor::of(q ? q : 1), Divisor::of(q + 1), Divisor::of(sp.split ? sp.split : 1), Divisor::of(KT)};
}

}  // namespace fq
