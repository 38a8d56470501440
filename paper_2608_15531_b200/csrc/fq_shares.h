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
// no such factor (0).  (Granlund and Montgomery, Division by invariant integers using multiplication, 1994.)  Of the compiler's divisions,
// each a chain of dependent instructions, up to ten stood between a CTA's last unit and its last sum: 14336 x 4096 at 16 rows 17.8 us,
// so 17.1; 4096 x 4096 at 16 8.6 and 8.3; 4096 x 28672 at 8 24.7 and 24.3.
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
// split tiles in a row.
struct Split {
    uint32_t grid, split, units_per_cta;
};
inline Split split_units(uint32_t NT, uint32_t KT, uint32_t sms, uint32_t slack) {
    const uint32_t grid = std::min<uint32_t>({sms, kMaxCtas, NT * KT}), units_per_cta = (NT * KT + grid - 1) / grid;
    const uint32_t c = std::min<uint32_t>(grid / NT, KT);
    if (c >= 2 && (KT + c - 1) / c <= units_per_cta + slack) return {NT * c, c, (KT + c - 1) / c};
    return {grid, 0, units_per_cta};
}
constexpr uint32_t kTwoGroups = 8;      // units per CTA from which the streaming kernel runs two groups of dense warps

// The streaming kernel's.  One unit more is always worth it, a second one where it costs less than the second split tile (about 1 us; with two CTAs to
// a tile, and so the fewest CTAs, less).  us, ranges / tiles:
//   the longer share brings the second group of dense warps: 2048 x 12800 at one row 9.7 / 8.5, at eight 11.0 / 9.9, 1920 x 7040 at eight
//     9.4 / 7.6; without outliers also where both shares are short, 1664 x 14336 at eight 7.9 / 7.4, 2432 x 14080 8.9 / 8.4, with them not (1408 x 13312 9.2 / 9.4)
//   up to four rows (one on tiles of 128 columns, whose units are worth half): three CTAs and more to a tile 8192 x 8192 at one 14.7 / 13.6, 8192 x 6400
//     13.6 / 12.5, 18688 x 8960 26.5 / 26.0; two, up to 16 units, 3200 x 15616 12.5 / 12.0, 3840 x 15360 13.7 / 13.3, 2816 x 13824 10.2 / 10.6, beyond them
//     5120 x 16384 16.0 / 16.1, 12288 x 17920 at four 34.8 / 35.6; without outliers up to 24, 6400 x 17152 15.8 / 15.4, 14976 x 18176 30.5 / 30.8
//   five rows and more, and two to four on tiles of 128 columns: no (3328 x 14592 at eight 13.2 / 14.3, 24320 x 3840 20.5 / 21.5, 11520 x 4224 15.9 / 16.9,
//     8192 x 6400 14.9 / 14.6; without outliers, where the CTAs, all at the same k-steps, take 4 to 9 % longer for a unit, 15232 x 18432 at eight
//     32.1 / 35.7, 10880 x 9088 at 16 23.5 / 25.9; 22656 x 2176 at four 15.9 / 16.2)
// (Seven units more, 28672 x 8192 at one row: 33.9 / 36.0.)
inline Split split_streaming(uint32_t BN, uint32_t NT, uint32_t KT, uint32_t sms, uint32_t rows, bool outliers) {
    const Split one = split_units(NT, KT, sms, 1), two = split_units(NT, KT, sms, 2);
    if (one.split || !two.split) return one;
    const uint32_t units = one.units_per_cta;                 // of a range
    if (units <= kTwoGroups && (two.units_per_cta >= kTwoGroups || !outliers)) return two;
    if (rows <= (BN == 256 ? 4 : 1) && (two.split > 2 || units * BN < (outliers ? 16u : 24u) * 256)) return two;
    return one;
}
// The tcgen05 kernel's.  us, ranges / tiles: three or four more at 33 to 64 rows and groups of 128, 5120 x 5120 16.2 / 14.8, 11008 x 4096 20.7 / 19.4, 2176 x
// 6400 13.9 / 11.4, 25344 x 9088 63.2 / 61.9, 3456 x 6400 at 40 13.1 / 13.3, six more 13824 x 5120 25.9 / 26.7; otherwise one: at 32 rows
// three more 14336 x 4096 18.6 / 19.0, at 128 33.6 / 34.1, with groups of 64 at 24 19.2 / 20.3.
inline Split split_tc(uint32_t NT, uint32_t KT, uint32_t sms, uint32_t nr, uint32_t group) {
    return split_units(NT, KT, sms, nr == 64 && group == 128 ? 4 : 1);
}
inline Shares shares_of(const Split& sp, uint32_t NT, uint32_t KT) {
    const uint32_t q = NT * KT / sp.grid, r = NT * KT % sp.grid;
    return {q, r, sp.split, Divisor::of(q ? q : 1), Divisor::of(q + 1), Divisor::of(sp.split ? sp.split : 1), Divisor::of(KT)};
}

}  // namespace fq
