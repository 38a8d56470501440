// Host side of the library: layout choice, INT4 group quantiser + packer (Eq. 2, Eq. 3),
// Tile-COO encoder / decoder / validator (Section 3.2).  Plain C++, no CUDA.
#include <omp.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>
#include <vector>

#include "fq_internal.h"

namespace fq {
char* error_buffer() {
    static thread_local char buf[512] = {0};
    return buf;
}

static inline uint16_t f32_to_bf16_rne(float f) {
    uint32_t u;
    std::memcpy(&u, &f, 4);
    if ((u & 0x7fffffffu) > 0x7f800000u) return (uint16_t)((u >> 16) | 0x40u);
    u += 0x7fffu + ((u >> 16) & 1u);
    return (uint16_t)(u >> 16);
}
static inline float bf16_to_f32(uint16_t h) {
    uint32_t u = (uint32_t)h << 16;
    float f;
    std::memcpy(&f, &u, 4);
    return f;
}

// Position of the code of (row kr, column cr) inside a 128 x BN chunk: word index and nibble.
static inline void wq_slot(uint32_t kr, uint32_t cr, uint32_t BN, uint32_t& word, uint32_t& nib) {
    const uint32_t j = kr >> 5, w = (kr >> 3) & 3, i = (kr >> 1) & 3, h = kr & 1;
    word = (j * BN + cr) * 4 + w;
    nib = i + 4 * h;
}
}  // namespace fq

using namespace fq;

extern "C" {

const char* fq_last_error(void) { return error_buffer(); }

fq_status_t fq_get_layout(uint32_t K, uint32_t N, uint32_t group, uint32_t bn_hint, uint32_t nb_hint,
                          fq_layout_t* out) {
    if (!out) return fail(FQ_ERR_INVALID_ARG, "fq_get_layout: null output");
    if (group != 64 && group != 128) return fail(FQ_ERR_UNSUPPORTED_SHAPE, "group must be 64 or 128, got %u", group);
    if (K == 0 || K % FQ_BK != 0) return fail(FQ_ERR_UNSUPPORTED_SHAPE, "K = %u is not a multiple of 128", K);
    uint32_t BN = bn_hint;
    if (BN == 0) BN = (N % 256 == 0) ? 256 : 128;
    if (BN != 128 && BN != 256) return fail(FQ_ERR_UNSUPPORTED_SHAPE, "BN must be 128 or 256, got %u", BN);
    if (N == 0 || N % BN != 0) return fail(FQ_ERR_UNSUPPORTED_SHAPE, "N = %u is not a multiple of BN = %u", N, BN);
    if (N / BN > kMaxTilesN) return fail(FQ_ERR_UNSUPPORTED_SHAPE, "N = %u has too many column tiles", N);
    // one bucket per group of four columns {g, g + 8, g + 16, g + 24} of a 32-column block
    const uint32_t NB = BN / 4;
    if (nb_hint != 0 && nb_hint != NB) return fail(FQ_ERR_UNSUPPORTED_SHAPE, "buckets per tile must be BN / 4 = %u, got %u", NB, nb_hint);
    std::memset(out, 0, sizeof(*out));
    out->abi = FQ_ABI_VERSION;
    out->K = K;
    out->N = N;
    out->group = group;
    out->BK = FQ_BK;
    out->BN = BN;
    out->buckets_per_tile = NB;
    out->wq_interleave = 3;
    out->coo_unit_bytes = 16;
    return FQ_OK;
}

// Tile column of column number j of bucket b (buckets are static: 8 * (c / 32) + c % 8).
static inline uint32_t column_of_bucket(uint32_t b, uint32_t j) { return ((b >> 3) << 5) | (b & 7u) | (j << 3); }

fq_status_t fq_pack_int4_sizes(const fq_layout_t* L, size_t* wq_bytes, size_t* scale_bytes, size_t* zero_bytes) {
    if (!layout_ok(L)) return fail(FQ_ERR_INVALID_ARG, "bad layout");
    if (wq_bytes) *wq_bytes = (size_t)L->K * L->N / 2;
    if (scale_bytes) *scale_bytes = (size_t)(L->K / L->group) * L->N * 2;
    if (zero_bytes) *zero_bytes = (size_t)(L->K / L->group) * L->N * 2;
    return FQ_OK;
}

}  // extern "C"

namespace {

// What bounds packing a K x N matrix is reading it (4 bytes a weight and 1 of mask) and one division a weight.  With the
// row loops below vectorised a 4096 x 4096 matrix takes 4.5 ms on 8 cores (21.6 with a branch and a library rounding call for
// each weight); a second pass over a chunk finds it in the core's L2.
// One chunk of the packer is compiled for AVX-512, AVX2 and the baseline instruction set, chosen when the library is
// loaded; the arithmetic is the same IEEE binary32 operations in each (-ffp-contract=off).
#define FQ_SIMD_CLONES __attribute__((target_clones("avx512f", "avx2", "default")))

constexpr uint32_t kMaxBN = 256;

// The loops below select with masks instead of branches, which is what lets the compiler vectorise them.  A mask of all
// ones or none from a truth value:
inline int32_t all_ones(bool b) { return -(int32_t)b; }
inline float select_or_zero(int32_t m, float f) {
    int32_t u;
    std::memcpy(&u, &f, 4);
    u &= m;
    std::memcpy(&f, &u, 4);
    return f;
}

// Range of a group's columns (g rows of W; masked weights count as 0, which the range contains anyway).
FQ_SIMD_CLONES void group_range(const float* W, size_t w_step, const uint8_t* mask, size_t m_step, uint32_t g, uint32_t BN, float* wmin, float* wmax) {
    for (uint32_t c = 0; c < BN; ++c) wmin[c] = 0.0f, wmax[c] = 0.0f;
    for (uint32_t k = 0; k < g; ++k) {
        const float* wr = W + k * w_step;
        const uint8_t* mr = mask + k * m_step;
        for (uint32_t c = 0; c < BN; ++c) {
            const float w = select_or_zero(all_ones(mr[c] == 0), wr[c]);
            wmin[c] = w < wmin[c] ? w : wmin[c];
            wmax[c] = w > wmax[c] ? w : wmax[c];
        }
    }
}

// Scales and zero-points of a group's columns.  A degenerate group (scale 1, zero-point 0, all codes 0) is divided by
// infinity.
FQ_SIMD_CLONES void group_scale(const float* wmin, const float* wmax, uint32_t BN, float* sf, float* zf, uint16_t* scale, uint16_t* zero) {
    for (uint32_t c = 0; c < BN; ++c) {
        const float s32 = (wmax[c] - wmin[c]) / 15.0f;
        uint32_t u;
        std::memcpy(&u, &s32, 4);
        u = (u + 0x7fffu + ((u >> 16) & 1u)) & 0xffff0000u;    // to BF16, nearest even (a NaN gives nothing that is > 0)
        float s;
        std::memcpy(&s, &u, 4);
        const int32_t m = all_ones(s > 0.0f);
        float zq = nearbyintf(-wmin[c] / s);
        zq = zq > 0.0f ? zq : 0.0f;
        zq = zq < 15.0f ? zq : 15.0f;
        zf[c] = select_or_zero(m, zq);                         // 0 to 15: exact in BF16
        uint32_t zu;
        std::memcpy(&zu, &zf[c], 4);
        u = (u & (uint32_t)m) | (0x7f800000u & ~(uint32_t)m);
        std::memcpy(&sf[c], &u, 4);
        scale[c] = (uint16_t)(((u >> 16) & (uint32_t)m) | (0x3f80u & ~(uint32_t)m));
        zero[c] = (uint16_t)(zu >> 16);
    }
}

// The words of eight rows (one word a column): nibble i + 4h is row 2i + h.  An outlier's place holds the zero-point.
FQ_SIMD_CLONES void eight_rows(const float* W, size_t w_step, const uint8_t* mask, size_t m_step, uint32_t BN, const float* sf, const float* zf,
                               uint32_t* words) {
    for (uint32_t c = 0; c < BN; ++c) words[c] = 0;
    for (uint32_t r = 0; r < 8; ++r) {
        const float* wr = W + r * w_step;
        const uint8_t* mr = mask + r * m_step;
        const uint32_t shift = 4 * ((r >> 1) + 4 * (r & 1));
        for (uint32_t c = 0; c < BN; ++c) {
            // clamped before the conversion (not a number gives 0); an outlier counts as 0, whose code is the zero-point
            float v = nearbyintf(select_or_zero(all_ones(mr[c] == 0), wr[c]) / sf[c]) + zf[c];
            v = v > 0.0f ? v : 0.0f;
            v = v < 15.0f ? v : 15.0f;
            words[c] |= (uint32_t)(int32_t)v << shift;
        }
    }
}

}  // namespace

extern "C" {

fq_status_t fq_pack_int4(const fq_layout_t* L, const float* W, const uint8_t* mask, void* wq_out,
                         uint16_t* scale, uint16_t* zero) {
    if (!layout_ok(L)) return fail(FQ_ERR_INVALID_ARG, "bad layout");
    if (!W || !wq_out || !scale || !zero) return fail(FQ_ERR_INVALID_ARG, "fq_pack_int4: null pointer");
    const uint32_t K = L->K, N = L->N, g = L->group, BN = L->BN;
    const uint32_t KT = K / FQ_BK, NT = N / BN, gpc = FQ_BK / g;  // groups per chunk
    uint32_t* wq = (uint32_t*)wq_out;
    const size_t chunk_words = (size_t)16 * BN;
    const std::vector<uint8_t> no_mask(mask ? 0 : FQ_BK * kMaxBN, 0);
    const size_t mask_step = mask ? N : kMaxBN;
    // k-steps outside, column tiles inside: threads that run at the same time read neighbouring parts of the same rows
#pragma omp parallel for schedule(dynamic, 2)
    for (int64_t ch = 0; ch < (int64_t)NT * KT; ++ch) {
        const uint32_t kt = (uint32_t)(ch / NT), tn = (uint32_t)(ch % NT);
        uint32_t* chunk = wq + ((size_t)tn * KT + kt) * chunk_words;
        const size_t n0 = (size_t)tn * BN;
        float wmin[kMaxBN], wmax[kMaxBN], sf[kMaxBN], zf[kMaxBN];
        uint32_t words[4][kMaxBN];
        for (uint32_t gi = 0; gi < gpc; ++gi) {
            const uint32_t k0 = kt * FQ_BK + gi * g;
            const size_t grow = (size_t)(k0 / g);
            const float* Wg = W + (size_t)k0 * N + n0;
            const uint8_t* mg = mask ? mask + (size_t)k0 * N + n0 : no_mask.data();
            group_range(Wg, N, mg, mask_step, g, BN, wmin, wmax);
            group_scale(wmin, wmax, BN, sf, zf, scale + grow * N + n0, zero + grow * N + n0);
            for (uint32_t j = 0; j < g / 32; ++j) {
                for (uint32_t w = 0; w < 4; ++w)
                    eight_rows(Wg + (size_t)(32 * j + 8 * w) * N, N, mg + (32 * j + 8 * w) * mask_step, mask_step, BN, sf, zf, words[w]);
                uint32_t* out = chunk + (size_t)(gi * (g / 32) + j) * BN * 4;
                for (uint32_t c = 0; c < BN; ++c)
                    for (uint32_t w = 0; w < 4; ++w) out[4 * c + w] = words[w][c];
            }
        }
    }
    return FQ_OK;
}

fq_status_t fq_repurpose_pad_slots(const fq_layout_t* L, const float* W, const uint8_t* mask, uint8_t* mask_out,
                                   uint64_t* added_out) {
    if (!layout_ok(L)) return fail(FQ_ERR_INVALID_ARG, "bad layout");
    if (!W || !mask || !mask_out) return fail(FQ_ERR_INVALID_ARG, "fq_repurpose_pad_slots: null pointer");
    const uint32_t K = L->K, N = L->N, g = L->group, BN = L->BN, NB = L->buckets_per_tile;
    const uint32_t KT = K / FQ_BK, NT = N / BN, gpc = FQ_BK / g;
    std::memcpy(mask_out, mask, (size_t)K * N);
    uint64_t added = 0;
#pragma omp parallel reduction(+ : added)
    {
        std::vector<double> err((size_t)FQ_BK * BN);          // quantisation error of every weight of the tile; < 0: not a candidate
        std::vector<uint32_t> count(BN);
        std::vector<std::pair<double, uint32_t>> cand;
#pragma omp for schedule(dynamic, 4)
        for (int64_t ch = 0; ch < (int64_t)NT * KT; ++ch) {
            const uint32_t tn = (uint32_t)(ch / KT), kt = (uint32_t)(ch % KT);
            const size_t n0 = (size_t)tn * BN;
            std::fill(count.begin(), count.end(), 0u);
            for (uint32_t gi = 0; gi < gpc; ++gi) {
                const uint32_t k0 = kt * FQ_BK + gi * g;
                for (uint32_t c = 0; c < BN; ++c) {
                    // Eq. 2 for this group and column under `mask`, as in fq_pack_int4
                    float wmin = 0.0f, wmax = 0.0f;
                    for (uint32_t k = k0; k < k0 + g; ++k) {
                        if (mask[(size_t)k * N + n0 + c]) continue;
                        const float w = W[(size_t)k * N + n0 + c];
                        wmin = std::min(wmin, w), wmax = std::max(wmax, w);
                    }
                    float s = bf16_to_f32(f32_to_bf16_rne((wmax - wmin) / 15.0f));
                    int z = 0;
                    const bool degenerate = !(s > 0.0f);
                    if (!degenerate) {
                        z = (int)nearbyintf(-wmin / s);
                        z = z < 0 ? 0 : (z > 15 ? 15 : z);
                    }
                    for (uint32_t k = k0; k < k0 + g; ++k) {
                        const size_t idx = (size_t)k * N + n0 + c;
                        const float w = W[idx];
                        const bool nonzero = (f32_to_bf16_rne(w) & 0x7fffu) != 0;
                        double e = -1.0;
                        if (mask[idx]) {
                            if (nonzero) ++count[c];
                        } else if (nonzero) {
                            int q = 0;
                            if (!degenerate) {
                                q = (int)nearbyintf(w / s) + z;
                                q = q < 0 ? 0 : (q > 15 ? 15 : q);
                            }
                            const double what = degenerate ? 0.0 : (double)s * ((double)q - (double)z);   // Eq. 3
                            e = std::fabs((double)w - what);
                        }
                        err[(size_t)(k - kt * FQ_BK) * BN + c] = e;
                    }
                }
            }
            for (uint32_t b = 0; b < NB; ++b) {
                uint32_t depth = 0;
                for (uint32_t j = 0; j < 4; ++j) depth = std::max(depth, count[column_of_bucket(b, j)]);
                if (depth > 32) continue;                      // a bucket with a tail keeps its padding
                for (uint32_t j = 0; j < 4; ++j) {
                    const uint32_t c = column_of_bucket(b, j), free_slots = depth - count[c];
                    if (!free_slots) continue;
                    cand.clear();
                    for (uint32_t r = 0; r < FQ_BK; ++r)
                        if (err[(size_t)r * BN + c] > 0.0) cand.emplace_back(err[(size_t)r * BN + c], r);
                    const size_t take = std::min<size_t>(free_slots, cand.size());
                    // larger error first, lower row first among equals
                    std::partial_sort(cand.begin(), cand.begin() + take, cand.end(),
                                      [](const std::pair<double, uint32_t>& x, const std::pair<double, uint32_t>& y) {
                                          return x.first != y.first ? x.first > y.first : x.second < y.second;
                                      });
                    for (size_t i = 0; i < take; ++i) mask_out[(size_t)(kt * FQ_BK + cand[i].second) * N + n0 + c] = 1;
                    added += take;
                }
            }
        }
    }
    if (added_out) *added_out = added;
    return FQ_OK;
}

fq_status_t fq_unpack_int4(const fq_layout_t* L, const void* wq_in, uint8_t* q) {
    if (!layout_ok(L)) return fail(FQ_ERR_INVALID_ARG, "bad layout");
    if (!wq_in || !q) return fail(FQ_ERR_INVALID_ARG, "fq_unpack_int4: null pointer");
    const uint32_t K = L->K, N = L->N, BN = L->BN, KT = K / FQ_BK, NT = N / BN;
    const uint32_t* wq = (const uint32_t*)wq_in;
#pragma omp parallel for schedule(static)
    for (int64_t ch = 0; ch < (int64_t)NT * KT; ++ch) {
        const uint32_t tn = (uint32_t)(ch / KT), kt = (uint32_t)(ch % KT);
        const uint32_t* chunk = wq + (size_t)ch * 16 * BN;
        for (uint32_t kr = 0; kr < FQ_BK; ++kr)
            for (uint32_t c = 0; c < BN; ++c) {
                uint32_t word, nib;
                wq_slot(kr, c, BN, word, nib);
                q[(size_t)(kt * FQ_BK + kr) * N + (size_t)tn * BN + c] = (uint8_t)((chunk[word] >> (4 * nib)) & 0xf);
            }
    }
    return FQ_OK;
}

}  // extern "C"

// ------------------------------------------------------------------ Tile-COO encoder

namespace {

struct Entry {
    uint8_t k, c;
    uint32_t v;      // the slot's 19 value bits
};

struct Encoded {
    std::vector<uint32_t> indptr;   // N_tile + 1
    std::vector<uint32_t> info;     // N_tile * NB
    uint32_t max_tile_packets = 0;
    uint32_t max_bucket_packets = 0;
    uint32_t max_tail_packets = 0;
    bool repeated = false;          // some position appears more than once
};

// Bucket of a tile column: the four columns {g, g + 8, g + 16, g + 24} of a 32-column block share
// bucket 8 * (c / 32) + c % 8.  These are the columns whose accumulators one group of four lanes
// holds in the kernels, so a bucket's outliers are applied in registers.
inline uint32_t bucket_of(uint32_t c) { return ((c >> 5) << 3) | (c & 7u); }
// Number of a column inside its bucket, and the way back.
inline uint32_t number_in_bucket(uint32_t c) { return (c >> 3) & 3u; }
inline uint32_t column_of(uint32_t b, uint32_t j) { return ((b >> 3) << 5) | (b & 7u) | (j << 3); }

// One outlier as a 32-bit word: the 19 value bits from bit 13 up, row * 32 in bits 5-11, the column's number
// inside the bucket in bits 3-4.
inline uint32_t entry_word(uint32_t k, uint32_t j, uint32_t v19) { return (v19 << fq::kSlotValueShift) | (j << fq::kSlotColShift) | (k << 5); }

// IEEE binary16 bits -> the FP32 number's bits (every binary16 number is an FP32 number with at most ten fraction
// bits), and back (exact for such numbers; `ok` says whether it was one).
inline uint32_t f16_to_f32_bits(uint16_t h) {
    const uint32_t sign = (uint32_t)(h & 0x8000u) << 16, e = (h >> 10) & 31u, f = h & 1023u;
    if (e == 31) return sign | 0x7f800000u | (f << 13);
    if (e != 0) return sign | ((e + 112u) << 23) | (f << 13);
    if (f == 0) return sign;
    int shift = 0;
    uint32_t m = f;
    while (!(m & 1024u)) m <<= 1, ++shift;                 // normalise the subnormal
    return sign | ((uint32_t)(113 - shift) << 23) | ((m & 1023u) << 13);
}
inline uint16_t f32_bits_to_f16(uint32_t u, bool* ok) {
    const uint16_t sign = (uint16_t)((u >> 16) & 0x8000u);
    const int e = (int)((u >> 23) & 255u) - 127;
    const uint32_t f = u & 0x7fffffu;
    uint16_t h;
    if (((u >> 23) & 255u) == 255u) h = (uint16_t)(sign | 0x7c00u | (f >> 13));
    else if ((u & 0x7fffffffu) == 0) h = sign;
    else if (e >= -14 && e <= 15) h = (uint16_t)(sign | ((uint32_t)(e + 15) << 10) | (f >> 13));
    else if (e >= -24 && e < -14) h = (uint16_t)(sign | ((0x800000u | f) >> (13 + (-14 - e))));
    else h = (uint16_t)(sign | 0x7c00u);                   // out of range
    *ok = f16_to_f32_bits(h) == u;
    return h;
}
// The caller's 16 value bits as the slot's 19 value bits, and back.
inline uint32_t value_field(uint16_t v, uint32_t value_type) {
    return value_type == FQ_VALUE_FP16 ? f16_to_f32_bits(v) >> fq::kSlotValueShift : (uint32_t)v << 3;
}

// A column with more entries than this in one tile gives its bucket a tail.
constexpr uint32_t kSlottedMax = 32;
// Column-slotted packets of a bucket that has a tail.
constexpr uint32_t kSlottedWithTail = 4;

// Encoding is two passes over the entries (count and move, by tile) and one over the tiles, each entry moved as one
// word; the packets of a tile are counted first, so that the second pass writes them where they belong.  168 thousand outliers
// of a 4096 x 4096 matrix: 3.4 ms on 8 cores (13.9 before, and twice that through a caller that asked for the sizes first); at 5 %
// of a 4096 x 8192 matrix 42 ms (290), where the search for a conflict-free order takes most of the time.
//
// The entries by tile (input order within a tile): a counting sort whose counting and moving are shared out over the
// threads, each with a contiguous part of the input.  Values of +-0 are dropped.
fq_status_t sort_by_tile(const fq_layout_t* L, const uint32_t* k, const uint32_t* n, const uint16_t* v, size_t nnz,
                         std::vector<size_t>& tstart, std::unique_ptr<Entry[]>& sorted) {
    const uint32_t K = L->K, N = L->N, KT = K / FQ_BK, bn_shift = L->BN == 256 ? 8 : 7;
    const size_t ntile = (size_t)KT * (N / L->BN);
    const int parts = (int)std::max<size_t>(1, std::min<size_t>({(size_t)omp_get_max_threads(), nnz / 4096, (size_t)64}));
    std::vector<uint32_t> place((size_t)parts * ntile, 0);
    size_t bad = nnz;
    auto tile_of = [&](size_t e) { return (size_t)(n[e] >> bn_shift) * KT + k[e] / FQ_BK; };
#pragma omp parallel for schedule(static, 1) reduction(min : bad)
    for (int t = 0; t < parts; ++t) {
        uint32_t* count = &place[(size_t)t * ntile];
        for (size_t e = nnz * t / parts; e < nnz * (t + 1) / parts; ++e) {
            if (k[e] >= K || n[e] >= N) { bad = std::min(bad, e); break; }
            if ((v[e] & 0x7fffu) != 0) ++count[tile_of(e)];
        }
    }
    if (bad < nnz) return fq::fail(FQ_ERR_INVALID_ARG, "outlier %zu at (%u, %u) is outside the %u x %u matrix", bad, k[bad], n[bad], K, N);
    tstart.assign(ntile + 1, 0);
    for (size_t tile = 0; tile < ntile; ++tile) {
        size_t in_tile = 0;
        for (int t = 0; t < parts; ++t) {
            const uint32_t c = place[(size_t)t * ntile + tile];
            place[(size_t)t * ntile + tile] = (uint32_t)in_tile;
            in_tile += c;
        }
        tstart[tile + 1] = tstart[tile] + in_tile;
    }
    sorted.reset(new Entry[std::max<size_t>(1, tstart[ntile])]);
#pragma omp parallel for schedule(static, 1)
    for (int t = 0; t < parts; ++t) {
        uint32_t* at = &place[(size_t)t * ntile];
        for (size_t e = nnz * t / parts; e < nnz * (t + 1) / parts; ++e) {
            if ((v[e] & 0x7fffu) == 0) continue;
            const size_t tile = tile_of(e);
            sorted[tstart[tile] + at[tile]++] = Entry{(uint8_t)(k[e] % FQ_BK), (uint8_t)(n[e] & (L->BN - 1)), value_field(v[e], L->value_type)};
        }
    }
    return FQ_OK;
}

// Packet counts of every tile and bucket: a bucket's depth is its longest column, or kSlottedWithTail when that column is
// too long; then the entries beyond each column's first kSlottedWithTail make the tail, four to a packet.
fq_status_t count_packets(const fq_layout_t* L, const std::vector<size_t>& tstart, const Entry* sorted, Encoded& E) {
    const uint32_t NB = L->buckets_per_tile;
    const size_t ntile = tstart.size() - 1;
    E.indptr.assign(ntile + 1, 0);
    E.info.resize(ntile * NB);
    int bad = 0;
    uint32_t max_bucket = 0, max_tail = 0, max_tile = 0;
#pragma omp parallel for schedule(dynamic, 16) reduction(max : max_bucket, max_tail, max_tile) reduction(| : bad)
    for (int64_t t = 0; t < (int64_t)ntile; ++t) {
        uint32_t count[kMaxBN] = {0};
        for (size_t e = tstart[t]; e < tstart[t + 1]; ++e) ++count[sorted[e].c];
        uint32_t off = 0;
        for (uint32_t b = 0; b < NB; ++b) {
            uint32_t longest = 0, rest = 0;
            for (uint32_t j = 0; j < 4; ++j) {
                const uint32_t c = count[column_of(b, j)];
                longest = std::max(longest, c);
                rest += c > kSlottedWithTail ? c - kSlottedWithTail : 0;
            }
            const uint32_t depth = longest > kSlottedMax ? kSlottedWithTail : longest;
            const uint32_t tail = longest > kSlottedMax ? (rest + 3) / 4 : 0;
            bad |= off > 0xffffu || tail > 0xffu;
            E.info[(size_t)t * NB + b] = (off & 0xffffu) | (depth << 16) | (tail << 24);
            max_bucket = std::max(max_bucket, depth + tail);
            max_tail = std::max(max_tail, tail);
            off += depth + tail;
        }
        E.indptr[t + 1] = off;
        max_tile = std::max(max_tile, off);
    }
    if (bad) return fq::fail(FQ_ERR_UNSUPPORTED_SHAPE, "a bucket exceeds the packet offset/count range of its descriptor");
    E.max_bucket_packets = max_bucket, E.max_tail_packets = max_tail, E.max_tile_packets = max_tile;
    uint64_t total = 0;
    for (size_t t = 0; t < ntile; ++t) {
        total += E.indptr[t + 1];
        if (total > 0xffffffffull) return fq::fail(FQ_ERR_UNSUPPORTED_SHAPE, "more than 2^32 packets");
        E.indptr[t + 1] = (uint32_t)total;
    }
    return FQ_OK;
}

// Which of its column-slotted packets holds which of a column's outliers is free (the sum is order-independent up to
// rounding).  By row: packet i holds the column's i-th.  Bank-aware (Section 3.2.2's element reordering, restated for a
// k-major FP32 copy of eight activation rows, 32 B per row, where rows with equal k mod 4 share banks): one load instruction
// of a warp reads slot j of packet d of its eight buckets and is served half a warp, i.e. four neighbouring buckets, at
// a time, in as many passes as the fullest bank group has different rows.  So for every four neighbouring buckets, slot j
// and packet number d in turn, the rows are chosen among what the four columns still have to place (or padding, row 0, where
// a column has places to spare) such that the passes are fewest; then such that the paddings are fewest (outliers placed
// early leave later packets more freedom); then the first combination, lowest rows first.
//
// The columns of one slot j of four neighbouring buckets: `list[q]` their entries by row, `todo[q]` how many of them go
// into packets, `depth[q]` the packets of the bucket; `out[q][d]` = index into the list + 1, 0 = padding.
void place_bank_aware(const Entry* const (&list)[4], const uint32_t (&todo)[4], const uint32_t (&depth)[4], uint8_t (&out)[4][kSlottedMax]) {
    uint32_t left[4], dmax = 0;                            // entries still to place, a bit each
    for (int q = 0; q < 4; ++q) {
        left[q] = todo[q] >= 32 ? ~0u : (1u << todo[q]) - 1;
        dmax = std::max(dmax, depth[q]);
    }
    for (uint32_t d = 0; d < dmax; ++d) {
        // candidates per bucket: up to four unplaced outliers (lowest rows first), padding if the column has a place to
        // spare; a bucket whose list has ended reads row 0 whatever happens
        int cand[4][5], ncand[4];
        uint32_t row[4][5], forced = 0;                    // forced: paddings that no choice avoids
        for (int q = 0; q < 4; ++q) {
            ncand[q] = 0;
            if (d < depth[q]) {
                for (uint32_t m = left[q]; m && ncand[q] < 4; m &= m - 1) {
                    cand[q][ncand[q]] = __builtin_ctz(m);
                    row[q][ncand[q]] = list[q][cand[q][ncand[q]]].k;
                    ++ncand[q];
                }
                forced += left[q] == 0;
            }
            if (d >= depth[q] || (uint32_t)__builtin_popcount(left[q]) < depth[q] - d) cand[q][ncand[q]] = -1, row[q][ncand[q]++] = 0;
        }
        // Two rows clash if they differ and share banks; the passes are the size of the largest set of rows that clash with
        // one another.  Passes and paddings only grow with every bucket that is added, so a beginning that is no better
        // than the best combination so far is given up, and a combination at the lower bound ends the search.
        auto clash = [](uint32_t a, uint32_t b) { return a != b && ((a ^ b) & 3u) == 0; };
        int best[4] = {0, 0, 0, 0};
        uint32_t best_cost = 1u << 30;
        const uint32_t bound = 16 + forced;
        for (int i0 = 0; i0 < ncand[0] && best_cost > bound; ++i0) {
            const uint32_t r0 = row[0][i0], pad0 = cand[0][i0] < 0 && d < depth[0];
            for (int i1 = 0; i1 < ncand[1] && best_cost > bound; ++i1) {
                const uint32_t r1 = row[1][i1], pad1 = pad0 + (cand[1][i1] < 0 && d < depth[1]);
                const bool c01 = clash(r0, r1);
                if ((c01 ? 32 : 16) + pad1 >= best_cost) continue;
                for (int i2 = 0; i2 < ncand[2] && best_cost > bound; ++i2) {
                    const uint32_t r2 = row[2][i2], pad2 = pad1 + (cand[2][i2] < 0 && d < depth[2]);
                    const bool c02 = clash(r0, r2), c12 = clash(r1, r2);
                    const uint32_t p3 = c01 && c02 && c12 ? 3 : (c01 || c02 || c12 ? 2 : 1);
                    if (p3 * 16 + pad2 >= best_cost) continue;
                    for (int i3 = 0; i3 < ncand[3]; ++i3) {
                        const uint32_t r3 = row[3][i3], pads = pad2 + (cand[3][i3] < 0 && d < depth[3]);
                        const bool c03 = clash(r0, r3), c13 = clash(r1, r3), c23 = clash(r2, r3);
                        uint32_t passes = p3;
                        if (p3 == 3 && c03 && c13 && c23) passes = 4;
                        else if ((c01 && c03 && c13) || (c02 && c03 && c23) || (c12 && c13 && c23)) passes = 3;
                        else if (c03 || c13 || c23) passes = std::max(passes, 2u);
                        const uint32_t cost = passes * 16 + pads;
                        if (cost < best_cost) best_cost = cost, best[0] = i0, best[1] = i1, best[2] = i2, best[3] = i3;
                    }
                }
            }
        }
        for (int q = 0; q < 4; ++q) {
            const int e = cand[q][best[q]];
            if (d < depth[q]) out[q][d] = (uint8_t)(e + 1);
            if (e >= 0) left[q] &= ~(1u << e);
        }
    }
}

// The packets of one tile: per bucket the column-slotted ones and, for a bucket with a long column, the tail (by (row, column),
// four to a packet).  True if a position appears twice.
bool write_tile(const fq_layout_t* L, const Entry* entries, size_t count, const uint32_t* info, uint32_t* words, std::vector<Entry>& by_col,
                std::vector<Entry>& rest) {
    const uint32_t NB = L->buckets_per_tile;
    // entries by column, then by row
    uint32_t start[kMaxBN + 1] = {0}, fill[kMaxBN];
    for (size_t e = 0; e < count; ++e) ++start[entries[e].c + 1];
    for (uint32_t c = 0; c < L->BN; ++c) start[c + 1] += start[c], fill[c] = start[c];
    if (by_col.size() < count) by_col.resize(count);
    for (size_t e = 0; e < count; ++e) by_col[fill[entries[e].c]++] = entries[e];
    bool repeated = false;
    for (uint32_t c = 0; c < L->BN; ++c) {
        Entry *a = by_col.data() + start[c], *b = by_col.data() + start[c + 1];
        bool sorted = true;
        for (Entry* e = a + 1; e < b; ++e) sorted &= e[-1].k <= e->k;
        if (a < b && !sorted) std::sort(a, b, [](const Entry& x, const Entry& y) { return x.k < y.k; });
        for (Entry* e = a + 1; e < b; ++e) repeated |= e[-1].k == e->k;
    }
    uint8_t place[4][4][kSlottedMax];                      // [bucket - b0][j][d]
    for (uint32_t b0 = 0; b0 < NB; b0 += 4) {
        const Entry* list[4][4];                           // [j][bucket - b0]
        uint32_t size[4][4], todo[4], depth[4];
        for (uint32_t q = 0; q < 4; ++q) depth[q] = (info[b0 + q] >> 16) & 0xffu;
        for (uint32_t j = 0; j < 4; ++j) {
            for (uint32_t q = 0; q < 4; ++q) {
                const uint32_t c = column_of(b0 + q, j);
                list[j][q] = by_col.data() + start[c];
                size[j][q] = start[c + 1] - start[c];
                todo[q] = std::min(size[j][q], depth[q]);
            }
            uint8_t slot[4][kSlottedMax];
            if (L->slot_order == 1) {
                for (uint32_t q = 0; q < 4; ++q)
                    for (uint32_t d = 0; d < depth[q]; ++d) slot[q][d] = d < todo[q] ? d + 1 : 0;
            } else {
                place_bank_aware(list[j], todo, depth, slot);
            }
            for (uint32_t q = 0; q < 4; ++q) std::memcpy(place[q][j], slot[q], depth[q]);
        }
        for (uint32_t q = 0; q < 4; ++q) {
            uint32_t* w = words + 4 * (size_t)(info[b0 + q] & 0xffffu);
            for (uint32_t d = 0; d < depth[q]; ++d)
                for (uint32_t j = 0; j < 4; ++j) {
                    const uint32_t e = place[q][j][d];
                    *w++ = e ? entry_word(list[j][q][e - 1].k, j, list[j][q][e - 1].v) : entry_word(0, j, 0);
                }
            const uint32_t tail = info[b0 + q] >> 24;
            if (!tail) continue;
            rest.clear();
            for (uint32_t j = 0; j < 4; ++j)
                if (size[j][q] > depth[q]) rest.insert(rest.end(), list[j][q] + depth[q], list[j][q] + size[j][q]);
            std::sort(rest.begin(), rest.end(), [](const Entry& x, const Entry& y) { return x.k != y.k ? x.k < y.k : x.c < y.c; });
            for (const Entry& e : rest) *w++ = entry_word(e.k, number_in_bucket(e.c), e.v);
            for (size_t z = rest.size(); z < (size_t)tail * 4; ++z) *w++ = 0;
        }
    }
    return repeated;
}

}  // namespace

extern "C" {

fq_status_t fq_encode_tilecoo_sizes(const fq_layout_t* L, const uint32_t* k, const uint32_t* n,
                                    const uint16_t* v, size_t nnz, size_t* n_indptr, size_t* n_bucket_info,
                                    size_t* n_packets, uint32_t* max_tile_packets) {
    if (!layout_ok(L)) return fail(FQ_ERR_INVALID_ARG, "bad layout");
    if (nnz && (!k || !n || !v)) return fail(FQ_ERR_INVALID_ARG, "fq_encode_tilecoo_sizes: null pointer");
    Encoded E;
    std::vector<size_t> tstart;
    std::unique_ptr<Entry[]> sorted;
    fq_status_t st = sort_by_tile(L, k, n, v, nnz, tstart, sorted);
    if (st == FQ_OK) st = count_packets(L, tstart, sorted.get(), E);
    if (st != FQ_OK) return st;
    if (n_indptr) *n_indptr = E.indptr.size();
    if (n_bucket_info) *n_bucket_info = E.info.size();
    if (n_packets) *n_packets = E.indptr.back();
    if (max_tile_packets) *max_tile_packets = E.max_tile_packets;
    return FQ_OK;
}

fq_status_t fq_encode_tilecoo(fq_layout_t* L, const uint32_t* k, const uint32_t* n, const uint16_t* v,
                              size_t nnz, uint32_t* tile_indptr, uint32_t* bucket_info, void* packed,
                              size_t n_packets) {
    if (!layout_ok(L)) return fail(FQ_ERR_INVALID_ARG, "bad layout");
    if ((nnz && (!k || !n || !v)) || !tile_indptr || !bucket_info) return fail(FQ_ERR_INVALID_ARG, "fq_encode_tilecoo: null pointer");
    Encoded E;
    std::vector<size_t> tstart;
    std::unique_ptr<Entry[]> sorted;
    fq_status_t st = sort_by_tile(L, k, n, v, nnz, tstart, sorted);
    if (st == FQ_OK) st = count_packets(L, tstart, sorted.get(), E);
    if (st != FQ_OK) return st;
    if (E.indptr.back() > n_packets) return fail(FQ_ERR_BUFFER_TOO_SMALL, "packed_outliers holds %zu packets, %zu needed", n_packets, (size_t)E.indptr.back());
    if (E.indptr.back() && !packed) return fail(FQ_ERR_INVALID_ARG, "fq_encode_tilecoo: null packet buffer");
    int repeated = 0;
#pragma omp parallel reduction(| : repeated)
    {
        std::vector<Entry> by_col, rest;
#pragma omp for schedule(dynamic, 4)
        for (int64_t t = 0; t < (int64_t)E.indptr.size() - 1; ++t)
            if (tstart[t + 1] > tstart[t])
                repeated |= write_tile(L, sorted.get() + tstart[t], tstart[t + 1] - tstart[t], &E.info[(size_t)t * L->buckets_per_tile],
                                       (uint32_t*)packed + 4 * (size_t)E.indptr[t], by_col, rest);
    }
    E.repeated = repeated != 0;
    std::memcpy(tile_indptr, E.indptr.data(), E.indptr.size() * 4);
    std::memcpy(bucket_info, E.info.data(), E.info.size() * 4);
    L->max_tile_packets = E.max_tile_packets;
    L->max_bucket_packets = E.max_bucket_packets;
    L->max_tail_packets = E.max_tail_packets;
    L->tilecoo_encoded = E.repeated ? 2 : 1;
    L->abi = FQ_ABI_ENCODED;
    return FQ_OK;
}

fq_status_t fq_decode_tilecoo(const fq_layout_t* L, const uint32_t* indptr, const uint32_t* info,
                              const void* packed, uint32_t* k, uint32_t* n, uint16_t* v, size_t* nnz_inout) {
    if (!layout_ok(L)) return fail(FQ_ERR_INVALID_ARG, "bad layout");
    if (!indptr || !info || !nnz_inout) return fail(FQ_ERR_INVALID_ARG, "fq_decode_tilecoo: null pointer");
    const uint32_t BN = L->BN, NB = L->buckets_per_tile, KT = L->K / FQ_BK, NT = L->N / BN;
    const uint32_t* pw = (const uint32_t*)packed;
    const size_t cap = *nnz_inout;
    size_t c = 0;
    for (uint32_t tn = 0; tn < NT; ++tn)
        for (uint32_t kt = 0; kt < KT; ++kt) {
            size_t t = (size_t)tn * KT + kt;
            for (uint32_t b = 0; b < NB; ++b) {
                const uint32_t inf = info[t * NB + b];
                const size_t i0 = (size_t)indptr[t] + (inf & 0xffffu), cnt = ((inf >> 16) & 0xffu) + (inf >> 24);
                for (size_t i = 0; i < cnt * 4; ++i) {
                    const uint32_t w = pw[i0 * 4 + i];
                    if ((w & fq::kSlotValueMask) == 0) continue;
                    if (c >= cap) return fail(FQ_ERR_BUFFER_TOO_SMALL, "decode buffer holds %zu entries", cap);
                    k[c] = kt * FQ_BK + ((w >> 5) & 127u);
                    n[c] = tn * BN + column_of(b, (w >> fq::kSlotColShift) & 3u);
                    if (L->value_type == FQ_VALUE_FP16) {
                        bool ok = true;
                        v[c] = f32_bits_to_f16(w & fq::kSlotValueMask, &ok);
                        if (!ok) return fail(FQ_ERR_FORMAT, "a value of tile %zu is not an IEEE binary16 number", t);
                    } else {
                        if (w & 0xe000u) return fail(FQ_ERR_FORMAT, "a value of tile %zu is not a BF16 number", t);
                        v[c] = (uint16_t)(w >> 16);
                    }
                    ++c;
                }
            }
        }
    *nnz_inout = c;
    return FQ_OK;
}

fq_status_t fq_validate_tilecoo(const fq_layout_t* L, const uint32_t* indptr, const uint32_t* info,
                                const void* packed, size_t n_packets) {
    if (!layout_ok(L)) return fail(FQ_ERR_INVALID_ARG, "bad layout");
    if (!indptr || !info || (n_packets && !packed)) return fail(FQ_ERR_INVALID_ARG, "fq_validate_tilecoo: null pointer");
    const uint32_t BN = L->BN, NB = L->buckets_per_tile;
    const size_t ntile = (size_t)(L->K / FQ_BK) * (L->N / BN);
    const uint32_t* pw = (const uint32_t*)packed;
    if (indptr[0] != 0) return fail(FQ_ERR_FORMAT, "tile_indptr[0] = %u, expected 0", indptr[0]);
    for (size_t t = 0; t < ntile; ++t) {
        if (indptr[t + 1] < indptr[t]) return fail(FQ_ERR_FORMAT, "tile_indptr decreases at tile %zu", t);
        const uint32_t tile_pk = indptr[t + 1] - indptr[t];
        if ((size_t)indptr[t + 1] > n_packets) return fail(FQ_ERR_FORMAT, "tile %zu ends at packet %u of %zu", t, indptr[t + 1], n_packets);
        for (uint32_t b = 0; b < NB; ++b) {
            const uint32_t inf = info[t * NB + b];
            const uint32_t off = inf & 0xffffu, depth = (inf >> 16) & 0xffu, tail = inf >> 24;
            if (off + depth + tail > tile_pk) return fail(FQ_ERR_FORMAT, "bucket %u of tile %zu covers packets [%u, %u) of %u", b, t, off, off + depth + tail, tile_pk);
            if (depth > kSlottedMax) return fail(FQ_ERR_FORMAT, "bucket %u of tile %zu has %u column-slotted packets, at most %u allowed", b, t, depth, kSlottedMax);
            for (uint32_t i = 0; i < (depth + tail) * 4; ++i) {
                const uint32_t w = pw[((size_t)indptr[t] + off) * 4 + i];
                if (L->value_type == FQ_VALUE_FP16) {
                    bool ok = true;
                    f32_bits_to_f16(w & fq::kSlotValueMask, &ok);
                    if (!ok) return fail(FQ_ERR_FORMAT, "a value in bucket %u of tile %zu is not an IEEE binary16 number", b, t);
                } else if (w & 0xe000u) {
                    return fail(FQ_ERR_FORMAT, "a value in bucket %u of tile %zu is not a BF16 number", b, t);
                }
                if (w & fq::kSlotStrayMask) return fail(FQ_ERR_FORMAT, "bits outside the fields are set in a slot of bucket %u, tile %zu", b, t);
                if (i < depth * 4 && ((w >> fq::kSlotColShift) & 3u) != (i & 3u))
                    return fail(FQ_ERR_FORMAT, "slot %u of a column-slotted packet of bucket %u, tile %zu, names column number %u", i & 3u, b, t, (w >> fq::kSlotColShift) & 3u);
            }
        }
    }
    if ((size_t)indptr[ntile] != n_packets) return fail(FQ_ERR_FORMAT, "tile_indptr ends at %u, %zu packets given", indptr[ntile], n_packets);
    return FQ_OK;
}

}  // extern "C"
