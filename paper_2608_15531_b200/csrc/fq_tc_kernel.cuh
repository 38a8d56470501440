// The fused operator on the fifth-generation tensor cores (tcgen05.mma kind::f16, FP32 accumulation), for launches of
// more rows than a warp-level MMA is made for.  Included by fq_kernels.cu inside namespace fq, after the PTX helpers.
//
// Arithmetic.  The A operand is the exact integers q - z as BF16 (weights on the M side, thread = output column), the
// B operand the BF16 activations as they are (batch rows on the N side).  Once per quantisation group the FP32 sums
// leave tensor memory and the scale is applied in FP32:
//     acc[m] += s * sum_k x (q - z)                                     (Eq. 3 inside Eq. 1)
// The outliers need no scale.  They are written, as they are, into a dense BF16 tile in shared memory that is zero
// elsewhere (Section 4.2's scatter, with the weights instead of the products as what is scattered), and a second MMA
// with the same activations adds X W_O into an accumulator of its own that stays in tensor memory over all of K.  A
// tile of zeros costs MMA time whatever the density, but none of the gathers, multiply-adds and registers of a step that
// adds each outlier for every batch row: with 32 rows and more, the tensor pipe does it in less time than the shared
// memory could deliver the activations to such a step.  An FP16 outlier (ten fraction bits) goes in two parts, each a
// BF16 number, one tile after the other.
//
// A unit is one k-step of 128 rows by 128 columns (a stored tile of 256 columns is two column tiles here).  One
// persistent CTA per SM walks a range of units through a ring of shared-memory stages (bulk copies + mbarrier
// expect_tx, Section 4.1).
//
//   warps 0, 2      producers: warp 0 copies a unit's codes, scales and zero-points, warp 2 its X block (tiled tensor
//                   copies, 128-byte swizzle: the K-major MMA operand)
//   warps 1, 3      tensor: per unit 8 MMAs of K = 16 with A from tensor memory (warp 1, dense) and 8 with A from shared
//                   memory (warp 3, outliers).  Two warps, because a warp's wait on a barrier costs it about 100 clocks
//                   even when the barrier is ready, and the MMAs of the other fill them
//   unpack warps    (8 or 12) per 32 rows one 128-bit load of a column's 32 codes, seven logic operations and four BF16 pair
//                   subtractions per eight codes, tcgen05.st into a ring of A operands
//   drain warps     thread = column, 32 batch rows (4 warps for each 32 rows): tcgen05.ld of the group's sums, one FMA per
//                   batch row; at the end of a piece the outlier accumulator, the split-tile settlement and the BF16
//                   store of Y
//   scatter warps   (4 to 12) thread = column: take the previous outliers out of the tile and put the unit's in
//
// What bounds it, per unit in SM clocks: HBM at the measured copy rate would need 425; 8 dense + 8 outlier MMAs issued back
// to back with their commits take 430 at N = 16, 490 at 32, 650 at 64, 1030 at 128 (an outlier MMA is bound by reading its 4 KB
// of A from shared memory up to N = 64).  The kernel takes 1100 at 32 rows and 1880 at 112 (8192 x 28672, 1 % of outliers: 53.4
// and 92.9 us).  That is instruction issue and latency: 2660 warp instructions a unit at 32 rows and 4530 at 128 fill 67 % of the issue
// slots (980 to 1210 of them on the half-rate integer pipe, half of those the unpacking, seven logic operations and four BF16 pair
// additions for eight codes), and every role's work on a unit is a chain of barriers and memory latencies of 800 clocks and
// more, which the groups of warps taking units in turn hide only in part.  At 128 rows the tensor pipe is busy 61 % of the time,
// the drain's FMAs come on top, and both variants spill.  Outliers cost little: 52.7 us without any at 32 rows, 57.0 at 3 %
// (1 %: 53.6).
// Before, launches of 17 to 32 rows ran on the 8-bit integer tensor path, activations as three limbs and outliers applied row
// by row (8192 x 28672 at 32 rows 124.5 us; 4096 x 28672 at 128 rows, in four launches, 305, now 53).

__device__ __forceinline__ bool elect_one() {
    uint32_t e;
    asm volatile("{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n selp.u32 %0, 1, 0, e;\n}" : "=r"(e));
    return e != 0;
}

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
        "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
// 16 or 32 consecutive 32-bit cells of this thread's tensor-memory lane
template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&r)[N]) {
    if constexpr (N == 16) {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]), "=f"(r[8]),
              "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
            : "r"(taddr) : "memory");
    } else {
        static_assert(N == 32, "unsupported tcgen05.ld width");
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
            "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
            : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]), "=f"(r[8]),
              "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15]), "=f"(r[16]),
              "=f"(r[17]), "=f"(r[18]), "=f"(r[19]), "=f"(r[20]), "=f"(r[21]), "=f"(r[22]), "=f"(r[23]), "=f"(r[24]),
              "=f"(r[25]), "=f"(r[26]), "=f"(r[27]), "=f"(r[28]), "=f"(r[29]), "=f"(r[30]), "=f"(r[31])
            : "r"(taddr) : "memory");
    }
}

// The eight MMAs of a unit, D[128 x N] (+)= A[128 x 16] * B[16 x N] for each 16 of its 128 k, BF16 in, FP32 out, and the
// commits that follow them.  Whole warp, converged, with warp-uniform operands; one elected lane issues.  One asm block, so
// that the address arithmetic is not in a divergent branch: there the operands of each MMA have to be moved into
// uniform registers one by one, and an MMA cost 45 to 120 clocks to issue instead of the 10 it runs (N = 16).
// `b0`, `b1`: lower words of the descriptors of the two halves of K, `b_hi` their upper word.
// Dense: A in tensor memory (8 columns to 16 k), the first four MMAs into d0 and the others into d1 (the second group's
// sums, starting afresh, or the same ones).
__device__ __forceinline__ void umma_dense(uint32_t d0, uint32_t d1, uint32_t acc1, uint32_t a, uint32_t b0, uint32_t b1, uint32_t b_hi,
                                           uint32_t idesc, uint32_t bar0, uint32_t bar1, uint32_t bar2) {
    asm volatile(
        "{\n .reg .pred e, f;\n .reg .b32 a, b;\n .reg .b64 x, y;\n elect.sync _|e, 0xffffffff;\n setp.ne.b32 f, %6, 0;\n"
        " add.u32 a, %1, 0;\n"
        " add.u32 b, %2, 0;\n mov.b64 y, {b, %4};\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [a], y, %5, f;\n"
        " setp.eq.b32 f, %6, %6;\n"
        " add.u32 a, %1, 8;\n"
        " add.u32 b, %2, 2;\n mov.b64 y, {b, %4};\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [a], y, %5, f;\n"
        " add.u32 a, %1, 16;\n"
        " add.u32 b, %2, 4;\n mov.b64 y, {b, %4};\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [a], y, %5, f;\n"
        " add.u32 a, %1, 24;\n"
        " add.u32 b, %2, 6;\n mov.b64 y, {b, %4};\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [a], y, %5, f;\n"
        " add.u32 a, %1, 32;\n"
        " add.u32 b, %3, 0;\n mov.b64 y, {b, %4};\n"
        " setp.ne.b32 f, %8, 0;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%7], [a], y, %5, f;\n"
        " setp.eq.b32 f, %6, %6;\n"
        " add.u32 a, %1, 40;\n"
        " add.u32 b, %3, 2;\n mov.b64 y, {b, %4};\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%7], [a], y, %5, f;\n"
        " add.u32 a, %1, 48;\n"
        " add.u32 b, %3, 4;\n mov.b64 y, {b, %4};\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%7], [a], y, %5, f;\n"
        " add.u32 a, %1, 56;\n"
        " add.u32 b, %3, 6;\n mov.b64 y, {b, %4};\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%7], [a], y, %5, f;\n"
        " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%9];\n"
        " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%10];\n"
        " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%11];\n}"
        ::"r"(d0), "r"(a), "r"(b0), "r"(b1), "r"(b_hi), "r"(idesc), "r"(0u), "r"(d1), "r"(acc1), "r"(bar0), "r"(bar1), "r"(bar2)
        : "memory");
}
// Outliers: A behind a shared-memory descriptor (4096 bytes to 16 k), all into d, which the first overwrites unless `acc`.
__device__ __forceinline__ void umma_outliers(uint32_t d, uint32_t a, uint32_t a_hi, uint32_t b0, uint32_t b1, uint32_t b_hi, uint32_t idesc,
                                              uint32_t acc, uint32_t bar0) {
    asm volatile(
        "{\n .reg .pred e, f;\n .reg .b32 a, b;\n .reg .b64 x, y;\n elect.sync _|e, 0xffffffff;\n setp.ne.b32 f, %6, 0;\n"
        " add.u32 a, %1, 0;\n"
        " add.u32 b, %2, 0;\n mov.b64 y, {b, %4};\n"
        " mov.b64 x, {a, %7};\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %5, f;\n"
        " setp.eq.b32 f, %6, %6;\n"
        " add.u32 a, %1, 256;\n"
        " add.u32 b, %2, 2;\n mov.b64 y, {b, %4};\n"
        " mov.b64 x, {a, %7};\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %5, f;\n"
        " add.u32 a, %1, 512;\n"
        " add.u32 b, %2, 4;\n mov.b64 y, {b, %4};\n"
        " mov.b64 x, {a, %7};\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %5, f;\n"
        " add.u32 a, %1, 768;\n"
        " add.u32 b, %2, 6;\n mov.b64 y, {b, %4};\n"
        " mov.b64 x, {a, %7};\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %5, f;\n"
        " add.u32 a, %1, 1024;\n"
        " add.u32 b, %3, 0;\n mov.b64 y, {b, %4};\n"
        " mov.b64 x, {a, %7};\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %5, f;\n"
        " add.u32 a, %1, 1280;\n"
        " add.u32 b, %3, 2;\n mov.b64 y, {b, %4};\n"
        " mov.b64 x, {a, %7};\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %5, f;\n"
        " add.u32 a, %1, 1536;\n"
        " add.u32 b, %3, 4;\n mov.b64 y, {b, %4};\n"
        " mov.b64 x, {a, %7};\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %5, f;\n"
        " add.u32 a, %1, 1792;\n"
        " add.u32 b, %3, 6;\n mov.b64 y, {b, %4};\n"
        " mov.b64 x, {a, %7};\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %5, f;\n"
        " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%8];\n}"
        ::"r"(d), "r"(a), "r"(b0), "r"(b1), "r"(b_hi), "r"(idesc), "r"(acc), "r"(a_hi), "r"(bar0)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// K-major operands.  No swizzle (the outlier tile): core matrices of 8 rows x 16 bytes, `lbo` bytes from one 16-byte
// column of K to the next, 128 bytes from one group of eight rows to the next.
__device__ __forceinline__ uint64_t desc_plain(uint32_t saddr, uint32_t lbo) {
    return (uint64_t)((saddr & 0x3ffffu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(128 >> 4) << 32) | (1ull << 46);
}
// 128-byte swizzle (the activations): rows of 64 K values, 1024 bytes from one group of eight rows to the next.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3ffffu) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t x, uint32_t y, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t add_bf16x2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("add.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// Bounded wait of a whole warp: every lane polls (the instructions after it want the warp converged), and the lanes give
// up together.
__device__ __forceinline__ bool wait_converged(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t* status) {
    const bool ok = mbar_wait(bar, parity, abort_flag, status);
    return __all_sync(0xffffffffu, ok);
}

// Groups of unpack and scatter warps of the variant for NR batch rows (see TcShape).
__host__ __device__ constexpr int tc_unpack_groups(int nr) { return nr == 16 ? 3 : 2; }
__host__ __device__ constexpr int tc_scatter_groups(int nr) { return nr <= 32 ? 3 : (nr <= 64 ? 2 : 1); }

// Shared memory of a launch of the variant for nr rows: its outlier tiles, and as many stages as fit beside them.  A stage holds X
// (nmma rows of 128 BF16 values), the codes, and the scales and zero-points of gps groups.
constexpr int kWoTile = 128 * 128 * 2;      // bytes of a unit's outlier tile
__host__ __device__ constexpr uint32_t tc_wo_bytes(int nr) { return (tc_scatter_groups(nr) == 1 ? 2 : tc_scatter_groups(nr)) * kWoTile; }
__host__ __device__ constexpr uint32_t tc_stage_bytes(uint32_t nmma, int gps) { return (256 * nmma + 8192 + 2 * gps * 256 + 1023) / 1024 * 1024; }
__host__ __device__ constexpr uint32_t tc_stages(int nr, uint32_t nmma, int gps) {
    const uint32_t fixed = 1024 /* alignment */ + 1024 /* barriers */ + tc_wo_bytes(nr), ug = tc_unpack_groups(nr);
    uint32_t s = (kSmemBudget - fixed) / tc_stage_bytes(nmma, gps);
    if (s > 12) s = 12;
    return s >= 2 * ug ? s - s % ug : s;                   // a stage then always returns to the same unpack group
}

struct TcParams {
    const uint8_t* wq;
    const uint16_t* scale;
    const uint16_t* zero;
    const uint32_t* indptr;
    const uint32_t* info;
    const uint4* packed;
    uint16_t* Y;
    uint32_t* status;
    uint32_t* counters;
    float* partials;
    uint32_t M, K, N, KT, NT;       // NT: column tiles of 128 columns
    uint32_t halves;                // such tiles to a stored tile (1 or 2)
    uint32_t max_tile_packets, stages;
    Shares shares;                  // as in the streaming kernel
    uint32_t nmma;                  // batch rows of the MMAs: M rounded up to 16
    uint32_t parts;                 // BF16 parts of an outlier: 1, or 2 (FP16 values)
    // shared-memory offsets (bytes); the first two are relative to a stage, whose X block is at 0
    uint32_t off_w, off_sz, stage_bytes, off_wo, off_bar;
};

constexpr int kScatterAhead = 8;            // slots of a column requested a unit ahead, and taken out one by one

// A variant's tensor-memory columns: NAB A operands of 64 columns, NDB sets of dense accumulators, one per group, and
// the outlier accumulators.  Its warps: four of copies and MMAs; UG groups of four unpack warps and SG groups of four
// scatter warps, which take the units in turn (their work on a unit is a chain of latencies of 800 to 1000 clocks, so that
// the rate comes from the groups side by side); and for each RT batch rows four drain warps.  A scatter group has TPG tiles.
template <int NR, int GROUP>
struct TcShape {
    static constexpr int GPS = kBK / GROUP, RT = NR < 32 ? NR : 32, SETS = NR / RT;
    static constexpr int NDB = 4 * 64 + 4 * GPS * NR + NR <= 512 ? 4 : (2 * 64 + 2 * GPS * NR + NR <= 512 ? 2 : 1);
    static constexpr int NAB = 4 * 64 + NDB * GPS * NR + NR <= 512 ? 4 : 2;
    static constexpr int D_BASE = NAB * 64, O_BASE = D_BASE + NDB * GPS * NR;
    static_assert(O_BASE + NR <= 512, "tensor memory");
    static constexpr int UG = tc_unpack_groups(NR), SG = tc_scatter_groups(NR), TPG = SG == 1 ? 2 : 1, NWO = SG * TPG;
    static constexpr int WARPS = 4 + 4 * UG + 4 * SETS + 4 * SG;
    static_assert(WARPS <= 32 && NWO <= 4, "warps, barriers");
    // Stages of the shortest ring that a launch of this variant gets (its MMAs have more than NR / 2 and at most NR rows).
    static constexpr uint32_t min_stages() {
        uint32_t least = tc_stages(NR, NR, GPS);
        for (uint32_t n = NR / 2 + 16; n < NR; n += 16)
            if (tc_stages(NR, n, GPS) < least) least = tc_stages(NR, n, GPS);
        return least;
    }
    // With this many stages an unpack group waits for a unit's stage before its A operand, so that the codes are on the way
    // while it waits for the operand; with fewer the other way round, which takes NAB (see the unpack warps).
    static constexpr uint32_t kStageFirst = UG + NAB;
    static_assert(min_stages() >= NAB && (NR == 128 || min_stages() >= kStageFirst), "stages");
};

// 16 bits to shared-memory address `addr`, unless that is 0 (predicated: no branch).
__device__ __forceinline__ void put_u16(uint32_t addr, uint32_t v) {
    asm volatile("{\n .reg .pred p;\n .reg .b16 h;\n setp.ne.u32 p, %0, 0;\n cvt.u16.u32 h, %1;\n @p st.shared.u16 [%0], h;\n}" ::"r"(addr), "r"(v) : "memory");
}
// Byte offset inside a column's row of the place of a slot's k (slot bits 5-11).
__device__ __forceinline__ uint32_t slot_place(uint32_t v) { return ((v & 0xf00u) << 3) | ((v >> 4) & 0xeu); }
// What a part of an outlier is: its BF16 bits, or (second part) the fraction bits that BF16 cuts off.
__device__ __forceinline__ uint32_t slot_bits(uint32_t v, uint32_t part) {
    if (part == 0) return v >> 16;
    return (v & 0x7f800000u) == 0x7f800000u ? 0u : float_to_bf16_bits(__uint_as_float(v & kSlotValueMask) - __uint_as_float(v & 0xffff0000u));
}

// The scatter warps' loop (see the kernel): group sg's units of [u_begin, u_end).
template <int NR, int GROUP, int PARTS>
__device__ __forceinline__ void tc_scatter(const TcParams& p, uint8_t* smem, uint32_t sg, uint32_t u_begin, uint32_t u_end, uint32_t bar_wo_full,
                                           uint32_t bar_wo_empty, volatile uint32_t* abort_flag) {
    using S_ = TcShape<NR, GROUP>;
    constexpr uint32_t SG = S_::SG, NWO = S_::NWO, TPG = S_::TPG;
    const uint32_t lane = threadIdx.x & 31, strip = (threadIdx.x >> 5) & 3, g = lane & 7, t = lane >> 3, KT = p.KT;
    const uint32_t row0 = smem_u32(smem) + p.off_wo + (strip * 32 + lane) * 16;
    auto clear_row = [&](uint32_t row) {
#pragma unroll 4
        for (int i = 0; i < 16; ++i) asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(row + i * 2048), "r"(0u) : "memory");
    };
    for (uint32_t b = sg; b < NWO; b += SG) clear_row(row0 + b * kWoTile);
    // a unit's bucket of this lane: its descriptor and the tile's packet range, then its checked form and first slots
    struct Raw { uint32_t info, a, b; };
    struct Bucket { const uint32_t* packets; uint32_t depth, tail, wd[kScatterAhead]; };
    uint32_t u = u_begin + sg, tn = p.shares.by_kt(u), kt = u - tn * KT;              // the next unit to request
    auto request = [&]() {
        Raw r = {0, 0, 0};
        if (p.info && u < u_end) {                         // (no descriptors: the dense half of the unfused pair)
            const uint32_t two = p.halves == 2, c = (tn >> two) * KT + kt;
            r.info = __ldg(p.info + (((size_t)c << two) + (tn & two)) * 32 + strip * 8 + g);
            r.a = __ldg(p.indptr + c), r.b = __ldg(p.indptr + c + 1);
        }
        u += SG;
        for (kt += SG; kt >= KT; kt -= KT) ++tn;
        return r;
    };
    auto fetch = [&](const Raw r) {
        Bucket k;
        const uint32_t off = r.info & 0xffffu;
        k.depth = (r.info >> 16) & 0xffu, k.tail = r.info >> 24;
        k.packets = reinterpret_cast<const uint32_t*>(p.packed + r.a + off) + t;
        if (off + k.depth + k.tail > min(r.b - r.a, p.max_tile_packets)) {
            // a descriptor that reaches past its tile, or past what the layout struct says a tile holds (struct and
            // arrays out of step): report it and skip the bucket
            asm volatile("griddepcontrol.wait;" ::: "memory");             // before the scratch is written
            atomicExch(p.status, (uint32_t)FQ_ERR_FORMAT);
            k.depth = 0, k.tail = 0;
        }
#pragma unroll
        for (uint32_t d = 0; d < kScatterAhead; ++d) k.wd[d] = d < k.depth ? __ldg(k.packets + d * 4) : 0u;
        return k;
    };
    // filled addresses of the group's tile in turn (0: none), how many of them to look at, and of its other tile
    uint32_t filled[TPG][kScatterAhead] = {}, deep[TPG] = {};              // deep: 0 = up to four, 1 = all, 2 = clear the row
    Bucket cur = fetch(request());
    Raw nxt = request();
    uint32_t wb = sg, use = 0;                                             // tile, how often it was handed over
    for (uint32_t it = sg; it < u_end - u_begin; it += SG) {
        const Bucket ahead = fetch(nxt);
        nxt = request();
        const uint32_t row = row0 + wb * kWoTile;
        const bool hot = __any_sync(0xffffffffu, cur.tail != 0 || cur.depth > kScatterAhead), more = __any_sync(0xffffffffu, cur.depth > 4);
#pragma unroll
        for (int part = 0; part < PARTS; ++part) {
            // ---- take out what the tile held; the MMAs that read it are complete
            const uint32_t n = use * PARTS + part;
            if (n > 0 && !wait_converged(bar_wo_empty + 8 * wb, (n - 1) & 1, abort_flag, p.status)) return;
            if (deep[0] < 2) {
#pragma unroll
                for (int d = 0; d < 4; ++d) put_u16(filled[0][d], 0);
                if (deep[0] == 1) {
#pragma unroll
                    for (int d = 4; d < kScatterAhead; ++d) put_u16(filled[0][d], 0);
                }
            } else {
                clear_row(row);
            }
            __syncwarp();
            // ---- put this unit's in (a padding slot has value 0)
            auto put = [&](uint32_t v) {
                const uint32_t at = (v & kSlotValueMask) ? row + slot_place(v) : 0u;
                put_u16(at, slot_bits(v, part));
                return at;
            };
#pragma unroll
            for (int d = 0; d < 4; ++d) filled[0][d] = put(cur.wd[d]);
            if (more) {
#pragma unroll
                for (int d = 4; d < kScatterAhead; ++d) filled[0][d] = put(cur.wd[d]);
            }
            deep[0] = more ? 1u : 0u;
            if (hot) {
                deep[0] = 2;
                for (uint32_t d = kScatterAhead; d < cur.depth; ++d) put(__ldg(cur.packets + d * 4));
                for (uint32_t left = __ballot_sync(0xffffffffu, cur.tail != 0); left;) {     // buckets with a tail: warp-uniform
                    const uint32_t b = (__ffs(left) - 1) & 7u;             // its four lanes b, b + 8, b + 16, b + 24 agree; t = 0 in lane b
                    left &= ~(0x01010101u << b);
                    const uint32_t* tp = reinterpret_cast<const uint32_t*>(
                        __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(cur.packets + cur.depth * 4), b));
                    const uint32_t words = 4 * __shfl_sync(0xffffffffu, cur.tail, b);
                    const uint32_t base = row + ((int)b - (int)lane) * 16;
                    for (uint32_t i = lane; i < words; i += 32) {
                        const uint32_t v = __ldg(tp + i);                  // a tail slot names its column
                        put_u16((v & kSlotValueMask) ? base + ((v >> kSlotColShift) & 3u) * 128 + slot_place(v) : 0u, slot_bits(v, part));
                    }
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_wo_full + 8 * wb);
        }
        if (TPG == 2) {
            wb ^= 1;                                                       // SG == 1: tiles 0 and 1 in turn
            use += wb == 0;
#pragma unroll
            for (int d = 0; d < kScatterAhead; ++d) {
                const uint32_t x = filled[0][d];
                filled[0][d] = filled[TPG - 1][d], filled[TPG - 1][d] = x;
            }
            const uint32_t x = deep[0];
            deep[0] = deep[TPG - 1], deep[TPG - 1] = x;
        } else {
            ++use;
        }
        cur = ahead;
    }
}

// COOP: who finishes a split tile that is the last of a CTA's range and to which the CTA was the last to add.  The drain warps that
// hold it, one to a scheduler, take 0.6 us for each contributor and 1 us to write 32 rows of Y, a chain of latencies; all warps of
// the CTA together, when their own work is done, about 1 us for everything.  us, by the drain warps / by the CTA: 8192 x 1024 at 24
// rows 14.7 / 9.0, 14336 x 4096 at 32 22.3 / 20.3, 4096 x 4096 at 32 11.0 / 10.0; with more rows see tc_coop.
template <int NR, int GROUP, bool COOP>
__global__ void __launch_bounds__(32 * TcShape<NR, GROUP>::WARPS, 1)
fq_tc_kernel(const __grid_constant__ CUtensorMap xmap, const TcParams p) {
    using S_ = TcShape<NR, GROUP>;
    constexpr int GPS = S_::GPS, NAB = S_::NAB, NDB = S_::NDB, SETS = S_::SETS, NWO = S_::NWO, UG = S_::UG;
    constexpr uint32_t W_BYTES = 8192, SZ_ROW = 256;
    static_assert(COOP || NR >= 64, "see tc_coop");
    constexpr bool DEFER = COOP && (NR == 32 || (NR == 16 && GROUP == 64));
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const uint32_t S = p.stages;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + p.off_bar);
    const uint32_t bar_full = smem_u32(bars), bar_empty = bar_full + 8 * S;      // [S] a unit's codes, scales, zero-points are here; the stage is free
    const uint32_t bar_a_full = bar_empty + 8 * S;        // [4] A operand written (unpack warps)
    const uint32_t bar_a_empty = bar_a_full + 32;         // [4] the MMAs that read it are complete
    const uint32_t bar_d_full = bar_a_empty + 32;         // [4] a unit's dense MMAs are complete
    const uint32_t bar_d_free = bar_d_full + 32;          // [4] its sums are read (drain warps)
    const uint32_t bar_wo_full = bar_d_free + 32;         // [4] outlier tile written (scatter warps)
    const uint32_t bar_wo_empty = bar_wo_full + 32;       // [4] the MMAs that read it are complete
    const uint32_t bar_o_full = bar_wo_empty + 32;        // the piece's outlier sums are complete
    const uint32_t bar_o_free = bar_o_full + 8;           // and read
    const uint32_t bar_final = bar_o_free + 8;
    // The activations' arrival, [S], has barriers of its own up to 32 rows, so that the first units are unpacked while the wait for the grid
    // before is still on (us, with / without: 4096 x 4096 at 32 rows 9.7 / 10.0, 8192 x 1024 at 24 8.7 / 9.0; with 64 rows no gain, with groups of 64
    // spills: 8192 x 28672 73.5 / 68.9).
    constexpr bool XB = NR <= 32;
    const uint32_t bar_x_full = XB ? bar_final + 32 : bar_full;
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(bars + 2 * S + 27);
    volatile uint32_t* tmem_slot = abort_flag + 1;
    // COOP: strips and sets (bit strip + 4 set) that the CTA finishes on its way out, of its range's last tile and (DEFER) of its first, of
    // which it seldom is the last contributor.  With 32 rows the sums in the drain warps' loop cost it registers (4096 x 28672 32.3 us, so 31.1;
    // 8192 x 28672 55.9 and 53.8), with 16 and groups of 64 too, 20 bytes of spills (28672 x 8192 52.6, so 50.9; 4096 x 28672 29.5 and 28.9;
    // but 8192 x 1024 at nine 7.6 and 7.8); with 16 and groups of 128 the sums of the first tile are better done at once (4096 x 28672
    // 28.3 and 29.0).
    uint32_t* settle = const_cast<uint32_t*>(abort_flag) + 2;

    if (tid == 0) {
        for (uint32_t s = 0; s < S; ++s) {
            mbar_init(bar_full + 8 * s, XB ? 1 : 2);                         // the producers' expect_tx arrivals
            if (XB) mbar_init(bar_x_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 4 + 4 * SETS + 2);                  // unpack and drain warps, the MMAs' commits
        }
        for (uint32_t i = 0; i < 4; ++i) {
            mbar_init(bar_a_full + 8 * i, 4);
            mbar_init(bar_a_empty + 8 * i, 1);
            mbar_init(bar_wo_full + 8 * i, 4);
            mbar_init(bar_wo_empty + 8 * i, 1);
            mbar_init(bar_d_full + 8 * i, 1);
            mbar_init(bar_d_free + 8 * i, 4 * SETS);
        }
        mbar_init(bar_o_full, 1);
        mbar_init(bar_o_free, 4 * SETS);
        mbar_init(bar_final, 2);
        *abort_flag = 0;
        if (COOP) settle[0] = settle[1] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        tmem_alloc(smem_u32((const void*)tmem_slot), kTmemCols);
        tmem_relinquish();
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // Where the allocation starts; the shuffle tells the compiler that every lane has the same.  Each role reads it for itself: kept
    // from here on it costs the drain warps of the larger variants a register that they do not have (4096 x 28672 at
    // 128 rows 55.0 us, so 53.9; groups of 64 63.7 and 61.0).  With 32 rows it is the other way round (8192 x 28672 with groups of 64
    // 61.4 us kept, 66.7 read again; groups of 128 54.4 and 55.1).
    auto tmem_base_read = [&]() { return __shfl_sync(0xffffffffu, *tmem_slot, 0); };
    const uint32_t tmem_base_kept = NR == 32 ? tmem_base_read() : 0u;
    auto tmem_base_of = [&]() { return NR == 32 ? tmem_base_kept : tmem_base_read(); };
    // The grid after this one in the stream may start now (it takes SMs as this grid's CTAs leave).  The weight arrays
    // are read at once (no kernel writes them while calls are in flight); whoever reads X or writes Y or the scratch
    // waits for the grids before this one.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const uint32_t KT = p.KT;
    uint32_t u_begin, u_end;
    p.shares.range(blockIdx.x, KT, u_begin, u_end);
    // stored tile of a unit (Tile-COO and codes) and the unit's half of it
    auto chunk_of = [&](uint32_t tn, uint32_t kt) { return (p.halves == 2 ? tn >> 1 : tn) * KT + kt; };

    if (warp < 4) {
        if (warp == 0) {
            // ---------------------------------------------------------------- producer of the dense arrays
            uint32_t issued = 0;
            bool ok = true;
            for (UnitIter w(u_begin, KT, p.shares.by_kt); w.u < u_end; w.next(S, KT)) {
                const uint32_t full = bar_full + 8 * w.s;
                if (!wait_converged(bar_empty + 8 * w.s, w.ph ^ 1, abort_flag, p.status)) { ok = false; break; }
                const uint32_t st = smem_u32(smem) + w.s * p.stage_bytes;
                if (elect_one()) {
                    mbar_arrive_expect_tx(full, W_BYTES + 2 * GPS * SZ_ROW);
                    if (p.halves == 2) {
                        const uint8_t* src = p.wq + (size_t)chunk_of(w.tn, w.kt) * 16384 + (w.tn & 1) * 2048;
#pragma unroll
                        for (int j = 0; j < 4; ++j) bulk_g2s(st + p.off_w + j * 2048, src + j * 4096, 2048, full);
                    } else {
                        bulk_g2s(st + p.off_w, p.wq + (size_t)w.u * W_BYTES, W_BYTES, full);
                    }
#pragma unroll
                    for (int gi = 0; gi < GPS; ++gi) {
                        const size_t row = (size_t)(w.kt * GPS + gi) * p.N + (size_t)w.tn * 128;
                        bulk_g2s(st + p.off_sz + gi * SZ_ROW, p.scale + row, SZ_ROW, full);
                        bulk_g2s(st + p.off_sz + (GPS + gi) * SZ_ROW, p.zero + row, SZ_ROW, full);
                    }
                }
                __syncwarp();
                issued = w.it + 1;
            }
            if (!ok) let_copies_land(bar_full, issued, S);
        } else if (warp == 2) {
            // ---------------------------------------------------------------- producer of X
            uint32_t issued = 0;
            bool ok = true;
            const uint32_t x_half = p.nmma * 128;                          // bytes of 64 K values of every batch row
            asm volatile("prefetch.tensormap [%0];" ::"l"(&xmap) : "memory");
            asm volatile("griddepcontrol.wait;" ::: "memory");
            for (UnitIter w(u_begin, KT, p.shares.by_kt); w.u < u_end; w.next(S, KT)) {
                const uint32_t full = bar_x_full + 8 * w.s;
                if (!wait_converged(bar_empty + 8 * w.s, w.ph ^ 1, abort_flag, p.status)) { ok = false; break; }
                const uint32_t st = smem_u32(smem) + w.s * p.stage_bytes;
                if (elect_one()) {
                    mbar_arrive_expect_tx(full, 2 * x_half);
                    tma_load_2d(st, &xmap, w.kt * kBK, 0, full);
                    tma_load_2d(st + x_half, &xmap, w.kt * kBK + 64, 0, full);
                }
                __syncwarp();
                issued = w.it + 1;
            }
            if (!ok) let_copies_land(bar_x_full, issued, S);
        } else if (warp == 1) {
            // ---------------------------------------------------------------- dense tensor warp
            // (without XB the unpack warps have waited for the whole stage, X block included, and their arrival hands that on: it is a release)
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((p.nmma >> 3) << 17) | (8u << 24), tmem_base = tmem_base_of();
            const uint32_t x_half = (p.nmma * 128) >> 4, stage = p.stage_bytes >> 4;
            const uint64_t xd0 = desc_sw128(smem_u32(smem));
            const uint32_t units = u_end - u_begin;
            uint32_t s = 0, ph = 0, xd = (uint32_t)xd0;
            bool ready = false;
            for (uint32_t it = 0; it < units; ++it) {
                const uint32_t ab = it % NAB, db = it % NDB, nx = it + 1;
                if (!ready) {
                    if (it >= NDB && !wait_converged(bar_d_free + 8 * db, (it / NDB - 1) & 1, abort_flag, p.status)) break;
                    if (XB && !wait_converged(bar_x_full + 8 * s, ph, abort_flag, p.status)) break;
                    if (!wait_converged(bar_a_full + 8 * ab, (it / NAB) & 1, abort_flag, p.status)) break;
                }
                tc_fence_after();
                // the next unit's barriers, tested while this one's MMAs are issued
                uint32_t seen = mbar_test_wait(bar_a_full + 8 * (nx % NAB), (nx / NAB) & 1) &
                                      (nx < NDB ? 1u : mbar_test_wait(bar_d_free + 8 * (nx % NDB), (nx / NDB - 1) & 1));
                const uint32_t d = tmem_base + S_::D_BASE + db * (GPS * NR);
                umma_dense(d, d + (GPS - 1) * NR, GPS == 1, tmem_base + ab * 64, xd, xd + x_half, (uint32_t)(xd0 >> 32), idesc, bar_d_full + 8 * db,
                           bar_a_empty + 8 * ab, bar_empty + 8 * s);
                xd += stage;
                if (++s == S) s = 0, xd = (uint32_t)xd0, ph ^= XB;
                if (XB) seen &= mbar_test_wait(bar_x_full + 8 * s, ph);
                ready = __all_sync(0xffffffffu, seen);
            }
            if (elect_one()) umma_commit(bar_final);     // fires when every MMA this warp issued has retired
            __syncwarp();
        } else {
            // ---------------------------------------------------------------- outlier tensor warp
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((p.nmma >> 3) << 17) | (8u << 24), tmem_base = tmem_base_of();
            const uint64_t wo0 = desc_plain(smem_u32(smem) + p.off_wo, 2048), xd0 = desc_sw128(smem_u32(smem));
            const uint32_t x_half = (p.nmma * 128) >> 4, stage = p.stage_bytes >> 4, o = tmem_base + S_::O_BASE;
            const uint32_t units = u_end - u_begin, parts = p.parts;
            uint32_t s = 0, ph = 0, wb = 0, wph = 0, xd = (uint32_t)xd0, acc = 0, left = KT - (u_begin - p.shares.by_kt(u_begin) * KT), piece = 0;    // left: units to the end of the tile
            bool ok = true, ready = false;
            for (uint32_t it = 0; it < units && ok; ++it) {
                if (!ready && !(wait_converged(bar_x_full + 8 * s, ph, abort_flag, p.status) &&
                                wait_converged(bar_wo_full + 8 * wb, wph, abort_flag, p.status))) break;
                tc_fence_after();
                umma_outliers(o, (uint32_t)wo0 + wb * (kWoTile >> 4), (uint32_t)(wo0 >> 32), xd, xd + x_half, (uint32_t)(xd0 >> 32), idesc, acc,
                              bar_wo_empty + 8 * wb);
                if (parts == 2) {                          // the second part of FP16 values, in the same tile
                    if (!wait_converged(bar_wo_full + 8 * wb, 1, abort_flag, p.status)) break;
                    tc_fence_after();
                    umma_outliers(o, (uint32_t)wo0 + wb * (kWoTile >> 4), (uint32_t)(wo0 >> 32), xd, xd + x_half, (uint32_t)(xd0 >> 32), idesc, 1,
                                  bar_wo_empty + 8 * wb);
                }
                if (elect_one()) umma_commit(bar_empty + 8 * s);
                __syncwarp();
                acc = 1;
                xd += stage;
                if (++s == S) s = 0, xd = (uint32_t)xd0, ph ^= 1;
                if (++wb == NWO) wb = 0, wph ^= parts & 1;
                // the next unit's barriers, tested while this one's MMAs run
                const uint32_t seen = mbar_test_wait(bar_x_full + 8 * s, ph) & mbar_test_wait(bar_wo_full + 8 * wb, wph);
                if (--left == 0 || it + 1 == units) {
                    // end of a piece: the drain warps take the sums before the next piece's overwrite them
                    if (elect_one()) umma_commit(bar_o_full);
                    __syncwarp();
                    if (it + 1 < units && !wait_converged(bar_o_free, piece & 1, abort_flag, p.status)) ok = false;
                    ++piece;
                    left = KT, acc = 0;
                }
                ready = __all_sync(0xffffffffu, seen);
            }
            if (elect_one()) umma_commit(bar_final);
            __syncwarp();
        }
    } else if (warp < 4 + 4 * UG) {
        // -------------------------------------------------------------------- unpack warps: thread = column
        const uint32_t ug = (warp - 4) >> 2;                               // takes the units it with it % UG == ug
        const uint32_t t_a = tmem_base_of() + ((uint32_t)((warp & 3) * 32) << 16);
        const uint32_t col = (warp & 3) * 32 + lane;
        const bool stage_first = NR < 128 || S >= S_::kStageFirst;
        for (UnitIter w(u_begin, KT, p.shares.by_kt); w.u < u_end; w.next(S, KT)) {
            if (w.it % UG != ug) continue;
            const uint32_t ab = w.it % NAB;
            const uint8_t* st = smem + w.s * p.stage_bytes;
            // A parity wait is only valid for a waiter that knows the phase before to be complete, and a group does not meet
            // the phases of the other groups' units.  What it knows: once the A operand of unit i is read, the stages of
            // all units up to i have been filled, since their MMAs were issued in order behind their unpacking.  So the stage's
            // phase before, that of unit it - S, is complete if the group has waited for the operand of unit it - NAB
            // (S >= NAB), or, with the stage's wait in front, of unit it - UG - NAB (S >= UG + NAB, see kStageFirst).  And the phase
            // cannot be over before the group has met it: the stage is not filled again until the group has released it.
            if (!stage_first && w.it >= NAB && !wait_converged(bar_a_empty + 8 * ab, (w.it / NAB - 1) & 1, abort_flag, p.status)) break;
            if (!wait_converged(bar_full + 8 * w.s, w.ph, abort_flag, p.status)) break;
            // (with 16 rows the A operand's barrier is tested while the codes load: 3 % faster there, 2 % slower at 32)
            uint32_t seen = 0;
            if constexpr (NR == 16) seen = w.it < NAB ? 1u : mbar_test_wait(bar_a_empty + 8 * ab, (w.it / NAB - 1) & 1);
            const uint4* wp = reinterpret_cast<const uint4*>(st + p.off_w) + col;
            uint4 w4[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) w4[j] = wp[j * 128];
            uint32_t nz[GPS];                                              // -(128 + z) twice
#pragma unroll
            for (int gi = 0; gi < GPS; ++gi) {
                const uint32_t z = reinterpret_cast<const uint16_t*>(st + p.off_sz + (GPS + gi) * SZ_ROW)[col];
                nz[gi] = 0x80008000u ^ add_bf16x2(z | (z << 16), 0x43004300u);
            }
            if (!stage_first || (NR == 16 && __all_sync(0xffffffffu, seen))) {}
            else if (w.it >= NAB && !wait_converged(bar_a_empty + 8 * ab, (w.it / NAB - 1) & 1, abort_flag, p.status)) break;
            tc_fence_after();
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t ww[4] = {w4[j].x, w4[j].y, w4[j].z, w4[j].w};
                uint32_t a[16];
#pragma unroll
                for (int x = 0; x < 4; ++x)
#pragma unroll
                    for (int i = 0; i < 4; ++i) a[4 * x + i] = add_bf16x2(codes_to_bf16x2(ww[x] >> (4 * i)), nz[j * GPS / 4]);
                tmem_st16(t_a + ab * 64 + j * 16, a);
            }
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(bar_a_full + 8 * ab);
                mbar_arrive(bar_empty + 8 * w.s);
            }
        }
    } else if (warp < 4 + 4 * UG + 4 * SETS) {
        // -------------------------------------------------------------------- drain warps: thread = column, RT batch rows
        const int set = (warp - 4 - 4 * UG) >> 2, dw = warp & 3;           // rows, strip of the unit
        const int col = dw * 32 + lane;
        constexpr int RT = S_::RT, CH = 16;                                // rows of a thread, rows per tensor-memory load
        const uint32_t r0 = set * RT;
        const uint32_t t_lane = tmem_base_of() + ((uint32_t)((warp & 3) * 32) << 16);
        float acc[RT];
#pragma unroll
        for (int i = 0; i < RT; ++i) acc[i] = 0.0f;
        bool ok = true;
        UnitIter w(u_begin, KT, p.shares.by_kt);
        uint32_t tn = p.shares.by_kt(u_begin), piece = 0;
        asm volatile("griddepcontrol.wait;" ::: "memory");
        // outer loop: the pieces of this CTA's range (a piece = its units of one column tile)
        for (uint32_t piece_first = u_begin; piece_first < u_end && ok; ++tn, ++piece) {
            const uint32_t piece_stop = min(u_end, (tn + 1) * KT);        // one past the piece's last unit
            piece_first = piece_stop;
            for (; w.u < piece_stop; w.next(S, KT)) {
                const uint32_t db = w.it % NDB;
                const uint8_t* st = smem + w.s * p.stage_bytes;
                if (!wait_converged(bar_full + 8 * w.s, w.ph, abort_flag, p.status)) { ok = false; break; }
                float sv[GPS];
#pragma unroll
                for (int gi = 0; gi < GPS; ++gi) sv[gi] = bf16_bits_to_float(reinterpret_cast<const uint16_t*>(st + p.off_sz + gi * SZ_ROW)[col]);
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_empty + 8 * w.s);       // the scales were all it needs of the stage
                if (!wait_converged(bar_d_full + 8 * db, (w.it / NDB) & 1, abort_flag, p.status)) { ok = false; break; }
                tc_fence_after();
#pragma unroll
                for (int gi = 0; gi < GPS; ++gi)
#pragma unroll
                    for (int c0 = 0; c0 < RT; c0 += CH)
                        if (r0 + c0 < p.nmma) {
                            float d[CH];
                            tmem_ld<CH>(t_lane + S_::D_BASE + (db * GPS + gi) * NR + r0 + c0, d);
                            tmem_wait_ld();
#pragma unroll
                            for (int i = 0; i < CH; ++i) acc[c0 + i] = fmaf(sv[gi], d[i], acc[c0 + i]);
                        }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_d_free + 8 * db);
            }
            if (!ok) break;
            // ---------------------------------------------------------------- end of a piece
            if (!wait_converged(bar_o_full, piece & 1, abort_flag, p.status)) { ok = false; break; }
            tc_fence_after();
#pragma unroll
            for (int c0 = 0; c0 < RT; c0 += CH)
                if (r0 + c0 < p.nmma) {
                    float d[CH];
                    tmem_ld<CH>(t_lane + S_::O_BASE + r0 + c0, d);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < CH; ++i) acc[c0 + i] += d[i];
                }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_o_free);
            const uint32_t kt = piece_stop - 1 - tn * KT;                 // k-step of the piece's last unit
            const uint32_t u_tile0 = tn * KT;
            const uint32_t piece_k0 = max(u_tile0, u_begin) - u_tile0;
            const bool full_piece = (piece_k0 == 0) && (kt == KT - 1);
            bool write_y = full_piece;
            if (!full_piece) {
                // Split tile.  Every warp settles its own 32 columns and rows, without CTA-wide barriers: FP32 partial, four
                // rows of a column to 16 bytes, then one arrival per (tile, strip, set of rows: a byte of the strip's
                // counter each); the last to arrive adds the partials in CTA order (the same order in every run) and writes Y:
                // this warp, or the whole CTA if the range ends here (COOP), and wherever it is the last (DEFER).
                constexpr uint32_t COLS = 128, SLOT = COLS * NR / 4;      // float4 per slot
                const uint32_t which = p.shares.slot_of(blockIdx.x, tn, KT);
                float4* slots = reinterpret_cast<float4*>(p.partials) + (size_t)(r0 / 4) * COLS + col;
                float4* slot = slots + ((size_t)blockIdx.x * 2 + which) * SLOT;
#pragma unroll
                for (int i = 0; i < RT / 4; ++i)
                    if (r0 + 4 * i < p.M) __stcg(slot + i * COLS, make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]));
                __syncwarp();
                uint32_t c_first, c_last;
                p.shares.owners(tn, KT, c_first, c_last);
                uint32_t* counter = p.counters + tn * 4 + dw;
                uint32_t last = 0;
                if (lane == 0) {
                    // one arrival, release and acquire at GPU scope: the warp's stores (ordered before this lane by
                    // the __syncwarp above) precede it, and the warp that finds itself last sees the stores of all
                    // contributors that arrived before
                    uint32_t old;
                    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(counter), "r"(1u << (8 * set)) : "memory");
                    last = (((old >> (8 * set)) & 0xffu) == c_last - c_first) ? 1u : 0u;
                }
                last = __shfl_sync(0xffffffffu, last, 0);
                __syncwarp();
                if (COOP && last && lane == 0) {
                    atomicSub(counter, (c_last - c_first + 1) << (8 * set));                     // ready for the next call
                    if (DEFER || piece_stop == u_end) atomicOr(settle + (piece_stop == u_end ? 0 : 1), 1u << (set * 4 + dw));
                }
                if constexpr (!DEFER) if (last && !(COOP && piece_stop == u_end)) {
                    write_y = true;
                    // 16 rows at a time, ND contributors' loads in flight; the additions keep CTA order
                    constexpr int ND = NR >= 64 ? 2 : 1;
#pragma unroll
                    for (int i0 = 0; i0 < RT / 4; i0 += 4)
                        if (r0 + 4 * i0 < p.M) {
#pragma unroll
                            for (int i = 0; i < 16; ++i) acc[4 * i0 + i] = 0.0f;
                            for (uint32_t c = c_first; c <= c_last; c += ND) {
                                float4 v[ND][4];
#pragma unroll
                                for (int dd = 0; dd < ND; ++dd) {
                                    const uint32_t cc = min(c + dd, c_last);
                                    const uint32_t wch = p.shares.slot_of(cc, tn, KT);
                                    const float4* sl = slots + ((size_t)cc * 2 + wch) * SLOT;
#pragma unroll
                                    for (int i = 0; i < 4; ++i) v[dd][i] = __ldcg(sl + (i0 + i) * COLS);
                                }
#pragma unroll
                                for (int dd = 0; dd < ND; ++dd)
                                    if (c + dd <= c_last) {
#pragma unroll
                                        for (int i = 0; i < 4; ++i) {
                                            acc[4 * (i0 + i) + 0] += v[dd][i].x;
                                            acc[4 * (i0 + i) + 1] += v[dd][i].y;
                                            acc[4 * (i0 + i) + 2] += v[dd][i].z;
                                            acc[4 * (i0 + i) + 3] += v[dd][i].w;
                                        }
                                    }
                            }
                        }
                    if (!COOP && lane == 0) atomicSub(counter, (c_last - c_first + 1) << (8 * set));      // ready for the next call
                }
            }
            if (write_y) {
                uint16_t* y = p.Y + (size_t)r0 * p.N + (size_t)tn * 128 + col;
#pragma unroll
                for (int m = 0; m < RT; ++m)
                    if (r0 + m < p.M) y[(size_t)m * p.N] = float_to_bf16_bits(acc[m]);
            }
#pragma unroll
            for (int i = 0; i < RT; ++i) acc[i] = 0.0f;
        }
    } else {
        // -------------------------------------------------------------------- scatter warps: thread = column
        // Column 32 strip + l of a half is column number t = l / 8 of bucket g = l % 8 of the strip: slot t of every
        // column-slotted packet of the bucket.  The thread owns the column's row of the tile (2 bytes per k, eight k
        // to 16 bytes, those 2048 bytes apart) and keeps the addresses that it has filled, to clear them for the next unit;
        // where they are more than kScatterAhead, or a tail was shared out over the warp, it clears the whole row.
        // The bucket descriptors and slots come from global memory straight into registers, requested two units and one unit
        // ahead.
        const uint32_t sg = (uint32_t)(warp - 4 - 4 * UG - 4 * SETS) >> 2;     // takes the units it with it % SG == sg
        if (p.parts == 1) tc_scatter<NR, GROUP, 1>(p, smem, sg, u_begin, u_end, bar_wo_full, bar_wo_empty, abort_flag);
        else tc_scatter<NR, GROUP, 2>(p, smem, sg, u_begin, u_end, bar_wo_full, bar_wo_empty, abort_flag);
    }

    // ---------------------------------------------------------------------- common exit
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        // every tcgen05 operation of this CTA must have retired before its tensor memory is released
        mbar_wait_leaving(bar_final, 0);
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base_of(), kTmemCols);
    }
    if constexpr (COOP) {
        for (uint32_t side = 0; side < (DEFER ? 2u : 1u); ++side) {
            const uint32_t mine = settle[side];
            if (!mine) continue;
            // The sums of the range's last tile, or (side 1) of its first (the drain warps' acquire is handed on by the barrier above): a
            // thread takes four rows of a column, with ND contributors' loads in flight.
            constexpr uint32_t COLS = 128, SLOT = COLS * NR / 4;
            constexpr int ND = 6;
            uint32_t begin = u_begin, end = u_end, c_first, c_last;
            if (NR >= 32) {                                   // the range anew, so that nothing of it is kept in registers until here
                uint32_t cta;
                asm volatile("mov.u32 %0, %%ctaid.x;" : "=r"(cta));
                p.shares.range(cta, p.KT, begin, end);
            }
            const uint32_t tn = p.shares.by_kt(side ? begin : end - 1);
            p.shares.owners(tn, p.KT, c_first, c_last);
            const float4* slots = reinterpret_cast<const float4*>(p.partials);
            for (uint32_t e = threadIdx.x; e < (p.M + 3) / 4 * COLS; e += blockDim.x) {
                const uint32_t i = e / COLS, col = e % COLS;
                if (!((mine >> (4 * i / S_::RT * 4 + col / 32)) & 1u)) continue;
                float4 sum = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                for (uint32_t c = c_first; c <= c_last; c += ND) {
                    float4 v[ND];
#pragma unroll
                    for (int d = 0; d < ND; ++d) {
                        const uint32_t wch = p.shares.slot_of(c + d, tn, p.KT);
                        if (c + d <= c_last) v[d] = __ldcg(slots + ((size_t)(c + d) * 2 + wch) * SLOT + e);
                    }
#pragma unroll
                    for (int d = 0; d < ND; ++d)
                        if (c + d <= c_last) sum.x += v[d].x, sum.y += v[d].y, sum.z += v[d].z, sum.w += v[d].w;
                }
                uint16_t* y = p.Y + (size_t)(4 * i) * p.N + (size_t)tn * COLS + col;
                const float rows[4] = {sum.x, sum.y, sum.z, sum.w};
#pragma unroll
                for (int m = 0; m < 4; ++m)
                    if (4 * i + m < p.M) y[(size_t)m * p.N] = float_to_bf16_bits(rows[m]);
            }
        }
    }
}
