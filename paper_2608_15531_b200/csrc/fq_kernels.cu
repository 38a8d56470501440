// CUDA side of the library (sm_100a): the fused W4A16 + Tile-COO outlier decode matmul
// (Eq. 1; Sections 3.1, 4.1, 4.2), its two unfused baselines and the launchers behind the C ABI.
//
// Three kernels serve the fused operator, chosen per launch from its rows and the layer's shape (tc_serves, direct_warps): a
// streaming kernel and a short-job kernel with warp-level MMAs for up to 16 rows (fq_mma_kernel.cuh,
// fq_direct_kernel.cuh) and a tcgen05 kernel for up to 128 (fq_tc_kernel.cuh).  The streaming kernels are
// persistent and warp-specialised: (tile, k-step) units of 128 rows stream through a ring of shared-memory stages
// (bulk copies + mbarrier expect_tx).  All feed the tensor cores exact integers and apply the scale once per group in FP32:
//     acc[m] += s * sum_k x (q - z)                                     (Eq. 3 inside Eq. 1)
//
// Units are split over CTAs as contiguous ranges (stream-K) or, for layers with few column tiles, as
// tile-aligned parts.  A tile whose k-range is shared by several CTAs is finished by the last to
// arrive, which adds the FP32 partials in CTA order; no CTA waits for another.  Every wait on a barrier
// is bounded: on expiry the CTA raises the scratch status word, drains and leaves through the common
// exit that frees its tensor memory.
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <mutex>

#include "fq_internal.h"
#include "fq_shares.h"

namespace cg = cooperative_groups;
namespace fq {

constexpr int kBK = 128;
constexpr int kSmemBudget = 232448;    // 227 KB per CTA on sm_100
constexpr uint32_t kSmemOneCta = 116736;   // of which no two CTAs fit on an SM: 228 KB, and 1 KB of a CTA is the system's
constexpr unsigned long long kWaitLimitNs = 2000000000ull;
constexpr uint32_t kTmemCols = 512;


// ----------------------------------------------------------------------------- PTX helpers

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
// A release, like every arrival here: also that of a consumer, whose reads of a stage come before the copy that fills it next,
// and that of a warp which has waited for a copy and tells the next warp so.
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}" ::"r"(bar), "r"(bytes)
                 : "memory");
}
// more bytes for the barrier's current phase, without arriving
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// A waiting thread sleeps in hardware for a while instead of spinning on the issue slots that the working warps of the
// CTA need.  No suspend-time hint: with one of 20 us the waits of the tcgen05 kernel returned later (8192 x 28672 at
// 32 rows 80.4 us, without it 78.0; spinning on test_wait instead 83.1).
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok;
}
__device__ __forceinline__ uint32_t mbar_test_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok;
}
__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait, slow part.  Inlined: a call in the pipeline loops constrains the register allocation of
// the code around it (measured: 3 % on the dense-only kernel).
__device__ __forceinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t* status) {
    uint32_t spins = 0;
    unsigned long long t0 = 0;
    while (!mbar_try_wait(bar, parity)) {
        if ((++spins & 0xf) == 0) {
            if (*abort_flag) return false;
            unsigned long long now = globaltimer_ns();
            if (t0 == 0) {
                t0 = now;
            } else if (now - t0 > kWaitLimitNs) {
                *abort_flag = 1;
                atomicExch(status, (uint32_t)FQ_ERR_TIMEOUT);
                return false;
            }
        }
    }
    return true;
}
// Bounded wait: false if this CTA is giving up (its own limit expired, or another warp's did).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag,
                                          uint32_t* status) {
    if (mbar_test_wait(bar, parity)) return true;   // already complete
    return mbar_wait_slow(bar, parity, abort_flag, status);
}
// Warp-uniform form: every lane waits, and the warp gives up together.  Every lane polls and the outcome is a vote, which
// the compiler knows to be the same in every lane; with one lane polling and a shuffle the loops around the waits were
// compiled as divergent (streaming kernel 5 to 7 % slower: 4096 x 28672 at one row 23.5 us, so 22.3).
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag, uint32_t* status) {
    const bool ok = mbar_wait(bar, parity, abort_flag, status);
    return __all_sync(0xffffffffu, ok);
}
// A wait of a CTA that is leaving: no status, no abort flag, at most 100 ms (and no fewer than 4096 polls: the clock also runs while
// the context is switched out).
__device__ __forceinline__ void mbar_wait_leaving(uint32_t bar, uint32_t parity) {
    const unsigned long long t0 = globaltimer_ns();
    for (uint32_t polls = 0; !mbar_try_wait(bar, parity); ++polls)
        if (polls >= 4096 && globaltimer_ns() - t0 > 100000000ull) return;
}
// What a producer does that gives up: it lets the copies already issued land before the CTA's shared memory goes away.
__device__ __forceinline__ void let_copies_land(uint32_t bar_full, uint32_t issued, uint32_t S) {
    for (uint32_t j = (issued > S ? issued - S : 0); j < issued; ++j) mbar_wait_leaving(bar_full + 8 * (j % S), (j / S) & 1);
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
// (w & 0x000f000f) | 0x43004300: two codes -> two BF16 values 128 + q
__device__ __forceinline__ uint32_t codes_to_bf16x2(uint32_t w) {
    uint32_t r;
    asm("lop3.b32 %0, %1, 0x000f000f, 0x43004300, 0xea;" : "=r"(r) : "r"(w));
    return r;
}
__device__ __forceinline__ float bf16lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }
__device__ __forceinline__ float bf16_bits_to_float(uint16_t v) { return __uint_as_float((uint32_t)v << 16); }
__device__ __forceinline__ uint16_t float_to_bf16_bits(float f) {
    return __bfloat16_as_ushort(__float2bfloat16_rn(f));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}

// ---- tcgen05 / tensor memory
__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// Walks a CTA's units without integer division: ring slot s with its parity, tile tn, k-step kt.
struct UnitIter {
    uint32_t u, it, s, ph, tn, kt;
    __device__ __forceinline__ UnitIter(uint32_t u_begin, uint32_t KT, const Divisor& by_kt) : u(u_begin), it(0), s(0), ph(0) {
        tn = by_kt(u_begin);
        kt = u_begin - tn * KT;
    }
    __device__ __forceinline__ void next(uint32_t S, uint32_t KT) {
        ++u;
        ++it;
        if (++s == S) { s = 0; ph ^= 1; }
        if (++kt == KT) { kt = 0; ++tn; }
    }
};

// Waits for the grid before this one, in a kernel without an outlier step.  That serves layers whose layout struct knows of no
// outliers; if the arrays hold some all the same (struct and arrays out of step), the warp that is told to `look` reports it.
// The load is on its way during the wait (at the end of the kernel it cost 2432 x 1152 at two rows 0.3 of 3.1 us).  `indptr` is
// null where there is no sparse part at all.
__device__ __forceinline__ void grid_wait_dense(bool look, const uint32_t* indptr, uint32_t tiles, uint32_t* status) {
    uint32_t packets = 0;
    if (look && indptr) packets = __ldg(indptr + tiles);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (packets) atomicExch(status, (uint32_t)FQ_ERR_FORMAT);
}

#include "fq_tc_kernel.cuh"
#include "fq_mma_kernel.cuh"
#include "fq_direct_kernel.cuh"

// ----------------------------------------------------------------------------- unfused SpMM

// Y += X * W_O as its own launch (the sparse half of the two-kernel baseline, Section 2.2).  One CTA per
// (column tile, slab of k-steps); the slabs of a tile form one thread-block cluster.  A warp owns a strip of
// 32 columns (lane = column = slot t of bucket g) and every second (fourth, for tiles of 128 columns) k-step of the slab.  The CTA stages the
// activations of eight k-steps at a time as a k-major BF16 tile in shared memory; while those loads are in
// flight every warp fetches the bucket descriptors and the first four packet slots of its k-steps, so one
// chunk costs three global-memory latencies whatever its length.  A lane multiplies-adds the slots of its
// column into RR FP32 registers (a padding slot has value 0 and reads row 0: a broadcast).  The warps of
// a strip add up in shared memory, the slabs of a tile through distributed shared memory (plain loads from
// the peers' tiles, each CTA taking its share of the elements in slab order: a fixed order, so the result
// is the same from run to run), and each element of Y is read, added to and written once.
constexpr int kSpmmChunk = 8;     // k-steps of activations staged at a time
constexpr int kSpmmThreads = 512; // 16 warps: 8 strips x 2 (tiles of 256 columns) or 4 strips x 4 (tiles of 128)
constexpr int kSpmmPer = 4;       // k-steps per warp and chunk, at most

template <int RR>
__device__ __forceinline__ void spmm_add(float (&acc)[RR], uint32_t w, const uint8_t* xrow) {
    const uint32_t k = (w >> 5) & 127u;
    const float v = __uint_as_float(w & kSlotValueMask);
    if constexpr (RR == 1) {
        acc[0] = fmaf(v, __uint_as_float((uint32_t)reinterpret_cast<const uint16_t*>(xrow)[k] << 16), acc[0]);
    } else {
#pragma unroll
        for (int c = 0; c < RR / 8; ++c) {
            const uint4 q = *reinterpret_cast<const uint4*>(xrow + k * (2 * RR) + 16 * c);
            const uint32_t x[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                acc[8 * c + 2 * i] = fmaf(v, bf16lo(x[i]), acc[8 * c + 2 * i]);
                acc[8 * c + 2 * i + 1] = fmaf(v, bf16hi(x[i]), acc[8 * c + 2 * i + 1]);
            }
        }
    }
}

template <int RR>
__global__ void __launch_bounds__(kSpmmThreads, 2) fq_spmm_kernel(const uint16_t* X, const uint32_t* __restrict__ indptr,
                                                    const uint32_t* __restrict__ info, const uint4* __restrict__ packed,
                                                    uint16_t* Y, uint32_t M, uint32_t K, uint32_t N,
                                                    uint32_t BN, uint32_t slabs) {
    extern __shared__ __align__(16) uint8_t spmm_smem[];
    const uint32_t NB = BN / 4, NS = BN / 32, KW = kSpmmThreads / 32 / NS, KT = K / kBK;
    float* red = reinterpret_cast<float*>(spmm_smem);                 // [RR][BN] sums of this slab
    uint8_t* xs = spmm_smem + (size_t)RR * BN * 4;                    // [kSpmmChunk * 128][RR] BF16, k-major
    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t strip = warp % NS, kw = warp / NS, g = lane & 7, t = lane >> 3;
    const uint32_t tile = blockIdx.x / slabs, slab = blockIdx.x - tile * slabs;
    const uint32_t kt0 = slab * KT / slabs, kt1 = (slab + 1) * KT / slabs;
    float acc[RR];
#pragma unroll
    for (int i = 0; i < RR; ++i) acc[i] = 0.0f;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (kt0 >= kt1) asm volatile("griddepcontrol.wait;" ::: "memory");     // a slab without k-steps still adds to Y below

    for (uint32_t c0 = kt0; c0 < kt1; c0 += kSpmmChunk) {
        const uint32_t nk = min((uint32_t)kSpmmChunk, kt1 - c0);
        uint32_t inf[kSpmmPer], base[kSpmmPer];
#pragma unroll
        for (int j = 0; j < kSpmmPer; ++j) {
            const uint32_t kl = kw + j * KW;
            inf[j] = 0, base[j] = 0;
            if (kl < nk) {
                const size_t u = (size_t)tile * KT + c0 + kl;
                inf[j] = __ldg(info + u * NB + strip * 8 + g);
                base[j] = __ldg(indptr + u);
            }
        }
        uint32_t w[kSpmmPer][4];
        const uint32_t* pk[kSpmmPer];
#pragma unroll
        for (int j = 0; j < kSpmmPer; ++j) {
            pk[j] = reinterpret_cast<const uint32_t*>(packed + base[j] + (inf[j] & 0xffffu));
            const uint32_t depth = (inf[j] >> 16) & 0xffu;
#pragma unroll
            for (int d = 0; d < 4; ++d) w[j][d] = (uint32_t)d < depth ? __ldg(pk[j] + d * 4 + t) : 0u;
        }
        // descriptors and packets are weights; X and Y may come from the grid before this one in the stream, so that they
        // are not read through the read-only path
        if (c0 == kt0) asm volatile("griddepcontrol.wait;" ::: "memory");
        // the chunk's activations: a thread takes eight consecutive k of one batch row at a time
        constexpr int XU = RR == 1 ? 1 : RR * 16 * kSpmmChunk / kSpmmThreads;
        uint4 xr[XU];
#pragma unroll
        for (int j = 0; j < XU; ++j) {
            const uint32_t e = tid + j * kSpmmThreads, m = e % RR, o = e / RR;
            xr[j] = make_uint4(0, 0, 0, 0);
            if (o < 16 * nk && m < M) xr[j] = __ldcg(reinterpret_cast<const uint4*>(X + (size_t)m * K + (size_t)c0 * kBK) + o);
        }
#pragma unroll
        for (int j = 0; j < XU; ++j) {
            const uint32_t e = tid + j * kSpmmThreads, m = e % RR, o = e / RR;
            if (o < 16 * kSpmmChunk) {
                if constexpr (RR == 1) {
                    *reinterpret_cast<uint4*>(xs + 16 * o) = xr[j];
                } else {
                    // value i of the eight goes to row 8 o + i; the lanes of a warp that hold other octets
                    // start at other i, so that one store instruction never hits a bank twice
                    const uint32_t v[4] = {xr[j].x, xr[j].y, xr[j].z, xr[j].w};
                    const uint32_t rot = (lane / RR) & 7u;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const uint32_t ii = (i + rot) & 7u;
                        const uint32_t word = ii & 4 ? (ii & 2 ? v[3] : v[2]) : (ii & 2 ? v[1] : v[0]);
                        *reinterpret_cast<uint16_t*>(xs + (size_t)(8 * o + ii) * (2 * RR) + 2 * m) =
                            (uint16_t)(ii & 1 ? word >> 16 : word);
                    }
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kSpmmPer; ++j) {
            const uint8_t* xrow = xs + (size_t)(kw + j * KW) * kBK * (2 * RR);
            const uint32_t depth = (inf[j] >> 16) & 0xffu, tail = inf[j] >> 24;
            const uint32_t dmax = __reduce_max_sync(0xffffffffu, depth);
#pragma unroll
            for (int d = 0; d < 4; ++d)
                if ((uint32_t)d < dmax) spmm_add<RR>(acc, w[j][d], xrow);
            for (uint32_t d = 4; d < depth; ++d) spmm_add<RR>(acc, __ldg(pk[j] + d * 4 + t), xrow);
            for (uint32_t d = depth; d < depth + tail; ++d) {             // tail: a slot names its column
                const uint4 q4 = __ldg(reinterpret_cast<const uint4*>(pk[j]) + d);
                const uint32_t wd[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (((wd[e] >> kSlotColShift) & 3u) == t) spmm_add<RR>(acc, wd[e], xrow);
            }
        }
        __syncthreads();                                                  // the tile is overwritten by the next chunk
    }

    // the warps of a strip, then the slabs of the tile
    const uint32_t col = strip * 32 + lane;
    for (uint32_t r = 0; r < KW; ++r) {
        if (kw == r) {
#pragma unroll
            for (int m = 0; m < RR; ++m) red[m * BN + col] = r ? red[m * BN + col] + acc[m] : acc[m];
        }
        __syncthreads();
    }
    cg::cluster_group cluster = cg::this_cluster();
    if (slabs > 1) cluster.sync(); else __syncthreads();
    const uint32_t E = M * BN, e0 = slab * E / slabs, e1 = (slab + 1) * E / slabs;
    for (uint32_t e = e0 + tid; e < e1; e += kSpmmThreads) {
        float sum = 0.0f;
        for (uint32_t s2 = 0; s2 < slabs; ++s2) sum += slabs > 1 ? cluster.map_shared_rank(red, s2)[e] : red[e];
        uint16_t* y = Y + (size_t)(e / BN) * N + (size_t)tile * BN + (e % BN);
        *y = float_to_bf16_bits(bf16_bits_to_float(*y) + sum);
    }
    if (slabs > 1) cluster.sync();                                        // peers may still be reading this tile
}

// ----------------------------------------------------------------------------- launch plumbing

static inline uint32_t round_up(uint32_t v, uint32_t a) { return (v + a - 1) / a * a; }

static int sm_count_cached() {
    static int cached[64];
    static std::once_flag once;
    std::call_once(once, [] { std::memset(cached, 0, sizeof(cached)); });
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
    if (cached[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
        cached[dev] = n;
    }
    return cached[dev];
}

// The tcgen05 kernel's variant for a launch: the batch rows its tensor memory and drain warps are laid out for.
static inline uint32_t tc_rows(uint32_t m) { return m <= 16 ? 16u : (m <= 32 ? 32u : (m <= 64 ? 64u : 128u)); }

struct TcPlan {
    TcParams p;
    uint32_t threads, smem, grid, nr;
    bool coop;      // the CTA, not its drain warps, finishes a split tile at the end of its range
};

// (See the kernel.  The CTA's sums cost one pass of its threads for each `threads` quads of rows of a column, the drain warps' one round trip for
// two contributors, and the drain warps of a tile's first CTAs are done while the last ones still run.  us, by the drain warps / by the CTA:
//   two CTAs to a tile in a split along the tiles, whose ends all come at once: 1536 x 9472 at 33 10.0 / 10.3, at 64 10.8 / 11.8, at 128 15.5 / 16.8
//   three and more, or ranges shorter than a tile, up to 56 rows (two passes): 3072 x 5120 at 33 11.0 / 10.5, at 56 11.7 / 11.3, 4096 x 4096 at 48 11.3 / 11.0,
//     2048 x 14336 at 48 16.1 / 15.8, 16384 x 5120 at 56 29.9 / 28.4, 8192 x 1024 at 48 15.5 / 11.9; but 1024 x 14336, a tile of eight units to ranges of
//     seven, at 33 11.4 / 11.7
//   57 to 64 rows (three passes): 4096 x 4096 at 64 12.0 / 12.5, 1024 x 1024, eight CTAs to a tile, 9.6 / 10.4, 2048 x 2048, nine, 11.4 / 11.3, 8192 x 1024, 18,
//     16.2 / 15.0; ranges 4096 x 8192, 2.3 to a tile, 18.45 / 18.55, 5120 x 5120 with groups of 64, 3.6 to a tile, 17.3 / 16.9
//   beyond: 3072 x 5120 at 65 14.9 / 13.8, at 128 17.2 / 17.05; ranges 1024 x 12800 at 128 18.1 / 18.9, 4096 x 8192 at 65 23.1 / 22.2, at 128 27.2 / 27.2
// With groups of 64 and 33 to 64 rows the loop of this variant is 1 % faster a unit besides, so that it is taken for long ranges too: 2048 x 57344,
// 65 units, at 33 39.3 / 38.6, at 64 41.35 / 41.5, 8192 x 38400, 130, 86.1 / 84.7 and 92.5 / 90.9, but 4096 x 28672, 49, at 64 40.1 / 40.6.)
static inline bool tc_coop(uint32_t nr, uint32_t group, uint32_t rows, uint32_t threads, uint32_t KT, const Split& sp) {
    const uint32_t units = sp.units_per_cta;
    if (nr == 128) return sp.split ? sp.split > 2 : KT >= 2 * units;
    if (nr <= 32 || (!sp.split && group == 64 && units >= 64)) return true;
    if ((rows + 3) / 4 * 128 <= 2 * threads) return sp.split ? sp.split > 2 : KT >= units + 2;
    return sp.split ? sp.split > 8 : KT >= 3 * units;
}

static fq_status_t make_plan_tc(const fq_layout_t* L, uint32_t M, TcPlan& pl) {
    TcParams& p = pl.p;
    std::memset(&p, 0, sizeof(p));
    pl.nr = tc_rows(M);
    const uint32_t GPS = kBK / L->group;
    const int sms = sm_count_cached();
    if (sms <= 0) return fail(FQ_ERR_CUDA, "no CUDA device: %s", cudaGetErrorString(cudaGetLastError()));
    p.M = M; p.K = L->K; p.N = L->N; p.KT = L->K / kBK; p.NT = L->N / 128;
    p.halves = L->BN / 128;
    p.nmma = round_up(M, 16);
    p.parts = L->value_type == FQ_VALUE_FP16 ? 2 : 1;
    const Split sp = split_tc(p.NT, p.KT, sms, pl.nr, L->group);
    p.shares = shares_of(sp, p.NT, p.KT);
    p.off_w = 256 * p.nmma;
    p.off_sz = p.off_w + 8192;
    p.stage_bytes = tc_stage_bytes(p.nmma, GPS);
    p.stages = tc_stages(pl.nr, p.nmma, GPS);
    p.max_tile_packets = L->max_tile_packets;
    p.off_wo = p.stages * p.stage_bytes;
    p.off_bar = p.off_wo + tc_wo_bytes(pl.nr);
    pl.smem = p.off_bar + 2048;
    const int ug = tc_unpack_groups(pl.nr), sg = tc_scatter_groups(pl.nr);
    pl.threads = 32 * (4 + 4 * ug + 4 * std::max<uint32_t>(1, pl.nr / 32) + 4 * sg);     // as TcShape::WARPS
    pl.grid = sp.grid;
    pl.coop = tc_coop(pl.nr, L->group, M, pl.threads, p.KT, sp);
    return FQ_OK;
}

// The tiled tensor map of a launch's activations: boxes of 64 K values by the MMA's batch rows, 128-byte swizzle;
// rows beyond M read as zero.
static fq_status_t encode_x_map(const fq_layout_t* L, const uint16_t* X, uint32_t M, uint32_t nmma, CUtensorMap* map) {
    typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                 const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static const EncodeFn fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult qr;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &qr) != cudaSuccess || qr != cudaDriverEntryPointSuccess) f = nullptr;
        return (EncodeFn)f;
    }();
    if (!fn) return fail(FQ_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
    const cuuint64_t dims[2] = {L->K, M}, strides[1] = {(cuuint64_t)L->K * 2};
    const cuuint32_t box[2] = {64, nmma}, ones[2] = {1, 1};
    const CUresult e = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)X, dims, strides, box, ones, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return e == CUDA_SUCCESS ? FQ_OK : fail(FQ_ERR_CUDA, "cuTensorMapEncodeTiled: %d", (int)e);
}

// Short jobs go to fq_direct_kernel: launches of up to 16 rows on layers with so few strips of 32 columns and
// so few k-steps that a CTA of the streaming kernel would get only a handful of units, and its fixed costs
// (ring start-up, settlement of split tiles) would be most of the call.  Returns the warps per CTA of the
// direct kernel, 0 = not a short job.  The bounds are where it measured faster than the streaming kernel
// on B200: every strip a CTA of its own on its own SM and at most two k-steps to a warp (32 warps up to 8 rows,
// 16 warps with twice the accumulators for 9-16 rows); for a single row also up to two CTAs of 16 warps to an SM.
// Not layers with tails, which its lanes read packet by packet from global memory (4096 x 4096 clustered at one, four, eight
// rows 14.5, 20.7, 24.5 us, on the streaming kernel 12.5, 13.5, 15.1; 2048 x 2048 at 16 rows 69 us, 8.1 on the tcgen05 kernel).
typedef void (*DirectFn)(const DirectParams);
static inline uint32_t direct_warps(const fq_layout_t* L, uint32_t rows, bool outliers) {
    const int sms = sm_count_cached();
    if (sms <= 0 || rows > 16 || L->kernel_hint == 1 || (outliers && L->max_tail_packets > 0)) return 0;
    const uint32_t strips = L->N / 32, KT = L->K / kBK;
    if (strips <= (uint32_t)sms) {
        if (rows <= 8) return KT <= 64 ? 32u : 0u;
        return KT <= 32 ? 16u : 0u;
    }
    return (rows == 1 && strips <= 2u * (uint32_t)sms && KT <= 32) ? 16u : 0u;
}
// UNI: whether the kernel tells the compiler that a warp's number is the same in all its lanes.  Without outliers that is
// always faster (4096 x 4096 at one row 4.8 us, so 4.1).  With outliers it goes both ways with the size of the job (us, without /
// with): at one to four rows, 8192 x 1024 at four 9.9 / 10.4, 4096 x 2176 at two 5.8 / 6.1, 2048 x 2048 4.2 / 4.2, 2048 x 4608 4.4 / 4.3, 8192 x 4736
// 11.0 / 10.8; at five to eight, 1024 x 1024 4.1 / 3.9, 2048 x 4608 5.3 / 5.0, 4096 x 4096 7.3 / 7.5, 8192 x 1024 11.5 / 12.0, 8192 x 4736 at five
// 12.5 / 12.0, and with groups of 64 1024 x 1024 4.1 / 4.05, 2048 x 2048 5.0 / 5.1, 8192 x 1024 11.8 / 12.5, 6016 x 4096 10.3 / 10.6.
static inline bool direct_uniform(const fq_layout_t* L, uint32_t rows) {
    const uint32_t strips = L->N / 32, KT = L->K / kBK;
    if (rows <= 4) return strips > 96;
    return L->group == 64 ? KT <= 8 : (KT <= 16 || strips * KT >= 4500);
}
template <int MO, int MS, int W, bool UNI>
static DirectFn pick_direct_group(uint32_t g) {
    return g == 64 ? (DirectFn)fq_direct_kernel<MO, MS, 64, true, W, UNI> : (DirectFn)fq_direct_kernel<MO, MS, 128, true, W, UNI>;
}
template <int W, bool UNI>
static DirectFn pick_direct_rows(uint32_t rows, uint32_t g) {
    if (rows == 1) return pick_direct_group<1, 1, W, UNI>(g);
    if (rows <= 4) return pick_direct_group<1, 4, W, UNI>(g);
    return pick_direct_group<1, 8, W, UNI>(g);
}
template <int MO, int W, bool UNI>
static DirectFn pick_direct_dense(uint32_t g) {
    return g == 64 ? (DirectFn)fq_direct_kernel<MO, 8 * MO, 64, false, W, UNI> : (DirectFn)fq_direct_kernel<MO, 8 * MO, 128, false, W, UNI>;
}
static DirectFn pick_direct(const fq_layout_t* L, uint32_t rows, uint32_t warps, bool sparse) {
    const uint32_t g = L->group;
    if (!sparse) return rows > 8 ? pick_direct_dense<2, 16, false>(g) : (warps == 32 ? pick_direct_dense<1, 32, true>(g) : pick_direct_dense<1, 16, false>(g));
    if (rows > 8) return pick_direct_group<2, 16, 16, false>(g);
    if (warps == 16) return pick_direct_group<1, 1, 16, false>(g);      // (two CTAs to an SM: a single row only)
    return direct_uniform(L, rows) ? pick_direct_rows<32, true>(rows, g) : pick_direct_rows<32, false>(rows, g);
}

// Which kernel serves a launch.  The tcgen05 kernel's time hardly depends on the rows (4096 x 28672, 1 % of outliers: 28.0 us
// at nine rows, 28.2 at 16, 31.1 at 32), the warp-level MMA kernels' grows (20.4 us at one row, 24.0 at eight, 34.8 at 16), and its start
// and end cost more than theirs (1024 x 4096 at nine 4.3 / 5.6).  It writes outliers into a tile instead of adding them, so an encoding that names a
// position twice (or may do so) stays with launches of 16 rows on the other kernels.  Times below: us, theirs / its, 1 % unless stated.
//   more than 16 rows   always
//   9 to 16 rows        with tails (2048 x 2048 8.8 / 6.2), or from 512 units of 128 x 128 weights up (4096 x 4096 10.4 / 8.2, 1024 x 8192
//                       7.5 / 6.5; 1024 x 6144, which is no short job either and stays with theirs, 8.1 / 6.2).  But not jobs of one k-step to a warp of
//                       the short-job kernel (2048 x 4096 6.2 / 6.35, at 0.5 % 5.6 / 6.3, 2048 x 4608 6.2 / 6.65), unless their buckets are
//                       deep (2 %: 8.5 / 6.5, 5 %: 12.5 / 7.5).
//   2 to 8 rows         tiles of 128 columns, where the streaming kernel has half the dense warps, at least 1024 units, no short job; and
//     with tails        always (4096 x 6272 at 2 % 14.4 / 12.1, 8 rows 17.1 / 12.2; 8192 x 16512 57.3 / 56.5, 71.2 / 56.6)
//     else              where the streaming kernel would run one group of dense warps (1024 x 16512 9.5 / 9.2, 8 rows 10.4 / 9.3), or two only by its split along
//                       the tiles and buckets are deep (2304 x 7296 at five 8.2 / 8.75, at 3 % 9.6 / 9.2, at four 8.7 / 9.2); from 4096 units at
//                       up to four rows (8192 x 16512 32.3 / 31.2, 2048 x 28800 16.7 / 16.8) if buckets are not deep (8192 x 16512 at 5 %
//                       37.5 / 46.1; at 2 %, which stays with theirs, 33.7 / 32.4); from 3072 at five and more (2048 x 28800 at 8 rows 17.9 /
//                       17.0, 8192 x 6272 at five 15.3 / 15.3), or from 2048 with buckets of middling depth (4096 x 9344 at 2 % at five 13.6 / 13.1,
//                       but at 1 % 12.3 / 12.7; at 5 % 16.7 / 17.2)
// Without outliers (the layer has none, or the call is the dense half of the unfused pair) it takes launches of more than 16
// rows, and the others, which have variants without the outlier step, those of up to 16 (4096 x 14336 at 16 rows 14.8 / 14.9); two or
// three launches of the short-job kernel are faster than one of it on small layers (1024 x 1024 at 32 rows 4.9 / 7.6, at 48 7.4 / 8.5, at 64
// 9.8 / 9.7; 2048 x 2048 at 32 7.1 / 8.3, at 48 10.6 / 9.2; 4096 x 4096 at 32 11.9 / 9.7).
static inline bool tc_serves(const fq_layout_t* L, uint32_t rows, bool outliers) {
    const uint32_t KT = L->K / kBK, depth = L->max_bucket_packets;
    const uint64_t units = (uint64_t)KT * (L->N / 128);
    if (!outliers) return rows > 16 && !(rows <= (units <= 128 ? 48u : 32u) && units <= 512 && direct_warps(L, 16, false));
    if (L->tilecoo_encoded != 1 || L->abi != FQ_ABI_ENCODED) return false;
    if (rows > 16) return true;
    const bool tails = L->max_tail_packets > 0;
    if (rows >= 9) return tails || (units >= 512 && !(KT <= 16 && depth <= 9 && direct_warps(L, rows, true)));
    if (L->BN != 128 || rows < 2 || units < 1024 || direct_warps(L, rows, true)) return false;
    const uint32_t sms = (uint32_t)sm_count_cached();
    const Split theirs = rows <= 4 || depth <= 10 ? split_streaming(128, L->N / 128, KT, sms, rows, true) : split_units(L->N / 128, KT, sms, 1);
    if (tails || theirs.units_per_cta < kTwoGroups) return true;
    return rows <= 4 ? units >= 4096 && depth <= 13 : units >= 3072 || (units >= 2048 && depth > 10 && depth <= 18);
}
static inline uint32_t rows_per_launch(const fq_layout_t* L, uint32_t rows_left, bool outliers) { return tc_serves(L, rows_left, outliers) ? rows_left : std::min<uint32_t>(rows_left, 16u); }

// Scratch layout: status word and header, tile-arrival counters, FP32 partial slots (two per CTA).
struct Scratch {
    size_t off_partials, total;
};
static Scratch scratch_layout(uint32_t BN, uint32_t rows) {
    Scratch sc;
    sc.off_partials = kWsHeaderBytes + kWsCounterBytes;
    // a slot: the columns of a stored tile by 16 rows, or the tcgen05 kernel's 128 columns by its rows (not less than the
    // stored tile by 32: FQ_STATIC_SCRATCH_MAX_M states what the built-in scratch holds)
    const size_t slot = rows <= 16 ? (size_t)BN * 16 : std::max<size_t>(128 * (size_t)tc_rows(rows), (size_t)BN * 32);
    sc.total = sc.off_partials + (size_t)kMaxCtas * 2 * slot * 4;
    return sc;
}

// The rows of the largest launch that `bytes` of scratch are enough for; 0: too few for this M.  fq_workspace_bytes states what one
// launch of all rows needs; with less, a larger M takes launches of 64, 32 or 16 rows.  The least that is accepted
// is the scratch of 32 rows (groups of 128) or 16 (groups of 64), or of M if that is fewer.
static uint32_t rows_for_scratch(const fq_layout_t* L, uint32_t M, size_t bytes) {
    const uint32_t least = std::min<uint32_t>(M, L->group == 64 ? 16 : 32);
    if (bytes < scratch_layout(L->BN, least).total) return 0;
    for (uint32_t rows : {M, 64u, 32u})
        if (rows <= M && bytes >= scratch_layout(L->BN, rows).total) return rows;
    return least;
}

struct MmaPlan {
    MmaParams p;
    uint32_t threads, smem, grid;
    uint32_t ngrp;   // groups of dense warps
    bool general;    // the layer needs the general form of the outlier step
};
typedef void (*MmaKernelFn)(const MmaParams);

// Plan of the streaming kernel (fq_mma_kernel): M <= 16 per launch.
static fq_status_t make_plan_mma(const fq_layout_t* L, uint32_t M, bool sparse, MmaPlan& pl) {
    const uint32_t BN = L->BN, NB = L->buckets_per_tile, GPS = kBK / L->group;
    const uint32_t MO = M <= 8 ? 1 : 2, ROWS = 8 * MO;
    const uint32_t NDW = BN / 32;
    MmaParams& p = pl.p;
    std::memset(&p, 0, sizeof(p));
    p.M = M; p.K = L->K; p.N = L->N; p.KT = L->K / kBK; p.NT = L->N / BN; p.NB = NB;
    const uint32_t w_bytes = 16 * BN * 4, sz_bytes = 2 * GPS * BN * 2;
    const uint32_t xt_bytes = sparse ? (M == 1 ? 512 : (M <= 4 ? 2048 : MO * 4096)) : 0;     // FP32 [k], [k][4] or [octet][k][8]
    // Two groups of dense warps (each takes every other unit) pay off when a CTA has enough units to
    // stream; short jobs keep one group.  With two octets of rows the second group fits only because
    // the outlier step of that variant prefetches less (96 registers per thread).
    const int sms = sm_count_cached();
    if (sms <= 0) return fail(FQ_ERR_CUDA, "no CUDA device: %s", cudaGetErrorString(cudaGetLastError()));
    const Split sp = split_streaming(BN, p.NT, p.KT, sms, M, sparse);
    p.shares = shares_of(sp, p.NT, p.KT);
    pl.ngrp = sp.units_per_cta >= kTwoGroups ? 2 : 1;
    const uint32_t xch_bytes = pl.ngrp > 1 ? BN * ROWS * 4 : 0;   // hand-over of a group's partial sums
    const uint32_t fixed = 1024 + xch_bytes;
    const uint32_t budget = kSmemBudget;
    uint32_t cap = 0;
    if (sparse) {
        cap = L->tilecoo_encoded ? std::max<uint32_t>(8, round_up(L->max_tile_packets, 8)) : 256;
        cap = std::min<uint32_t>(cap, 1024);
    }
    uint32_t stage = 0, S = 0;
    for (;;) {
        p.off_sz = w_bytes;
        p.off_xcan = p.off_sz + round_up(sz_bytes, 128);
        p.off_xsum = p.off_xcan + round_up(ROWS * kXPitch, 128);
        p.off_xt = p.off_xsum + round_up(GPS * ROWS * 4, 128);          // stage-relative in this kernel
        p.off_info = p.off_xt + xt_bytes;
        p.off_coo = p.off_info + (sparse ? round_up(NB * 4, 128) : 0);
        stage = round_up(p.off_coo + cap * 16, 128);
        // An even number of stages: the activation warps and the dense groups take alternate units, and
        // a parity wait is only valid for a waiter that meets every phase of the barrier.  With S even a
        // stage always comes back to the same activation warp and the same dense group.
        S = std::min<uint32_t>(8, (budget - fixed) / stage) & ~1u;
        if (S >= 4 || cap <= 64) break;
        cap = std::max<uint32_t>(64, cap / 2);
    }
    if (S < 4) return fail(FQ_ERR_UNSUPPORTED_SHAPE, "shared-memory stages do not fit");
    p.coo_cap = cap; p.stages = S; p.stage_bytes = stage;
    // hot columns, tiles larger than the staged part, or an encoding whose sizes were not recorded
    pl.general = sparse && (L->max_tail_packets > 0 || L->max_tile_packets > cap || !L->tilecoo_encoded);
    p.off_shc = S * stage;
    p.off_bar = p.off_shc + xch_bytes;
    // One CTA to an SM, also where two would fit: the next call's grid is there before this one ends (programmatic dependent launch), and if
    // a grid has fewer CTAs than the GPU SMs, the free SMs take two of the next one's, which then last longest (us, two fit / one: without
    // outliers on tiles of 128 columns 9472 x 1408, 143 CTAs, at one row 7.4 / 6.3, at 16 11.5 / 8.9, 6272 x 8832, 138 CTAs, 17.4 / 11.9; with them
    // 8448 x 1152 at one 7.6 / 7.0; and of grids that fill the GPU 14336 x 4224 13.05 / 12.9, 1024 x 11136 6.3 / 6.2).
    pl.smem = std::max<uint32_t>(p.off_bar + 1024, kSmemOneCta);
    pl.threads = 32 * (1 + kActWarps + pl.ngrp * NDW);
    pl.grid = sp.grid;
    return FQ_OK;
}

// MS: form of the outlier step (1: single batch row, one column per lane; 8: rows split over the lanes);
// NGRP: groups of dense warps; HOT: general form of the outlier step
// (long bucket lists shared out, packets beyond the staged part of a tile)
template <int BN, int MO, int G, bool HOT>
static MmaKernelFn pick_mma_sparse(bool sparse, uint32_t ms, uint32_t ngrp) {
    if constexpr (MO == 1) {
        if (ngrp == 2) {
            if (!sparse) return (MmaKernelFn)fq_mma_kernel<BN, MO, G, false, 8, 2, false>;
            if (ms == 1) return (MmaKernelFn)fq_mma_kernel<BN, MO, G, true, 1, 2, HOT>;
            if (ms == 4) return (MmaKernelFn)fq_mma_kernel<BN, MO, G, true, 4, 2, HOT>;
            return (MmaKernelFn)fq_mma_kernel<BN, MO, G, true, 8, 2, HOT>;
        }
        if (sparse && ms == 1) return (MmaKernelFn)fq_mma_kernel<BN, MO, G, true, 1, 1, HOT>;
        if (sparse && ms == 4) return (MmaKernelFn)fq_mma_kernel<BN, MO, G, true, 4, 1, HOT>;
    }
    if constexpr (MO == 2) {
        if (ngrp == 2) return sparse ? (MmaKernelFn)fq_mma_kernel<BN, MO, G, true, 8, 2, HOT> : (MmaKernelFn)fq_mma_kernel<BN, MO, G, false, 8, 2, false>;
    }
    if (!sparse) return (MmaKernelFn)fq_mma_kernel<BN, MO, G, false, 8, 1, false>;
    return (MmaKernelFn)fq_mma_kernel<BN, MO, G, true, 8, 1, HOT>;
}
template <int BN, int MO>
static MmaKernelFn pick_mma_group(uint32_t g, bool sparse, uint32_t ms, uint32_t ngrp, bool hot) {
    if (g == 64) return hot ? pick_mma_sparse<BN, MO, 64, true>(sparse, ms, ngrp) : pick_mma_sparse<BN, MO, 64, false>(sparse, ms, ngrp);
    return hot ? pick_mma_sparse<BN, MO, 128, true>(sparse, ms, ngrp) : pick_mma_sparse<BN, MO, 128, false>(sparse, ms, ngrp);
}
static MmaKernelFn pick_mma_kernel(uint32_t bn, uint32_t M, uint32_t g, bool sparse, uint32_t ngrp, bool hot) {
    const uint32_t mo = M <= 8 ? 1 : 2, ms = M <= 1 ? 1 : (M <= 4 ? 4 : 8);
    if (bn == 128) return mo == 1 ? pick_mma_group<128, 1>(g, sparse, ms, ngrp, hot) : pick_mma_group<128, 2>(g, sparse, ms, ngrp, hot);
    return mo == 1 ? pick_mma_group<256, 1>(g, sparse, ms, ngrp, hot) : pick_mma_group<256, 2>(g, sparse, ms, ngrp, hot);
}

typedef void (*TcKernelFn)(const CUtensorMap, const TcParams);
template <int NR, bool COOP>
static TcKernelFn pick_tc_group(uint32_t g) { return g == 64 ? (TcKernelFn)fq_tc_kernel<NR, 64, COOP> : (TcKernelFn)fq_tc_kernel<NR, 128, COOP>; }
static TcKernelFn pick_tc_kernel(uint32_t nr, uint32_t g, bool coop) {             // (coop: always, up to 32 rows)
    if (nr == 128) return coop ? pick_tc_group<128, true>(g) : pick_tc_group<128, false>(g);
    if (nr == 64) return coop ? pick_tc_group<64, true>(g) : pick_tc_group<64, false>(g);
    return nr == 32 ? pick_tc_group<32, true>(g) : pick_tc_group<16, true>(g);
}

// cudaFuncSetAttribute costs several microseconds: do it once per (kernel, device).
static cudaError_t ensure_smem_attr(const void* fn, int bytes) {
    struct Seen { const void* fn; int dev; };
    static Seen seen[256];
    static int nseen = 0;
    static std::mutex mu;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    for (int i = 0; i < nseen; ++i)
        if (seen[i].fn == fn && seen[i].dev == dev) return cudaSuccess;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && nseen < 256) seen[nseen++] = Seen{fn, dev};
    return e;
}

static bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

// Argument checks of the device entry points: nothing is enqueued when one fails.
static fq_status_t check_gemm_args(const fq_layout_t* L, const void* X, uint32_t M, const void* wq, const void* scale,
                                   const void* zero, const void* indptr, const void* info, const void* packed, void* Y,
                                   void* workspace, bool sparse) {
    if (!layout_ok(L)) return fail(FQ_ERR_INVALID_ARG, "bad layout");
    if (M < 1 || M > FQ_MAX_M) return fail(FQ_ERR_INVALID_ARG, "M = %u outside [1, %u]", M, FQ_MAX_M);
    if (!X || !wq || !scale || !zero || !Y || !workspace) return fail(FQ_ERR_INVALID_ARG, "null device pointer");
    if (sparse && (!indptr || !info)) return fail(FQ_ERR_INVALID_ARG, "null Tile-COO pointer");
    if (sparse && !packed && (L->max_tile_packets || !L->tilecoo_encoded)) return fail(FQ_ERR_INVALID_ARG, "null packet pointer");
    if (!aligned(X, 16) || !aligned(Y, 16) || !aligned(wq, 128) || !aligned(scale, 128) || !aligned(zero, 128) ||
        !aligned(workspace, 128) || (sparse && (!aligned(indptr, 4) || !aligned(info, 128) || !aligned(packed, 128))))
        return fail(FQ_ERR_INVALID_ARG, "misaligned device pointer");
    return FQ_OK;
}

static fq_status_t launch_gemm(const fq_layout_t* L, const void* X, uint32_t M, const void* wq, const void* scale,
                               const void* zero, const void* indptr, const void* info, const void* packed, void* Y,
                               void* workspace, size_t workspace_bytes, void* stream, bool sparse) {
    fq_status_t st = check_gemm_args(L, X, M, wq, scale, zero, indptr, info, packed, Y, workspace, sparse);
    if (st != FQ_OK) return st;
    const bool outliers = sparse && !(L->tilecoo_encoded && L->max_tile_packets == 0);
    const Scratch sc = scratch_layout(L->BN, M);
    const uint32_t most_rows = rows_for_scratch(L, M, workspace_bytes);
    if (!most_rows) return fail(FQ_ERR_BUFFER_TOO_SMALL, "workspace holds %zu bytes, %zu needed", workspace_bytes, sc.total);
    cudaLaunchAttribute attr[1];
    std::memset(attr, 0, sizeof(attr));
    // Programmatic dependent launch: a grid may become resident while the kernel before it in the stream
    // drains.  Its producer warps then already stream weights (which no kernel writes); everything that touches
    // X, Y or the scratch first executes griddepcontrol.wait, after which all memory operations of the earlier
    // grids are complete and visible.
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    for (uint32_t m0 = 0; m0 < M;) {
        const uint32_t mb = rows_per_launch(L, std::min(M - m0, most_rows), outliers);
        const uint16_t* Xm = (const uint16_t*)X + (size_t)m0 * L->K;
        uint16_t* Ym = (uint16_t*)Y + (size_t)m0 * L->N;
        cudaLaunchConfig_t cfg;
        std::memset(&cfg, 0, sizeof(cfg));
        cfg.stream = (cudaStream_t)stream;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cudaError_t e;
        if (tc_serves(L, mb, outliers)) {
            TcPlan pl;
            st = make_plan_tc(L, mb, pl);
            if (st != FQ_OK) return st;
            TcParams& p = pl.p;
            p.Y = Ym;
            p.wq = (const uint8_t*)wq; p.scale = (const uint16_t*)scale; p.zero = (const uint16_t*)zero;
            p.indptr = (const uint32_t*)indptr; p.info = (const uint32_t*)info; p.packed = (const uint4*)packed;
            p.status = (uint32_t*)workspace;
            p.counters = (uint32_t*)((uint8_t*)workspace + kWsHeaderBytes);
            p.partials = (float*)((uint8_t*)workspace + sc.off_partials);
            CUtensorMap xmap;
            st = encode_x_map(L, Xm, mb, p.nmma, &xmap);
            if (st != FQ_OK) return st;
            TcKernelFn fn = pick_tc_kernel(pl.nr, L->group, pl.coop);
            e = ensure_smem_attr((const void*)fn, (int)kSmemBudget);
            if (e != cudaSuccess) return fail(FQ_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
            cfg.gridDim = dim3(pl.grid);
            cfg.blockDim = dim3(pl.threads);
            cfg.dynamicSmemBytes = pl.smem;
            e = cudaLaunchKernelEx(&cfg, fn, xmap, p);
        } else if (direct_warps(L, mb, outliers)) {
            DirectParams p;
            std::memset(&p, 0, sizeof(p));
            p.X = Xm; p.Y = Ym;
            p.wq = (const uint8_t*)wq; p.scale = (const uint16_t*)scale; p.zero = (const uint16_t*)zero;
            p.indptr = (const uint32_t*)indptr; p.info = (const uint32_t*)info; p.packed = (const uint4*)packed;
            p.status = (uint32_t*)workspace;
            p.M = mb; p.K = L->K; p.N = L->N; p.KT = L->K / kBK; p.BN = L->BN; p.NB = L->buckets_per_tile;
            const uint32_t warps = direct_warps(L, mb, outliers);
            cfg.gridDim = dim3(L->N / 32);
            cfg.blockDim = dim3(32 * warps);
            // per warp: rows of activations, their k-major copy, scale and zero rows, staged packets; the warps'
            // sums reuse those bytes
            cfg.dynamicSmemBytes = warps * kDirectWarpBytes;
            DirectFn dfn = pick_direct(L, mb, warps, outliers);
            e = ensure_smem_attr((const void*)dfn, 32 * kDirectWarpBytes);
            if (e != cudaSuccess) return fail(FQ_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
            e = cudaLaunchKernelEx(&cfg, dfn, p);
        } else {
            MmaPlan pl;
            st = make_plan_mma(L, mb, outliers, pl);
            if (st != FQ_OK) return st;
            MmaParams& p = pl.p;
            p.X = Xm; p.Y = Ym;
            p.wq = (const uint8_t*)wq; p.scale = (const uint16_t*)scale; p.zero = (const uint16_t*)zero;
            p.indptr = (const uint32_t*)indptr; p.info = (const uint32_t*)info; p.packed = (const uint4*)packed;
            p.status = (uint32_t*)workspace;
            p.counters = (uint32_t*)((uint8_t*)workspace + kWsHeaderBytes);
            p.partials = (float*)((uint8_t*)workspace + sc.off_partials);
            MmaKernelFn fn = pick_mma_kernel(L->BN, mb, L->group, outliers, pl.ngrp, pl.general);
            e = ensure_smem_attr((const void*)fn, (int)kSmemBudget);
            if (e != cudaSuccess) return fail(FQ_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
            cfg.gridDim = dim3(pl.grid);
            cfg.blockDim = dim3(pl.threads);
            cfg.dynamicSmemBytes = pl.smem;
            e = cudaLaunchKernelEx(&cfg, fn, p);
        }
        if (e != cudaSuccess) return fail(FQ_ERR_CUDA, "kernel launch: %s", cudaGetErrorString(e));
        m0 += mb;
    }
    return FQ_OK;
}

template <int RR>
static cudaError_t launch_spmm(const fq_layout_t* L, const uint16_t* X, uint32_t M, const void* indptr, const void* info,
                               const void* packed, uint16_t* Y, uint32_t slabs, cudaStream_t stream) {
    const uint32_t smem = (uint32_t)RR * L->BN * 4 + kSpmmChunk * kBK * RR * 2;
    cudaError_t e = ensure_smem_attr((const void*)fq_spmm_kernel<RR>, 64 * 1024);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(L->N / L->BN * slabs);
    cfg.blockDim = dim3(kSpmmThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[2];
    std::memset(at, 0, sizeof(at));
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = slabs, at[0].val.clusterDim.y = 1, at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;        // as the fused launches: the descriptors
    at[1].val.programmaticStreamSerializationAllowed = 1;                 // and first slots load during the tail of
    cfg.attrs = at, cfg.numAttrs = 2;                                     // the kernel before (the dense half)
    return cudaLaunchKernelEx(&cfg, fq_spmm_kernel<RR>, X, (const uint32_t*)indptr, (const uint32_t*)info,
                              (const uint4*)packed, Y, M, L->K, L->N, L->BN, slabs);
}

}  // namespace fq

using namespace fq;

extern "C" {

fq_status_t fq_workspace_bytes(const fq_layout_t* L, uint32_t M, size_t* bytes) {
    if (!layout_ok(L) || !bytes) return fail(FQ_ERR_INVALID_ARG, "bad layout or null output");
    if (M < 1 || M > FQ_MAX_M) return fail(FQ_ERR_INVALID_ARG, "M = %u outside [1, %u]", M, FQ_MAX_M);
    *bytes = scratch_layout(L->BN, M).total;
    return FQ_OK;
}

fq_status_t fq_fused_w4a16_outlier_gemm(const fq_layout_t* L, const void* X, uint32_t M, const void* wq,
                                        const void* scale, const void* zero, const void* tile_indptr,
                                        const void* bucket_info, const void* packed_outliers, void* Y,
                                        void* workspace, size_t workspace_bytes, void* cuda_stream) {
    return launch_gemm(L, X, M, wq, scale, zero, tile_indptr, bucket_info, packed_outliers, Y, workspace,
                       workspace_bytes, cuda_stream, true);
}

// ---- the entry point that allocates nothing -------------------------------------------------
// Scratch for callers that cannot allocate device memory: lives in the library's own image on
// every GPU that loads it, for the life of the process.
static __device__ __align__(256) unsigned char g_static_scratch[FQ_STATIC_SCRATCH_BYTES];

// Device address of g_static_scratch on the current device.  In host code the array's name is only
// a handle; the address a kernel can use comes from cudaGetSymbolAddress, asked once per device
// with that device current.
static fq_status_t static_scratch_address(void** out) {
    static void* addr[64] = {nullptr};
    static std::mutex mu;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return fail(FQ_ERR_CUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
    if (dev < 0 || dev >= 64) return fail(FQ_ERR_CUDA, "device ordinal %d is outside the supported range", dev);
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void* ptr = nullptr;
        e = cudaGetSymbolAddress(&ptr, g_static_scratch);
        if (e != cudaSuccess || !ptr) return fail(FQ_ERR_CUDA, "cudaGetSymbolAddress: %s", cudaGetErrorString(e));
        addr[dev] = ptr;
    }
    *out = addr[dev];
    return FQ_OK;
}

fq_status_t fq_fused_w4a16_outlier_gemm_noalloc(const fq_layout_t* L, const void* X, uint32_t M, const void* wq,
                                                const void* scale, const void* zero, const void* tile_indptr,
                                                const void* bucket_info, const void* packed_outliers, void* Y,
                                                void* cuda_stream) {
    // every argument error is reported before anything is put on the stream (the scratch pointer stands in for itself)
    fq_status_t st = check_gemm_args(L, X, M, wq, scale, zero, tile_indptr, bucket_info, packed_outliers, Y, (void*)256, true);
    if (st != FQ_OK) return st;
    const size_t need = scratch_layout(L->BN, M).total;
    if (need > (size_t)FQ_STATIC_SCRATCH_BYTES && (L->group != 64 || !rows_for_scratch(L, M, FQ_STATIC_SCRATCH_BYTES)))
        return fail(FQ_ERR_BUFFER_TOO_SMALL,
                    "this call needs %zu bytes of scratch but the built-in scratch holds %zu (M <= %u always fits); "
                    "use fq_fused_w4a16_outlier_gemm with caller-allocated scratch",
                    need, (size_t)FQ_STATIC_SCRATCH_BYTES, (unsigned)FQ_STATIC_SCRATCH_MAX_M);
    void* scratch = nullptr;
    st = static_scratch_address(&scratch);
    if (st != FQ_OK) return st;
    // the status word and the tile-arrival counters must start at zero; the previous user of the
    // shared array may have been interrupted
    cudaError_t e = cudaMemsetAsync(scratch, 0, kWsHeaderBytes + kWsCounterBytes, (cudaStream_t)cuda_stream);
    if (e != cudaSuccess) return fail(FQ_ERR_CUDA, "clearing the built-in scratch: %s", cudaGetErrorString(e));
    return launch_gemm(L, X, M, wq, scale, zero, tile_indptr, bucket_info, packed_outliers, Y, scratch,
                       (size_t)FQ_STATIC_SCRATCH_BYTES, cuda_stream, true);
}

fq_status_t fq_unfused_gemm(const fq_layout_t* L, const void* X, uint32_t M, const void* wq, const void* scale,
                            const void* zero, void* Y, void* workspace, size_t workspace_bytes, void* cuda_stream) {
    return launch_gemm(L, X, M, wq, scale, zero, nullptr, nullptr, nullptr, Y, workspace, workspace_bytes,
                       cuda_stream, false);
}

fq_status_t fq_unfused_spmm(const fq_layout_t* L, const void* X, uint32_t M, const void* tile_indptr,
                            const void* bucket_info, const void* packed_outliers, void* Y, void* cuda_stream) {
    if (!layout_ok(L)) return fail(FQ_ERR_INVALID_ARG, "bad layout");
    if (M < 1 || M > FQ_MAX_M) return fail(FQ_ERR_INVALID_ARG, "M = %u outside [1, %u]", M, FQ_MAX_M);
    if (!X || !tile_indptr || !bucket_info || !Y) return fail(FQ_ERR_INVALID_ARG, "null device pointer");
    if (!packed_outliers && (L->max_tile_packets || !L->tilecoo_encoded)) return fail(FQ_ERR_INVALID_ARG, "null packet pointer");
    if (!aligned(X, 16) || !aligned(Y, 16) || !aligned(packed_outliers, 16))
        return fail(FQ_ERR_INVALID_ARG, "misaligned device pointer");
    const int sms = sm_count_cached();
    if (sms <= 0) return fail(FQ_ERR_CUDA, "no CUDA device: %s", cudaGetErrorString(cudaGetLastError()));
    const uint32_t NT = L->N / L->BN, KT = L->K / kBK;
    // slabs of a tile = one cluster (at most eight CTAs): as many as it takes to put about two CTAs on every SM
    const uint32_t slabs = std::max<uint32_t>(1, std::min<uint32_t>(std::min<uint32_t>(8, KT), (uint32_t)(2 * sms) / NT));
    for (uint32_t m0 = 0; m0 < M; m0 += 16) {
        const uint32_t mb = std::min<uint32_t>(16, M - m0);
        const uint16_t* Xm = (const uint16_t*)X + (size_t)m0 * L->K;
        uint16_t* Ym = (uint16_t*)Y + (size_t)m0 * L->N;
        cudaStream_t st = (cudaStream_t)cuda_stream;
        cudaError_t e = mb == 1 ? launch_spmm<1>(L, Xm, mb, tile_indptr, bucket_info, packed_outliers, Ym, slabs, st)
                      : mb <= 8 ? launch_spmm<8>(L, Xm, mb, tile_indptr, bucket_info, packed_outliers, Ym, slabs, st)
                                : launch_spmm<16>(L, Xm, mb, tile_indptr, bucket_info, packed_outliers, Ym, slabs, st);
        if (e != cudaSuccess) return fail(FQ_ERR_CUDA, "spmm launch: %s", cudaGetErrorString(e));
    }
    return FQ_OK;
}

// The copies of X and Y.  A copy engine's copy between two kernels of a stream costs far more than its transfer: four
// calls at 8 rows with their eight copies (1.1 MB) took 177 us where the kernels alone take 61.  A kernel that reads or
// writes the pinned host memory itself starts like any other of the chain, its CTAs resident before the one before it ends:
// 118 us.  So short copies of pinned memory are copied by a kernel, and the engine keeps pageable memory, which
// only it can read, and long copies, where its transfer rate is what counts (host to host, us, engine / kernel: 4096 x 4096 at one row 29.9 / 20.6,
// at 32 48.9 / 38.7, at 128 83.2 / 74.6, with 1 MB each way; 4096 x 16384 at 128, with 1 and 4 MB, 159 / 157; 8192 x 28672 at 128,
// with 2 and 7 MB, 293 / 300, and with the kernel for X only 292).
constexpr size_t kKernelCopyMax = 4u << 20;
// (the loads are coherent ones, in program order behind the wait: the kernel before may still be writing `src` when this grid starts)
__device__ __forceinline__ uint4 load_coherent(const uint4* p) {
    uint4 v;
    asm volatile("ld.relaxed.sys.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__global__ void __launch_bounds__(256) fq_copy_kernel(const uint4* src, uint4* dst, uint32_t n) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t i0 = blockIdx.x * 1024 + threadIdx.x;
    uint4 v[4];                                            // four loads in flight: a read of host memory takes over a microsecond
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (i0 + 256 * j < n) v[j] = load_coherent(src + i0 + 256 * j);
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (i0 + 256 * j < n) dst[i0 + 256 * j] = v[j];
}
// Device address of `bytes` of pinned host memory, or null: not pinned, or not all of it (a kernel, unlike a copy engine's copy, would
// read on past the end of what is pinned, and fault).
static void* pinned_view(const void* host, size_t bytes) {
    typedef CUresult (*AttributesFn)(unsigned int, CUpointer_attribute*, void**, CUdeviceptr);
    static const AttributesFn fn = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult qr;
        if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &f, cudaEnableDefault, &qr) != cudaSuccess || qr != cudaDriverEntryPointSuccess) f = nullptr;
        return (AttributesFn)f;
    }();
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, host) != cudaSuccess) {
        cudaGetLastError();                                // not an error here
        return nullptr;
    }
    if (!fn || at.type != cudaMemoryTypeHost || !at.devicePointer) return nullptr;
    CUdeviceptr start = 0;
    size_t size = 0;
    CUpointer_attribute what[2] = {CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    void* out[2] = {&start, &size};
    if (fn(2, what, out, (CUdeviceptr)host) != CUDA_SUCCESS) return nullptr;
    const size_t before = (size_t)((CUdeviceptr)host - start);
    return before <= size && bytes <= size - before ? at.devicePointer : nullptr;
}
// `host`: the one of the two that is host memory.
static cudaError_t enqueue_copy(void* dst, const void* src, const void* host, size_t bytes, cudaMemcpyKind kind, cudaStream_t s) {
    if (bytes <= kKernelCopyMax && bytes % 16 == 0 && aligned(src, 16) && aligned(dst, 16)) {
        if (void* view = pinned_view(host, bytes)) {
            const uint32_t n = (uint32_t)(bytes / 16);
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((n + 1023) / 1024);
            cfg.blockDim = dim3(256);
            cfg.stream = s;
            cudaLaunchAttribute pdl[1];
            std::memset(pdl, 0, sizeof(pdl));
            pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            pdl[0].val.programmaticStreamSerializationAllowed = 1;
            cfg.attrs = pdl, cfg.numAttrs = 1;
            return cudaLaunchKernelEx(&cfg, fq_copy_kernel, (const uint4*)(src == host ? view : src),
                                      (uint4*)(dst == host ? view : dst), n);
        }
    }
    return cudaMemcpyAsync(dst, src, bytes, kind, s);
}

fq_status_t fq_fused_host_io_async(const fq_layout_t* L, const void* X_host, uint32_t M, void* x_dev, const void* wq,
                                   const void* scale, const void* zero, const void* tile_indptr,
                                   const void* bucket_info, const void* packed_outliers, void* y_dev, void* Y_host,
                                   void* workspace, size_t workspace_bytes, void* cuda_stream) {
    if (!layout_ok(L)) return fail(FQ_ERR_INVALID_ARG, "bad layout");
    if (!X_host || !Y_host || !x_dev || !y_dev) return fail(FQ_ERR_INVALID_ARG, "null pointer");
    if (M < 1 || M > FQ_MAX_M) return fail(FQ_ERR_INVALID_ARG, "M = %u outside [1, %u]", M, FQ_MAX_M);
    cudaStream_t s = (cudaStream_t)cuda_stream;
    cudaError_t e = enqueue_copy(x_dev, X_host, X_host, (size_t)M * L->K * 2, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return fail(FQ_ERR_CUDA, "copy of X: %s", cudaGetErrorString(e));
    fq_status_t st = fq_fused_w4a16_outlier_gemm(L, x_dev, M, wq, scale, zero, tile_indptr, bucket_info,
                                                 packed_outliers, y_dev, workspace, workspace_bytes, cuda_stream);
    if (st != FQ_OK) return st;
    e = enqueue_copy(Y_host, y_dev, Y_host, (size_t)M * L->N * 2, cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return fail(FQ_ERR_CUDA, "copy of Y: %s", cudaGetErrorString(e));
    return FQ_OK;
}

fq_status_t fq_fused_host_io(const fq_layout_t* L, const void* X_host, uint32_t M, void* x_dev, const void* wq,
                             const void* scale, const void* zero, const void* tile_indptr, const void* bucket_info,
                             const void* packed_outliers, void* y_dev, void* Y_host, void* workspace,
                             size_t workspace_bytes, void* cuda_stream) {
    fq_status_t st = fq_fused_host_io_async(L, X_host, M, x_dev, wq, scale, zero, tile_indptr, bucket_info,
                                            packed_outliers, y_dev, Y_host, workspace, workspace_bytes, cuda_stream);
    if (st != FQ_OK) return st;
    cudaError_t e = cudaStreamSynchronize((cudaStream_t)cuda_stream);
    if (e != cudaSuccess) return fail(FQ_ERR_CUDA, "stream synchronisation: %s", cudaGetErrorString(e));
    return FQ_OK;
}

fq_status_t fq_check_status(void* workspace, void* cuda_stream) {
    if (!workspace) return fail(FQ_ERR_INVALID_ARG, "null workspace");
    cudaStream_t s = (cudaStream_t)cuda_stream;
    uint32_t word = 0;
    cudaError_t e = cudaMemcpyAsync(&word, workspace, 4, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return fail(FQ_ERR_CUDA, "status read: %s", cudaGetErrorString(e));
    if (word != 0) {
        // A call that gave up left some tile-arrival counters short: clear the status word and all of them, so
        // that the next call on this scratch starts from a clean state (Y of the failed call is undefined).
        cudaMemsetAsync(workspace, 0, kWsHeaderBytes + kWsCounterBytes, s);
        cudaStreamSynchronize(s);
        return fail((fq_status_t)(int32_t)word, "the device reported status %d (-5: a bounded wait expired, -6: Tile-COO descriptors do not match the staged packets)", (int32_t)word);
    }
    return FQ_OK;
}

}  // extern "C"
