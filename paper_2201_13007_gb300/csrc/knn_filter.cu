// knn_filter.cu -- brute-force k nearest neighbours over BF16 rows as a
// tensor-core filter followed by an exact pass over the few rows that pass it.
//
// The scan kernel of knn.cu keeps its sorted lists beside the tiles, and at
// 200,000 rows spends most of a tile's 8,000 cycles on appends and merges, not
// on the product (73 ms for 200,000 x 96, 104 TFLOP/s). Here the product runs
// on tcgen05 and its epilogue only compares: a value that is not below its
// query row's bound is dropped, and the bound does not change inside a launch.
//
//   segments  The base is taken in nested samples: first every 2^J-th row (at
//             most 256 rows), then the rows halfway between those, and so on
//             to the odd rows, so each launch doubles the rows seen. A segment
//             is one strided tensor map, and whatever order the base is in,
//             each sample is spread over all of it.
//   filter    Per segment, every value F = |x|^2 - 2<q, x> (or -<q, x>) at or
//             below the row's bound goes to the row's list: about k per row
//             and segment, since the bound is the k-th of as many rows again.
//   tighten   Per segment and row, the k-th smallest F seen so far becomes the
//             next bound, and only the values within it are kept.
//   finish    The values kept at the end (k and a few) are computed again with
//             mma.sync, in the order of the scan kernel, and ranked by their
//             exact (key, id): results do not depend on tcgen05's sums.
//
// Bounds are widened by the largest difference that FP32 accumulation in any
// order can make (knn_row_margin), so no row that belongs to a result is
// dropped. Where a list runs over (many equal distances, a base that defeats
// the sampling, values that are not finite), the 128 query rows concerned are
// done again by the scan kernel; a row given up meets no bound from then on.
//
// Measured, all rows against all, k = 64, whole call: 200,000 x 96 in 73.5 ms
// before and 11.6 ms now (662 TFLOP/s), 20,000 x 128 in 2.93 and 0.92 ms. Of
// the 11.6 ms the filter takes 8.7, the tightens 1.8, the finish 0.8.
#include <cuda.h>

#include <algorithm>
#include <atomic>

#include "knn_common.cuh"

namespace ann {
namespace {

constexpr int FN = 256;         // base rows per tile (one UMMA: 128 x 256, K = 16 a step)
constexpr int FEPI = 16;        // epilogue warps: four per quarter of the accumulator's rows
constexpr int FCOLS = FN / (FEPI / 4);      // columns of a tile that one of them reads
constexpr int FCAP = FCOLS;                 // values one epilogue thread can append per segment (the first tile's: all)
constexpr int FTHREADS = 128 + 32 * FEPI;   // warp 0 TMA, warp 1 UMMA, warp 2 TMEM, then the epilogue
constexpr int FKEEP = 128;      // values kept per row between segments
constexpr int FMERGE = 384;     // values of one row that a tighten can take
constexpr int FSEG = 32;        // most segments
// A bound every value meets (|F| stays below 1e30, see knn_query_rows), and the segments' padding does not: bias rows
// of the byte kPadByte, three times -6.2e32.
constexpr float kOpen = 1e31f;
constexpr int kPadByte = 0xF5;
// Most tries of one wait; each may suspend for up to 20 us, so a wait that never ends costs 0.33 s at most. The longest
// that ends, an epilogue in which every value passes, takes some 100 us.
constexpr uint32_t kWaits = 1u << 14;

// ---------------------------------------------------------------- PTX
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Waits for the phase of the given parity; false if it did not come within
// the limit, or if another warp of the CTA has given up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *gave_up) {
    for (uint32_t i = 0; i < kWaits; ++i) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred p;\n"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 20000;\n"
            "selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if ((i & 63) == 63 && *gave_up) return false;
    }
    *gave_up = 1;
    return false;
}
__device__ __forceinline__ void tma_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void umma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool acc) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
        ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"((uint32_t)acc)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// 32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t (&r)[32], uint32_t addr) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(addr));
}
// The loads issued so far are complete; naming the registers keeps their uses behind the wait.
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                   "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                   "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :
                 : "memory");
}
// The sign bits of v[0..8) - lim, v[0]'s highest of the low eight.
__device__ __forceinline__ uint32_t signs_below(const uint32_t *v, float lim) {
    unsigned long long neg;
    asm("mov.b64 %0, {%1, %1};" : "=l"(neg) : "f"(-lim));
    uint32_t m = 0;
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
        uint32_t lo, hi;
        asm("{\n.reg .b64 x;\nmov.b64 x, {%2, %3};\nadd.rn.f32x2 x, x, %4;\nmov.b64 {%0, %1}, x;\n}\n"
            : "=r"(lo), "=r"(hi)
            : "r"(v[j]), "r"(v[j + 1]), "l"(neg));
        m = __funnelshift_l(lo, m, 1);
        m = __funnelshift_l(hi, m, 1);
    }
    return m;
}

// Shared-memory operand descriptor of K-major rows of 128 bytes (64 elements)
// with the 128-byte swizzle, or of 64 bytes with the 64-byte one: groups of
// eight rows lie 1024 or 512 bytes apart.
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, bool wide) {
    return (uint64_t)((saddr & 0x3FFFF) >> 4) | (1ull << 16) | ((uint64_t)((wide ? 1024 : 512) >> 4) << 32) |
           (1ull << 46) | ((wide ? 2ull : 4ull) << 61);
}
// The operands' last K step (see kBiasRow): no swizzle, eight rows of 16 bytes
// lie 128 bytes apart from the next eight; `kstep` is the distance of the step's
// second half.
__device__ __forceinline__ uint64_t umma_desc_plain(uint32_t saddr, uint32_t kstep) {
    return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)(kstep >> 4) << 16) | ((uint64_t)(128 >> 4) << 32) | (1ull << 46);
}
// BF16 x BF16 -> FP32, both operands K-major, 128 x 256.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((FN / 8) << 17) | ((KBM / 16) << 24);

// ---------------------------------------------------------------- layout
__host__ __device__ constexpr int filter_stages(int kd) { return kd == 4 ? 2 : kd == 3 ? 3 : 4; }
// One more K step adds the base row's bias to the product: the query's side is
// 1 1 1 0 ... in every row, the base row's the bias in three BF16 parts (24
// bits: exact), then values that meet zeros. It costs 128 cycles of the tensor
// pipe a tile; adding the bias in the epilogue cost a packed fma and a quarter
// of a load for each value, 768 issue slots a tile. Both sides are stored as
// the step's first eight elements of all rows, then its second eight.
constexpr int kBiasRow = 32;  // bytes of it per base row
__host__ __device__ constexpr int filter_a_bytes(int kd) { return KBM * kd * 64; }
__host__ __device__ constexpr int filter_b_bytes(int kd) { return FN * (kd * 64 + kBiasRow); }
// alignment, query rows twice, their bias step, base tiles, barriers and flags
__host__ __device__ constexpr int filter_smem(int kd) {
    return 1024 + 2 * filter_a_bytes(kd) + KBM * 32 + filter_stages(kd) * filter_b_bytes(kd) + 256;
}

// Rows of d = 32 KD elements: a tensor map of their 64-element pieces and one
// of the last 32 elements (odd KD). A TMA request fetches one piece of one row,
// so wide pieces halve the requests (of no effect on the time while the
// epilogue bounds a tile).
struct RowMaps {
    CUtensorMap wide, narrow;
};

template <int KD>
__device__ __forceinline__ void load_rows(uint32_t dst, const RowMaps &map, int rows, int y, uint32_t bar) {
#pragma unroll
    for (int w = 0; w < KD / 2; ++w) tma_2d(dst + w * rows * 128, &map.wide, w * 64, y, bar);
    if (KD & 1) tma_2d(dst + KD / 2 * rows * 128, &map.narrow, KD / 2 * 64, y, bar);
}

struct FilterArgs {
    const unsigned char *bias;  // this segment's bias rows, padded to whole tiles
    const float *thr;       // per query row: the bound
    uint2 *lists;           // [row][subs][FCAP] of (F, id)
    int32_t *counts;        // [row][subs]
    int *over;              // per 128 query rows: 1 = a list ran over
    int *err;               // set to 2 if a wait ran out; a launch that finds it set does nothing
    uint32_t first;         // the segment: base rows first, first + 2^shift, ...
    int no_loads;           // 1 = load nothing, so that every wait for data runs out (the error path, for tests)
    int shift, subs;
    int tiles, blocks, splits;
};

// Work items are (128 query rows, every splits-th tile of the segment); a CTA
// takes every gridDim.x-th. Three kinds of warps run through the same items:
// one lane issues the TMA loads (query rows double-buffered by item, base
// tiles in a ring), one lane the UMMAs into two 128 x 256 accumulators, sixteen
// warps read them, one query row a thread and a quarter of the columns a warp.
//
// Bound: at d = 96 a tile of 128 x 256 is 7 UMMAs of 128 cycles. The epilogue
// takes a three-way maximum for every two values; measured, a tile costs 1,120
// cycles, and each value that passes about 14 more (45 instructions of one
// warp, almost alone in its branch): 64 a row and segment, half of the time at
// 200,000 rows, little at 10 million. Sixteen epilogue warps, as eight waited
// on their own latencies (tile of the last segment, 200,000 rows: 2,340 cycles
// with eight, 1,880 with sixteen; 1,440 with the bias in the product).
template <int KD>
__global__ void __launch_bounds__(FTHREADS, 1)
    knn_filter_kernel(const __grid_constant__ RowMaps map_q, const __grid_constant__ RowMaps map_x,
                      const FilterArgs a) {
    constexpr int WIDE = KD / 2;  // pieces of 64 elements of a row; an odd KD has one of 32 after them
    constexpr int ST = filter_stages(KD);
    constexpr int A_BYTES = filter_a_bytes(KD), B_BYTES = filter_b_bytes(KD);
    extern __shared__ unsigned char smem_raw[];
    const uint32_t smem0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char *smem = smem_raw + (smem0 - smem_u32(smem_raw));
    const uint32_t sA = smem0, sOne = smem0 + 2 * A_BYTES, sB = sOne + KBM * 32;
    unsigned char *tail = smem + 2 * A_BYTES + KBM * 32 + ST * B_BYTES;
    const uint32_t bars = smem_u32(tail);
    auto b_full = [&](int i) { return bars + 8u * i; };
    auto b_empty = [&](int i) { return bars + 8u * (ST + i); };
    auto a_full = [&](int i) { return bars + 8u * (2 * ST + i); };
    auto a_empty = [&](int i) { return bars + 8u * (2 * ST + 2 + i); };
    auto acc_full = [&](int i) { return bars + 8u * (2 * ST + 4 + i); };
    auto acc_empty = [&](int i) { return bars + 8u * (2 * ST + 6 + i); };
    const uint32_t drained = bars + 8u * (2 * ST + 8);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(tail + 8 * (2 * ST + 9));
    volatile int *gave_up = reinterpret_cast<volatile int *>(tmem_slot + 1), *failed = gave_up + 1;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    if (tid == 0) {
        for (int i = 0; i < ST; ++i) {
            mbar_init(b_full(i), 1);
            mbar_init(b_empty(i), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(a_full(i), 1);
            mbar_init(a_empty(i), 1);
            mbar_init(acc_full(i), 1);
            mbar_init(acc_empty(i), FEPI);  // one arrival per epilogue warp
        }
        mbar_init(drained, 1);
        *gave_up = 0;
        *failed = *static_cast<volatile int *>(a.err);  // read once: other CTAs of this launch may set it
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid >= 128 && tid < 128 + KBM) {  // the query's side of the bias step: eight elements 1 1 1 0 ..., then eight zeros
        uint4 *one = reinterpret_cast<uint4 *>(smem + 2 * A_BYTES);
        one[tid - 128] = make_uint4(0x3F803F80u, 0x00003F80u, 0u, 0u);
        one[tid] = make_uint4(0u, 0u, 0u, 0u);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 2) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(tmem_slot);
    const int items = *failed ? 0 : a.blocks * a.splits;

    if (warp == 0) {
        if (lane == 0 && !a.no_loads) {
            uint32_t nb = 0, ni = 0;  // tiles and items loaded
            bool ok = true;
            for (int it = blockIdx.x; ok && it < items; it += gridDim.x) {
                const int block = it / a.splits, split = it - block * a.splits;
                const int as = ni & 1;
                ok = mbar_wait(a_empty(as), ((ni >> 1) & 1) ^ 1, gave_up);
                if (!ok) break;
                mbar_expect(a_full(as), A_BYTES);
                load_rows<KD>(sA + as * A_BYTES, map_q, KBM, block * KBM, a_full(as));
                ++ni;
                for (int t = split; t < a.tiles; t += a.splits) {
                    const int st = nb % ST;
                    ok = mbar_wait(b_empty(st), ((nb / ST) & 1) ^ 1, gave_up);
                    if (!ok) break;
                    mbar_expect(b_full(st), B_BYTES);
                    load_rows<KD>(sB + st * B_BYTES, map_x, FN, t * FN, b_full(st));
                    bulk_copy(sB + st * B_BYTES + FN * KD * 64, a.bias + (size_t)t * (FN * kBiasRow), FN * kBiasRow,
                              b_full(st));
                    ++nb;
                }
            }
            if (*gave_up) {  // let the copies in flight land before the CTA leaves
                volatile int never = 0;
                for (uint32_t i = nb > (uint32_t)ST ? nb - ST : 0; i < nb && !never; ++i)
                    mbar_wait(b_full(i % ST), (i / ST) & 1, &never);
                for (uint32_t i = ni > 2 ? ni - 2 : 0; i < ni && !never; ++i)
                    mbar_wait(a_full(i & 1), (i >> 1) & 1, &never);
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            uint32_t nb = 0, ni = 0;
            bool ok = true;
            for (int it = blockIdx.x; ok && it < items; it += gridDim.x, ++ni) {
                const int block = it / a.splits, split = it - block * a.splits;
                const int as = ni & 1;
                ok = mbar_wait(a_full(as), (ni >> 1) & 1, gave_up);
                for (int t = split; ok && t < a.tiles; t += a.splits) {
                    const int st = nb % ST, ac = nb & 1;
                    ok = mbar_wait(acc_empty(ac), ((nb >> 1) & 1) ^ 1, gave_up) &&
                         mbar_wait(b_full(st), (nb / ST) & 1, gave_up);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t pa = sA + as * A_BYTES, pb = sB + st * B_BYTES;
#pragma unroll
                    for (int k = 0; k < 4 * WIDE; ++k)
                        umma_bf16(tmem + ac * FN, umma_desc(pa + (k >> 2) * (KBM * 128) + (k & 3) * 32, true),
                                  umma_desc(pb + (k >> 2) * (FN * 128) + (k & 3) * 32, true), kIdesc, k > 0);
#pragma unroll
                    for (int k = 4 * WIDE; k < 2 * KD; ++k)
                        umma_bf16(tmem + ac * FN, umma_desc(pa + WIDE * (KBM * 128) + (k & 1) * 32, false),
                                  umma_desc(pb + WIDE * (FN * 128) + (k & 1) * 32, false), kIdesc, k > 0);
                    umma_bf16(tmem + ac * FN, umma_desc_plain(sOne, KBM * 16),
                              umma_desc_plain(pb + FN * KD * 64, FN * 16), kIdesc, true);
                    umma_commit(b_empty(st));
                    umma_commit(acc_full(ac));
                    ++nb;
                }
                umma_commit(a_empty(as));
            }
            // nothing is in flight when the accumulators are freed, on the way out early too
            umma_commit(drained);
            volatile int never = 0;
            mbar_wait(drained, 0, &never);
        }
    } else if (warp >= 4) {
        const int part = (warp - 4) >> 2, quad = warp & 3;  // a warp reads the TMEM rows of its number mod 4
        uint32_t nb = 0;
        bool ok = true;
        for (int it = blockIdx.x; ok && it < items; it += gridDim.x) {
            const int block = it / a.splits, split = it - block * a.splits;
            const size_t row = (size_t)block * KBM + quad * 32 + lane;
            const size_t sub = row * a.subs + split * (FEPI / 4) + part;
            uint2 *const list = a.lists + sub * FCAP;
            int at = 0;
            bool over = false;
            float lim = -a.thr[row];  // the accumulator holds -F
            for (int t = split; t < a.tiles; t += a.splits) {
                const int ac = nb & 1;
                ok = mbar_wait(acc_full(ac), (nb >> 1) & 1, gave_up);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t src = tmem + ((uint32_t)(quad * 32) << 16) + ac * FN + part * FCOLS;
                uint32_t v[FCOLS / 32][32];
                static_assert(FCOLS == 64, "two loads of 32 columns");
                // both halves are read, and the accumulator handed back, before either is looked at: values that pass
                // then delay this warp alone and not the next product
                tmem_ld32(v[0], src);
                tmem_ld32(v[1], src + 32);
                tmem_wait(v[0]);
                tmem_wait(v[1]);
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(acc_empty(ac));
#pragma unroll
                for (int c = 0; c < FCOLS / 32; ++c) {
                    uint32_t(&w)[32] = v[c];
                    float m[4];
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        const uint32_t *x = w + g * 8;
                        m[g] = fmaxf(__uint_as_float(x[0]), __uint_as_float(x[1]));
#pragma unroll
                        for (int j = 2; j < 8; j += 2)
                            m[g] = fmaxf(fmaxf(m[g], __uint_as_float(x[j])), __uint_as_float(x[j + 1]));
                    }
                    if (fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3])) >= lim) {
                        const uint32_t id0 = a.first + ((uint32_t)(t * FN + part * FCOLS + c * 32) << a.shift);
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            if (m[g] >= lim) {
                                uint32_t hits = ~signs_below(w + g * 8, lim) & 0xFFu;
                                do {
                                    const int j = __clz(hits) - 24;  // the first value is the highest bit
                                    hits &= ~(0x80u >> j);
                                    const uint32_t *x = w + g * 8;
                                    const uint32_t x01 = j & 1 ? x[1] : x[0], x23 = j & 1 ? x[3] : x[2];
                                    const uint32_t x45 = j & 1 ? x[5] : x[4], x67 = j & 1 ? x[7] : x[6];
                                    const uint32_t xl = j & 2 ? x23 : x01, xh = j & 2 ? x67 : x45;
                                    if (at < FCAP)
                                        list[at++] = make_uint2((j & 4 ? xh : xl) ^ 0x80000000u,
                                                                id0 + ((uint32_t)(g * 8 + j) << a.shift));
                                    else
                                        over = true;
                                } while (hits);
                            }
                        }
                        if (over) lim = __int_as_float(0x7F800000);  // these query rows are scanned instead
                    }
                }
                ++nb;
            }
            a.counts[sub] = at;
            if (over) a.over[block] = 1;
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (tid == 0 && *gave_up) atomicExch(a.err, 2);
    if (warp == 2)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

// ---------------------------------------------------------------- segments
// Segment 0 holds base rows 0, 2^levels, 2 * 2^levels, ...; segment s > 0 the
// rows halfway between those seen by then: 2^(levels - s) and on by twice that.
__host__ __device__ inline int segment_shift(int levels, int s) { return s == 0 ? levels : levels - s + 1; }
__host__ __device__ inline int64_t segment_first(int levels, int s) { return s == 0 ? 0 : int64_t(1) << (levels - s); }
__host__ __device__ inline int64_t segment_count(int64_t n, int levels, int s) {
    const int64_t step = int64_t(1) << segment_shift(levels, s);
    return (n - segment_first(levels, s) + step - 1) / step;
}
// The first bias row of segment s: each is padded to whole tiles.
__host__ __device__ inline int64_t segment_row0(int64_t n, int levels, int s) {
    int64_t at = 0;
    for (int i = 0; i < s; ++i) at += (segment_count(n, levels, i) + FN - 1) / FN * FN;
    return at;
}

// ---------------------------------------------------------------- rows
// Norms of the base rows in order (as the scan kernel wants them: zeros up to
// n_pad), the bias rows (-|x|^2 / 2, or 0; none if bias is null) in segment
// order, and the largest norm (its bits).
__global__ void knn_base_rows(const __nv_bfloat16 *__restrict__ x, int64_t n, int64_t n_pad, int d, int levels, bool l2,
                              float *__restrict__ norms, unsigned char *__restrict__ bias,
                              unsigned *__restrict__ top) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    float nrm = 0.f;
    if (i < n) {
        nrm = bf16_norm(x + i * d, d);
        // segment 0: the multiples of 2^levels; segment s > 0: the odd multiples of 2^(levels - s)
        const int low = i == 0 ? levels : min(levels, __ffsll(i) - 1);
        const int64_t at = low == levels ? i >> levels
                                         : segment_row0(n, levels, levels - low) + (i >> (low + 1));
        if (bias) {
            const float b = l2 ? -0.5f * nrm : 0.f;
            const __nv_bfloat16 h = __float2bfloat16_rn(b);
            const float r = b - __bfloat162float(h);
            const __nv_bfloat16 m = __float2bfloat16_rn(r);
            const __nv_bfloat16 l = __float2bfloat16_rn(r - __bfloat162float(m));
            const uint4 part = make_uint4((uint32_t)__bfloat16_as_ushort(h) | (uint32_t)__bfloat16_as_ushort(m) << 16,
                                          (uint32_t)__bfloat16_as_ushort(l), 0u, 0u);
            *reinterpret_cast<uint4 *>(bias + at / FN * (FN * kBiasRow) + at % FN * 16) = part;
        }
    }
    if (i < n_pad) norms[i] = nrm;
    unsigned m = __float_as_uint(nrm);  // not finite: above every finite value
    m = __reduce_max_sync(0xFFFFFFFFu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(top, m);
}

// By how much a bound on F = |x|^2 / 2 - <q, x> (or -<q, x>) is widened, so
// that every row is kept whose exact key is among the k smallest. With u =
// 2^-22, a product sum of d elements in FP32 is off by at most (d + 16) u |q| |x|
// in any order and with truncated sums, F by at most (d + 32) u (|q| |x| + |x|^2 / 2);
// keys take two more sums, 8 units in the last place of (|q| + |x|)^2. That
// holds down to the smallest normal number, 2^-126; below it a product, a sum or
// a part of the bias (BF16 ends at 2^-133) can lose up to 2^-126 each, 2 d + 64
// of them at most. The k-th F, the k-th key and the key at hand can each be off:
// three times. Vectors so short that this second part decides (|x| below 1e-15)
// all meet the bound, and their blocks are scanned.
__device__ __forceinline__ float knn_row_margin(float qn, float top, int d) {
    const float q = sqrtf(qn), x = sqrtf(top);
    return 3.f * ((d + 32) * 2.4e-7f * (2.f * q * x + x * x) + 8.f * 1.2e-7f * (q + x) * (q + x) + (d + 32) * 0x1p-125f);
}

// Per query row of a chunk (padded to whole blocks): its norm, margin, first
// bound, and no values kept. A row whose values could pass 1e30, or are not
// finite, meets no bound and has its block scanned.
__global__ void knn_query_rows(const __nv_bfloat16 *__restrict__ q, int64_t nq, int rows, int d,
                               const unsigned *__restrict__ top, float *__restrict__ qnorm, float *__restrict__ margin,
                               float *__restrict__ thr, int32_t *__restrict__ kept_n, int *__restrict__ over) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= rows) return;
    const float qn = r < nq ? bf16_norm(q + (size_t)r * d, d) : 0.f;
    const float e = knn_row_margin(qn, __uint_as_float(*top), d);  // at least 2.9e-6 (|q| + |x|)^2
    const bool fine = r < nq && e < 1e24f;
    qnorm[r] = qn;
    margin[r] = e;
    thr[r] = fine ? kOpen : -__int_as_float(0x7F800000);
    kept_n[r] = 0;
    if (r < nq && !fine) over[r / KBM] = 1;
}

// The smallest of n values (b[0..n).x) such that at least kk of them are
// below or equal, or a bound little above it: bisection of the values' range,
// ended early when no more than kk + 3 values meet it. n <= 32 PER.
template <int PER>
__device__ __forceinline__ float knn_kth_bound(const uint2 *b, int n, int kk, int lane) {
    const float inf = __int_as_float(0x7F800000);
    float f[PER];
    float lo = inf, hi = -inf;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const bool in = i * 32 + lane < n;
        f[i] = in ? __uint_as_float(b[i * 32 + lane].x) : inf;
        lo = fminf(lo, f[i]);
        if (in) hi = fmaxf(hi, f[i]);
    }
    for (int off = 16; off > 0; off >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xFFFFFFFFu, lo, off));
        hi = fmaxf(hi, __shfl_xor_sync(0xFFFFFFFFu, hi, off));
    }
    for (int it = 0; it < 24; ++it) {  // at least kk values are <= hi throughout
        const float mid = 0.5f * lo + 0.5f * hi;
        if (!(mid > lo && mid < hi)) break;
        int c = 0;
#pragma unroll
        for (int i = 0; i < PER; ++i) c += f[i] <= mid;
        c = __reduce_add_sync(0xFFFFFFFFu, c);
        if (c >= kk) {
            hi = mid;
            if (c <= kk + 3) break;
        } else {
            lo = mid;
        }
    }
    return hi;
}

// One warp per query row: the next bound from the values kept and those
// appended by the last segment (about 2 k of them), widened by the row's
// margin; the values within it are kept. Bound by its instructions, some 800 a
// row: 43 us for 58,000 rows. The counts of the row's lists are
// read at once, one lane each, so that all lists are copied without waiting
// for one another.
__global__ void __launch_bounds__(256) knn_tighten_kernel(const uint2 *__restrict__ lists,
                                                          const int32_t *__restrict__ counts, int subs, int used,
                                                          int rows, int kk, const float *__restrict__ margin,
                                                          float *__restrict__ thr, uint2 *__restrict__ kept,
                                                          int32_t *__restrict__ kept_n, int *__restrict__ over) {
    __shared__ uint2 buf[8][FMERGE];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row = blockIdx.x * 8 + warp;
    if (row >= rows) return;
    uint2 *b = buf[warp];
    uint2 *keep = kept + (size_t)row * FKEEP;
    const int had = kept_n[row];
    const float last = thr[row], wide = margin[row];
    for (int i = lane; i < had; i += 32) b[i] = keep[i];
    int n = had;
    for (int s0 = 0; s0 < used; s0 += 32) {
        // (after a wait that ran out, counts and lists may hold anything: nothing here goes by the values of a list)
        const int c = s0 + lane < used ? min(max(counts[(size_t)row * subs + s0 + lane], 0), FCAP) : 0;
        int end = c;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, end, off);
            if (lane >= off) end += y;
        }
        const int total = __shfl_sync(0xFFFFFFFFu, end, 31);
        const uint2 *src = lists + ((size_t)row * subs + s0) * FCAP;
#pragma unroll 4
        for (int i0 = 0; i0 < total; i0 += 32) {
            const int i = i0 + lane;
            int s = 0;  // the list that holds value i: the lists that end at or before it
#pragma unroll
            for (int step = 16; step > 0; step >>= 1) {
                const int e = __shfl_sync(0xFFFFFFFFu, end, min(s + step - 1, 31));
                if (e <= i) s += step;
            }
            const int first = __shfl_sync(0xFFFFFFFFu, end - c, s & 31);
            if (i < total && n + i < FMERGE) b[n + i] = src[s * FCAP + i - first];
        }
        n += total;
    }
    const bool full = n > FMERGE;
    n = min(n, FMERGE);
    __syncwarp();
    float bound = kOpen;
    if (n >= kk)
        bound = wide + (n <= 160 ? knn_kth_bound<5>(b, n, kk, lane) : knn_kth_bound<FMERGE / 32>(b, n, kk, lane));
    int out = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
        const int i = i0 + lane;
        const uint2 e = i < n ? b[i] : make_uint2(0u, 0u);
        const bool take = i < n && __uint_as_float(e.x) <= bound;
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, take);
        const int at = out + __popc(bal & ((1u << lane) - 1u));
        if (take && at < FKEEP) keep[at] = e;
        out += __popc(bal);
    }
    if (lane == 0) {
        // No more values of a row that is the scan's: where the norms are far above the distances all of them would
        // pass, in every segment (20,000 x 96 rows at an offset of 30: 4.67 ms; with none 3.33, the scan alone 2.86)
        const bool lost = full || out > FKEEP;
        kept_n[row] = lost ? 0 : out;
        if (last > -kOpen) thr[row] = lost ? -__int_as_float(0x7F800000) : bound;
        if (lost) over[row / KBM] = 1;
    }
}

// Writes the first k of c distinct keys in ascending order: each lane ranks
// up to U of them against all (two a load). KMAX is left out.
template <int U>
__device__ __forceinline__ void knn_rank(const unsigned long long *keys, int c, int lane, int k, int32_t *out_ids,
                                         float *out_d) {
    unsigned long long x[U];
    int rank[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        x[u] = u * 32 + lane < c ? keys[u * 32 + lane] : KMAX;
        rank[u] = 0;
    }
    for (int j = 0; j < c; j += 2) {
        const ulonglong2 y = *reinterpret_cast<const ulonglong2 *>(keys + j);
#pragma unroll
        for (int u = 0; u < U; ++u) rank[u] += (y.x < x[u]) + (y.y < x[u]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (x[u] != KMAX && rank[u] < k) {
            out_ids[rank[u]] = (int32_t)(uint32_t)x[u];
            out_d[rank[u]] = ord_dec((uint32_t)(x[u] >> 32));
        }
}

// One warp per query row: the exact keys of the rows kept, ranked. Sixteen
// rows at a time are multiplied with the query as the scan kernel does: the
// query in the first row of A, the same order of K, so a key has the same bits
// wherever it is computed. It gathers about 66 rows a query and is bound by
// their latency, so every lane loads its part of B straight from the rows (all
// of 16 rows in flight) and no shared memory but the keys limits the warps:
// 229 us for 58,000 queries of 96 elements, 239 us with the rows staged in
// shared memory.
template <int KS, bool L2>
__global__ void __launch_bounds__(256)
    knn_finish_kernel(const __nv_bfloat16 *__restrict__ base, const float *__restrict__ bnorm,
                      const __nv_bfloat16 *__restrict__ queries, const float *__restrict__ qnorm, int64_t nq,
                      int64_t self0, int k, const uint2 *__restrict__ kept, const int32_t *__restrict__ kept_n,
                      int32_t *__restrict__ out_ids, float *__restrict__ out_d, const int *__restrict__ err) {
    constexpr int D = KS * 16;
    __shared__ __align__(16) unsigned long long key_buf[8][FKEEP];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t row = (int64_t)blockIdx.x * 8 + warp;
    if (row >= nq) return;
    unsigned long long *keys = key_buf[warp];
    const int c = *err ? 0 : kept_n[row];  // after a wait that ran out the ids kept may be anything
    const int g = lane >> 2, t = lane & 3;
    uint32_t a[KS][4];
    const uint32_t *q = reinterpret_cast<const uint32_t *>(queries + row * D);
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
        a[ks][0] = g == 0 ? q[ks * 8 + t] : 0u;
        a[ks][2] = g == 0 ? q[ks * 8 + 4 + t] : 0u;
        a[ks][1] = a[ks][3] = 0u;
    }
    const float qn = qnorm[row];
    const int64_t self = self0 >= 0 ? self0 + row : -1;
    const uint2 *mine = kept + (size_t)row * FKEEP;
    bool mine_self = false;  // this lane met the query's own row
    for (int i0 = 0; i0 < c; i0 += 16) {
        // rows i0 + g and i0 + 8 + g (of B, column g of either product); past the end: the query's first row kept
        uint32_t b[2][KS][2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = i0 + h * 8 + g;
            const uint32_t *x = reinterpret_cast<const uint32_t *>(base + (size_t)mine[i < c ? i : 0].y * D);
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
                b[h][ks][0] = __ldg(x + ks * 8 + t);
                b[h][ks][1] = __ldg(x + ks * 8 + 4 + t);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float acc[4] = {};
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) mma_bf16_16816(acc, a[ks], b[h][ks][0], b[h][ks][1]);
            if (g == 0) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int i = i0 + h * 8 + 2 * t + e;
                    if (i < c) {
                        const uint32_t id = mine[i].y;
                        const float dist = knn_dist<L2>(acc[e], L2 ? bnorm[id] : 0.f, qn);
                        mine_self |= (int64_t)id == self;
                        keys[i] = (int64_t)id == self ? KMAX : ((unsigned long long)ord_enc(dist) << 32) | id;
                    }
                }
            }
        }
    }
    if (lane == 0 && (c & 1)) keys[c] = KMAX;  // the ranking reads two at a time
    __syncwarp();
    // rank = entries below (keys are distinct: every base row is kept once); the query's own row ranks last
    const int have = c - __popc(__ballot_sync(0xFFFFFFFFu, mine_self));
    if (c <= 96)
        knn_rank<3>(keys, c, lane, k, out_ids + (size_t)row * k, out_d + (size_t)row * k);
    else
        knn_rank<FKEEP / 32>(keys, c, lane, k, out_ids + (size_t)row * k, out_d + (size_t)row * k);
    for (int i = have + lane; i < k; i += 32) {
        out_ids[(size_t)row * k + i] = -1;
        out_d[(size_t)row * k + i] = __int_as_float(0x7F800000);
    }
}

// ---------------------------------------------------------------- host
typedef CUresult (*EncodeTiled)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

cudaError_t encode_rows_map(RowMaps *maps, const void *rows, int64_t count, int64_t pitch, int d, int box_rows) {
    static std::atomic<void *> entry{nullptr};  // the driver's function, the same for every thread and device
    void *fn = entry.load(std::memory_order_acquire);
    if (!fn) {
        cudaDriverEntryPointQueryResult found;
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found);
        if (e != cudaSuccess) return e;
        if (found != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
        entry.store(fn, std::memory_order_release);
    }
    for (int wide = 0; wide < 2; ++wide) {
        if (wide && d < 64) continue;  // no 64-element piece to load
        const cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)count};
        const cuuint64_t strides[1] = {(cuuint64_t)pitch};
        const cuuint32_t box[2] = {wide ? 64u : 32u, (cuuint32_t)box_rows}, steps[2] = {1, 1};
        const CUresult r = reinterpret_cast<EncodeTiled>(fn)(
            wide ? &maps->wide : &maps->narrow, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(rows), dims,
            strides, box, steps, CU_TENSOR_MAP_INTERLEAVE_NONE,
            wide ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    }
    return cudaSuccess;
}

template <int KD>
cudaError_t launch_filter(const RowMaps &q, const RowMaps &x, const FilterArgs &a, int grid, cudaStream_t s) {
    cudaError_t e = ensure_dyn_smem(reinterpret_cast<const void *>(knn_filter_kernel<KD>), filter_smem(KD));
    if (e != cudaSuccess) return e;
    knn_filter_kernel<KD><<<grid, FTHREADS, filter_smem(KD), s>>>(q, x, a);
    return cudaGetLastError();
}

template <int KS, bool L2>
cudaError_t launch_finish(const void *base, const float *norms, const void *q, const float *qnorm, int64_t nq,
                          int64_t self0, int k, const uint2 *kept, const int32_t *kept_n, int32_t *ids, float *dists,
                          const int *err, cudaStream_t s) {
    knn_finish_kernel<KS, L2><<<(unsigned)((nq + 7) / 8), 256, 0, s>>>(
        reinterpret_cast<const __nv_bfloat16 *>(base), norms, reinterpret_cast<const __nv_bfloat16 *>(q), qnorm, nq,
        self0, k, kept, kept_n, ids, dists, err);
    return cudaGetLastError();
}

}  // namespace

size_t knn_scan_bytes(int64_t n) { return 256 + (size_t)knn_norms_rows(n) * 4; }

cudaError_t launch_knn_scan_all(void *ws, const void *base, int64_t n, int d, const void *queries, int64_t nq,
                                int64_t self0, int metric, int k, int32_t *ids, float *dists, cudaStream_t s) {
    unsigned char *w = static_cast<unsigned char *>(ws);
    float *norms = reinterpret_cast<float *>(w + 256);
    const int64_t np = knn_norms_rows(n);
    cudaError_t e = cudaMemsetAsync(w, 0, 256, s);
    if (e != cudaSuccess) return e;
    knn_base_rows<<<(unsigned)((np + 255) / 256), 256, 0, s>>>(reinterpret_cast<const __nv_bfloat16 *>(base), n, np, d, 0,
                                                               metric == ANN_METRIC_L2, norms, nullptr,
                                                               reinterpret_cast<unsigned *>(w + 4));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return launch_knn_scan(base, n, d, queries, nq, self0, metric, k, ids, dists, norms, nullptr,
                           reinterpret_cast<int *>(w), s);
}

// The filter costs a few launches more than the scan, and an allocation of over 2 MB (640 queries) 125 us. Scan and
// filter, us, 128-d rows, k = 64 (32-d rows): one query of 64 rows 47 / 62 (38 / 58), of 257 rows 83 / 81 (60 / 76), of
// 512 rows 93 / 84 (73 / 78), 16 queries of 64 rows 50 / 70 (47 / 58), of 257 rows 96 / 87 (74 / 79), 32 of 64 rows
// 61 / 70 (50 / 58); 1,000 queries of 64 rows 96 / 183, of 257 rows 219 / 208, 4,000 of 257 rows 224 / 240, of 400 rows
// 261 / 253; 512 queries of 64 rows 96 / 71.
bool knn_scan_is_faster(int64_t n, int64_t nq) {
    return n <= 128 ? nq <= 16 || nq > 640 : n <= 320 && (nq <= 4 || nq > 640);
}

KnnPlan knn_plan(int64_t n, int64_t nq, int sms) {
    KnnPlan p;
    p.no_loads = 0;
    p.levels = 0;
    while ((n + (int64_t(1) << p.levels) - 1) >> p.levels > FN) ++p.levels;
    // three rounds of 128 query rows per SM in a chunk: a segment's launch is long enough to fill the chip
    const int64_t blocks = (nq + KBM - 1) / KBM;
    p.chunk_blocks = (int)std::min<int64_t>(blocks, 3 * (int64_t)sms);
    // fewer blocks than SMs could share evenly: several CTAs take every splits-th tile of one block. chunk_blocks x splits
    // stays below six rounds of SMs, so a chunk's lists (2 KB a query and split) below 241 MB on 152 SMs. At least four
    // tiles of the last segment, half of the base, for each: with 32 CTAs whatever the base, 1,000 rows against themselves
    // took 69 MB and 383 us (now 3 MB and 256 us), and 512 such 347 us (now 116: its workspace stays below the 2 MB from
    // which on an allocation costs 125 us)
    const int64_t tiles = (segment_count(n, p.levels, p.levels) + FN - 1) / FN;
    p.splits = 1;
    while (p.splits < 32 && p.chunk_blocks * p.splits < 3 * sms) p.splits *= 2;
    p.splits = (int)std::min<int64_t>(p.splits, (tiles + 3) / 4);
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o += (bytes + 255) / 256 * 256;
        return at;
    };
    const size_t rows = (size_t)p.chunk_blocks * KBM;
    p.err = take(256);  // [0] error, [1] the largest norm's bits
    p.norms = take((size_t)knn_norms_rows(n) * 4);
    p.bias = take((size_t)segment_row0(n, p.levels, p.levels + 1) * kBiasRow);
    p.over = take((size_t)p.chunk_blocks * 4);
    p.qnorm = take(rows * 4);
    p.margin = take(rows * 4);
    p.thr = take(rows * 4);
    p.kept_n = take(rows * 4);
    p.counts = take(rows * (FEPI / 4) * p.splits * 4);
    p.kept = take(rows * FKEEP * 8);
    p.lists = take(rows * (FEPI / 4) * p.splits * FCAP * 8);
    p.bytes = o;
    return p;
}

cudaError_t launch_knn_bf16(const KnnPlan &p, void *ws, const void *base, int64_t n, int d, const void *queries,
                            int64_t nq, int64_t self0, int metric, int k, int32_t *ids, float *dists, int sms,
                            cudaStream_t s) {
    const bool l2 = metric == ANN_METRIC_L2;
    unsigned char *w = static_cast<unsigned char *>(ws);
    int *err = reinterpret_cast<int *>(w + p.err);
    unsigned *top = reinterpret_cast<unsigned *>(w + p.err + 4);
    float *norms = reinterpret_cast<float *>(w + p.norms);
    unsigned char *bias = w + p.bias;
    int *over = reinterpret_cast<int *>(w + p.over);
    float *qnorm = reinterpret_cast<float *>(w + p.qnorm), *margin = reinterpret_cast<float *>(w + p.margin);
    float *thr = reinterpret_cast<float *>(w + p.thr);
    int32_t *kept_n = reinterpret_cast<int32_t *>(w + p.kept_n), *counts = reinterpret_cast<int32_t *>(w + p.counts);
    uint2 *kept = reinterpret_cast<uint2 *>(w + p.kept), *lists = reinterpret_cast<uint2 *>(w + p.lists);
    const int64_t bias_rows = segment_row0(n, p.levels, p.levels + 1), np = knn_norms_rows(n);
    cudaError_t e;
    if ((e = cudaMemsetAsync(w + p.err, 0, 256, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(bias, kPadByte, (size_t)bias_rows * kBiasRow, s)) != cudaSuccess) return e;
    knn_base_rows<<<(unsigned)((np + 255) / 256), 256, 0, s>>>(reinterpret_cast<const __nv_bfloat16 *>(base), n, np, d,
                                                               p.levels, l2, norms, bias, top);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int segs = p.levels + 1;
    RowMaps map_x[FSEG] = {};
    for (int i = 0; i < segs; ++i) {
        const int64_t first = segment_first(p.levels, i), count = segment_count(n, p.levels, i);
        const int64_t pitch = (int64_t)d * 2 << segment_shift(p.levels, i);
        e = encode_rows_map(&map_x[i], static_cast<const char *>(base) + first * d * 2, count, pitch, d, FN);
        if (e != cudaSuccess) return e;
    }
    for (int64_t r0 = 0; r0 < nq; r0 += (int64_t)p.chunk_blocks * KBM) {
        const int64_t cq = std::min<int64_t>(nq - r0, (int64_t)p.chunk_blocks * KBM);
        const int blocks = (int)((cq + KBM - 1) / KBM), rows = blocks * KBM;
        const char *q = static_cast<const char *>(queries) + r0 * d * 2;
        const int64_t cself = self0 >= 0 ? self0 + r0 : -1;
        RowMaps map_q = {};
        if ((e = encode_rows_map(&map_q, q, cq, (int64_t)d * 2, d, KBM)) != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(over, 0, (size_t)blocks * 4, s)) != cudaSuccess) return e;
        knn_query_rows<<<(rows + 255) / 256, 256, 0, s>>>(reinterpret_cast<const __nv_bfloat16 *>(q), cq, rows, d, top,
                                                          qnorm, margin, thr, kept_n, over);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        for (int i = 0; i < segs; ++i) {
            FilterArgs a = {};
            a.first = (uint32_t)segment_first(p.levels, i);
            a.shift = segment_shift(p.levels, i);
            a.bias = bias + segment_row0(n, p.levels, i) * kBiasRow;
            a.thr = thr;
            a.lists = lists;
            a.counts = counts;
            a.over = over;
            a.err = err;
            a.no_loads = p.no_loads;
            a.subs = FEPI / 4 * p.splits;
            a.tiles = (int)((segment_count(n, p.levels, i) + FN - 1) / FN);
            a.blocks = blocks;
            a.splits = std::min(p.splits, a.tiles);
            const int grid = (int)std::min<int64_t>((int64_t)blocks * a.splits, sms);
            switch (d / 32) {
                case 1: e = launch_filter<1>(map_q, map_x[i], a, grid, s); break;
                case 2: e = launch_filter<2>(map_q, map_x[i], a, grid, s); break;
                case 3: e = launch_filter<3>(map_q, map_x[i], a, grid, s); break;
                case 4: e = launch_filter<4>(map_q, map_x[i], a, grid, s); break;
                default: return cudaErrorInvalidValue;
            }
            if (e != cudaSuccess) return e;
            knn_tighten_kernel<<<(rows + 7) / 8, 256, 0, s>>>(lists, counts, a.subs, FEPI / 4 * a.splits, rows,
                                                              k + (self0 >= 0 ? 1 : 0), margin, thr, kept, kept_n,
                                                              over);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        int32_t *oi = ids + r0 * k;
        float *od = dists + r0 * k;
#define ANN_KNN_FINISH(KS)                                                                                     \
    case KS:                                                                                                   \
        e = l2 ? launch_finish<KS, true>(base, norms, q, qnorm, cq, cself, k, kept, kept_n, oi, od, err, s)    \
               : launch_finish<KS, false>(base, norms, q, qnorm, cq, cself, k, kept, kept_n, oi, od, err, s);  \
        break;
        switch (d / 16) {
            ANN_KNN_FINISH(2)
            ANN_KNN_FINISH(4)
            ANN_KNN_FINISH(6)
            ANN_KNN_FINISH(8)
            default: return cudaErrorInvalidValue;
        }
#undef ANN_KNN_FINISH
        if (e != cudaSuccess) return e;
        // the blocks whose lists ran over
        if ((e = launch_knn_scan(base, n, d, q, cq, cself, metric, k, oi, od, norms, over, err, s)) != cudaSuccess)
            return e;
    }
    return cudaSuccess;
}

}  // namespace ann
