// Device helpers shared by the warp-specialised TMA kernels: mbarrier
// operations, bounded waits, bulk copies into shared memory, and the warp's
// realigning copy of a compacted segment to global memory.
#pragma once

#include "ka_dev.cuh"

namespace ka {
namespace tma {

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return uint32_t(__cvta_generic_to_shared(p)); }

// 32-bit store to a shared-memory address (a cvta-to-shared address).
__device__ __forceinline__ void st_shared_u32(uint32_t addr, uint32_t v) {
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t *m, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(m)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *m) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(m)) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *m, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(m)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *m, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_addr(m)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Non-blocking test of the same (try_wait may suspend the thread for a while
// when the phase is not complete; test_wait returns at once).
__device__ __forceinline__ bool mbar_test_wait(uint64_t *m, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_addr(m)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Waits until the phase of parity `parity` of m has completed. Gives up after
// kWaitNs of wall time and returns false.
constexpr uint64_t kWaitNs = 2000000000ull;
__device__ __forceinline__ bool mbar_wait(uint64_t *m, uint32_t parity) {
    if (mbar_try_wait(m, parity)) return true;
    const uint64_t t0 = global_ns();
    for (uint32_t i = 1;; ++i) {
        if (mbar_try_wait(m, parity)) return true;
        if ((i & 15u) == 0u && global_ns() - t0 > kWaitNs) return false;
    }
}

// Bulk copy global -> this block's shared memory, completing on mbarrier m.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *m) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(m))
                 : "memory");
}

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

constexpr int kSeg = 512;         // entries per compute warp and tile (32 lanes x 4 rows x 4)


// Keep mask of a lane's entries (entry c of row r: bit 4 r + c) and, above it, the kept entries of each row (row r: bits 16 + 4 r .. 19 + 4 r), both by
// one addition under the test's predicate: two instructions an entry for most
// kinds. (Bool values shifted into place cost three to four, and the counts
// four population counts more.)
template <int K, int ROWS>
__device__ __forceinline__ uint32_t tally(const PredDev &p, const uint32_t (&v)[ROWS][4]) {
    static_assert(ROWS <= 4, "16 mask bits and four counts");
    if constexpr (K == kAll) return 0x4444FFFFu & (0xFFFFu >> (16 - 4 * ROWS)) * 0x10001u;
    uint32_t t[4] = {0u, 0u, 0u, 0u};
    auto add = [&](auto keep) {
#pragma unroll
        for (int r = 0; r < ROWS; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t one = (1u << (4 * r + c)) | (1u << (16 + 4 * r));
                if constexpr (K == kPopcOdd)
                    // (in one piece: the low bit goes straight to a predicate)
                    asm("{\n .reg .pred q;\n .reg .b32 b;\n and.b32 b, %1, 1;\n setp.ne.u32 q, b, 0;\n"
                        " @q add.u32 %0, %0, %2;\n}"
                        : "+r"(t[r])
                        : "r"(uint32_t(__popc(v[r][c]))), "r"(one));
                else if (keep(v[r][c]))
                    t[r] += one;
            }
    };
    if (K == kModNe0 && p.s == 0u) add([&](uint32_t x) { return x * p.a > p.b; });  // odd divisors: no rotation
    else add([&](uint32_t x) { return keep_k<K>(p, x); });
    return (t[0] + t[1]) + (t[2] + t[3]);
}

// The tally for the set of tests MASK: the tests of an entry are one chain of
// predicates, and only the last makes a bit and a count.
template <int MASK, int ROWS>
__device__ __forceinline__ uint32_t set_tally(const PredSet &p, const uint32_t (&v)[ROWS][4]) {
    static_assert(ROWS <= 4, "16 mask bits and four counts");
    uint32_t t[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint32_t x = v[r][c];
            bool keep = true;
            if (MASK & kSetAnd) keep = keep && (x & p.and_mask) == 0u;
            if (MASK & kSetLt) keep = keep && x < p.lt;
            if (MASK & kSetNe) keep = keep && x != p.ne;
            if (MASK & kSetMod) keep = keep && rotr32(x * p.mod_a, p.mod_s) > p.mod_b;
            if (MASK & kSetPopc) keep = keep && (__popc(x) & 1u) != 0u;
            if (keep) t[r] += (1u << (4 * r + c)) | (1u << (16 + 4 * r));
        }
    return (t[0] + t[1]) + (t[2] + t[3]);
}

// The tally of a keep mask alone.
__device__ __forceinline__ uint32_t tally_of(uint32_t mask) {
    uint32_t t = mask;
#pragma unroll
    for (int r = 0; r < 4; ++r) t += uint32_t(__popc(mask & (0xFu << (4 * r)))) << (16 + 4 * r);
    return t;
}

// Applies a chain to a lane's entries: v becomes the last values; the tally of
// those that pass every test. The kind is switched on once per test for all
// of the lane's entries.
template <int ROWS>
__device__ __forceinline__ uint32_t chain_tally(const PredChain &ch, uint32_t (&v)[ROWS][4]) {
    // (unrolled: every parameter is then read at a fixed place, as an operand)
    uint32_t m = 0xFFFFu >> (16 - 4 * ROWS);
#pragma unroll
    for (uint32_t i = 0; i < kChainMax; ++i) {
        if (i >= ch.n) break;
        const PredDev &p = ch.op[i].pred;
        if (ch.op[i].mul != 1u) {
#pragma unroll
            for (int r = 0; r < ROWS; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) v[r][c] *= ch.op[i].mul;
        }
        switch (p.kind) {
        case kAndMaskEq0: m &= tally<kAndMaskEq0>(p, v); break;
        case kLt: m &= tally<kLt>(p, v); break;
        case kPopcOdd: m &= tally<kPopcOdd>(p, v); break;
        case kModNe0: m &= tally<kModNe0>(p, v); break;
        case kNe: m &= tally<kNe>(p, v); break;
        default: break;
        }
    }
    return tally_of(m);
}

// The tally cut to entries [vlo, vhi) of the segment.
__device__ __forceinline__ uint32_t cut_tally(uint32_t t, uint32_t vlo, uint32_t vhi, int lane) {
    uint32_t m = 0u;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const uint32_t e0 = uint32_t(r * 128 + lane * 4);
        const uint32_t skip = vlo > e0 ? min(vlo - e0, 4u) : 0u;
        const uint32_t left = vhi > e0 ? vhi - e0 : 0u;
        m |= (((0xFu << skip) & (left >= 4 ? 0xFu : ((1u << left) - 1u))) & 0xFu) << (4 * r);
    }
    return tally_of(t & m);
}

// Ranks of a lane's kept entries from its tally. The row counts, in 8-bit
// fields (a row of the warp keeps at most 128), are scanned across the warp:
// byte r of `excl` counts the kept entries of row r in the lanes before this
// one, byte r of `rows` those of the whole row; `total` is the segment's. The
// shuffle's own in-range predicate guards each addition.
struct Ranks {
    uint32_t excl, rows, total;
};
__device__ __forceinline__ Ranks rank_tally(uint32_t t) {
    uint32_t packed = ((t >> 16) * 0x101u) & 0x00FF00FFu;  // nibbles to bytes
    packed = (packed * 0x11u) & 0x0F0F0F0Fu;
    uint32_t incl = packed;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1)
        asm volatile(
            "{\n .reg .pred q;\n .reg .b32 t;\n shfl.sync.up.b32 t|q, %0, %1, 0, 0xffffffff;\n"
            " @q add.u32 %0, %0, t;\n}"
            : "+r"(incl)
            : "r"(d));
    Ranks k;
    k.excl = incl - packed;
    k.rows = __shfl_sync(kFull, incl, 31);
    k.total = __dp4a(k.rows, 0x01010101u, 0u);
    return k;
}

// One warp copies cnt compacted entries from shared memory (16-byte aligned)
// to dst (4-byte aligned): single entries up to dst's next 16-byte boundary,
// then 16-byte stores, each assembled from two aligned 16-byte shared loads,
// then the remaining single entries. cnt <= kSeg.
// The 16-byte loops are kept rolled: a lane makes at most 4 trips, and in a
// kernel with registers to spare the compiler unrolled them into predicated
// stores that issue even when switched off. Those cost the held write-out
// throughput (same array, same process: 273 -> 263 us at 50 % kept and 346
// -> 324 us at 99 % in the five-stage shape, 352 -> 338 us at 99 % in the
// four-stage one; the store instructions dropped from 578 K to 508 K).
__device__ __forceinline__ void warp_copy_out(const uint32_t *src, uint32_t *dst, uint32_t cnt, int lane) {
    const uint32_t to16 = uint32_t((16u - (reinterpret_cast<uintptr_t>(dst) & 15u)) & 15u) >> 2;
    const uint32_t head = to16 < cnt ? to16 : cnt;
    if (uint32_t(lane) < head) dst[lane] = src[lane];
    const uint32_t body = (cnt - head) >> 2;
    const uint4 *s4 = reinterpret_cast<const uint4 *>(src);
    uint4 *d4 = reinterpret_cast<uint4 *>(dst + head);
    // Output chunk i holds src[head + 4i .. head + 4i + 3]: the tail of source
    // chunk i and the front of chunk i + 1 (index <= 127 since cnt <= 512).
    switch (head) {
    case 0:
#pragma unroll 1
        for (uint32_t i = uint32_t(lane); i < body; i += 32) d4[i] = s4[i];
        break;
    case 1:
#pragma unroll 1
        for (uint32_t i = uint32_t(lane); i < body; i += 32) {
            const uint4 x = s4[i], y = s4[i + 1];
            d4[i] = make_uint4(x.y, x.z, x.w, y.x);
        }
        break;
    case 2:
#pragma unroll 1
        for (uint32_t i = uint32_t(lane); i < body; i += 32) {
            const uint4 x = s4[i], y = s4[i + 1];
            d4[i] = make_uint4(x.z, x.w, y.x, y.y);
        }
        break;
    default:
#pragma unroll 1
        for (uint32_t i = uint32_t(lane); i < body; i += 32) {
            const uint4 x = s4[i], y = s4[i + 1];
            d4[i] = make_uint4(x.w, y.x, y.y, y.z);
        }
        break;
    }
    const uint32_t t0 = head + 4 * body;
    if (uint32_t(lane) < cnt - t0) dst[t0 + lane] = src[t0 + lane];
}

// One warp writes cnt entries out of its ring (RW words, a power of two;
// the entries start at word q), one per lane: few enough that realigning them
// to 16 bytes would take more instructions than it saves.
template <uint32_t RW>
__device__ __forceinline__ void warp_ring_out(const uint32_t *ring, uint32_t q, uint32_t *dst, uint32_t cnt,
                                              int lane) {
#pragma unroll 1
    for (uint32_t i = uint32_t(lane); i < cnt; i += 32) dst[i] = ring[(q + i) & (RW - 1u)];
}

}  // namespace tma
}  // namespace ka
