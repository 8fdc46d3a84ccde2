#pragma once
// The warp-specialised TMA kernels: fused single-pass compaction
// (k_compact_tma) and single-pass exclusive scan (k_scan_tma), each one
// persistent kernel fed by bulk copies, whose compute warps never wait for one
// another.
//
// Layout of the work. The grid holds exactly the blocks that fit on the GPU at
// once (cooperative launch), G of them; block b owns tiles b, b + G, b + 2G, ...
// (iteration j of block b is tile t = j G + b). A tile is CWW segments of 512
// entries; compute warp w owns segment w of every tile. Tiles start on
// 16-byte boundaries: an input that starts 4, 8 or 12 bytes past one is read
// from that boundary, and the 1-3 entries before its start belong to no tile.
//
// Inside a block:
//   * a producer warp streams tiles into a ring of S shared-memory stages with
//     cp.async.bulk (completion on the stage's "full" mbarrier), and refills a
//     stage once every compute warp has released it ("empty");
//   * each compute warp counts (compaction) or scans (scan) its segment of
//     tile j and posts the result ("counted" mbarrier of tile j); the last
//     warp to post publishes the tile aggregate at once (an atomic on a shared
//     word tells it that it is last);
//   * one look-back warp resolves the tiles' exclusive prefixes in order,
//     anchored on the block's own previous tile: prefix(t) = prefix(t - G) +
//     agg(t - G) + the aggregates of the G - 1 tiles t - G + 1 .. t - 1, which
//     the other blocks publish as soon as they have counted. So no block waits
//     for another block's look-back, and a tile costs one batch of independent
//     loads. This is the decoupled look-back of Merrill & Garland (2016)
//     reorganised around a round-robin persistent grid.
//
// The look-back's loads queue behind the SM's own stream of bulk copies, so a
// round trip takes about as long as a tile's copy (1-2 us). The two kernels
// keep it off the copy stream's critical path in different ways:
//   * scan: every segment is written out whole, from its stage, LAG tiles
//     after it was scanned (the "prefix" mbarrier says its offset is ready),
//     and only then is the stage released. One round trip per tile.
//   * compaction: a block that keeps few entries moves them out of the stage
//     into a ring of kept entries per warp and releases the stage at once; one
//     that keeps many holds them in the stage until they are written out (see
//     tma_compact_pass). While the oldest pending tile keeps little, the
//     look-back resolves every tile counted so far (up to BMAX) in one round
//     trip; otherwise that tile alone, whose write-out waits for it.
// One lane per warp arrives on an mbarrier, after __syncwarp: 32 arrivals on
// one barrier word serialise. Every wait is bounded (a few seconds); on
// time-out the kernel records a device error and still finishes.
#include "ka_internal.h"
#include "ka_tma.cuh"

namespace ka {
namespace tma {

// What the scan needs, and no more: with the compaction's chain and set behind it
// as kernel parameters too, the scan of (512, 16) spilled registers and took 360
// us at N = 2^28 instead of 334.
struct TmaBase {
    const uint32_t *in;  // input rounded down to 16 bytes: entry i of the input is in[lead + i]
    uint32_t *out;
    const uint32_t *n_ptr;
    uint32_t *count;
    WsHeader *ws;
    uint64_t *status;
    uint32_t n;
    uint32_t status_cap;
    uint32_t mul;
    uint32_t lead;     // 0..3 entries before the input's first entry
    uint32_t out_vec;  // scan: out - lead is 16-byte aligned (output entries align with input entries)
    PredDev pred;
};

struct TmaArgs : TmaBase {
    // the chain kernels (PK == kChainKind): their tests, and for an
    // interleaved input its second array
    const uint32_t *in2;
    PredChain chain;
    PredSet set;  // the set kernels' tests
};

// Predicate kind of the kernels that run a chain of tests (TmaArgs::chain), and
// of those made for a set of tests (kSetKind + its mask).
constexpr int kChainKind = -1, kSetKind = 64;

// Kept entries of a segment up to which they are stored one by one.
constexpr uint32_t kFewKept = 20;
// Kept entries a pending tile up to which four, or two, are written out at a
// time.
constexpr uint32_t kGroup4 = 64, kGroup2 = 100;

// Offset of a tile's segments when its look-back gave up (no segment that
// keeps an entry can start there: counts are at most 2^32 - 1).
constexpr uint32_t kNoOffset = 0xFFFFFFFFu;

// Block set-up shared by both passes (thread 0): the live length, the spin
// limit and the launch epoch (one ticket per block; the last block resets).
// With INTER, n and *n_ptr count pairs: the input has twice as many entries.
template <bool INTER = false>
__device__ __forceinline__ void tma_block_setup(const TmaBase &a, uint32_t *s_n, uint32_t *s_spin,
                                                uint32_t *s_epoch) {
    uint32_t n = a.n;
    if (a.n_ptr) {
        const uint32_t d = *a.n_ptr;
        n = d < n ? d : n;
    }
    *s_n = INTER ? 2u * n : n;
    const uint32_t sl = a.ws->spin_limit;
    *s_spin = sl ? sl : kDefaultSpinLimit;
    uint32_t ep;
    bool last;
    take_ticket(a.ws, 0u, &ep, &last);
    *s_epoch = ep;
}

// The producer warp's loop of a scan block (lane 0 only): tiles b, b + G, ... of
// the full tiles into the S-stage ring; the ragged last tile is read by the compute
// warps. Waits (bounded) for its last copies before returning, so none lands
// after the block exits.
template <int S, int T>
__device__ __forceinline__ void tma_produce(const TmaBase &a, uint32_t *stage_mem, uint64_t *full_bar,
                                            uint64_t *empty_bar, uint32_t my_tiles, uint32_t full_tiles) {
    const uint32_t G = gridDim.x, b = blockIdx.x;
    uint32_t issued = 0;
    for (uint32_t jj = 0; jj < my_tiles; ++jj) {
        const uint32_t tile = b + jj * G;
        if (tile >= full_tiles) break;
        const int s = int(jj % S);
        if (jj >= uint32_t(S) && !mbar_wait(&empty_bar[s], ((jj / S) - 1u) & 1u)) {
            record_error(a.ws, kDevErrTimeout, tile);
            break;
        }
        // the status sector of this block's tile two ahead: in L2 before its
        // aggregate is stored and polled
        if (jj + 2 < my_tiles) prefetch_l2(status_at(a.status, uint64_t(tile) + 2u * G));
        fence_proxy_async();  // the compute warps' accesses to this stage precede the copy into it
        mbar_expect_tx(&full_bar[s], uint32_t(T) * 4u);
        // two copies of half a tile each, both completing on the stage's barrier
        static_assert(T % 8 == 0, "each half is whole 16-byte chunks");
        bulk_g2s(stage_mem + size_t(s) * T, a.in + size_t(tile) * T, uint32_t(T / 2) * 4u, &full_bar[s]);
        bulk_g2s(stage_mem + size_t(s) * T + T / 2, a.in + size_t(tile) * T + T / 2, uint32_t(T / 2) * 4u,
                 &full_bar[s]);
        issued = jj + 1;
    }
    for (uint32_t jj = issued > uint32_t(S) ? issued - S : 0u; jj < issued; ++jj)
        mbar_wait(&full_bar[jj % S], (jj / S) & 1u);
}

// A scan warp's segment of tile j in shared memory: waits for the copy, or
// reads the ragged last tile with plain loads (zeros outside the input).
// Entries [vlo, vhi) of the segment are input entries.
__device__ __forceinline__ void tma_segment_ready(const TmaBase &a, uint32_t *seg, uint64_t *full_bar_s,
                                                  uint32_t parity, bool full_tile, uint64_t base, uint32_t vlo,
                                                  uint32_t vhi, uint32_t tile, int lane) {
    if (full_tile) {
        if (!mbar_wait(full_bar_s, parity) && lane == 0) record_error(a.ws, kDevErrTimeout, tile);
    } else {
        const uint32_t *src = a.in + base;
        for (uint32_t e = uint32_t(lane); e < uint32_t(kSeg); e += 32)
            seg[e] = e >= vlo && e < vhi ? src[e] : 0u;
        __syncwarp();
    }
}

// ============================================================================ scan
// Exclusive prefix sum: CWW compute warps (tile = CWW * 512 entries), S
// stages, write-out LAG tiles after scanning, at most MAXG blocks.
template <int CWW, int S, int LAG, int MAXG>
__device__ __forceinline__ void tma_scan_pass(const TmaBase &a) {
    constexpr int T = CWW * kSeg, ROWS = 4;
    constexpr int K = (MAXG + 31) / 32;
    static_assert(LAG >= 1 && LAG < S && LAG <= 3, "a stage is written out before its refill; slots repeat every 4");
    static_assert(CWW <= 32, "the look-back warp holds one segment sum per lane");
    extern __shared__ __align__(128) uint32_t stage_mem[];
    __shared__ __align__(8) uint64_t full_bar[S], empty_bar[S], count_bar[4], prefix_bar[4];
    __shared__ uint32_t s_wcnt[4][CWW], s_woff[4][CWW], s_err[4];
    __shared__ uint32_t s_pack[4];  // per tile slot: segments scanned
    __shared__ uint32_t s_n, s_epoch, s_spin;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t G = gridDim.x, b = blockIdx.x;

    if (tid == 0) {
        tma_block_setup(a, &s_n, &s_spin, &s_epoch);
        for (int s = 0; s < S; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], CWW);
        }
        for (int k = 0; k < 4; ++k) {
            s_pack[k] = 0;
            mbar_init(&count_bar[k], CWW);
            mbar_init(&prefix_bar[k], 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const uint32_t n_in = s_n, n = n_in + a.lead;
    const uint32_t epoch = s_epoch, want = epoch & kEpochMask, spin = s_spin;
    const uint32_t live = uint32_t((uint64_t(n) + T - 1) / T);
    const uint32_t full_tiles = n / uint32_t(T);
    if (uint64_t(live) > a.status_cap) {
        if (tid == 0 && b == 0) record_error(a.ws, kDevErrWorkspace, 0);
        return;
    }
    if (n_in == 0) {
        if (tid == 0 && b == 0) *a.count = 0u;
        return;
    }
    const uint32_t my_tiles = live > b ? (live - b + G - 1) / G : 0u;
    uint64_t *agg_words = a.status;  // entry per tile

    if (warp == CWW + 1) {
        if (lane == 0) tma_produce<S, T>(a, stage_mem, full_bar, empty_bar, my_tiles, full_tiles);
        return;
    }

    if (warp == CWW) {
        // ---------------------------------------------------------------- look-back warp
        uint32_t incl_prev = 0;  // inclusive prefix of this block's previous tile
        bool broken = false;     // an earlier look-back of this block gave up
        for (uint32_t j = 0; j < my_tiles; ++j) {
            const uint32_t k = j & 3u, tile = b + j * G;
            bool failed = !mbar_wait(&count_bar[k], (j >> 2) & 1u);  // every segment of tile j scanned
            if (failed && lane == 0) record_error(a.ws, kDevErrTimeout, tile);
            const uint32_t wc = lane < CWW ? s_wcnt[k][lane] : 0u;
            const uint32_t wincl = warp_incl_scan(wc, lane);
            const uint32_t agg = __shfl_sync(kFull, wincl, 31);  // (published by the last warp to scan)
            const uint32_t lo = j == 0 ? 0u : tile - G + 1u;     // first tile of the window
            const uint32_t wn = tile - lo;                       // window length, < G
            uint32_t sum = 0, polls = 0, sleep_ns = 0;
            failed = failed || broken;
            while (!failed) {
                uint64_t raw[K];
#pragma unroll
                for (int kk = 0; kk < K; ++kk) {
                    const uint32_t i = uint32_t(lane) + 32u * kk;
                    raw[kk] = i < wn ? ld_relaxed_u64(status_at(agg_words, uint64_t(lo) + i)) : 0ull;
                }
                bool all = true;
                sum = 0;
#pragma unroll
                for (int kk = 0; kk < K; ++kk) {
                    const uint32_t i = uint32_t(lane) + 32u * kk;
                    if (i < wn) {
                        const uint32_t f =
                            uint32_t(raw[kk] >> 34) == want ? uint32_t(raw[kk] >> 32) & 3u : kFlagInvalid;
                        if (f == kFlagAggregate) sum += uint32_t(raw[kk]);
                        else all = false;
                    }
                }
                if (__all_sync(kFull, all)) break;
                if (++polls >= spin) {
                    failed = true;
                    if (lane == 0) record_error(a.ws, kDevErrTimeout, tile);
                    break;
                }
                if (polls > 2) {
                    __nanosleep(sleep_ns);
                    sleep_ns = sleep_ns < 128 ? sleep_ns * 2 + 32 : 128;
                }
            }
            const uint32_t prefix = incl_prev + warp_sum(sum);
            broken = failed;
            incl_prev = prefix + agg;
            if (lane < CWW) s_woff[k][lane] = prefix + wincl - wc;
            if (lane == 0) {
                if (!failed && tile == live - 1) *a.count = prefix + agg;
                s_err[k] = failed ? 1u : 0u;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&prefix_bar[k]);  // offsets of tile j ready
        }
        return;
    }

    // ---------------------------------------------------------------- compute warps
    // Iteration j: write out this warp's segment of tile j-LAG (every input
    // entry plus the segment's offset), whose offset the look-back warp has
    // had LAG iterations to resolve, and release its stage; then scan the
    // segment of tile j in place and post its sum.
    const int w = warp;
    uint32_t *const seg_base = stage_mem + w * kSeg;
    for (uint32_t j = 0; j < my_tiles + uint32_t(LAG); ++j) {
        if (j >= uint32_t(LAG)) {
            const uint32_t jp = j - uint32_t(LAG), k = jp & 3u;
            const int s = int(jp % S);
            const bool ok = mbar_wait(&prefix_bar[k], (jp >> 2) & 1u);
            if (!ok && lane == 0) record_error(a.ws, kDevErrTimeout, b + jp * G);
            const uint32_t off = s_woff[k][w];
            __syncwarp();
            if (ok && s_err[k] == 0u) {
                const uint64_t base = uint64_t(b + jp * G) * T + uint32_t(w) * kSeg;
                const uint32_t vlo = base < a.lead ? a.lead - uint32_t(base) : 0u;
                const uint32_t vhi = n > base ? uint32_t(min(n - base, uint64_t(kSeg))) : 0u;
                const uint32_t *sg = seg_base + size_t(s) * T;
                uint32_t *dst = a.out - a.lead + base;  // entry i of the output is a.out[i]
#pragma unroll
                for (int r = 0; r < ROWS; ++r) {
                    const uint32_t e0 = uint32_t(r * 128 + lane * 4);
                    uint4 q = *reinterpret_cast<const uint4 *>(sg + e0);
                    q.x += off;
                    q.y += off;
                    q.z += off;
                    q.w += off;
                    if (a.out_vec && e0 >= vlo && e0 + 4 <= vhi) {
                        *reinterpret_cast<uint4 *>(dst + e0) = q;
                    } else {
                        if (e0 >= vlo && e0 < vhi) dst[e0] = q.x;
                        if (e0 + 1 >= vlo && e0 + 1 < vhi) dst[e0 + 1] = q.y;
                        if (e0 + 2 >= vlo && e0 + 2 < vhi) dst[e0 + 2] = q.z;
                        if (e0 + 3 >= vlo && e0 + 3 < vhi) dst[e0 + 3] = q.w;
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty_bar[s]);  // this warp is done with the stage
        }
        if (j < my_tiles) {
            const uint32_t tile = b + j * G, k = j & 3u;
            const int s = int(j % S);
            uint32_t *seg = seg_base + size_t(s) * T;
            // entries [vlo, vhi) of this segment are input entries (64-bit
            // position: the last tile's later segments can lie past 2^32 when
            // T does not divide 2^32)
            const uint64_t base = uint64_t(tile) * T + uint32_t(w) * kSeg;
            const uint32_t vlo = base < a.lead ? a.lead - uint32_t(base) : 0u;
            const uint32_t vhi = n > base ? uint32_t(min(n - base, uint64_t(kSeg))) : 0u;
            tma_segment_ready(a, seg, &full_bar[s], (j / S) & 1u, tile < full_tiles, base, vlo, vhi, tile, lane);
            uint32_t v[ROWS][4];
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const uint32_t e0 = uint32_t(r * 128 + lane * 4);
                const uint4 q = *reinterpret_cast<const uint4 *>(seg + e0);
                v[r][0] = q.x;
                v[r][1] = q.y;
                v[r][2] = q.z;
                v[r][3] = q.w;
                if (vlo != 0u || vhi != uint32_t(kSeg)) {
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (e0 + c < vlo || e0 + c >= vhi) v[r][c] = 0u;
                }
            }
            uint32_t rs[ROWS], incl[ROWS], rowbase = 0;
#pragma unroll
            for (int r = 0; r < ROWS; ++r) rs[r] = v[r][0] + v[r][1] + v[r][2] + v[r][3];
#pragma unroll
            for (int r = 0; r < ROWS; ++r) incl[r] = warp_incl_scan(rs[r], lane);
            // in place: every lane rewrites only the entries it read
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const uint32_t e0 = uint32_t(r * 128 + lane * 4);
                uint32_t x = rowbase + incl[r] - rs[r];
                uint4 o;
                o.x = x;
                x += v[r][0];
                o.y = x;
                x += v[r][1];
                o.z = x;
                x += v[r][2];
                o.w = x;
                *reinterpret_cast<uint4 *>(seg + e0) = o;
                rowbase += __shfl_sync(kFull, incl[r], 31);
            }
            if (lane == 0) {
                s_wcnt[k][w] = rowbase;
                // segment sums are full 32-bit values: the last warp adds them up
                __threadfence_block();
                if (atomicAdd(&s_pack[k], 1u) == uint32_t(CWW - 1)) {
                    __threadfence_block();
                    uint32_t agg = 0;
                    for (int q = 0; q < CWW; ++q) agg += s_wcnt[k][q];
                    s_pack[k] = 0;
                    st_relaxed_u64(status_at(agg_words, tile), pack_status(epoch, kFlagAggregate, agg));
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&count_bar[k]);
        }
    }
}

// ====================================================================== compaction
// Fused compaction with predicate kind PK (a PredKind, or kChainKind: the
// tests of a.chain, one after the other; or kSetKind + a mask: those of a.set
// at once): CWW compute warps (tile = CWW * 512
// entries), at most MAXG blocks, NS tile slots (counts, offsets, barriers), at
// most BMAX tiles resolved per round trip of the look-back.
//
// Shared memory holds SH tiles. A block uses them in one of two ways, chosen
// by what its first tile keeps:
//   * ring (at most kRingNum / kRingDen of the entries kept): SR stages, and
//     the other SH - SR tiles as one ring of kept entries per compute warp. A
//     warp moves the kept entries of its segment into its ring, releases the
//     stage at once, and writes tiles out when the ring or the tile slots run
//     out of room. So every stage is in flight or being counted, and the
//     look-back has many tiles of time. What bounds it is the compute warps'
//     instructions (250-340 a segment, 68 % of the issue slots), so tiles that
//     keep little are written out four or two at a time.
//   * hold (more kept): SH stages; a segment is compacted in place in its
//     stage and written out LAG tiles later, and SH - LAG stages are in
//     flight. What bounds it is HBM (0.98-1.01 of the copy rate). Above a
//     fifth kept it is the faster of the two (17 % kept: ring 211 us, hold
//     220 us; 25 %: 240 us and 216 us).
// Both are correct for any data. The general chain, whose switches are
// instructions too, holds from kRingNumChain / kRingDen.
//
// A block that holds goes over to rings (FOLLOW) when a tile in every lap of its
// stages says so, at a sixteenth less than the first choice: held, data that
// thins out waits for the look-back of every third tile. N = 2^28, 2 M entries
// at 50 % and the rest at 0 / 1 / 2 / 5 %, us: 209 / 210 / 214 / 216 held to the
// end, 165 / 168 / 172 / 179 so. (First tiles that keep little and a dense rest
// stay in rings: 251 us at 50 %, where holding from the start takes 242. Following
// the data in both directions cost every call: loops that are left and entered
// again came out 4 to 20 % slower.) The small shapes hold to the end: following
// cost them registers. Against a choice for every segment they lose 5 to 12 % on
// such data, and gain 5 to 15 % on uniform data.
//
// N = 2^28, shape (768, 16), s = 1 / 5 / 10 / 25 / 50 / 99 % kept, us: 163 /
// 174 / 187 / 216 / 241 / 310. Before, four stages of 26 segments, each held
// until its write-out unless every segment of the tile kept at most 16
// entries: 176 / 223 / 227 / 237 / 266 / 331 (one stage in flight).
//
// A segment's count is posted before its entries are stored: the other blocks
// wait for it. A warp waits for an older tile's offset only after it has
// posted every tile up to that one, so no two blocks wait for each other.
//
// INTER: the input is the interleave of two arrays of a.n entries (entry 2i is
// a.in[i], entry 2i + 1 is a.in2[i]; both 16-byte aligned, a.lead 0) that
// exists nowhere in memory: a stage holds half a tile of each array, warp w's
// segment is 256 entries of either half, and a held segment is compacted into
// its own 256 words of the first half, then of the second.
constexpr uint32_t kRingNum = 3, kRingNumChain = 2, kRingDen = 16;

// The producer warp's loop of a compaction block (lane 0 only): as
// tma_produce, for SR stages or SH, whichever the compute warps choose after
// the first tile (the first SR tiles go to the same stages either way), or, if
// FOLLOW, after a lap of SH stages (every stage then has had the same number of
// tiles, so the parities are the same for all).
template <int SR, int SH, int T, bool INTER, bool FOLLOW>
__device__ __forceinline__ void compact_produce(const TmaArgs &a, uint32_t *stage_mem, uint64_t *full_bar,
                                                uint64_t *empty_bar, uint64_t *mode_bar, const uint32_t *s_ring,
                                                uint64_t *lap_bar, const uint32_t *s_leave, uint32_t my_tiles,
                                                uint32_t full_tiles) {
    const uint32_t G = gridDim.x, b = blockIdx.x;
    uint32_t stages = SR, s = 0, lap = 0;  // tile jj goes to stage s, which has had lap tiles before
    uint32_t held = 0;                     // laps of SH stages
    bool hold = false;
    for (uint32_t jj = 0; jj < my_tiles; ++jj) {
        const uint32_t tile = b + jj * G;
        if (tile >= full_tiles) break;
        if (jj == uint32_t(SR)) {
            if (!mbar_wait(mode_bar, 0u)) {
                record_error(a.ws, kDevErrTimeout, tile);
                break;
            }
            if (*s_ring == 0u) {
                hold = true;
                stages = SH;
                s = SR;
                lap = 0;
            }
        }
        if (FOLLOW && hold && s == 0u) {
            // (about as long as the wait for stage 0 would take)
            if (!mbar_wait(lap_bar, (lap - 1u) & 1u)) {
                record_error(a.ws, kDevErrTimeout, tile);
                break;
            }
            if (*s_leave != 0u) {
                hold = false;
                stages = SR;
                held = lap;
            }
        }
        if (lap != 0u && !mbar_wait(&empty_bar[s], (lap - 1u) & 1u)) {
            record_error(a.ws, kDevErrTimeout, tile);
            break;
        }
        // the status sector of this block's tile two ahead: in L2 before its
        // aggregate is stored and polled (first touches by those went to
        // DRAM; 1 % faster at s = 1 %)
        if (jj + 2 < my_tiles) prefetch_l2(status_at(a.status, uint64_t(tile) + 2u * G));
        fence_proxy_async();  // the compute warps' accesses to this stage precede the copy into it
        mbar_expect_tx(&full_bar[s], uint32_t(T) * 4u);
        // two copies of half a tile each, both completing on the stage's
        // barrier (measured 0.5 % faster than one at 1 % and 50 % kept)
        static_assert(T % 8 == 0, "each half is whole 16-byte chunks");
        const uint32_t *const h0 = INTER ? a.in + size_t(tile) * (T / 2) : a.in + size_t(tile) * T;
        const uint32_t *const h1 = INTER ? a.in2 + size_t(tile) * (T / 2) : h0 + T / 2;
        bulk_g2s(stage_mem + size_t(s) * T, h0, uint32_t(T / 2) * 4u, &full_bar[s]);
        bulk_g2s(stage_mem + size_t(s) * T + T / 2, h1, uint32_t(T / 2) * 4u, &full_bar[s]);
        if (++s == stages) {
            s = 0;
            ++lap;
        }
    }
    // waits (bounded) for the last copy into each stage, so none lands after the block exits
    for (uint32_t q = 0; q < uint32_t(SH); ++q) {
        const uint32_t tiles = q < s ? lap + 1u : q < stages ? lap : held;
        if (tiles != 0u) mbar_wait(&full_bar[q], (tiles - 1u) & 1u);
    }
}

template <int PK, int CWW, int SR, int SH, int LAG, int MAXG, int NS, int BMAX, bool INTER = false>
__device__ __forceinline__ void tma_compact_pass(const TmaArgs &a) {
    constexpr int T = CWW * kSeg, ROWS = 4, HALF = kSeg / 2;
    constexpr uint32_t RW = uint32_t(SH - SR) * kSeg;  // words of a warp's ring
    constexpr int KB = (MAXG - 1 + 31) / 32;  // loads per lane for the G - 1 words before one tile
    constexpr bool FOLLOW = SR == 3 && SH == 5;  // the shape (768, 16)
    constexpr uint32_t RING_NUM = PK == kChainKind ? kRingNumChain : kRingNum;
    static_assert(NS >= 2 && (NS & (NS - 1)) == 0, "tile slots: a power of two");
    static_assert(SR >= 2 && SH > SR && (RW & (RW - 1)) == 0 && RW >= kSeg, "a ring: a power of two, one segment fits");
    static_assert(LAG >= 1 && LAG < SH && LAG < NS, "a held segment is written out before its stage is refilled");
    static_assert(BMAX >= 1 && BMAX <= NS, "a batch of tiles fits the tile slots");
    static_assert(CWW <= 32, "the look-back warp holds one segment count per lane");
    static_assert(CWW * kSeg < 65536, "a tile aggregate fits the 16 low bits of s_pack");
    static_assert(kSeg < 65536 && RW <= 65536, "count and ring word of a segment share a word");
    extern __shared__ __align__(128) uint32_t stage_mem[];
    __shared__ __align__(8) uint64_t full_bar[SH], empty_bar[SH], count_bar[NS], prefix_bar[NS], mode_bar;
    __shared__ uint32_t s_wcnt[NS][CWW];  // per tile slot: segment counts (low half; above: first ring word)
    __shared__ uint32_t s_woff[NS][CWW];  // per tile slot: segment offsets in the output
    __shared__ uint32_t s_pack[NS];  // per tile slot: (segments counted << 16) | kept so far
    __shared__ uint32_t s_n, s_epoch, s_spin, s_ring;
    // a block that holds: phase n - 1 of lap_bar: *s_leave says whether it goes
    // over to the rings after lap n; left_bar: every compute warp has
    __shared__ __align__(8) uint64_t lap_bar, left_bar;
    __shared__ uint32_t s_leave;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t G = gridDim.x, b = blockIdx.x;

    if (tid == 0) {
        allow_dependents();
        tma_block_setup<INTER>(a, &s_n, &s_spin, &s_epoch);
        for (int s = 0; s < SH; ++s) {
            mbar_init(&full_bar[s], 1);
            mbar_init(&empty_bar[s], CWW);
        }
        for (int k = 0; k < NS; ++k) {
            s_pack[k] = 0;
            mbar_init(&count_bar[k], CWW);
            mbar_init(&prefix_bar[k], 1);
        }
        mbar_init(&mode_bar, 1);
        s_ring = 0u;
        if (FOLLOW) {
            mbar_init(&lap_bar, 1);
            mbar_init(&left_bar, CWW);
            s_leave = 0u;
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const uint32_t n_in = s_n, n = n_in + a.lead;
    const uint32_t epoch = s_epoch, want = epoch & kEpochMask, spin = s_spin;
    const uint32_t live = uint32_t((uint64_t(n) + T - 1) / T);
    const uint32_t full_tiles = n / uint32_t(T);
    if (uint64_t(live) > a.status_cap) {
        if (tid == 0 && b == 0) record_error(a.ws, kDevErrWorkspace, 0);
        return;
    }
    if (n_in == 0) {
        if (tid == 0 && b == 0) *a.count = 0u;
        return;
    }
    const uint32_t my_tiles = live > b ? (live - b + G - 1) / G : 0u;
    uint64_t *const agg_words = a.status;  // entry per tile
    if (my_tiles == 0) return;

    if (warp == CWW + 1) {
        if (lane == 0)
            compact_produce<SR, SH, T, INTER, FOLLOW>(a, stage_mem, full_bar, empty_bar, &mode_bar, &s_ring, &lap_bar,
                                                      &s_leave, my_tiles, full_tiles);
        return;
    }

    if (warp == CWW) {
        // ---------------------------------------------------------------- look-back warp
        // Tiles r, r + 1, ... of this block (iterations) are resolved in
        // order. One round trip loads, for every tile counted so far (up to
        // BMAX), the words of the G - 1 tiles between it and this block's
        // previous tile (for r = 0: the tiles before it); word i is tile lo + i,
        // lo following this block's last resolved tile, and batch tile t sits
        // at i = e_t = (t + 1) G - c. The tiles whose words before them are
        // all published are resolved; the rest wait for the next trip.
        uint32_t r = 0, incl_prev = 0, polls = 0, sleep_ns = 0;
        bool broken = false;  // a wait of this block's look-back gave up: no later tile is resolved
        while (r < my_tiles) {
            const uint32_t k0 = r & uint32_t(NS - 1);
            if (!mbar_wait(&count_bar[k0], (r / NS) & 1u) && !broken) {
                if (lane == 0) record_error(a.ws, kDevErrTimeout, b + r * G);
                broken = true;
            }
            if (broken) {
                // releases the waiters on this tile (once it is counted, so
                // that the barriers' phases stay in step); its output is not
                // written
                if (lane < CWW) s_woff[k0][lane] = kNoOffset;
                __syncwarp();
                if (lane == 0) mbar_arrive(&prefix_bar[k0]);
                ++r;
                continue;
            }
            // Batching pays when the compute warps run ahead (a ring that
            // holds every tile slot's entries); when segments keep more, their
            // write-outs wait for this tile alone, and a batch would only
            // lengthen the trip.
            const uint32_t wc0 = lane < CWW ? s_wcnt[k0][lane] & 0xFFFFu : 0u;
            const bool held0 = __any_sync(kFull, wc0 > RW / uint32_t(NS - 1));
            uint32_t m = 1;
            while (!held0 && m < uint32_t(BMAX) && r + m < my_tiles &&
                   mbar_test_wait(&count_bar[(r + m) & uint32_t(NS - 1)], ((r + m) / NS) & 1u))
                ++m;
            const uint32_t lo = r == 0 ? 0u : b + (r - 1u) * G + 1u;
            const uint32_t c = r == 0 ? G - b : 1u;
            uint32_t bsum[BMAX], first_bad = 0xFFFFFFFFu;  // first word not yet published
#pragma unroll
            for (int t = 0; t < BMAX; ++t) bsum[t] = 0u;
            // per batch tile: this lane's segment offset within the tile, and
            // the tile aggregate; computed while the window's loads are in flight
            uint32_t wexcl[BMAX], wagg[BMAX];
            auto scan_counts = [&]() {
#pragma unroll
                for (int t = 0; t < BMAX; ++t) {
                    if (uint32_t(t) < m) {
                        const uint32_t k = (r + uint32_t(t)) & uint32_t(NS - 1);
                        const uint32_t wc = lane < CWW ? s_wcnt[k][lane] & 0xFFFFu : 0u;
                        const uint32_t wincl = warp_incl_scan(wc, lane);
                        wexcl[t] = wincl - wc;
                        wagg[t] = __shfl_sync(kFull, wincl, 31);
                    }
                }
            };
            if (m == 1) {
                // one tile pending (the look-back keeps up): its G - 1 words only
                const uint32_t end = G - c;
                uint64_t raw[KB];
#pragma unroll
                for (int kk = 0; kk < KB; ++kk) {
                    const uint32_t i = uint32_t(lane) + 32u * kk;
                    raw[kk] = i < end ? ld_relaxed_u64(status_at(agg_words, uint64_t(lo + i))) : 0ull;
                }
                scan_counts();
#pragma unroll
                for (int kk = 0; kk < KB; ++kk) {
                    const uint32_t i = uint32_t(lane) + 32u * kk;
                    if (i < end) {
                        if (uint32_t(raw[kk] >> 34) == want && (uint32_t(raw[kk] >> 32) & 3u) == kFlagAggregate)
                            bsum[0] += uint32_t(raw[kk]);
                        else
                            first_bad = i;
                    }
                }
                if (!__all_sync(kFull, first_bad == 0xFFFFFFFFu)) first_bad = 0u;
            } else {
                // several tiles counted: the words before each of them, all in one round trip
                uint64_t raw[BMAX][KB];
#pragma unroll
                for (int t = 0; t < BMAX; ++t) {
                    if (uint32_t(t) < m) {
                        const uint32_t start = t == 0 ? 0u : uint32_t(t) * G - c + 1u, end = uint32_t(t + 1) * G - c;
#pragma unroll
                        for (int kk = 0; kk < KB; ++kk) {
                            const uint32_t i = start + uint32_t(lane) + 32u * kk;
                            raw[t][kk] = i < end ? ld_relaxed_u64(status_at(agg_words, uint64_t(lo + i))) : 0ull;
                        }
                    }
                }
                scan_counts();
#pragma unroll
                for (int t = 0; t < BMAX; ++t) {
                    if (uint32_t(t) < m) {
                        const uint32_t start = t == 0 ? 0u : uint32_t(t) * G - c + 1u, end = uint32_t(t + 1) * G - c;
#pragma unroll
                        for (int kk = 0; kk < KB; ++kk) {
                            const uint32_t i = start + uint32_t(lane) + 32u * kk;
                            const uint64_t wv = raw[t][kk];
                            if (i < end) {
                                if (uint32_t(wv >> 34) == want && (uint32_t(wv >> 32) & 3u) == kFlagAggregate)
                                    bsum[t] += uint32_t(wv);
                                else
                                    first_bad = min(first_bad, i);
                            }
                        }
                    }
                }
                first_bad = __reduce_min_sync(kFull, first_bad);
            }
            uint32_t nres = 0;  // batch tile t is resolved when every word before it is published
            while (nres < m && (nres + 1u) * G - c <= first_bad) ++nres;
            if (nres == 0) {
                if (++polls >= spin) {
                    if (lane == 0) record_error(a.ws, kDevErrTimeout, b + r * G);
                    broken = true;
                } else if (polls > 2) {
                    __nanosleep(sleep_ns);
                    sleep_ns = sleep_ns < 128 ? sleep_ns * 2 + 32 : 128;
                }
                continue;
            }
            polls = 0;
            sleep_ns = 0;
            uint32_t before = incl_prev;  // inclusive prefix of the tile before batch tile t
#pragma unroll
            for (int t = 0; t < BMAX; ++t) {
                if (uint32_t(t) < nres) {
                    const uint32_t part = warp_sum(bsum[t]);
                    const uint32_t tt = r + uint32_t(t), k = tt & uint32_t(NS - 1);
                    const uint32_t prefix = before + part, agg = wagg[t];
                    before = prefix + agg;
                    if (lane < CWW) s_woff[k][lane] = prefix + wexcl[t];
                    if (lane == 0 && b + tt * G == live - 1) *a.count = prefix + agg;
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&prefix_bar[k]);  // offsets of tile tt ready
                }
            }
            incl_prev = before;
            r += nres;
        }
        return;
    }

    // ---------------------------------------------------------------- compute warps
    const int w = warp;
    const uint32_t mul = a.mul;
    uint32_t *const seg_base = stage_mem + w * (INTER ? HALF : kSeg);
    const uint32_t lead_tiles = a.lead != 0u ? 1u : 0u;  // tile 0 starts before the input

    // Segment of iteration j (tile `tile`, stage s) in shared memory, its
    // entries [vlo, vhi) being input entries: all of them except in the first
    // tile of an input with lead entries and in the ragged last tile, the only
    // tiles that compute the bounds (64-bit position: the last tile's later
    // segments can lie past 2^32 when T does not divide 2^32). The ragged tile
    // is read with plain loads.
    uint32_t vlo, vhi;
    auto arrive = [&](uint32_t tile, uint32_t *seg, int s, uint32_t parity) {
        vlo = 0u;
        vhi = uint32_t(kSeg);
        const bool full_tile = tile < full_tiles;
        if (!full_tile || tile < lead_tiles) {
            const uint64_t base = uint64_t(tile) * T + uint32_t(w) * kSeg;
            vlo = base < a.lead ? a.lead - uint32_t(base) : 0u;
            vhi = n > base ? uint32_t(min(n - base, uint64_t(kSeg))) : 0u;
            if (!full_tile) {
                // 16 bytes at a time, all in flight: up to 3 entries past the
                // input's end are read, in the same 16 bytes as its last one;
                // they and what is not read are cut from the tally
                if constexpr (INTER) {
                    // (base is even, and so is vhi: whole pairs)
                    const uint64_t pair = base / 2;
                    uint4 p[2], q[2];
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const uint32_t e = uint32_t(r * 128 + lane * 4);
                        if (2u * e < vhi) {
                            p[r] = *reinterpret_cast<const uint4 *>(a.in + pair + e);
                            q[r] = *reinterpret_cast<const uint4 *>(a.in2 + pair + e);
                        }
                    }
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const uint32_t e = uint32_t(r * 128 + lane * 4);
                        if (2u * e < vhi) {
                            *reinterpret_cast<uint4 *>(seg + e) = p[r];
                            *reinterpret_cast<uint4 *>(seg + T / 2 + e) = q[r];
                        }
                    }
                } else {
                    uint4 q[ROWS];
#pragma unroll
                    for (int r = 0; r < ROWS; ++r) {
                        const uint32_t e = uint32_t(r * 128 + lane * 4);
                        if (e < vhi) q[r] = *reinterpret_cast<const uint4 *>(a.in + base + e);
                    }
#pragma unroll
                    for (int r = 0; r < ROWS; ++r) {
                        const uint32_t e = uint32_t(r * 128 + lane * 4);
                        if (e < vhi) *reinterpret_cast<uint4 *>(seg + e) = q[r];
                    }
                }
                __syncwarp();
            }
        }
        if (full_tile && !mbar_wait(&full_bar[s], parity) && lane == 0) record_error(a.ws, kDevErrTimeout, tile);
    };
    // The segment's entries (after the transform) and their ranks.
    uint32_t v[ROWS][4], tl;
    auto count = [&](const uint32_t *seg) -> Ranks {
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const uint32_t e0 = uint32_t(r * 128 + lane * 4);
            if constexpr (INTER) {
                const uint2 p = *reinterpret_cast<const uint2 *>(seg + e0 / 2);
                const uint2 q = *reinterpret_cast<const uint2 *>(seg + T / 2 + e0 / 2);
                v[r][0] = p.x;
                v[r][1] = q.x;
                v[r][2] = p.y;
                v[r][3] = q.y;
            } else {
                const uint4 q = *reinterpret_cast<const uint4 *>(seg + e0);
                v[r][0] = q.x;
                v[r][1] = q.y;
                v[r][2] = q.z;
                v[r][3] = q.w;
            }
        }
        if constexpr (PK == kChainKind) {
            tl = chain_tally(a.chain, v);
        } else {
            if (mul != 1u) {
#pragma unroll
                for (int r = 0; r < ROWS; ++r)
#pragma unroll
                    for (int c = 0; c < 4; ++c) v[r][c] *= mul;
            }
            if constexpr (PK > kSetKind) tl = set_tally<PK - kSetKind>(a.set, v);
            else tl = tally<PK>(a.pred, v);
        }
        if (vlo != 0u || vhi != uint32_t(kSeg)) tl = cut_tally(tl, vlo, vhi, lane);
        return rank_tally(tl);
    };
    // Posts the count of iteration j's segment, whose entries start at word p
    // of the warp's ring. The last segment counted publishes the tile aggregate
    // at once, and that of the block's first tile decides how the block uses
    // its memory (of the held tiles, one in every lap decides again, early enough
    // for the producer, which is at most SH tiles ahead). (A warp of its own
    // that waits for the counts and publishes takes the atomic's round trip off
    // the compute warps, but publishes later: 241 -> 248 us at N = 2^28 and 50 %
    // kept.)
    auto post = [&](uint32_t j, uint32_t tile, uint32_t total, uint32_t p, auto held) {
        if (lane == 0) {
            const uint32_t k = j & uint32_t(NS - 1);
            s_wcnt[k][w] = p << 16 | total;
            const uint32_t prev = atomicAdd(&s_pack[k], (1u << 16) | total);
            if ((prev >> 16) == uint32_t(CWW - 1)) {
                const uint32_t agg = (prev & 0xFFFFu) + total;
                s_pack[k] = 0;
                st_relaxed_u64(status_at(agg_words, tile), pack_status(epoch, kFlagAggregate, agg));
                if (j == 0) {
                    s_ring = agg * kRingDen <= uint32_t(T) * RING_NUM ? 1u : 0u;
                    mbar_arrive(&mode_bar);
                } else if (FOLLOW && decltype(held)::value && j % uint32_t(SH) == uint32_t(SH - 3)) {
                    s_leave = agg * kRingDen <= uint32_t(T) * (RING_NUM - 1u) ? 1u : 0u;
                    mbar_arrive(&lap_bar);
                }
            }
            mbar_arrive(&count_bar[k]);
        }
    };
    // Offset of iteration j's segment once its tile is resolved (kNoOffset:
    // the look-back gave up).
    auto offset = [&](uint32_t j) -> uint32_t {
        const uint32_t k = j & uint32_t(NS - 1);
        if (!mbar_wait(&prefix_bar[k], (j / NS) & 1u)) {
            if (lane == 0) record_error(a.ws, kDevErrTimeout, b + j * G);
            return kNoOffset;
        }
        return s_woff[k][w];
    };

    arrive(b, seg_base, 0, 0u);
    post(0, b, count(seg_base).total, 0u, std::false_type{});
    if (!mbar_wait(&mode_bar, 0u) && lane == 0) record_error(a.ws, kDevErrTimeout, b);

    // -------------------------------------------------------------- ring
    // Tiles from j0 on, from stage 0 with the parity p0 on.
    auto ring_tiles = [&](uint32_t j0, uint32_t p0) __attribute__((always_inline)) {
        // Tile jq is the oldest one not written out; `used` ring words are
        // taken, and the next entries go to word p. A tile's entries start on
        // a 16-byte boundary.
        uint32_t *const ring = stage_mem + size_t(SR) * T + size_t(w) * RW;
        uint32_t jq = j0, p = 0, used = 0, s = 0, parity = p0;
        auto flush = [&]() {  // the oldest tile
            const uint32_t c = s_wcnt[jq & uint32_t(NS - 1)][w], cnt = c & 0xFFFFu, off = offset(jq);
            if (off != kNoOffset) warp_ring_out<RW>(ring, c >> 16, a.out + off, cnt, lane);
            __syncwarp();  // read before the ring's words are written again
            used -= (cnt + 3u) & ~3u;
            ++jq;
        };
        // The oldest N, 32 / N lanes each (tiles are resolved in order: the
        // last one's offset comes last): one wait and one chain of dependent
        // loads where there would be N.
        auto flush_group = [&](auto group) {
            constexpr uint32_t N = decltype(group)::value, LANES = 32u / N;
            const uint32_t k = (jq + uint32_t(lane) / LANES) & uint32_t(NS - 1);
            const uint32_t c = s_wcnt[k][w], cnt = c & 0xFFFFu;
            if (offset(jq + N - 1u) != kNoOffset) {
                const uint32_t off = s_woff[k][w];
                if (off != kNoOffset) {
                    uint32_t *const dst = a.out + off;
                    const uint32_t q = c >> 16;
#pragma unroll 1
                    for (uint32_t i = uint32_t(lane) % LANES; i < cnt; i += 2u * LANES) {
                        const uint32_t i2 = i + LANES;
                        const uint32_t x = ring[(q + i) & (RW - 1u)], x2 = ring[(q + i2) & (RW - 1u)];
                        dst[i] = x;
                        if (i2 < cnt) dst[i2] = x2;
                    }
                }
            }
            uint32_t room = (cnt + 3u) & ~3u;
#pragma unroll
            for (uint32_t d = LANES; d < 32u; d *= 2u) room += __shfl_xor_sync(kFull, room, d);
            __syncwarp();  // read before the ring's words are written again
            used -= room;
            jq += N;
        };
        // The oldest tiles out, of `pend` pending: several at once while they
        // are small (the youngest of them has had three tiles' time to be
        // resolved).
        auto write_out = [&](uint32_t pend) {
            if (NS >= 8 && pend >= 7u && used <= pend * kGroup4) flush_group(std::integral_constant<uint32_t, 4>{});
            else if (NS >= 8 && pend >= 5u && used <= pend * kGroup2) flush_group(std::integral_constant<uint32_t, 2>{});
            else flush();
        };
        uint32_t tile = b + j0 * G;
        for (uint32_t j = j0; j < my_tiles; ++j, tile += G) {
            if (j - jq >= uint32_t(NS)) write_out(j - jq);  // tile j's slot
            uint32_t *const seg = seg_base + size_t(s) * T;
            if (j != 0) arrive(tile, seg, int(s), parity);
            const Ranks rk = count(seg);
            if (j != 0) post(j, tile, rk.total, p, std::false_type{});
            const uint32_t room = (rk.total + 3u) & ~3u;
            // room for its entries, which stay in registers meanwhile: the
            // count is known, so nothing is written out before it has to be
            while (used + room > RW) write_out(j - jq);
            if (rk.total <= kFewKept) {
                // Few entries for the whole warp: each lane stores only its
                // own kept entries, in order, reading each back from the stage
                // (as many trips as the busiest lane has kept entries; most
                // lanes hold none, where the 16 predicated stores below cost
                // every lane 16 slots). Entry r * 128 + 4 lane + c of the
                // segment is bit 4 r + c of the lane's mask; its place is the
                // lane's first in row r (byte r of `first`: the rows before r
                // plus the lanes before this one in row r; no byte carries)
                // plus its kept entries in row r already stored.
                const uint32_t orig = tl & 0xFFFFu;
                const uint32_t first = rk.excl + rk.rows * 0x01010100u;
                const uint32_t *const mine = seg + uint32_t(lane) * (INTER ? 2u : 4u);
                for (uint32_t left = orig; left != 0u; left &= left - 1u) {
                    const uint32_t i = uint32_t(__ffs(int(left))) - 1u, r = i >> 2;
                    const uint32_t pos =
                        ((first >> (8u * r)) & 0xFFu) + __popc((orig ^ left) & (0xFu << (4u * r)));
                    const uint32_t x = INTER ? mine[r * 64u + ((i >> 1) & 1u) + (i & 1u) * uint32_t(T / 2)]
                                             : mine[r * 128u + (i & 3u)];
                    ring[(p + pos) & (RW - 1u)] = x * mul;
                }
            } else {
                const uint32_t dst = smem_addr(ring);
                auto store = [&](auto wrap) {  // wrap: p + total passes the ring's end
                    uint32_t rowbase = p;
#pragma unroll
                    for (int r = 0; r < ROWS; ++r) {
                        uint32_t pos = rowbase + ((rk.excl >> (8 * r)) & 0xFFu);
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            if ((tl >> (4 * r + c)) & 1u) {
                                st_shared_u32(dst + 4u * (wrap ? pos & (RW - 1u) : pos), v[r][c]);
                                ++pos;
                            }
                        }
                        rowbase += (rk.rows >> (8 * r)) & 0xFFu;
                    }
                };
                if (p + rk.total <= RW) store(std::false_type{});
                else store(std::true_type{});
            }
            p = (p + room) & (RW - 1u);
            used += room;
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty_bar[s]);  // nothing of this tile is left in the stage
            if (++s == uint32_t(SR)) {
                s = 0;
                parity ^= 1u;
            }
        }
        while (jq < my_tiles) flush();
    };

    if (s_ring != 0u) {
        ring_tiles(0u, 0u);
    } else {
        // -------------------------------------------------------------- hold
        uint32_t s = 0, parity = 0, so = 0;  // stages of tiles j and j - LAG
        uint32_t end = my_tiles;             // the first tile that is not held
        uint32_t tile = b;
        for (uint32_t j = 0; j < end + uint32_t(LAG); ++j, tile += G) {
            if (j >= uint32_t(LAG)) {
                const uint32_t jp = j - uint32_t(LAG), cnt = s_wcnt[jp & uint32_t(NS - 1)][w] & 0xFFFFu,
                               off = offset(jp);
                if (off != kNoOffset) {
                    const uint32_t *const held = seg_base + size_t(so) * T;
                    if constexpr (INTER) {
                        warp_copy_out(held, a.out + off, min(cnt, uint32_t(HALF)), lane);
                        if (cnt > uint32_t(HALF)) warp_copy_out(held + T / 2, a.out + off + HALF, cnt - HALF, lane);
                    } else {
                        warp_copy_out(held, a.out + off, cnt, lane);
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty_bar[so]);  // this warp is done with the stage
                if (++so == uint32_t(SH)) so = 0;
            }
            if (j < end) {
                uint32_t *const seg = seg_base + size_t(s) * T;
                if (j != 0) arrive(tile, seg, int(s), parity);
                const Ranks rk = count(seg);
                if (j != 0) post(j, tile, rk.total, 0u, std::true_type{});
                // in place, at the front of the segment (an explicit st.shared
                // to the segment's shared-memory address)
                const uint32_t dst = smem_addr(seg);
                __syncwarp();  // every lane holds its entries before any is overwritten
                uint32_t rowbase = 0;
#pragma unroll
                for (int r = 0; r < ROWS; ++r) {
                    uint32_t pos = rowbase + ((rk.excl >> (8 * r)) & 0xFFu);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        if ((tl >> (4 * r + c)) & 1u) {
                            if constexpr (INTER)
                                st_shared_u32(dst + 4u * pos + (pos >= uint32_t(HALF) ? 4u * (T / 2 - HALF) : 0u),
                                              v[r][c]);
                            else
                                st_shared_u32(dst + 4u * pos, v[r][c]);
                            ++pos;
                        }
                    }
                    rowbase += (rk.rows >> (8 * r)) & 0xFFu;
                }
                __syncwarp();
                if (++s == uint32_t(SH)) {
                    s = 0;
                    parity ^= 1u;
                    if (FOLLOW && j + 1u < my_tiles) {
                        if (!mbar_wait(&lap_bar, parity ^ 1u) && lane == 0)
                            record_error(a.ws, kDevErrTimeout, tile);
                        if (__any_sync(kFull, s_leave != 0u)) end = j + 1u;
                    }
                }
            }
        }
        if (FOLLOW && end != my_tiles) {
            // Every tile before tile `end` is written out by this warp; the
            // rings lie in stages that other warps may still be writing out of.
            if (lane == 0) mbar_arrive(&left_bar);
            if (!mbar_wait(&left_bar, 0u) && lane == 0) record_error(a.ws, kDevErrTimeout, b + end * G);
            ring_tiles(end, parity);
        }
    }
}

template <int PK, int CWW, int SR, int SH, int LAG, int MAXG, int MINB, int NS, int BMAX, bool INTER = false>
__global__ void __launch_bounds__((CWW + 2) * 32, MINB) k_compact_tma(const TmaArgs a) {
    tma_compact_pass<PK, CWW, SR, SH, LAG, MAXG, NS, BMAX, INTER>(a);
}

template <int CWW, int S, int LAG, int MAXG, int MINB>
__global__ void __launch_bounds__((CWW + 2) * 32, MINB) k_scan_tma(const TmaBase a) {
    tma_scan_pass<CWW, S, LAG, MAXG>(a);
}

// Cooperative launch of `kern` with `smem` bytes of dynamic shared memory:
// one block per tile up to the blocks resident at once (at most MAXG),
// found once per device.
template <int BLOCK, int T, int MAXG, class Kern, class Args>
ka_status launch_tma_kernel(Kern kern, PerDeviceInt &grid_cache, size_t smem, const Args &a, uint64_t cap,
                            cudaStream_t stream) {
    const int resident = per_device_value(grid_cache, current_device(), [&] {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess)
            return -1;
        int occ = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, BLOCK, smem) != cudaSuccess || occ < 1)
            return -1;
        const int g = device_info().sm_count * occ;
        return g > MAXG ? MAXG : g;
    });
    if (resident <= 0) return launch_setup_error();
    uint64_t grid = (cap + T - 1) / T;
    if (grid > uint64_t(resident)) grid = uint64_t(resident);
    if (grid < 1) grid = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(grid));
    cfg.blockDim = dim3(BLOCK);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return launch_status(cudaLaunchKernelEx(&cfg, kern, a));
}

template <int PK, int CWW, int SR, int SH, int LAG, int MAXG, int MINB, int NS, int BMAX, bool INTER = false>
ka_status launch_compact_shape(const TmaArgs &a, uint64_t cap, cudaStream_t stream) {
    constexpr int BLOCK = (CWW + 2) * 32, T = CWW * kSeg;
    const size_t smem = size_t(SH) * T * 4;
    static PerDeviceInt grid_cache;
    return launch_tma_kernel<BLOCK, T, MAXG>(k_compact_tma<PK, CWW, SR, SH, LAG, MAXG, MINB, NS, BMAX, INTER>, grid_cache,
                                             smem, a, cap, stream);
}

// The general chain's kernels of a configuration: one array, or the interleave
// of two.
template <int CWW, int SR, int SH, int LAG, int MAXG, int MINB, int NS, int BMAX>
ka_status launch_chain_config(const TmaArgs &a, uint64_t cap, cudaStream_t stream) {
    if (a.in2) return launch_compact_shape<kChainKind, CWW, SR, SH, LAG, MAXG, MINB, NS, BMAX, true>(a, cap, stream);
    return launch_compact_shape<kChainKind, CWW, SR, SH, LAG, MAXG, MINB, NS, BMAX>(a, cap, stream);
}

// One configuration's compaction for predicate kind pk (every kind has its
// own kernel); with INTER, of the interleave of two arrays.
template <int CWW, int SR, int SH, int LAG, int MAXG, int MINB, int NS, int BMAX, bool INTER = false>
ka_status launch_compact_config(const TmaArgs &a, int32_t pk, uint64_t cap, cudaStream_t stream) {
    switch (pk) {
#define KA_CASE(K) \
    case K: return launch_compact_shape<K, CWW, SR, SH, LAG, MAXG, MINB, NS, BMAX, INTER>(a, cap, stream);
        KA_CASE(kAndMaskEq0)
        KA_CASE(kLt)
        KA_CASE(kPopcOdd)
        KA_CASE(kModNe0)
        KA_CASE(kNe)
        KA_CASE(kAll)
#undef KA_CASE
    default: return KA_E_ARG;
    }
}

// One configuration's scan.
template <int CWW, int S, int LAG, int MAXG, int MINB>
ka_status launch_scan_config(const TmaArgs &a, uint64_t cap, cudaStream_t stream) {
    constexpr int BLOCK = (CWW + 2) * 32, T = CWW * kSeg;
    static PerDeviceInt grid_cache;
    return launch_tma_kernel<BLOCK, T, MAXG>(k_scan_tma<CWW, S, LAG, MAXG, MINB>, grid_cache, size_t(S) * T * 4,
                                             static_cast<const TmaBase &>(a), cap, stream);
}

// One translation unit per tile shape instantiates its configuration.
ka_status launch_tma_768(const TmaArgs &a, bool scan, int32_t pk, uint64_t cap, cudaStream_t stream);
ka_status launch_tma_512(const TmaArgs &a, bool scan, int32_t pk, uint64_t cap, cudaStream_t stream);
ka_status launch_tma_256(const TmaArgs &a, bool scan, int32_t pk, uint64_t cap, cudaStream_t stream);
ka_status launch_chain_768(const TmaArgs &a, uint64_t cap, cudaStream_t stream);
ka_status launch_chain_512(const TmaArgs &a, uint64_t cap, cudaStream_t stream);
// Shape (768, 16): one test on an interleave; a set of tests (k_tma_sets_*.cu:
// KA_E_UNSUPPORTED for a mask of another file).
ka_status launch_inter_768(const TmaArgs &a, int32_t pk, uint64_t cap, cudaStream_t stream);
ka_status launch_sets_768_a(const TmaArgs &a, int mask, uint64_t cap, cudaStream_t stream);
ka_status launch_sets_768_b(const TmaArgs &a, int mask, uint64_t cap, cudaStream_t stream);
ka_status launch_sets_768_c(const TmaArgs &a, int mask, uint64_t cap, cudaStream_t stream);
ka_status launch_sets_768_d(const TmaArgs &a, int mask, uint64_t cap, cudaStream_t stream);

}  // namespace tma
}  // namespace ka
