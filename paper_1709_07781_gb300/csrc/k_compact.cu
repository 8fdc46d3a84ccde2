// Fused single-pass stream compaction (Sec. 4.1's flag, prefix-sum and move
// phases in one kernel; the paper's own OpenCL version fuses only the last
// two, and Sec. 3.6 names "several kernels inside one actor" as the way to
// avoid inter-stage traffic). The per-tile work is compact_tile (ka_tile.cuh).
// Blocks are persistent (grid = resident blocks) and take tiles by ticket.
// Output offsets never exceed input positions, so out == in is safe: a tile
// writes only after all its predecessors have loaded their input.
//
// An array whose tiles all run at once (up to 4.98 M entries in the largest of the
// shapes) has a kernel of its own, k_compact_wave: such a call is a chain of
// latencies, not of bytes.
#include <algorithm>

#include "ka_internal.h"
#include "ka_tile.cuh"
#include "ka_tma.cuh"

namespace ka {

struct CompactArgs {
    const uint32_t *in;
    uint32_t *out;
    const uint32_t *n_ptr;
    uint32_t *count;
    WsHeader *ws;
    uint64_t *status;
    uint32_t n;
    uint32_t status_cap;
    uint32_t mul;
    uint32_t vec_ok;
    PredDev pred;
};

template <int BLOCK, int IPT>
__global__ void __launch_bounds__(BLOCK) k_compact_fused(const CompactArgs a) {
    constexpr int T = BLOCK * IPT;
    __shared__ CompactSmem<BLOCK, IPT> sm;
    __shared__ uint32_t s_ticket, s_epoch, s_n, s_spin;
    const int tid = threadIdx.x;

    if (tid == 0) {
        uint32_t n = a.n;
        if (a.n_ptr) {
            const uint32_t d = *a.n_ptr;
            n = d < n ? d : n;
        }
        s_n = n;
        const uint32_t sl = a.ws->spin_limit;
        s_spin = sl ? sl : kDefaultSpinLimit;
    }
    __syncthreads();
    const uint32_t n = s_n;
    const uint32_t spin = s_spin;
    const uint32_t live_tiles = uint32_t((uint64_t(n) + T - 1) / T);
    if (live_tiles > a.status_cap) {
        if (tid == 0 && blockIdx.x == 0) record_error(a.ws, kDevErrWorkspace, 0);
        return;
    }

    for (;;) {
        if (tid == 0) {
            uint32_t ep;
            bool last;
            const uint32_t t = take_ticket(a.ws, live_tiles, &ep, &last);
            if (last && live_tiles == 0) *a.count = 0u;
            s_ticket = t;
            s_epoch = ep;
        }
        __syncthreads();
        const uint32_t tile = s_ticket;
        const uint32_t epoch = s_epoch;
        if (tile >= live_tiles) break;
        const uint32_t base = tile * uint32_t(T);
        const uint32_t valid = (n - base) < uint32_t(T) ? (n - base) : uint32_t(T);
        compact_tile<BLOCK, IPT>(sm, a.in + base, a.out, valid, a.vec_ok != 0u, a.mul, a.pred, a.status, tile, 0u,
                                 epoch, spin, a.ws, tile == live_tiles - 1 ? a.count : nullptr);
    }
}

constexpr uint32_t kWaveMaxTiles = 1216;  // every tile reads a status word of each before it (152 SMs x 8 blocks)

// One tile per block, every block running at once. What bounds it is the chain
// ticket, loads, counts, offset, stores, a round trip to L2 or more each; so
//   * a block loads the tile of its own index before its ticket is back, and
//     only loads again if the ticket names another tile (tickets come in block
//     order nearly always; they guarantee that every tile before this one is
//     running). With a device length, the loads wait for the length;
//   * a tile waits for no look-back of another: it adds up the counts of all
//     tiles before it, one status word per thread, all in flight together,
//     where a decoupled look-back walks 32 at a time and waits for prefixes;
//   * warp w of a block owns 32 IPT consecutive entries, so one barrier of the
//     warps' totals ranks the whole tile;
//   * the tile starts on a 16-byte boundary of the input (up to 3 entries
//     before it, in the same 16 bytes as its first, are read and ignored).
// A tile whose wait gives up records the error and writes nothing. It has posted
// its count by then, so unlike in the ticketed kernel the tiles after it are not
// stopped: they go on with offsets that are right, and the last of them may store
// the count. (Outputs and count are undefined once an error is recorded.)
// A ka_compact call among others in a CUDA graph, us, at 50 % kept, against the
// ticketed kernel below in the same shape: (256, 4), 2^16 entries 5.3 -> 4.2,
// 2^18 6.1 -> 5.4, 2^20 9.2 -> 7.9; (512, 8), 2^18 5.4 -> 4.9, 2^20 6.4 -> 5.4,
// 2^21 8.7 -> 7.3.
struct WaveArgs {
    const uint32_t *in;  // input rounded down to 16 bytes: entry i of the input is in[lead + i]
    uint32_t *out;
    const uint32_t *n_ptr;
    uint32_t *count;
    WsHeader *ws;
    uint64_t *status;
    uint32_t n;
    uint32_t status_cap;
    uint32_t lead;
    PredChain chain;
};

template <int BLOCK, int IPT>
__global__ void __launch_bounds__(BLOCK, 2048 / BLOCK) k_compact_wave(const WaveArgs a) {
    constexpr int ROWS = IPT / 4, WARPS = BLOCK / 32, SEG = 32 * IPT;
    constexpr uint32_t T = BLOCK * IPT;
    static_assert(ROWS >= 1 && ROWS <= 4 && WARPS <= 32, "a lane's tally, and one warp scans the warps");
    __shared__ uint32_t s_out[T];
    __shared__ uint32_t s_wtot[WARPS], s_part[WARPS];
    __shared__ uint32_t s_ticket, s_epoch, s_n, s_spin, s_bad;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    uint32_t v[ROWS][4];
    auto load = [&](uint32_t tile, uint32_t n) {  // n: entries from the 16-byte boundary
        const uint64_t base = uint64_t(tile) * T + uint32_t(warp) * SEG;
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const uint64_t e = base + uint32_t(r * 128 + lane * 4);
            uint4 q = make_uint4(0u, 0u, 0u, 0u);
            if (e < n) q = *reinterpret_cast<const uint4 *>(a.in + e);
            v[r][0] = q.x;
            v[r][1] = q.y;
            v[r][2] = q.z;
            v[r][3] = q.w;
        }
    };
    wait_for_prior();
    if (!a.n_ptr) load(blockIdx.x, a.n + a.lead);
    if (tid == 0) {
        allow_dependents();
        uint32_t ep;
        bool last;
        s_ticket = take_ticket(a.ws, 0u, &ep, &last);  // one ticket per block: the last one starts the next epoch
        s_epoch = ep;
        uint32_t n = a.n;
        if (a.n_ptr) {
            const uint32_t d = *a.n_ptr;
            n = d < n ? d : n;
        }
        s_n = n;
        const uint32_t sl = a.ws->spin_limit;
        s_spin = sl ? sl : kDefaultSpinLimit;
        s_bad = 0u;
    }
    __syncthreads();
    const uint32_t n = s_n ? s_n + a.lead : 0u, tile = s_ticket, epoch = s_epoch;
    const uint32_t live = (n + T - 1u) / T;
    if (live > a.status_cap) {
        if (tid == 0 && tile == 0u) record_error(a.ws, kDevErrWorkspace, 0);
        return;
    }
    if (tile >= live) {
        if (tid == 0 && live == 0u && tile == 0u) *a.count = 0u;
        return;
    }
    if (a.n_ptr || tile != blockIdx.x) load(tile, n);

    uint32_t tl = tma::chain_tally(a.chain, v);
    {
        const uint32_t base = tile * T + uint32_t(warp) * SEG;
        const uint32_t vlo = base < a.lead ? a.lead - base : 0u;
        const uint32_t vhi = n > base ? min(n - base, uint32_t(SEG)) : 0u;
        if (vlo != 0u || vhi != uint32_t(SEG)) tl = tma::cut_tally(tl, vlo, vhi, lane);
    }
    const tma::Ranks rk = tma::rank_tally(tl);
    if (lane == 0) s_wtot[warp] = rk.total;
    __syncthreads();
    const uint32_t wt = lane < WARPS ? s_wtot[lane] : 0u;
    const uint32_t wincl = warp_incl_scan(wt, lane);
    const uint32_t agg = __shfl_sync(kFull, wincl, 31);
    if (tid == 0) st_relaxed_u64(status_at(a.status, tile), pack_status(epoch, kFlagAggregate, agg));

    // the kept entries in tile order, while the other tiles' counts arrive
    uint32_t rowbase = __shfl_sync(kFull, wincl - wt, warp);
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        uint32_t pos = rowbase + ((rk.excl >> (8 * r)) & 0xFFu);
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if ((tl >> (4 * r + c)) & 1u) s_out[pos++] = v[r][c];
        rowbase += (rk.rows >> (8 * r)) & 0xFFu;
    }

    const uint32_t want = epoch & kEpochMask, spin = s_spin;
    uint32_t sum = 0, polls = 0, sleep_ns = 0;
    for (uint32_t i = uint32_t(tid); i < tile;) {
        const uint64_t w = ld_relaxed_u64(status_at(a.status, i));
        if (uint32_t(w >> 34) == want && (uint32_t(w >> 32) & 3u) == kFlagAggregate) {
            sum += uint32_t(w);
            i += BLOCK;
            continue;
        }
        if (++polls >= spin) {
            record_error(a.ws, kDevErrTimeout, tile);
            s_bad = 1u;
            break;
        }
        if (polls > 4) {
            __nanosleep(sleep_ns);
            sleep_ns = sleep_ns < 128 ? sleep_ns * 2 + 32 : 128;
        }
    }
    sum = warp_sum(sum);
    if (lane == 0) s_part[warp] = sum;
    __syncthreads();
    const uint32_t prefix = warp_sum(lane < WARPS ? s_part[lane] : 0u);
    if (s_bad) return;  // (recorded; nothing of this tile is written)
    if (tid == 0 && tile == live - 1u) *a.count = prefix + agg;
    uint32_t *const dst = a.out + prefix;
    for (uint32_t k = uint32_t(tid); k < agg; k += BLOCK) dst[k] = s_out[k];
}

template <int BLOCK, int IPT>
static uint32_t wave_tiles() {  // tiles that run at once
    static PerDeviceInt cache;
    return uint32_t(per_device_value(cache, current_device(), [] {
        int occ = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_compact_wave<BLOCK, IPT>, BLOCK, 0);
        return occ > 0 ? occ * device_info().sm_count : 1;
    }));
}

// The wave kernel of a register shape, if every tile of L runs at once.
// KA_E_UNSUPPORTED: it does not.
template <int BLOCK, int IPT>
static ka_status launch_wave_shape(WaveArgs a, uint64_t cap, cudaStream_t stream) {
    const uint64_t tiles = tiles_for(cap + a.lead, BLOCK * IPT);
    if (tiles > wave_tiles<BLOCK, IPT>() || tiles > kWaveMaxTiles) return KA_E_UNSUPPORTED;
    return launch_dependent(k_compact_wave<BLOCK, IPT>, unsigned(tiles ? tiles : 1), BLOCK, stream, a);
}

static ka_status launch_wave(const ChainLaunch &L, ka_tile t, cudaStream_t stream) {
    if (L.n > uint64_t(kWaveMaxTiles) * t.block * t.ipt) return KA_E_UNSUPPORTED;
    WaveArgs a{};
    const AlignedView view = aligned_view(L.in, L.n);
    a.lead = view.lead;
    a.in = view.in;
    a.out = L.out;
    a.n_ptr = L.n_ptr;
    a.count = L.count;
    a.ws = static_cast<WsHeader *>(L.ws);
    a.status = reinterpret_cast<uint64_t *>(static_cast<char *>(L.ws) + kWsHeaderBytes);
    a.n = uint32_t(L.n);
    a.status_cap = status_capacity(L.ws_bytes);
    a.chain = L.chain;
    switch (shape_key(t.block, t.ipt)) {
#define KA_CASE(B, I) \
    case shape_key(B, I): return launch_wave_shape<B, I>(a, L.n, stream);
        KA_FOR_EACH_SHAPE(KA_CASE)
#undef KA_CASE
    default: return KA_E_UNSUPPORTED;
    }
}

ka_status launch_compact_chain(const ChainLaunch &L, cudaStream_t stream) {
    const uint64_t entries = L.in2 ? 2 * L.n : L.n;
    if (entries > kChainEntries || L.chain.n == 0 || L.chain.n > kChainMax) return KA_E_ARG;
    if (L.n && (!L.in || !L.out)) return KA_E_ARG;
    if (!L.count || L.n_ptr == L.count) return KA_E_ARG;
    if (L.in2 && ((reinterpret_cast<uintptr_t>(L.in) | reinterpret_cast<uintptr_t>(L.in2)) & 15u)) return KA_E_ARG;
    ka_tile t = resolve_tile(KA_KERNEL_COMPACT, entries, nullptr);
    // A chain is a request somebody waits for, not a call among others, so what
    // counts is its own latency: the TMA kernels' is the lower one from about
    // 0.4 M entries (three actors on 2^20: 24.4 us, and 25.0 us on the wave kernel).
    if (!L.in2 && entries < (3ull << 17) && !tma_shape(t.block, t.ipt)) {
        const ka_status ws_ok = check_workspace(L.ws, L.ws_bytes, tiles_for(entries, t.block * t.ipt));
        if (ws_ok != KA_OK) return ws_ok;
        const ka_status s = launch_wave(L, t, stream);
        if (s != KA_E_UNSUPPORTED) return s;
    }
    return launch_chain_tma(L, t, stream);
}

template <int BLOCK, int IPT>
static ka_status launch_shape(const CompactArgs &a, uint64_t cap, cudaStream_t stream) {
    constexpr int T = BLOCK * IPT;
    static PerDeviceInt occ_cache;
    const int occupancy = per_device_value(occ_cache, current_device(), [] {
        int occ = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_compact_fused<BLOCK, IPT>, BLOCK, 0);
        return occ > 0 ? occ : 1;
    });
    uint64_t grid = (cap + T - 1) / T;
    const uint64_t resident = uint64_t(device_info().sm_count) * occupancy;
    if (grid > resident) grid = resident;
    if (grid < 1) grid = 1;
    k_compact_fused<BLOCK, IPT><<<unsigned(grid), BLOCK, 0, stream>>>(a);
    return cuda_status(cudaGetLastError());
}

ka_status launch_compact(const CompactLaunch &L, cudaStream_t stream) {
    if (L.n > 0xFFFFFFFFull) return KA_E_ARG;
    if (L.n && (!L.in || !L.out)) return KA_E_ARG;
    if (!L.count) return KA_E_ARG;
    if (L.n_ptr && L.n_ptr == L.count) return KA_E_ARG;
    const ka_tile t = L.tile;
    if (!tile_supported_for(KA_KERNEL_COMPACT, t.block, t.ipt)) return KA_E_ARG;
    const uint64_t tiles = std::max(L.ws_tiles, tiles_for(L.n, t.block * t.ipt));
    const ka_status ws_ok = check_workspace(L.ws, L.ws_bytes, tiles);
    if (ws_ok != KA_OK) return ws_ok;
    ChainLaunch one{L.in, nullptr, L.out, L.n_ptr, L.count, L.n, {}, L.ws, L.ws_bytes};
    one.chain.n = 1;
    one.chain.mul_all = L.mul;
    one.chain.op[0].pred = L.pred;
    one.chain.op[0].mul = L.mul;
    if (!tma_shape(t.block, t.ipt)) {
        const ka_status wave = launch_wave(one, t, stream);
        if (wave != KA_E_UNSUPPORTED) return wave;
    }
    if (L.any_kernel) {
        // tiles of 8192 entries that all run at once (4.98 M entries), in place
        // of a TMA shape, or of a register shape (tuned for a smaller array of
        // the same power of two) whose tiles do not. Among others on a stream,
        // 1 % / 50 % kept: 3.0 M entries 8.3 / 9.5 us on the TMA kernel, 6.8 /
        // 8.2 us here; 4.9 M 10.3 / 10.3 and 7.7 / 8.8.
        const ka_status s = launch_wave(one, ka_tile{512, 16}, stream);
        if (s != KA_E_UNSUPPORTED) return s;
    }
    if (compact_tma_eligible(L)) return launch_compact_tma(L, stream);
    if (!tile_supported(t.block, t.ipt)) return KA_E_ARG;  // a TMA-only shape beyond its size limit
    CompactArgs a;
    a.in = L.in;
    a.out = L.out;
    a.n_ptr = L.n_ptr;
    a.count = L.count;
    a.ws = static_cast<WsHeader *>(L.ws);
    a.status = reinterpret_cast<uint64_t *>(static_cast<char *>(L.ws) + kWsHeaderBytes);
    a.n = uint32_t(L.n);
    a.status_cap = status_capacity(L.ws_bytes);
    a.mul = L.mul;
    a.vec_ok = (reinterpret_cast<uintptr_t>(L.in) & 15u) == 0 ? 1u : 0u;
    a.pred = L.pred;
    switch (shape_key(t.block, t.ipt)) {
#define KA_CASE(B, I) \
    case shape_key(B, I): return launch_shape<B, I>(a, L.n, stream);
        KA_FOR_EACH_SHAPE(KA_CASE)
#undef KA_CASE
    default: return KA_E_ARG;
    }
}

}  // namespace ka

using namespace ka;

extern "C" ka_status ka_compact(const uint32_t *d_in, uint64_t n, const uint32_t *d_n, int32_t pred, uint32_t param,
                                uint32_t xform, uint32_t *d_out, uint32_t *d_count, void *d_ws, uint64_t ws_bytes,
                                const ka_tile *tile, void *stream) {
    CompactLaunch L;
    const ka_status s = make_pred(pred, param, &L.pred);
    if (s != KA_OK) return s;
    if (xform != KA_XFORM_NONE && xform != KA_XFORM_HASH) return KA_E_ARG;
    L.in = d_in;
    L.out = d_out;
    L.n_ptr = d_n;
    L.count = d_count;
    L.n = n;
    L.mul = xform == KA_XFORM_HASH ? kHashMul : 1u;
    L.ws = d_ws;
    L.ws_bytes = ws_bytes;
    L.any_kernel = !(tile && tile->block && tile->ipt);
    L.tile = resolve_tile(KA_KERNEL_COMPACT, n, tile, &L.ws_tiles);
    return launch_compact(L, static_cast<cudaStream_t>(stream));
}
