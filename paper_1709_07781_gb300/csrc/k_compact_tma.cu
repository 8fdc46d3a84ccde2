// Entry points of the warp-specialised TMA kernel (ka_tma_pass.cuh): the
// fused compaction and the exclusive scan for the TMA tile shapes, with any
// 4-byte-aligned input (tiles are shifted back to a 16-byte boundary). The
// kernels are instantiated in k_tma_<shape>.cu, one file per tile shape.
#include <algorithm>

#include "ka_tma_pass.cuh"

namespace ka {

using namespace tma;

namespace {

// Compaction, tile (768, 16): 22 compute warps, 11264 entries, 5 tiles of 44 KiB, 1 block per SM;
//             tile (512, 16): 16 compute warps, 8192 entries, 3 tiles of 32 KiB, 2 blocks per SM;
//             tile (256, 16): 8 compute warps, 4096 entries, 4 tiles of 16 KiB, 3 blocks per SM.
// Scan: the same, except 26 compute warps and 4 stages of 52 KiB for (768, 16).
ka_status launch_tma(const TmaArgs &a, ka_tile tile, bool scan, int32_t pk, uint64_t cap, cudaStream_t stream) {
    if (tile.block == 768) return launch_tma_768(a, scan, pk, cap, stream);
    if (tile.block == 512) return launch_tma_512(a, scan, pk, cap, stream);
    return launch_tma_256(a, scan, pk, cap, stream);
}

}  // namespace

bool tma_shape(uint32_t block, uint32_t ipt) {
    return ipt == 16 && (block == 256 || block == 512 || block == 768);
}

bool compact_tma_eligible(const CompactLaunch &L) {
    // the shifted length n + lead must fit 32 bits
    return tma_shape(L.tile.block, L.tile.ipt) && L.n <= 0xFFFFFFFCull;
}

ka_status launch_compact_tma(const CompactLaunch &L, cudaStream_t stream) {
    TmaArgs a{};
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
    a.mul = L.mul;
    a.pred = L.pred;
    a.out_vec = 0;
    return launch_tma(a, L.tile, false, L.pred.kind, L.n + a.lead, stream);
}

namespace {

// A chain as something simpler with the same result: one test, or a set of
// different ones. Products that come before every test may go in front of them
// all; tests of one kind combine (two upper bounds are the lower of them) or, if
// they do not, and where a product stands between or after tests, the chain
// stays as it is (mask -1). mask 0: keep everything.
struct Simplified {
    int mask = -1;
    uint32_t mul = 1;
    PredSet set{};
    PredDev one{};  // the test, when the mask has one bit or none
};

Simplified simplify(const PredChain &c) {
    Simplified s;
    s.one.kind = kAll;
    int mask = 0;
    for (uint32_t i = 0; i < c.n; ++i) {
        const PredDev &p = c.op[i].pred;
        if (c.op[i].mul != 1u) {
            if (mask != 0) return s;
            s.mul *= c.op[i].mul;
        }
        int bit = 0;
        switch (p.kind) {
        case kAndMaskEq0:
            bit = kSetAnd;
            s.set.and_mask |= p.a;
            break;
        case kLt:
            bit = kSetLt;
            s.set.lt = mask & bit ? std::min(s.set.lt, p.a) : p.a;
            break;
        case kPopcOdd: bit = kSetPopc; break;
        case kModNe0:
            bit = kSetMod;
            if (mask & bit && (s.set.mod_a != p.a || s.set.mod_b != p.b || s.set.mod_s != p.s)) return s;
            s.set.mod_a = p.a;
            s.set.mod_b = p.b;
            s.set.mod_s = p.s;
            break;
        case kNe:
            bit = kSetNe;
            if (mask & bit && s.set.ne != p.a) return s;
            s.set.ne = p.a;
            break;
        default: continue;  // kAll
        }
        mask |= bit;
        s.one = p;
    }
    if (mask == kSetAnd) s.one.a = s.set.and_mask;
    if (mask == kSetLt) s.one.a = s.set.lt;
    s.mask = mask;
    return s;
}

}  // namespace

bool chain_is_set(const PredChain &c) { return simplify(c).mask >= 0; }

// The chain kernel tests an entry with each op in turn, for any ops, at the cost
// of a switch and a mask per op (16 entries: 20 to 30 instructions) and of two
// to four instructions an entry; the kernels made for one test or for a set
// only have the latter. Which is which is settled here, on the host.
ka_status launch_chain_tma(const ChainLaunch &L, ka_tile t, cudaStream_t stream) {
    const uint64_t entries = L.in2 ? 2 * L.n : L.n;
    // two of the shapes have chain kernels: the smaller of them for any other
    if (t.block != 768) t = ka_tile{512, 16};
    const ka_status ws_ok = check_workspace(L.ws, L.ws_bytes, tiles_for(entries, t.block * t.ipt));
    if (ws_ok != KA_OK) return ws_ok;
    TmaArgs a{};
    const AlignedView view = aligned_view(L.in, L.n);
    a.lead = view.lead;
    a.in = view.in;
    a.in2 = L.in2;
    a.out = L.out;
    a.n_ptr = L.n_ptr;
    a.count = L.count;
    a.ws = static_cast<WsHeader *>(L.ws);
    a.status = reinterpret_cast<uint64_t *>(static_cast<char *>(L.ws) + kWsHeaderBytes);
    a.n = uint32_t(L.n);
    a.status_cap = status_capacity(L.ws_bytes);
    a.mul = L.chain.mul_all;
    a.chain = L.chain;
    const uint64_t cap = entries + a.lead;
    const Simplified s = simplify(L.chain);
    if (s.mask >= 0) {
        const bool single = (s.mask & (s.mask - 1)) == 0;
        a.mul = s.mul;
        a.pred = s.one;
        a.set = s.set;
        if (single && !L.in2) return launch_tma(a, t, false, s.one.kind, cap, stream);
        if (single && t.block == 768) return launch_inter_768(a, s.one.kind, cap, stream);
        if (!single && !L.in2 && t.block == 768)
            for (auto sets : {launch_sets_768_a, launch_sets_768_b, launch_sets_768_c, launch_sets_768_d}) {
                const ka_status r = sets(a, s.mask, cap, stream);
                if (r != KA_E_UNSUPPORTED) return r;
            }
        a.mul = L.chain.mul_all;
    }
    return t.block == 768 ? launch_chain_768(a, cap, stream) : launch_chain_512(a, cap, stream);
}

ka_status launch_scan_tma(const uint32_t *in, uint64_t n, const uint32_t *n_ptr, uint32_t *out, uint32_t *total,
                          void *ws, uint64_t ws_bytes, ka_tile tile, cudaStream_t stream) {
    TmaArgs a{};
    const AlignedView view = aligned_view(in, n);
    a.lead = view.lead;
    a.in = view.in;
    a.out = out;
    a.out_vec = ((reinterpret_cast<uintptr_t>(out) - 4u * a.lead) & 15u) == 0 ? 1u : 0u;
    a.n_ptr = n_ptr;
    a.count = total;
    a.ws = static_cast<WsHeader *>(ws);
    a.status = reinterpret_cast<uint64_t *>(static_cast<char *>(ws) + kWsHeaderBytes);
    a.n = uint32_t(n);
    a.status_cap = status_capacity(ws_bytes);
    a.mul = 1u;
    a.pred = PredDev{};
    return launch_tma(a, tile, true, kAll, n + a.lead, stream);
}

}  // namespace ka
