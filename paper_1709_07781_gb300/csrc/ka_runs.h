// Runs of stages issued as one kernel: which stages of a composition share one, and
// the chain of tests that they come to. Used by the actor layer and by the loop
// that launches the same kernels without it.
//
// A compaction keeps the entries that pass its test, in order, so compacting a
// compacted array keeps the entries that pass both tests; a hash map multiplies
// each entry; flag map, exclusive scan and move together are a compaction; and the
// interleave only orders what the compaction after it reads. A run of such stages
// is therefore one pass over the run's input (launch_compact_chain), which leaves
// the arrays between the stages unwritten: nobody but the next stage could have
// read them. Request to response, 4-stage pipeline of N = 2^26: 267 us (four
// kernels, 1.1 GB) became 90 us (one, 0.31 GB); interleave and zero removal of 2^24
// pairs: 110 us became 60 us; flag map, scan and move of 2^20 entries: 41 us became
// 25 us.
#pragma once

#include "ka_internal.h"

namespace ka {

// A stage as far as runs need to know it.
struct RunStage {
    int32_t kind;
    PredDev pred;  // of a compaction or a flag map
    uint32_t mul;  // of a compaction
    bool shaped;   // the caller has chosen its tile shape, and with it its kernel
};

struct FusedRun {
    int stages = 0;  // stages of the run, from the first (0: no run here)
    PredChain chain{};
    bool inter = false;  // the run starts with the interleave
};

// From this many entries on, a run of one array is one that kernels are made
// for. The kernel for any chain makes every test on every entry, 1.05 us per 2^20
// entries whatever they keep, where stages one by one stop reading what the first
// has dropped. Three stages with a hash after the first test, which keeps 0 / 1 /
// 10 / 50 %, one by one and as a general chain, us: 2^25 entries 47 / 58 / 71 / 97
// and 50 / 51 / 54 / 58; 2^26 66 / 83 / 104 / 161 and 83 / 85 / 90 / 98; 2^28 173 /
// 208 / 305 / 508 and 284 / 287 / 306 / 340. (A second phase in that kernel, for the
// few entries that pass its first test, took longer than the tests it saved.) Runs
// that start with the interleave gain more than that by not writing it. The
// kernels made for a set are slower than their stages one by one only from 2^27
// entries on and where the first test keeps next to nothing: lt, popc odd, mod 3
// at 2^28, 0 / 0.1 / 1 / 10 %: 194 / 193 / 200 / 222 against 172 / 186 / 208 / 300.
// (Cheap tests first, and the others on what passes them, where the warp's last
// segment kept little: 166 / 168 / 190 / 232, and every other run 1 to 7 % longer.)
constexpr uint64_t kSetsOnlyFrom = 1ull << 25;

// Appends one test to the chain; false when it is full, or when the run would
// no longer be one that kernels are made for, and has to be.
inline bool chain_add(FusedRun *f, const PredDev &p, uint32_t mul, bool sets_only) {
    if (f->chain.n == kChainMax) return false;
    PredChain c = f->chain;
    c.op[c.n].pred = p;
    c.op[c.n].mul = mul;
    c.n += 1;
    c.mul_all *= mul;
    if (sets_only && !chain_is_set(c)) return false;
    f->chain = c;
    return true;
}

// The longest run of at least two of the `count` stages that starts with the
// first and holds a test, as far as it can be issued as one kernel: no tile
// shape asked for, and an input that the chain kernels take (x; with the interleave
// in front also y; `capacity` entries each). stage(i) is stage i, usable(i) whether
// it may take part.
template <class Stage, class Usable>
FusedRun plan_run(const void *x, const void *y, uint64_t capacity, size_t count, Stage stage, Usable usable) {
    const FusedRun none;
    FusedRun f;
    f.chain.mul_all = 1u;
    if (count < 2 || !usable(0)) return none;
    size_t i = 0;
    uint64_t entries = capacity;
    if (stage(0).kind == KA_STAGE_PREPARE) {
        if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) & 15u) return none;
        if (!x || !y) return none;  // (the stage itself settles whether there is anything to read)
        f.inter = true;
        entries = 2 * capacity;
        ++i;
    }
    if (entries > kChainEntries) return none;
    const PredDev all = {kAll, 0, 0, 0};
    const bool sets_only = !f.inter && entries >= kSetsOnlyFrom;
    bool tests = false;
    while (i < count && usable(i)) {
        const RunStage st = stage(i);
        if (st.kind == KA_STAGE_MAP_HASH) {
            if (!chain_add(&f, all, kHashMul, sets_only)) break;
            i += 1;
        } else if (st.kind == KA_STAGE_COMPACT && !st.shaped) {
            if (!chain_add(&f, st.pred, st.mul, sets_only)) break;
            tests = true;
            i += 1;
        } else if (st.kind == KA_STAGE_PREDICATE && i + 2 < count && stage(i + 1).kind == KA_STAGE_EXSCAN &&
                   stage(i + 2).kind == KA_STAGE_SCATTER && usable(i + 1) && usable(i + 2) && !stage(i + 1).shaped) {
            if (!chain_add(&f, st.pred, 1u, sets_only)) break;
            tests = true;
            i += 3;
        } else {
            break;
        }
    }
    if (!tests || i < 2) return none;
    f.stages = int(i);
    return f;
}

}  // namespace ka
