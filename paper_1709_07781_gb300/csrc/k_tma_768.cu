// Kernels of the TMA tile shape (768, 16) (see ka_tma_pass.cuh). Compaction: 22
// compute warps (tiles of 11264 entries), five tiles of shared memory (220
// KiB), the largest tile for which five fit: as a ring kernel three stages and
// 1024 ring words a warp, as a hold kernel five stages, two in flight. 16 tile
// slots (against 8: 164 against 168 us at 1 % kept and N = 2^28). Scan: 26
// compute warps, four stages.
#include "ka_tma_pass.cuh"

namespace ka {
namespace tma {

ka_status launch_tma_768(const TmaArgs &a, bool scan, int32_t pk, uint64_t cap, cudaStream_t stream) {
    if (scan) return launch_scan_config<26, 4, 3, 160, 1>(a, cap, stream);
    return launch_compact_config<22, 3, 5, 3, 160, 1, 16, 3>(a, pk, cap, stream);
}

ka_status launch_chain_768(const TmaArgs &a, uint64_t cap, cudaStream_t stream) {
    return launch_chain_config<22, 3, 5, 3, 160, 1, 16, 3>(a, cap, stream);
}

}  // namespace tma
}  // namespace ka
