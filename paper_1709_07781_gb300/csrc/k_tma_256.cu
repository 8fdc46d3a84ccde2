// Kernels of the TMA tile shape (256, 16): the compaction for every predicate
// kind and the scan (see ka_tma_pass.cuh).
#include "ka_tma_pass.cuh"

namespace ka {
namespace tma {

ka_status launch_tma_256(const TmaArgs &a, bool scan, int32_t pk, uint64_t cap, cudaStream_t stream) {
    if (scan) return launch_scan_config<8, 4, 2, 480, 3>(a, cap, stream);
    return launch_compact_config<8, 2, 4, 2, 480, 3, 4, 1>(a, pk, cap, stream);
}

}  // namespace tma
}  // namespace ka
