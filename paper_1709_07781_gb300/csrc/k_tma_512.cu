// Kernels of the TMA tile shape (512, 16): the compaction for every predicate
// kind and the scan (see ka_tma_pass.cuh).
#include "ka_tma_pass.cuh"

namespace ka {
namespace tma {

ka_status launch_tma_512(const TmaArgs &a, bool scan, int32_t pk, uint64_t cap, cudaStream_t stream) {
    if (scan) return launch_scan_config<16, 3, 2, 320, 2>(a, cap, stream);
    return launch_compact_config<16, 2, 3, 2, 320, 2, 4, 1>(a, pk, cap, stream);
}

ka_status launch_chain_512(const TmaArgs &a, uint64_t cap, cudaStream_t stream) {
    return launch_chain_config<16, 2, 3, 2, 320, 2, 4, 1>(a, cap, stream);
}

}  // namespace tma
}  // namespace ka
