// Compaction kernels of the TMA tile shape (768, 16) for one test on the
// interleave of two arrays (see ka_tma_pass.cuh).
#include "ka_tma_pass.cuh"

namespace ka {
namespace tma {

ka_status launch_inter_768(const TmaArgs &a, int32_t pk, uint64_t cap, cudaStream_t stream) {
    return launch_compact_config<22, 3, 5, 3, 160, 1, 16, 3, true>(a, pk, cap, stream);
}

}  // namespace tma
}  // namespace ka
