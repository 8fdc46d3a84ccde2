// Compaction kernels of the TMA tile shape (768, 16) made for a set of two to
// four tests, as many as a chain holds (see k_compact_tma.cu); one of four files.
#include "ka_tma_pass.cuh"

namespace ka {
namespace tma {

ka_status launch_sets_768_a(const TmaArgs &a, int mask, uint64_t cap, cudaStream_t stream) {
    switch (mask) {
#define KA_CASE(M) \
    case M: return launch_compact_shape<kSetKind + M, 22, 3, 5, 3, 160, 1, 16, 3>(a, cap, stream);
        KA_CASE(3)
        KA_CASE(9)
        KA_CASE(13)
        KA_CASE(18)
        KA_CASE(22)
        KA_CASE(26)
        KA_CASE(30)
#undef KA_CASE
    default: return KA_E_UNSUPPORTED;
    }
}

}  // namespace tma
}  // namespace ka
