// laq_gemm_batch.cu -- the batch GEMM kernel's plain-X instances, compiled apart from the general
// kernel's so that the sets build in parallel.
#include "laq_gemm_batch.cuh"

namespace laq {

const void* gemm_batch_plain_kernel(int bits, int nb, int tw) {
    return bits == 4 ? pick_batch<4, false>(nb, tw) : pick_batch<3, false>(nb, tw);
}

}  // namespace laq
