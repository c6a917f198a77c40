// laq_gemm_prologue.cu -- the GEMM kernel instances whose X staging applies a fused prologue
// (RMSNorm of the residual sum, or SiLU(gate) * up), compiled apart from the plain instances so
// the two sets build in parallel.
#include "laq_gemm_batch.cuh"

namespace laq {

const void* gemm_prologue_kernel(int bits, int mp, int nt) {
    return bits == 4 ? pick_mp<4, true>(mp, nt) : pick_mp<3, true>(mp, nt);
}

const void* gemm_batch_prologue_kernel(int bits, int nb, int tw) {
    return bits == 4 ? pick_batch<4, true>(nb, tw) : pick_batch<3, true>(nb, tw);
}

}  // namespace laq
