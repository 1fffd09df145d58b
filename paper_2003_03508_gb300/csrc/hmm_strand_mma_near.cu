// Strands on the tensor cores, 48 to 80 states, with the affine emission forms
// (hmm_strand_mma.cuh).
#include "hmm_strand_mma.cuh"

namespace hmm {

cudaError_t launch_strand_mma_near(int n_prop, int K, int init_mode, const ConstLayout &lay, int precision,
                                   const float *cblock, const float *pi, const float2 *head, const float2 *packed,
                                   const StrandPtrs &sp, cudaStream_t st) {
    switch (lay.KP) {
        case 48: return launch_kp<48, F_NEAR>(n_prop, K, init_mode, lay, precision, cblock, pi, head, packed, sp, st);
        case 64: return launch_kp<64, F_NEAR>(n_prop, K, init_mode, lay, precision, cblock, pi, head, packed, sp, st);
        case 80: return launch_kp<80, F_NEAR>(n_prop, K, init_mode, lay, precision, cblock, pi, head, packed, sp, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace hmm
