// Strands on the tensor cores up to 32 states, and the choice by padded count
// (hmm_strand_mma.cuh; the wider ones are in hmm_strand_mma_near.cu and _far.cu, so
// that all compile side by side).
#include "hmm_strand_mma.cuh"

namespace hmm {

int strand_mma_per_warp(int KP) { return KP <= 32 ? 16 : 32; }

cudaError_t launch_strand_mma(int n_prop, int K, int init_mode, const ConstLayout &lay, int precision,
                              const float *cblock, const float *pi, const float2 *head, const float2 *packed,
                              const StrandPtrs &sp, cudaStream_t st) {
    if (sp.n == 0) return cudaSuccess;
    switch (lay.KP) {
        case 16: return launch_kp<16, F_BOTH>(n_prop, K, init_mode, lay, precision, cblock, pi, head, packed, sp, st);
        case 32: return launch_kp<32, F_BOTH>(n_prop, K, init_mode, lay, precision, cblock, pi, head, packed, sp, st);
        default: break;
    }
    const cudaError_t e = launch_strand_mma_near(n_prop, K, init_mode, lay, precision, cblock, pi, head, packed, sp, st);
    return e != cudaSuccess ? e : launch_strand_mma_far(n_prop, K, init_mode, lay, precision, cblock, pi, head, packed, sp, st);
}

}  // namespace hmm
