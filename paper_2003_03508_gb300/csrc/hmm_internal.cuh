// Internal declarations shared by the library's translation units.
//
// Data layout in HBM (per call, carved out of one context-owned workspace):
//   cblock  [n_prop][cstride] f32  per-proposal constants written by the prep
//                                  kernel: emission coefficients (log2 domain,
//                                  EM_ALL x KP SoA), P padded to KP x KP in FP32,
//                                  and the tensor-core operand images of P.
//   packed  [n_packed] float2      chain observations x_1..x_{T-1} of every
//                                  segment, each segment starting on a
//                                  64-step boundary; x = NaN marks "no tremor".
//   head    [n_seg] float2         first observation x_0 of each segment.
//   chunks  [n_chunks] ChunkDesc   chunk table shared by all proposals.
//   A0/e0   [n_prop][n_chunks]     chunk products (KP x KP f32) and per-row
//                                  int32 power-of-two exponents.
//   A_l/e_l levels of the product tree (int64 exponents).
//   strands                        StrandPtrs: two vectors, exponent and scale per
//                                  strand and proposal, the routes and the list
//                                  of proposals left to the chunk products.
//   qtab/qexp [n_prop][nb] run-length shortcut table (KP x KP f32 and KP int32
//                                  row exponents per power), only when it is on.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "hmm_gb300.h"

namespace hmm {

// device status word bits
enum : unsigned {
    ST_EINVAL = 1u,
    ST_ENUMERIC = 2u,
    ST_ETIMEOUT = 4u,
};

// emission coefficient rows in the const block (each row is KP floats)
enum {
    EM_MUX = 0,
    EM_MUY = 1,
    EM_QA = 2,   // -0.5 log2(e) syy / det
    EM_QB = 3,   //      log2(e) sxy / det
    EM_QC = 4,   // -0.5 log2(e) sxx / det
    EM_CTR = 5,  // log2 p - log2(2 pi) - 0.5 log2 det
    EM_CNO = 6,  // log2 (1 - p)
    EM_ROWS = 8,
    // the strands' form of the same density (hmm_strand.cuh)
    EM_OFF = 8,  // [0], [1]: whole numbers next above the row maxima of EM_CTR and EM_CNO; with 16 states and more
                 // [2], [3]: the states' centre, [4]: 1 where the affine forms serve (hmm_strand.cuh), else 0
    EM_UX = 9,   // u = ux dx + uy dy, w = wy dy, from the mean: log2 density = ctr - u^2 - w^2
    EM_UY = 10,
    EM_WY = 11,
    EM_U0 = 12,  // u = ux x + uy y + u0, w = wy y + w0, from the centre
    EM_W0 = 13,
    EM_SC = 14,  // the strands' offset [0] - log2 constant of a tremor
    EM_QF = 15,  // and their factor of a step without one: (1 - p) 2^-offset [1]
    EM_ALL = 16,
};

// a step whose best state has log2-emission below -EXP_LIMIT is not representable
// (keeps a chunk's exponent sum, <= 16384 steps, inside int32)
constexpr int EXP_LIMIT = 1 << 16;
// exponent recorded for an all-zero row (its scale is irrelevant); the tree
// aligns rows to the largest exponent, so zero rows must never win that max
constexpr int32_t ZERO_ROW_EXP32 = INT32_MIN;
constexpr long long ZERO_ROW_EXP64 = -(1LL << 62);
constexpr int MAX_LEVELS = 10;
constexpr int TREE_GROUP = 16;
constexpr int OBS_WIN = 64;   // steps per observation window; chunk lengths are multiples

struct ChunkDesc {
    int64_t pstart;  // index of the chunk's first step in `packed`
    int32_t len;     // steps in this chunk (1..L)
    int32_t seg;     // segment it belongs to
};

// One strand: the forward vector of one proposal carried over `len` steps of a
// segment (hmm_strand.cuh). It starts `warm` steps earlier, from a flat vector
// or, when that reaches the segment's start, from the head vector.
struct StrandDesc {
    int64_t pstart;  // index of the piece's first step in `packed` (a multiple of OBS_WIN)
    int32_t len;     // steps in the piece (>= 1)
    int32_t warm;    // steps run before the piece (a multiple of OBS_WIN)
    int32_t seg;     // segment it belongs to
    int32_t flags;   // SD_HEAD (starts at the head vector), SD_FIRST, SD_LAST (of its segment)
};
enum { SD_HEAD = 1, SD_FIRST = 2, SD_LAST = 4 };

// How a proposal's log L is formed (route[q]): by strands, by chunk products
// (listed in todo[1..], todo[0] of them), or not at all (invalid parameters)
enum { ROUTE_STRANDS = 0, ROUTE_CHUNKS = 1, ROUTE_BAD = 2 };

struct StrandPtrs {
    const StrandDesc *desc = nullptr;  // [n], by segment and position
    const int32_t *order = nullptr;    // [n], longest first: the warps' order
    int n = 0;
    float *vs = nullptr;       // [n_prop][n][KP] vector at the piece's start
    float *ve = nullptr;       // [n_prop][n][KP] vector at its end
    long long *ex = nullptr;   // [n_prop][n] power-of-two exponent of ve relative to vs
    double *logr = nullptr;    // [n_prop][n] log scale of the true vector over the strand of piece `jump`
    int *jump = nullptr;       // [n_prop][n] piece where the vectors met: itself, a later one, or -1 (at the segment's end)
    int *jumps = nullptr;      // [n_prop] some piece's jump is not itself
    int *route = nullptr;      // [n_prop]
    int *todo = nullptr;       // [1 + n_prop]
    int *spent = nullptr;      // [n_prop] steps that the proposal's joins have run on
    int most = 0;              // how many a join may run on,
    int budget = 0;            // and a proposal's together, before the chunk products are the quicker way
    bool bad_too = false;      // invalid parameters take the chunk products as well (they fill every output)
};

// The posterior of one sequence by strands (hmm_smooth.cu). Row t belongs to
// observation t; u's row t to the step from t to t + 1.
constexpr int SMOOTH_PARTS = 456;  // partial sums of the E-step statistics
struct SmoothPtrs {
    int warm = 0;              // warm-up steps of the backward strands
    int most = 0;              // steps of the pieces that a chain of rows may pass
    float *alpha = nullptr;    // [T][KP] forward vectors, any scale (null: no posterior)
    float *gamma = nullptr;    // [T][K]
    float *u = nullptr;        // [T][KP] d o b / S of every step (null: no statistics)
    float *bs = nullptr;       // [n][KP] backward vector at the piece's end
    float *be = nullptr;       // [n][KP] and at its start
    float *carry = nullptr;    // [n][KP] true vector where a piece ended unmet
    int *unmet = nullptr;      // [n] 2 x rows written again, + 1 where the piece ended first
    double *part = nullptr;    // [SMOOTH_PARTS][K K + 7 K]
    double *g0 = nullptr;      // [K]
    double *stats = nullptr;   // K K + 8 K, as hmm_expected_stats
};

// The most probable path by strands (hmm_vit_strand.cu). Row i belongs to step i.
struct VitPtrs {
    int most = 0;              // steps of the pieces that a chain may pass
    float *lp = nullptr;       // [KP][KP] log2 P
    double *lp64 = nullptr;    // [KP][KP] log P
    double *em64 = nullptr;    // [K][8] emission constants of the score
    float *vs = nullptr;       // [n][KP] vector at the piece's start
    float *ve = nullptr;       // [n][KP] and at its end
    float *carry = nullptr;    // [n][KP] true vector where a piece ended unmet
    int *unmet = nullptr;      // [n] 2 x rows written again, + 1 where the piece ended first
    int *bstate = nullptr;     // [n] state at the piece's end
    uint8_t *map = nullptr;    // [n][KP] leaving state -> state before the piece
    uint8_t *bp = nullptr;     // [steps][KP] back-pointers
    double *part = nullptr;    // [n] the pieces' parts of the score
    int *chunks = nullptr;     // set: the chunk products take the sequence
};

struct ConstLayout {
    int KP;         // padded state count used by the chunk kernel
    int off_emis;   // EM_ALL * KP floats
    int off_p32;    // KP * KP floats, row-major, zero padded
    int off_tc;     // tensor-core B-operand images (path dependent)
    int tc_floats;  // size of the tensor-core section
    int stride;     // floats per proposal (multiple of 32)
};

struct TreeGroup {
    int32_t src;  // first matrix (index within one proposal's level buffer)
    int32_t cnt;  // matrices to multiply, in order
    int32_t dst;  // output index in the next level
    int32_t pad;
};

struct SegFinal {
    int64_t T;      // observations in the segment
    int32_t level;  // level holding the segment's product (-1: no product)
    int32_t idx;    // index within one proposal's slice of that level
};

struct LevelPtrs {
    float *A[MAX_LEVELS];
    void *e[MAX_LEVELS];     // level 0: int32, others: int64
    int32_t n[MAX_LEVELS];   // matrices per proposal at each level
};

// ---------------- small device helpers ----------------

// floor(log2(m)) for a positive normal float, as the exponent field.
__device__ __forceinline__ int float_exponent(float m) {
    return ((__float_as_int(m) >> 23) & 0xff) - 127;
}

// 2^k as a float for k in [-126, 127]
__device__ __forceinline__ float pow2f(int k) {
    return __int_as_float((k + 127) << 23);
}

// log2 of the emission of state k for observation (x, y) (Eq. "emission-matrix").
__device__ __forceinline__ float log2_emission(const float *__restrict__ em, int KP, int k,
                                               float x, float y, bool tremor) {
    if (!tremor) return em[EM_CNO * KP + k];
    float dx = x - em[EM_MUX * KP + k];
    float dy = y - em[EM_MUY * KP + k];
    float acc = em[EM_CTR * KP + k];
    acc = fmaf(em[EM_QC * KP + k] * dy, dy, acc);
    acc = fmaf(em[EM_QB * KP + k] * dx, dy, acc);
    acc = fmaf(em[EM_QA * KP + k] * dx, dx, acc);
    return acc;
}

// ---------------- launchers (host side, one per translation unit) ----------------

ConstLayout make_layout(int K, int precision);

cudaError_t launch_prep_pack(int n_prop, int K, const ConstLayout &lay, int precision, const float *pi,
                             const float *P, const float *p, const float *mu, const float *cov, float *cblock,
                             int *prop_bad, const StrandPtrs &sp, int n_seg, const int64_t *d_offsets,
                             const int64_t *d_pbase, int64_t T_total, const float *xy, const uint8_t *tremor,
                             float2 *packed, float2 *head, int *obs_bad, unsigned *status, cudaStream_t st);

cudaError_t launch_chunk_simt(int n_prop, int n_chunks, int L, int renorm, const ConstLayout &lay,
                              const float *cblock, const ChunkDesc *chunks, const float2 *packed,
                              float *A0, int32_t *e0, unsigned *status, const int *todo, cudaStream_t st);

// Strands (hmm_strand_simt.cu) and their join (hmm_join.cu). strand_simt_kp: the
// padded state count (0: K too large).
int strand_simt_kp(int K);
int strand_simt_per_warp(int KP);
cudaError_t launch_strand_simt(int n_prop, int K, int init_mode, const ConstLayout &lay,
                               const float *cblock, const float *pi, const float2 *head, const float2 *packed,
                               const StrandPtrs &sp, float *alpha, cudaStream_t st);
cudaError_t launch_smooth(int K, int KP, int64_t steps, const ConstLayout &lay, const float *cblock, const float2 *head,
                          const float2 *packed, const StrandPtrs &sp, const SmoothPtrs &sm, cudaStream_t st);
cudaError_t launch_vit_strands(int K, int KP, int init_mode, const ConstLayout &lay, const float *cb, const float *pi,
                               const float *P, const float *p, const float *mu, const float *cov, const float2 *head,
                               const float2 *packed, const StrandPtrs &sp, const VitPtrs &vp, int32_t *path,
                               double *score, cudaStream_t st);
int strand_mma_per_warp(int KP);
cudaError_t launch_strand_mma(int n_prop, int K, int init_mode, const ConstLayout &lay, int precision,
                              const float *cblock, const float *pi, const float2 *head, const float2 *packed,
                              const StrandPtrs &sp, cudaStream_t st);
// beyond 32 states: the proposals whose emissions take the affine forms, and the others
cudaError_t launch_strand_mma_near(int n_prop, int K, int init_mode, const ConstLayout &lay, int precision,
                                   const float *cblock, const float *pi, const float2 *head, const float2 *packed,
                                   const StrandPtrs &sp, cudaStream_t st);
cudaError_t launch_strand_mma_far(int n_prop, int K, int init_mode, const ConstLayout &lay, int precision,
                                  const float *cblock, const float *pi, const float2 *head, const float2 *packed,
                                  const StrandPtrs &sp, cudaStream_t st);
cudaError_t launch_join(int n_prop, int K, int KP, const ConstLayout &lay, int precision, bool tensor, const float *cblock,
                        const float2 *packed, const StrandPtrs &sp, cudaStream_t st);

// The chunk-product kernels and the tree take a list of the proposals to work
// on, todo[0] of them in todo[1..] (null: all n_prop).

// run-length shortcut (FP32 on the CUDA cores): table of M_0^(2^b), b < nb,
// then chunk products that apply runs of >= min_run no-tremor steps from it
int rle_levels(int L);
cudaError_t launch_rle_table(int n_prop, int nb, const ConstLayout &lay, const float *cblock, float *qtab,
                             int32_t *qexp, unsigned *status, const int *todo, cudaStream_t st);
cudaError_t launch_chunk_rle(int n_prop, int n_chunks, int renorm, int min_run, int nb, const ConstLayout &lay,
                             const float *cblock, const float *qtab, const int32_t *qexp, const ChunkDesc *chunks,
                             const float2 *packed, float *A0, int32_t *e0, unsigned *status, const int *todo, cudaStream_t st);

bool chunk_tc_supported(int K, int precision);
int chunk_tc_chunks_per_item(int KP, int precision);
cudaError_t launch_posterior(int K, int KP, int init_mode, int n_chunks, int L, const ChunkDesc *chunks,
                             const float *pi, const float *P, const float *em, const float2 *head,
                             const float2 *packed, const float *A0, const int32_t *e0, float *fvec, float *bvec,
                             float *gamma, double *stats_part, double *g0, double *stats, const int *todo,
                             cudaStream_t st);
int chunk_tc_wide_chunks_per_item(int KP, int precision);
cudaError_t launch_viterbi(int K, int init_mode, int n_chunks, int L, const ConstLayout &lay, const ChunkDesc *chunks,
                           const float *pi, const float *P, const float *cblock, const float2 *head,
                           const float2 *packed, float *V, double *voff, int32_t *ptr, int32_t *bstate, uint8_t *bp,
                           int32_t *path, double *score, const int *todo, cudaStream_t st);
cudaError_t launch_chunk_tc_wide(int n_prop, int n_chunks, int renorm, int precision, const ConstLayout &lay,
                                 const float *cblock, const ChunkDesc *chunks, const float2 *packed, float *A0,
                                 int32_t *e0, unsigned *status, const int *todo, cudaStream_t st);
cudaError_t launch_chunk_tc(int n_prop, int n_chunks, int L, int renorm, int precision,
                            const ConstLayout &lay, const float *cblock, const ChunkDesc *chunks,
                            const float2 *packed, float *A0, int32_t *e0, unsigned *status,
                            const int *todo, cudaStream_t st);

// Fisher-identity gradient and EM M-step from the E-step statistics (hmm_grad.cu)
cudaError_t launch_fisher_grad(int K, int init_mode, const float *pi, const float *P, const float *p, const float *mu,
                               const float *cov, const double *stats, double *grad, cudaStream_t st);
cudaError_t launch_em_mstep(int K, const float *pi, const float *P, const float *p, const float *mu, const float *cov,
                            const double *stats, float *pi_out, float *P_out, float *p_out, float *mu_out,
                            float *cov_out, cudaStream_t st);

cudaError_t launch_tree_level(int n_prop, int KP, int level, int n_groups, const TreeGroup *groups,
                              const LevelPtrs &lv, unsigned *status, const int *todo, cudaStream_t st);

cudaError_t launch_final(int n_prop, int K, int init_mode, int n_seg, const SegFinal *segs,
                         const float2 *head, const LevelPtrs &lv, int KP, const float *pi,
                         const float *P, const float *p, const float *mu, const float *cov,
                         const int *prop_bad, const int *obs_bad, double *out, const StrandPtrs &sp, int strand_kp, cudaStream_t st);

}  // namespace hmm
