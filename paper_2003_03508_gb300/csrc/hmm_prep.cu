// Parameter preparation and observation packing.
//
// prep (one CTA per proposal): checks a parameter set and turns it into the
// constants the later kernels read -- the emission coefficients of Eq.
// "emission-matrix" in the log2 domain, P padded to KP x KP, and the
// tensor-core operand images of P.
//
// pack: copies the observations of every segment into an aligned buffer the
// chunk kernels read in 64-step windows (x = NaN marks "no tremor"), and
// checks that every flagged tremor has a finite location.
#include <cuda_bf16.h>
#include <math.h>

#include "hmm_strand.cuh"

namespace hmm {

static int round_up(int x, int m) { return (x + m - 1) / m * m; }

ConstLayout make_layout(int K, int precision) {
    ConstLayout L{};
    int KP;
    if (precision == HMM_PREC_FP32_SIMT) {
        KP = K <= 4 ? 4 : K <= 8 ? 8 : K <= 16 ? 16 : K <= 32 ? 32 : round_up(K, 16);
    } else {
        KP = round_up(K < 16 ? 16 : K, 16);
    }
    L.KP = KP;
    L.off_emis = 0;
    L.off_p32 = round_up(EM_ALL * KP, 32);
    L.off_tc = round_up(L.off_p32 + KP * KP, 32);
    switch (precision) {
        case HMM_PREC_TF32: L.tc_floats = KP * KP; break;            // P_hi (tf32)
        case HMM_PREC_TF32_SPLIT: L.tc_floats = 2 * KP * KP; break;  // P_hi, P_lo (tf32)
        case HMM_PREC_BF16: L.tc_floats = KP * KP; break;            // P_hi, P_lo (bf16)
        default: L.tc_floats = 0;
    }
    L.stride = round_up(L.off_tc + L.tc_floats, 32);
    return L;
}

__device__ __forceinline__ float to_tf32(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return __uint_as_float(r);
}

// Offset (in elements) of B-operand element (n, k) in the canonical K-major,
// no-swizzle layout: 8-row x 16-byte core matrices, adjacent along K at
// 128 bytes, 8-row groups at (KP * esize / 16) * 128 bytes.
__device__ __forceinline__ int kmajor_offset(int n, int k, int KP, int elems16) {
    int sbo_elems = (KP / elems16) * 8 * elems16;  // one 8-row group spans all of K
    return (n >> 3) * sbo_elems + (k / elems16) * (8 * elems16) + (n & 7) * elems16 + (k % elems16);
}

constexpr int PREP_THREADS = 256;

// One proposal's constants, by one CTA. FP64 is two lanes per cycle and SM here,
// so the chain of a state's logarithms and square roots is spread over four
// threads (14 us for a lone proposal when one thread took them in turn).
__device__ __forceinline__ void prep_proposal(int q, int K, const ConstLayout &lay, int precision,
                                              const float *__restrict__ pi, const float *__restrict__ P,
                                              const float *__restrict__ p, const float *__restrict__ mu,
                                              const float *__restrict__ cov, float *__restrict__ cblock,
                                              int *__restrict__ prop_bad, unsigned *__restrict__ status,
                                              const StrandPtrs &sp) {
    const int KP = lay.KP;
    pi += (size_t)q * K;
    P += (size_t)q * K * K;
    p += (size_t)q * K;
    mu += (size_t)q * 2 * K;
    cov += (size_t)q * 3 * K;
    float *cb = cblock + (size_t)q * lay.stride;
    float *em = cb + lay.off_emis;
    __shared__ float s_ctr[80], s_cno[80], s_centre[2];
    __shared__ double s_ctr64[80], s_quiet[80];
    const int lane = threadIdx.x & 31;
    bool bad = false, small = false, far = false;

    // per-state emission constants (log2 domain), padded states emit nothing
    const double LOG2E = 1.4426950408889634074;
    const double LOG2_2PI = 2.6514961294723187980;
    const int job = threadIdx.x >> 6;
    float cx = 0.0f, cy = 0.0f;
    if (job == 3) {
        // the states' centre: the affine forms take coordinates from it
        for (int k = lane; k < K; k += 32) {
            cx += mu[2 * k] / (float)K;
            cy += mu[2 * k + 1] / (float)K;
        }
        for (int o = 16; o > 0; o >>= 1) {
            cx += __shfl_xor_sync(0xffffffffu, cx, o);
            cy += __shfl_xor_sync(0xffffffffu, cy, o);
        }
        if (threadIdx.x == 192) {
            s_centre[0] = cx;
            s_centre[1] = cy;
        }
    }
    for (int k = threadIdx.x & 63; k < KP; k += 64) {
        const bool in = k < K;
        const double pk = in ? p[k] : 0.0;
        const double sxx = in ? cov[3 * k] : 1.0, sxy = in ? cov[3 * k + 1] : 0.0, syy = in ? cov[3 * k + 2] : 1.0;
        const double det = sxx * syy - sxy * sxy;
        const float mx = in ? mu[2 * k] : 0.0f, my = in ? mu[2 * k + 1] : 0.0f;
        const bool ok = isfinite(pk) && pk >= 0.0 && pk <= 1.0 && isfinite(sxx) && isfinite(sxy) && isfinite(syy) &&
                        sxx > 0.0 && syy > 0.0 && det > 0.0 && isfinite(mx) && isfinite(my);
        if (!ok) bad = true;
        const bool use = in && ok;
        if (job == 0) {
            em[EM_MUX * KP + k] = use ? mx : 0.0f;
            em[EM_MUY * KP + k] = use ? my : 0.0f;
            const double inv = LOG2E / det;
            em[EM_QA * KP + k] = use ? (float)(-0.5 * syy * inv) : 0.0f;
            em[EM_QB * KP + k] = use ? (float)(sxy * inv) : 0.0f;
            em[EM_QC * KP + k] = use ? (float)(-0.5 * sxx * inv) : 0.0f;
        } else if (job == 1) {
            const double v64 = use ? 0.5 * log2(pk * pk / det) - LOG2_2PI : -INFINITY;
            const float v = (float)v64;
            em[EM_CTR * KP + k] = v;
            s_ctr[k] = v;
            s_ctr64[k] = v64;
        } else if (job == 2) {
            const float v = use ? (float)log2(1.0 - pk) : -INFINITY;
            em[EM_CNO * KP + k] = v;
            s_cno[k] = v;
            s_quiet[k] = use ? 1.0 - pk : 0.0;
        } else {
            // the quadratic form as two squares (Cholesky factor of the precision matrix)
            const double ux = use ? sqrt(0.5 * LOG2E * syy / det) : 0.0, wy = use ? sqrt(0.5 * LOG2E / syy) : 0.0;
            const double uy = use ? -ux * sxy / syy : 0.0, dx = (double)mx - cx, dy = (double)my - cy;
            em[EM_UX * KP + k] = (float)ux;
            em[EM_UY * KP + k] = (float)uy;
            em[EM_WY * KP + k] = (float)wy;
            em[EM_U0 * KP + k] = use ? (float)-(ux * dx + uy * dy) : 0.0f;
            em[EM_W0 * KP + k] = use ? (float)(-wy * dy) : 0.0f;
            far = far || (use && !(fabs(ux * dx) + fabs(uy * dy) <= EMIS_NEAR && fabs(wy * dy) <= EMIS_NEAR));
        }
    }
    // rows of P and pi: non-negative, finite, summing to 1 within 1e-5 (a warp
    // per row; row K is pi)
    for (int i = threadIdx.x >> 5; i <= K; i += PREP_THREADS / 32) {
        const float *row = i < K ? P + i * K : pi;
        double s = 0.0;
        bool ok = true, tiny = false;
        for (int j = lane; j < K; j += 32) {
            const float v = row[j];
            ok = ok && isfinite(v) && v >= 0.0f;
            tiny = tiny || v < STRAND_PMIN;
            s += v;
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        bad = bad || !ok || !(fabs(s - 1.0) <= 1e-5);
        small = small || (i < K && tiny);
    }
    // P padded to KP x KP (FP32, row-major) and the tensor-core images
    for (int idx = threadIdx.x; idx < KP * KP; idx += PREP_THREADS) {
        int i = idx / KP, j = idx % KP;
        float v = (i < K && j < K) ? P[i * K + j] : 0.0f;
        cb[lay.off_p32 + idx] = v;
        // B operand is P itself: B[k = i][n = j]
        if (precision == HMM_PREC_TF32 || precision == HMM_PREC_TF32_SPLIT) {
            float hi = to_tf32(v);
            cb[lay.off_tc + kmajor_offset(j, i, KP, 4)] = hi;
            if (precision == HMM_PREC_TF32_SPLIT)
                cb[lay.off_tc + KP * KP + kmajor_offset(j, i, KP, 4)] = to_tf32(v - hi);
        } else if (precision == HMM_PREC_BF16) {
            __nv_bfloat16 *img = reinterpret_cast<__nv_bfloat16 *>(cb + lay.off_tc);
            __nv_bfloat16 hi = __float2bfloat16_rn(v);
            __nv_bfloat16 lo = __float2bfloat16_rn(v - __bfloat162float(hi));
            img[kmajor_offset(j, i, KP, 8)] = hi;
            img[KP * KP + kmajor_offset(j, i, KP, 8)] = lo;
        }
    }
    bad = __syncthreads_or(bad);
    small = __syncthreads_or(small);
    far = __syncthreads_or(far);
    if (threadIdx.x < 32) {
        // EM_OFF: the emissions' largest constants, rounded up to whole numbers
        float mt = -INFINITY, mn = -INFINITY;
        for (int k = lane; k < K; k += 32) {
            mt = fmaxf(mt, s_ctr[k]);
            mn = fmaxf(mn, s_cno[k]);
        }
        for (int o = 16; o > 0; o >>= 1) {
            mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, o));
            mn = fmaxf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        }
        mt = isfinite(mt) ? ceilf(mt) : 0.0f;
        mn = isfinite(mn) ? ceilf(mn) : 0.0f;
        // The strands' constants, rounded once from 64 bits. EX2_BIAS: what
        // ex2.approx loses in the mean, for arguments below 0 as all are here
        // (-5.0e-8 of its value, measured), spread over the states by the rounding.
        // The quiet steps' factor is no exponential at all: that loss, the same at
        // every quiet step, was most of log L's error (rare tremors: 6.0e-8 of it).
        constexpr double EX2_BIAS = 7.2e-8;
        for (int k = lane; k < KP; k += 32) {
            em[EM_SC * KP + k] = (float)((double)mt - s_ctr64[k] - EX2_BIAS);
            em[EM_QF * KP + k] = (float)(s_quiet[k] * (double)pow2f(-(int)mn));
        }
        if (lane == 0) {
            em[EM_OFF * KP] = mt;
            em[EM_OFF * KP + 1] = mn;
            if (KP >= 16) {
                em[EM_OFF * KP + 2] = s_centre[0];
                em[EM_OFF * KP + 3] = s_centre[1];
                em[EM_OFF * KP + 4] = far ? 0.0f : 1.0f;
            }
            prop_bad[q] = bad;
            if (bad) atomicOr(status, ST_EINVAL);
            if (sp.route) {
                // strands need P's entries above STRAND_PMIN and constants of ordinary size
                const bool fits = !small && fabsf(mt) <= 1000.0f && fabsf(mn) <= 1000.0f;
                sp.route[q] = bad ? ROUTE_BAD : ROUTE_STRANDS;
                sp.jumps[q] = 0;
                sp.spent[q] = 0;
                if (bad ? sp.bad_too : !fits) {
                    sp.route[q] = ROUTE_CHUNKS;
                    sp.todo[1 + atomicAdd(&sp.todo[0], 1)] = q;
                }
            }
        }
    }
}

// One thread per observation; the segment is found by binary search.
__device__ __forceinline__ void pack_observations(int block, int blocks, int n_seg, const int64_t *__restrict__ offs,
                                                  const int64_t *__restrict__ pbase, int64_t T_total,
                                                  const float2 *__restrict__ xy, const uint8_t *__restrict__ tremor,
                                                  float2 *__restrict__ packed, float2 *__restrict__ head,
                                                  int *__restrict__ obs_bad, unsigned *__restrict__ status) {
    for (int64_t t = block * (int64_t)PREP_THREADS + threadIdx.x; t < T_total; t += (int64_t)blocks * PREP_THREADS) {
        int lo = 0, hi = n_seg - 1;  // last s with offs[s] <= t
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (offs[mid] <= t) lo = mid; else hi = mid - 1;
        }
        // skip empty segments that share the offset
        int s = lo;
        float2 v = xy[t];
        bool tr = tremor[t] != 0;
        if (tr && !(isfinite(v.x) && isfinite(v.y))) {
            *obs_bad = 1;
            atomicOr(status, ST_EINVAL);
        }
        float2 o = tr ? v : make_float2(__int_as_float(0x7fc00000), 0.0f);
        int64_t u = t - offs[s];
        if (u == 0) head[s] = o;
        else packed[pbase[s] + u - 1] = o;
    }
}

// Both in one launch: the first n_prop CTAs take a proposal each, the rest the
// observations.
__global__ void __launch_bounds__(PREP_THREADS)
prep_pack_kernel(int n_prop, int K, ConstLayout lay, int precision, const float *__restrict__ pi,
                 const float *__restrict__ P, const float *__restrict__ p, const float *__restrict__ mu,
                 const float *__restrict__ cov, float *__restrict__ cblock, int *__restrict__ prop_bad,
                 StrandPtrs sp, int n_seg, const int64_t *__restrict__ offs, const int64_t *__restrict__ pbase,
                 int64_t T_total, const float2 *__restrict__ xy, const uint8_t *__restrict__ tremor,
                 float2 *__restrict__ packed, float2 *__restrict__ head, int *__restrict__ obs_bad,
                 unsigned *__restrict__ status) {
    if ((int)blockIdx.x < n_prop)
        prep_proposal(blockIdx.x, K, lay, precision, pi, P, p, mu, cov, cblock, prop_bad, status, sp);
    else
        pack_observations(blockIdx.x - n_prop, gridDim.x - n_prop, n_seg, offs, pbase, T_total, xy, tremor, packed,
                          head, obs_bad, status);
}

cudaError_t launch_prep_pack(int n_prop, int K, const ConstLayout &lay, int precision, const float *pi,
                             const float *P, const float *p, const float *mu, const float *cov, float *cblock,
                             int *prop_bad, const StrandPtrs &sp, int n_seg, const int64_t *d_offsets,
                             const int64_t *d_pbase, int64_t T_total, const float *xy, const uint8_t *tremor,
                             float2 *packed, float2 *head, int *obs_bad, unsigned *status, cudaStream_t st) {
    int64_t blocks = (T_total + PREP_THREADS - 1) / PREP_THREADS;
    if (blocks > 152 * 16) blocks = 152 * 16;
    prep_pack_kernel<<<(unsigned)(n_prop + blocks), PREP_THREADS, 0, st>>>(
        n_prop, K, lay, precision, pi, P, p, mu, cov, cblock, prop_bad, sp, n_seg, d_offsets, d_pbase, T_total,
        reinterpret_cast<const float2 *>(xy), tremor, packed, head, obs_bad, status);
    return cudaGetLastError();
}

}  // namespace hmm
