// Parameter preparation and observation packing.
//
// prep (one CTA per proposal): checks a parameter set and turns it into the
// constants the chunk kernels read -- the emission coefficients of Eq.
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

__global__ void __launch_bounds__(PREP_THREADS) prep_kernel(int K, ConstLayout lay, int precision, const float *__restrict__ pi,
                            const float *__restrict__ P, const float *__restrict__ p,
                            const float *__restrict__ mu, const float *__restrict__ cov,
                            float *__restrict__ cblock, int *__restrict__ prop_bad,
                            unsigned *__restrict__ status, StrandPtrs sp) {
    const int q = blockIdx.x;
    const int KP = lay.KP;
    pi += (size_t)q * K;
    P += (size_t)q * K * K;
    p += (size_t)q * K;
    mu += (size_t)q * 2 * K;
    cov += (size_t)q * 3 * K;
    float *cb = cblock + (size_t)q * lay.stride;
    __shared__ int bad, small;
    __shared__ float centre[2];
    if (threadIdx.x == 0) bad = small = 0;
    if (threadIdx.x < 32) {
        // the states' centre: the strands take coordinates from it
        float sx = 0.0f, sy = 0.0f;
        for (int k = threadIdx.x; k < K; k += 32) {
            sx += mu[2 * k] / (float)K;
            sy += mu[2 * k + 1] / (float)K;
        }
        for (int o = 16; o > 0; o >>= 1) {
            sx += __shfl_xor_sync(0xffffffffu, sx, o);
            sy += __shfl_xor_sync(0xffffffffu, sy, o);
        }
        if (threadIdx.x == 0) {
            centre[0] = sx;
            centre[1] = sy;
        }
    }
    __syncthreads();

    // rows of P and pi: non-negative, finite, summing to 1 within 1e-5 (a warp
    // per row; row K is pi)
    for (int i = threadIdx.x >> 5; i <= K; i += blockDim.x >> 5) {
        const float *row = i < K ? P + i * K : pi;
        const int lane = threadIdx.x & 31;
        double s = 0.0;
        bool ok = true, tiny = false;
        for (int j = lane; j < K; j += 32) {
            const float v = row[j];
            ok = ok && isfinite(v) && v >= 0.0f;
            tiny = tiny || v < STRAND_PMIN;
            s += v;
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (!ok || (lane == 0 && !(fabs(s - 1.0) <= 1e-5))) bad = 1;
        if (i < K && tiny) small = 1;
    }
    // per-state emission constants (log2 domain), padded states emit nothing
    const double LOG2E = 1.4426950408889634074;
    const double LOG2_2PI = 2.6514961294723187980;
    for (int k = threadIdx.x; k < KP; k += blockDim.x) {
        float mx = 0.f, my = 0.f, qa = 0.f, qb = 0.f, qc = 0.f;
        float ctr = -INFINITY, cno = -INFINITY;
        double ux = 0.0, uy = 0.0, u0 = 0.0, wy = 0.0, w0 = 0.0;
        if (k < K) {
            double pk = p[k];
            double sxx = cov[3 * k], sxy = cov[3 * k + 1], syy = cov[3 * k + 2];
            double det = sxx * syy - sxy * sxy;
            bool ok = isfinite(pk) && pk >= 0.0 && pk <= 1.0 && isfinite(sxx) && isfinite(sxy) &&
                      isfinite(syy) && sxx > 0.0 && syy > 0.0 && det > 0.0 &&
                      isfinite(mu[2 * k]) && isfinite(mu[2 * k + 1]);
            if (!ok) {
                bad = 1;
            } else {
                mx = mu[2 * k];
                my = mu[2 * k + 1];
                qa = (float)(-0.5 * LOG2E * syy / det);
                qb = (float)(LOG2E * sxy / det);
                qc = (float)(-0.5 * LOG2E * sxx / det);
                ctr = (float)(log2(pk) - LOG2_2PI - 0.5 * log2(det));
                cno = (float)log2(1.0 - pk);
                // the quadratic form as two squares (Cholesky factor of the precision matrix)
                ux = sqrt(0.5 * LOG2E * syy / det);
                uy = -ux * sxy / syy;
                wy = sqrt(0.5 * LOG2E / syy);
                const double cx = (double)mx - centre[0], cy = (double)my - centre[1];
                u0 = -(ux * cx + uy * cy);
                w0 = -wy * cy;
            }
        }
        float *em = cb + lay.off_emis;
        em[EM_MUX * KP + k] = mx;
        em[EM_MUY * KP + k] = my;
        em[EM_QA * KP + k] = qa;
        em[EM_QB * KP + k] = qb;
        em[EM_QC * KP + k] = qc;
        em[EM_CTR * KP + k] = ctr;
        em[EM_CNO * KP + k] = cno;
        em[EM_UX * KP + k] = (float)ux;
        em[EM_UY * KP + k] = (float)uy;
        em[EM_U0 * KP + k] = (float)u0;
        em[EM_WY * KP + k] = (float)wy;
        em[EM_W0 * KP + k] = (float)w0;
    }
    // P padded to KP x KP (FP32, row-major) and the tensor-core images
    for (int idx = threadIdx.x; idx < KP * KP; idx += blockDim.x) {
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
    __syncthreads();
    if (threadIdx.x < 32) {
        // EM_OFF: the emissions' largest constants, rounded up to whole numbers
        float *em = cb + lay.off_emis;
        float mt = -INFINITY, mn = -INFINITY;
        for (int k = threadIdx.x; k < K; k += 32) {
            mt = fmaxf(mt, em[EM_CTR * KP + k]);
            mn = fmaxf(mn, em[EM_CNO * KP + k]);
        }
        for (int o = 16; o > 0; o >>= 1) {
            mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, o));
            mn = fmaxf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        }
        if (threadIdx.x == 0) {
            mt = isfinite(mt) ? ceilf(mt) : 0.0f;
            mn = isfinite(mn) ? ceilf(mn) : 0.0f;
            em[EM_OFF * KP] = mt;
            em[EM_OFF * KP + 1] = mn;
            em[EM_OFF * KP + 2] = centre[0];
            em[EM_OFF * KP + 3] = centre[1];
            prop_bad[q] = bad;
            if (bad) atomicOr(status, ST_EINVAL);
            if (sp.route) {
                // strands need P's entries above STRAND_PMIN and constants of ordinary size
                const bool fits = !small && fabsf(mt) <= 1000.0f && fabsf(mn) <= 1000.0f;
                sp.route[q] = bad ? ROUTE_BAD : ROUTE_STRANDS;
                sp.jumps[q] = 0;
                if (!bad && !fits) {
                    sp.route[q] = ROUTE_CHUNKS;
                    sp.todo[1 + atomicAdd(&sp.todo[0], 1)] = q;
                }
            }
        }
    }
}

cudaError_t launch_prep(int n_prop, int K, const ConstLayout &lay, int precision, int init_mode,
                        const float *pi, const float *P, const float *p, const float *mu,
                        const float *cov, float *cblock, int *prop_bad, unsigned *status,
                        const StrandPtrs &sp, cudaStream_t st) {
    (void)init_mode;
    prep_kernel<<<n_prop, PREP_THREADS, 0, st>>>(K, lay, precision, pi, P, p, mu, cov, cblock, prop_bad,
                                        status, sp);
    return cudaGetLastError();
}

// One thread per observation; the segment is found by binary search.
__global__ void pack_kernel(int n_seg, const int64_t *__restrict__ offs,
                            const int64_t *__restrict__ pbase, int64_t T_total,
                            const float2 *__restrict__ xy, const uint8_t *__restrict__ tremor,
                            float2 *__restrict__ packed, float2 *__restrict__ head,
                            int *__restrict__ obs_bad, unsigned *__restrict__ status) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < T_total;
         t += (int64_t)gridDim.x * blockDim.x) {
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

cudaError_t launch_pack(int n_seg, const int64_t *d_offsets, const int64_t *d_pbase,
                        int64_t T_total, const float *xy, const uint8_t *tremor, float2 *packed,
                        float2 *head, int *obs_bad, unsigned *status, cudaStream_t st) {
    if (T_total == 0) return cudaSuccess;
    int64_t blocks = (T_total + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    pack_kernel<<<(int)blocks, 256, 0, st>>>(n_seg, d_offsets, d_pbase, T_total,
                                             reinterpret_cast<const float2 *>(xy), tremor, packed,
                                             head, obs_bad, status);
    return cudaGetLastError();
}

}  // namespace hmm
