// Joining the strands of a segment (hmm_strand.cuh): one warp per piece that
// is not its segment's first compares the vector its strand had at the piece's
// start, g, with the end of the strand before, a. If a = r g within the
// tolerance in every entry, log r is noted. Otherwise both vectors run on
// through the piece, with exact scaling, until they meet. Where the piece ends
// first, a goes on against the strand of the next piece, and the pieces passed
// over are taken from it (jump). After sp.most steps of one piece, or sp.budget of
// all of a proposal's, the proposal is sent to the chunk products, which would have
// taken twice as long by then (strand_limits in hmm_api.cu).
//
// Most pieces meet at once (the warm-up covers the usual distance), so the
// kernel reads 2 KP floats a piece; the rest are up to some hundred steps of one
// warp each, bound by the latency of a step: 0.2 us with P's column in registers
// (K <= 32), four steps between two looks and two renormalisations (0.3 us with a
// look at every step). Beyond 32 states a CTA's four pieces are of one proposal
// and share its P in shared memory, loaded where one of them has not met: 0.55 us
// a step, eight rows' loads in flight (about 1 with four), 3.4 where every step
// fetched it through the cache (K = 48, 16 proposals, T = 5000: 0.475 ms for the
// call, which chunk products make in 0.44; 0.23 now).
#include "hmm_strand.cuh"

namespace hmm {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int JOIN_WARPS = 4;
constexpr float JOIN_TOL = 3.0517578125e-5f;  // 2^-15: what FP32 vectors run on to

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(FULL, v, o));
    return v;
}
__device__ __forceinline__ float warp_min(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(FULL, v, o));
    return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}

// NC: states per lane (KP <= 32 NC)
template <int NC>
__global__ void __launch_bounds__(32 * JOIN_WARPS)
join_kernel(int n_prop, int K, int KP, ConstLayout lay, bool round_tf32, float tol0, const float *__restrict__ cblock,
            const float2 *__restrict__ packed, StrandPtrs sp) {
    __shared__ __align__(16) float2 sag[JOIN_WARPS][32 * NC];
    extern __shared__ float sP[];  // NC > 1: P, rows of 32 NC floats
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int q, s;
    if (NC == 1) {
        const long long id = (long long)blockIdx.x * JOIN_WARPS + warp;
        q = (int)(id / sp.n);
        s = (int)(id % sp.n);
        if (q >= n_prop) return;
    } else {  // CTAs of one proposal
        const int cpp = (sp.n + JOIN_WARPS - 1) / JOIN_WARPS;
        q = blockIdx.x / cpp;
        s = (blockIdx.x % cpp) * JOIN_WARPS + warp;
    }
    // (another warp may change the route meanwhile: what this one does does not hang on when it looks)
    const bool mine = s < sp.n && __shfl_sync(FULL, sp.route[q], 0) == ROUTE_STRANDS;
    StrandDesc d = sp.desc[mine ? s : 0];
    const size_t idx = (size_t)q * sp.n + s;
    const bool first = (d.flags & SD_FIRST) != 0, joins = mine && !first;
    if (mine && first && lane == 0) {
        sp.logr[idx] = 0.0;
        sp.jump[idx] = s;
    }
    float a[NC], g[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const int k = lane + 32 * c;
        a[c] = joins && k < K ? sp.ve[(idx - 1) * KP + k] : 0.0f;
        g[c] = joins && k < K ? sp.vs[idx * KP + k] : 0.0f;
    }
    // in every entry; never where one is not a number (fmin and fmax pass those over) or none is large enough
    auto met = [&](float tol) {
        float lo = INFINITY, hi = 0.0f;
        bool numbers = true;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            numbers = numbers && a[c] == a[c] && g[c] == g[c];
            if (a[c] > STRAND_TINY || g[c] > STRAND_TINY) {
                const float r = a[c] / g[c];
                lo = fminf(lo, r);
                hi = fmaxf(hi, r);
            }
        }
        lo = warp_min(lo);
        hi = warp_max(hi);
        return __all_sync(FULL, numbers) && hi > 0.0f && hi < INFINITY && hi <= lo * (1.0f + tol);
    };
    int ea = 0, eg = 0;  // exponents gathered while running on: a's from this piece's start, g's from piece `at`'s
    long long xa = 0, xg = 0;  // their sums
    long long off = 0;  // whole offsets of the current piece's steps: common to both vectors
    int at = s;
    bool over = false;  // the segment ended before the vectors met
    bool ok = met(tol0);
    const float *cb = cblock + (size_t)q * lay.stride;
    const int KPl = lay.KP;
    auto load_p = [&](int i, int k) {
        float v = i < KPl && k < KPl ? cb[lay.off_p32 + i * KPl + k] : 0.0f;
        if (round_tf32) {
            uint32_t r;
            asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(v));
            v = __uint_as_float(r);
        }
        return v;
    };
    if (NC > 1 && __syncthreads_or(joins && !ok)) {
        for (int x = threadIdx.x; x < KP * 32 * NC; x += 32 * JOIN_WARPS) sP[x] = load_p(x / (32 * NC), x % (32 * NC));
        __syncthreads();
    }
    if (!joins) return;
    if (!ok) {
        const float *em = cb + lay.off_emis;
        f32x2 pc[NC == 1 ? 32 : 1];  // this lane's column of P, each entry twice
        if (NC == 1) {
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const float v = load_p(i, lane);
                pc[NC == 1 ? i : 0] = pack2(v, v);
            }
        }
        float c[NC][7];
        const float offt = em[EM_OFF * KPl], offn = em[EM_OFF * KPl + 1];
        const int ct = (int)offt, cn = (int)offn;
#pragma unroll
        for (int n = 0; n < NC; ++n) {
            const int k = lane + 32 * n;
#pragma unroll
            for (int r = 0; r < 7; ++r) c[n][r] = k < K ? em[r * KPl + k] : r >= EM_CTR ? -INFINITY : 0.0f;
            c[n][EM_CTR] -= offt;
            c[n][EM_CNO] -= offn;
        }
        // log2 emission factor of state lane + 32 n, relative to the whole offsets
        auto emission = [&](int n, float x, float y) {
            const float dx = x - c[n][EM_MUX], dy = y - c[n][EM_MUY];
            const float l = fmaf(fmaf(c[n][EM_QA], dx, c[n][EM_QB] * dy), dx, fmaf(c[n][EM_QC] * dy, dy, c[n][EM_CTR]));
            return isnan(x) ? c[n][EM_CNO] : l;
        };
        // one step of both vectors: (a, g) <- ((a, g) P) f
        auto step = [&](const float (&f)[NC]) {
#pragma unroll
            for (int n = 0; n < NC; ++n) sag[warp][lane + 32 * n] = make_float2(a[n], g[n]);
            __syncwarp();
            f32x2 acc[NC][4];
#pragma unroll
            for (int n = 0; n < NC; ++n) acc[n][0] = acc[n][1] = acc[n][2] = acc[n][3] = 0ull;
            if (NC == 1) {
#pragma unroll
                for (int i = 0; i < 32; i += 2) {
                    const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(&sag[warp][i]);
                    acc[0][i & 2] = fma2(x.x, pc[NC == 1 ? i : 0], acc[0][i & 2]);
                    acc[0][(i & 2) + 1] = fma2(x.y, pc[NC == 1 ? i + 1 : 0], acc[0][(i & 2) + 1]);
                }
            } else {
#pragma unroll 8
                for (int i = 0; i < KP; i += 2) {
                    const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(&sag[warp][i]);
#pragma unroll
                    for (int n = 0; n < NC; ++n) {
                        const float v = sP[i * 32 * NC + lane + 32 * n], w = sP[(i + 1) * 32 * NC + lane + 32 * n];
                        acc[n][0] = fma2(x.x, pack2(v, v), acc[n][0]);
                        acc[n][1] = fma2(x.y, pack2(w, w), acc[n][1]);
                    }
                }
            }
            __syncwarp();
#pragma unroll
            for (int n = 0; n < NC; ++n) {
                unpack2(add2(add2(acc[n][0], acc[n][1]), add2(acc[n][2], acc[n][3])), a[n], g[n]);
                a[n] *= f[n];
                g[n] *= f[n];
            }
        };
        // both back to [1, 2); false when one left the range
        auto rescale = [&]() {
            float ma = 0.0f, mg = 0.0f;
#pragma unroll
            for (int n = 0; n < NC; ++n) {
                ma = fmaxf(ma, a[n]);
                mg = fmaxf(mg, g[n]);
            }
            ma = warp_max(ma);
            mg = warp_max(mg);
            if (!(ma >= STRAND_SHRINK && mg >= STRAND_SHRINK && ma <= STRAND_GROW && mg <= STRAND_GROW)) return false;
            const int pa = float_exponent(ma), pg = float_exponent(mg);
            const float fa = pow2f(-pa), fg = pow2f(-pg);
#pragma unroll
            for (int n = 0; n < NC; ++n) {
                a[n] *= fa;
                g[n] *= fg;
            }
            ea += pa;
            eg += pg;
            return true;
        };
        bool alive = true;
        int t0 = 0;
        for (int done = 0; !ok && alive && done < sp.most; done += 32, t0 += 32) {
            // Every 64 steps: what all joins of a proposal need is the same in any order, so whether it is
            // above the budget is too. Another one may have given up: nothing to do here then.
            if (done && done % 64 == 0) {
                int sum = 0, route = ROUTE_STRANDS;
                if (lane == 0) {
                    sum = atomicAdd(&sp.spent[q], 64) + 64;
                    route = *(volatile const int *)&sp.route[q];
                }
                if (__shfl_sync(FULL, route, 0) != ROUTE_STRANDS) return;
                if (__shfl_sync(FULL, sum, 0) > sp.budget) break;
            }
            if (t0 >= d.len) {
                // this piece is over: on against the next one's strand
                xa += off;
                off = xg = 0;
                if (d.flags & SD_LAST) {
                    over = true;
                    break;
                }
                ++at;
                d = sp.desc[at];
                t0 = 0;
#pragma unroll
                for (int n = 0; n < NC; ++n) {
                    const int k = lane + 32 * n;
                    g[n] = k < K ? sp.vs[((size_t)q * sp.n + at) * KP + k] : 0.0f;
                }
                ok = met(JOIN_TOL);
                if (ok) break;
            }
            // 32 steps' observations, one per lane (the packed sequence is padded to whole windows)
            const float2 ob = packed[d.pstart + t0 + lane];
            for (int t = t0; t < min(t0 + 32, d.len) && !ok && alive; t += 4) {
                const int m = min(4, d.len - t);
                float ka[NC], kg[NC];
#pragma unroll
                for (int n = 0; n < NC; ++n) {
                    ka[n] = a[n];
                    kg[n] = g[n];
                }
                bool fine = m == 4;
                int o4 = 0;
                if (fine) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float x = __shfl_sync(FULL, ob.x, t - t0 + j), y = __shfl_sync(FULL, ob.y, t - t0 + j);
                        float f[NC];
                        o4 += isnan(x) ? cn : ct;
#pragma unroll
                        for (int n = 0; n < NC; ++n) f[n] = ex2(emission(n, x, y));
                        step(f);
                    }
                    fine = rescale();
                }
                if (!fine) {
                    o4 = 0;
                    // step by step with exact scaling (as in the strands)
#pragma unroll
                    for (int n = 0; n < NC; ++n) {
                        a[n] = ka[n];
                        g[n] = kg[n];
                    }
                    for (int j = 0; j < m && alive; ++j) {
                        const float x = __shfl_sync(FULL, ob.x, t - t0 + j), y = __shfl_sync(FULL, ob.y, t - t0 + j);
                        float f[NC], mx = -INFINITY;
#pragma unroll
                        for (int n = 0; n < NC; ++n) {
                            f[n] = emission(n, x, y);
                            mx = fmaxf(mx, f[n]);
                        }
                        mx = warp_max(mx);
                        alive = mx + (isnan(x) ? offn : offt) >= -(float)EXP_LIMIT;
                        const float fm = alive ? floorf(mx) : 0.0f;
                        o4 += (int)fm + (isnan(x) ? cn : ct);
#pragma unroll
                        for (int n = 0; n < NC; ++n) f[n] = ex2(f[n] - fm);
                        step(f);
                        alive = alive && rescale();
                    }
                }
                off += o4;
                ok = alive && met(JOIN_TOL);
            }
            xa += ea;
            xg += eg;
            ea = eg = 0;
        }
    }
    double sa = 0.0, sg = 0.0;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        sa += a[c];
        sg += g[c];
    }
    sa = warp_sum(sa);
    sg = warp_sum(sg);
    if (lane == 0) {
        if (ok || over) {
            sp.logr[idx] = log(ok ? sa / sg : sa) + 0.69314718055994530942 * (double)(xa - xg);
            sp.jump[idx] = ok ? at : -1;
            if (at != s || over) sp.jumps[q] = 1;
        } else {
            send_to_chunks(sp, q);
        }
    }
}

}  // namespace

cudaError_t launch_join(int n_prop, int K, int KP, const ConstLayout &lay, int precision, bool tensor, const float *cblock,
                        const float2 *packed, const StrandPtrs &sp, cudaStream_t st) {
    if (sp.n == 0) return cudaSuccess;
    // Vectors that have met differ by the rounding of their strands: a few
    // 2^-20 in FP32, 2^-11 with TF32 operands, 2^-16 with BF16 hi + lo. What is
    // taken as met at a piece's start is wider by eight; the ratio of the sums
    // then carries the rounding of one step, where the piece has that of 64 and
    // more. The rest runs on in FP32 to JOIN_TOL (K=80 BF16, 32 proposals:
    // 1000 us when every boundary had to).
    const float tol = !tensor ? JOIN_TOL : precision == HMM_PREC_BF16 ? 2.44140625e-4f : 3.90625e-3f;
    const bool rt = tensor && precision == HMM_PREC_TF32;  // P as the strands have it
    const long long warps = (long long)n_prop * sp.n;
    const int nc = KP <= 32 ? 1 : KP <= 64 ? 2 : 3;
    const unsigned grid = (unsigned)(nc == 1 ? (warps + JOIN_WARPS - 1) / JOIN_WARPS
                                             : (long long)n_prop * ((sp.n + JOIN_WARPS - 1) / JOIN_WARPS));
    const size_t smem = nc == 1 ? 0 : sizeof(float) * KP * 32 * nc;  // at most 30 KB
    auto kern = nc == 1 ? join_kernel<1> : nc == 2 ? join_kernel<2> : join_kernel<3>;
    kern<<<grid, 32 * JOIN_WARPS, smem, st>>>(n_prop, K, KP, lay, rt, tol, cblock, packed, sp);
    return cudaGetLastError();
}

}  // namespace hmm
