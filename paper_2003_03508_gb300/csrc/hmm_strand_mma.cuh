// Strands on the tensor cores, for batches in HMM_PREC_TF32, _TF32_SPLIT and
// _BF16. See hmm_strand.cuh for the method.
//
// A warp carries 16 MT strands of one proposal as the rows of mma.sync
// fragments. The accumulator fragment of one step (row l/4, columns 2(l%4) and
// 2(l%4)+1 of every eight) is, lane for lane, the A fragment of the next one
// once the rows of P are taken in the matching order, so the vectors never
// leave their registers: no exchange, no barrier, no tensor memory round trip.
// That is why this is mma.sync and not tcgen05: a tcgen05 step has to go
// through tensor memory and an mbarrier, some 1100 cycles as the chunk-product
// kernels measure it, and here a step's arithmetic (with emissions that differ
// in every row) is larger than its matrix work, which mma.sync covers at 8
// cycles per 16 x 8 x 8 block (TF32) or 16 x 8 x 16 block (BF16).
//
// Operands: TF32 rounds the vector and P to TF32; TF32_SPLIT carries P as
// hi + lo; BF16 carries both the vector and P as hi + lo and takes three of
// the four products, which costs half as much again as one TF32 product.
// Accumulation is FP32, and everything between two products stays FP32.
//
// P's fragments are in registers up to KP = 32 and in shared memory above, where
// two row blocks a warp (MT = 2) halve the loads; the emission constants are in
// registers up to KP = 32 as well, but for BF16 at 32, whose hi and lo words need
// the room (5.9 against 7.4 ms at T = 2^20, 256 proposals).
//
// What bounds it: MMAs, packed FMAs and selects share the register ports and do
// not overlap (4 MMAs of 32 cycles and 16 packed FMAs of 36 take 68), so a step
// of a warp costs their sum: at KP = 32 TF32 about 300 cycles for 16 strands,
// 128 of them MMAs. K=32, T=2^20, 256 proposals: 4.35 ms TF32, 6.5 ms TF32_SPLIT,
// 5.9 ms BF16; 13.5 ms on the CUDA cores, 60.5 ms by chunk products. Two warps a
// scheduler without spills (4.37 ms) beat three with (4.81) and four (6.64); two
// row blocks a warp at KP = 32 took 6.8 ms.
#pragma once

#include <cuda_bf16.h>

#include "hmm_strand.cuh"

namespace hmm {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int WPC = 4;  // warps per CTA

enum { M_TF32 = 0, M_SPLIT = 1, M_BF16 = 2 };

template <int KP_, int MODE_>
struct MmaTile {
    static constexpr int KP = KP_;
    static constexpr int MODE = MODE_;
    static constexpr bool REGS = KP <= 32;             // P's fragments in registers
    static constexpr bool EREG = KP <= 16 || (KP == 32 && MODE != M_BF16);  // emission constants too
    static constexpr int MT = REGS ? 1 : 2;            // row blocks per warp
    static constexpr int NT = KP / 8;                  // column blocks
    static constexpr int NS = MODE == M_BF16 ? KP / 16 : KP / 8;  // k slices
    static constexpr int NB = MODE == M_TF32 ? 2 : 4;  // words of one B fragment (hi, then lo)
    static constexpr int ROWS = 16 * MT;               // strands per warp
    static constexpr int B_WORDS = REGS ? 0 : NS * NT * 32 * NB;
    static constexpr int E_WORDS = NT * 4 * 16;          // per warp (REGS) or CTA
    static constexpr int E_ALL = EREG ? 0 : REGS ? WPC * E_WORDS : E_WORDS;
    static constexpr int SMEM = 4 * (B_WORDS + E_ALL) + WPC * ROWS * 4 * 8;
};

__device__ __forceinline__ void mma_tf32(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t rna(float x) { return __float_as_uint(x) + 0x1000u; }  // nearest TF32 (low bits ignored)
// TF32: the raw bits, which the tensor core truncates; the emissions carry the
// mean loss back (TRUNC_LOG2). TF32_SPLIT: rounded to nearest.
template <int MODE>
__device__ __forceinline__ uint32_t operand(float x) {
    return MODE == M_TF32 ? __float_as_uint(x) : rna(x);
}
// -log2(1 - c), c = 2^-11 / (2 ln 2) the mean relative loss of truncating a
// float with a log-uniform mantissa to 10 bits
constexpr float TRUNC_LOG2 = 5.0820e-4f;
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// (a, b) as bf16 hi and lo words
__device__ __forceinline__ void split_bf16(float a, float b, uint32_t &hi, uint32_t &lo) {
    hi = pack_bf16(a, b);
    lo = pack_bf16(a - __uint_as_float(hi << 16), b - __uint_as_float(hi & 0xffff0000u));
}

// Words of the B fragment of k slice s and column block n for lane l. Slices
// of eight (TF32) take the rows 8 s + 2 (l%4), + 1 in the places l%4, l%4 + 4.
template <class C>
__device__ __forceinline__ void b_fragment(const float *__restrict__ P, int KPl, int s, int n, int l, uint32_t (&b)[C::NB]) {
    const int col = 8 * n + (l >> 2), t = l & 3;
    auto at = [&](int i) { return i < KPl && col < KPl ? P[i * KPl + col] : 0.0f; };
    if (C::MODE == M_BF16) {
        const float p0 = at(16 * s + 2 * t), p1 = at(16 * s + 2 * t + 1);
        const float p2 = at(16 * s + 2 * t + 8), p3 = at(16 * s + 2 * t + 9);
        split_bf16(p0, p1, b[0], b[C::NB - 2]);
        split_bf16(p2, p3, b[1], b[C::NB - 1]);
    } else {
        const float p[2] = {at(8 * s + 2 * t), at(8 * s + 2 * t + 1)};
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            b[u] = rna(p[u]) & 0xffffe000u;
            if (C::MODE == M_SPLIT) b[C::NB - 2 + u] = rna(p[u] - __uint_as_float(b[u])) & 0xffffe000u;
        }
    }
}

// One warp's strands. NEAR: with the affine emission forms (hmm_strand.cuh)
template <class C, bool NEAR>
__device__ __forceinline__ void
carry_strands(int q, int wq, int wpp, int K, int init_mode, const ConstLayout &lay, const float *__restrict__ cb,
              const float *__restrict__ pi_all, const float2 *__restrict__ head, const float2 *__restrict__ packed,
              const StrandPtrs &sp) {
    constexpr int KP = C::KP, MT = C::MT, NT = C::NT, NS = C::NS, NB = C::NB, ROWS = C::ROWS, NR = 2 * MT;
    extern __shared__ __align__(16) uint32_t smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gid = lane >> 2, tig = lane & 3;
    const float *em = cb + lay.off_emis;
    const float *P = cb + lay.off_p32;
    const int KPl = lay.KP;
    const bool mine = __shfl_sync(FULL, sp.route[q], 0) == ROUTE_STRANDS;  // the warp agrees
    StrandBase base;
    base.load(em, KPl);
    const float cx = NEAR ? em[EM_OFF * KPl + 2] : 0.0f, cy = NEAR ? em[EM_OFF * KPl + 3] : 0.0f;
    // the factors' offsets; TF32 operands lose TRUNC_LOG2 a step
    const float lost = C::MODE == M_TF32 ? TRUNC_LOG2 : 0.0f;

    uint32_t breg[C::REGS ? NS : 1][C::REGS ? NT : 1][NB];
    EmisPair<NEAR> ereg[C::EREG ? NT : 1];
    uint32_t *sB = smem;
    f32x2 *sE = reinterpret_cast<f32x2 *>(smem + C::B_WORDS + (C::REGS ? warp * C::E_WORDS : 0));  // [NT][4][8]
    float2 *sObs = reinterpret_cast<float2 *>(smem + C::B_WORDS + C::E_ALL) + warp * ROWS * 4;  // [ROWS][4]
    auto fill_emission = [&](int first, int step) {
        for (int i = first; i < NT * 4; i += step) {
            EmisPair<NEAR> e;
            e.load(em, KPl, 8 * (i / 4) + 2 * (i % 4), lost);
            // pairs (u, u + 1) of a lane side by side: 16-byte loads
            f32x2 *d = sE + (i / 4) * 32 + (i % 4) * 2;
            d[0] = e.p; d[1] = e.q; d[8] = e.ux; d[9] = e.uy; d[16] = e.wy; d[17] = e.nctr;
            d[24] = pack2(e.quiet0, e.quiet1);
        }
    };
    if (C::REGS) {
        if (!mine || wq >= wpp) return;
#pragma unroll
        for (int s = 0; s < (C::REGS ? NS : 1); ++s)
#pragma unroll
            for (int n = 0; n < (C::REGS ? NT : 1); ++n) b_fragment<C>(P, KPl, s, n, lane, breg[s][n]);
        if (C::EREG) {
#pragma unroll
            for (int n = 0; n < (C::EREG ? NT : 1); ++n) ereg[n].load(em, KPl, 8 * n + 2 * tig, lost);
        } else {
            fill_emission(lane, 32);
            __syncwarp();
        }
    } else {
        // `route` may change while the strands run: what this CTA does with
        // the barrier below does not depend on it
        for (int i = threadIdx.x; i < NS * NT * 32; i += 32 * WPC) {
            uint32_t b[NB];
            b_fragment<C>(P, KPl, (i >> 5) / NT, (i >> 5) % NT, i & 31, b);
#pragma unroll
            for (int u = 0; u < NB; ++u) sB[i * NB + u] = b[u];
        }
        fill_emission(threadIdx.x, 32 * WPC);
        __syncthreads();
        if (!mine || wq >= wpp) return;
    }
    auto emis = [&](int n) -> EmisPair<NEAR> {
        if (C::EREG) return ereg[C::EREG ? n : 0];
        EmisPair<NEAR> e;
        const f32x2 *d = sE + n * 32 + tig * 2;
        const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(d), b = *reinterpret_cast<const ulonglong2 *>(d + 8),
                         c = *reinterpret_cast<const ulonglong2 *>(d + 16);
        e.p = a.x; e.q = a.y; e.ux = b.x; e.uy = b.y; e.wy = c.x; e.nctr = c.y;
        unpack2(d[24], e.quiet0, e.quiet1);
        return e;
    };
    const int ct = (int)base.offt, cn = (int)base.offn;
    const int w0 = wq * ROWS;

    // this thread's rows: gid + 8 r
    int total[NR], warm[NR], sid[NR], e32[NR], nwin = 0;
    long long e64[NR];
    unsigned bad = 0;
    float v[MT][NT][4];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int k = w0 + gid + 8 * r;
        sid[r] = k < sp.n ? sp.order[k] : -1;
        const StrandDesc d = sp.desc[sid[r] < 0 ? 0 : sid[r]];
        total[r] = sid[r] < 0 ? 0 : d.warm + d.len;
        warm[r] = d.warm;
        e32[r] = 0;
        e64[r] = 0;
        nwin = max(nwin, (total[r] + 3) / 4);
        const bool at_head = (d.flags & SD_HEAD) != 0;
        const float2 o = head[d.seg];
        const bool tr = !isnan(o.x);
        const float hx = NEAR ? o.x - cx : o.x, hy = NEAR ? o.y - cy : o.y;
        float l[NT][2], m = -INFINITY;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            emis(n).sizes(hx, hy, tr, l[n][0], l[n][1]);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int k2 = 8 * n + 2 * tig + u;
                float w = 0.0f;
                if (k2 < K) {
                    if (init_mode == HMM_INIT_TRANSITION_FIRST) {
                        double s = 0.0;
                        for (int i = 0; i < K; ++i) s += (double)pi_all[(size_t)q * K + i] * (double)P[i * KPl + k2];
                        w = (float)s;
                    } else {
                        w = pi_all[(size_t)q * K + k2];
                    }
                }
                v[r / 2][n][2 * (r & 1) + u] = w;
                if (w > 0.0f) m = fmaxf(m, l[n][u]);
            }
        }
        m = fmaxf(m, __shfl_xor_sync(FULL, m, 1));
        m = fmaxf(m, __shfl_xor_sync(FULL, m, 2));
        const bool emits = m + base.off(tr) >= -(float)EXP_LIMIT;
        const float fm = emits ? floorf(m) : 0.0f;
        if (at_head && !emits) bad |= 1u << r;
        if (at_head && emits) e32[r] = (int)fm + (tr ? ct : cn);
        // no product here, nothing truncated: `lost` comes off again (3.5e-4 a segment otherwise)
        const float kept = C::MODE == M_TF32 ? exp2f(-lost) : 1.0f;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            emis(n).factors(hx, hy, tr, fm, l[n][0], l[n][1]);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                float &x = v[r / 2][n][2 * (r & 1) + u];
                if (at_head && emits) x = x > 0.0f ? x * (l[n][u] * kept) : 0.0f;
                else x = 8 * n + 2 * tig + u < K ? 1.0f : 0.0f;
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nwin = max(nwin, __shfl_xor_sync(FULL, nwin, o));

    // y = v P, block of columns by block, each handed to put(n, acc)
    auto advance = [&](auto put) {
        uint32_t a[MT][NS][4], alo[MT][C::MODE == M_BF16 ? NS : 1][4];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                if (C::MODE == M_BF16) {
                    const int s2 = C::MODE == M_BF16 ? s : 0;
                    const float(&x)[4] = v[mt][C::MODE == M_BF16 ? 2 * s : 0];
                    const float(&y)[4] = v[mt][C::MODE == M_BF16 ? 2 * s + 1 : 0];
                    split_bf16(x[0], x[1], a[mt][s][0], alo[mt][s2][0]);
                    split_bf16(x[2], x[3], a[mt][s][1], alo[mt][s2][1]);
                    split_bf16(y[0], y[1], a[mt][s][2], alo[mt][s2][2]);
                    split_bf16(y[2], y[3], a[mt][s][3], alo[mt][s2][3]);
                } else {
                    const float(&x)[4] = v[mt][C::MODE == M_BF16 ? 0 : s];
                    a[mt][s][0] = operand<C::MODE>(x[0]);
                    a[mt][s][1] = operand<C::MODE>(x[2]);
                    a[mt][s][2] = operand<C::MODE>(x[1]);
                    a[mt][s][3] = operand<C::MODE>(x[3]);
                }
            }
#pragma unroll
        for (int n = 0; n < NT; n += 2) {
            float acc[2][MT][4] = {};
#pragma unroll
            for (int s = 0; s < NS; ++s)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t b[NB];
                    if (C::REGS) {
#pragma unroll
                        for (int u = 0; u < NB; ++u) b[u] = breg[C::REGS ? s : 0][C::REGS ? n + h : 0][u];
                    } else if (NB == 4) {
                        const uint4 t = *reinterpret_cast<const uint4 *>(sB + ((s * NT + n + h) * 32 + lane) * NB);
                        b[0] = t.x; b[1] = t.y; b[NB - 2] = t.z; b[NB - 1] = t.w;
                    } else {
                        const uint2 t = *reinterpret_cast<const uint2 *>(sB + ((s * NT + n + h) * 32 + lane) * NB);
                        b[0] = t.x; b[1] = t.y;
                    }
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        if (C::MODE == M_BF16) {
                            mma_bf16(acc[h][mt], a[mt][s], b[NB - 2], b[NB - 1]);
                            mma_bf16(acc[h][mt], alo[mt][C::MODE == M_BF16 ? s : 0], b[0], b[1]);
                            mma_bf16(acc[h][mt], a[mt][s], b[0], b[1]);
                        } else {
                            if (C::MODE == M_SPLIT) mma_tf32(acc[h][mt], a[mt][s], b[NB - 2], b[NB - 1]);
                            mma_tf32(acc[h][mt], a[mt][s], b[0], b[1]);
                        }
                    }
                }
#pragma unroll
            for (int h = 0; h < 2; ++h) put(n + h, acc[h]);
        }
    };

    // Observations: lane i brings those of row i (MT = 2), or half a window of
    // row i / 2 (MT = 1), a window ahead, through shared memory.
    const int lrow = MT == 2 ? lane : lane >> 1;
    const float4 *lobs;
    int ltotal;
    {
        const int k = w0 + lrow;
        const StrandDesc d = sp.desc[k < sp.n ? sp.order[k] : 0];
        ltotal = k < sp.n ? d.warm + d.len : 0;
        lobs = reinterpret_cast<const float4 *>(packed + d.pstart - d.warm) + (MT == 2 ? 0 : lane & 1);
    }
    float4 na = make_float4(0.f, 0.f, 0.f, 0.f), nb = na;
    if (ltotal > 0) {
        na = lobs[0];
        if (MT == 2) nb = lobs[1];
    }
    for (int w = 0; w < nwin; ++w) {
        {
            if (NEAR) {
                na.x -= cx; na.y -= cy; na.z -= cx; na.w -= cy;
                nb.x -= cx; nb.y -= cy; nb.z -= cx; nb.w -= cy;
            }
            float4 *d = reinterpret_cast<float4 *>(sObs + lrow * 4) + (MT == 2 ? 0 : lane & 1);
            d[0] = na;
            if (MT == 2) d[1] = nb;
        }
        __syncwarp();
        if (4 * (w + 1) < ltotal) {
            na = lobs[2 * (w + 1)];
            if (MT == 2) nb = lobs[2 * (w + 1) + 1];
        }
        float keep[MT][NT][4];
        int step_e[NR];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int u = 0; u < 4; ++u) keep[mt][n][u] = v[mt][n][u];
#pragma unroll
        for (int r = 0; r < NR; ++r) step_e[r] = 0;
#pragma unroll(KP <= 32 ? 4 : 1)
        for (int j = 0; j < 4; ++j) {
            float2 o[NR];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                o[r] = sObs[(gid + 8 * r) * 4 + j];
                step_e[r] += isnan(o[r].x) ? cn : ct;
            }
            advance([&](int n, const float (&acc)[MT][4]) {
                const EmisPair<NEAR> e = emis(n);
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    float f0, f1;
                    e.factors(o[r].x, o[r].y, !isnan(o[r].x), 0.0f, f0, f1);
                    v[r / 2][n][2 * (r & 1)] = acc[r / 2][2 * (r & 1)] * f0;
                    v[r / 2][n][2 * (r & 1) + 1] = acc[r / 2][2 * (r & 1) + 1] * f1;
                }
            });
        }
        unsigned redo = 0;
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            float m = 0.0f;
#pragma unroll
            for (int n = 0; n < NT; ++n) m = fmaxf(m, fmaxf(v[r / 2][n][2 * (r & 1)], v[r / 2][n][2 * (r & 1) + 1]));
            m = fmaxf(m, __shfl_xor_sync(FULL, m, 1));
            m = fmaxf(m, __shfl_xor_sync(FULL, m, 2));
            const int left = total[r] - 4 * w;
            const bool fine = left >= 4 && m >= STRAND_SHRINK && m <= STRAND_GROW;
            if (left > 0 && !fine) redo |= 1u << r;
            const int x = float_exponent(m);
            const float s = pow2f(-x);
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    float &y = v[r / 2][n][2 * (r & 1) + u];
                    y = fine ? y * s : keep[r / 2][n][2 * (r & 1) + u];
                }
            e32[r] += fine ? step_e[r] + x : 0;
        }
        if (__any_sync(FULL, redo != 0)) {
            // one step at a time with exact scaling: a window that shrank too
            // far, or a piece's last steps
            for (int j = 0; j < 4; ++j) {
                float2 o[NR];
                float mx[NR];
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    o[r] = sObs[(gid + 8 * r) * 4 + j];
                    mx[r] = -INFINITY;
                }
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    const EmisPair<NEAR> e = emis(n);
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        float l0, l1;
                        e.sizes(o[r].x, o[r].y, !isnan(o[r].x), l0, l1);
                        mx[r] = fmaxf(mx[r], fmaxf(l0, l1));
                    }
                }
                bool emits[NR];
                float fm[NR];
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    mx[r] = fmaxf(mx[r], __shfl_xor_sync(FULL, mx[r], 1));
                    mx[r] = fmaxf(mx[r], __shfl_xor_sync(FULL, mx[r], 2));
                    emits[r] = mx[r] + base.off(!isnan(o[r].x)) >= -(float)EXP_LIMIT;
                    fm[r] = emits[r] ? floorf(mx[r]) : 0.0f;
                }
                float z[MT][NT][4];
                advance([&](int n, const float (&acc)[MT][4]) {
                    const EmisPair<NEAR> e = emis(n);
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        float f0, f1;
                        e.factors(o[r].x, o[r].y, !isnan(o[r].x), fm[r], f0, f1);
                        z[r / 2][n][2 * (r & 1)] = acc[r / 2][2 * (r & 1)] * f0;
                        z[r / 2][n][2 * (r & 1) + 1] = acc[r / 2][2 * (r & 1) + 1] * f1;
                    }
                });
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    float m = 0.0f;
#pragma unroll
                    for (int n = 0; n < NT; ++n) m = fmaxf(m, fmaxf(z[r / 2][n][2 * (r & 1)], z[r / 2][n][2 * (r & 1) + 1]));
                    m = fmaxf(m, __shfl_xor_sync(FULL, m, 1));
                    m = fmaxf(m, __shfl_xor_sync(FULL, m, 2));
                    const bool fine = emits[r] && m >= STRAND_SHRINK && m <= STRAND_GROW;
                    const bool act = (redo >> r & 1) && j < total[r] - 4 * w;
                    if (act && !fine) bad |= 1u << r;  // the chunk products decide
                    if (act && fine) {
                        const int x = float_exponent(m);
                        const float s = pow2f(-x);
#pragma unroll
                        for (int n = 0; n < NT; ++n)
#pragma unroll
                            for (int u = 0; u < 2; ++u)
                                v[r / 2][n][2 * (r & 1) + u] = z[r / 2][n][2 * (r & 1) + u] * s;
                        e32[r] += (int)fm[r] + (isnan(o[r].x) ? cn : ct) + x;
                    }
                }
            }
        }
        __syncwarp();  // everyone has read the window
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            if ((w & 63) == 63) {
                e64[r] += e32[r];
                e32[r] = 0;
            }
            if (4 * (w + 1) == warm[r] && total[r] > 0) {
                // the piece starts here
                float *dst = sp.vs + ((size_t)q * sp.n + sid[r]) * KP + 2 * tig;
#pragma unroll
                for (int n = 0; n < NT; ++n)
                    *reinterpret_cast<float2 *>(dst + 8 * n) = make_float2(v[r / 2][n][2 * (r & 1)], v[r / 2][n][2 * (r & 1) + 1]);
                e64[r] = 0;
                e32[r] = 0;
            }
        }
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        if (sid[r] < 0) continue;
        const size_t idx = (size_t)q * sp.n + sid[r];
        float *dst = sp.ve + idx * KP + 2 * tig;
#pragma unroll
        for (int n = 0; n < NT; ++n)
            *reinterpret_cast<float2 *>(dst + 8 * n) = make_float2(v[r / 2][n][2 * (r & 1)], v[r / 2][n][2 * (r & 1) + 1]);
        if (tig == 0) {
            sp.ex[idx] = e64[r] + e32[r];
            if (bad >> r & 1) send_to_chunks(sp, q);
        }
    }
}

// FORMS: which proposals this kernel takes. Up to 32 states one kernel holds both
// forms; beyond, where one alone takes a minute to compile, a kernel each, and
// the CTAs of the other's proposals leave at once (2 us a launch).
enum { F_FAR = 0, F_NEAR = 1, F_BOTH = 2 };

template <class C, int FORMS>
__global__ void __launch_bounds__(32 * WPC, C::KP <= 16 ? 4 : 2)
strand_mma_kernel(int n_prop, int K, int init_mode, ConstLayout lay, const float *__restrict__ cblock,
                  const float *__restrict__ pi_all, const float2 *__restrict__ head,
                  const float2 *__restrict__ packed, StrandPtrs sp) {
    const int warp = threadIdx.x >> 5;
    const int wpp = (sp.n + C::ROWS - 1) / C::ROWS;  // warps per proposal
    int q, wq;
    if (C::REGS) {  // warps on their own
        const long long wid = (long long)blockIdx.x * WPC + warp;
        q = (int)(wid / wpp);
        wq = (int)(wid % wpp);
    } else {        // CTAs of one proposal
        const int cpp = (wpp + WPC - 1) / WPC;
        q = blockIdx.x / cpp;
        wq = (blockIdx.x % cpp) * WPC + warp;
    }
    if (q >= n_prop) return;
    const float *cb = cblock + (size_t)q * lay.stride;
    const bool near = cb[lay.off_emis + EM_OFF * lay.KP + 4] != 0.0f;
    if (FORMS != F_FAR && near) carry_strands<C, FORMS != F_FAR>(q, wq, wpp, K, init_mode, lay, cb, pi_all, head, packed, sp);
    if (FORMS != F_NEAR && !near) carry_strands<C, FORMS == F_NEAR>(q, wq, wpp, K, init_mode, lay, cb, pi_all, head, packed, sp);
}

template <int KP, int MODE, int FORMS>
cudaError_t launch_t(int n_prop, int K, int init_mode, const ConstLayout &lay, const float *cblock, const float *pi,
                     const float2 *head, const float2 *packed, const StrandPtrs &sp, cudaStream_t st) {
    using C = MmaTile<KP, MODE>;
    const long long wpp = (sp.n + C::ROWS - 1) / C::ROWS;
    const long long ctas = C::REGS ? (n_prop * wpp + WPC - 1) / WPC : n_prop * ((wpp + WPC - 1) / WPC);
    auto kern = strand_mma_kernel<C, FORMS>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)ctas, 32 * WPC, C::SMEM, st>>>(n_prop, K, init_mode, lay, cblock, pi, head, packed, sp);
    return cudaGetLastError();
}

template <int KP, int FORMS>
cudaError_t launch_kp(int n_prop, int K, int init_mode, const ConstLayout &lay, int precision, const float *cblock,
                      const float *pi, const float2 *head, const float2 *packed, const StrandPtrs &sp,
                      cudaStream_t st) {
    switch (precision) {
        case HMM_PREC_TF32: return launch_t<KP, M_TF32, FORMS>(n_prop, K, init_mode, lay, cblock, pi, head, packed, sp, st);
        case HMM_PREC_TF32_SPLIT: return launch_t<KP, M_SPLIT, FORMS>(n_prop, K, init_mode, lay, cblock, pi, head, packed, sp, st);
        case HMM_PREC_BF16: return launch_t<KP, M_BF16, FORMS>(n_prop, K, init_mode, lay, cblock, pi, head, packed, sp, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace
}  // namespace hmm
