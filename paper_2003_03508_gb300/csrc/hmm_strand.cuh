// Strands: the forward vector carried over pieces of a segment.
//
// log L needs the row vector pi D_1 P D_2 ... only. A chunk product carries K
// such rows because the row entering the chunk is not known when the chunk
// runs; but the products of a chain that mixes forget where they started: any
// two positive vectors run through the same steps become proportional, after
// some 25 steps at the median and 250 at most on tremor data (about 800 where
// tremors are rare). So every piece of a segment carries ONE vector, 2 K^2
// flops a step in place of 2 K^3:
//   * a strand starts `warm` steps before its piece from a flat vector, notes
//     the vector g at the piece's start, and runs on to the piece's end, with
//     the power-of-two exponents of its scaling;
//   * the strand of the piece before ends with the vector a at the same place.
//     If a = r g within a small tolerance in EVERY entry, then, all factors
//     being non-negative, the true vector stays within that tolerance of r
//     times the strand's for the rest of the chain: the piece contributes
//     log r + its exponents, and the error is at most the tolerance, once per
//     piece. If it is not, the join runs both vectors on until it is.
//   * a proposal whose joins would run on for longer than its chunk products
//     take (a chain that does not mix), or whose P has an entry below PMIN (next
//     paragraph), goes to the chunk products as a whole.
//
// Range. Entries below 2^-126 flush to zero. The vector is renormalised every
// four steps and the steps between are checked to shrink it by no more than
// 2^-60 (else they are repeated one by one with exact scaling), so what is
// lost is below 2^-66 of the largest entry l, while the next prediction of any
// state j is at least P_lj >= PMIN = 2^-40 of it: a loss below K 2^-26, and
// far less on any data, since it needs the smallest P_lj to meet the largest
// flushed entry at the same step.
#pragma once

#include "hmm_internal.cuh"

namespace hmm {

constexpr float STRAND_PMIN = 9.094947017729282e-13f;   // 2^-40
constexpr float STRAND_SHRINK = 8.673617379884035e-19f; // 2^-60
constexpr float STRAND_SHRINK_KEEP = 5.960464477539063e-08f;  // 2^-24: where every step's vector is kept
constexpr float STRAND_TINY = 8.470329472543003e-22f;   // 2^-70: an entry this far below the largest cannot matter (PMIN)
constexpr float STRAND_GROW = 1.2676506002282294e30f;   // 2^100

typedef unsigned long long f32x2;  // two packed floats

__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// What all states of a proposal share: the whole offsets of the factors, taken
// out of ctr and cno so that every factor is at most 1.
struct StrandBase {
    float offt, offn;

    __device__ __forceinline__ void load(const float *__restrict__ em, int KPl) {
        offt = em[EM_OFF * KPl];
        offn = em[EM_OFF * KPl + 1];
    }
    __device__ __forceinline__ float off(bool tremor) const { return tremor ? offt : offn; }
};

// Emission constants of two states. The density's exponent is two squares of
// linear forms of the difference from the mean, seven packed operations a pair.
// AFFINE: five, as affine forms of the location from the states' centre, which
// lose the bits that the mean's distance has over the state's width (s = |u0|,
// |w0|: 2^-23 s |u| of a log2 factor). FP32 never takes them: they
// cost the CUDA cores nothing (log L, host and run-length calls within 1.5%), and
// at 25 states 0.2 km wide log L was 1.5e-6 off with them, 1.7e-7 without. The
// tensor cores' strands do where s is at most EMIS_NEAR for every state (the
// synthetic recipe stays below 40): 2e-5 of a factor at three deviations, a tenth
// of the rounding of a TF32 operand; K=32, T=2^20, 256 proposals 4.35 ms with
// them, 4.57 without.
constexpr float EMIS_NEAR = 64.0f;

template <bool AFFINE>
struct EmisPair {
    f32x2 p, q, ux, uy, wy, nctr;  // p, q: minus the mean (AFFINE: u0, w0); nctr: offset - constant
    float quiet0, quiet1;          // factors of a step without a tremor

    // `up`: log2 of what every factor is made larger by
    __device__ __forceinline__ void load(const float *__restrict__ em, int KPl, int k0, float up = 0.0f) {
        constexpr int rows[5] = {AFFINE ? EM_U0 : EM_MUX, AFFINE ? EM_W0 : EM_MUY, EM_UX, EM_UY, EM_WY};
        float v[2][7];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int k = k0 + u;
            const bool in = k < KPl;
#pragma unroll
            for (int r = 0; r < 5; ++r) {
                v[u][r] = in ? em[rows[r] * KPl + k] : 0.0f;
                if (!AFFINE && r < 2) v[u][r] = -v[u][r];
            }
            v[u][5] = in ? em[EM_SC * KPl + k] - up : INFINITY;
            v[u][6] = in ? em[EM_QF * KPl + k] : 0.0f;
            if (up != 0.0f) v[u][6] *= exp2f(up);
        }
        p = pack2(v[0][0], v[1][0]);
        q = pack2(v[0][1], v[1][1]);
        ux = pack2(v[0][2], v[1][2]);
        uy = pack2(v[0][3], v[1][3]);
        wy = pack2(v[0][4], v[1][4]);
        nctr = pack2(v[0][5], v[1][5]);
        quiet0 = v[0][6];
        quiet1 = v[1][6];
    }
    // log2 factors of a tremor at (x, y) (AFFINE: from the centre)
    __device__ __forceinline__ void density(float x, float y, float &l0, float &l1) const {
        const f32x2 xx = pack2(x, x), yy = pack2(y, y);
        f32x2 u, w;
        if (AFFINE) {
            u = fma2(ux, xx, fma2(uy, yy, p));
            w = fma2(wy, yy, q);
        } else {
            const f32x2 dx = add2(xx, p), dy = add2(yy, q);
            u = fma2(ux, dx, mul2(uy, dy));
            w = mul2(wy, dy);
        }
        float n0, n1;
        unpack2(fma2(w, w, fma2(u, u, nctr)), n0, n1);
        l0 = -n0;
        l1 = -n1;
    }
    // emission factors of an observation, a tremor's relative to 2^fm
    __device__ __forceinline__ void factors(float x, float y, bool tremor, float fm, float &f0, float &f1) const {
        density(x, y, f0, f1);
        f0 = tremor ? ex2(f0 - fm) : quiet0;
        f1 = tremor ? ex2(f1 - fm) : quiet1;
    }
    // What fm is taken from: log2 factors of a tremor; without one 0 for every
    // state that emits (their factors are in (2^-25, 1], the largest above 1/2).
    __device__ __forceinline__ void sizes(float x, float y, bool tremor, float &l0, float &l1) const {
        density(x, y, l0, l1);
        if (!tremor) {
            l0 = quiet0 > 0.0f ? 0.0f : -INFINITY;
            l1 = quiet1 > 0.0f ? 0.0f : -INFINITY;
        }
    }
};
using Emis2 = EmisPair<false>;

// Marks proposal q for the chunk products (once).
__device__ __forceinline__ void send_to_chunks(const StrandPtrs &sp, int q) {
    if (atomicCAS(&sp.route[q], ROUTE_STRANDS, ROUTE_CHUNKS) == ROUTE_STRANDS)
        sp.todo[1 + atomicAdd(&sp.todo[0], 1)] = q;
}

}  // namespace hmm
