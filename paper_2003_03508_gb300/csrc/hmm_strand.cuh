// Strands: the forward vector carried over pieces of a segment.
//
// log L needs the row vector pi D_1 P D_2 ... only. A chunk product carries K
// such rows because the row entering the chunk is not known when the chunk
// runs; but the products of a chain that mixes forget where they started: any
// two positive vectors run through the same steps become proportional, after
// some 25 steps at the median and 200 at most on tremor data (about 800 where
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
//   * a piece whose two vectors do not meet before its end (a chain that does
//     not mix: P = I), and a P with an entry below PMIN (next paragraph), send
//     the whole proposal to the chunk products.
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
// out of ctr and cno so that every factor is at most 1, and the centre that the
// strands' coordinates are taken from.
struct StrandBase {
    float offt, offn, cx, cy;

    __device__ __forceinline__ void load(const float *__restrict__ em, int KPl) {
        offt = em[EM_OFF * KPl];
        offn = em[EM_OFF * KPl + 1];
        cx = em[EM_OFF * KPl + 2];
        cy = em[EM_OFF * KPl + 3];
    }
    __device__ __forceinline__ float off(bool tremor) const { return tremor ? offt : offn; }
};

// Emission constants of two states. The density's exponent is taken as two
// squares of affine forms of the centred location, five packed operations a
// pair where differences from the mean and their products take seven; the FMA
// pipe is what the strands run on. Its rounding is that of the location itself
// (float32, at most 2^-24 of the states' spread): 1e-5 in log2 at three
// deviations of a state 1/60 of the box wide, without bias over a chain.
struct Emis2 {
    f32x2 ux, uy, u0, wy, w0, nctr;  // nctr = -(ctr - offset)
    float cno0, cno1;

    __device__ __forceinline__ void load(const float *__restrict__ em, int KPl, int k0, float offt, float offn) {
        float v[2][7];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int k = k0 + u;
            const bool in = k < KPl;
#pragma unroll
            for (int r = 0; r < 5; ++r) v[u][r] = in ? em[(EM_UX + r) * KPl + k] : 0.0f;
            v[u][5] = in ? offt - em[EM_CTR * KPl + k] : INFINITY;
            v[u][6] = in ? em[EM_CNO * KPl + k] - offn : -INFINITY;
        }
        ux = pack2(v[0][0], v[1][0]);
        uy = pack2(v[0][1], v[1][1]);
        u0 = pack2(v[0][2], v[1][2]);
        wy = pack2(v[0][3], v[1][3]);
        w0 = pack2(v[0][4], v[1][4]);
        nctr = pack2(v[0][5], v[1][5]);
        cno0 = v[0][6];
        cno1 = v[1][6];
    }
    // log2 emission factors of the centred observation (x, y)
    __device__ __forceinline__ void eval(float x, float y, bool tremor, float &l0, float &l1) const {
        const f32x2 xx = pack2(x, x), yy = pack2(y, y);
        const f32x2 u = fma2(ux, xx, fma2(uy, yy, u0)), w = fma2(wy, yy, w0);
        float n0, n1;
        unpack2(fma2(w, w, fma2(u, u, nctr)), n0, n1);
        l0 = tremor ? -n0 : cno0;
        l1 = tremor ? -n1 : cno1;
    }
};

// Marks proposal q for the chunk products (once).
__device__ __forceinline__ void send_to_chunks(const StrandPtrs &sp, int q) {
    if (atomicCAS(&sp.route[q], ROUTE_STRANDS, ROUTE_CHUNKS) == ROUTE_STRANDS)
        sp.todo[1 + atomicAdd(&sp.todo[0], 1)] = q;
}

}  // namespace hmm
