// What the CUDA-core strand kernels share (hmm_strand_simt.cu forward,
// hmm_smooth.cu backward): how a strand's vector is spread over threads and
// multiplied by P.
#pragma once

#include "hmm_strand.cuh"

namespace hmm {

constexpr int STRAND_WPC = 4;  // warps per CTA

// A strand is carried by G threads. Each holds the four columns of the matrix
// it is responsible for (KP / H of their rows) in registers, as pairs over the
// row index, so a step reads the vector from shared memory as 16-byte
// broadcasts (one load feeds 16 FMAs) and nothing else: one step of KP = 32 is
// 64 packed FMAs and 8 loads per thread, and a warp carries four strands. With
// H = 2 twice the threads take half of the rows each and swap two partial sums:
// for KP = 64, whose columns do not fit one thread otherwise, and for sequences
// with too few strands to give every scheduler a warp, where a step's latency is
// what counts (strand_rows).
template <int KP_, int H_ = (KP_ > 32 ? 2 : 1)>
struct SimtTile {
    static constexpr int KP = KP_;
    static constexpr int H = H_;                 // row split
    static constexpr int CG = KP / 4;            // column groups
    static constexpr int G = CG * H;             // threads per strand
    static constexpr int NI = KP / H;            // rows per thread
    static constexpr int NS = 4 / H;             // states a thread owns
    static constexpr int PER_WARP = 32 / G;      // strands per warp
    static constexpr int MIN_CTAS = KP >= 32 ? 2 : KP >= 8 ? 3 : 4;
    // one strand's vector in shared memory, padded so that the broadcasts of
    // different strands (and of the two row halves) fall on different banks
    static constexpr int STRIDE = KP + 4 * H;
    static __device__ __forceinline__ int at(int i) { return H == 1 ? i : i + 4 * (i / NI); }
};

// Row split for n strands in all: two while one row block would leave schedulers
// without a warp (4 on each of 152 SMs). Posterior K=25, T=105,000: forward 53 ->
// 43 us, backward 98 -> 81; Viterbi's strands 148 -> 98.
inline int strand_rows(int KP, int n) {
    return KP == 64 ? 2 : (KP == 32 && n <= 4 * 608) || (KP == 16 && n <= 8 * 608) ? 2 : 1;
}

template <class C>
struct SimtStrand {
    f32x2 p[4][C::NI / 2];
    float *row;  // this strand's place in the warp's first buffer
    int slot, cg, h, own, buf;

    // `mem`: the warp's two buffers of C::PER_WARP vectors
    __device__ __forceinline__ void init(float *mem, int lane) {
        const int g = lane % C::G;
        slot = lane / C::G;
        cg = g % C::CG;
        h = g / C::CG;
        own = 4 * cg + C::NS * h;  // first state this thread owns
        row = mem + slot * C::STRIDE;
        buf = 0;
    }
    // the matrix: P (row vector times P), or with `transposed` P^T (P times a column vector)
    __device__ __forceinline__ void load(const float *__restrict__ P, int KPl, bool transposed) {
#pragma unroll
        for (int i = 0; i < C::NI / 2; ++i)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float v[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int r = h * C::NI + 2 * i + u, k = 4 * cg + c;
                    v[u] = r < KPl && k < KPl ? P[transposed ? k * KPl + r : r * KPl + k] : 0.0f;
                }
                p[c][i] = pack2(v[0], v[1]);
            }
    }
    // y = x times the matrix, this thread's owned states of both
    __device__ __forceinline__ void mul(const float (&x)[C::NS], float (&y)[C::NS]) {
        constexpr int NS = C::NS;
        float *const b = row + buf * C::PER_WARP * C::STRIDE;
        if (C::KP > 4) {
            if (NS == 4) *reinterpret_cast<float4 *>(b + C::at(own)) = make_float4(x[0], x[1], x[NS - 2], x[NS - 1]);
            else *reinterpret_cast<float2 *>(b + C::at(own)) = make_float2(x[0], x[1]);
            __syncwarp();
        }
        f32x2 acc[4] = {0ull, 0ull, 0ull, 0ull};
        const float *src = b + C::at(h * C::NI);
#pragma unroll
        for (int i = 0; i < C::NI / 4; ++i) {
            f32x2 t, w;
            if (C::KP == 4) {
                t = pack2(x[0], x[1]);
                w = pack2(x[NS - 2], x[NS - 1]);
            } else {
                const ulonglong2 z = *reinterpret_cast<const ulonglong2 *>(src + 4 * i);
                t = z.x;
                w = z.y;
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[c] = fma2(t, p[c][2 * i], acc[c]);
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[c] = fma2(w, p[c][2 * i + 1], acc[c]);
        }
        float s[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float lo, hi;
            unpack2(acc[c], lo, hi);
            s[c] = lo + hi;
        }
        if (C::H == 1) {
#pragma unroll
            for (int u = 0; u < NS; ++u) y[u] = s[u];
        } else {
            // the other half's rows: swap the two sums each half does not own
            const float t0 = __shfl_xor_sync(0xffffffffu, h ? s[0] : s[2], C::CG);
            const float t1 = __shfl_xor_sync(0xffffffffu, h ? s[1] : s[3], C::CG);
            y[0] = (h ? s[2] : s[0]) + t0;
            y[1] = (h ? s[3] : s[1]) + t1;
        }
        buf ^= 1;
    }
    // over the strand's threads
    static __device__ __forceinline__ float max_all(float m) {
#pragma unroll
        for (int o = 1; o < C::G; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        return m;
    }
    static __device__ __forceinline__ float sum_all(float m) {
#pragma unroll
        for (int o = 1; o < C::G; o <<= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
        return m;
    }
    static __device__ __forceinline__ float max_own(const float (&v)[C::NS]) {
        return fmaxf(fmaxf(v[0], v[1]), fmaxf(v[C::NS - 2], v[C::NS - 1]));
    }
    // this thread's states of a row of KP floats
    __device__ __forceinline__ void store(float *r, const float (&v)[C::NS]) const {
        if (C::NS == 4) *reinterpret_cast<float4 *>(r + own) = make_float4(v[0], v[1], v[C::NS - 2], v[C::NS - 1]);
        else *reinterpret_cast<float2 *>(r + own) = make_float2(v[0], v[1]);
    }
    __device__ __forceinline__ void fetch(const float *r, float (&v)[C::NS]) const {
        if (C::NS == 4) {
            const float4 t = *reinterpret_cast<const float4 *>(r + own);
            v[0] = t.x; v[1] = t.y; v[C::NS - 2] = t.z; v[C::NS - 1] = t.w;
        } else {
            const float2 t = *reinterpret_cast<const float2 *>(r + own);
            v[0] = t.x; v[1] = t.y;
        }
    }
};

}  // namespace hmm
