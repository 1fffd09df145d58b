// Strands on the CUDA cores (FP32): HMM_PREC_FP32_SIMT, and the other precisions
// where the batch has too few strands for the tensor cores' rows (with P rounded
// to TF32 for HMM_PREC_TF32). See hmm_strand.cuh for the method.
//
// A strand is carried by G threads. Each holds the four columns of P it is
// responsible for (KP / H of their rows) in registers, as pairs over the row
// index, so a step reads the vector from shared memory as 16-byte broadcasts
// (one load feeds 16 FMAs) and nothing else: one step of KP = 32 is 64 packed
// FMAs and 8 loads per thread, and a warp carries four strands. The threads
// exchange the vector through a double buffer of their own warp (one
// __syncwarp per step). For KP = 64 two half-warps take half of the rows each
// and swap two partial sums.
//
// What bounds it: the FMA pipe, 2 K^2 flops per strand-step at 128 lanes per
// SM and cycle, plus seven packed operations and one EX2 per two emissions.
#include "hmm_strand.cuh"

namespace hmm {

namespace {

constexpr int WPC = 4;  // warps per CTA

template <int KP_, int R_>
struct SimtTile {
    static constexpr int KP = KP_;
    static constexpr int R = R_;                  // strands per thread group
    static constexpr int H = KP > 32 ? 2 : 1;     // row split
    static constexpr int CG = KP / 4;             // column groups
    static constexpr int G = CG * H;              // threads per strand
    static constexpr int NI = KP / H;             // rows of P per thread
    static constexpr int NS = 4 / H;              // states a thread owns
    static constexpr int PER_WARP = (32 / G) * R; // strands per warp
    // one strand's vector in shared memory, padded so that the broadcasts of
    // different strands (and of the two row halves) fall on different banks
    static constexpr int STRIDE = KP + 4 * H;
    static __device__ __forceinline__ int at(int i) { return H == 1 ? i : i + 4 * (i / 32); }
};

template <class C>
__global__ void __launch_bounds__(32 * WPC, C::KP >= 32 ? 2 : C::KP >= 8 ? 3 : 4)
strand_simt_kernel(int n_prop, int K, int init_mode, ConstLayout lay, bool round_tf32, const float *__restrict__ cblock,
                   const float *__restrict__ pi_all, const float2 *__restrict__ head,
                   const float2 *__restrict__ packed, StrandPtrs sp) {
    constexpr int KP = C::KP, R = C::R, G = C::G, NI = C::NI, NS = C::NS, H = C::H;
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ __align__(16) float sv[WPC][2][KP == 4 ? 1 : C::PER_WARP][KP == 4 ? 4 : C::STRIDE];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wpp = (sp.n + C::PER_WARP - 1) / C::PER_WARP;  // warps per proposal
    const long long wid = (long long)blockIdx.x * WPC + warp;
    const int q = (int)(wid / wpp);
    if (q >= n_prop) return;
    // one lane's answer for the warp: another warp may change it meanwhile (whole warps leave: no CTA barrier below)
    if (__shfl_sync(FULL, sp.route[q], 0) != ROUTE_STRANDS) return;
    const int w0 = (int)(wid % wpp) * C::PER_WARP;
    const int g = lane % G, slot = lane / G;
    const int cg = g % C::CG, h = g / C::CG;
    const int own = 4 * cg + NS * h;  // first state this thread owns
    const float *cb = cblock + (size_t)q * lay.stride;
    const float *em = cb + lay.off_emis;
    const int KPl = lay.KP;

    // P columns 4 cg .. 4 cg + 3, rows h NI .. (pairs), and emission constants
    f32x2 p[4][NI / 2];
#pragma unroll
    for (int i = 0; i < NI / 2; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float v[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int row = h * NI + 2 * i + u, col = 4 * cg + c;
                v[u] = row < KPl && col < KPl ? cb[lay.off_p32 + row * KPl + col] : 0.0f;
                if (round_tf32) {
                    uint32_t r;
                    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(v[u]));
                    v[u] = __uint_as_float(r);
                }
            }
            p[c][i] = pack2(v[0], v[1]);
        }
    StrandBase base;
    base.load(em, KPl);
    const int ct = (int)base.offt, cn = (int)base.offn;
    Emis2 ec[NS / 2];
#pragma unroll
    for (int u = 0; u < NS / 2; ++u) ec[u].load(em, KPl, own + 2 * u, base.offt, base.offn);

    // this thread's strands
    const float4 *obs[R];
    int total[R], warm[R], sid[R];
    bool bad[R];
    float v[R][NS];
    int e32[R];
    long long e64[R];
    int nwin = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int k = w0 + slot + r * (32 / G);
        sid[r] = k < sp.n ? sp.order[k] : -1;
        const StrandDesc d = sp.desc[sid[r] < 0 ? 0 : sid[r]];
        total[r] = sid[r] < 0 ? 0 : d.warm + d.len;
        warm[r] = d.warm;
        obs[r] = reinterpret_cast<const float4 *>(packed + d.pstart - d.warm);
        bad[r] = false;
        e32[r] = 0;
        e64[r] = 0;
        nwin = max(nwin, (total[r] + 3) / 4);
        // start: the head vector, or flat
        const bool at_head = (d.flags & SD_HEAD) != 0;
        const float2 o = head[d.seg];
        const bool tr = !isnan(o.x);
        float l[NS], m = -INFINITY;
#pragma unroll
        for (int u = 0; u < NS / 2; ++u) ec[u].eval(o.x - base.cx, o.y - base.cy, tr, l[2 * u], l[2 * u + 1]);
#pragma unroll
        for (int u = 0; u < NS; ++u) {
            const int k = own + u;
            float w = 0.0f;
            if (k < K) {
                if (init_mode == HMM_INIT_TRANSITION_FIRST) {
                    double s = 0.0;
                    for (int i = 0; i < K; ++i) s += (double)pi_all[(size_t)q * K + i] * (double)cb[lay.off_p32 + i * KPl + k];
                    w = (float)s;
                } else {
                    w = pi_all[(size_t)q * K + k];
                }
            }
            v[r][u] = w;
            if (w > 0.0f) m = fmaxf(m, l[u]);
        }
#pragma unroll
        for (int o = 1; o < G; o <<= 1) m = fmaxf(m, __shfl_xor_sync(FULL, m, o));
        if (at_head) {
            if (m + base.off(tr) >= -(float)EXP_LIMIT) {
                const float fm = floorf(m);
                e32[r] = (int)fm + (tr ? ct : cn);
#pragma unroll
                for (int u = 0; u < NS; ++u) v[r][u] = v[r][u] > 0.0f ? v[r][u] * ex2(l[u] - fm) : 0.0f;
            } else {
                bad[r] = true;
            }
        }
        if (!at_head || bad[r])
#pragma unroll
            for (int u = 0; u < NS; ++u) v[r][u] = own + u < K ? 1.0f : 0.0f;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nwin = max(nwin, __shfl_xor_sync(FULL, nwin, o));

    int buf = 0;
    // w = v P for every strand of the warp (this thread's owned states)
    auto advance = [&](const float (&x)[R][NS], float (&y)[R][NS]) {
        if (KP > 4) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float *dst = &sv[warp][buf][slot + r * (32 / G)][C::at(own)];
                if (NS == 4) *reinterpret_cast<float4 *>(dst) = make_float4(x[r][0], x[r][1], x[r][NS - 2], x[r][NS - 1]);
                else *reinterpret_cast<float2 *>(dst) = make_float2(x[r][0], x[r][1]);
            }
            __syncwarp();
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            f32x2 acc[4] = {0ull, 0ull, 0ull, 0ull};
            const float *src = &sv[warp][buf][KP == 4 ? 0 : slot + r * (32 / G)][KP == 4 ? 0 : C::at(h * NI)];
#pragma unroll
            for (int i = 0; i < NI / 4; ++i) {
                f32x2 a, b;
                if (KP == 4) {
                    a = pack2(x[r][0], x[r][1]);
                    b = pack2(x[r][NS - 2], x[r][NS - 1]);
                } else {
                    const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(src + 4 * i);
                    a = t.x;
                    b = t.y;
                }
                // a and b each four times in a row: their registers are read once
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[c] = fma2(a, p[c][2 * i], acc[c]);
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[c] = fma2(b, p[c][2 * i + 1], acc[c]);
            }
            float s[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float lo, hi;
                unpack2(acc[c], lo, hi);
                s[c] = lo + hi;
            }
            if (H == 1) {
#pragma unroll
                for (int u = 0; u < NS; ++u) y[r][u] = s[u];
            } else {
                // the other half's rows: swap the two sums each half does not own
                const float t0 = __shfl_xor_sync(FULL, h ? s[0] : s[2], 16);
                const float t1 = __shfl_xor_sync(FULL, h ? s[1] : s[3], 16);
                y[r][0] = (h ? s[2] : s[0]) + t0;
                y[r][1] = (h ? s[3] : s[1]) + t1;
            }
        }
        buf ^= 1;
    };

    float4 na[R], nb[R];  // the next window's observations
#pragma unroll
    for (int r = 0; r < R; ++r) {
        na[r] = total[r] > 0 ? obs[r][0] : make_float4(0.f, 0.f, 0.f, 0.f);
        nb[r] = total[r] > 0 ? obs[r][1] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int w = 0; w < nwin; ++w) {
        float ox[R][4], oy[R][4], keep[R][NS];
        int step_e[R];
        bool ok = true;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            ox[r][0] = na[r].x; oy[r][0] = na[r].y; ox[r][1] = na[r].z; oy[r][1] = na[r].w;
            ox[r][2] = nb[r].x; oy[r][2] = nb[r].y; ox[r][3] = nb[r].z; oy[r][3] = nb[r].w;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                ox[r][j] -= base.cx;
                oy[r][j] -= base.cy;
            }
            if (4 * (w + 1) < total[r]) {
                na[r] = obs[r][2 * (w + 1)];
                nb[r] = obs[r][2 * (w + 1) + 1];
            }
#pragma unroll
            for (int u = 0; u < NS; ++u) keep[r][u] = v[r][u];
            step_e[r] = 0;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float f[R][NS], y[R][NS];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const bool tr = !isnan(ox[r][j]);
                step_e[r] += tr ? ct : cn;
#pragma unroll
                for (int u = 0; u < NS / 2; ++u) {
                    ec[u].eval(ox[r][j], oy[r][j], tr, f[r][2 * u], f[r][2 * u + 1]);
                    f[r][2 * u] = ex2(f[r][2 * u]);
                    f[r][2 * u + 1] = ex2(f[r][2 * u + 1]);
                }
            }
            advance(v, y);
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int u = 0; u < NS; ++u) v[r][u] = y[r][u] * f[r][u];
        }
        bool redo[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float m = fmaxf(fmaxf(v[r][0], v[r][1]), fmaxf(v[r][NS - 2], v[r][NS - 1]));
#pragma unroll
            for (int o = 1; o < G; o <<= 1) m = fmaxf(m, __shfl_xor_sync(FULL, m, o));
            const int left = total[r] - 4 * w;  // steps of this strand still to do
            const bool fine = left >= 4 && m >= STRAND_SHRINK && m <= STRAND_GROW;
            redo[r] = left > 0 && !fine;
            ok = ok && !redo[r];
            const int x = float_exponent(m);
            const float s = pow2f(-x);
#pragma unroll
            for (int u = 0; u < NS; ++u) v[r][u] = fine ? v[r][u] * s : keep[r][u];
            e32[r] += fine ? step_e[r] + x : 0;
        }
        if (!__all_sync(FULL, ok)) {
            // one step at a time with exact scaling: a window that shrank too
            // far, or a piece's last steps
            for (int j = 0; j < 4; ++j) {
                float y[R][NS];
                advance(v, y);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float x = j == 0 ? ox[r][0] : j == 1 ? ox[r][1] : j == 2 ? ox[r][2] : ox[r][3];
                    const float yy = j == 0 ? oy[r][0] : j == 1 ? oy[r][1] : j == 2 ? oy[r][2] : oy[r][3];
                    const bool tr = !isnan(x);
                    float l[NS], m = -INFINITY;
#pragma unroll
                    for (int u = 0; u < NS / 2; ++u) ec[u].eval(x, yy, tr, l[2 * u], l[2 * u + 1]);
#pragma unroll
                    for (int u = 0; u < NS; ++u) m = fmaxf(m, l[u]);
#pragma unroll
                    for (int o = 1; o < G; o <<= 1) m = fmaxf(m, __shfl_xor_sync(FULL, m, o));
                    const bool emits = m + base.off(tr) >= -(float)EXP_LIMIT;
                    const float fm = emits ? floorf(m) : 0.0f;
                    float z[NS], mx = 0.0f;
#pragma unroll
                    for (int u = 0; u < NS; ++u) {
                        z[u] = y[r][u] * ex2(l[u] - fm);
                        mx = fmaxf(mx, z[u]);
                    }
#pragma unroll
                    for (int o = 1; o < G; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, o));
                    const bool fine = emits && mx >= STRAND_SHRINK && mx <= STRAND_GROW;
                    const bool mine = redo[r] && j < total[r] - 4 * w;
                    if (mine && fine) {
                        const int ex = float_exponent(mx);
                        const float s = pow2f(-ex);
#pragma unroll
                        for (int u = 0; u < NS; ++u) v[r][u] = z[u] * s;
                        e32[r] += (int)fm + (tr ? ct : cn) + ex;
                    } else if (mine) {
                        bad[r] = true;  // the chunk products decide (zero likelihood, range, invalid data)
                    }
                }
            }
        }
        if ((w & 63) == 63) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                e64[r] += e32[r];
                e32[r] = 0;
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (4 * (w + 1) == warm[r] && total[r] > 0) {
                // the piece starts here
                float *dst = sp.vs + ((size_t)q * sp.n + sid[r]) * KP + own;
#pragma unroll
                for (int u = 0; u < NS; ++u) dst[u] = v[r][u];
                e64[r] = 0;
                e32[r] = 0;
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (sid[r] < 0) continue;
        const size_t idx = (size_t)q * sp.n + sid[r];
#pragma unroll
        for (int u = 0; u < NS; ++u) sp.ve[idx * KP + own + u] = v[r][u];
        if (g == 0) {
            sp.ex[idx] = e64[r] + e32[r];
            if (bad[r]) send_to_chunks(sp, q);
        }
    }
}

template <int KP, int R>
cudaError_t launch_t(int n_prop, int K, int init_mode, const ConstLayout &lay, bool round_tf32, const float *cblock,
                     const float *pi, const float2 *head, const float2 *packed, const StrandPtrs &sp,
                     cudaStream_t st) {
    using C = SimtTile<KP, R>;
    const long long warps = (long long)n_prop * ((sp.n + C::PER_WARP - 1) / C::PER_WARP);
    strand_simt_kernel<C><<<(unsigned)((warps + WPC - 1) / WPC), 32 * WPC, 0, st>>>(
        n_prop, K, init_mode, lay, round_tf32, cblock, pi, head, packed, sp);
    return cudaGetLastError();
}

}  // namespace

int strand_simt_kp(int K) { return K <= 4 ? 4 : K <= 8 ? 8 : K <= 16 ? 16 : K <= 32 ? 32 : K <= 64 ? 64 : 0; }

cudaError_t launch_strand_simt(int n_prop, int K, int init_mode, const ConstLayout &lay, int precision,
                               const float *cblock, const float *pi, const float2 *head, const float2 *packed,
                               const StrandPtrs &sp, cudaStream_t st) {
    if (sp.n == 0) return cudaSuccess;
    const bool rt = precision == HMM_PREC_TF32;
    switch (strand_simt_kp(K)) {
        case 4: return launch_t<4, 1>(n_prop, K, init_mode, lay, rt, cblock, pi, head, packed, sp, st);
        case 8: return launch_t<8, 1>(n_prop, K, init_mode, lay, rt, cblock, pi, head, packed, sp, st);
        case 16: return launch_t<16, 1>(n_prop, K, init_mode, lay, rt, cblock, pi, head, packed, sp, st);
        case 32: return launch_t<32, 1>(n_prop, K, init_mode, lay, rt, cblock, pi, head, packed, sp, st);
        case 64: return launch_t<64, 1>(n_prop, K, init_mode, lay, rt, cblock, pi, head, packed, sp, st);
        default: return cudaErrorInvalidValue;
    }
}

int strand_simt_per_warp(int KP) {
    switch (KP) {
        case 4: return SimtTile<4, 1>::PER_WARP;
        case 8: return SimtTile<8, 1>::PER_WARP;
        case 16: return SimtTile<16, 1>::PER_WARP;
        case 32: return SimtTile<32, 1>::PER_WARP;
        default: return SimtTile<64, 1>::PER_WARP;
    }
}

}  // namespace hmm
