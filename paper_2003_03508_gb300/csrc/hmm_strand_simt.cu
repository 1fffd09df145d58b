// Strands on the CUDA cores: FP32 whatever the call's precision, for
// HMM_PREC_FP32_SIMT, for the other precisions where the batch has too few
// strands for the tensor cores' rows, and for the posterior of one sequence,
// which keeps the vector of every step (hmm_smooth.cu; its backward vectors are
// FP32 too, so P is never rounded here: forward vectors on a P rounded to TF32
// put gamma off by up to 2.6e-3). See hmm_strand.cuh for the method and
// hmm_strand_simt.cuh for the layout.
//
// What bounds it: the FMA pipe's register ports. One step of a warp at KP = 32
// is 64 packed FMAs of 2.2 cycles (the vector's pair repeats over four columns;
// three distinct pairs take 3), 10 for the emissions, and some 60 other issues:
// 250 cycles for four strands with two warps per scheduler, 63 a strand-step.
#include "hmm_strand_simt.cuh"

namespace hmm {

namespace {

constexpr unsigned FULL = 0xffffffffu;

// KEEP: alpha [steps + 1][KP] receives the (scaled) vector of every step
template <class C, bool KEEP>
__global__ void __launch_bounds__(32 * STRAND_WPC, C::MIN_CTAS)
strand_simt_kernel(int n_prop, int K, int init_mode, ConstLayout lay, const float *__restrict__ cblock,
                   const float *__restrict__ pi_all, const float2 *__restrict__ head,
                   const float2 *__restrict__ packed, StrandPtrs sp, float *__restrict__ alpha) {
    constexpr int KP = C::KP, G = C::G, NS = C::NS;
    // posterior rows multiply a forward by a backward vector: less room to shrink
    constexpr float SHRINK = KEEP ? STRAND_SHRINK_KEEP : STRAND_SHRINK;
    __shared__ __align__(16) float sv[STRAND_WPC][2 * C::PER_WARP * C::STRIDE];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wpp = (sp.n + C::PER_WARP - 1) / C::PER_WARP;  // warps per proposal
    const long long wid = (long long)blockIdx.x * STRAND_WPC + warp;
    const int q = (int)(wid / wpp);
    if (q >= n_prop) return;
    // one lane's answer for the warp: another warp may change it meanwhile (whole warps leave: no CTA barrier below)
    if (__shfl_sync(FULL, sp.route[q], 0) != ROUTE_STRANDS) return;
    const float *cb = cblock + (size_t)q * lay.stride;
    const float *em = cb + lay.off_emis;
    const int KPl = lay.KP;

    SimtStrand<C> S;
    S.init(sv[warp], lane);
    S.load(cb + lay.off_p32, KPl, false);
    const int own = S.own;
    StrandBase base;
    base.load(em, KPl);
    const int ct = (int)base.offt, cn = (int)base.offn;
    Emis2 ec[NS / 2];
#pragma unroll
    for (int u = 0; u < NS / 2; ++u) ec[u].load(em, KPl, own + 2 * u);

    const int k = (int)(wid % wpp) * C::PER_WARP + S.slot;
    const int sid = k < sp.n ? sp.order[k] : -1;
    const StrandDesc d = sp.desc[sid < 0 ? 0 : sid];
    const int total = sid < 0 ? 0 : d.warm + d.len;
    const float4 *obs = reinterpret_cast<const float4 *>(packed + d.pstart - d.warm);
    float *arow = KEEP ? alpha + ((size_t)d.pstart - d.warm + 1) * KP : nullptr;  // row of the first step's observation
    bool bad = false;
    float v[NS];
    int e32 = 0;
    long long e64 = 0;
    int nwin = (total + 3) / 4;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nwin = max(nwin, __shfl_xor_sync(FULL, nwin, o));

    {  // start: the head vector, or flat
        const bool at_head = (d.flags & SD_HEAD) != 0;
        const float2 o = head[d.seg];
        const bool tr = !isnan(o.x);
        float l[NS], m = -INFINITY;
#pragma unroll
        for (int u = 0; u < NS / 2; ++u) ec[u].sizes(o.x, o.y, tr, l[2 * u], l[2 * u + 1]);
#pragma unroll
        for (int u = 0; u < NS; ++u) {
            const int s = own + u;
            float w = 0.0f;
            if (s < K) {
                if (init_mode == HMM_INIT_TRANSITION_FIRST) {
                    double t = 0.0;
                    for (int i = 0; i < K; ++i) t += (double)pi_all[(size_t)q * K + i] * (double)cb[lay.off_p32 + i * KPl + s];
                    w = (float)t;
                } else {
                    w = pi_all[(size_t)q * K + s];
                }
            }
            v[u] = w;
            if (w > 0.0f) m = fmaxf(m, l[u]);
        }
        m = S.max_all(m);
        const bool emits = m + base.off(tr) >= -(float)EXP_LIMIT;
        const float fm = emits ? floorf(m) : 0.0f;
        if (at_head && emits) e32 = (int)fm + (tr ? ct : cn);
        bad = at_head && !emits;
#pragma unroll
        for (int u = 0; u < NS / 2; ++u) ec[u].factors(o.x, o.y, tr, fm, l[2 * u], l[2 * u + 1]);
#pragma unroll
        for (int u = 0; u < NS; ++u) {
            if (at_head && emits) v[u] = v[u] > 0.0f ? v[u] * l[u] : 0.0f;
            else v[u] = own + u < K ? 1.0f : 0.0f;
        }
        if (KEEP && (d.flags & SD_FIRST) && sid >= 0) S.store(alpha, v);
    }

    float4 na = make_float4(0.f, 0.f, 0.f, 0.f), nb = na;  // the next window's observations
    if (total > 0) {
        na = obs[0];
        nb = obs[1];
    }
    for (int w = 0; w < nwin; ++w) {
        const float ox[4] = {na.x, na.z, nb.x, nb.z}, oy[4] = {na.y, na.w, nb.y, nb.w};
        if (4 * (w + 1) < total) {
            na = obs[2 * (w + 1)];
            nb = obs[2 * (w + 1) + 1];
        }
        float keep[NS];
        int step_e = 0;
#pragma unroll
        for (int u = 0; u < NS; ++u) keep[u] = v[u];
        const int left = total - 4 * w;  // steps of this strand still to do
        const bool own_steps = KEEP && left >= 4 && 4 * w >= d.warm;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float f[NS], y[NS];
            const bool tr = !isnan(ox[j]);
            step_e += tr ? ct : cn;
#pragma unroll
            for (int u = 0; u < NS / 2; ++u) ec[u].factors(ox[j], oy[j], tr, 0.0f, f[2 * u], f[2 * u + 1]);
            S.mul(v, y);
#pragma unroll
            for (int u = 0; u < NS; ++u) v[u] = y[u] * f[u];
            if (own_steps) S.store(arow + (size_t)(4 * w + j) * KP, v);
        }
        const float m = S.max_all(S.max_own(v));
        const bool fine = left >= 4 && m >= SHRINK && m <= STRAND_GROW;
        const bool redo = left > 0 && !fine;
        {
            const int x = float_exponent(m);
            const float s = pow2f(-x);
#pragma unroll
            for (int u = 0; u < NS; ++u) v[u] = fine ? v[u] * s : keep[u];
            e32 += fine ? step_e + x : 0;
        }
        if (__any_sync(FULL, redo)) {
            // one step at a time with exact scaling: a window that shrank too
            // far, or a piece's last steps
            for (int j = 0; j < 4; ++j) {
                float y[NS], l[NS], z[NS], mx = -INFINITY;
                S.mul(v, y);
                const float x = j == 0 ? ox[0] : j == 1 ? ox[1] : j == 2 ? ox[2] : ox[3];
                const float yy = j == 0 ? oy[0] : j == 1 ? oy[1] : j == 2 ? oy[2] : oy[3];
                const bool tr = !isnan(x);
#pragma unroll
                for (int u = 0; u < NS / 2; ++u) ec[u].sizes(x, yy, tr, l[2 * u], l[2 * u + 1]);
                mx = S.max_all(S.max_own(l));
                const bool emits = mx + base.off(tr) >= -(float)EXP_LIMIT;
                const float fm = emits ? floorf(mx) : 0.0f;
#pragma unroll
                for (int u = 0; u < NS / 2; ++u) ec[u].factors(x, yy, tr, fm, l[2 * u], l[2 * u + 1]);
#pragma unroll
                for (int u = 0; u < NS; ++u) z[u] = y[u] * l[u];
                mx = S.max_all(S.max_own(z));
                const bool can = emits && mx >= STRAND_SHRINK && mx <= STRAND_GROW;
                const bool mine = redo && j < left;
                if (mine && can) {
                    const int ex = float_exponent(mx);
                    const float s = pow2f(-ex);
#pragma unroll
                    for (int u = 0; u < NS; ++u) v[u] = z[u] * s;
                    e32 += (int)fm + (tr ? ct : cn) + ex;
                    if (KEEP && 4 * w + j >= d.warm) S.store(arow + (size_t)(4 * w + j) * KP, v);
                } else if (mine) {
                    bad = true;  // the chunk products decide (zero likelihood, range, invalid data)
                }
            }
        }
        if ((w & 63) == 63) {
            e64 += e32;
            e32 = 0;
        }
        if (4 * (w + 1) == d.warm && total > 0) {
            // the piece starts here
            S.store(sp.vs + ((size_t)q * sp.n + sid) * KP, v);
            e64 = 0;
            e32 = 0;
        }
    }
    if (sid < 0) return;
    const size_t idx = (size_t)q * sp.n + sid;
    S.store(sp.ve + idx * KP, v);
    if (lane % G == 0) {
        sp.ex[idx] = e64 + e32;
        if (bad) send_to_chunks(sp, q);
    }
}

template <int KP>
cudaError_t launch_t(int n_prop, int K, int init_mode, const ConstLayout &lay, const float *cblock,
                     const float *pi, const float2 *head, const float2 *packed, const StrandPtrs &sp, float *alpha,
                     cudaStream_t st) {
    auto go = [&](auto kern, int per_warp) {
        const long long warps = (long long)n_prop * ((sp.n + per_warp - 1) / per_warp);
        kern<<<(unsigned)((warps + STRAND_WPC - 1) / STRAND_WPC), 32 * STRAND_WPC, 0, st>>>(
            n_prop, K, init_mode, lay, cblock, pi, head, packed, sp, alpha);
        return cudaGetLastError();
    };
    using C = SimtTile<KP>;
    constexpr bool two = KP == 16 || KP == 32;
    using C2 = SimtTile<KP, two ? 2 : C::H>;
    if (two && (long long)n_prop * sp.n < (1 << 20) && strand_rows(KP, n_prop * sp.n) == 2)
        return alpha ? go(strand_simt_kernel<C2, true>, C2::PER_WARP) : go(strand_simt_kernel<C2, false>, C2::PER_WARP);
    return alpha ? go(strand_simt_kernel<C, true>, C::PER_WARP) : go(strand_simt_kernel<C, false>, C::PER_WARP);
}

}  // namespace

int strand_simt_kp(int K) { return K <= 4 ? 4 : K <= 8 ? 8 : K <= 16 ? 16 : K <= 32 ? 32 : K <= 64 ? 64 : 0; }

cudaError_t launch_strand_simt(int n_prop, int K, int init_mode, const ConstLayout &lay,
                               const float *cblock, const float *pi, const float2 *head, const float2 *packed,
                               const StrandPtrs &sp, float *alpha, cudaStream_t st) {
    if (sp.n == 0) return cudaSuccess;
    switch (strand_simt_kp(K)) {
        case 4: return launch_t<4>(n_prop, K, init_mode, lay, cblock, pi, head, packed, sp, alpha, st);
        case 8: return launch_t<8>(n_prop, K, init_mode, lay, cblock, pi, head, packed, sp, alpha, st);
        case 16: return launch_t<16>(n_prop, K, init_mode, lay, cblock, pi, head, packed, sp, alpha, st);
        case 32: return launch_t<32>(n_prop, K, init_mode, lay, cblock, pi, head, packed, sp, alpha, st);
        case 64: return launch_t<64>(n_prop, K, init_mode, lay, cblock, pi, head, packed, sp, alpha, st);
        default: return cudaErrorInvalidValue;
    }
}

int strand_simt_per_warp(int KP) {
    switch (KP) {
        case 4: return SimtTile<4>::PER_WARP;
        case 8: return SimtTile<8>::PER_WARP;
        case 16: return SimtTile<16>::PER_WARP;
        case 32: return SimtTile<32>::PER_WARP;
        default: return SimtTile<64>::PER_WARP;
    }
}

}  // namespace hmm
