// Posterior probabilities and E-step statistics of one sequence by strands
// (hmm_strand.cuh), in place of two scans over chunk products on one CTA.
//
// The forward strands keep their vector of every step (alpha, any scale). The
// backward vectors b_t = P (d_{t+1} o b_{t+1}) of a piece are carried the same
// way: from a flat vector some steps behind the piece (or from the sequence's
// end, where it is exact) down to the piece's start, checked against the
// strand of the piece behind where the two meet. Each step in the piece gives
//     w = d_t o b_t,  y = P w,  S = sum_i alpha_{t-1}(i) y(i),
//     gamma_{t-1} = alpha_{t-1} o y / S,
// and w / S is what the expected transition counts need:
//     N_ij = P_ij sum_t alpha_{t-1}(i) w_t(j) / S_t,
// a K x T by T x K product taken over blocks of 64 steps in FP32 and summed in
// FP64. The gamma-weighted moments keep what their FP32 products and sums drop.
//
// Vectors that have not met at a piece's edge run on from the true one, and the
// rows passed are written again (rows_join_kernel).
//
// What bounds it: a step of a lone warp, 0.2 us, times warm-up and piece, in
// each direction; at T = 2^20 also the FMA pipe (K=25: 130 us a direction). The
// rows are written once and read once or twice: 0.27 GB at K=32, T=2^20, 40 us.
#include "hmm_strand_simt.cuh"

namespace hmm {

namespace {

constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ float rcp(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// ---- backward strands ----
template <class C>
__global__ void __launch_bounds__(32 * STRAND_WPC, C::MIN_CTAS)
strand_back_kernel(int K, int64_t steps, int warm, ConstLayout lay, const float *__restrict__ cb,
                   const float2 *__restrict__ packed, StrandPtrs sp, SmoothPtrs sm) {
    constexpr int KP = C::KP, NS = C::NS;
    __shared__ __align__(16) float sv[STRAND_WPC][2 * C::PER_WARP * C::STRIDE];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wid = blockIdx.x * STRAND_WPC + warp;
    if (wid * C::PER_WARP >= sp.n) return;
    if (__shfl_sync(FULL, sp.route[0], 0) != ROUTE_STRANDS) return;
    const float *em = cb + lay.off_emis;
    const int KPl = lay.KP;

    SimtStrand<C> S;
    S.init(sv[warp], lane);
    S.load(cb + lay.off_p32, KPl, true);
    const int own = S.own;
    StrandBase base;
    base.load(em, KPl);
    Emis2 ec[NS / 2];
#pragma unroll
    for (int u = 0; u < NS / 2; ++u) ec[u].load(em, KPl, own + 2 * u);

    const int k = wid * C::PER_WARP + S.slot;
    const int sid = k < sp.n ? k : -1;
    const StrandDesc d = sp.desc[sid < 0 ? 0 : sid];
    const int64_t a = d.pstart, b = a + d.len;                // the piece's steps
    const int64_t e = sid < 0 ? a : min(b + (int64_t)warm, steps);  // where the strand starts
    const int64_t wtop = (e + 3) / 4 - 1;
    const int mine = sid < 0 ? 0 : (int)(wtop - a / 4 + 1);
    int nwin = mine;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nwin = max(nwin, __shfl_xor_sync(FULL, nwin, o));
    bool bad = false;
    float v[NS];
#pragma unroll
    for (int u = 0; u < NS; ++u) v[u] = own + u < K ? 1.0f : 0.0f;

    // gamma's row t of the strand's own states from alpha's row and y. gamma is
    // the caller's: any float address, so 16-byte stores only where it allows them
    const bool wide = (K & 3) == 0 && ((uintptr_t)sm.gamma & 15) == 0;
    auto put_gamma = [&](int64_t t, const float (&al)[NS], const float (&y)[NS], float r) {
        float *g = sm.gamma + t * K + own;
        if (wide && NS == 4) {
            if (own < K) *reinterpret_cast<float4 *>(g) = make_float4(al[0] * y[0] * r, al[1] * y[1] * r, al[NS - 2] * y[NS - 2] * r, al[NS - 1] * y[NS - 1] * r);
        } else {
#pragma unroll
            for (int u = 0; u < NS; ++u)
                if (own + u < K) g[u] = al[u] * y[u] * r;
        }
    };
    {  // the sequence's last row
        const bool last = sid >= 0 && (d.flags & SD_LAST);
        float al[NS], t = 0.0f;
#pragma unroll
        for (int u = 0; u < NS; ++u) al[u] = 0.0f;
        if (last) S.fetch(sm.alpha + steps * KP, al);
#pragma unroll
        for (int u = 0; u < NS; ++u) t += al[u];
        t = S.sum_all(t);
        if (last) put_gamma(steps, al, v, 1.0f / t);
    }

    const float4 *obs = reinterpret_cast<const float4 *>(packed);
    float4 na = make_float4(0.f, 0.f, 0.f, 0.f), nb = na;
    if (mine > 0) {
        na = obs[2 * wtop];
        nb = obs[2 * wtop + 1];
    }
    for (int it = 0; it < nwin; ++it) {
        const int64_t w = wtop - it;
        const bool act = it < mine;
        const float ox[4] = {na.x, na.z, nb.x, nb.z};
        const float oy[4] = {na.y, na.w, nb.y, nb.w};
        if (it + 1 < mine) {
            na = obs[2 * (w - 1)];
            nb = obs[2 * (w - 1) + 1];
        }
        if (act && 4 * (w + 1) == b && !(d.flags & SD_LAST)) S.store(sm.bs + (size_t)sid * KP, v);  // the piece begins
        const bool own_steps = act && 4 * w < b;
        const int valid = act ? (int)min((int64_t)4, e - 4 * w) : 0;
        if (it + 1 < mine && 4 * (w - 1) < b) {
            // alpha's rows of the next window
#pragma unroll
            for (int j = 0; j < 4; ++j)
                asm volatile("prefetch.global.L1 [%0];" ::"l"(sm.alpha + (4 * (w - 1) + j) * KP + own));
        }
        float keep[NS];
#pragma unroll
        for (int u = 0; u < NS; ++u) keep[u] = v[u];
        // two steps at a time: the recursion first, then both rows' sums, whose
        // shuffles would otherwise stand between the steps
#pragma unroll
        for (int j2 = 2; j2 >= 0; j2 -= 2) {
            float f[2][NS], y[2][NS], al[2][NS], s[2] = {0.0f, 0.0f};
#pragma unroll
            for (int h = 1; h >= 0; --h) {
                const int j = j2 + h;
#pragma unroll
                for (int u = 0; u < NS / 2; ++u) ec[u].factors(ox[j], oy[j], !isnan(ox[j]), 0.0f, f[h][2 * u], f[h][2 * u + 1]);
#pragma unroll
                for (int u = 0; u < NS; ++u) f[h][u] *= v[u];
                S.mul(f[h], y[h]);
#pragma unroll
                for (int u = 0; u < NS; ++u) v[u] = y[h][u];
            }
            if (!__any_sync(FULL, own_steps && valid == 4)) continue;  // all of the warp's strands are warming up
#pragma unroll
            for (int h = 1; h >= 0; --h) {
#pragma unroll
                for (int u = 0; u < NS; ++u) al[h][u] = 0.0f;
                if (own_steps && valid == 4) S.fetch(sm.alpha + (4 * w + j2 + h) * KP, al[h]);
#pragma unroll
                for (int u = 0; u < NS; ++u) s[h] = fmaf(al[h][u], y[h][u], s[h]);
            }
#pragma unroll
            for (int o = 1; o < C::G; o <<= 1) {
                s[0] += __shfl_xor_sync(FULL, s[0], o);
                s[1] += __shfl_xor_sync(FULL, s[1], o);
            }
            if (own_steps && valid == 4) {
#pragma unroll
                for (int h = 1; h >= 0; --h) {
                    const int64_t i = 4 * w + j2 + h;
                    const float r = rcp(s[h]);
                    put_gamma(i, al[h], y[h], r);
                    if (sm.u) {
#pragma unroll
                        for (int u = 0; u < NS; ++u) f[h][u] *= r;
                        S.store(sm.u + i * KP, f[h]);
                    }
                }
            }
        }
        const float m = S.max_all(S.max_own(v));
        const bool fine = valid == 4 && m >= STRAND_SHRINK_KEEP && m <= STRAND_GROW;
        const bool redo = act && !fine;
        const float sc = pow2f(-float_exponent(m));
#pragma unroll
        for (int u = 0; u < NS; ++u) v[u] = fine ? v[u] * sc : keep[u];
        if (__any_sync(FULL, redo)) {
            for (int j = 3; j >= 0; --j) {
                const int64_t i = 4 * w + j;
                const float x = j == 0 ? ox[0] : j == 1 ? ox[1] : j == 2 ? ox[2] : ox[3];
                const float yy = j == 0 ? oy[0] : j == 1 ? oy[1] : j == 2 ? oy[2] : oy[3];
                const bool todo = redo && j < valid;
                float l[NS], y[NS], al[NS], s = 0.0f;
#pragma unroll
                for (int u = 0; u < NS; ++u) al[u] = 0.0f;
                if (todo && own_steps) S.fetch(sm.alpha + i * KP, al);
#pragma unroll
                for (int u = 0; u < NS / 2; ++u) ec[u].sizes(x, yy, !isnan(x), l[2 * u], l[2 * u + 1]);
                float mx = S.max_all(S.max_own(l));
                const bool emits = mx + base.off(!isnan(x)) >= -(float)EXP_LIMIT;
                const float fm = emits ? floorf(mx) : 0.0f;
#pragma unroll
                for (int u = 0; u < NS / 2; ++u) ec[u].factors(x, yy, !isnan(x), fm, l[2 * u], l[2 * u + 1]);
#pragma unroll
                for (int u = 0; u < NS; ++u) l[u] *= v[u];
                S.mul(l, y);
                mx = S.max_all(S.max_own(y));
                const bool can = emits && mx >= STRAND_SHRINK && mx <= STRAND_GROW;
                const float sy = can ? pow2f(-float_exponent(mx)) : 1.0f;
#pragma unroll
                for (int u = 0; u < NS; ++u) {
                    y[u] *= sy;
                    l[u] *= sy;
                    s = fmaf(al[u], y[u], s);
                }
                s = S.sum_all(s);
                if (todo && can) {
#pragma unroll
                    for (int u = 0; u < NS; ++u) v[u] = y[u];
                    if (own_steps) {
                        const float r = rcp(s);
                        put_gamma(i, al, y, r);
                        if (sm.u) {
#pragma unroll
                            for (int u = 0; u < NS; ++u) l[u] *= r;
                            S.store(sm.u + i * KP, l);
                        }
                    }
                } else if (todo) {
                    bad = true;
                }
            }
        }
    }
    if (sid < 0) return;
    S.store(sm.be + (size_t)sid * KP, v);
    if (lane % C::G == 0 && bad) send_to_chunks(sp, 0);
}

// ---- pieces whose vectors had not met at their edge: rows written again ----
// BACK = false: strand c's first rows of alpha, from the end of strand c - 1.
// BACK = true: strand c's last rows of gamma (and u), from the end of strand
// c + 1. One warp per piece, one step after another with exact scaling. A piece
// that ends first is noted with its true vector (unmet, carry), and a second
// launch (`chain`) takes those on through the pieces that follow once every
// piece has written its rows; after sm.most steps, or where two of them
// touch, the sequence is left to the chunk products.

template <int NC, bool BACK>
__global__ void __launch_bounds__(128)
rows_join_kernel(int K, int KP, bool chain, ConstLayout lay, const float *__restrict__ cb,
                 const float2 *__restrict__ packed, StrandPtrs sp, SmoothPtrs sm) {
    __shared__ __align__(16) float2 sag[4][32 * NC];
    // NC > 1: P, or its transpose, where the step reads it (rows of 64 floats);
    // through the cache a step took some 1.1 us
    __shared__ float sP[NC == 1 ? 1 : 32 * NC][NC == 1 ? 1 : 32 * NC];
    // Every row is a result, so vectors have met where they differ by little more
    // than FP32's rounding: with rare tremors 2^-19.8 of an entry at the median and
    // 2^-18.7 at most of the time for K = 16, 2^-18.8 and 2^-17.8 for K = 32, 2^-17.9
    // and 2^-16.8 for K = 64 (a float32 replay). With 2^-15, which the likelihood's
    // join takes, gamma was up to 1.3e-5 off (K = 16), 5.4e-6 now.
    const float tol = KP <= 16 ? 3.814697265625e-6f : KP <= 32 ? 7.62939453125e-6f : 1.52587890625e-5f;  // 2^-18, -17, -16
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (NC == 1 && __shfl_sync(FULL, sp.route[0], 0) != ROUTE_STRANDS) return;
    const float *em = cb + lay.off_emis, *P = cb + lay.off_p32;
    const int KPl = lay.KP;
    if (NC > 1) {
        for (int x = threadIdx.x; x < 32 * NC * 32 * NC; x += 128) {
            const int i = x / (32 * NC), k = x % (32 * NC);
            sP[NC == 1 ? 0 : BACK ? k : i][NC == 1 ? 0 : BACK ? i : k] = i < K && k < K ? P[i * KPl + k] : 0.0f;
        }
        __syncthreads();
        if (__shfl_sync(FULL, sp.route[0], 0) != ROUTE_STRANDS) return;
    }
    float a[NC], g[NC];
    auto all_max = [&](float v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(FULL, v, o));
        return v;
    };
    auto all_sum = [&](float v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
        return v;
    };
    auto met = [&]() {
        float lo = INFINITY, hi = 0.0f;
        bool numbers = true;  // fmin and fmax pass over what is not
#pragma unroll
        for (int n = 0; n < NC; ++n) {
            numbers = numbers && a[n] == a[n] && g[n] == g[n];
            if (a[n] > STRAND_TINY || g[n] > STRAND_TINY) {
                const float r = a[n] / g[n];
                lo = fminf(lo, r);
                hi = fmaxf(hi, r);
            }
        }
        hi = all_max(hi);
        return __all_sync(FULL, numbers) && hi > 0.0f && hi < INFINITY && hi <= -all_max(-lo) * (1.0f + tol);
    };
    auto fetch = [&](const float *row, float (&x)[NC]) {
#pragma unroll
        for (int n = 0; n < NC; ++n) x[n] = lane + 32 * n < K ? row[lane + 32 * n] : 0.0f;
    };
    float pc[NC == 1 ? 32 : 1];  // this lane's column of P (row, backward)
    // runs a and piece c's own vector through the piece, writing a's rows, at
    // least `least` of them: 1 they met, 0 the piece ended, -1 out of range
    int rows = 0;
    auto run = [&](int c, int least) {
        const StrandDesc d = sp.desc[c];
        fetch((BACK ? sm.bs : sp.vs) + (size_t)c * KP, g);
        rows = 0;
        if (least == 0 && met()) return 1;
        if (NC == 1) {
#pragma unroll
            for (int j = 0; j < 32; ++j) pc[NC == 1 ? j : 0] = j < K && lane < K ? (BACK ? P[lane * KPl + j] : P[j * KPl + lane]) : 0.0f;
        }
        // emissions relative to the whole offsets, as the strands have them; a
        // step that shrinks too far is made again with exact scaling
        const float offt = em[EM_OFF * KPl], offn = em[EM_OFF * KPl + 1];
        float ec[NC][7];  // in registers: the rows written below could alias them
#pragma unroll
        for (int n = 0; n < NC; ++n) {
            const int k = lane + 32 * n;
#pragma unroll
            for (int r = 0; r < 7; ++r) ec[n][r] = k < K ? em[r * KPl + k] : r >= EM_CTR ? -INFINITY : 0.0f;
            ec[n][EM_CTR] -= offt;
            ec[n][EM_CNO] -= offn;
        }
        float2 ob = make_float2(0.0f, 0.0f);  // 32 steps' observations, one a lane
        for (int &s = rows; s < least || (s & 3) || !met(); ++s) {
            if (s >= d.len) return 0;
            const int64_t i = BACK ? d.pstart + d.len - 1 - s : d.pstart + s;
            if ((s & 31) == 0) {
                const int64_t x = BACK ? i - lane : i + lane;
                if (BACK ? x >= d.pstart : x < d.pstart + d.len) ob = packed[x];
                if (BACK && x >= d.pstart) {
                    // alpha's rows of these steps, ahead of their turn
                    for (int k = 0; k < KP; k += 32) asm volatile("prefetch.global.L1 [%0];" ::"l"(sm.alpha + x * KP + k));
                }
            }
            const float ox = __shfl_sync(FULL, ob.x, s & 31), oy = __shfl_sync(FULL, ob.y, s & 31);
            const bool tr = !isnan(ox);
            float l[NC], f[NC], wa[NC], ka[NC], kg[NC], al[NC], ma, mg;
#pragma unroll
            for (int n = 0; n < NC; ++n) {
                const int k = lane + 32 * n;
                al[n] = BACK && k < K ? sm.alpha[i * KP + k] : 0.0f;  // early: used after the step
                const float dx = ox - ec[n][EM_MUX], dy = oy - ec[n][EM_MUY];
                l[n] = fmaf(fmaf(ec[n][EM_QA], dx, ec[n][EM_QB] * dy), dx, fmaf(ec[n][EM_QC] * dy, dy, ec[n][EM_CTR]));
                l[n] = tr ? l[n] : ec[n][EM_CNO];
                f[n] = ex2(l[n]);
                ka[n] = a[n];
                kg[n] = g[n];
            }
            for (int attempt = 0;; ++attempt) {
#pragma unroll
                for (int n = 0; n < NC; ++n) {
                    wa[n] = BACK ? ka[n] * f[n] : ka[n];
                    sag[warp][lane + 32 * n] = make_float2(wa[n], BACK ? kg[n] * f[n] : kg[n]);
                    a[n] = g[n] = 0.0f;
                }
                __syncwarp();
                if (NC == 1) {
                    f32x2 t[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
                    for (int j = 0; j < 32; j += 2) {
                        const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(&sag[warp][j]);
                        const float p0 = pc[NC == 1 ? j : 0], p1 = pc[NC == 1 ? j + 1 : 0];
                        t[j & 2] = fma2(x.x, pack2(p0, p0), t[j & 2]);
                        t[(j & 2) + 1] = fma2(x.y, pack2(p1, p1), t[(j & 2) + 1]);
                    }
                    unpack2(add2(add2(t[0], t[1]), add2(t[2], t[3])), a[0], g[0]);
                } else {
#pragma unroll 8
                    for (int j = 0; j < K; ++j) {
                        const float2 x = sag[warp][j];
#pragma unroll
                        for (int n = 0; n < NC; ++n) {
                            const float p = sP[NC == 1 ? 0 : j][NC == 1 ? 0 : lane + 32 * n];
                            a[n] = fmaf(x.x, p, a[n]);
                            g[n] = fmaf(x.y, p, g[n]);
                        }
                    }
                }
                __syncwarp();
                ma = mg = 0.0f;
#pragma unroll
                for (int n = 0; n < NC; ++n) {
                    if (!BACK) {
                        a[n] *= f[n];
                        g[n] *= f[n];
                    }
                    ma = fmaxf(ma, a[n]);
                    mg = fmaxf(mg, g[n]);
                }
                ma = all_max(ma);
                mg = all_max(mg);
                if (ma >= STRAND_SHRINK_KEEP && mg >= STRAND_SHRINK_KEEP && ma <= STRAND_GROW && mg <= STRAND_GROW) break;
                if (attempt) {
                    if (ma >= STRAND_SHRINK && mg >= STRAND_SHRINK && ma <= STRAND_GROW && mg <= STRAND_GROW) break;
                    return -1;
                }
                float mx = l[0];
#pragma unroll
                for (int n = 1; n < NC; ++n) mx = fmaxf(mx, l[n]);
                mx = all_max(mx);
                if (!(mx + (tr ? offt : offn) >= -(float)EXP_LIMIT)) return -1;
#pragma unroll
                for (int n = 0; n < NC; ++n) f[n] = ex2(l[n] - floorf(mx));
            }
            const float fa = pow2f(-float_exponent(ma)), fg = pow2f(-float_exponent(mg));
            float z = 0.0f;
#pragma unroll
            for (int n = 0; n < NC; ++n) {
                const int k = lane + 32 * n;
                a[n] *= fa;
                g[n] *= fg;
                wa[n] *= fa;
                if (BACK) {
                    z = fmaf(al[n], a[n], z);
                } else if (k < KP) {
                    sm.alpha[(i + 1) * KP + k] = a[n];
                }
            }
            if (BACK) {
                const float r = rcp(all_sum(z));
#pragma unroll
                for (int n = 0; n < NC; ++n) {
                    const int k = lane + 32 * n;
                    if (k < K) sm.gamma[i * K + k] = al[n] * a[n] * r;
                    if (k < KP && sm.u) sm.u[i * KP + k] = wa[n] * r;
                }
            }
        }
        return 1;
    };
    if (!chain) {
        const int c = blockIdx.x * 4 + warp;
        if (c >= sp.n) return;
        int how = 1;
        if (!(sp.desc[c].flags & (BACK ? SD_LAST : SD_FIRST))) {
            fetch(BACK ? sm.be + (size_t)(c + 1) * KP : sp.ve + (size_t)(c - 1) * KP, a);
            how = run(c, 0);
        }
        if (how == 0)
#pragma unroll
            for (int n = 0; n < NC; ++n)
                if (lane + 32 * n < K) sm.carry[(size_t)c * KP + lane + 32 * n] = a[n];
        if (lane == 0) {
            sm.unmet[c] = 2 * rows + (how == 0 ? 1 : 0);
            if (how < 0) send_to_chunks(sp, 0);
        }
        return;
    }
    // one warp per piece: those unmet whose neighbour behind had met (its end is
    // the true vector) go on, up to the next such piece. Where the true vector
    // meets the strand of a piece that is itself noted as unmet (against the
    // untrue end of the one behind), the next piece's own run did set out from the
    // truth; if that run ended unmet too, no warp of its own takes it on (its
    // neighbour behind is noted), so this one goes on from what it ended with.
    const int x0 = blockIdx.x * 4 + warp;  // in the recursion's direction
    if (x0 >= sp.n) return;
    auto piece = [&](int x) { return BACK ? sp.n - 1 - x : x; };
    auto starts = [&](int x) { return (sm.unmet[piece(x)] & 1) && (x == 0 || !(sm.unmet[piece(x - 1)] & 1)); };
    if (!starts(x0)) return;
    fetch(sm.carry + (size_t)piece(x0) * KP, a);
    int how = 0;
    int64_t spent = 0;
    for (int x = x0 + 1; x < sp.n && how == 0; ++x) {
        // (all the rows that the piece's own run wrote, from a vector that was not the true one)
        how = starts(x) || spent > sm.most ? -1 : run(piece(x), sm.unmet[piece(x)] >> 1);
        spent += sp.desc[piece(x)].len;
        if (how == 1 && x + 1 < sp.n && (sm.unmet[piece(x)] & 1) && (sm.unmet[piece(x + 1)] & 1)) {
            ++x;
            fetch(sm.carry + (size_t)piece(x) * KP, a);
            how = 0;
        }
    }
    if (how < 0 && lane == 0) send_to_chunks(sp, 0);
}

// ---- E-step statistics ----
constexpr int SX_THREADS = 256, SX_BLOCK = 64, SX_GROUP = 8, SX_FLUSH = 64;

// hi + lo += x, what the addition drops kept in lo (Knuth's two-sum)
__device__ __forceinline__ void add_kept(float &hi, float &lo, float x) {
    const float s = __fadd_rn(hi, x), b = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(x, b)));
    hi = s;
}

// One CTA per range of steps: sum of alpha_i (x) u_i times P, and the gamma
// moments. Sums as in 64 bits: every term of N rounded to
// FP32, groups of SX_GROUP products in FP32 (a quiet stretch adds nearly the same
// term again and again, whose rounding would repeat), what their additions drop
// kept beside them for up to SX_FLUSH blocks of 64 steps, FP64 across those. FP64
// additions and conversions run at two a cycle and SM here: eleven sums a thread
// and block were most of this kernel (EM step, K=12,
// T=200,003: 216 us in all with one addition each, 252 with two, 209 with none). The CTAs'
// sums are added in order by a later kernel.
template <int KP>
__global__ void __launch_bounds__(SX_THREADS)
stats_kernel(int K, int64_t steps, int64_t per, ConstLayout lay, const float *__restrict__ cb,
             const float2 *__restrict__ head, const float2 *__restrict__ packed, StrandPtrs sp, SmoothPtrs sm,
             double *__restrict__ part, double *__restrict__ g0) {
    constexpr int CQ = KP / 4;                                        // column quads
    constexpr int NR = KP * CQ <= SX_THREADS ? 1 : KP * CQ / SX_THREADS;  // rows of N per thread
    constexpr int SL = KP * CQ <= SX_THREADS ? SX_THREADS / (KP * CQ) : 1;  // step slices of N
    constexpr int GROUP = SX_BLOCK / SL < SX_GROUP ? SX_BLOCK / SL : SX_GROUP;  // products of one slice in FP32
    constexpr int MS = SX_THREADS / KP;                               // step slices of the moments
    __shared__ __align__(16) float sA[SX_BLOCK][KP], sU[SX_BLOCK][KP];
    __shared__ float2 sO[SX_BLOCK];
    __shared__ double red[SX_THREADS][4];
    if (sp.route[0] != ROUTE_STRANDS) return;
    const int tid = threadIdx.x;
    const int64_t i0 = (int64_t)blockIdx.x * per, i1 = min(i0 + per, steps);
    double *out = part + (size_t)blockIdx.x * (K * K + 7 * K);

    const int cq = tid % CQ, row = (tid / CQ) % (KP / NR), sl = tid / (CQ * (KP / NR));
    double acc[NR][4] = {};
    const int mk = tid % KP, msl = tid / KP;
    double mom[7] = {};
    // gamma rows: i + 1 for each of this CTA's steps i, and row 0 for the first CTA
    // (products with what their rounding drops: a sum of squares near the origin
    // by a mean far from it would be lost in squares about the mean)
    auto add = [&](float (&s)[7], float (&l)[7], float g, float2 o) {
        add_kept(s[0], l[0], g);
        if (!isnan(o.x)) {
            const float gx = __fmul_rn(g, o.x), gy = __fmul_rn(g, o.y);
            const float ex = fmaf(g, o.x, -gx), ey = fmaf(g, o.y, -gy);
            auto square = [&](int c, float h, float e, float z) {
                const float q = __fmul_rn(h, z);
                add_kept(s[c], l[c], q);
                l[c] += fmaf(e, z, fmaf(h, z, -q));
            };
            add_kept(s[1], l[1], g);
            add_kept(s[2], l[2], gx);
            l[2] += ex;
            add_kept(s[3], l[3], gy);
            l[3] += ey;
            square(4, gx, ex, o.x);
            square(5, gx, ex, o.y);
            square(6, gy, ey, o.y);
        }
    };
    float hi[NR][4] = {}, lo[NR][4] = {}, m[7] = {}, ml[7] = {};
    auto flush = [&]() {
#pragma unroll
        for (int r = 0; r < NR; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                acc[r][c] += (double)hi[r][c] + (double)lo[r][c];
                hi[r][c] = lo[r][c] = 0.0f;
            }
#pragma unroll
        for (int c = 0; c < 7; ++c) {
            mom[c] += (double)m[c] + (double)ml[c];
            m[c] = ml[c] = 0.0f;
        }
    };
    int done = 0;
    for (int64_t b = i0; b < i1; b += SX_BLOCK) {
        const int n = (int)min((int64_t)SX_BLOCK, i1 - b);
        __syncthreads();
        for (int x = tid; x < SX_BLOCK * CQ; x += SX_THREADS) {
            const int s = x / CQ;
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
            reinterpret_cast<float4 *>(&sA[0][0])[x] = s < n ? reinterpret_cast<const float4 *>(sm.alpha + b * KP)[x] : zero;
            reinterpret_cast<float4 *>(&sU[0][0])[x] = s < n ? reinterpret_cast<const float4 *>(sm.u + b * KP)[x] : zero;
        }
        for (int x = tid; x < n; x += SX_THREADS) sO[x] = packed[b + x];
        __syncthreads();
        if (sl < SL) {
            for (int s0 = sl; s0 < SX_BLOCK; s0 += SL * GROUP) {
                float t[NR][4] = {};
#pragma unroll
                for (int g = 0; g < GROUP; ++g) {
                    const int s = s0 + g * SL;
                    const float4 u = *reinterpret_cast<const float4 *>(&sU[s][4 * cq]);
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        const float al = sA[s][row + r * (KP / NR)];
                        t[r][0] = fmaf(al, u.x, t[r][0]);
                        t[r][1] = fmaf(al, u.y, t[r][1]);
                        t[r][2] = fmaf(al, u.z, t[r][2]);
                        t[r][3] = fmaf(al, u.w, t[r][3]);
                    }
                }
#pragma unroll
                for (int r = 0; r < NR; ++r)
#pragma unroll
                    for (int c = 0; c < 4; ++c) add_kept(hi[r][c], lo[r][c], t[r][c]);
            }
        }
        if (msl < MS && mk < K)
            for (int s = msl; s < n; s += MS) add(m, ml, sm.gamma[(b + s + 1) * K + mk], sO[s]);
        if (++done % SX_FLUSH == 0) flush();
    }
    if (blockIdx.x == 0 && msl == 0 && mk < K) {
        const float g = sm.gamma[mk];
        add(m, ml, g, head[0]);
        g0[mk] = g;
    }
    flush();
    // the slices together, in order
    const float *P = cb + lay.off_p32;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 4; ++c) red[tid][c] = acc[r][c];
        __syncthreads();
        if (sl == 0) {
            const int i = row + r * (KP / NR);
            for (int c = 0; c < 4; ++c) {
                const int j = 4 * cq + c;
                double v = 0.0;
                for (int x = 0; x < SL; ++x) v += red[tid + x * CQ * (KP / NR)][c];
                if (i < K && j < K) out[i * K + j] = v * (double)P[i * lay.KP + j];
            }
        }
    }
    double s[7];
    for (int c = 0; c < 7; ++c) {
        __syncthreads();
        red[tid][0] = mom[c];
        __syncthreads();
        s[c] = 0.0;
        if (msl == 0)
            for (int x = 0; x < MS; ++x) s[c] += red[tid + x * KP][0];
    }
    if (msl == 0 && mk < K) {
        for (int c = 0; c < 7; ++c) out[K * K + c * K + mk] = s[c];
    }
}

// stats = [N, G0, Gs, Gr, Sx, Sy, Sxx, Sxy, Syy]: a warp per entry adds the
// CTAs' sums in a fixed order
__global__ void stats_sum_kernel(int K, int n_parts, const double *__restrict__ part, const double *__restrict__ g0,
                                 const int *__restrict__ route, double *stats) {
    if (route[0] != ROUTE_STRANDS) return;
    const int n = K * K + 7 * K;
    const int lane = threadIdx.x & 31;
    for (int e = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32; e < n; e += gridDim.x * (blockDim.x / 32)) {
        double acc = 0.0;
        for (int c = lane; c < n_parts; c += 32) acc += part[(size_t)c * n + e];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
        if (lane == 0) stats[e < K * K ? e : e + K] = acc;
    }
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < K; k += gridDim.x * blockDim.x) stats[K * K + k] = g0[k];
}

template <int KP, int H>
cudaError_t back_t(int K, int64_t steps, const ConstLayout &lay, const float *cb, const float2 *packed,
                   const StrandPtrs &sp, const SmoothPtrs &sm, cudaStream_t st) {
    using C = SimtTile<KP, H>;
    const int warps = (sp.n + C::PER_WARP - 1) / C::PER_WARP;
    strand_back_kernel<C><<<(warps + STRAND_WPC - 1) / STRAND_WPC, 32 * STRAND_WPC, 0, st>>>(K, steps, sm.warm, lay, cb,
                                                                                           packed, sp, sm);
    return cudaGetLastError();
}

template <int KP>
cudaError_t stats_t(int K, int64_t steps, const ConstLayout &lay, const float *cb, const float2 *head,
                    const float2 *packed, const StrandPtrs &sp, const SmoothPtrs &sm, cudaStream_t st) {
    const int64_t blocks = (steps + SX_BLOCK - 1) / SX_BLOCK;
    const int64_t per = (blocks + SMOOTH_PARTS - 1) / SMOOTH_PARTS * SX_BLOCK;
    const int ctas = (int)((steps + per - 1) / per);
    stats_kernel<KP><<<ctas, SX_THREADS, 0, st>>>(K, steps, per, lay, cb, head, packed, sp, sm, sm.part, sm.g0);
    stats_sum_kernel<<<(K * K + 7 * K + 7) / 8, 256, 0, st>>>(K, ctas, sm.part, sm.g0, sp.route, sm.stats);
    return cudaGetLastError();
}

template <bool BACK>
cudaError_t join_t(int K, int KP, const ConstLayout &lay, const float *cb, const float2 *packed, const StrandPtrs &sp,
                   const SmoothPtrs &sm, cudaStream_t st) {
    auto kern = KP <= 32 ? rows_join_kernel<1, BACK> : rows_join_kernel<2, BACK>;
    kern<<<(sp.n + 3) / 4, 128, 0, st>>>(K, KP, false, lay, cb, packed, sp, sm);
    kern<<<(sp.n + 3) / 4, 128, 0, st>>>(K, KP, true, lay, cb, packed, sp, sm);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_smooth(int K, int KP, int64_t steps, const ConstLayout &lay, const float *cblock, const float2 *head,
                          const float2 *packed, const StrandPtrs &sp, const SmoothPtrs &sm, cudaStream_t st) {
    cudaError_t e = join_t<false>(K, KP, lay, cblock, packed, sp, sm, st);
    if (e != cudaSuccess) return e;
#define HMM_SMOOTH_CASE(KPV, HV)                                                   \
    case KPV:                                                                      \
        e = strand_rows(KPV, sp.n) == 2 ? back_t<KPV, HV>(K, steps, lay, cblock, packed, sp, sm, st) \
                                        : back_t<KPV, HV == 2 && KPV < 64 ? 1 : HV>(K, steps, lay, cblock, packed, sp, sm, st); \
        if (e == cudaSuccess) e = join_t<true>(K, KP, lay, cblock, packed, sp, sm, st); \
        if (e == cudaSuccess && sm.stats) e = stats_t<KPV>(K, steps, lay, cblock, head, packed, sp, sm, st); \
        return e;
    switch (KP) {
        HMM_SMOOTH_CASE(4, 1)
        HMM_SMOOTH_CASE(8, 1)
        HMM_SMOOTH_CASE(16, 2)
        HMM_SMOOTH_CASE(32, 2)
        HMM_SMOOTH_CASE(64, 2)
        default: return cudaErrorInvalidValue;
    }
#undef HMM_SMOOTH_CASE
}

}  // namespace hmm
