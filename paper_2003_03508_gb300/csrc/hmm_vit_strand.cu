// The most probable path by strands: one max-plus vector per piece of the
// sequence in place of K (hmm_viterbi.cu's chunk products, kept for chains whose
// paths do not coalesce). Best paths into all states of a step share their
// beginning a few dozen steps back, so two vectors that start apart become
// equal up to a constant, which is checked where pieces meet:
//   strands   every piece's vector from a warm-up, and its back-pointers;
//   rejoin    a piece whose vector had not met the one before it at its start
//             runs again from that one until they meet, over its own
//             back-pointers (and on through the next pieces where it must);
//   maps      every piece's back-pointers as one map, leaving to entering state;
//   compose   the maps in order: the state at every piece's end;
//   trace     every piece back from there, and the path's score in FP64.
// A row of back-pointers is one byte a lane, so a step of a trace is a shuffle.
//
// The recursion's scores are FP32 relative to the largest, renormalised every
// four steps; the comparison and the order of the sums are those of
// hmm_viterbi.cu (v_i + log2 P_ij, the smallest i on ties, then the emission).
//
// What bounds it: one step of a lone warp (128 candidates a thread, four
// instructions each), 0.3 us, times warm-up and piece.
#include "hmm_strand_simt.cuh"

namespace hmm {

namespace {

constexpr unsigned FULL = 0xffffffffu;
// Vectors whose paths have coalesced differ by rounding alone, which renormalising
// at the same steps makes alike: 0 nearly always, 2e-6 at most in a float32 replay
// (K = 4 to 64, scores to -3000). Those that have not may differ by any amount,
// and a difference passed over is a path given up for a worse one.
constexpr float VIT_TOL = 7.62939453125e-6f;  // 2^-17

// log2 P in FP32 for the recursion, and what the path's score takes in FP64:
// log P and each state's emission constants
__global__ void vit_table_kernel(int K, int KP, const float *__restrict__ P, const float *__restrict__ p,
                                 const float *__restrict__ mu, const float *__restrict__ cov, VitPtrs vp) {
    const int n = KP * KP;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int r = i / KP, c = i % KP;
        const float v = r < K && c < K ? P[r * K + c] : 0.0f;
        vp.lp[i] = v > 0.0f ? log2f(v) : -INFINITY;
        vp.lp64[i] = log((double)v);
    }
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < K; k += gridDim.x * blockDim.x) {
        const double sxx = cov[3 * k], sxy = cov[3 * k + 1], syy = cov[3 * k + 2], det = sxx * syy - sxy * sxy;
        double *e = vp.em64 + 8 * k;
        e[0] = mu[2 * k];
        e[1] = mu[2 * k + 1];
        e[2] = -0.5 * syy / det;
        e[3] = sxy / det;
        e[4] = -0.5 * sxx / det;
        e[5] = log((double)p[k]) - 1.8378770664093454836 - 0.5 * log(det);
        e[6] = log(1.0 - (double)p[k]);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *vp.chunks = 0;
}

// emissions relative to the whole offsets, in the form that hmm_viterbi.cu has
struct VitEmis {
    float mx, my, qa, qb, qc, ctr, cno;
    __device__ __forceinline__ void load(const float *__restrict__ em, int KPl, int K, int k, float offt, float offn) {
        const bool in = k < K;
        mx = in ? em[EM_MUX * KPl + k] : 0.0f;
        my = in ? em[EM_MUY * KPl + k] : 0.0f;
        qa = in ? em[EM_QA * KPl + k] : 0.0f;
        qb = in ? em[EM_QB * KPl + k] : 0.0f;
        qc = in ? em[EM_QC * KPl + k] : 0.0f;
        ctr = in ? em[EM_CTR * KPl + k] - offt : -INFINITY;
        cno = in ? em[EM_CNO * KPl + k] - offn : -INFINITY;
    }
    __device__ __forceinline__ float eval(float x, float y) const {
        const float dx = x - mx, dy = y - my;
        float acc = fmaf(qc * dy, dy, ctr);
        acc = fmaf(qb * dx, dy, acc);
        acc = fmaf(qa * dx, dx, acc);
        return isnan(x) ? cno : acc;
    }
};

template <class C>
__global__ void __launch_bounds__(32 * STRAND_WPC, C::MIN_CTAS)
vit_strand_kernel(int K, int init_mode, ConstLayout lay, const float *__restrict__ cb, const float *__restrict__ pi,
                  const float2 *__restrict__ head, const float2 *__restrict__ packed, StrandPtrs sp, VitPtrs vp) {
    constexpr int KP = C::KP, NS = C::NS, NI = C::NI;
    __shared__ __align__(16) float sv[STRAND_WPC][2 * C::PER_WARP * C::STRIDE];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wid = blockIdx.x * STRAND_WPC + warp;
    if (wid * C::PER_WARP >= sp.n) return;
    const float *em = cb + lay.off_emis;
    const int KPl = lay.KP;
    const int g = lane % C::G, slot = lane / C::G, cg = g % C::CG, h = g / C::CG;
    const int own = 4 * cg + NS * h;
    float *const row = sv[warp] + slot * C::STRIDE;
    float lp[4][NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const float4 t = *reinterpret_cast<const float4 *>(vp.lp + (h * NI + i) * KP + 4 * cg);
        lp[0][i] = t.x; lp[1][i] = t.y; lp[2][i] = t.z; lp[3][i] = t.w;
    }
    const float offt = em[EM_OFF * KPl], offn = em[EM_OFF * KPl + 1];
    VitEmis ec[NS];
#pragma unroll
    for (int u = 0; u < NS; ++u) ec[u].load(em, KPl, K, own + u, offt, offn);

    const int k = wid * C::PER_WARP + slot;
    const int sid = k < sp.n ? k : -1;
    const StrandDesc d = sp.desc[sid < 0 ? 0 : sid];
    const int total = sid < 0 ? 0 : d.warm + d.len;
    const float2 *obs = packed + d.pstart - d.warm;
    uint8_t *bp = vp.bp + ((size_t)d.pstart - d.warm) * KP + own;  // row of the first step
    int steps = total;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) steps = max(steps, __shfl_xor_sync(FULL, steps, o));
    auto top = [&](const float (&x)[NS]) {
        float m = fmaxf(fmaxf(x[0], x[1]), fmaxf(x[NS - 2], x[NS - 1]));
#pragma unroll
        for (int o = 1; o < C::G; o <<= 1) m = fmaxf(m, __shfl_xor_sync(FULL, m, o));
        return m;
    };

    float v[NS];
    bool bad = false;
    {
        const float2 o = head[0];
        const bool at_head = (d.flags & SD_HEAD) != 0;
#pragma unroll
        for (int u = 0; u < NS; ++u) {
            const int s = own + u;
            double w = 0.0;
            if (s < K) {
                if (init_mode == HMM_INIT_TRANSITION_FIRST)
                    for (int i = 0; i < K; ++i) w += (double)pi[i] * (double)cb[lay.off_p32 + i * KPl + s];
                else
                    w = pi[s];
            }
            v[u] = !at_head ? (s < K ? 0.0f : -INFINITY) : w > 0.0 ? (float)log2(w) + ec[u].eval(o.x, o.y) : -INFINITY;
        }
        const float m = top(v);
        bad = !(m > -INFINITY);
#pragma unroll
        for (int u = 0; u < NS; ++u) v[u] = bad ? 0.0f : v[u] - m;
    }
    auto store = [&](float *r) {
        if (NS == 4) *reinterpret_cast<float4 *>(r + own) = make_float4(v[0], v[1], v[NS - 2], v[NS - 1]);
        else *reinterpret_cast<float2 *>(r + own) = make_float2(v[0], v[1]);
    };
    float2 next = total > 0 ? obs[0] : make_float2(0.f, 0.f);
    int buf = 0;
    for (int t = 0; t < steps; ++t) {
        const float2 o = next;
        if (t + 1 < total) next = obs[t + 1];
        float l[NS];
#pragma unroll
        for (int u = 0; u < NS; ++u) l[u] = ec[u].eval(o.x, o.y);
        float *const b = row + buf * C::PER_WARP * C::STRIDE;
        if (KP > 4) {
            if (NS == 4) *reinterpret_cast<float4 *>(b + C::at(own)) = make_float4(v[0], v[1], v[NS - 2], v[NS - 1]);
            else *reinterpret_cast<float2 *>(b + C::at(own)) = make_float2(v[0], v[1]);
            __syncwarp();
        }
        float best[4];
        int arg[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            best[c] = -INFINITY;
            arg[c] = h * NI;
        }
#pragma unroll
        for (int i4 = 0; i4 < NI / 4; ++i4) {
            float x[4];
            if (KP == 4) {
                x[0] = v[0]; x[1] = v[1]; x[2] = v[NS - 2]; x[3] = v[NS - 1];
            } else {
                const float4 z = *reinterpret_cast<const float4 *>(b + C::at(h * NI) + 4 * i4);
                x[0] = z.x; x[1] = z.y; x[2] = z.z; x[3] = z.w;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float w = x[u] + lp[c][4 * i4 + u];
                    const bool gt = w > best[c];
                    best[c] = gt ? w : best[c];
                    arg[c] = gt ? h * NI + 4 * i4 + u : arg[c];
                }
        }
        buf ^= 1;
        float y[NS];
        unsigned pack = 0;
        if (C::H == 1) {
#pragma unroll
            for (int u = 0; u < NS; ++u) y[u] = best[u];
            pack = (unsigned)arg[0] | (unsigned)arg[1] << 8 | (unsigned)arg[2] << 16 | (unsigned)arg[3] << 24;
        } else {
            // the other half's rows: the first half wins ties (smaller indices)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const float ob = __shfl_xor_sync(FULL, h ? best[u] : best[2 + u], C::CG);
                const int oa = __shfl_xor_sync(FULL, h ? arg[u] : arg[2 + u], C::CG);
                const float mb = h ? best[2 + u] : best[u];
                const int ma = h ? arg[2 + u] : arg[u];
                const bool take = h ? ob >= mb : ob > mb;
                y[u] = take ? ob : mb;
                pack |= (unsigned)(take ? oa : ma) << (8 * u);
            }
        }
        const bool act = t < total;
        if (act) {
#pragma unroll
            for (int u = 0; u < NS; ++u) v[u] = y[u] + l[u];
            if (t >= d.warm) {
                if (NS == 4) *reinterpret_cast<unsigned *>(bp + (size_t)t * KP) = pack;
                else *reinterpret_cast<uint16_t *>(bp + (size_t)t * KP) = (uint16_t)pack;
            }
        }
        if ((t & 3) == 3 || __any_sync(FULL, t + 1 == total)) {  // the warp agrees
            const float m = top(v);
            bad = bad || !(m > -INFINITY);
#pragma unroll
            for (int u = 0; u < NS; ++u) v[u] = m > -INFINITY ? v[u] - m : v[u];
        }
        if (t + 1 == d.warm && act) {
            store(vp.vs + (size_t)sid * KP);
        }
    }
    if (sid < 0) return;
    store(vp.ve + (size_t)sid * KP);
    if (g == 0 && bad) *vp.chunks = 1;
}

// Pieces whose vector had not met the one before at their start. The first
// launch runs each against its own strand; one that ends first is noted, and a
// second launch (`chain`) carries those on, as rows_join_kernel does.
template <int NC>
__global__ void __launch_bounds__(128)
vit_rejoin_kernel(int K, int KP, bool chain, ConstLayout lay, const float *__restrict__ cb,
                  const float2 *__restrict__ packed, StrandPtrs sp, VitPtrs vp) {
    __shared__ float sag[4][2][32 * NC];
    __shared__ float slp[32 * NC][32 * NC];  // log2 P
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c0 = blockIdx.x * 4 + warp;
    for (int x = threadIdx.x; x < 32 * NC * 32 * NC; x += 128) {
        const int i = x / (32 * NC), k = x % (32 * NC);
        slp[i][k] = i < K && k < K ? vp.lp[i * KP + k] : -INFINITY;
    }
    __syncthreads();
    if (c0 >= sp.n || __shfl_sync(FULL, *vp.chunks, 0)) return;
    const float *em = cb + lay.off_emis;
    const float offt = em[EM_OFF * lay.KP], offn = em[EM_OFF * lay.KP + 1];
    float a[NC], g[NC];
    int rows = 0;
    auto all_max = [&](float v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(FULL, v, o));
        return v;
    };
    auto met = [&]() {
        float lo = INFINITY, hi = -INFINITY;
#pragma unroll
        for (int n = 0; n < NC; ++n)
            if (a[n] > -INFINITY || g[n] > -INFINITY) {
                const float r = a[n] - g[n];  // +-inf where only one is possible
                lo = fminf(lo, r);
                hi = fmaxf(hi, r);
            }
        hi = all_max(hi);
        lo = -all_max(-lo);
        return hi >= lo && hi - lo <= VIT_TOL;  // false for infinities, and where no entry was compared
    };
    auto fetch = [&](const float *r, float (&x)[NC]) {
#pragma unroll
        for (int n = 0; n < NC; ++n) x[n] = lane + 32 * n < K ? r[lane + 32 * n] : -INFINITY;
    };
    // 1 they met, 0 the piece ended, -1 no path left
    auto run = [&](int c, int least) {
        const StrandDesc d = sp.desc[c];
        fetch(vp.vs + (size_t)c * KP, g);
        rows = 0;
        if (least == 0 && met()) return 1;
        VitEmis ec[NC];
#pragma unroll
        for (int n = 0; n < NC; ++n) ec[n].load(em, lay.KP, K, lane + 32 * n, offt, offn);
        for (int &s = rows; s < least || (s & 3) || !met(); ++s) {
            if (s >= d.len) return 0;
            const int64_t i = d.pstart + s;
            const float2 o = packed[i];
#pragma unroll
            for (int n = 0; n < NC; ++n) {
                sag[warp][0][lane + 32 * n] = a[n];
                sag[warp][1][lane + 32 * n] = g[n];
            }
            __syncwarp();
            int arg[NC] = {};
#pragma unroll
            for (int n = 0; n < NC; ++n) a[n] = g[n] = -INFINITY;
#pragma unroll 8
            for (int j = 0; j < K; ++j) {
                const float xa = sag[warp][0][j], xg = sag[warp][1][j];
#pragma unroll
                for (int n = 0; n < NC; ++n) {
                    const float p = slp[j][lane + 32 * n];
                    const float w = xa + p;
                    if (w > a[n]) {
                        a[n] = w;
                        arg[n] = j;
                    }
                    g[n] = fmaxf(g[n], xg + p);
                }
            }
            __syncwarp();
            float ma = -INFINITY, mg = -INFINITY;
#pragma unroll
            for (int n = 0; n < NC; ++n) {
                const int k = lane + 32 * n;
                if (k < KP) vp.bp[i * KP + k] = (uint8_t)arg[n];
                const float l = ec[n].eval(o.x, o.y);
                a[n] += l;
                g[n] += l;
                ma = fmaxf(ma, a[n]);
                mg = fmaxf(mg, g[n]);
            }
            ma = all_max(ma);
            mg = all_max(mg);
            if (!(ma > -INFINITY && mg > -INFINITY)) return -1;
#pragma unroll
            for (int n = 0; n < NC; ++n) {
                a[n] -= ma;
                g[n] -= mg;
            }
        }
        return 1;
    };
    if (!chain) {
        int how = 1;
        if (!(sp.desc[c0].flags & SD_FIRST)) {
            fetch(vp.ve + (size_t)(c0 - 1) * KP, a);
            how = run(c0, 0);
        }
        if (how == 0) {
#pragma unroll
            for (int n = 0; n < NC; ++n)
                if (lane + 32 * n < K) vp.carry[(size_t)c0 * KP + lane + 32 * n] = a[n];
        }
        if (lane == 0) {
            vp.unmet[c0] = 2 * rows + (how == 0 ? 1 : 0);
            if (how < 0) *vp.chunks = 1;
        }
        return;
    }
    auto starts = [&](int x) { return (vp.unmet[x] & 1) && !(vp.unmet[x - 1] & 1); };
    if (c0 == 0 || !starts(c0)) return;
    fetch(vp.carry + (size_t)c0 * KP, a);
    int how = 0;
    int64_t spent = 0;
    for (int x = c0 + 1; x < sp.n && how == 0; ++x) {
        how = starts(x) || spent > vp.most ? -1 : run(x, vp.unmet[x] >> 1);
        spent += sp.desc[x].len;
        if (how == 1 && x + 1 < sp.n && (vp.unmet[x] & 1) && (vp.unmet[x + 1] & 1)) {
            ++x;
            fetch(vp.carry + (size_t)x * KP, a);
            how = 0;
        }
    }
    if (how < 0 && lane == 0) *vp.chunks = 1;
    if (how == 0) {  // to the sequence's end: this is its last vector
#pragma unroll
        for (int n = 0; n < NC; ++n)
            if (lane + 32 * n < K) vp.ve[(size_t)(sp.n - 1) * KP + lane + 32 * n] = a[n];
    }
}

// every piece's map: leaving state -> the state before its first step
// (NC lanes' worth of states: a row is one byte a lane, or two)
template <int NC>
__global__ void __launch_bounds__(128)
vit_map_kernel(int K, int KP, StrandPtrs sp, VitPtrs vp) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c = blockIdx.x * 4 + warp;
    if (c >= sp.n || __shfl_sync(FULL, *vp.chunks, 0)) return;
    const StrandDesc d = sp.desc[c];
    const uint8_t *bp = vp.bp + (size_t)d.pstart * KP;
    int s0 = lane, s1 = lane + 32;
#pragma unroll 8
    for (int t = d.len - 1; t >= 0; --t) {
        const int r0 = lane < KP ? bp[(size_t)t * KP + lane] : 0;
        const int a0 = __shfl_sync(FULL, r0, s0 & 31);
        if (NC == 1) {
            s0 = a0;
        } else {
            const int r1 = lane + 32 < KP ? bp[(size_t)t * KP + lane + 32] : 0;
            const int a1 = __shfl_sync(FULL, r1, s0 & 31);
            const int b0 = __shfl_sync(FULL, r0, s1 & 31), b1 = __shfl_sync(FULL, r1, s1 & 31);
            s0 = s0 < 32 ? a0 : a1;
            s1 = s1 < 32 ? b0 : b1;
        }
    }
    if (lane < KP) vp.map[(size_t)c * KP + lane] = (uint8_t)s0;
    if (NC > 1 && lane + 32 < KP) vp.map[(size_t)c * KP + lane + 32] = (uint8_t)s1;
}

// One CTA: each warp composes the maps of a run of pieces, the runs are walked
// from the best last state, and each warp walks its run again from its own end.
constexpr int VC = 1024;
__global__ void __launch_bounds__(VC)
vit_compose_kernel(int K, int KP, StrandPtrs sp, VitPtrs vp) {
    __shared__ uint8_t run_map[32][64];
    __shared__ int run_end[32];
    if (*vp.chunks) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n = sp.n;
    const int per = (n + 31) / 32, lo = min(n, warp * per), hi = min(n, lo + per);
    auto walk = [&](int c, int s) {
        const int r0 = lane < KP ? vp.map[(size_t)c * KP + lane] : 0, r1 = lane + 32 < KP ? vp.map[(size_t)c * KP + lane + 32] : 0;
        const int a0 = __shfl_sync(FULL, r0, s & 31), a1 = __shfl_sync(FULL, r1, s & 31);
        return s < 32 ? a0 : a1;
    };
    int s0 = lane, s1 = lane + 32;
#pragma unroll 4
    for (int c = hi - 1; c >= lo; --c) {
        s0 = walk(c, s0);
        s1 = walk(c, s1);
    }
    run_map[warp][lane] = (uint8_t)s0;
    run_map[warp][lane + 32] = (uint8_t)s1;
    __syncthreads();
    if (threadIdx.x == 0) {
        // the best last state, the smallest on ties
        const float *v = vp.ve + (size_t)(n - 1) * KP;
        int s = 0;
        for (int k = 1; k < K; ++k)
            if (v[k] > v[s]) s = k;
        for (int w = 31; w >= 0; --w) {
            run_end[w] = s;
            s = run_map[w][s];
        }
    }
    __syncthreads();
    int s = run_end[warp];
#pragma unroll 4
    for (int c = hi - 1; c >= lo; --c) {
        if (lane == 0) vp.bstate[c] = s;
        s = walk(c, s);
    }
}

// A piece's states from its last one, and their part of the path's score: the
// transitions into and the emissions of its observations (and of the first).
template <int NC>
__global__ void __launch_bounds__(128)
vit_trace_kernel(int K, int KP, int init_mode, const float *__restrict__ pi, const float *__restrict__ P,
                 const float2 *__restrict__ head, const float2 *__restrict__ packed, StrandPtrs sp, VitPtrs vp,
                 int32_t *__restrict__ path) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c = blockIdx.x * 4 + warp;
    if (c >= sp.n || __shfl_sync(FULL, *vp.chunks, 0)) return;
    const StrandDesc d = sp.desc[c];
    const uint8_t *bp = vp.bp + (size_t)d.pstart * KP;
    int32_t *out = path + d.pstart + 1;  // observation of the piece's first step
    auto emission = [&](int k, float2 o) {
        const double *e = vp.em64 + 8 * k;
        if (isnan(o.x)) return e[6];
        const double dx = (double)o.x - e[0], dy = (double)o.y - e[1];
        return e[5] + e[2] * dx * dx + e[3] * dx * dy + e[4] * dy * dy;
    };
    int s = vp.bstate[c];
    double part = 0.0;
    for (int t1 = d.len; t1 > 0; t1 -= 32) {
        const int t0 = max(0, t1 - 32), n = t1 - t0;
        int to = 0, from = 0;
#pragma unroll 8
        for (int t = t1 - 1; t >= t0; --t) {
            const int r0 = lane < KP ? bp[(size_t)t * KP + lane] : 0;
            int before = __shfl_sync(FULL, r0, s & 31);
            if (NC > 1) {
                const int r1 = lane + 32 < KP ? bp[(size_t)t * KP + lane + 32] : 0;
                const int a1 = __shfl_sync(FULL, r1, s & 31);
                before = s < 32 ? before : a1;
            }
            if (lane == t - t0) {
                to = s;
                from = before;
            }
            s = before;
        }
        if (lane < n) {
            out[t0 + lane] = to;
            part += vp.lp64[from * KP + to] + emission(to, packed[d.pstart + t0 + lane]);
        }
    }
    if (c == 0 && lane == 0) {
        path[0] = s;
        double w = 0.0;
        if (init_mode == HMM_INIT_TRANSITION_FIRST)
            for (int i = 0; i < K; ++i) w += (double)pi[i] * (double)P[i * K + s];
        else
            w = pi[s];
        part += log(w) + emission(s, head[0]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(FULL, part, o);
    if (lane == 0) vp.part[c] = part;
}

__global__ void __launch_bounds__(256) vit_score_kernel(int n, VitPtrs vp, double *score) {
    __shared__ double red[256];
    if (*vp.chunks) return;
    double s = 0.0;
    for (int c = threadIdx.x; c < n; c += 256) s += vp.part[c];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) *score = red[0];
}

template <int KP, int H>
cudaError_t vit_t(int K, int init_mode, const ConstLayout &lay, const float *cb, const float *pi, const float2 *head,
                  const float2 *packed, const StrandPtrs &sp, const VitPtrs &vp, cudaStream_t st) {
    using C = SimtTile<KP, H>;
    const int warps = (sp.n + C::PER_WARP - 1) / C::PER_WARP;
    vit_strand_kernel<C><<<(warps + STRAND_WPC - 1) / STRAND_WPC, 32 * STRAND_WPC, 0, st>>>(K, init_mode, lay, cb, pi,
                                                                                          head, packed, sp, vp);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_vit_strands(int K, int KP, int init_mode, const ConstLayout &lay, const float *cb, const float *pi,
                               const float *P, const float *p, const float *mu, const float *cov, const float2 *head,
                               const float2 *packed, const StrandPtrs &sp, const VitPtrs &vp, int32_t *path,
                               double *score, cudaStream_t st) {
    vit_table_kernel<<<(KP * KP + 127) / 128, 128, 0, st>>>(K, KP, P, p, mu, cov, vp);
    cudaError_t e = cudaSuccess;
    switch (KP) {
        case 4: e = vit_t<4, 1>(K, init_mode, lay, cb, pi, head, packed, sp, vp, st); break;
        case 8: e = vit_t<8, 1>(K, init_mode, lay, cb, pi, head, packed, sp, vp, st); break;
        case 16:
            e = strand_rows(KP, sp.n) == 2 ? vit_t<16, 2>(K, init_mode, lay, cb, pi, head, packed, sp, vp, st)
                                           : vit_t<16, 1>(K, init_mode, lay, cb, pi, head, packed, sp, vp, st);
            break;
        case 32:
            e = strand_rows(KP, sp.n) == 2 ? vit_t<32, 2>(K, init_mode, lay, cb, pi, head, packed, sp, vp, st)
                                           : vit_t<32, 1>(K, init_mode, lay, cb, pi, head, packed, sp, vp, st);
            break;
        case 64: e = vit_t<64, 2>(K, init_mode, lay, cb, pi, head, packed, sp, vp, st); break;
        default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    const int ctas = (sp.n + 3) / 4;
    auto rejoin = KP <= 32 ? vit_rejoin_kernel<1> : vit_rejoin_kernel<2>;
    rejoin<<<ctas, 128, 0, st>>>(K, KP, false, lay, cb, packed, sp, vp);
    rejoin<<<ctas, 128, 0, st>>>(K, KP, true, lay, cb, packed, sp, vp);
    if (KP <= 32) vit_map_kernel<1><<<ctas, 128, 0, st>>>(K, KP, sp, vp);
    else vit_map_kernel<2><<<ctas, 128, 0, st>>>(K, KP, sp, vp);
    vit_compose_kernel<<<1, VC, 0, st>>>(K, KP, sp, vp);
    auto trace = KP <= 32 ? vit_trace_kernel<1> : vit_trace_kernel<2>;
    trace<<<ctas, 128, 0, st>>>(K, KP, init_mode, pi, P, head, packed, sp, vp, path);
    vit_score_kernel<<<1, 256, 0, st>>>(sp.n, vp, score);
    return cudaGetLastError();
}

}  // namespace hmm
