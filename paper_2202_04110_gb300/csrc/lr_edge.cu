// Log-ratio iterations of binary graphs with high-degree variables -- pairwise factors (an RBM's
// layers), or OR and AND factors in max-product (deconvolution): one number per edge, d = m(1) - m(0), in edge order. The variable pass sums a variable's d into
// its total D (float-float); the factor pass forms both variable-to-factor log-ratios as D - d,
// updates both messages and stores them in place.
//
// An iteration of the edge-state form moves 16 bytes of messages per edge twice over and gathers
// 64 bytes of state totals per factor; this one reads 4 and writes 4 bytes per edge, gathers 16
// bytes of totals per factor and reads the tables as they are. The first iteration reads the
// caller's messages and the last one writes them, so a run has no conversion passes and needs
// no memory beyond the edge-state form's (d, and explicit sums where a term is infinite, in its
// second message buffer, D in its beliefs).
//
// Measured against the edge-state launches (GB300, whole calls, us per iteration), T = 1: 784 x 500
// (392,000 factors) 22.7 -> 9.7, 1000 x 1000 35.4 -> 17.5, 2000 x 128 22.9 -> 12.5, 100 x 150 10.7 ->
// 4.0, 70 x 80 10.6 -> 3.6 (two launches' latency); deconvolution of 100 images (T = 0, 1.8 million
// AND factors, 22,500 ORs of up to 180 parents) 125 -> 91: per launch, events included, AND 42.8 ->
// 27.1, OR 36.2 -> 24.9, the two variable launches 24.8 -> 22.1 and 32 -> 28.7, which are bound by
// gathers of 4 bytes a sector. Error against 64 bits, relative: RBM messages 7.7e-7 -> 9.4e-8,
// deconvolution 1.7e-7 -> 9.7e-8.
#include <algorithm>

#include "bp_common.cuh"

namespace pgm {
namespace {

// An edge's stored log-ratio; both entries -inf (which only a caller's messages can hold) is
// the NaN pattern of lam_encode.
__device__ __forceinline__ float edge_encode(float2 q) {
    if (q.x == kNegInf && q.y == kNegInf) return __uint_as_float(kLamBothNegInf);
    return lr_encode(q.x, q.y);
}

__device__ __forceinline__ float2 load_pair(const float *__restrict__ m) {
    return __ldcg(reinterpret_cast<const float2 *>(m));
}

// d of the edge whose states start at es: from the caller's messages m in the first
// iteration, else from d.
__device__ __forceinline__ float edge_ratio(const float *__restrict__ d, const float *__restrict__ m, int es) {
    return m != nullptr ? edge_encode(load_pair(m + es)) : __ldcg(d + (es >> 1));
}

__device__ __forceinline__ bool aligned16(const float *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// The next launch may be scheduled once every block of this one has its inputs: where they are
// all resident (784 x 500: 164,000 and 196,000 threads; 152 SMs hold 311,000). Blocks that still queue
// need the places. (By threads, since these kernels' blocks have 128 to 1,024; the edge-state
// kernels' rule, pdl_launch_if_small, counts blocks of mostly 256 and more registers.)
__device__ __forceinline__ void pdl_launch_if_one_wave() {
    if ((int64_t)gridDim.x * gridDim.y * blockDim.x <= 300000) pdl_launch_dependents();
}

// A state's total as hd_pair takes it: the float-float sum of the finite terms and the count
// of the -inf ones.
__device__ __forceinline__ void add_term(FF &s, float &c, float q) {
    if (q == kNegInf) c += 1.f;
    else s = ff_add(s, q);
}

// A clamped variable -- one state's evidence -inf, the other's finite -- whose messages are finite and
// far from overflow has every leave-one-out log-ratio at that infinity, whatever the messages: its
// total says so (edge_lam), without the explicit sums (784 x 500, all visible variables clamped: 20.6 us per
// iteration with them, 10.4 so; the edge-state form takes 22.4). 0: not such a variable.
constexpr float kClampedMax = 1e30f;  // (times the largest degree far below the largest number)
__device__ __forceinline__ float clamped_ratio(float2 e) {
    if (e.x == kNegInf && isfinite(e.y)) return CUDART_INF_F;
    if (e.y == kNegInf && isfinite(e.x)) return kNegInf;
    return 0.f;
}

// Block per variable of more than kVarBlockDegree factors, 128 threads (1024 on graphs with
// variables of more than kLrEdgeMaxDegree) with 8 edges each in flight. The gathers' latency bounds it: every block is resident at once (1284 blocks for 784 x
// 500), the edge list is read before the previous pass ends, and each thread adds its edges in
// float-float before two levels of block sums.
constexpr int kEdgeVarItems = 8;
template <int B>
__global__ void __launch_bounds__(B) k_edge_var_block(DevGraph G, const int32_t *__restrict__ list,
                                                                    const float *__restrict__ ev,
                                                                    const float *__restrict__ d,
                                                                    const float *__restrict__ m,
                                                                    float2 *__restrict__ Dv) {
    __shared__ float sh[3 * B / 32];
    const int64_t smp = sample_select(G);  // multi-sample launches: this block's sample
    ev += smp * G.s_vs;
    d += smp * G.s_es;
    if (m) m += smp * G.s_es;
    Dv += smp * (G.s_vs / 2);
    constexpr int N = kEdgeVarItems;
    const int v = list ? __ldg(list + blockIdx.x) : (int)blockIdx.x;
    const int k0 = __ldg(G.vin_off + v), k1 = __ldg(G.vin_off + v + 1);
    int es[N];
    auto load_es = [&](int base) {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int j = base + i * B + (int)threadIdx.x;
            es[i] = j < k1 ? __ldg(G.vin_es + j) : -1;
        }
    };
    load_es(k0);
    pdl_wait();  // the previous pass's messages
    pdl_launch_if_one_wave();
    const float2 e = make_float2(__ldg(ev + 2 * (size_t)v), __ldg(ev + 2 * (size_t)v + 1));
    FF s = ff_make(0.f);
    bool fin = true, big = false;
    for (int base = k0;;) {
        float q[N];
#pragma unroll
        for (int i = 0; i < N; ++i) q[i] = es[i] >= 0 ? edge_ratio(d, m, es[i]) : 0.f;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            fin &= isfinite(q[i]);
            big |= fabsf(q[i]) > kClampedMax;
            s = ff_add_nc(s, q[i]);
        }
        base += N * B;
        if (base >= k1) break;
        load_es(base);
    }
    float c = !fin ? 1.f : big ? 1.f / 65536.f : 0.f;  // below 1: every thread's are finite
    const FF tot = block_sum_count(s, c, sh);
    FF D = ff_add_nc(ff_make(e.y), -e.x);
    D = ff_add(D, tot);
    if (c < 1.f && isfinite(D.hi) && isfinite(D.lo)) {
        if (threadIdx.x == 0) Dv[v] = make_float2(D.hi, D.lo);
        return;
    }
    const float inf = c == 0.f ? clamped_ratio(e) : 0.f;
    if (inf != 0.f) {
        if (threadIdx.x == 0) Dv[v] = make_float2(inf, 0.f);
        return;
    }
    // an infinite (or NaN) term, the same for the whole block: the two states' totals apart
    for (int x = 0; x < 2; ++x) {
        FF sx = ff_make(0.f);
        float cx = 0.f;
        for (int j = k0 + (int)threadIdx.x; j < k1; j += B) {
            const float2 q = lam_decode(edge_ratio(d, m, __ldg(G.vin_es + j)));
            add_term(sx, cx, x ? q.y : q.x);
        }
        FF t = block_sum_count(sx, cx, sh);
        add_term(t, cx, x ? e.y : e.x);
        if (threadIdx.x == 0)
            reinterpret_cast<float4 *>(G.hd_b)[2 * (size_t)v + x] = make_float4(t.hi, t.lo, cx, 0.f);
    }
    if (threadIdx.x == 0) Dv[v] = make_float2(__uint_as_float(kDvSlow), 0.f);
}

// The graph's other variables: thread per variable.
__global__ void __launch_bounds__(256) k_edge_var_thread(DevGraph G, const int32_t *__restrict__ list, int n,
                                                         const float *__restrict__ ev, const float *__restrict__ d,
                                                         const float *__restrict__ m, float2 *__restrict__ Dv) {
    const int64_t smp = sample_select(G);  // multi-sample launches: this block's sample
    ev += smp * G.s_vs;
    d += smp * G.s_es;
    if (m) m += smp * G.s_es;
    Dv += smp * (G.s_vs / 2);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int v = i < n ? (list ? __ldg(list + i) : i) : 0;
    const int k0 = __ldg(G.vin_off + v), k1 = __ldg(G.vin_off + v + 1);
    pdl_wait();  // the previous pass's messages
    pdl_launch_if_one_wave();
    if (i >= n) return;
    const float2 e = make_float2(__ldg(ev + 2 * (size_t)v), __ldg(ev + 2 * (size_t)v + 1));
    FF D = ff_add_nc(ff_make(e.y), -e.x);
    bool fin = true, big = false;
    for (int k = k0; k < k1; k += 4) {
        float q[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) q[j] = k + j < k1 ? edge_ratio(d, m, __ldg(G.vin_es + k + j)) : 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            fin &= isfinite(q[j]);
            big |= fabsf(q[j]) > kClampedMax;
            D = ff_add_nc(D, q[j]);
        }
    }
    if (fin && isfinite(D.hi) && isfinite(D.lo)) {
        Dv[v] = make_float2(D.hi, D.lo);
        return;
    }
    const float inf = fin && !big ? clamped_ratio(e) : 0.f;
    if (inf != 0.f) {
        Dv[v] = make_float2(inf, 0.f);
        return;
    }
    // an infinite (or NaN) term: each edge's explicit sums without its own message
    float *lam = const_cast<float *>(d) + G.E;
    for (int k = k0; k < k1; ++k) {
        FF l0 = ff_make(e.x), l1 = ff_make(e.y);
        for (int o = k0; o < k1; ++o) {
            if (o == k) continue;
            const float2 q = lam_decode(edge_ratio(d, m, __ldg(G.vin_es + o)));
            l0 = ff_add(l0, q.x);
            l1 = ff_add(l1, q.y);
        }
        lam[__ldg(G.vin_es + k) >> 1] = lam_encode(l0, l1);
    }
    Dv[v] = make_float2(__uint_as_float(kDvSlow), 0.f);
}

// The leave-one-out log-ratio of edge e (vs: its edge_vs, mo its d) of a variable with an infinite
// term: a high-degree variable's from its two state totals, another's from the explicit sums.
__device__ __noinline__ float edge_lam_slow(const DevGraph &G, const float *d, int e, int vs, float mo) {
    if (vs >= 0) return __ldcg(d + G.E + e);
    const float2 q = lam_decode(mo);
    const float m2[2] = {q.x, q.y};
    float l[2];
    hd_v2f<2>(G, vs, m2, l);
    return lam_encode(ff_make(l[0]), ff_make(l[1]));
}

__device__ __forceinline__ float edge_lam(const DevGraph &G, float2 D, const float *d, int e, int vs, float mo) {
    if (__float_as_uint(D.x) == kDvSlow) return edge_lam_slow(G, d, e, vs, mo);
    const FF l = ff_add(FF{D.x, D.y}, -mo);
    return l.hi + l.lo;
}

// sp_T(x) - sp_T(y), x - y = D, E = expm1(-|D| / T), u the larger of x and y: with sigma = sigma(u / T)
// the ratio of 1 + e^(smaller / T) to 1 + e^(u / T) is 1 + E sigma, so the difference is
// -+ T log1p(E sigma). Weak couplings make it small against the two values, whose difference on
// the SFU (lr_dir) loses what the messages' sums are made of: on 784 x 500 with couplings of 0.1
// the messages' error against 64 bits was 1.3e-6 with it, 7e-7 in the edge-state form. Where the
// ratio is below a half the two values are apart and their difference is taken as it is.
__device__ __forceinline__ float softplus_diff(float x, float y, float D, float E, float T, float invT) {
    const float u = (D >= 0.f ? x : y) * invT;
    const float t = expf(-fabsf(u)), r = __fdividef(1.f, 1.f + t);
    const float a = E * (u >= 0.f ? r : t * r);
    if (a > -0.5f) return copysignf(1.f, D) * (-T * log1pf(a));
    const float sx = fmaf(T, log1pf(expf(-fabsf(x) * invT)), fmaxf(x, 0.f));
    const float sy = fmaf(T, log1pf(expf(-fabsf(y) * invT)), fmaxf(y, 0.f));
    return sx - sy;
}

// lr_dir with that difference; D = p - q and its E are the same in both directions.
template <bool MAXP>
__device__ __forceinline__ float edge_dir(float r, float p, float q, float D, float E, float l, float mo, float T, float invT,
                                          float damping, float w) {
    if constexpr (MAXP) return lr_dir<true>(r, p, q, l, mo, 0.f, 0.f, damping, w);
    return fmaf(damping, mo, w * (r + softplus_diff(p + l, q + l, D, E, T, invT)));
}

template <bool MAXP>
__device__ __noinline__ float edge_exact(float4 t, int side, float l, float mo, float k, float Tln2, float damping,
                                         uint32_t *flags) {
    if (__float_as_uint(mo) == kLamBothNegInf && damping != 0.f) {  // damping keeps both entries at -inf
        atomicOr(flags, kFlagContradiction);
        return 0.f;
    }
    const float t4[4] = {t.x, t.y, t.z, t.w};
    return lr_dir_exact<MAXP>(t4, side, l, mo, k, Tln2, damping, flags);
}

// Thread per two consecutive factors: 16-byte loads of d, the edges' variables and each table.
// The variables' totals (8 bytes each, a few KB in all for an RBM) are the only gather. m_in /
// m_out: the caller's messages in the first / last iteration, nullptr in the others.
template <bool MAXP>
__global__ void __launch_bounds__(256) k_edge_pair(DevGraph G, const EnumSeg *__restrict__ segs, int n_seg, int F,
                                                   const float *__restrict__ pot, const float2 *__restrict__ Dv,
                                                   float *__restrict__ d, const float *m_in, float *m_out, float T,
                                                   float invT, float k, float Tln2, float damping) {
    const int64_t smp = sample_select(G);  // multi-sample launches: this block's sample
    pot += smp * G.s_pot;
    d += smp * G.s_es;
    if (m_in) m_in += smp * G.s_es;
    if (m_out) m_out += smp * G.s_es;
    Dv += smp * (G.s_vs / 2);
    const int g = 2 * (int)(blockIdx.x * blockDim.x + threadIdx.x);
    const int n = min(2, F - g);
    int4 vs = make_int4(0, 0, 0, 0);
    float4 tab[2];
    if (n == 2) {
        vs = __ldg(reinterpret_cast<const int4 *>(G.edge_vs + 2 * (size_t)g));
        tab[1] = lr_table(segs, n_seg, pot, g + 1);
    } else if (n == 1) {
        const int2 q = __ldg(reinterpret_cast<const int2 *>(G.edge_vs + 2 * (size_t)g));
        vs = make_int4(q.x, q.y, q.x, q.y);
    }
    if (n > 0) tab[0] = lr_table(segs, n_seg, pot, g);
    if (n < 2) tab[1] = tab[0];
    pdl_wait();  // the variable pass's totals
    pdl_launch_if_one_wave();
    if (n <= 0) return;
    float mo[4];
    if (m_in != nullptr) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            mo[i] = i < 2 * n ? edge_encode(load_pair(m_in + 4 * (size_t)g + 2 * i)) : 0.f;
    } else if (n == 2) {
        const float4 q = __ldcg(reinterpret_cast<const float4 *>(d + 2 * (size_t)g));
        mo[0] = q.x, mo[1] = q.y, mo[2] = q.z, mo[3] = q.w;
    } else {
        const float2 q = __ldcg(reinterpret_cast<const float2 *>(d + 2 * (size_t)g));
        mo[0] = q.x, mo[1] = q.y, mo[2] = 0.f, mo[3] = 0.f;
    }
    const int v[4] = {vs.x, vs.y, vs.z, vs.w};
    float2 D[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) D[i] = __ldca(Dv + ((v[i] & 0x7fffffff) >> 1));
    const float w = 1.f - damping;
    float o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int f = 0; f < 2; ++f) {
        if (f >= n) break;
        const float4 t = tab[f];
        const bool fin = isfinite(t.x) & isfinite(t.y) & isfinite(t.z) & isfinite(t.w);
        const float c = fin ? t.z - t.x : CUDART_NAN_F;  // as k_lr_params
        const float al = fin ? t.w - t.z : CUDART_NAN_F;
        const float be = fin ? t.y - t.x : CUDART_NAN_F;
        const float m0 = mo[2 * f], m1 = mo[2 * f + 1];
        const int e = 2 * (g + f);
        const float l0 = edge_lam(G, D[2 * f], d, e, v[2 * f], m0), l1 = edge_lam(G, D[2 * f + 1], d, e + 1, v[2 * f + 1], m1);
        const float dpq = al - be, E = MAXP ? 0.f : expm1f(-fabsf(dpq) * invT);
        float a = edge_dir<MAXP>(c, al, be, dpq, E, l1, m0, T, invT, damping, w);
        float b = edge_dir<MAXP>(be, c + dpq, c, dpq, E, l0, m1, T, invT, damping, w);
        if (lr_dir_rare(a, l1)) a = edge_exact<MAXP>(t, 0, l1, m0, k, Tln2, damping, G.flags);
        if (lr_dir_rare(b, l0)) b = edge_exact<MAXP>(t, 1, l0, m1, k, Tln2, damping, G.flags);
        o[2 * f] = a;
        o[2 * f + 1] = b;
    }
    if (m_out != nullptr) {
        float *p = m_out + 4 * (size_t)g;
        const bool al = aligned16(p);
#pragma unroll
        for (int f = 0; f < 2; ++f) {
            if (f >= n) break;
            const float2 a = lr_decode(o[2 * f]), b = lr_decode(o[2 * f + 1]);
            if (al) {
                reinterpret_cast<float4 *>(p)[f] = make_float4(a.x, a.y, b.x, b.y);
            } else {
                p[4 * f] = a.x, p[4 * f + 1] = a.y, p[4 * f + 2] = b.x, p[4 * f + 3] = b.y;
            }
        }
    } else if (n == 2) {
        *reinterpret_cast<float4 *>(d + 2 * (size_t)g) = make_float4(o[0], o[1], o[2], o[3]);
    } else {
        *reinterpret_cast<float2 *>(d + 2 * (size_t)g) = make_float2(o[0], o[1]);
    }
}

// ---- OR / AND factors, max-product ------------------------------------------------------
//
// The closed forms of k_logic_small and k_logic_warp on log-odds x = +-lam, which the log-ratio
// form has at hand: no states to gather and subtract.

__device__ __forceinline__ float edge_odds(const DevGraph &G, const float2 *Dv, const float *d, int e, int vs, float mo,
                                           float sgn) {
    const float l = edge_lam(G, __ldca(Dv + ((vs & 0x7fffffff) >> 1)), d, e, vs, mo);
    return __float_as_uint(l) == kLamBothNegInf ? 0.f : sgn * l;  // (log_odds of a contradiction)
}
// The stored d of edge e, and the new one written.
__device__ __forceinline__ float edge_load(const float *d, const float *m_in, int e) {
    return m_in != nullptr ? edge_encode(load_pair(m_in + 2 * (size_t)e)) : __ldcg(d + e);
}
__device__ __noinline__ float edge_finish(float o, float mo, float damping, uint32_t *flags) {
    const float2 q = lam_decode(mo);
    const float old[2] = {q.x, q.y};
    float t[2] = {o >= 0.f ? -o : 0.f, o >= 0.f ? 0.f : o};  // as write_logic_edge
    finish_k<2>(t, old, damping, flags);
    return t[1] - t[0];
}
__device__ __forceinline__ void edge_store(float *d, float *m_out, int e, float o, float mo, float damping,
                                           uint32_t *flags) {
    float n = fmaf(damping, mo, (1.f - damping) * o);
    if (!isfinite(n)) n = edge_finish(o, mo, damping, flags);
    if (m_out != nullptr) reinterpret_cast<float2 *>(m_out)[e] = lr_decode(n);
    else d[e] = n;
}

// Thread per factor of at most F parents. A factor's edges and those of the next thread are
// neighbours in d, and so are most of their variables' totals (L1).
template <int F>
__global__ void __launch_bounds__(256) k_edge_logic_small(DevGraph G, const LogicSeg *__restrict__ segs, int n_seg,
                                                          const float2 *Dv, float *d, const float *m_in, float *m_out,
                                                          float damping) {
    const int64_t smp = sample_select(G);  // multi-sample launches: this block's sample
    d += smp * G.s_es;
    if (m_in) m_in += smp * G.s_es;
    if (m_out) m_out += smp * G.s_es;
    Dv += smp * (G.s_vs / 2);
    const LogicSeg *S = segs + find_seg(segs, n_seg, blockIdx.x);
    const int f = (blockIdx.x - __ldg(&S->block_begin)) * blockDim.x + threadIdx.x;
    const bool have = f < __ldg(&S->n_fac);
    const float sgn = __ldg(&S->kind) == PGM_LOGIC_AND ? -1.f : 1.f;
    int n = 0, e0 = 0, vs[F], vc = 0;
    if (have) {
        const int *po = G.paroff_pool + __ldg(&S->paroff_base);
        const int p0 = __ldg(po + f);
        n = __ldg(po + f + 1) - p0;
        e0 = __ldg(&S->edge_base) + p0 + f;
#pragma unroll
        for (int k = 0; k < F; ++k) vs[k] = k < n ? __ldg(G.edge_vs + e0 + k) : 0;
        vc = __ldg(G.edge_vs + e0 + n);
    }
    pdl_wait();  // the variable pass's totals
    pdl_launch_if_one_wave();
    if (!have) return;
    float x[F], mo[F];
#pragma unroll
    for (int k = 0; k < F; ++k) mo[k] = k < n ? edge_load(d, m_in, e0 + k) : 0.f;
    const float moc = edge_load(d, m_in, e0 + n);
#pragma unroll
    for (int k = 0; k < F; ++k) x[k] = k < n ? edge_odds(G, Dv, d, e0 + k, vs[k], mo[k], sgn) : 0.f;
    const float xc = edge_odds(G, Dv, d, e0 + n, vc, moc, sgn);
    float A = 0.f, M = kNegInf;
#pragma unroll
    for (int j = 0; j < F; ++j)
        if (j < n) {
            A += fmaxf(x[j], 0.f);
            M = fmaxf(M, x[j]);
        }
    edge_store(d, m_out, e0 + n, sgn * (A + (M < 0.f ? M : 0.f)), moc, damping, G.flags);
#pragma unroll
    for (int i = 0; i < F; ++i) {
        if (i >= n) break;
        float Si = 0.f, Mi = kNegInf;
#pragma unroll
        for (int j = 0; j < F; ++j)
            if (j < n && j != i) {
                Si += fmaxf(x[j], 0.f);
                Mi = fmaxf(Mi, x[j]);
            }
        edge_store(d, m_out, e0 + i, sgn * or_parent_max(Si, Mi, xc), mo[i], damping, G.flags);
    }
}

// Warp per factor of at most 32 R parents, R a lane. Every edge of the factor is in flight at
// once and its indices are read before the variable pass ends; the parents' leave-one-out terms
// come from the total (float-float, +inf terms counted) less their own and from the two largest
// log-odds, instead of a scan in each direction.
template <int R>
__global__ void __launch_bounds__(128) k_edge_logic_warp(DevGraph G, const LogicSeg *__restrict__ segs, int n_seg,
                                                         const float2 *Dv, float *d, const float *m_in, float *m_out,
                                                         float damping) {
    const int64_t smp = sample_select(G);  // multi-sample launches: this block's sample
    d += smp * G.s_es;
    if (m_in) m_in += smp * G.s_es;
    if (m_out) m_out += smp * G.s_es;
    Dv += smp * (G.s_vs / 2);
    const int lane = threadIdx.x & 31;
    const LogicSeg *S = segs + find_seg(segs, n_seg, blockIdx.x);
    const int f = (blockIdx.x - __ldg(&S->block_begin)) * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const bool have = f < __ldg(&S->n_fac);  // the whole warp
    const float sgn = __ldg(&S->kind) == PGM_LOGIC_AND ? -1.f : 1.f;
    int n = 0, e0 = 0, vs[R], vc = 0;
    if (have) {
        const int *po = G.paroff_pool + __ldg(&S->paroff_base);
        const int p0 = __ldg(po + f);
        n = __ldg(po + f + 1) - p0;
        e0 = __ldg(&S->edge_base) + p0 + f;
#pragma unroll
        for (int r = 0; r < R; ++r) vs[r] = lane + 32 * r < n ? __ldg(G.edge_vs + e0 + lane + 32 * r) : 0;
        vc = __ldg(G.edge_vs + e0 + n);
    }
    pdl_wait();  // the variable pass's totals
    pdl_launch_if_one_wave();
    if (!have) return;
    float x[R], mo[R];
#pragma unroll
    for (int r = 0; r < R; ++r) mo[r] = lane + 32 * r < n ? edge_load(d, m_in, e0 + lane + 32 * r) : 0.f;
    const float moc = edge_load(d, m_in, e0 + n);
    const float xc = edge_odds(G, Dv, d, e0 + n, vc, moc, sgn);
    FF A = ff_make(0.f);
    float c = 0.f, M1 = kNegInf, M2 = kNegInf;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        x[r] = kNegInf;
        if (lane + 32 * r < n) {
            x[r] = edge_odds(G, Dv, d, e0 + lane + 32 * r, vs[r], mo[r], sgn);
            if (x[r] == CUDART_INF_F) c += 1.f;
            else A = ff_add(A, fmaxf(x[r], 0.f));
            if (x[r] == x[r]) M2 = fmaxf(M2, fminf(M1, x[r]));  // (a NaN counts as nothing)
            M1 = fmaxf(M1, x[r]);
        }
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        A = ff_add(A, FF{__shfl_xor_sync(0xffffffffu, A.hi, s), __shfl_xor_sync(0xffffffffu, A.lo, s)});
        c += __shfl_xor_sync(0xffffffffu, c, s);
        const float o1 = __shfl_xor_sync(0xffffffffu, M1, s), o2 = __shfl_xor_sync(0xffffffffu, M2, s);
        M2 = fmaxf(fminf(M1, o1), fmaxf(M2, o2));
        M1 = fmaxf(M1, o1);
    }
    if (lane == 0) {
        const float a = c > 0.f ? CUDART_INF_F : A.hi + A.lo;
        edge_store(d, m_out, e0 + n, sgn * (a + (M1 < 0.f ? M1 : 0.f)), moc, damping, G.flags);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (lane + 32 * r >= n) break;
        const bool inf = x[r] == CUDART_INF_F;
        float Si = CUDART_INF_F;
        if (c == (inf ? 1.f : 0.f)) {
            const FF a = inf ? A : ff_add(A, -fmaxf(x[r], 0.f));
            Si = fmaxf(a.hi + a.lo, 0.f);
        }
        edge_store(d, m_out, e0 + lane + 32 * r, sgn * or_parent_max(Si, x[r] == M1 ? M2 : M1, xc), mo[r], damping,
                   G.flags);
    }
}

template <typename... KArgs, typename... Args>
cudaError_t launch_after(void (*kernel)(KArgs...), int blocks, int S, int threads, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks, (unsigned)S);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace

cudaError_t launch_edge_var_pass(const DevGraph &G, const Plan &P, const float *ev, const float *d, const float *m_in,
                                 float2 *Dv, cudaStream_t s, int S, const LaunchHook *hook) {
    for (const VarLaunch &L : P.var) {
        if (L.n == 0) continue;
        const cudaError_t e =
            L.kind == kVarBlock
                ? (P.edge_var_threads == 128 ? launch_after(k_edge_var_block<128>, L.n, S, 128, s, G, L.list, ev, d, m_in, Dv)
                                             : launch_after(k_edge_var_block<1024>, L.n, S, 1024, s, G, L.list, ev, d, m_in, Dv))
                : launch_after(k_edge_var_thread, (L.n + 255) / 256, S, 256, s, G, L.list, L.n, ev, d, m_in, Dv);
        if (e != cudaSuccess) return e;
        if (hook) hook->after(hook->ctx);
    }
    return cudaSuccess;
}

cudaError_t launch_edge_factor_pass(const DevGraph &G, const Plan &P, const float *log_pot, const float2 *Dv, float *d,
                                    const float *m_in, float *m_out, float T, float damping, cudaStream_t s,
                                    int S, const LaunchHook *hook) {
    // lse2_fast constants: k = log2(e) / T, T ln 2
    const float k = T > 0.f ? (float)(1.4426950408889634 / (double)T) : 0.f;
    const float Tln2 = (float)((double)T * 0.6931471805599453);
    const int F = G.E / 2;
    for (const FactorLaunch &L : P.factor) {
        if (L.n_blocks == 0) continue;
        const LogicSeg *ls = static_cast<const LogicSeg *>(L.segs);
        cudaError_t e;
        if (L.variant == kPair2) {  // the one launch: every factor
            e = launch_after(T == 0.f ? k_edge_pair<true> : k_edge_pair<false>, (F + 511) / 512, S, 256, s, G,
                             static_cast<const EnumSeg *>(L.segs), L.n_seg, F, log_pot, Dv, d, m_in, m_out, T,
                             T > 0.f ? 1.f / T : 0.f, k, Tln2, damping);
        } else if (L.variant == kLogicSmall) {
            e = launch_after(L.max_fan <= 2 ? k_edge_logic_small<2> : k_edge_logic_small<kLogicSmallFan>, L.n_blocks, S,
                             L.threads, s, G, ls, L.n_seg, Dv, d, m_in, m_out, damping);
        } else {
            auto kern = L.max_fan <= 64    ? k_edge_logic_warp<2>
                        : L.max_fan <= 128 ? k_edge_logic_warp<4>
                        : L.max_fan <= 192 ? k_edge_logic_warp<6>
                                           : k_edge_logic_warp<8>;
            e = launch_after(kern, L.n_blocks, S, L.threads, s, G, ls, L.n_seg, Dv, d, m_in, m_out, damping);
        }
        if (e != cudaSuccess) return e;
        if (hook) hook->after(hook->ctx);
    }
    return cudaSuccess;
}

}  // namespace pgm
