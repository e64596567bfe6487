// Log-ratio iterations of binary pairwise graphs with high-degree variables (an RBM's layers):
// one number per edge, d = m(1) - m(0), in edge order. The variable pass sums a variable's d into
// its total D (float-float); the factor pass forms both variable-to-factor log-ratios as D - d,
// updates both messages and stores them in place.
//
// An iteration of the edge-state form moves 16 bytes of messages per edge twice over and gathers
// 64 bytes of state totals per factor; this one reads 4 and writes 4 bytes per edge, gathers 16
// bytes of totals per factor and reads the tables as they are. The first iteration reads the
// caller's messages and the last one writes them, so a run has no conversion passes and needs
// no memory beyond the edge-state form's (d in its second message buffer, D in its beliefs).
//
// Measured against the edge-state launches (GB300, T = 1, whole calls, us per iteration): 784 x 500
// (392,000 factors) 22.7 -> 11.1, 1000 x 1000 35.4 -> 17.5, 2000 x 128 22.9 -> 12.5, 100 x 150 10.7 ->
// 4.0, 70 x 80 10.6 -> 3.6 (two launches' latency). Error of the messages against 64 bits, relative:
// 7.7e-7 -> 9.4e-8.
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

// A state's total as hd_pair takes it: the float-float sum of the finite terms and the count
// of the -inf ones.
__device__ __forceinline__ void add_term(FF &s, float &c, float q) {
    if (q == kNegInf) c += 1.f;
    else s = ff_add(s, q);
}

// Block per variable of more than kVarBlockDegree factors, 128 threads with 8 edges each in
// flight. The gathers' latency bounds it: every block is resident at once (1284 blocks for 784 x
// 500), the edge list is read before the previous pass ends, and each thread adds its edges in
// float-float before two levels of block sums.
constexpr int kEdgeVarThreads = 128, kEdgeVarItems = 8;
__global__ void __launch_bounds__(kEdgeVarThreads) k_edge_var_block(DevGraph G, const int32_t *__restrict__ list,
                                                                    const float *__restrict__ ev,
                                                                    const float *__restrict__ d,
                                                                    const float *__restrict__ m,
                                                                    float2 *__restrict__ Dv) {
    __shared__ float sh[3 * kEdgeVarThreads / 32];
    const int64_t smp = sample_select(G);  // multi-sample launches: this block's sample
    ev += smp * G.s_vs;
    d += smp * G.s_es;
    if (m) m += smp * G.s_es;
    Dv += smp * (G.s_vs / 2);
    constexpr int N = kEdgeVarItems, B = kEdgeVarThreads;
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
    pdl_launch_dependents();
    const float2 e = make_float2(__ldg(ev + 2 * (size_t)v), __ldg(ev + 2 * (size_t)v + 1));
    FF s = ff_make(0.f);
    bool fin = isfinite(e.x) & isfinite(e.y);
    for (int base = k0;;) {
        float q[N];
#pragma unroll
        for (int i = 0; i < N; ++i) q[i] = es[i] >= 0 ? edge_ratio(d, m, es[i]) : 0.f;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            fin &= isfinite(q[i]);
            s = ff_add_nc(s, q[i]);
        }
        base += N * B;
        if (base >= k1) break;
        load_es(base);
    }
    float c = fin ? 0.f : 1.f;
    const FF tot = block_sum_count(s, c, sh);
    FF D = ff_add_nc(ff_make(e.y), -e.x);
    D = ff_add(D, tot);
    if (c == 0.f && isfinite(D.hi) && isfinite(D.lo)) {
        if (threadIdx.x == 0) Dv[v] = make_float2(D.hi, D.lo);
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
    pdl_launch_dependents();
    if (i >= n) return;
    const float2 e = make_float2(__ldg(ev + 2 * (size_t)v), __ldg(ev + 2 * (size_t)v + 1));
    FF D = ff_add_nc(ff_make(e.y), -e.x);
    bool fin = isfinite(e.x) & isfinite(e.y);
    for (int k = k0; k < k1; k += 4) {
        float q[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) q[j] = k + j < k1 ? edge_ratio(d, m, __ldg(G.vin_es + k + j)) : 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            fin &= isfinite(q[j]);
            D = ff_add_nc(D, q[j]);
        }
    }
    if (fin && isfinite(D.hi) && isfinite(D.lo)) {
        Dv[v] = make_float2(D.hi, D.lo);
        return;
    }
    FF s0 = ff_make(0.f), s1 = ff_make(0.f);
    float c0 = 0.f, c1 = 0.f;
    for (int k = k0; k < k1; ++k) {
        const float2 q = lam_decode(edge_ratio(d, m, __ldg(G.vin_es + k)));
        add_term(s0, c0, q.x);
        add_term(s1, c1, q.y);
    }
    add_term(s0, c0, e.x);
    add_term(s1, c1, e.y);
    float4 *t = reinterpret_cast<float4 *>(G.hd_b) + 2 * (size_t)v;
    t[0] = make_float4(s0.hi, s0.lo, c0, 0.f);
    t[1] = make_float4(s1.hi, s1.lo, c1, 0.f);
    Dv[v] = make_float2(__uint_as_float(kDvSlow), 0.f);
}

// The leave-one-out log-ratio of an edge from its variable's two state totals.
__device__ __noinline__ float edge_lam_slow(const DevGraph &G, int v, float mo) {
    const float2 q = lam_decode(mo);
    const float2 a = hd_pair(G, 2 * v, 0, q.x), b = hd_pair(G, 2 * v, 1, q.y);
    return lam_encode(FF{a.x, a.y}, FF{b.x, b.y});
}

__device__ __forceinline__ float edge_lam(const DevGraph &G, float2 D, int v, float mo) {
    if (__float_as_uint(D.x) == kDvSlow) return edge_lam_slow(G, v, mo);
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
    pdl_launch_dependents();
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
    const int v[4] = {(vs.x & 0x7fffffff) >> 1, (vs.y & 0x7fffffff) >> 1, (vs.z & 0x7fffffff) >> 1,
                      (vs.w & 0x7fffffff) >> 1};
    float2 D[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) D[i] = __ldcg(Dv + v[i]);
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
        const float l0 = edge_lam(G, D[2 * f], v[2 * f], m0), l1 = edge_lam(G, D[2 * f + 1], v[2 * f + 1], m1);
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
                ? launch_after(k_edge_var_block, L.n, S, kEdgeVarThreads, s, G, L.list, ev, d, m_in, Dv)
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
    for (const FactorLaunch &L : P.factor) {  // the one kPair2 launch: every factor
        if (L.n_blocks == 0) continue;
        const cudaError_t e = launch_after(T == 0.f ? k_edge_pair<true> : k_edge_pair<false>, (F + 511) / 512, S, 256,
                                           s, G, static_cast<const EnumSeg *>(L.segs), L.n_seg, F, log_pot, Dv, d, m_in,
                                           m_out, T, T > 0.f ? 1.f / T : 0.f, k, Tln2, damping);
        if (e != cudaSuccess) return e;
        if (hook) hook->after(hook->ctx);
    }
    return cudaSuccess;
}

}  // namespace pgm
