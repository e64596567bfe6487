// One direction of a dense K-state pairwise factor (K = 4, 8, 16), thread-local, shared by
// the kernel forms that give the same bits (kernels.cu: k_pair_thr, k_pair_dir, k_pair_quad;
// pair_fused.cu). From the source variable's values v, the target's message is
//   o(t) = T log sum_s exp((phi(s, t) + v(s)) / T)   (max_s phi(s, t) + v(s) at T = 0),
// up to a constant per message, which the normalisation that follows removes.
//
// What bounds it: the bytes a warp takes from shared memory (the return path gives 128 a
// cycle, broadcast or not) and issue slots. At K = 16 the direction is 256 multiply-adds, 16
// exponentials and 16 logarithms. Here two targets share an instruction (fma.rn.f32x2 and its add
// and mul, Blackwell's packed FP32, rounding each half as the scalar does), and the tables are
// stored source-major so that a 16-byte load brings four targets of one source. The operations
// and their order are the scalar form's (w = __expf, sources 3, 2, 1, 0, 7, 6, ..., T logf(s) + max
// v + max phi, two normalisations): grids with strong couplings amplify any change of rounding by
// 10^4 over 100 iterations. (A polynomial logarithm and one normalisation measured 1.2x faster.)
#pragma once

#include "bp_common.cuh"

namespace pgm {
namespace {

typedef unsigned long long F2;  // two floats, the first in the low half

__device__ __forceinline__ F2 f2(float a, float b) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 f2_get(F2 a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

template <int K>
__device__ __forceinline__ float f2_max(const F2 (&a)[K / 2]) {
    float mx = kNegInf;
#pragma unroll
    for (int i = 0; i < K / 2; ++i) {
        const float2 q = f2_get(a[i]);
        mx = fmaxf(mx, fmaxf(q.x, q.y));
    }
    return mx;
}

__device__ __forceinline__ float ex2_ftz(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Two weights exp((v - vmax) / T) (__expf, but a result below the normal numbers is 0: beside the
// largest weight, 1, it adds nothing).
__device__ __forceinline__ float2 pair_weights(F2 v, float vmax, float invT) {
    const F2 x = f2_mul(f2_mul(f2_add(v, f2(-vmax, -vmax)), f2(invT, invT)), f2(1.4426950408889634f, 1.4426950408889634f));
    const float2 q = f2_get(x);
    return make_float2(ex2_ftz(q.x), ex2_ftz(q.y));
}

// Two outputs of the linear form from their sums.
__device__ __forceinline__ F2 pair_log(F2 s, float T, float vmax, float tmax) {
    const float2 q = f2_get(s);
    return f2_add(f2_fma(f2(T, T), f2(logf(q.x), logf(q.y)), f2(vmax, vmax)), f2(tmax, tmax));
}

// Linear form (sum-product, a shared table of range at most 60 T): S[s K + t] = exp((phi(s, t) -
// tmax) / T) in shared memory, 16-byte aligned, tmax = max phi; o = T log(sum_s S(s, t) w(s)) + vmax +
// tmax. The sum is at least exp(-range / T), a normal number.
template <int K>
__device__ __forceinline__ void pair_linear(const F2 (&v)[K / 2], F2 (&o)[K / 2], const float *S, float tmax, float T,
                                            float invT) {
    const float vmax = f2_max<K>(v);
    if (vmax == kNegInf) {
#pragma unroll
        for (int i = 0; i < K / 2; ++i) o[i] = f2(kNegInf, kNegInf);
        return;
    }
    float w[K];
#pragma unroll
    for (int i = 0; i < K / 2; ++i) {
        const float2 q = pair_weights(v[i], vmax, invT);
        w[2 * i] = q.x;
        w[2 * i + 1] = q.y;
        o[i] = f2(0.f, 0.f);
    }
#pragma unroll
    for (int j = 0; j < K / 4; ++j)
#pragma unroll
        for (int i = 3; i >= 0; --i) {
            const ulonglong2 *row = reinterpret_cast<const ulonglong2 *>(S + (4 * j + i) * K);
            const F2 ws = f2(w[4 * j + i], w[4 * j + i]);
#pragma unroll
            for (int q = 0; q < K / 4; ++q) {
                const ulonglong2 a = row[q];
                o[2 * q] = f2_fma(a.x, ws, o[2 * q]);
                o[2 * q + 1] = f2_fma(a.y, ws, o[2 * q + 1]);
            }
        }
#pragma unroll
    for (int i = 0; i < K / 2; ++i) o[i] = pair_log(o[i], T, vmax, tmax);
}

// Max-product with a shared table, S[s K + t] = phi(s, t) in shared memory.
template <int K>
__device__ __forceinline__ void pair_max(const F2 (&v)[K / 2], F2 (&o)[K / 2], const float *S) {
    float m[K];
#pragma unroll
    for (int t = 0; t < K; ++t) m[t] = kNegInf;
#pragma unroll
    for (int s = 0; s < K; ++s) {
        const ulonglong2 *row = reinterpret_cast<const ulonglong2 *>(S + s * K);
        const float2 p = f2_get(v[s / 2]);
        const F2 vs = (s & 1) ? f2(p.y, p.y) : f2(p.x, p.x);
#pragma unroll
        for (int q = 0; q < K / 4; ++q) {
            const ulonglong2 a = row[q];
            const float2 x = f2_get(f2_add(a.x, vs)), y = f2_get(f2_add(a.y, vs));
            m[4 * q] = fmaxf(m[4 * q], x.x);
            m[4 * q + 1] = fmaxf(m[4 * q + 1], x.y);
            m[4 * q + 2] = fmaxf(m[4 * q + 2], y.x);
            m[4 * q + 3] = fmaxf(m[4 * q + 3], y.y);
        }
    }
#pragma unroll
    for (int i = 0; i < K / 2; ++i) o[i] = f2(m[2 * i], m[2 * i + 1]);
}

// Any table, entry by entry: phi(s, t) at phi[s step_s + t step_t].
template <int K, bool MAXP>
__device__ __forceinline__ void pair_entries(const float (&v)[K], float (&o)[K], const float *phi, int step_s, int step_t,
                                             float T, float invT) {
#pragma unroll
    for (int t = 0; t < K; ++t) {
        float z[K];
#pragma unroll
        for (int s = 0; s < K; ++s) z[s] = phi[s * step_s + t * step_t] + v[s];
        o[t] = lse_row<K, MAXP>(z, T, invT);
    }
}

// normalise, damp, normalise (finish_k): o becomes the new message.
template <int K>
__device__ __forceinline__ void f2_normalise(F2 (&t)[K / 2], uint32_t *flags) {
    const float mx = f2_max<K>(t);
    if (mx == kNegInf) {
        atomicOr(flags, kFlagContradiction);
#pragma unroll
        for (int i = 0; i < K / 2; ++i) t[i] = f2(0.f, 0.f);
        return;
    }
    const F2 n = f2(-mx, -mx);
#pragma unroll
    for (int i = 0; i < K / 2; ++i) t[i] = f2_add(t[i], n);
}
template <int K>
__device__ __forceinline__ void pair_finish(F2 (&o)[K / 2], const F2 (&mo)[K / 2], float damping, uint32_t *flags) {
    f2_normalise<K>(o, flags);
    if (damping != 0.f) {
        const float w = 1.f - damping;
        const F2 d2 = f2(damping, damping), w2 = f2(w, w);
#pragma unroll
        for (int i = 0; i < K / 2; ++i) o[i] = f2_fma(d2, mo[i], f2_mul(w2, o[i]));
    }
    f2_normalise<K>(o, flags);
}

template <int K>
__device__ __forceinline__ void f2_load(F2 (&d)[K / 2], const float *__restrict__ p) {
    float q[K];
    load_n<K>(q, p);
#pragma unroll
    for (int i = 0; i < K / 2; ++i) d[i] = f2(q[2 * i], q[2 * i + 1]);
}
template <int K>
__device__ __forceinline__ void f2_store(float *__restrict__ p, const F2 (&d)[K / 2]) {
    float q[K];
#pragma unroll
    for (int i = 0; i < K / 2; ++i) {
        const float2 a = f2_get(d[i]);
        q[2 * i] = a.x;
        q[2 * i + 1] = a.y;
    }
    store_n<K>(p, q);
}
// needs_exact of any entry (a NaN entry too).
template <int K>
__device__ __forceinline__ bool f2_needs_exact(const F2 (&m)[K / 2]) {
    bool any = false;
#pragma unroll
    for (int i = 0; i < K / 2; ++i) {
        const float2 q = f2_get(m[i]);
        any |= !(fmaxf(fabsf(q.x), fabsf(q.y)) <= kExactThreshold) | (q.x != q.x) | (q.y != q.y);
    }
    return any;
}

// One direction through the guarded arithmetic, out of line: the source edge is one of a
// high-degree variable or has a stored entry that is -inf or large (gather_v2f). phi(s, t) as in
// pair_entries, in shared or global memory.
template <int K, bool MAXP>
__device__ __noinline__ void pair_dir_rare(const DevGraph &G, const float *phi, int step_s, int step_t, const float *b,
                                           const float *ev, const float *m_old, float *m_new, int vs_s, int es_s,
                                           int es_t, float T, float invT, float damping) {
    float mo[K], v[K], o[K];
    load_n<K>(mo, m_old + es_s);
    gather_v2f<K>(G, b, ev, m_old, vs_s, es_s, mo, v);
    pair_entries<K, MAXP>(v, o, phi, step_s, step_t, T, invT);
    F2 o2[K / 2], m2[K / 2];
#pragma unroll
    for (int i = 0; i < K / 2; ++i) o2[i] = f2(o[2 * i], o[2 * i + 1]);
    f2_load<K>(m2, m_old + es_t);
    pair_finish<K>(o2, m2, damping, G.flags);
    f2_store<K>(m_new + es_t, o2);
}

// One direction of a factor whose source edge is regular: v becomes the source's values (in),
// the new message goes to m_new + es_t. lin: S holds the linear table; else, for max-product
// with a shared table, phi itself; else phi entry by entry.
template <int K, bool MAXP>
__device__ __forceinline__ void pair_direction(const F2 (&v)[K / 2], bool lin, float tmax, bool shared, const float *S,
                                               const float *phi, int step_s, int step_t, const float *m_old,
                                               float *m_new, int es_t, float T, float invT, float damping,
                                               uint32_t *flags) {
    F2 o[K / 2], mo[K / 2];
    f2_load<K>(mo, m_old + es_t);
    if (!MAXP && lin) {
        pair_linear<K>(v, o, S, tmax, T, invT);
    } else if (MAXP && shared) {
        pair_max<K>(v, o, S);
    } else {
        float vv[K], oo[K];
#pragma unroll
        for (int i = 0; i < K / 2; ++i) {
            const float2 q = f2_get(v[i]);
            vv[2 * i] = q.x;
            vv[2 * i + 1] = q.y;
        }
        pair_entries<K, MAXP>(vv, oo, phi, step_s, step_t, T, invT);
#pragma unroll
        for (int i = 0; i < K / 2; ++i) o[i] = f2(oo[2 * i], oo[2 * i + 1]);
    }
    pair_finish<K>(o, mo, damping, flags);
    f2_store<K>(m_new + es_t, o);
}

// A group's shared table for a block (all threads): the raw entries in tab (row-major) and, for
// the fast forms, source-major tables S0 (source: variable 0) and S1 (source: variable 1):
// exp((phi - max) / T) when lin (returned: sum-product and a range of at most 60 T, red[0] = max),
// phi for max-product. red: 2 floats per warp.
template <int K>
__device__ __forceinline__ void table_store(float *S0, float *S1, int i, float e) {
    S0[i] = e;
    S1[(i % K) * K + i / K] = e;
}
// The raw entries (pair_tables_load), then, after a barrier, the fast forms' (pair_tables_make).
// NT: threads of the block, 0 if known at run time only.
template <int K, int NT = 0>
__device__ __forceinline__ void pair_tables_load(const float *__restrict__ phi, float *tab) {
#pragma unroll
    for (int i = threadIdx.x; i < K * K; i += NT ? NT : blockDim.x) tab[i] = __ldg(phi + i);
}
template <int K, bool MAXP, int NT = 0>
__device__ __forceinline__ bool pair_tables_make(const float *tab, float *S0, float *S1, float *red, float invT) {
    const int nt = NT ? NT : (int)blockDim.x, nw = nt >> 5, w = threadIdx.x >> 5;
    float mx = kNegInf, mn = CUDART_INF_F;
    for (int i = threadIdx.x; i < K * K; i += nt) {
        const float t = tab[i];
        if (MAXP) table_store<K>(S0, S1, i, t);
        mx = fmaxf(mx, t);
        mn = fminf(mn, t);
    }
    bool lin = false;
    if constexpr (!MAXP) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
            mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, d));
        }
        if ((threadIdx.x & 31) == 0) {
            red[2 * w] = mx;
            red[2 * w + 1] = mn;
        }
        __syncthreads();
        for (int j = 0; j < nw; ++j) {
            mx = fmaxf(mx, red[2 * j]);
            mn = fminf(mn, red[2 * j + 1]);
        }
        lin = isfinite(mx) && isfinite(mn) && (mx - mn) * invT <= 60.f;
        if (lin)
            for (int i = threadIdx.x; i < K * K; i += nt) table_store<K>(S0, S1, i, expf((tab[i] - mx) * invT));
        __syncthreads();
        if (threadIdx.x == 0) red[0] = mx;
    }
    __syncthreads();
    return lin;
}
template <int K, bool MAXP>
__device__ __forceinline__ bool pair_tables(const float *__restrict__ phi, float *tab, float *S0, float *S1, float *red,
                                            float invT) {
    pair_tables_load<K>(phi, tab);
    __syncthreads();
    return pair_tables_make<K, MAXP>(tab, S0, S1, red, invT);
}

}  // namespace
}  // namespace pgm
