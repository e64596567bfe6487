// Device functions shared by the edge-state kernels (kernels.cu, pair_fused.cu): launch
// overlap, vector access, variable-to-factor values, log-sum-exp, the message epilogue,
// samples and batch members.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>
#include <math_constants.h>

#include "lr_math.cuh"
#include "pgm_internal.h"

namespace pgm {
namespace {

// Programmatic dependent launch (griddepcontrol): a kernel launched with the
// programmatic-serialization attribute may be scheduled before the previous kernel of
// its stream has finished. pdl_wait() returns once that kernel has completed and its
// writes are visible (at once for a kernel launched without the attribute);
// pdl_launch_dependents() lets the next kernel be scheduled before this one ends.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;"); }
// The same for a grid of at most kPdlBlocks blocks. The next launch's blocks wait on the SMs for
// this one to end: that hides a launch when the grid is small (4 blocks per SM), but where blocks
// of this grid still queue, the waiting ones take their places (a 256 x 256 grid of K = 8: 8.7 us
// per iteration without, 11.2 with; deconvolution of 100 images 118 without, 125 with).
constexpr unsigned kPdlBlocks = 640;
__device__ __forceinline__ bool pdl_small() { return gridDim.x * gridDim.y <= kPdlBlocks; }
__device__ __forceinline__ void pdl_launch_if_small() {
    if (pdl_small()) pdl_launch_dependents();
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class Seg>
__device__ __forceinline__ int find_seg(const Seg *__restrict__ segs, int n, int blk) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (__ldg(&segs[mid].block_begin) <= blk) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// ---- vector loads / stores with a run-time alignment check -------------------------

template <int N>
__device__ __forceinline__ void load_n(float (&d)[N], const float *__restrict__ p) {
    if constexpr (N % 4 == 0) {
        if ((reinterpret_cast<uintptr_t>(p) & 15u) == 0) {
#pragma unroll
            for (int i = 0; i < N / 4; ++i) {
                float4 q = __ldg(reinterpret_cast<const float4 *>(p) + i);
                d[4 * i] = q.x; d[4 * i + 1] = q.y; d[4 * i + 2] = q.z; d[4 * i + 3] = q.w;
            }
            return;
        }
    }
    if constexpr (N % 2 == 0) {
        if ((reinterpret_cast<uintptr_t>(p) & 7u) == 0) {
#pragma unroll
            for (int i = 0; i < N / 2; ++i) {
                float2 q = __ldg(reinterpret_cast<const float2 *>(p) + i);
                d[2 * i] = q.x; d[2 * i + 1] = q.y;
            }
            return;
        }
    }
#pragma unroll
    for (int i = 0; i < N; ++i) d[i] = __ldg(p + i);
}

// Streaming load of data read once per iteration (messages).
template <int N>
__device__ __forceinline__ void load_n_stream(float (&d)[N], const float *__restrict__ p) {
    if constexpr (N % 4 == 0) {
        if ((reinterpret_cast<uintptr_t>(p) & 15u) == 0) {
#pragma unroll
            for (int i = 0; i < N / 4; ++i) {
                float4 q = __ldcs(reinterpret_cast<const float4 *>(p) + i);
                d[4 * i] = q.x; d[4 * i + 1] = q.y; d[4 * i + 2] = q.z; d[4 * i + 3] = q.w;
            }
            return;
        }
    }
    load_n<N>(d, p);
}

template <int N>
__device__ __forceinline__ void store_n(float *__restrict__ p, const float (&s)[N]) {
    if constexpr (N % 4 == 0) {
        if ((reinterpret_cast<uintptr_t>(p) & 15u) == 0) {
#pragma unroll
            for (int i = 0; i < N / 4; ++i)
                reinterpret_cast<float4 *>(p)[i] = make_float4(s[4 * i], s[4 * i + 1], s[4 * i + 2], s[4 * i + 3]);
            return;
        }
    }
    if constexpr (N % 2 == 0) {
        if ((reinterpret_cast<uintptr_t>(p) & 7u) == 0) {
#pragma unroll
            for (int i = 0; i < N / 2; ++i)
                reinterpret_cast<float2 *>(p)[i] = make_float2(s[2 * i], s[2 * i + 1]);
            return;
        }
    }
#pragma unroll
    for (int i = 0; i < N; ++i) p[i] = s[i];
}

// a > b, compared exactly on the float-float values
__device__ __forceinline__ bool ff_gt(FF a, FF b) {
    if (a.hi == kNegInf) return false;
    if (b.hi == kNegInf) return true;
    return ff_diff(a, b) > 0.f;
}

// What r = ff_diff(a, b) dropped: (a - b) - r, from the two-sum of the high parts plus
// the low parts; 0 where a or b is not finite.
__device__ __forceinline__ float ff_diff_lo(FF a, FF b, float r) {
    if (!isfinite(a.hi) || !isfinite(b.hi)) return 0.f;
    const float th = a.hi - b.hi, bb = th - a.hi;
    const float te = (a.hi - (th - bb)) + (-b.hi - bb);
    return (th - r) + (te + (a.lo - b.lo));
}

// Belief residuals of a binary variable whose relative beliefs (r0, r1) came from the
// float-float sums (s0, s1): the larger state is exact (0), the other keeps what its
// rounding dropped.
__device__ __forceinline__ void write_b_lo2(float *p, FF s0, FF s1, float r0, float r1) {
    float l0 = 0.f, l1 = 0.f;
    if (r0 != 0.f || r1 != 0.f) {
        if (r1 == 0.f) l0 = ff_diff_lo(s0, s1, r0);
        else l1 = ff_diff_lo(s1, s0, r1);
    }
    reinterpret_cast<float2 *>(p)[0] = make_float2(l0, l1);
}

// ---- variable-to-factor value -------------------------------------------------------

// Explicit leave-one-out values of one edge: v(x) = e_v(x) + sum over the variable's
// other incoming edges of m(x), float-float summed, for all K states of the edge. Used
// when b - m would be unreliable: a stored entry is -inf (-inf - -inf) or very large
// (cancellation). Its per-edge constant differs from the fast path's, which the factor
// update does not see (it is invariant to a constant added to one edge's values).
constexpr float kExactThreshold = 128.f;

__device__ __noinline__ void v2f_slow_edge(const DevGraph G, const float *__restrict__ ev,
                                           const float *__restrict__ m, int vs, int es, int K,
                                           float *__restrict__ out) {
    int lo = 0, hi = G.V - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (G.vs_off[mid] <= vs) lo = mid;
        else hi = mid - 1;
    }
    const int k0 = G.vin_off[lo], k1 = G.vin_off[lo + 1];
    for (int x = 0; x < K; ++x) {
        FF s = ff_make(ev[vs + x]);
        for (int k = k0; k < k1; ++k) {
            const int e2 = G.vin_es[k];
            if (e2 != es) s = ff_add(s, m[e2 + x]);
        }
        out[x] = s.hi + s.lo;
    }
}

__device__ __forceinline__ bool needs_exact(float mv) { return !(fabsf(mv) <= kExactThreshold); }

// High-degree variables (more than kVarBlockDegree factors; their edges carry edge_vs
// with the sign bit set, the variable's first state in the other bits): the variable pass
// keeps, per state, the float-float sum of the finite evidence and incoming entries and
// the count of the -inf ones (G.hd_b, float4 (hi, lo, count, 0)). An edge's exact
// leave-one-out value is that sum less the edge's own entry -- -inf when another entry
// or the evidence is -inf -- formed in float-float from the four numbers and the entry,
// so that the pass writes nothing per edge. Returned as a (hi, lo) pair.
__device__ __forceinline__ float2 hd_pair(const DevGraph &G, int vs, int x, float mo) {
    const float4 t = __ldg(reinterpret_cast<const float4 *>(G.hd_b) + (vs & 0x7fffffff) + x);
    const bool own = (mo == -CUDART_INF_F);
    if (t.z > (own ? 1.f : 0.f)) return make_float2(-CUDART_INF_F, 0.f);
    if (own) return make_float2(t.x, t.y);
    const float sh = t.x - mo;
    if (!isfinite(sh)) return make_float2(sh, 0.f);
    // two-sum of the high parts, then the low part, renormalised
    const float bb = sh - t.x;
    const float err = (t.x - (sh - bb)) + (-mo - bb);
    const float lo = err + t.y;
    const float hi = sh + lo;
    return make_float2(hi, lo - (hi - sh));
}

__device__ __forceinline__ float hd_rel(float2 a, float2 mx) {
    if (!isfinite(a.x) || !isfinite(mx.x)) return a.x - mx.x;
    return (a.x - mx.x) + (a.y - mx.y);
}

__device__ __forceinline__ bool hd_gt(float2 a, float2 b) {
    if (a.x == -CUDART_INF_F) return false;
    if (b.x == -CUDART_INF_F) return true;
    return hd_rel(a, b) > 0.f;
}

// The variable-to-factor values of an edge of a high-degree variable (vs: its edge_vs,
// mo: the edge's stored entries), relative to the edge's largest state.
template <int K>
__device__ __forceinline__ void hd_v2f(const DevGraph &G, int vs, const float (&mo)[K], float (&v)[K]) {
    float2 d[K];
    int arg = 0;
#pragma unroll
    for (int x = 0; x < K; ++x) {
        d[x] = hd_pair(G, vs, x, mo[x]);
        if (x > 0 && hd_gt(d[x], d[arg])) arg = x;
    }
    float2 mx = d[0];
#pragma unroll
    for (int x = 1; x < K; ++x)
        if (x == arg) mx = d[x];
    if (mx.x == -CUDART_INF_F) {
#pragma unroll
        for (int x = 0; x < K; ++x) v[x] = -CUDART_INF_F;
        return;
    }
#pragma unroll
    for (int x = 0; x < K; ++x) v[x] = hd_rel(d[x], mx);
}

// Block-wide float-float sum of v and plain sum of c (a count) in a fixed order; sh holds
// 3 floats per warp.
__device__ __forceinline__ FF block_sum_count(FF v, float &c, float *sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        v = ff_add(v, ff_shfl_down(v, d));
        c += __shfl_down_sync(0xffffffffu, c, d);
    }
    if (lane == 0) {
        sh[3 * warp] = v.hi;
        sh[3 * warp + 1] = v.lo;
        sh[3 * warp + 2] = c;
    }
    __syncthreads();
    FF tot = ff_make(0.f);
    c = 0.f;
    for (int w = 0; w < nw; ++w) {
        tot = ff_add(tot, FF{sh[3 * w], sh[3 * w + 1]});
        c += sh[3 * w + 2];
    }
    __syncthreads();
    return tot;
}

// Variable-to-factor values of one K-state edge. Edges of high-degree variables
// (edge_vs < 0) take the exact leave-one-out values from the variable's totals (hd_pair);
// all others use b - m, or the explicit sum when an entry needs it.
template <int K>
__device__ __forceinline__ void gather_v2f(const DevGraph &G, const float *__restrict__ b,
                                           const float *__restrict__ ev, const float *__restrict__ m_old,
                                           int vs, int es, const float (&mo)[K], float (&v)[K]) {
    if (vs < 0) {
        hd_v2f<K>(G, vs, mo, v);
        return;
    }
    bool exact = false;
#pragma unroll
    for (int x = 0; x < K; ++x) exact |= needs_exact(mo[x]);
    if (exact) {
        v2f_slow_edge(G, ev, m_old, vs, es, K, v);
        return;
    }
    load_n<K>(v, b + vs);
#pragma unroll
    for (int x = 0; x < K; ++x) v[x] -= mo[x];
}

// ---- log-sum-exp helpers -------------------------------------------------------------


// T > 0 logical factors: the closed forms chain several exp / log evaluations per edge;
// in FP32 their rounding errors are biased, which long runs on logical-factor graphs
// amplify. They are therefore evaluated in FP64 from the FP32 inputs (the outputs are
// rounded once to FP32). Sums of softplus terms s(x_j / T) are kept as logarithms,
// log A = LSE_j log s(x_j / T), so that very negative log-odds do not underflow.

// log(s(u)), s(u) = log(1 + e^u)
__device__ __forceinline__ double log_softplus_d(double u) {
    if (u < -30.0) return u + log1p(-0.5 * exp(u));
    if (u > 0.0) return log(u + log1p(exp(-u)));
    return log(log1p(exp(u)));
}

__device__ __forceinline__ double lse2_d(double a, double b) {
    const double mx = fmax(a, b);
    if (mx == -CUDART_INF || mx == CUDART_INF) return mx;
    return mx + log1p(exp(fmin(a, b) - mx));
}

// log(e^a - 1) from la = log a
__device__ __forceinline__ double log_expm1_from_log_d(double la) {
    if (la == -CUDART_INF) return -CUDART_INF;
    if (la == CUDART_INF) return CUDART_INF;
    if (la > 0.0) {
        const double a = exp(la);
        return a + log(-expm1(-a));
    }
    if (la > -700.0) {
        const double a = exp(la);
        return la + log(expm1(a) / a);
    }
    return la;
}

// -log(1 - e^{-a}) from la = log a
__device__ __forceinline__ double neg_log_1mexp_from_log_d(double la) {
    if (la == CUDART_INF) return 0.0;
    if (la > 0.0) return -log(-expm1(-exp(la)));
    if (la > -700.0) {
        const double a = exp(la);
        return -la - log(-expm1(-a) / a);
    }
    return -la;
}

// OR update to parent i (T > 0): la = log of the leave-one-out softplus sum (units of
// T), xc = child log-odds.
__device__ __forceinline__ float or_parent_soft(double la, float xc_f, double T) {
    const double xc = xc_f;
    if (la == -CUDART_INF) return xc_f;
    const double y = xc + T * log_expm1_from_log_d(la);
    if (y >= 0.0) return (float)(T * neg_log_1mexp_from_log_d(la) - T * log1p(exp(-y / T)));
    return (float)(xc + T * exp(la) - T * log1p(exp(y / T)));
}

// OR update to parent i (T = 0): S = leave-one-out sum of max(x_j, 0), M = leave-one-out max.
__device__ __forceinline__ float or_parent_max(float S, float M, float xc) {
    float mn = M < 0.f ? M : 0.f;
    float z = xc + S + mn;
    return (z >= 0.f) ? -mn : xc + S;
}

// XOR (parity) factors: the parents and the child have even parity, and a member's
// message depends on all the others alike. With log-odds a_j = x_j / T of the others,
// the product rule of parity checks gives D = prod tanh(-a_j / 2) and the log-odds
// T log((1 - D) / (1 + D)). The magnitude is carried as l_j = log u_j,
// u_j = -log tanh(|a_j| / 2) = log1p(2 / expm1(|a_j|)) (log 2 - |a_j| beyond 30), and the
// others' LSE lambda of the l_j gives log((1 - |D|) / (1 + |D|)) =
// log(-expm1(-e^lambda)) - log1p(e^-e^lambda) (lambda - log 2 once e^lambda < 1e-9); the
// sign is the parity of the others' positive log-odds. T = 0: the others' smallest |x|,
// positive when an odd number of them is positive. FP64 at T > 0, as the OR / AND forms.
__device__ __forceinline__ double xor_log_u(double a) {
    a = fabs(a);
    if (a == 0.0) return CUDART_INF;
    if (isinf(a)) return -CUDART_INF;
    if (a > 30.0) return 0.6931471805599453 - a;
    return log(log1p(2.0 / expm1(a)));
}

// XOR output (T > 0) from the others' LSE lambda and their parity.
__device__ __forceinline__ float xor_out_soft(double lam, bool odd, double T) {
    double r;
    if (lam == CUDART_INF) r = 0.0;
    else if (lam == -CUDART_INF) r = -CUDART_INF;
    else if (lam < -20.7) r = lam - 0.6931471805599453;
    else {
        const double u = exp(lam);
        r = log(-expm1(-u)) - log1p(exp(-u));
    }
    return (float)(T * (odd ? -r : r));
}

__device__ __forceinline__ float xor_out_max(float mn, bool odd) { return odd ? mn : -mn; }

__device__ __forceinline__ float log_odds(float a0, float a1) {
    return (a0 == kNegInf && a1 == kNegInf) ? 0.f : a1 - a0;
}

// ---- message epilogue: normalise, damp, normalise ------------------------------------

template <int K>
__device__ __forceinline__ void normalise_k(float (&t)[K], uint32_t *flags) {
    float mx = kNegInf;
#pragma unroll
    for (int x = 0; x < K; ++x)
        if (t[x] > mx) mx = t[x];
    if (mx == kNegInf) {
#pragma unroll
        for (int x = 0; x < K; ++x) t[x] = 0.f;
        atomicOr(flags, kFlagContradiction);
        return;
    }
#pragma unroll
    for (int x = 0; x < K; ++x) t[x] -= mx;
}

template <int K>
__device__ __forceinline__ void finish_k(float (&t)[K], const float (&mo)[K], float damping,
                                         uint32_t *flags) {
    normalise_k<K>(t, flags);
    if (damping != 0.f) {
        const float w = 1.f - damping;
#pragma unroll
        for (int x = 0; x < K; ++x) t[x] = damping * mo[x] + w * t[x];
    }
    normalise_k<K>(t, flags);
}

__device__ __forceinline__ void normalise_rt(float *t, int K, uint32_t *flags) {
    float mx = kNegInf;
    for (int x = 0; x < K; ++x)
        if (t[x] > mx) mx = t[x];
    if (mx == kNegInf) {
        for (int x = 0; x < K; ++x) t[x] = 0.f;
        atomicOr(flags, kFlagContradiction);
        return;
    }
    for (int x = 0; x < K; ++x) t[x] -= mx;
}

// ---- LSE_T over a row of K values ---------------------------------------------------

template <int K, bool MAXP>
__device__ __forceinline__ float lse_row(const float (&z)[K], float T, float invT) {
    float mx = kNegInf;
#pragma unroll
    for (int y = 0; y < K; ++y) mx = fmaxf(mx, z[y]);
    if (MAXP || mx == kNegInf) return mx;
    if constexpr (K == 2) {
        // log(1 + e^-d), d >= 0, with the SFU exp2 / log2 (absolute error below 3e-7)
        return mx + T * __logf(1.f + __expf((fminf(z[0], z[1]) - mx) * invT));
    } else {
        float s = 0.f;
#pragma unroll
        for (int y = 0; y < K; ++y) s += expf((z[y] - mx) * invT);
        return mx + T * logf(s);
    }
}

// Multi-sample launches (pgm_run_bp_multi on graphs without the joint log-ratio path;
// the kernels' MS instantiations): gridDim.y samples share the index arrays; a block
// works on sample blockIdx.y, whose
// messages, beliefs, evidence and log-potentials lie at the DevGraph strides (0 for an
// ordinary launch) and whose scratch (exact leave-one-out sums, belief residuals) is the
// sample's slice.
__device__ __forceinline__ int64_t sample_select(DevGraph &G) {
    const int64_t smp = blockIdx.y;
    if (smp != 0) {
        if (G.hd_b) G.hd_b += smp * 4 * G.s_vs;
        if (G.b_lo) G.b_lo += smp * G.s_vs;
    }
    return smp;
}

// A batch member whose early exit has frozen it: the factor pass leaves its messages
// alone (a block, or a chunk of the persistent kernel, lies in one member's group).
__device__ __forceinline__ bool member_frozen(const DevGraph &G, int member) {
    return G.frozen != nullptr && __ldg(G.frozen + member) != 0;
}

// A batch run with parameters per member (pgm_run_bp_batch): the member's T, 1 / T and
// damping replace the launch's, and the launch of the other kind (max-product or not)
// skips it. Also true for a frozen member.
template <bool MAXP>
__device__ __forceinline__ bool member_skip(const DevGraph &G, int member, float &T, float &invT, float &damping) {
    if (member_frozen(G, member)) return true;
    if (G.mem_prm != nullptr) {
        const float4 p = __ldg(reinterpret_cast<const float4 *>(G.mem_prm) + member);
        if ((p.x == 0.f) != MAXP) return true;
        T = p.x;
        invT = p.y;
        damping = p.z;
    }
    return false;
}

}  // namespace
}  // namespace pgm
