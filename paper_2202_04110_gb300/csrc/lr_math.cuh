// Arithmetic of the log-ratio form of an iteration (binary pairwise graphs), shared by the
// multi-launch kernels (kernels.cu) and the one-launch runs (lr_run.cu): one definition, so
// that every form gives the same bits.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>
#include <math_constants.h>

#include "pgm_internal.h"

namespace pgm {
namespace {

constexpr uint32_t kFlagContradiction = 1u;
constexpr uint32_t kFlagNaN = 2u;

#define kNegInf (-CUDART_INF_F)

// ---- compensated (float-float) sums ----------------------------------------------------
// A value hi + lo with |lo| << |hi|: TwoSum keeps the rounding error of every addition,
// giving about 44 significant bits at FP32 speed (FP64 is a small fraction of the FP32
// rate on this GPU). Infinite sums keep lo = 0.
struct FF {
    float hi, lo;
};

__device__ __forceinline__ FF ff_make(float v) { return FF{v, 0.f}; }

__device__ __forceinline__ FF ff_add(FF a, float v) {
    const float s = a.hi + v;
    if (!isfinite(s)) return FF{s, 0.f};
    const float bp = s - a.hi;
    const float e = (a.hi - (s - bp)) + (v - bp);
    return FF{s, a.lo + e};
}

__device__ __forceinline__ FF ff_add(FF a, FF b) {
    FF r = ff_add(a, b.hi);
    if (!isfinite(r.hi)) return r;
    r.lo += b.lo;
    return r;
}

__device__ __forceinline__ FF ff_shfl_down(FF v, int d) {
    return FF{__shfl_down_sync(0xffffffffu, v.hi, d), __shfl_down_sync(0xffffffffu, v.lo, d)};
}

// a - b for float-float values, rounded to FP32 (exact up to that rounding when a and b
// are close). -inf - finite = -inf.
__device__ __forceinline__ float ff_diff(FF a, FF b) {
    if (!isfinite(a.hi) || !isfinite(b.hi)) return a.hi - b.hi;
    return (a.hi - b.hi) + (a.lo - b.lo);
}

constexpr uint32_t kLamBothNegInf = 0x7fc00001u;


__device__ __forceinline__ float2 lr_decode(float d) {
    return d > 0.f ? make_float2(-d, 0.f) : make_float2(0.f, d);
}

__device__ __forceinline__ float lr_encode(float m0, float m1) { return m1 - m0; }

__device__ __forceinline__ float2 lam_decode(float l) {
    if (__float_as_uint(l) == kLamBothNegInf) return make_float2(kNegInf, kNegInf);
    return lr_decode(l);
}

__device__ __forceinline__ float lam_encode(FF l0, FF l1) {
    if (l0.hi == kNegInf && l1.hi == kNegInf) return __uint_as_float(kLamBothNegInf);
    return ff_diff(l1, l0);
}

// ff_add for operands known to be finite: an overflow shows as a non-finite result,
// which the caller tests.
__device__ __forceinline__ FF ff_add_nc(FF a, float v) {
    const float s = a.hi + v;
    const float bp = s - a.hi;
    const float e = (a.hi - (s - bp)) + (v - bp);
    return FF{s, a.lo + e};
}

// Variable-to-factor log-ratios of one variable: the leave-one-out value of edge k is
//   lam_k = l_k(1) - l_k(0) = (e(1) - e(0)) + sum over j != k of d_j = D - d_k,
// linear in the stored log-ratios, with D = (e(1) - e(0)) + sum_j d_j kept float-float
// (the evidence difference exactly, by TwoSum), so lam_k is exact up to its final
// rounding. lr_var_slow handles a variable with an infinite evidence entry or message
// (hard constraints) by the per-state explicit sums l_k(x) instead (d = 0 of an unused
// slot decodes to (0, 0) and adds nothing there either).
__device__ __noinline__ void lr_var_slow(float2 e, const float *dk, const int *pos, int n, float *lam) {
    for (int k = 0; k < n; ++k) {
        FF l0 = ff_make(e.x), l1 = ff_make(e.y);
        for (int j = 0; j < n; ++j) {
            if (j == k) continue;
            const float2 q = lr_decode(dk[j]);
            l0 = ff_add(l0, q.x);
            l1 = ff_add(l1, q.y);
        }
        lam[pos[k]] = lam_encode(l0, l1);
    }
}

constexpr uint32_t kDvSlow = 0x7fc00002u;

__device__ __forceinline__ float lr_lam_from_D(float2 D, float dk) {
    const FF l = ff_add_nc(FF{D.x, D.y}, -dk);
    return l.hi + l.lo;
}

// LSE_T of two values for the log-ratio factor pass:
//   max + T ln(1 + e^((min - max) / T)) = max + (T ln 2) log2(1 + 2^((min - max) k)),
// k = log2(e) / T, on the SFU's base-2 exponential and logarithm (flush-to-zero forms;
// the argument of log2 lies in [1, 2], the result's absolute error is below 3e-7 T).
__device__ __forceinline__ float lse2_fast(float a, float b, float k, float Tln2) {
    const float mx = fmaxf(a, b), mn = fminf(a, b);
    float p, l;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(p) : "f"((mn - mx) * k));
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(1.f + p));
    return fmaf(Tln2, l, mx);
}

// The same with the -inf case (both values -inf) returning -inf.
template <bool MAXP>
__device__ __forceinline__ float lse2_lr(float a, float b, float k, float Tln2) {
    if constexpr (MAXP) return fmaxf(a, b);
    if (fmaxf(a, b) == kNegInf) return kNegInf;
    return lse2_fast(a, b, k, Tln2);
}

template <bool MAXP>
__device__ __forceinline__ float lse2_fast_t(float a, float b, float k, float Tln2) {
    if constexpr (MAXP) return fmaxf(a, b);
    else return lse2_fast(a, b, k, Tln2);
}

// The normalise-damp-normalise epilogue (finish_k) in log-ratio form: from the factor's
// values a(0), a(1) and the stored message d_old, the new message's log-ratio. The
// decoded pairs are those finish_k sees, so the result is the one it would store; a
// contradiction (both entries -inf) gives zeros and the flag.
__device__ __forceinline__ float lr_finish(float a0, float a1, float d_old, float damping, uint32_t *flags) {
    float dt;
    if (a0 == kNegInf && a1 == kNegInf) {
        atomicOr(flags, kFlagContradiction);
        dt = 0.f;
    } else {
        dt = a1 - a0;
    }
    if (damping == 0.f) return dt;
    const float2 o = lr_decode(dt), mo = lr_decode(d_old);
    const float w = 1.f - damping;
    const float t0 = damping * mo.x + w * o.x, t1 = damping * mo.y + w * o.y;
    if (t0 == kNegInf && t1 == kNegInf) {
        atomicOr(flags, kFlagContradiction);
        return 0.f;
    }
    return t1 - t0;
}

// One factor's new log-ratio message towards its neighbour `side` with every special case
// handled: a variable-to-factor pair l (from the other neighbour) that is -inf in both
// states, table entries of -inf, an infinite stored message mo, damping 0 (the update of
// finish_k, decoded).
template <bool MAXP>
__device__ __noinline__ float lr_dir_exact(const float *phi, int side, float l, float mo, float k, float Tln2,
                                           float damping, uint32_t *flags) {
    const float2 v = lam_decode(l);
    const int a = side ? 2 : 1;  // table step of the other neighbour's state; 3 - a: of this one's
    const float a0 = lse2_lr<MAXP>(phi[0] + v.x, phi[a] + v.y, k, Tln2);
    const float a1 = lse2_lr<MAXP>(phi[3 - a] + v.x, phi[3] + v.y, k, Tln2);
    return lr_finish(a0, a1, mo, damping, flags);
}

// The segment of global factor g (segments in factor order, segment i starting at
// factor segs[i].edge_base / 2).
__device__ __forceinline__ int lr_seg_of(const EnumSeg *__restrict__ segs, int n_seg, int g) {
    int lo = 0, hi = n_seg - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((__ldg(&segs[mid].edge_base) >> 1) <= g) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// The table of global factor g: its own 4 entries, or the segment's shared table.
__device__ __forceinline__ float4 lr_table(const EnumSeg *__restrict__ segs, int n_seg,
                                           const float *__restrict__ pot, int g) {
    const EnumSeg *S = segs + lr_seg_of(segs, n_seg, g);
    const int shared = __ldg(&S->shared);
    const float *t = pot + __ldg(&S->pot_base) + (shared ? 0 : (size_t)4 * (g - (__ldg(&S->edge_base) >> 1)));
    if ((reinterpret_cast<uintptr_t>(t) & 15u) == 0)
        return shared ? __ldg(reinterpret_cast<const float4 *>(t)) : __ldcs(reinterpret_cast<const float4 *>(t));
    return make_float4(__ldg(t), __ldg(t + 1), __ldg(t + 2), __ldg(t + 3));
}

// sp_T(x) = T ln(1 + e^(x / T)) = max(x, 0) + (T ln 2) log2(1 + 2^(-|x| k)), k = log2(e) / T,
// on the SFU's base-2 exponential and logarithm (flush-to-zero forms; the argument of
// log2 lies in [1, 2], absolute error below 3e-7 T); max(x, 0) for T = 0.
template <bool MAXP>
__device__ __forceinline__ float softplus_t(float x, float k, float Tln2) {
    if constexpr (MAXP) {
        return fmaxf(x, 0.f);
    } else {
        float p, l;
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(p) : "f"(-fabsf(x) * k));
        asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(1.f + p));
        return fmaf(Tln2, l, fmaxf(x, 0.f));
    }
}

// With the variable-to-factor log-ratio l of one neighbour and the table numbers
// (c = phi(1,0) - phi(0,0), al = phi(1,1) - phi(1,0), be = phi(0,1) - phi(0,0)), LSE_T over that
// neighbour's states gives the other's new log-ratio
//   to neighbour 0: c  + sp_T(al + l1) - sp_T(be + l1),
//   to neighbour 1: be + sp_T(al + c - be + l0) - sp_T(c + l0)   (al + c - be = phi(1,1) - phi(0,1)),
// r + sp_T(p + l) - sp_T(q + l) either way. With o, mo the decoded new and stored messages
// (one entry of each exactly 0), the damped pair t = damping mo + (1 - damping) o has
// log-ratio damping d_old + (1 - damping) dt, since min(x, 0) + max(x, 0) = x; the final
// normalisation does not change it. Every input that needs the guarded arithmetic (a
// non-finite table entry, l = +inf, an infinite stored message, damping 0 against an
// infinite stored message) makes the result non-finite; that and a NaN l (the
// contradiction pattern) send the message to lr_dir_exact with its table. (l = -inf gives
// the finite limit r + sp_T(-inf) - sp_T(-inf) = r.) Each direction decides for itself:
// it reads nothing of the other, so the blocks of a one-launch run can compute the two
// directions of a factor apart.
template <bool MAXP>
__device__ __forceinline__ float lr_dir(float r, float p, float q, float l, float mo, float k, float Tln2,
                                        float damping, float w) {
    const float dt = r + softplus_t<MAXP>(p + l, k, Tln2) - softplus_t<MAXP>(q + l, k, Tln2);
    return fmaf(damping, mo, w * dt);
}
__device__ __forceinline__ bool lr_dir_rare(float dn, float l) { return !(isfinite(dn) && l == l); }

// Both messages of a factor of which at least one is rare: one call, so that the callers' common
// path keeps nothing across two.
template <bool MAXP>
__device__ __noinline__ float2 lr_pair_exact(float4 t, float l0, float l1, float mo0, float mo1, float2 dn, float k,
                                             float Tln2, float damping, uint32_t *flags) {
    const float t4[4] = {t.x, t.y, t.z, t.w};
    if (lr_dir_rare(dn.x, l1)) dn.x = lr_dir_exact<MAXP>(t4, 0, l1, mo0, k, Tln2, damping, flags);
    if (lr_dir_rare(dn.y, l0)) dn.y = lr_dir_exact<MAXP>(t4, 1, l0, mo1, k, Tln2, damping, flags);
    return dn;
}

}  // namespace
}  // namespace pgm
