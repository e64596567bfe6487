// Variable pass and factor pass of dense K-state pairwise groups (K = 4, 8, 16) in one kernel,
// for variables with at most 4 factors, all of one group (grids, chains, lattices).
//
// Method: one flooding iteration of PGMax's damped updates (arXiv 2202.04110, Sec. 3; dense
// pairwise enumeration factors, Sec. 5.2). A message from factor to variable depends on one
// variable-to-factor value, so an iteration can be computed source by source: the lanes of a
// variable sum its beliefs (the arithmetic of k_var_group) and then form the message that
// leaves each of its edges (the arithmetic of pair_direction, lane by lane), so the messages
// are bitwise those of the two passes.
//
// Why: the two passes moved 18 K floats per variable and iteration, 13 K here (the beliefs stay
// in registers), and paid two launch boundaries. What bounded the factor pass was not its
// arithmetic but the L1: a thread that loads its own 4 K-byte rows touches 32 lines with every
// 16-byte load of a warp, one line per cycle, and reads the whole table for every message.
// Here K / 4 lanes share a variable, four states each: a warp's load covers whole rows, and a
// lane reads the four targets' part of the table, once for two edges of the same side. A block
// loads its indices and table before it waits for the previous launch.
// Measured against the two passes it replaces (GB300, T = 1, whole calls, us per iteration): K =
// 16 on 181 x 181 17.9 -> 9.1; K = 8 on 178 x 178 9.3 -> 5.5; K = 4 on 64 x 64 6.0 -> 3.3 (two
// launches' latency -> one); per launch on 128 uneven grids K = 16 (662,000 variables) 60 + 222
// -> 160 us, K = 8 (800,000) 43 + 88 -> 93, K = 4 (672,000) 28 + 46 -> 48. What bounds it now: the
// L1's data path (wavefronts 70 to 75 % of its rate) and issue slots (49 % at K = 4, 64 % at K = 16);
// more resident blocks win against fewer spills (K = 16: 2, 3, 4 blocks of 256 per SM 232, 183,
// 171 us, when the kernel had a second round that no plan reached; without it 160). Edges with entries
// that are -inf, large or NaN, and tables of range above 60 T, go to team_rare.
#include <cstdint>

#include "pair_math.cuh"

namespace pgm {
namespace {

template <int L>
__device__ __forceinline__ float team_max(float v) {
#pragma unroll
    for (int d = L / 2; d > 0; d >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, d, L));
    return v;
}
// Subtracts the team's maximum and returns it.
template <int L>
__device__ __forceinline__ float team_normalise(F2 (&t)[2]) {
    const float mx = team_max<L>(f2_max<4>(t));
    const F2 n = f2(-mx, -mx);
    t[0] = f2_add(t[0], n);
    t[1] = f2_add(t[1], n);
    return mx;
}
// Four floats; AL: 16-byte aligned.
template <bool AL>
__device__ __forceinline__ void row_load(float (&d)[4], const float *p) {
    if constexpr (AL) {
        const float4 q = __ldg(reinterpret_cast<const float4 *>(p));
        d[0] = q.x, d[1] = q.y, d[2] = q.z, d[3] = q.w;
    } else {
        load_n<4>(d, p);
    }
}

// A team's variable: its incoming edges (es_base where there is none) and their number.
struct TeamVar {
    int v, deg, es[4];
};
__device__ __forceinline__ TeamVar team_var(const DevGraph &G, const int32_t *list, int pos, bool valid, int es_base) {
    TeamVar t;
    t.v = list ? __ldg(list + pos) : pos;
    const int k0 = __ldg(G.vin_off + t.v);
    t.deg = valid ? __ldg(G.vin_off + t.v + 1) - k0 : 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) t.es[i] = i < t.deg ? __ldg(G.vin_es + k0 + i) : es_base;
    return t;
}

// The edges that team_edges leaves out (bits of mask, the same for the team; every lane of the warp
// calls): all of them with a sum-product table of range above 60 T, else those whose stored entries
// are -inf, large or NaN, or that met a maximum of -inf. The variable-to-factor values of an edge with
// such entries are the explicit sums without its own message (v2f_slow_edge's), of another the beliefs
// less the message, and each target's sum runs over the table's entries (lse_row): the operations of
// pair_dir_rare and of the two passes' entry form, lane by lane, so the same bits. Out of line: its
// registers are not the main path's. us per iteration on 181 x 181 by the two passes, by one thread
// per edge, which this replaces, and so: T = 0.02 (a range of 100 T and more) K = 4 8.1, 19.6, 8.3, K = 8
// 13.5, 21.2, 13.0, K = 16 35.3, 45.0, 29.3; max-product with messages above 128 K = 4 16.8, 25.9, 8.9, K =
// 16 68, 91, 21.6. What bounds it: the accurate exponentials (K^2 per edge) and the edges one after
// the other.
template <int K, bool MAXP>
__device__ __noinline__ void team_rare(const DevGraph &G, const float *tab, const float *ev, const float *m_old,
                                       float *m_new, const TeamVar &t, int l, int es_base, float *xs, unsigned mask,
                                       float T, float invT, float damping) {
    constexpr int L = K / 4;
    mask &= (1u << t.deg) - 1u;  // (a maximum of -inf marks edges that are not there, too)
    const float *e = ev + __ldg(G.vs_off + t.v) + 4 * l;
    // beliefs relative to the best state (the largest rounded sum, lowest state on ties). The messages
    // are read again where they are used: held, they would spill
    unsigned odd = 0;
    float b[4];
    {
        FF sum[4];
        float e4[4], mx = kNegInf;
        int arg = 4 * l;
        load_n<4>(e4, e);
#pragma unroll
        for (int x = 0; x < 4; ++x) sum[x] = ff_make(e4[x]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i < t.deg) {
                float q[4];
                load_n<4>(q, m_old + t.es[i] + 4 * l);
                if (needs_exact(q[0]) | needs_exact(q[1]) | needs_exact(q[2]) | needs_exact(q[3])) odd |= 1u << i;
#pragma unroll
                for (int x = 0; x < 4; ++x) sum[x] = ff_add(sum[x], q[x]);
            }
        FF best = sum[0];
#pragma unroll
        for (int x = 0; x < 4; ++x)
            if (sum[x].hi + sum[x].lo > mx) {
                mx = sum[x].hi + sum[x].lo;
                arg = 4 * l + x;
                best = sum[x];
            }
#pragma unroll
        for (int d = L / 2; d > 0; d >>= 1) {
            odd |= __shfl_xor_sync(0xffffffffu, odd, d, L);
            const float ov = __shfl_xor_sync(0xffffffffu, mx, d, L), oh = __shfl_xor_sync(0xffffffffu, best.hi, d, L),
                        ol = __shfl_xor_sync(0xffffffffu, best.lo, d, L);
            const int oi = __shfl_xor_sync(0xffffffffu, arg, d, L);
            if (ov > mx || (ov == mx && oi < arg)) {
                mx = ov;
                arg = oi;
                best = FF{oh, ol};
            }
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) b[x] = best.hi == kNegInf ? kNegInf : 4 * l + x == arg ? 0.f : ff_diff(sum[x], best);
    }
    const float w = 1.f - damping;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool mine = (mask >> i) & 1;
        if (!__any_sync(0xffffffffu, mine)) continue;
        const int side = ((t.es[i] - es_base) / K) & 1, es_t = side ? t.es[i] - K : t.es[i] + K;
        F2 mo[2] = {f2(0.f, 0.f), f2(0.f, 0.f)};
        float v[4] = {0.f, 0.f, 0.f, 0.f};
        if (mine) {
            f2_load<4>(mo, m_old + es_t + 4 * l);
            if ((odd >> i) & 1) {  // the explicit sums
                float q[4];
                FF s[4];
                load_n<4>(q, e);
#pragma unroll
                for (int x = 0; x < 4; ++x) s[x] = ff_make(q[x]);
                for (int k = 0; k < t.deg; ++k)
                    if (k != i) {
                        load_n<4>(q, m_old + t.es[k] + 4 * l);
#pragma unroll
                        for (int x = 0; x < 4; ++x) s[x] = ff_add(s[x], q[x]);
                    }
#pragma unroll
                for (int x = 0; x < 4; ++x) v[x] = s[x].hi + s[x].lo;
            } else {
                load_n<4>(v, m_old + t.es[i] + 4 * l);
#pragma unroll
                for (int x = 0; x < 4; ++x) v[x] = b[x] - v[x];
            }
        }
        __syncwarp();
#pragma unroll
        for (int x = 0; x < 4; ++x) xs[4 * l + x] = v[x];
        __syncwarp();
        const float *p = tab + (side ? 4 * l * K : 4 * l);  // phi(s, 4 l + j) at p[s ss + j sj]
        const int ss = side ? 1 : K, sj = side ? K : 1;
        float mx[4];
        constexpr int N = K == 4 ? 2 : 1;  // targets at a time: N K values in registers
#pragma unroll
        for (int j = 0; j < 4; j += N) {
            float z[N][K];
#pragma unroll
            for (int s = 0; s < K; ++s) {
                const float v = xs[s];
#pragma unroll
                for (int n = 0; n < N; ++n) z[n][s] = p[s * ss + (j + n) * sj] + v;
            }
#pragma unroll
            for (int n = 0; n < N; ++n) mx[j + n] = lse_row<K, MAXP>(z[n], T, invT);
        }
        // pair_finish
        F2 o[2] = {f2(mx[0], mx[1]), f2(mx[2], mx[3])};
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (team_normalise<L>(o) == kNegInf) {
                if (mine && l == 0) atomicOr(G.flags, kFlagContradiction);
                o[0] = o[1] = f2(0.f, 0.f);
            }
            if (r == 0 && damping != 0.f) {
                o[0] = f2_fma(f2(damping, damping), mo[0], f2_mul(f2(w, w), o[0]));
                o[1] = f2_fma(f2(damping, damping), mo[1], f2_mul(f2(w, w), o[1]));
            }
        }
        if (mine) f2_store<4>(m_new + es_t + 4 * l, o);
    }
}

// The four states of lane l (of a team of K / 4): the beliefs' sums s + evidence and the stored
// messages q, then the message that leaves each edge. Returns the edges (bit i, the same for
// the whole team) that team_rare has to take: stored entries that are -inf, large or NaN, or
// a maximum of -inf on the way (contradictions and their flags are left to it).
template <int K, bool MAXP, bool AL>
__device__ __forceinline__ unsigned team_edges(const TeamVar &t, const float (&e4)[4], const float (&q)[4][4], int l,
                                               int es_base, const float *S0, const float *S1, float tmax, float *xs, int xs_step,
                                               const float *m_old, float *m_new, float T, float invT, float damping) {
    constexpr int L = K / 4;
    const F2 minus1 = f2(-1.f, -1.f);
    F2 qa[4], qb[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        qa[i] = f2(q[i][0], q[i][1]);
        qb[i] = f2(q[i][2], q[i][3]);
    }
    // beliefs relative to the variable's best state (k_var_group, kVarIter): ff_add on two
    // states at a time; a sum that is not finite has lo = 0, set once at the end
    F2 b[2];
    {
        F2 hi[2] = {f2(e4[0], e4[1]), f2(e4[2], e4[3])}, lo[2] = {f2(0.f, 0.f), f2(0.f, 0.f)};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const F2 v = h ? qb[i] : qa[i];
                const F2 s = f2_add(hi[h], v), bp = f2_fma(hi[h], minus1, s);
                const F2 ea = f2_fma(f2_fma(bp, minus1, s), minus1, hi[h]), eb = f2_fma(bp, minus1, v);
                lo[h] = f2_add(lo[h], f2_add(ea, eb));
                hi[h] = s;
            }
        float sh[4], sl[4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 x = f2_get(hi[h]), y = f2_get(lo[h]);
            sh[2 * h] = x.x;
            sh[2 * h + 1] = x.y;
            sl[2 * h] = isfinite(x.x) ? y.x : 0.f;
            sl[2 * h + 1] = isfinite(x.y) ? y.y : 0.f;
        }
        // the best state: the largest rounded sum, lowest state on ties; its sum comes along
        float lmx = kNegInf, bh = sh[0], bl = sl[0];
        int larg = 4 * l;
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const float rs = sh[x] + sl[x];
            if (rs > lmx) {
                lmx = rs;
                larg = 4 * l + x;
                bh = sh[x];
                bl = sl[x];
            }
        }
#pragma unroll
        for (int d = L / 2; d > 0; d >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, lmx, d, L);
            const int oi = __shfl_xor_sync(0xffffffffu, larg, d, L);
            const float oh = __shfl_xor_sync(0xffffffffu, bh, d, L), ol = __shfl_xor_sync(0xffffffffu, bl, d, L);
            if (ov > lmx || (ov == lmx && oi < larg)) {
                lmx = ov;
                larg = oi;
                bh = oh;
                bl = ol;
            }
        }
        float r[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) r[x] = 4 * l + x == larg ? 0.f : (sh[x] - bh) + (sl[x] - bl);  // ff_diff
        if (bh == kNegInf) r[0] = r[1] = r[2] = r[3] = kNegInf;
        b[0] = f2(r[0], r[1]);
        b[1] = f2(r[2], r[3]);
    }
    unsigned rare = 0;
    {
        float big = 0.f, sum = 0.f;  // sum: NaN if an entry is
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            big = fmaxf(big, fmaxf(fmaxf(fabsf(q[i][0]), fabsf(q[i][1])), fmaxf(fabsf(q[i][2]), fabsf(q[i][3]))));
            sum += (q[i][0] + q[i][1]) + (q[i][2] + q[i][3]);
        }
        if (!(big <= kExactThreshold) | (sum != sum))  // seldom: which edges
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (needs_exact(q[i][0]) | needs_exact(q[i][1]) | needs_exact(q[i][2]) | needs_exact(q[i][3])) rare |= 1u << i;
    }
#pragma unroll
    for (int d = L / 2; d > 0; d >>= 1) rare |= __shfl_xor_sync(0xffffffffu, rare, d, L);
    // two edges at a time
#pragma unroll
    for (int p = 0; p < 4; p += 2) {
        if (!__any_sync(0xffffffffu, t.deg > p)) break;
        const int side0 = ((t.es[p] - es_base) / K) & 1, side1 = ((t.es[p + 1] - es_base) / K) & 1;  // the sources' places
        float vmax[2];
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // the source's values or weights, each twice: pairs for two targets
            const F2 v[2] = {f2_fma(qa[p + h], minus1, b[0]), f2_fma(qb[p + h], minus1, b[1])};
            float2 wa = f2_get(v[0]), wb = f2_get(v[1]);
            if constexpr (!MAXP) {
                vmax[h] = team_max<L>(f2_max<4>(v));
                if (vmax[h] == kNegInf) rare |= 1u << (p + h);
                wa = pair_weights(v[0], vmax[h], invT);
                wb = pair_weights(v[1], vmax[h], invT);
            }
            float4 *x = reinterpret_cast<float4 *>(xs + h * xs_step + 8 * l);
            x[0] = make_float4(wa.x, wa.x, wa.y, wa.y);
            x[1] = make_float4(wb.x, wb.x, wb.y, wb.y);
        }
        __syncwarp();
        F2 acc[2][2];
        float mxp[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            acc[h][0] = acc[h][1] = f2(0.f, 0.f);
            mxp[h][0] = mxp[h][1] = mxp[h][2] = mxp[h][3] = kNegInf;
        }
        auto step = [&](int h, const ulonglong2 a, const F2 w) {
            if constexpr (MAXP) {  // pair_max
                const float2 x = f2_get(f2_add(a.x, w)), y = f2_get(f2_add(a.y, w));
                mxp[h][0] = fmaxf(mxp[h][0], x.x);
                mxp[h][1] = fmaxf(mxp[h][1], x.y);
                mxp[h][2] = fmaxf(mxp[h][2], y.x);
                mxp[h][3] = fmaxf(mxp[h][3], y.y);
            } else {  // pair_linear
                acc[h][0] = f2_fma(a.x, w, acc[h][0]);
                acc[h][1] = f2_fma(a.y, w, acc[h][1]);
            }
        };
        const ulonglong2 *S4 = reinterpret_cast<const ulonglong2 *>(side0 ? S1 : S0) + l;  // row s: S4[s L]
        if (__all_sync(0xffffffffu, side0 == side1 || p + 1 >= t.deg)) {  // one reading of the table for both
#pragma unroll
            for (int c = 0; c < K / 4; ++c)
#pragma unroll
                for (int i = 2; i >= 0; i -= 2) {  // sources 4 c + 3, 4 c + 2, then 4 c + 1, 4 c
                    const ulonglong2 w0 = *reinterpret_cast<const ulonglong2 *>(xs + 2 * (4 * c + i));
                    const ulonglong2 w1 = *reinterpret_cast<const ulonglong2 *>(xs + xs_step + 2 * (4 * c + i));
                    const ulonglong2 hi = S4[(4 * c + i + 1) * L], lo = S4[(4 * c + i) * L];
                    step(0, hi, w0.y);
                    step(1, hi, w1.y);
                    step(0, lo, w0.x);
                    step(1, lo, w1.x);
                }
        } else {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (h == 1) S4 = reinterpret_cast<const ulonglong2 *>(side1 ? S1 : S0) + l;
#pragma unroll
                for (int c = 0; c < K / 4; ++c)
#pragma unroll
                    for (int i = 2; i >= 0; i -= 2) {
                        const ulonglong2 w = *reinterpret_cast<const ulonglong2 *>(xs + h * xs_step + 2 * (4 * c + i));
                        step(h, S4[(4 * c + i + 1) * L], w.y);
                        step(h, S4[(4 * c + i) * L], w.x);
                    }
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int es_t = (h ? side1 : side0) ? t.es[p + h] - K : t.es[p + h] + K;
            const bool have = p + h < t.deg;
            float mo4[4] = {0.f, 0.f, 0.f, 0.f};
            if (have) row_load<AL>(mo4, m_old + es_t + 4 * l);
            const F2 mo[2] = {f2(mo4[0], mo4[1]), f2(mo4[2], mo4[3])};
            F2 o[2];
            bool none = false;
            if constexpr (MAXP) {
                o[0] = f2(mxp[h][0], mxp[h][1]);
                o[1] = f2(mxp[h][2], mxp[h][3]);
            } else {
                o[0] = pair_log(acc[h][0], T, vmax[h], tmax);
                o[1] = pair_log(acc[h][1], T, vmax[h], tmax);
            }
            // pair_finish
            none = team_normalise<L>(o) == kNegInf;
            if (damping != 0.f) {
                const float w = 1.f - damping;
                o[0] = f2_fma(f2(damping, damping), mo[0], f2_mul(f2(w, w), o[0]));
                o[1] = f2_fma(f2(damping, damping), mo[1], f2_mul(f2(w, w), o[1]));
            }
            none |= team_normalise<L>(o) == kNegInf;
            if (none) rare |= 1u << (p + h);
            if (have && !((rare >> (p + h)) & 1)) {
                if constexpr (AL) {
                    ulonglong2 x;
                    x.x = o[0];
                    x.y = o[1];
                    *reinterpret_cast<ulonglong2 *>(m_new + es_t + 4 * l) = x;
                } else {
                    f2_store<4>(m_new + es_t + 4 * l, o);
                }
            }
        }
    }
    return rare;
}

// NT: threads of a block.
template <int K, bool MAXP, bool MS, int NT>
__global__ void __launch_bounds__(NT, (K == 16 ? 1024 : 1280) / NT)
k_pair_fused(const __grid_constant__ DevGraph G, const FuseBlock *__restrict__ blocks, const int32_t *__restrict__ list,
             const float *__restrict__ pot, const float *__restrict__ ev, const float *__restrict__ m_old,
             float *__restrict__ m_new, float T, float invT, float damping) {
    constexpr int L = K / 4;                  // lanes per variable
    constexpr int kTeams = NT / L;            // the block's variables at most (fuse_plan, capi.cu)
    constexpr int kRow = K == 4 ? 8 : 2 * K + 4;  // a team's exchange row: few bank conflicts between teams
    __shared__ __align__(16) float S0[K * K], S1[K * K];
    __shared__ __align__(16) float xch[2 * kTeams * kRow];
    __shared__ float tab[K * K];
    __shared__ float red[2 * NT / 32];
    if constexpr (MS) {  // multi-sample launches: this block's sample
        const int64_t smp = blockIdx.y;
        pot += smp * G.s_pot;
        ev += smp * G.s_vs;
        m_old += smp * G.s_es;
        m_new += smp * G.s_es;
    }
    // before the previous launch has finished: what is fixed for the run (indices, the table). The
    // table is the caller's, so a run's first launch is an ordinary one (launch_k): nothing of it
    // runs before the caller's work on the stream is done
    const int4 B = __ldg(reinterpret_cast<const int4 *>(blocks + blockIdx.x));  // pos, n, es_base, pot_base
    const int es_base = B.z, n = B.y;
    const int l = threadIdx.x & (L - 1), team = threadIdx.x / L;
    float *xs = xch + team * kRow;
    TeamVar t = team_var(G, list, B.x + (team < n ? team : 0), team < n, es_base);
    int vs = __ldg(G.vs_off + t.v);
    pair_tables_load<K, NT>(pot + B.w, tab);
    pdl_wait();  // messages of the previous launch
    __syncthreads();
    if (member_skip<MAXP>(G, __ldg(&blocks[blockIdx.x].member), T, invT, damping)) return;  // the whole block
    const bool lin = pair_tables_make<K, MAXP, NT>(tab, S0, S1, red, invT);
    if (!MAXP && !lin) {
        team_rare<K, MAXP>(G, tab, ev, m_old, m_new, t, l, es_base, xs, (1u << t.deg) - 1u, T, invT, damping);
        return;
    }
    pdl_launch_if_small();  // the next launch may be scheduled (it waits likewise)
    // rows are 16-byte aligned or not for the whole run (K is a multiple of 4)
    const bool al = ((reinterpret_cast<uintptr_t>(m_old + es_base) | reinterpret_cast<uintptr_t>(m_new + es_base) |
                      reinterpret_cast<uintptr_t>(ev + vs)) & 15u) == 0;
    const bool all_al = __syncthreads_and(al);
    float e4[4], q[4][4];
    unsigned rare;
    if (all_al) {
        row_load<true>(e4, ev + vs + 4 * l);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (i < t.deg) row_load<true>(q[i], m_old + t.es[i] + 4 * l);
            else q[i][0] = q[i][1] = q[i][2] = q[i][3] = 0.f;  // adds exactly nothing
        }
        rare = team_edges<K, MAXP, true>(t, e4, q, l, es_base, S0, S1, red[0], xs, kTeams * kRow, m_old, m_new, T, invT,
                                         damping);
    } else {
        row_load<false>(e4, ev + vs + 4 * l);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (i < t.deg) row_load<false>(q[i], m_old + t.es[i] + 4 * l);
            else q[i][0] = q[i][1] = q[i][2] = q[i][3] = 0.f;
        }
        rare = team_edges<K, MAXP, false>(t, e4, q, l, es_base, S0, S1, red[0], xs, kTeams * kRow, m_old, m_new, T, invT,
                                          damping);
    }
    if (__any_sync(0xffffffffu, rare != 0))
        team_rare<K, MAXP>(G, tab, ev, m_old, m_new, t, l, es_base, xs, rare, T, invT, damping);
    if (!pdl_small()) pdl_launch_dependents();
}

template <int K, bool MAXP, bool MS>
cudaError_t launch_k(const DevGraph &G, const FactorLaunch &L, const float *pot, const float *ev, const float *m_old,
                     float *m_new, float T, float damping, int S, bool later, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)L.fuse_blocks, (unsigned)S);
    cfg.blockDim = dim3((unsigned)L.fuse_threads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = later ? 1 : 0;  // a run's first launch starts after the caller's work, which may write pot
    auto kern = L.fuse_threads == 128 ? k_pair_fused<K, MAXP, MS, 128> : k_pair_fused<K, MAXP, MS, 256>;
    return cudaLaunchKernelEx(&cfg, kern, G, L.fuse, L.fuse_list, pot, ev, m_old, m_new, T, MAXP ? 0.f : 1.f / T,
                              damping);
}

template <int K>
cudaError_t launch_pick(const DevGraph &G, const FactorLaunch &L, const float *pot, const float *ev, const float *m_old,
                        float *m_new, float T, float damping, int S, bool later, cudaStream_t s) {
    if (S > 1)
        return T == 0.f ? launch_k<K, true, true>(G, L, pot, ev, m_old, m_new, T, damping, S, later, s)
                        : launch_k<K, false, true>(G, L, pot, ev, m_old, m_new, T, damping, S, later, s);
    return T == 0.f ? launch_k<K, true, false>(G, L, pot, ev, m_old, m_new, T, damping, 1, later, s)
                    : launch_k<K, false, false>(G, L, pot, ev, m_old, m_new, T, damping, 1, later, s);
}

}  // namespace

cudaError_t launch_pair_fused(const DevGraph &G, const FactorLaunch &L, const float *pot, const float *ev,
                              const float *m_old, float *m_new, float T, float damping, int S, bool later, cudaStream_t s) {
    switch (L.variant) {
        case kPairF4: return launch_pick<4>(G, L, pot, ev, m_old, m_new, T, damping, S, later, s);
        case kPairF8: return launch_pick<8>(G, L, pot, ev, m_old, m_new, T, damping, S, later, s);
        case kPairF16: return launch_pick<16>(G, L, pot, ev, m_old, m_new, T, damping, S, later, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace pgm
