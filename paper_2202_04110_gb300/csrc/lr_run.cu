// One-launch runs of binary pairwise graphs (every variable binary with at most 4 factors,
// every factor a 2 x 2 table): every iteration of a pgm_run_bp call inside one kernel, the
// messages resident in shared memory from the first iteration to the last.
//
// Method: the log-ratio form of PGMax's damped flooding updates (arXiv 2202.04110, Sec. 3)
// with the arithmetic of lr_math.cuh, item for item that of the multi-launch kernels, so
// messages and flags are bitwise theirs.
//
// Why: the multi-launch run moves 112 bytes per variable and iteration through L2 and pays
// two launch boundaries; on a 1000 x 1000 grid that took 17.4 us per iteration, on grids of
// 10^4 .. 10^5 variables 3 .. 4 us, nearly all of it boundaries. A block here owns a
// contiguous range of Vc variables: their incoming messages d and the variable-to-factor values
// lam (4 slots each) live in its shared memory (32 bytes per variable: 7,250 per SM, 1.1 million on
// 152 SMs; larger graphs keep d and the totals D, 24 bytes, up to 1.47 million),
// factors between two variables of one block are updated in place, and only
// the factors that join two blocks exchange anything: one variable-to-factor value in each
// direction per iteration. Each of the two blocks computes the message to its own variable.
//
// One iteration of a block:
//   1. thread per variable: D = (e(1) - e(0)) + sum of its d (float-float), lam = D - d;
//   2. publish: for every split factor, its lam into the other block's inbox;
//   3. whole factors: thread per factor, both messages in place;
//   4. split factors: wait for the other block's value, one message in place;
// with a block barrier after 1 and after 4. Step 3 runs while the values travel.
// Measured against the multi-launch run (whole calls, GB300): 1000 x 1000, 200 iterations
// 3.65 -> 1.80 ms (8.9 us per iteration), 317 x 241 max-product, 50 iterations 213 -> 87 us,
// 32 evidence sets of 256 x 256, 100 iterations 4.22 -> 2.16 ms. Messages that need the guarded
// arithmetic (towards or from clamped variables, tables with -inf) are done where they are met, each
// three dependent loads away from its table at half the warps of the launches: where records are
// streamed that costs more than the launches from some per cent of such messages on (1000 x 1000, T = 1,
// 10 % of the tables with -inf: 49.6 us per iteration against 30.6). Putting them on a list that all
// threads take up after the loop was measured: 24.7 us there, but 1.80 -> 1.89 ms on finite inputs; dropped.
//
// Inbox words carry their iteration: one 8-byte store holds (value, iteration), and the
// reader polls its own word until the iteration is the one it is in; no fence, flag or
// grid-wide barrier is needed. Two parities suffice: a block can publish iteration t + 2
// only after its own step 4 of t + 1, which waited for the other side's t + 1, which that
// side published after it had finished reading t. Inboxes are cleared in the prologue,
// before the one barrier of all blocks (per sample they exchange with; the launch's).
//   - a cluster of up to 16 blocks (graphs of 701 .. 16,384 variables): the inboxes are in the
//     reader's shared memory, written through distributed shared memory, so a poll is a
//     local read;
//   - a cooperative grid of up to one block per SM (above that): the inboxes are in global
//     memory (L2).
// Every wait is bounded: after LrWait::polls polls a block raises PGM_FLAG_TIMEOUT in the status
// word and the caller's (LrWait::host), stops waiting and runs to its end. (The barrier's words are right
// again by then: every block of a launch arrives, also one that gives up, and the last one to
// arrive resets the count.)
#include <algorithm>
#include <cstdint>
#include <mutex>

#include <cuda_runtime.h>

#include "lr_math.cuh"
#include "pgm_internal.h"

namespace pgm {
namespace {

constexpr uint32_t kFlagTimeout = PGM_FLAG_TIMEOUT;

struct LrRun {
    int32_t V, E;
    const int4 *tab4;       // each variable's incoming edge-states (DevGraph::vin_tab4)
    const int32_t *lr_pos;  // each edge's slot k V + v
    const EnumSeg *segs;
    int n_seg;
    const float *pot, *ev;
    float *msgs, *lam;      // lam: explicit sums of variables with infinite entries, lam_floats per sample
    int64_t pot_stride, ev_stride, msg_stride;  // per sample (pot_stride 0: one table set)
    int64_t lam_stride;                         // (lam_floats)
    uint32_t *flags;
    float k, Tln2, damping;
    int n_iters;
    int nb, Vc;             // blocks per sample, variables per block
    int f_cap, h_cap;       // items per block that the arrays below have room for
    const int2 *off;        // kGrid, one sample: first whole / split item of each block; else null
    int32_t *dir;           // [4 V] per sample: a split slot's item in its block
    unsigned long long *box0, *box1;  // kGrid inboxes of the even / odd iterations
    float4 *rec;            // whole factors' records when not in shared memory
    float4 *hrec;           // split factors' records when not in shared memory
    uint32_t *hdst;         // and the other block's inbox word
    uint32_t *bar;          // launch-wide barrier: arrivals, generation
    LrWait wait;
};

// A wait of this run has run out.
__device__ __noinline__ void wait_failed(const LrRun &A) {
    atomicOr(A.flags, kFlagTimeout);
    if (A.wait.host) {
        *(volatile uint32_t *)A.wait.host = 1u;
        __threadfence_system();
    }
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// The shared::cluster address of the same shared-memory location in block `rank`.
__device__ __forceinline__ uint32_t rank_addr(uint32_t a, uint32_t rank) {
    uint32_t out;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"(a), "r"(rank));
    return out;
}

// (value, iteration) as one 8-byte word.
__device__ __forceinline__ unsigned long long box_word(float v, uint32_t it) {
    return ((unsigned long long)it << 32) | __float_as_uint(v);
}

// All blocks of the launch (co-resident: a cooperative launch), once. The last to arrive
// resets the count and moves the generation on, so the words need no clearing between
// launches.
__device__ __forceinline__ bool grid_barrier_once(uint32_t *bar, uint32_t n_blocks, int limit) {
    bool ok = true;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile uint32_t *gen = bar + 1;
        const uint32_t g0 = *gen;
        __threadfence();
        if (atomicAdd(bar, 1u) == n_blocks - 1) {
            atomicExch(bar, 0u);
            __threadfence();
            atomicAdd(bar + 1, 1u);
        } else {
            int polls = 0;
            while (*gen == g0 && ++polls < limit) __nanosleep(64);
            ok = *gen != g0;
        }
        __threadfence();
    }
    return __syncthreads_and(ok || threadIdx.x != 0);
}

// The message into slot (v, kk) with every special case handled: its factor's table, its side.
template <bool MAXP>
__device__ __noinline__ float run_exact(const LrRun &A, const float *pot, int v0, int s, float l, float mo) {
    const int kk = s / A.Vc, v = v0 + s - kk * A.Vc;
    const int4 t = __ldg(A.tab4 + v);
    const int es = kk == 0 ? t.x : kk == 1 ? t.y : kk == 2 ? t.z : t.w;
    const float4 q = lr_table(A.segs, A.n_seg, pot, es >> 2);
    const float phi[4] = {q.x, q.y, q.z, q.w};
    return lr_dir_exact<MAXP>(phi, (es >> 1) & 1, l, mo, A.k, A.Tln2, A.damping, A.flags);
}

// A clamped variable -- one state's evidence -inf, the other's finite -- whose messages are finite and
// far from overflow has every leave-one-out log-ratio at that infinity; 0: not such a variable.
__device__ __forceinline__ float clamped_ratio(float2 e, float d0, float d1, float d2, float d3) {
    const float big = fmaxf(fmaxf(fabsf(d0), fabsf(d1)), fmaxf(fabsf(d2), fabsf(d3))), sum = d0 + d1 + d2 + d3;
    if (!(big < 1e37f) || sum != sum) return 0.f;
    if (e.x == kNegInf && fabsf(e.y) < 1e37f) return CUDART_INF_F;
    if (e.y == kNegInf && fabsf(e.x) < 1e37f) return kNegInf;
    return 0.f;
}

// A variable whose values do not come out finite: its four lam by the explicit sums, or, clamped, without
// (30 % of the variables clamped, us per iteration, the launches per pass / sums / so: 64 x 64 3.75 / 4.2 /
// 3.8, 317 x 241 8.7 / 5.5 / 4.8, 1000 x 1000 38.7 / 64.8 / 56.4).
__device__ __noinline__ void run_var_slow(float *lam, int lv, int Vc, float2 e, float d0, float d1, float d2, float d3) {
    if (const float inf = clamped_ratio(e, d0, d1, d2, d3); inf != 0.f) {
        lam[lv] = lam[Vc + lv] = lam[2 * Vc + lv] = lam[3 * Vc + lv] = inf;
        return;
    }
    const float dk[4] = {d0, d1, d2, d3};
    const int pos[4] = {lv, Vc + lv, 2 * Vc + lv, 3 * Vc + lv};
    lr_var_slow(e, dk, pos, 4, lam);
}

// A block's explicit sums in global memory, by local slot: 4 Vc a block, so that the last one's, of
// fewer variables, end inside. (Formed where it is used: the streamed forms are at 60 to 64 registers,
// and an index by variable, or a call in the factor loop, cost 3 to 6 % on 32 samples of 256 x 256.)
__device__ __forceinline__ float *run_sums(const LrRun &A, int smp, int v0) {
    return A.lam + (size_t)smp * A.lam_stride + 4 * (size_t)v0;
}

__device__ __forceinline__ bool is_slow(float2 D) { return __float_as_uint(D.x) == kDvSlow; }

// X: how blocks exchange values; RES: the records (and evidence) are in shared memory too,
// else they are streamed from L2 (16 bytes per whole factor and iteration, loaded one item
// ahead; the loads do not depend on the messages, so the block barriers do not delay them).
// A record: three table numbers and the local slots k Vc + (v - v0) of the two messages, 16 bits
// each. LAM: lam is kept per slot, so a factor reads d and lam at the same two offsets; else the
// totals are kept per variable (8 bytes less) and a factor forms lam from them.
template <bool MAXP, int X, bool RES, bool LAM>
__global__ void __launch_bounds__(kLrRunThreads, 1) k_lr_run(const __grid_constant__ LrRun A) {
    extern __shared__ __align__(16) char lr_sm[];
    __shared__ int s_n[2];
    __shared__ int s_abort;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    const int V = A.V, Vc = A.Vc;
    int b, smp;  // block within the sample, sample
    if constexpr (X == kCluster) {
        b = (int)cluster_rank();
        smp = 0;
    } else {
        smp = (int)blockIdx.x / A.nb;
        b = (int)blockIdx.x - smp * A.nb;
    }
    const int v0 = b * Vc, nv = max(0, min(Vc, V - v0));
    const float *pot = A.pot + (size_t)smp * A.pot_stride;
    const float2 *ev = reinterpret_cast<const float2 *>(A.ev + (size_t)smp * A.ev_stride) + v0;
    float *msgs = A.msgs + (size_t)smp * A.msg_stride;
    int32_t *dir = A.dir + (size_t)smp * 4 * V;
    // shared memory: [records, split records,] lam or totals, [evidence,] [inbox,] slots, [addresses]
    char *sp = lr_sm;
    float4 *rec, *hrec;
    uint32_t *hdst;
    float2 *es_sh = nullptr;
    unsigned long long *box = nullptr;
    size_t f_base = 0, h_base = 0;  // this block's first item in the global arrays
    if constexpr (X == kGrid) {
        f_base = A.off ? (size_t)A.off[b].x : (size_t)blockIdx.x * A.f_cap;
        h_base = A.off ? (size_t)A.off[b].y : (size_t)blockIdx.x * A.h_cap;
    } else if (!RES) {
        f_base = (size_t)blockIdx.x * A.f_cap;
    }
    if constexpr (RES) {
        rec = reinterpret_cast<float4 *>(sp);
        sp += 16 * (size_t)A.f_cap;
        hrec = reinterpret_cast<float4 *>(sp);
        sp += 16 * (size_t)A.h_cap;
    } else {
        rec = A.rec + f_base;
        hrec = A.hrec + h_base;
        hdst = A.hdst + h_base;
    }
    float2 *Dv = reinterpret_cast<float2 *>(sp);
    float *lam = reinterpret_cast<float *>(sp);
    sp += (LAM ? 16 : 8) * (size_t)Vc;
    if constexpr (RES) {
        es_sh = reinterpret_cast<float2 *>(sp);
        sp += 8 * (size_t)Vc;
    }
    if constexpr (X == kCluster) {
        box = reinterpret_cast<unsigned long long *>(sp);
        sp += 16 * (size_t)A.h_cap;
    }
    float *d = reinterpret_cast<float *>(sp);
    sp += 16 * (size_t)Vc;
    if constexpr (RES) hdst = reinterpret_cast<uint32_t *>(sp);

    // ---- prologue: slots from msgs, the block's items ----
    if (tid < 2) s_n[tid] = 0;
    if (tid == 0) s_abort = X != kAlone && A.wait.polls == 0;
    __syncthreads();
    for (int l0 = 0; l0 < nv; l0 += nt) {
        const int lv = l0 + tid, v = v0 + lv;
        const int4 t = lv < nv ? __ldg(A.tab4 + v) : make_int4(-1, -1, -1, -1);
        if (RES && lv < nv) es_sh[lv] = __ldg(ev + lv);
        const int es[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bool have = es[q] >= 0;
            float m = 0.f;
            int u = 0, uk = 0;
            if (have) {
                m = lr_encode(__ldcg(msgs + es[q]), __ldcg(msgs + es[q] + 1));
                const int p = __ldg(A.lr_pos + ((es[q] >> 1) ^ 1));  // the factor's other slot
                uk = (p >= V) + (p >= 2 * V) + (p >= 3 * V);
                u = p - uk * V;
            }
            if (lv < nv) d[q * Vc + lv] = m;
            const bool local = X == kAlone || (u >= v0 && u < v0 + nv);
            const int side = (es[q] >> 1) & 1;
            const bool whole = have && local && side == 0, split = have && !local;
            float c = 0.f, al = 0.f, be = 0.f;
            if (whole || split) {
                const float4 tb = lr_table(A.segs, A.n_seg, pot, es[q] >> 2);
                const bool fin = isfinite(tb.x) & isfinite(tb.y) & isfinite(tb.z) & isfinite(tb.w);
                c = fin ? tb.z - tb.x : CUDART_NAN_F;  // as k_lr_params
                al = fin ? tb.w - tb.z : CUDART_NAN_F;
                be = fin ? tb.y - tb.x : CUDART_NAN_F;
            }
            // runs of consecutive variables stay together: coalesced, without bank conflicts
            const unsigned mw = __ballot_sync(0xffffffffu, whole), mh = __ballot_sync(0xffffffffu, split);
            int bw = 0, bh = 0;
            if (lane == 0) {
                if (mw) bw = atomicAdd(&s_n[0], __popc(mw));
                if (mh) bh = atomicAdd(&s_n[1], __popc(mh));
            }
            bw = __shfl_sync(0xffffffffu, bw, 0) + __popc(mw & ((1u << lane) - 1u));
            bh = __shfl_sync(0xffffffffu, bh, 0) + __popc(mh & ((1u << lane) - 1u));
            if (whole)
                rec[bw] = make_float4(c, al, be, __uint_as_float((uint32_t)(q * Vc + lv) | (uint32_t)(uk * Vc + u - v0) << 16));
            if (X != kAlone && split) {
                hrec[bh] = side == 0 ? make_float4(c, al, be, __uint_as_float((uint32_t)(q * Vc + lv)))
                                     : make_float4(be, al + c - be, c, __uint_as_float((uint32_t)(q * Vc + lv)));
                __stcg(dir + (size_t)q * V + v, bh);
            }
        }
    }
    __syncthreads();
    const int nF = s_n[0], nH = X == kAlone ? 0 : s_n[1];
    bool ok = true;
    if constexpr (X == kCluster) {
        for (int h = tid; h < 2 * A.h_cap; h += nt) box[h] = 0;
        cluster_barrier();
    } else if constexpr (X == kGrid) {
        for (int h = tid; h < nH; h += nt) {
            __stcg(A.box0 + h_base + h, 0ull);
            __stcg(A.box1 + h_base + h, 0ull);
        }
        ok = grid_barrier_once(A.bar, gridDim.x, A.wait.polls);
    }
    if (X == kGrid && !ok) {  // (a block that got past the barrier times out in its waits)
        if (tid == 0) wait_failed(A);
        return;
    }
    for (int h = tid; h < nH; h += nt) {  // where each split factor's value goes
        const int s = (int)__float_as_uint(hrec[h].w), q = s / Vc, lv = s - q * Vc;
        const int4 t = __ldg(A.tab4 + v0 + lv);
        const int es = q == 0 ? t.x : q == 1 ? t.y : q == 2 ? t.z : t.w;
        const int p = __ldg(A.lr_pos + ((es >> 1) ^ 1));
        const int u = p - V * ((p >= V) + (p >= 2 * V) + (p >= 3 * V));
        const int ub = u / Vc, at = __ldcg(dir + p);
        if constexpr (X == kCluster) hdst[h] = rank_addr(smem_addr(box + at), (uint32_t)ub);
        else hdst[h] = (uint32_t)((A.off ? A.off[ub].y : (smp * A.nb + ub) * A.h_cap) + at);
    }
    __syncthreads();

    // ---- iterations ----
    const float k = A.k, Tln2 = A.Tln2, damping = A.damping, w = 1.f - damping;
    // a total kept per variable: the local variable of slot s, and lam from the total
    auto var_of = [&](int s) { return s - Vc * ((s >= Vc) + (s >= 2 * Vc) + (s >= 3 * Vc)); };
    auto lam_of = [&](int s, float dk) {
        if constexpr (LAM) return lam[s];
        else {
            const float2 D = Dv[var_of(s)];
            return is_slow(D) ? __ldcg(run_sums(A, smp, v0) + s) : lr_lam_from_D(D, dk);
        }
    };
    // what the thread reads first in steps 1 and 3 is fixed for the run: in registers when the
    // records are streamed (each step would otherwise begin with an L2 latency)
    const float2 e_first = !RES && tid < nv ? __ldg(ev + tid) : make_float2(0.f, 0.f);
    const float4 r_first = !RES && tid < nF ? rec[tid] : make_float4(0.f, 0.f, 0.f, 0.f);
    for (int it = 1; it <= A.n_iters; ++it) {
        // 1. totals
        float2 e_next = e_first;
        for (int lv = tid; lv < nv; lv += nt) {
            const float2 e = RES ? es_sh[lv] : e_next;
            if (!RES && lv + nt < nv) e_next = __ldg(ev + lv + nt);
            const float d0 = d[lv], d1 = d[Vc + lv], d2 = d[2 * Vc + lv], d3 = d[3 * Vc + lv];
            FF D = ff_add_nc(ff_make(e.y), -e.x);
            D = ff_add_nc(D, d0);
            D = ff_add_nc(D, d1);
            D = ff_add_nc(D, d2);
            D = ff_add_nc(D, d3);
            float2 Df = make_float2(D.hi, D.lo);
            const float big = fmaxf(fmaxf(fabsf(d0), fabsf(d1)), fmaxf(fabsf(d2), fabsf(d3)));
            const float l0 = lr_lam_from_D(Df, d0), l1 = lr_lam_from_D(Df, d1), l2 = lr_lam_from_D(Df, d2),
                        l3 = lr_lam_from_D(Df, d3);
            bool slow = false;
            if (!(fabsf(D.hi) + big < 1e38f))  // an infinite entry, NaN, or near overflow
                slow = !(isfinite(e.x) && isfinite(e.y) && isfinite(d0) && isfinite(d1) && isfinite(d2) && isfinite(d3) &&
                         isfinite(l0) && isfinite(l1) && isfinite(l2) && isfinite(l3));
            if (slow) {
                if constexpr (LAM) {
                    run_var_slow(lam, lv, Vc, e, d0, d1, d2, d3);
                } else {
                    run_var_slow(run_sums(A, smp, v0), lv, Vc, e, d0, d1, d2, d3);
                    Dv[lv] = make_float2(__uint_as_float(kDvSlow), 0.f);
                }
            } else if constexpr (LAM) {
                lam[lv] = l0;
                lam[Vc + lv] = l1;
                lam[2 * Vc + lv] = l2;
                lam[3 * Vc + lv] = l3;
            } else {
                Dv[lv] = Df;
            }
        }
        __syncthreads();
        // 2. publish
        if constexpr (X != kAlone) {
            for (int h = tid; h < nH; h += nt) {
                const int s = (int)__float_as_uint(RES ? hrec[h].w : __ldcg(&hrec[h].w));
                const unsigned long long wd = box_word(lam_of(s, LAM ? 0.f : d[s]), (uint32_t)it);
                if constexpr (X == kCluster) {
                    const uint32_t a = hdst[h] + ((it & 1) ? 8u * (uint32_t)A.h_cap : 0u);
                    asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(wd) : "memory");
                } else {
                    unsigned long long *p = ((it & 1) ? A.box1 : A.box0) + (RES ? hdst[h] : __ldcg(hdst + h));
                    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(wd) : "memory");
                }
            }
        }
        // 3. whole factors
        {
            int i = tid;
            float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
            if (RES && i < nF) r = rec[i];
            if (!RES) r = r_first;
            while (i < nF) {
                const int in = i + nt;
                float4 rn = r;
                if (!RES && in < nF) rn = __ldcg(rec + in);
                const uint32_t pk = __float_as_uint(r.w);
                const int s0 = pk & 0xffff, s1 = pk >> 16;
                const float mo0 = d[s0], mo1 = d[s1];
                const float l0 = lam_of(s0, mo0), l1 = lam_of(s1, mo1);
                float n0 = lr_dir<MAXP>(r.x, r.y, r.z, l1, mo0, k, Tln2, damping, w);
                float n1 = lr_dir<MAXP>(r.z, r.y + r.x - r.z, r.x, l0, mo1, k, Tln2, damping, w);
                // (a NaN lam makes a sum-product message NaN by itself)
                if (!(fabsf(n0) + fabsf(n1) < CUDART_INF_F) || (MAXP && !(l0 == l0 && l1 == l1))) {
                    if (lr_dir_rare(n0, l1)) n0 = run_exact<MAXP>(A, pot, v0, s0, l1, mo0);
                    if (lr_dir_rare(n1, l0)) n1 = run_exact<MAXP>(A, pot, v0, s1, l0, mo1);
                }
                d[s0] = n0;
                d[s1] = n1;
                i = in;
                if (RES) {
                    if (i < nF) r = rec[i];
                } else {
                    r = rn;
                }
            }
        }
        // 4. split factors
        if constexpr (X != kAlone) {
            for (int h = tid; h < nH; h += nt) {
                const float4 r = RES ? hrec[h] : __ldcg(hrec + h);
                unsigned long long wd = 0;
                int polls = 0;
                while (true) {
                    if constexpr (X == kCluster) {
                        const uint32_t a = smem_addr(box + h) + ((it & 1) ? 8u * (uint32_t)A.h_cap : 0u);
                        asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(wd) : "r"(a) : "memory");
                    } else {
                        const unsigned long long *p = ((it & 1) ? A.box1 : A.box0) + h_base + h;
                        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(wd) : "l"(p) : "memory");
                    }
                    if ((uint32_t)(wd >> 32) == (uint32_t)it) break;
                    if (*(volatile int *)&s_abort) break;
                    if (++polls >= A.wait.polls) {
                        *(volatile int *)&s_abort = 1;
                        break;
                    }
                }
                const float l = __uint_as_float((uint32_t)wd);
                const int s = (int)__float_as_uint(r.w);
                const float mo = d[s];
                float n = lr_dir<MAXP>(r.x, r.y, r.z, l, mo, k, Tln2, damping, w);
                if (lr_dir_rare(n, l)) n = run_exact<MAXP>(A, pot, v0, s, l, mo);
                d[s] = n;
            }
        }
        __syncthreads();
    }

    if (X != kAlone && tid == 0 && s_abort) wait_failed(A);  // (here, not in the wait loop: 2 to 3 %)

    // ---- epilogue: every slot's two entries back into msgs (as k_lr_unpack) ----
    const bool aligned = (reinterpret_cast<uintptr_t>(msgs) & 7u) == 0;
    for (int lv = tid; lv < nv; lv += nt) {
        const int4 t = __ldg(A.tab4 + v0 + lv);
        const int es[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (es[q] < 0) continue;
            const float2 o = lr_decode(d[q * Vc + lv]);
            if (aligned) {
                reinterpret_cast<float2 *>(msgs)[es[q] >> 1] = o;
            } else {
                msgs[es[q]] = o.x;
                msgs[es[q] + 1] = o.y;
            }
        }
    }
    if constexpr (X == kCluster) cluster_barrier();  // no block leaves while another may write to its inbox
}

// ---- one block: graphs of up to kLrBlockAutoV variables ----
//
// Thread per directed edge: from the total of its variable and the message that came in along
// the edge it sends the new message to the factor's other variable, into the other of two copies
// of d. What the thread alone uses (its message, table numbers, addresses) stays in registers.
//   TWO = false, up to kPushOneE edges: the thread forms the total itself from the variable's
//     four messages. The four threads of a variable repeat it, but an iteration is one chain --
//     read, sum, update, write, barrier. Bound by that chain's latency.
//   TWO = true: a thread per variable forms the totals, a barrier, then the edges. Two chains,
//     but 1.6x fewer instructions, which is what bounds a block of 1,024 threads.
__device__ __noinline__ float push_lam_slow(float2 e, float d0, float d1, float d2, float d3, int k) {
    if (const float inf = clamped_ratio(e, d0, d1, d2, d3); inf != 0.f) return inf;
    const float dk[4] = {d0, d1, d2, d3};
    FF l0 = ff_make(e.x), l1 = ff_make(e.y);
    for (int j = 0; j < 4; ++j) {  // as lr_var_slow
        if (j == k) continue;
        const float2 q = lr_decode(dk[j]);
        l0 = ff_add(l0, q.x);
        l1 = ff_add(l1, q.y);
    }
    return lam_encode(l0, l1);
}

// The total of a variable from its evidence and four messages; false (and what the slow path
// needs left to the caller) when a leave-one-out value would not come out finite.
__device__ __forceinline__ bool push_total(float2 e, float d0, float d1, float d2, float d3, float2 &Df) {
    FF D = ff_add_nc(ff_make(e.y), -e.x);
    D = ff_add_nc(D, d0);
    D = ff_add_nc(D, d1);
    D = ff_add_nc(D, d2);
    D = ff_add_nc(D, d3);
    Df = make_float2(D.hi, D.lo);
    const float big = fmaxf(fmaxf(fabsf(d0), fabsf(d1)), fmaxf(fabsf(d2), fabsf(d3)));
    if (fabsf(D.hi) + big < 1e38f) return true;
    // an infinite entry, NaN, or near overflow
    return isfinite(e.x) && isfinite(e.y) && isfinite(d0) && isfinite(d1) && isfinite(d2) && isfinite(d3) &&
           isfinite(lr_lam_from_D(Df, d0)) && isfinite(lr_lam_from_D(Df, d1)) && isfinite(lr_lam_from_D(Df, d2)) &&
           isfinite(lr_lam_from_D(Df, d3));
}

template <bool MAXP, int NE, bool TWO>
__global__ void __launch_bounds__(kLrRunThreads, 1) k_lr_push(const LrRun A) {
    extern __shared__ __align__(16) char lr_sm[];
    const int V = A.V, E = A.E, tid = threadIdx.x, nt = blockDim.x, smp = blockIdx.x;
    const float *pot = A.pot + (size_t)smp * A.pot_stride;
    const float2 *ev = reinterpret_cast<const float2 *>(A.ev + (size_t)smp * A.ev_stride);
    float *msgs = A.msgs + (size_t)smp * A.msg_stride;
    float *cur = reinterpret_cast<float *>(lr_sm), *nxt = cur + 4 * V;
    float2 *Dv = reinterpret_cast<float2 *>(nxt + 4 * V);  // TWO
    for (int i = tid; i < 8 * V; i += nt) cur[i] = 0.f;  // (unused slots stay 0)
    __syncthreads();
    int v[NE], k[NE], dst[NE];
    float r[NE], p[NE], q[NE], mo[NE];
    float2 e[TWO ? 1 : NE];
    if (TWO) e[0] = tid < V ? __ldg(ev + tid) : make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < NE; ++j) {
        const int i = tid + j * nt;  // the edge this thread sends along, from its variable
        v[j] = k[j] = dst[j] = 0;
        r[j] = p[j] = q[j] = mo[j] = 0.f;
        if (!TWO) e[j] = make_float2(0.f, 0.f);
        if (i >= E) continue;
        const int s = __ldg(A.lr_pos + i);
        k[j] = (s >= V) + (s >= 2 * V) + (s >= 3 * V);
        v[j] = s - k[j] * V;
        dst[j] = __ldg(A.lr_pos + (i ^ 1));
        if (!TWO) e[j] = __ldg(ev + v[j]);
        mo[j] = lr_encode(__ldcg(msgs + 2 * (i ^ 1)), __ldcg(msgs + 2 * (i ^ 1) + 1));
        const float4 t = lr_table(A.segs, A.n_seg, pot, i >> 1);
        const bool fin = isfinite(t.x) & isfinite(t.y) & isfinite(t.z) & isfinite(t.w);
        const float c = fin ? t.z - t.x : CUDART_NAN_F, al = fin ? t.w - t.z : CUDART_NAN_F;
        const float be = fin ? t.y - t.x : CUDART_NAN_F;
        const bool to1 = (i & 1) == 0;  // from variable 0 to variable 1
        r[j] = to1 ? be : c;
        p[j] = to1 ? al + c - be : al;
        q[j] = to1 ? c : be;
        cur[dst[j]] = mo[j];
    }
    __syncthreads();
    const float w = 1.f - A.damping;
    for (int it = 0; it < A.n_iters; ++it) {
        if constexpr (TWO) {
            if (tid < V) {
                float2 Df;
                const bool ok = push_total(e[0], cur[tid], cur[V + tid], cur[2 * V + tid], cur[3 * V + tid], Df);
                Dv[tid] = ok ? Df : make_float2(__uint_as_float(kDvSlow), 0.f);
            }
            __syncthreads();
        }
#pragma unroll
        for (int j = 0; j < NE; ++j) {
            if (tid + j * nt >= E) continue;
            float l;
            if constexpr (TWO) {
                const float2 Df = Dv[v[j]];
                l = lr_lam_from_D(Df, cur[k[j] * V + v[j]]);
                if (is_slow(Df))
                    l = push_lam_slow(__ldg(ev + v[j]), cur[v[j]], cur[V + v[j]], cur[2 * V + v[j]], cur[3 * V + v[j]], k[j]);
            } else {
                const float d0 = cur[v[j]], d1 = cur[V + v[j]], d2 = cur[2 * V + v[j]], d3 = cur[3 * V + v[j]];
                float2 Df;
                const bool ok = push_total(e[j], d0, d1, d2, d3, Df);
                l = lr_lam_from_D(Df, k[j] == 0 ? d0 : k[j] == 1 ? d1 : k[j] == 2 ? d2 : d3);
                if (!ok) l = push_lam_slow(e[j], d0, d1, d2, d3, k[j]);
            }
            float n = lr_dir<MAXP>(r[j], p[j], q[j], l, mo[j], A.k, A.Tln2, A.damping, w);
            if (lr_dir_rare(n, l)) {
                const int i = tid + j * nt;
                const float4 t = lr_table(A.segs, A.n_seg, pot, i >> 1);
                const float phi[4] = {t.x, t.y, t.z, t.w};
                n = lr_dir_exact<MAXP>(phi, (i & 1) ^ 1, l, mo[j], A.k, A.Tln2, A.damping, A.flags);
            }
            mo[j] = n;
            nxt[dst[j]] = n;
        }
        __syncthreads();
        float *t = cur;
        cur = nxt;
        nxt = t;
    }
#pragma unroll
    for (int j = 0; j < NE; ++j) {
        const int i = tid + j * nt;
        if (i >= E) continue;
        const float2 o = lr_decode(mo[j]);
        msgs[2 * (i ^ 1)] = o.x;
        msgs[2 * (i ^ 1) + 1] = o.y;
    }
}

// ---- gradient in one launch ----
//
// pgm_grad of a graph with a table per factor: the forward iterations of k_lr_run from zero
// messages, with each iteration's lam also kept in global memory (16 bytes per variable and
// iteration), the read-out, and the reverse steps, in the same blocks with the same exchange.
// The launches it replaces (a 64 x 64 grid, 100 iterations: 590 of 2.4 us, half of them to
// recompute the forward from checkpoints) were bound by their latency; here a step forward or
// back costs one exchange between blocks, and nothing is recomputed.
//
// In log-ratios one step is d' = damping d + w (r + sp_T(p + lam) - sp_T(q + lam)) per message, lam =
// D - d, so with the adjoint a of the new message into a slot and the lam of the slot it came
// from, s_p = sigma((p + lam) / T), s_q likewise:
//   g = w a (s_p - s_q) is lam's adjoint, and w a s_p, w a (1 - s_p), -w a s_q, -w a (1 - s_q) those
//   of the table entries that p and q are differences of;
//   the stored message of slot k gets damping a_k + the g of the variable's other slots, the
//   evidence difference the sum of all four.
// A whole factor's two messages are done by one thread; of a split factor each block does the
// message that left it, for which the blocks exchange a instead of lam. The table's gradient is
// kept per factor and written once; the two blocks of a split factor add theirs to zeros (a sum of
// two terms: the same bits in either order), so repeated calls give the same bits.
// Tables with non-finite entries, contradictions and infinite messages (a lam of +-inf is
// fine: its sigmas are 0 or 1) set *bail, and so does a wait that runs out: the caller's launches
// take over. What shows in the inputs -- tables, evidence of -inf in both states -- ends the kernel in
// its prologue (64 x 64, 60 iterations, a table with -inf: 894 us by the launches alone, 1,097 with the
// kernel run to its end first, 941 so).
// Measured (GB300, whole calls): 64 x 64, 100 iterations, checkpoints every 10: 1.59 ms as ~590
// dependent launches of 2.4 us, 0.313 in one (0.311 with plain sums over a variable's factors, which
// lose what cancelling adjoints leave); with lr_dir's SFU forms 0.28, but the table gradients' error
// against 64 bits rose from 2.3e-7 to 2.7e-7 (mean of 15 grids). What bounds it:
// two barriers and an exchange per step of 200.
struct LrGrad {
    LrRun A;                // msgs unused
    const float *gnb;       // [2 V] cotangent of the normalised log-beliefs
    float *d_pot, *d_ev;
    float *hist;            // [n_iters][blocks][4 Vc]
    int *bail;              // and, at bail + 1, whether it was set in the prologue (both zeroed by the caller)
    float T;
};

// sigma(x / T) and 1 - sigma(x / T), each to a few ulp of itself (the launches' weights are exp of a
// difference of log-sum-exps, off by as many ulp of the exponent; a correctly rounded quotient costs
// 6 % of the call and leaves the gradients' error where it is).
struct Sigma {
    float s, c;
};
__device__ __forceinline__ Sigma sigma_t(float x, float invT) {
    const float t = expf(-fabsf(x) * invT), big = __fdividef(1.f, 1.f + t), small = t * big;
    return x >= 0.f ? Sigma{big, small} : Sigma{small, big};
}

// lr_dir (T > 0) with the accurate exponential and logarithm: its 3e-7 T would be the largest
// error of the gradient's forward messages.
__device__ __forceinline__ float grad_dir(float r, float p, float q, float l, float mo, float T, float invT,
                                          float damping, float w) {
    const float x = p + l, y = q + l;
    const float sx = fmaf(T, log1pf(expf(-fabsf(x) * invT)), fmaxf(x, 0.f));
    const float sy = fmaf(T, log1pf(expf(-fabsf(y) * invT)), fmaxf(y, 0.f));
    return fmaf(damping, mo, w * (r + sx - sy));
}

// The gradients of one direction's four table entries -- the two that p and the two that q are
// differences of, each weight formed as itself, since the differences of sums over the
// iterations would lose to cancellation -- and of the lam it came from.
struct DirGrad {
    float p1, p0, q1, q0, lam;
};
__device__ __forceinline__ DirGrad dir_grad(float p, float q, float l, float wa, float invT) {
    const Sigma P = sigma_t(p + l, invT), Q = sigma_t(q + l, invT);
    return DirGrad{wa * P.s, wa * P.c, -wa * Q.s, -wa * Q.c, wa * (P.s * Q.c - Q.s * P.c)};
}

// One value per split slot: out in step st, and in from the other block.
template <int X>
__device__ __forceinline__ void grad_publish(const LrRun &A, const float *val, const float4 *hrec, const uint32_t *hdst,
                                             int nH, int st) {
    if (X == kAlone) return;
    for (int h = threadIdx.x; h < nH; h += blockDim.x) {
        const unsigned long long wd = box_word(val[__float_as_uint(hrec[h].w) & 0xffff], (uint32_t)st);
        if (X == kCluster) {
            const uint32_t a = hdst[h] + ((st & 1) ? 8u * (uint32_t)A.h_cap : 0u);
            asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(wd) : "memory");
        } else {
            unsigned long long *p = ((st & 1) ? A.box1 : A.box0) + hdst[h];
            asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(wd) : "memory");
        }
    }
}
template <int X>
__device__ __forceinline__ float grad_receive(const LrRun &A, const unsigned long long *box, size_t h_base, int h, int st,
                                              int *s_abort) {
    unsigned long long wd = 0;
    int polls = 0;
    while (true) {
        if (X == kCluster) {
            const uint32_t a = smem_addr(box + h) + ((st & 1) ? 8u * (uint32_t)A.h_cap : 0u);
            asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(wd) : "r"(a) : "memory");
        } else {
            const unsigned long long *p = ((st & 1) ? A.box1 : A.box0) + h_base + h;
            asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(wd) : "l"(p) : "memory");
        }
        if ((uint32_t)(wd >> 32) == (uint32_t)st) return __uint_as_float((uint32_t)wd);
        if (*(volatile int *)s_abort) break;
        if (++polls >= A.wait.polls) {
            *(volatile int *)s_abort = 1;
            break;
        }
    }
    return 0.f;
}

template <int X>
__global__ void __launch_bounds__(kLrRunThreads, 1) k_lr_grad(const __grid_constant__ LrGrad P) {
    extern __shared__ __align__(16) char lr_sm[];
    __shared__ int s_n[2];
    __shared__ int s_abort;
    const LrRun &A = P.A;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    const int V = A.V, Vc = A.Vc;
    const int b = X == kCluster ? (int)cluster_rank() : (int)blockIdx.x;
    const int v0 = b * Vc, nv = max(0, min(Vc, V - v0));
    const size_t h_base = X == kGrid ? (size_t)A.off[b].y : 0;
    float *hist = P.hist + (size_t)b * 4 * Vc;
    const size_t hist_step = (size_t)A.nb * 4 * Vc;
    // shared memory
    char *sp = lr_sm;
    float4 *rec = reinterpret_cast<float4 *>(sp);  // c, al, be, slots
    sp += 16 * (size_t)A.f_cap;
    float4 *hrec = reinterpret_cast<float4 *>(sp);  // c, al, be, slot | side << 16
    sp += 16 * (size_t)A.h_cap;
    float4 *racc = reinterpret_cast<float4 *>(sp);  // gradients of a table's entries
    sp += 16 * (size_t)A.f_cap;
    float4 *hacc = reinterpret_cast<float4 *>(sp);
    sp += 16 * (size_t)A.h_cap;
    float2 *es_sh = reinterpret_cast<float2 *>(sp);
    sp += 8 * (size_t)Vc;
    unsigned long long *box = reinterpret_cast<unsigned long long *>(sp);
    if (X == kCluster) sp += 16 * (size_t)A.h_cap;
    float *lam = reinterpret_cast<float *>(sp);  // reverse: g
    sp += 16 * (size_t)Vc;
    float *d = reinterpret_cast<float *>(sp);    // reverse: a
    sp += 16 * (size_t)Vc;
    float *dD = reinterpret_cast<float *>(sp);   // the evidence difference's gradient
    sp += 4 * (size_t)Vc;
    uint32_t *hdst = reinterpret_cast<uint32_t *>(sp);

    if (tid < 2) s_n[tid] = 0;
    if (tid == 0) s_abort = X != kAlone && A.wait.polls == 0;
    for (int i = tid; i < A.f_cap; i += nt) racc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i = tid; i < A.h_cap; i += nt) hacc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    bool bad = false;
    for (int l0 = 0; l0 < nv; l0 += nt) {  // as k_lr_run's prologue
        const int lv = l0 + tid, v = v0 + lv;
        const int4 t = lv < nv ? __ldg(A.tab4 + v) : make_int4(-1, -1, -1, -1);
        if (lv < nv) {
            const float2 e = __ldg(reinterpret_cast<const float2 *>(A.ev) + v);
            es_sh[lv] = e;
            bad |= (e.x == kNegInf && e.y == kNegInf) | (e.x != e.x) | (e.y != e.y);
        }
        const int es[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bool have = es[q] >= 0;
            int u = 0, uk = 0;
            if (have) {
                const int p = __ldg(A.lr_pos + ((es[q] >> 1) ^ 1));  // the factor's other slot
                uk = (p >= V) + (p >= 2 * V) + (p >= 3 * V);
                u = p - uk * V;
            }
            if (lv < nv) d[q * Vc + lv] = 0.f;
            const bool local = X == kAlone || (u >= v0 && u < v0 + nv);
            const int side = (es[q] >> 1) & 1;
            const bool whole = have && local && side == 0, split = have && !local;
            float c = 0.f, al = 0.f, be = 0.f;
            if (whole || split) {
                const float4 tb = lr_table(A.segs, A.n_seg, A.pot, es[q] >> 2);
                c = tb.z - tb.x;
                al = tb.w - tb.z;
                be = tb.y - tb.x;
                bad |= !(isfinite(tb.x) & isfinite(tb.y) & isfinite(tb.z) & isfinite(tb.w));
            }
            const unsigned mw = __ballot_sync(0xffffffffu, whole), mh = __ballot_sync(0xffffffffu, split);
            int bw = 0, bh = 0;
            if (lane == 0) {
                if (mw) bw = atomicAdd(&s_n[0], __popc(mw));
                if (mh) bh = atomicAdd(&s_n[1], __popc(mh));
            }
            bw = __shfl_sync(0xffffffffu, bw, 0) + __popc(mw & ((1u << lane) - 1u));
            bh = __shfl_sync(0xffffffffu, bh, 0) + __popc(mh & ((1u << lane) - 1u));
            if (whole)
                rec[bw] = make_float4(c, al, be, __uint_as_float((uint32_t)(q * Vc + lv) | (uint32_t)(uk * Vc + u - v0) << 16));
            if (X != kAlone && split) {
                hrec[bh] = make_float4(c, al, be, __uint_as_float((uint32_t)(q * Vc + lv) | (uint32_t)side << 16));
                __stcg(A.dir + (size_t)q * V + v, bh);
            }
        }
    }
    // tables and evidence that the kernel hands back show here: every block learns of them at the
    // barrier, and none begins
    if (__syncthreads_or(bad)) {
        if (tid == 0) {
            *(volatile int *)P.bail = 1;
            *(volatile int *)(P.bail + 1) = 1;
            __threadfence();
        }
        if (X == kAlone) return;
    }
    const int nF = s_n[0], nH = X == kAlone ? 0 : s_n[1];
    bool ok = true;
    if constexpr (X == kCluster) {
        for (int h = tid; h < 2 * A.h_cap; h += nt) box[h] = 0;
        cluster_barrier();
    } else if constexpr (X == kGrid) {
        for (int h = tid; h < nH; h += nt) {
            __stcg(A.box0 + h_base + h, 0ull);
            __stcg(A.box1 + h_base + h, 0ull);
        }
        ok = grid_barrier_once(A.bar, gridDim.x, A.wait.polls);
    }
    if (X == kGrid && !ok) {
        if (tid == 0) *(volatile int *)P.bail = 1;
        return;
    }
    if (X != kAlone && *(volatile int *)(P.bail + 1) != 0) return;  // (written before the barrier only)
    for (int h = tid; h < nH; h += nt) {
        const int s = (int)(__float_as_uint(hrec[h].w) & 0xffff), q = s / Vc, lv = s - q * Vc;
        const int4 t = __ldg(A.tab4 + v0 + lv);
        const int es = q == 0 ? t.x : q == 1 ? t.y : q == 2 ? t.z : t.w;
        const int p = __ldg(A.lr_pos + ((es >> 1) ^ 1));
        const int u = p - V * ((p >= V) + (p >= 2 * V) + (p >= 3 * V));
        const int ub = u / Vc, at = __ldcg(A.dir + p);
        if constexpr (X == kCluster) hdst[h] = rank_addr(smem_addr(box + at), (uint32_t)ub);
        else hdst[h] = (uint32_t)(A.off[ub].y + at);
    }
    __syncthreads();

    const float T = P.T, invT = 1.f / P.T, damping = A.damping, w = 1.f - damping;
    // a message that lr_dir could not form
    auto rare = [&](int s, float l, float mo) {
        const float n = l == l ? run_exact<false>(A, A.pot, v0, s, l, mo) : 0.f;
        bad |= !(l == l) | !isfinite(n);
        return n;
    };

    // ---- forward ----
    for (int it = 1; it <= A.n_iters; ++it) {
        float *H = hist + (size_t)(it - 1) * hist_step;
        for (int lv = tid; lv < nv; lv += nt) {
            const float2 e = es_sh[lv];
            const float d0 = d[lv], d1 = d[Vc + lv], d2 = d[2 * Vc + lv], d3 = d[3 * Vc + lv];
            float2 Df;
            if (push_total(e, d0, d1, d2, d3, Df)) {
                lam[lv] = lr_lam_from_D(Df, d0);
                lam[Vc + lv] = lr_lam_from_D(Df, d1);
                lam[2 * Vc + lv] = lr_lam_from_D(Df, d2);
                lam[3 * Vc + lv] = lr_lam_from_D(Df, d3);
            } else {
                run_var_slow(lam, lv, Vc, e, d0, d1, d2, d3);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) __stcg(H + q * Vc + lv, lam[q * Vc + lv]);
        }
        __syncthreads();
        grad_publish<X>(A, lam, hrec, hdst, nH, it);
        for (int i = tid; i < nF; i += nt) {
            const float4 r = rec[i];
            const uint32_t pk = __float_as_uint(r.w);
            const int s0 = pk & 0xffff, s1 = pk >> 16;
            const float mo0 = d[s0], mo1 = d[s1], l0 = lam[s0], l1 = lam[s1];
            float n0 = grad_dir(r.x, r.y, r.z, l1, mo0, T, invT, damping, w);
            float n1 = grad_dir(r.z, r.y + r.x - r.z, r.x, l0, mo1, T, invT, damping, w);
            if (!(fabsf(n0) + fabsf(n1) < CUDART_INF_F)) {
                if (lr_dir_rare(n0, l1)) n0 = rare(s0, l1, mo0);
                if (lr_dir_rare(n1, l0)) n1 = rare(s1, l0, mo1);
            }
            d[s0] = n0;
            d[s1] = n1;
        }
        for (int h = tid; h < nH; h += nt) {
            const float4 r = hrec[h];
            const uint32_t pk = __float_as_uint(r.w);
            const int s = pk & 0xffff;
            const bool one = (pk >> 16) != 0;  // the message into the factor's variable 1
            const float mo = d[s], l = grad_receive<X>(A, box, h_base, h, it, &s_abort);
            float n = one ? grad_dir(r.z, r.y + r.x - r.z, r.x, l, mo, T, invT, damping, w)
                          : grad_dir(r.x, r.y, r.z, l, mo, T, invT, damping, w);
            if (lr_dir_rare(n, l)) n = rare(s, l, mo);
            d[s] = n;
        }
        __syncthreads();
    }
    // ---- the read-out: L = sum g (b - LSE(b)), dL/dD = g1 - (g0 + g1) sigma(D) ----
    for (int lv = tid; lv < nv; lv += nt) {
        float2 D;
        if (!push_total(es_sh[lv], d[lv], d[Vc + lv], d[2 * Vc + lv], d[3 * Vc + lv], D)) {
            const float2 e = es_sh[lv];  // (finite messages: an infinite evidence entry, or none)
            D = make_float2(e.y - e.x, 0.f);
            bad |= !(D.x == D.x) | !(fabsf(d[lv]) + fabsf(d[Vc + lv]) + fabsf(d[2 * Vc + lv]) + fabsf(d[3 * Vc + lv]) < CUDART_INF_F);
        }
        const float *gp = P.gnb + 2 * (size_t)(v0 + lv);  // (the caller's, at any 4-byte address)
        const float2 g = make_float2(__ldg(gp), __ldg(gp + 1));
        const float x = D.x + D.y, a = g.y * sigma_t(x, 1.f).c - g.x * sigma_t(x, 1.f).s;
        dD[lv] = a;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            d[q * Vc + lv] = a;
            lam[q * Vc + lv] = 0.f;  // unused slots have no g
        }
    }
    __syncthreads();
    // ---- reverse ----
    for (int it = A.n_iters; it >= 1; --it) {
        const float *H = hist + (size_t)(it - 1) * hist_step;
        const int st = 2 * A.n_iters + 1 - it;
        grad_publish<X>(A, d, hrec, hdst, nH, st);
        for (int i = tid; i < nF; i += nt) {
            const float4 r = rec[i];
            const uint32_t pk = __float_as_uint(r.w);
            const int s0 = pk & 0xffff, s1 = pk >> 16;
            const float l0 = __ldcg(H + s0), l1 = __ldcg(H + s1);
            const DirGrad a = dir_grad(r.y, r.z, l1, w * d[s0], invT), c = dir_grad(r.y + r.x - r.z, r.x, l0, w * d[s1], invT);
            lam[s1] = a.lam;
            lam[s0] = c.lam;
            float4 t = racc[i];  // to variable 0: p = phi11 - phi10, q = phi01 - phi00; to 1: phi11 - phi01, phi10 - phi00
            t.x += a.q0 + c.q0;
            t.y += a.q1 + c.p0;
            t.z += a.p0 + c.q1;
            t.w += a.p1 + c.p1;
            racc[i] = t;
        }
        for (int h = tid; h < nH; h += nt) {  // the message that left slot s, towards the other block
            const float4 r = hrec[h];
            const uint32_t pk = __float_as_uint(r.w);
            const int s = pk & 0xffff;
            const bool one = (pk >> 16) != 0;  // the source is variable 1: the message to variable 0
            const float l = __ldcg(H + s), a = w * grad_receive<X>(A, box, h_base, h, st, &s_abort);
            const DirGrad g = one ? dir_grad(r.y, r.z, l, a, invT) : dir_grad(r.y + r.x - r.z, r.x, l, a, invT);
            lam[s] = g.lam;
            float4 t = hacc[h];
            t.x += g.q0;
            t.y += one ? g.q1 : g.p0;
            t.z += one ? g.p0 : g.q1;
            t.w += g.p1;
            hacc[h] = t;
        }
        __syncthreads();
        for (int lv = tid; lv < nv; lv += nt) {
            const float g0 = lam[lv], g1 = lam[Vc + lv], g2 = lam[2 * Vc + lv], g3 = lam[3 * Vc + lv];
            FF S = ff_add_nc(ff_make(g0), g1);  // float-float, as k_adj_var_tab4's sums
            S = ff_add_nc(S, g2);
            S = ff_add_nc(S, g3);
            const float2 t = make_float2(S.hi, S.lo);
            d[lv] = fmaf(damping, d[lv], lr_lam_from_D(t, g0));
            d[Vc + lv] = fmaf(damping, d[Vc + lv], lr_lam_from_D(t, g1));
            d[2 * Vc + lv] = fmaf(damping, d[2 * Vc + lv], lr_lam_from_D(t, g2));
            d[3 * Vc + lv] = fmaf(damping, d[3 * Vc + lv], lr_lam_from_D(t, g3));
            dD[lv] += S.hi + S.lo;
        }
        __syncthreads();
    }
    // ---- out ----
    for (int lv = tid; lv < nv; lv += nt) {
        P.d_ev[2 * (size_t)(v0 + lv)] = -dD[lv];
        P.d_ev[2 * (size_t)(v0 + lv) + 1] = dD[lv];
    }
    auto table_of = [&](int s) {  // the table of slot s's factor in d_pot
        const int q = s / Vc, v = v0 + s - q * Vc;
        const int4 t = __ldg(A.tab4 + v);
        const int g = (q == 0 ? t.x : q == 1 ? t.y : q == 2 ? t.z : t.w) >> 2;
        const EnumSeg *S = A.segs + lr_seg_of(A.segs, A.n_seg, g);
        return P.d_pot + __ldg(&S->pot_base) + 4 * (size_t)(g - (__ldg(&S->edge_base) >> 1));
    };
    for (int i = tid; i < nF; i += nt) {
        float *t = table_of((int)(__float_as_uint(rec[i].w) & 0xffff));
        const float4 a = racc[i];
        t[0] = a.x;
        t[1] = a.y;
        t[2] = a.z;
        t[3] = a.w;
    }
    for (int h = tid; h < nH; h += nt) {
        float *t = table_of((int)(__float_as_uint(hrec[h].w) & 0xffff));
        const float4 a = hacc[h];
        atomicAdd(t, a.x);
        atomicAdd(t + 1, a.y);
        atomicAdd(t + 2, a.z);
        atomicAdd(t + 3, a.w);
    }
    if (bad || (X != kAlone && s_abort)) *P.bail = 1;
    if constexpr (X == kCluster) cluster_barrier();
}

__global__ void k_set_condition(cudaGraphConditionalHandle h, const int *__restrict__ word) {
    cudaGraphSetConditional(h, *word != 0 ? 1u : 0u);
}

using RunKernel = void (*)(const LrRun);
// LAM where it fits: always with the records in shared memory.
template <bool MAXP>
RunKernel run_kernel_t(int x, bool res, bool lam) {
    if (x == kCluster) return k_lr_run<MAXP, kCluster, true, true>;
    if (x == kAlone) return res ? k_lr_run<MAXP, kAlone, true, true>
                                : lam ? k_lr_run<MAXP, kAlone, false, true> : k_lr_run<MAXP, kAlone, false, false>;
    return res ? k_lr_run<MAXP, kGrid, true, true>
               : lam ? k_lr_run<MAXP, kGrid, false, true> : k_lr_run<MAXP, kGrid, false, false>;
}
RunKernel run_kernel(bool maxp, int x, bool res, bool lam) {
    return maxp ? run_kernel_t<true>(x, res, lam) : run_kernel_t<false>(x, res, lam);
}

// What the device offers, asked once: SMs, shared memory for a block, cluster size, whether
// it takes cooperative launches. The kernels' attributes are set here too.
struct RunDevice {
    bool ready = false;
    int n_sm = 0, smem = 0, cluster = 0;
    bool coop = false;
};
const RunDevice &run_device() {
    static RunDevice devs[64];
    static std::mutex mu;
    static const RunDevice none;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return none;
    std::lock_guard<std::mutex> lk(mu);
    RunDevice &R = devs[dev];
    if (R.ready) return R;
    int optin = 0, coop = 0;
    if (cudaDeviceGetAttribute(&R.n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess) {
        cudaGetLastError();
        return none;
    }
    R.smem = optin - 256;  // less the kernels' static shared memory
    for (int x = 0; x < 3; ++x)
        for (int m = 0; m < 2; ++m)
            for (int r = 0; r < 3; ++r) {
                RunKernel kern = run_kernel(m, x, r == 2, r >= 1);
                cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, R.smem);
                if (x == kCluster) cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            }
    for (auto kern : {k_lr_grad<kAlone>, k_lr_grad<kCluster>, k_lr_grad<kGrid>})
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, R.smem);
    cudaFuncSetAttribute(k_lr_grad<kCluster>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    for (int C : {kLrClusterMax, 8}) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(C);
        cfg.blockDim = dim3(kLrRunThreads);
        cfg.dynamicSmemBytes = run_smem(kCluster, true, true, kLrSmallMaxV, 2 * kLrSmallMaxV, 4 * kLrSmallMaxV);
        if ((int)cfg.dynamicSmemBytes > R.smem) break;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = C;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n0 = 0, n1 = 0;
        if (cudaOccupancyMaxActiveClusters(&n0, k_lr_run<true, kCluster, true, true>, &cfg) == cudaSuccess && n0 > 0 &&
            cudaOccupancyMaxActiveClusters(&n1, k_lr_run<false, kCluster, true, true>, &cfg) == cudaSuccess && n1 > 0) {
            R.cluster = C;
            break;
        }
    }
    R.coop = coop != 0;
    for (int m = 0; m < 2 && R.coop; ++m)
        for (int r = 0; r < 3; ++r) {
            int n = 0;
            R.coop = R.coop && cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, run_kernel(m, kGrid, r == 2, r >= 1),
                                                                             kLrRunThreads, R.smem) == cudaSuccess && n >= 1;
        }
    cudaGetLastError();  // a refused query leaves no error behind
    R.ready = true;
    return R;
}

template <class Args>
cudaError_t launch(void (*kern)(const Args), const Args &A, int blocks, int threads, size_t smem, int x, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    if (x == kCluster) {
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = (unsigned)blocks;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
    } else {
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
    }
    cfg.attrs = at;
    cfg.numAttrs = x == kAlone ? 0 : 1;
    return cudaLaunchKernelEx(&cfg, kern, A);
}

// The push form of one block per sample (lr_block_fits).
template <bool MAXP>
RunKernel push_kernel(const PushShape &p) {
    if (!p.two) return k_lr_push<MAXP, 1, false>;
    return p.edges == 1 ? k_lr_push<MAXP, 1, true> : p.edges == 2 ? k_lr_push<MAXP, 2, true> : k_lr_push<MAXP, 4, true>;
}
cudaError_t launch_push(const LrRun &A, bool maxp, int samples, cudaStream_t s) {
    const PushShape p = push_shape(A.V, A.E);
    return launch(maxp ? push_kernel<true>(p) : push_kernel<false>(p), A, samples, p.threads, p.smem, kAlone, s);
}

LrRun run_args(const DevGraph &G, const EnumSeg *segs, int n_seg, const float *pot, const float *ev, float *msgs,
               float *lam, float T, float damping, int n_iters, const LrWait &wait) {
    LrRun A{};
    A.wait = wait;
    A.V = G.V;
    A.E = G.E;
    A.tab4 = G.vin_tab4;
    A.lr_pos = G.lr_pos;
    A.segs = segs;
    A.n_seg = n_seg;
    A.pot = pot;
    A.ev = ev;
    A.msgs = msgs;
    A.lam = lam;
    A.flags = G.flags;
    A.bar = G.flags + 16;
    // softplus_t constants: k = log2(e) / T, T ln 2
    A.k = T > 0.f ? (float)(1.4426950408889634 / (double)T) : 0.f;
    A.Tln2 = (float)((double)T * 0.6931471805599453);
    A.damping = damping;
    A.n_iters = n_iters;
    A.nb = 1;
    A.Vc = G.V;
    return A;
}

// The one launch that covers every factor of a log-ratio graph.
const FactorLaunch *only_launch(const Plan &P) {
    for (const FactorLaunch &L : P.factor)
        if (L.n_blocks > 0) return &L;
    return nullptr;
}

}  // namespace

int lr_cluster_size() { return run_device().cluster; }

cudaError_t launch_lr_small_run(const DevGraph &G, const Plan &P, const float *log_pot, const float *ev, float *msgs,
                                float *lam, int32_t *dir, float T, float damping, int n_iters, bool cluster,
                                const LrWait &wait, cudaStream_t s) {
    const int F = G.E / 2, V = G.V;
    if (!(cluster ? lr_cluster_fits(V, F) : lr_block_fits(V, F)) || G.vin_tab4 == nullptr || G.lr_pos == nullptr)
        return cudaErrorInvalidValue;
    const FactorLaunch *L = only_launch(P);
    if (L == nullptr || n_iters <= 0) return cudaSuccess;
    run_device();  // the kernels' attributes
    LrRun A = run_args(G, static_cast<const EnumSeg *>(L->segs), L->n_seg, log_pot, ev, msgs, lam, T, damping, n_iters, wait);
    A.dir = dir;
    if (!cluster) return launch_push(A, T == 0.f, 1, s);
    const int C = lr_cluster_size();
    A.nb = C;
    A.Vc = (V + C - 1) / C;
    A.f_cap = 2 * A.Vc;  // a block's variables have 4 slots each, a whole factor takes two
    A.h_cap = 4 * A.Vc;
    return launch(run_kernel(T == 0.f, kCluster, true, true), A, C, run_threads(A.Vc, (F + C - 1) / C),
                  run_smem(kCluster, true, true, A.Vc, A.f_cap, A.h_cap), kCluster, s);
}

// ---- the grid form of one sample ----

int lr_grid_device() { return run_device().coop ? run_device().n_sm : 0; }
int lr_grid_smem() { return run_device().smem; }

bool lr_grid_fits(const LrGridPlan &g, int V, int F) {
    const RunDevice &R = run_device();
    if (g.nb < 2 || !R.coop || g.nb > R.n_sm) return false;
    const int64_t split = g.n_split;
    // the workspace: see launch_lr_grid_run
    if (run_smem(kGrid, true, true, g.Vc, g.f_max, g.h_max) <= (size_t)R.smem) return 2 * split <= 3 * (int64_t)F;
    return 20 * split <= 12 * (int64_t)F && 16 * split <= 8 * (int64_t)V;
}

// Workspace from the graph's multi-launch scratch, which a one-launch run does not otherwise
// use (bytes, F factors, V variables): m_tmp [16 F], b [8 V], d [16 V], prm [12 F]. The slot
// directory (16 V) is in d. Records in shared memory: the inboxes (8 bytes per split slot
// each) in m_tmp and prm. Records in global memory: whole factors' in m_tmp (16 each), split
// factors' (16 + 4) in prm, the inboxes in b. lr_grid_fits has checked that they fit.
cudaError_t launch_lr_grid_run(const DevGraph &G, const Plan &P, const LrGridPlan &g, const float *log_pot,
                               const float *ev, float *msgs, float *lam, float *m_tmp, float *b, float *d, float *prm,
                               float T, float damping, int n_iters, const LrWait &wait, cudaStream_t s) {
    const int F = G.E / 2, V = G.V;
    if (!lr_grid_fits(g, V, F)) return cudaErrorInvalidValue;
    const FactorLaunch *L = only_launch(P);
    if (L == nullptr || n_iters <= 0) return cudaSuccess;
    const RunDevice &R = run_device();
    LrRun A = run_args(G, static_cast<const EnumSeg *>(L->segs), L->n_seg, log_pot, ev, msgs, lam, T, damping, n_iters, wait);
    A.dir = reinterpret_cast<int32_t *>(d);
    A.nb = g.nb;
    A.Vc = g.Vc;
    A.f_cap = g.f_max;
    A.h_cap = g.h_max;
    A.off = g.off;
    const size_t smem = run_smem(kGrid, true, true, g.Vc, g.f_max, g.h_max);
    const bool res = smem <= (size_t)R.smem;
    if (res) {
        A.box0 = reinterpret_cast<unsigned long long *>(m_tmp);
        A.box1 = reinterpret_cast<unsigned long long *>(prm);
    } else {
        A.rec = reinterpret_cast<float4 *>(m_tmp);
        A.hrec = reinterpret_cast<float4 *>(prm);
        A.hdst = reinterpret_cast<uint32_t *>(prm) + 4 * g.n_split;
        A.box0 = reinterpret_cast<unsigned long long *>(b);
        A.box1 = A.box0 + g.n_split;
    }
    const bool lam_sh = run_smem(kGrid, false, true, g.Vc, 0, 0) <= (size_t)R.smem;
    return launch(run_kernel(T == 0.f, kGrid, res, lam_sh), A, g.nb, run_threads(g.Vc, g.f_max),
                  res ? smem : run_smem(kGrid, false, lam_sh, g.Vc, 0, 0), kGrid, s);
}

// ---- many samples of one graph ----

LrMultiPlan lr_multi_plan(int V, int S, bool local) {
    const RunDevice &R = run_device();
    return lr_multi_plan(V, S, local, R.n_sm, R.smem, R.coop);
}

cudaError_t launch_lr_multi_run(const DevGraph &G, const Plan &P, const LrMultiPlan &p, int S, int64_t pot_stride,
                                const float *log_pot, const float *ev, float *msgs, char *work, float T, float damping,
                                int n_iters, const LrWait &wait, cudaStream_t s) {
    const FactorLaunch *L = only_launch(P);
    if (S < 1 || S > p.S || G.vin_tab4 == nullptr) return cudaErrorInvalidValue;
    if (L == nullptr || n_iters <= 0) return cudaSuccess;
    const size_t V = (size_t)G.V, blocks = (size_t)S * p.nb;
    LrRun A = run_args(G, static_cast<const EnumSeg *>(L->segs), L->n_seg, log_pot, ev, msgs, nullptr, T, damping, n_iters, wait);
    A.pot_stride = pot_stride;
    A.ev_stride = G.VS;
    A.msg_stride = G.ES;
    A.nb = p.nb;
    A.Vc = p.Vc;
    A.lam_stride = (int64_t)lam_floats(p.nb, p.Vc);
    A.f_cap = p.f_cap;
    A.h_cap = p.h_cap;
    // 16-byte records first, then 8-byte inboxes, then words
    if (!p.res) {
        A.rec = reinterpret_cast<float4 *>(work);
        A.hrec = A.rec + blocks * p.f_cap;
        work = reinterpret_cast<char *>(A.hrec + blocks * p.h_cap);
    }
    A.box0 = reinterpret_cast<unsigned long long *>(work);
    A.box1 = A.box0 + blocks * p.h_cap;
    A.hdst = reinterpret_cast<uint32_t *>(A.box1 + blocks * p.h_cap);
    A.lam = reinterpret_cast<float *>(A.hdst + (p.res ? 0 : blocks * p.h_cap));
    A.dir = reinterpret_cast<int32_t *>(A.lam + lam_floats(p.nb, p.Vc) * S);
    if (p.nb == 1 && G.V <= kLrBlockAutoV && lr_block_fits(G.V, G.E / 2)) return launch_push(A, T == 0.f, S, s);
    const int x = p.nb > 1 ? kGrid : kAlone;
    const bool lam_sh = run_smem(x, false, true, p.Vc, 0, 0) <= (size_t)run_device().smem;
    return launch(run_kernel(T == 0.f, x, p.res, lam_sh), A, (int)blocks, run_threads(p.Vc, (2 * G.V + p.nb - 1) / p.nb),
                  p.res ? run_smem(x, true, true, p.Vc, p.f_cap, p.h_cap) : run_smem(x, false, lam_sh, p.Vc, 0, 0), x, s);
}

// ---- gradient ----

LrGradPlan lr_grad_plan(const LrGridPlan &g, int V, int F, int n_iters) {
    const RunDevice &R = run_device();
    LrGradPlan p;
    if (V < 1 || F < 1 || n_iters < 1 || n_iters > (1 << 28)) return p;
    const int C = R.cluster;
    if (V <= kLrBlockAutoV && F <= kLrBlockAutoF && grad_smem(kAlone, V, F, 0) <= (size_t)R.smem) {
        p.form = 1;
        p.nb = 1;
        p.Vc = V;
        p.f_cap = F;
    } else if (C > 0 && V <= kLrClusterAutoV && grad_smem(kCluster, (V + C - 1) / C, 2 * ((V + C - 1) / C), 4 * ((V + C - 1) / C)) <= (size_t)R.smem) {
        p.form = 2;
        p.nb = C;
        p.Vc = (V + C - 1) / C;
        p.f_cap = 2 * p.Vc;
        p.h_cap = 4 * p.Vc;
    } else if (g.nb >= 2 && R.coop && g.nb <= R.n_sm && grad_smem(kGrid, g.Vc, g.f_max, g.h_max) <= (size_t)R.smem &&
               2 * g.n_split <= 3 * (int64_t)F) {  // (the inboxes, as launch_lr_grid_run)
        p.form = 3;
        p.nb = g.nb;
        p.Vc = g.Vc;
        p.f_cap = g.f_max;
        p.h_cap = g.h_max;
    } else {
        return p;
    }
    p.hist_bytes = (size_t)n_iters * p.nb * 16 * (size_t)p.Vc;
    if (p.hist_bytes > kLrGradHistory) p.form = 0;
    return p;
}

cudaError_t launch_lr_grad(const DevGraph &G, const Plan &P, const LrGradPlan &p, const float *log_pot, const float *ev,
                           const float *gnb, float *d_pot, float *d_ev, float *hist, int *bail, float *m_tmp, float *d,
                           float *prm, float T, float damping, int n_iters, const LrWait &wait, cudaStream_t s) {
    const FactorLaunch *L = only_launch(P);
    if (L == nullptr || p.form == 0) return cudaErrorInvalidValue;
    const EnumSeg *segs = static_cast<const EnumSeg *>(L->segs);
    LrGrad a{};
    a.A = run_args(G, segs, L->n_seg, log_pot, ev, nullptr, nullptr, T, damping, n_iters, wait);
    a.A.nb = p.nb;
    a.A.Vc = p.Vc;
    a.A.f_cap = p.f_cap;
    a.A.h_cap = p.h_cap;
    a.A.off = P.grid.off;
    a.A.dir = reinterpret_cast<int32_t *>(d);
    a.A.box0 = reinterpret_cast<unsigned long long *>(m_tmp);
    a.A.box1 = reinterpret_cast<unsigned long long *>(prm);
    a.gnb = gnb;
    a.d_pot = d_pot;
    a.d_ev = d_ev;
    a.hist = hist;
    a.bail = bail;
    a.T = T;
    const int x = p.form == 1 ? kAlone : p.form == 2 ? kCluster : kGrid;
    auto kern = p.form == 1 ? k_lr_grad<kAlone> : p.form == 2 ? k_lr_grad<kCluster> : k_lr_grad<kGrid>;
    const int items = p.form == 3 ? p.f_cap : (G.E / 2 + p.nb - 1) / p.nb;
    return launch(kern, a, p.nb, run_threads(p.Vc, items), grad_smem(x, p.Vc, p.f_cap, p.h_cap), x, s);
}

cudaError_t launch_set_condition(cudaGraphConditionalHandle h, const int *word, cudaStream_t s) {
    k_set_condition<<<1, 1, 0, s>>>(h, word);
    return cudaGetLastError();
}

}  // namespace pgm
