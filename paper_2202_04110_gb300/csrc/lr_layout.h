// Launch shapes and shared-memory layouts of the one-launch log-ratio runs (lr_run.cu): host
// arithmetic alone, so that it is checked without a device.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>

namespace pgm {

constexpr int kLrRunThreads = 1024, kLrSmallMaxV = 1024, kLrSmallMaxF = 2048;
constexpr int kLrClusterMax = 16;
// Setting 1 of PGM_OPT_SMALL_RUN: one block up to this many variables and factors, the cluster
// up to kLrClusterAutoV variables, the grid form above (us per iteration, T = 1, square grids:
// 22 x 22 block 0.65, cluster 0.82; 24 x 24 1.03, 0.81; 90 x 90 cluster 1.17; 128 x 128 cluster
// 1.75, grid 1.22).
constexpr int kLrBlockAutoV = 700, kLrBlockAutoF = 1024, kLrClusterAutoV = 9000;
constexpr int kLrGridMinV = 256;  // variables per block of the grid form at least
constexpr int kLrAloneV = 1536;   // pgm_run_bp_multi: up to this many variables a sample takes one block
// A GB300's SMs and a block's shared memory (less the kernels' static part), for sizes that are
// stated without asking a device (pgm_check_desc, serving budgets).
constexpr int kPlanSms = 152, kPlanSmem = 232448 - 256;

// Where a block's items and exchanged values live.
enum LrExchange : int { kAlone = 0, kCluster = 1, kGrid = 2 };

// Shared memory of a block of k_lr_run: Vc variables, f_cap whole and h_cap split factors. res: the
// records and the evidence too; lam: lam per slot (16 bytes a variable), else the totals (8).
inline size_t run_smem(int x, bool res, bool lam, int Vc, int f_cap, int h_cap) {
    size_t n = (lam ? 32 : 24) * (size_t)Vc;
    if (res) n += 8 * (size_t)Vc + 16 * (size_t)f_cap + 20 * (size_t)h_cap;
    if (x == kCluster) n += 16 * (size_t)h_cap;
    return n + 16;
}

// Explicit sums in global memory (the form with totals): 4 Vc a block, fewer than 4 nb floats more than
// 4 V in all, of which a graph's scratch has room for up to kLrMaxBlocks blocks.
constexpr int kLrMaxBlocks = 256;
inline size_t lam_floats(int nb, int Vc) { return 4 * (size_t)nb * Vc; }
inline size_t lam_floats_max(int64_t slots) { return (size_t)slots + 4 * kLrMaxBlocks; }

// Shared memory of a gradient block.
inline size_t grad_smem(int x, int Vc, int f_cap, int h_cap) {
    return 44 * (size_t)Vc + 32 * (size_t)f_cap + (x == kCluster ? 52 : 36) * (size_t)h_cap + 16;
}

inline int run_threads(int Vc, int items) {
    const int per = std::max(Vc, items);
    return std::min(kLrRunThreads, std::max(32, (per + 31) / 32 * 32));
}

// k_lr_push, one block per sample, a thread per directed edge (1, 2 or 4 of them): up to kPushOneE
// edges a thread forms its variable's total itself, above that a thread per variable does.
constexpr int kPushOneE = 600;
struct PushShape {
    int edges, threads;
    bool two;
    size_t smem;  // two copies of d, 16 bytes a variable each, and the totals (two)
};
inline PushShape push_shape(int V, int E) {
    const int n = E <= kLrRunThreads ? 1 : E <= 2 * kLrRunThreads ? 2 : 4;
    const bool two = E > kPushOneE;
    return PushShape{n, run_threads(V, (E + n - 1) / n), two, (two ? 40 : 32) * (size_t)V};
}

// The grid form: blocks for V variables on n_sm SMs with smem bytes a block (0: none).
inline int lr_grid_blocks(int V, int n_sm, int smem) {
    if (n_sm < 1 || V < 2) return 0;
    n_sm = std::min(n_sm, kLrMaxBlocks);
    const int Vc = std::max((V + n_sm - 1) / n_sm, kLrGridMinV);
    const int nb = (V + Vc - 1) / Vc;
    return nb >= 2 && run_smem(kGrid, false, false, Vc, 0, 0) <= (size_t)smem && Vc < (1 << 14) ? nb : 0;
}

// Many samples of one graph: nb blocks each, up to S samples a launch.
struct LrMultiPlan {
    int S = 0;  // samples per launch; 0: the device takes no such launch
    int nb = 0, Vc = 0, f_cap = 0, h_cap = 0;
    bool res = false;
    size_t sample_bytes = 0;
};
// A sample that several blocks do not divide well still takes one block up to kLrAloneMaxV variables, and
// above that where S >= (V / 800)^2 samples keep as many SMs busy: one block is slower than the launches
// of all samples together until they are that many (us per iteration, grids numbered at random, launches
// against one block: 3,600 variables 3.7 / 4.5 with 8 samples, 5.1 / 4.5 with 32; 5,625 6.1 / 7.2 with 32,
// 9.1 / 7.2 with 64; 9,409 13.5 / 14.2 with 64, 29 / 14.5 with 152).
constexpr int kLrAloneMaxV = 3000;
// coop: the device takes cooperative launches; local: few factors join different blocks (LrGridPlan).
inline LrMultiPlan lr_multi_plan(int V, int S, bool local, int n_sm, int smem, bool coop) {
    LrMultiPlan p;
    if (n_sm < 1 || V < 1 || S < 1) return p;
    const int v_max = std::min((1 << 14) - 1, (smem - 16) / 24);  // variables one block can own
    const int nb_min = (V + v_max - 1) / v_max;
    int nb = 1, Sc = S;
    if (V > kLrAloneV && coop && local && nb_min <= n_sm) {
        const int chunks = (S + n_sm / nb_min - 1) / (n_sm / nb_min);
        Sc = (S + chunks - 1) / chunks;
        nb = std::min(n_sm / Sc, (V + kLrGridMinV - 1) / kLrGridMinV);
    } else if (nb_min > 1 || (V > kLrAloneMaxV && (int64_t)V * V > (int64_t)640000 * S)) {
        return p;
    }
    p.Vc = (V + nb - 1) / nb;
    p.nb = (V + p.Vc - 1) / p.Vc;
    p.f_cap = 2 * p.Vc;  // a block's variables have 4 slots each, a whole factor takes two
    p.h_cap = p.nb > 1 ? 4 * p.Vc : 0;
    p.res = run_smem(p.nb > 1 ? kGrid : kAlone, true, true, p.Vc, p.f_cap, p.h_cap) <= (size_t)smem;
    // per sample: lam and directory, then each block's items (launch_lr_multi_run's layout)
    p.sample_bytes = 4 * lam_floats(p.nb, p.Vc) + 16 * (size_t)V + (size_t)p.nb * (16 * (size_t)p.h_cap + (p.res ? 0 : 16 * (size_t)p.f_cap + 20 * (size_t)p.h_cap));
    if (p.nb == 1) Sc = (int)std::min<int64_t>(S, std::max<int64_t>(1, ((int64_t)1 << 28) / (int64_t)p.sample_bytes));
    p.S = Sc;
    return p;
}

}  // namespace pgm
