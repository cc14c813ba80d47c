// On-chip CG engine: the layout rule (host).
#pragma once

#include "hh_onchip.cuh"

namespace hh {

// Dynamic shared memory a block may ask for: the 227 KB a block can have, less
// the kernels' static part.  The kernels' limit is set to it, whatever a
// launch uses, so that threads launching different layouts do not race on it.
constexpr int kOcStaticSmem = 2048;
constexpr int kOcMaxSmem = 227 * 1024 - kOcStaticSmem;

// Dynamic shared memory of a block whose tile is at most so x st columns of P
// sites (the kernel's layout).
inline size_t oc_smem(int d, long long P, int so, int st, bool mixed, bool cheb, bool x_global)
{
    const long long C = P * so * st, E = P * (so + 2) * (st + 1), Lk = P * so * (st + 1);
    const long long vals = 3 * E + Lk + (x_global ? 0 : C) + (cheb ? 2 * C : 0);
    return (size_t)(vals * (mixed ? 4 : 8) + (d == 3 ? P * so : 0) + 16);
}

// Column form: a tile's row of so P sites, one per thread, st slices each, with
// one halo column per edge thread, or two when tiles have one o position (d = 3).
inline bool cols_candidate(int d, long long P, int nx, int go, int so, int st, bool mixed, bool cheb, bool ex, int *K,
                           int *sides, int *threads)
{
    const long long row = P * so;
    if (row > kColMaxRow || st > (cheb || ex ? 4 : 8)) return false;
    *sides = nx / go >= 2 ? 1 : 2;
    if (*sides == 2 && (d == 1 || so != 1)) return false;
    *K = st <= 2 ? 2 : st <= 4 ? 4 : 8;
    *threads = (int)((row + 31) / 32 * 32) + 32;
    return *threads <= col_max_threads(mixed ? 4 : 8, *K);
}

// The layout of least cost for nsys systems (ok = 0: none fits).  regs_of: registers per
// thread of a layout's kernel; fits: whether its blocks run on the chip at once, which
// has the last word (when it refuses the best layout, the best one of another form or
// number of blocks per SM is taken).  forms as for oc_plan.
template <typename Regs, typename Fits>
OcPlan oc_choose(int d, int nx, int ntau, int nsys, bool mixed, bool cheb, bool ex, int nsm, size_t smem_sm,
                 size_t smem_blk, int forms, Regs &&regs_of, Fits &&fits)
{
    constexpr int kMaxBlocks = 4, kForms = 3;
    OcPlan found[kMaxBlocks][kForms] = {};      // best by blocks per SM and form
    double costs[kMaxBlocks][kForms];
    int order[kMaxBlocks][kForms], seen = 0;    // equal costs: the first one met
    const long long P = d == 3 ? (long long)nx * nx : 1;
    constexpr size_t kStatic = kOcStaticSmem;    // static and reserved shared memory per block
    for (int m = 1; m <= kMaxBlocks; ++m) {
        const int G = (int)((long long)nsm * m / nsys) < kOcMaxTiles ? nsm * m / nsys : kOcMaxTiles;
        if (G < 1) continue;
        const int max_threads = kOcMaxThreads / m / 32 * 32;    // whole warps: the kernels sum by warps
        // Tile extents that differ: so = ceil(nx / go), st = ceil(ntau / gt), with the fewest tiles each.
        for (int go = 1; go <= nx && go <= G; ++go) {
            const int so = (nx + go - 1) / go;
            if (go > 1 && (nx + go - 2) / (go - 1) == so) continue;
            for (int st = 1, gt; st <= ntau; st = gt == 1 ? ntau + 1 : (ntau + gt - 2) / (gt - 1)) {
                gt = (ntau + st - 1) / st;
                if ((long long)go * gt > G) continue;
                const long long C = P * so * st, H = P * (2 * st + so);
                for (int form = forms == 2 ? 1 : 0; form < (forms == 3 || ex ? 1 : 3); ++form) {
                    // form 0: columns; 1, 2: tile form with x in shared or global memory
                    int K = 0, sides = 1, thr = 0;
                    size_t sm;
                    // Clocks of one iteration on an SM holding m tiles, fitted to times over so, st
                    // and m; what counts is their order.  Times of 500 drawn lattices over this cost,
                    // median (8 in 10 of them): FP64 columns 1.03 (0.97 - 1.10), tiles 0.94 (0.87 -
                    // 1.06); mixed columns 1.25 (1.18 - 1.35), tiles 1.26 (1.04 - 1.37).  Of a whole
                    // preconditioned step (n = 8): columns 10.6 (9.5 - 12.9), tiles 12.7 (10.7 - 15.8).
                    double cost;
                    if (form == 0) {
                        if (!cols_candidate(d, P, nx, go, so, st, mixed, cheb, ex, &K, &sides, &thr)) continue;
                        sm = oc_cols_smem(d, mixed, cheb, ex, K, thr);
                        const double warps = (thr - 32) / 32;
                        cost = (mixed ? 5000.0 : 7000.0) + 20.0 * go * gt + (sides == 2 ? 2500.0 : 0.0) +
                               (cheb && K > 2 ? 1500.0 : 0.0) + (K == 8 ? (mixed ? 1500.0 : 2500.0) : 0.0) +
                               (mixed ? 300.0 : 500.0) * st +
                               m * (warps * st * (mixed ? 30.0 : 16.0 * (d == 1 ? 12 : 20)) + 0.5 * H);
                    } else {
                        sm = oc_smem(d, P, so, st, mixed, cheb, form == 2);
                        // FP32: a thread per item of 4 slices.  FP64: more than 8 warps only lengthen
                        // the block's barriers while a thread has few sites.
                        const long long items = mixed ? P * so * ((st + 3) / 4) : C;
                        thr = items < max_threads ? (int)((items + 31) / 32 * 32) : max_threads;
                        if (!mixed && thr > 256 && C <= 2048) thr = 256;
                        if (thr < 64) thr = 64;
                        if (mixed) {
                            cost = 2600.0 + 20.0 * go * gt + m * (1.6 * C + 1.6 * items + 0.7 * H);
                            if (cost < 11000.0) cost = 11000.0;
                        } else {
                            cost = 9500.0 + 20.0 * go * gt + m * ((d == 1 ? 6.5 : 13.0) * C + 0.7 * H);
                        }
                        if (form == 2) cost += 0.5 * m * C;
                    }
                    if (sm > kOcMaxSmem || sm + kStatic > smem_blk || (sm + kStatic) * m > smem_sm) continue;
                    OcPlan &best = found[m - 1][form];
                    if (best.ok && cost >= costs[m - 1][form]) continue;
                    OcPlan p = {};
                    p.ok = 1;
                    p.go = go;
                    p.gt = gt;
                    p.so = so;
                    p.st = st;
                    p.x_global = form == 2;
                    p.mixed = mixed;
                    p.cheb = cheb;
                    p.ex = ex;
                    p.cols = K;
                    p.sides = sides;
                    p.smem = sm;
                    p.threads = thr;
                    // Co-resident, as its blocks wait on one another: by registers (a
                    // warp's are one of the 4 partitions', 16384 each) and shared memory.
                    const int regs = (regs_of(p) + 7) / 8 * 8;
                    const int parts = (thr / 32 + 3) / 4;    // warps of a block per partition
                    if (regs <= 0 || 16384 / (regs * 32) / parts < m) continue;
                    costs[m - 1][form] = cost;
                    order[m - 1][form] = seen++;
                    best = p;
                }
            }
        }
    }
    for (;;) {
        int bm = -1, bf = 0;
        for (int m = 0; m < kMaxBlocks; ++m)
            for (int f = 0; f < kForms; ++f) {
                if (!found[m][f].ok) continue;
                if (bm < 0 || costs[m][f] < costs[bm][bf] ||
                    (costs[m][f] == costs[bm][bf] && order[m][f] < order[bm][bf])) {
                    bm = m;
                    bf = f;
                }
            }
        if (bm < 0) return OcPlan{};
        if (fits(found[bm][bf])) return found[bm][bf];
        found[bm][bf].ok = 0;
    }
}

}  // namespace hh
