// On-chip CG engine, column form: the vectors of a tile in registers.
//
// The engine of hh_onchip.cu with the same tiles, packets and sums, for tiles
// whose row of spatial sites is at most one block wide: a thread owns one
// spatial site and its K time slices (at most) of the tile, and keeps r, p, t,
// x and the links of that column in registers (but for some spills, below).  The time neighbours of a site
// are then in the same thread, the row before the tile and the one after it
// are read from their packets straight into registers, and shared memory only
// carries the 2d spatial neighbours, at constant strides.  The threads at the
// tile's o edges fetch the halo columns, one each, or both when the tile has one
// o position (SIDES).  Warp 0 does nothing but wait for sums, decide and
// publish; the other warps hand it their partial sums at a barrier they do not
// wait on.
//
// Why: with a few warps per SM each instruction is 4-8 clocks of the chain exchange -
// barrier - phase - sum that bounds it, and the index arithmetic, edge tests and
// addresses of the shared-memory form are most of its instructions.  Counted over
// 200-step solves with two right-hand sides, thread instructions per site and
// iteration (polls and the control warp included): 12^3 x 64 mixed 164, tile form
// 479; 8^3 x 40 FP64 380, tile form 962.  Measured, us per iteration, two
// right-hand sides, against the tile form (and the grid engine): d = 1 32 x 64
// FP64 4.3, 4.8 (11.5), mixed 3.5, 4.3 (9.8); 731 x 96 mixed 4.6, 5.5 (11.3);
// 1024 x 128 mixed 5.4, 5.9 (10.9); d = 3 8^3 x 40 FP64 6.5, 7.3 (17.1);
// 12^3 x 64 mixed 4.9, 6.8 (14.7).  The tile form stays for tiles that do not fit
// (wider rows, more slices than registers) and where it is faster: 16^3 x 64
// mixed, one right-hand side, 6.7 against 8.4.  Not all of a column stays in registers:
// the FP64 kernels of 4 slices spill 16 to 108 bytes a thread (52 to 120 in the
// exact-block form, 124 to 212 preconditioned), of 8 slices 220 to 284, the preconditioned
// one of 2 slices with two halo columns 40, and the FP32 ones of 8 slices 8 to 140.  The exact-block form of M to first order exists in this form
// only, with at most 4 slices: observables on 10^3 x 48 FP64, 4 noise vectors, 38.6 ms
// on the grid engine (scalar loops that recompute the hops), 22 here; that is the most
// slices 10^3 can have with 4 vectors.
#include "hh_onchip_dev.cuh"

namespace hh {

namespace {

// Barriers (the roles run different code, so all of them are numbered ones).
constexpr int kBarStage = 1;    // compute warps: a vector is staged
constexpr int kBarSum = 2;      // compute warps arrive, warp 0 waits: partial sums in red
constexpr int kBarAll = 3;      // the whole block

__device__ __forceinline__ void bar_sync(int id, int n)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

__device__ __forceinline__ void bar_arrive(int id, int n)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// Barrier of the whole block: whether any thread comes with bad set.
__device__ __forceinline__ bool bar_all(int n, bool bad)
{
    int any;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %3, 0;\n\tbar.red.or.pred q, %1, %2, p;\n\t"
                 "selp.s32 %0, 1, 0, q;\n\t}"
                 : "=r"(any)
                 : "r"(kBarAll), "r"(n), "r"((int)bad)
                 : "memory");
    return any != 0;
}

// What the two roles share.
template <typename T>
struct ColShared {
    EngSystem sys;
    EngState st;
    ISum red[kColMaxThreads / 32];
    double redd[kColMaxThreads / 32];   // signed sums
    double tolbb, dmax;                 // tol^2 |b|^2 and delta^2 maxr2 of the fast decision
    T scal;                             // beta or alpha of the phase about to run
    int restart;                        // beta = 0: p starts anew
    int hand;                           // a mixed system leaves for FP64 steps in the grid engine
};

// Warp 0: waits for the tiles' sums, decides, hands scalars and modes over, and
// publishes the block's sums.  Follows the same sequence of modes and barriers
// as the compute warps; returns the phases run.
template <typename T, bool CHEB>
__device__ __forceinline__ uint32_t control_warp(const OcLaunch &L, ColShared<T> &S, int sid, int tile)
{
    constexpr bool MIXED = sizeof(T) == 4;
    const EngSystem &Y = S.sys;
    const int tid = (int)threadIdx.x, nthr = (int)blockDim.x, ncw = (nthr >> 5) - 1;
    const int tiles = L.go * L.gt;
    EngCtl *const ctl = L.ctl;
    Raw16 *const slots = (Raw16 *)L.slots + (size_t)sid * 2 * kOcReplicas * kOcMaxTiles;
    const Raw16 *const my_slots = slots + (size_t)(tile % kOcReplicas) * 2 * kOcMaxTiles;
    const uint32_t ph0 = (uint32_t)L.seq[0];
    uint32_t ph = ph0;
    int par = 0;
    const bool drop = L.drop != 0 && L.drop - 1 == tile && sid == 0;
    const int cheb2 = CHEB ? 2 * Y.cheb_n : 0;

    auto publish_value = [&](double v) {
        if (tid < kOcReplicas && !drop)
            st_raw(slots + (size_t)(2 * tid + par) * kOcMaxTiles + tile,
                   (unsigned long long)__double_as_longlong(v), ph);
    };
    // The block's sum, published under the current phase number.
    auto publish = [&]() {
        bar_sync(kBarSum, nthr);
        ISum a = {0ull, 1};
        if (tid < ncw) a = S.red[tid];
        publish_value(isum_value(warp_isum_parts(a)));
    };
    auto publish_signed = [&]() {
        bar_sync(kBarSum, nthr);
        double v = tid < ncw ? S.redd[tid] : 0.0;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        publish_value(__shfl_sync(0xffffffffu, v, 0));
    };
    auto wait = [&](double &sum) -> bool {
        return sum_slots<true>(my_slots + par * kOcMaxTiles, tiles, ph, ctl, sum);
    };
    // A barrier over the system's tiles that also orders plain global accesses.
    auto tile_barrier = [&]() -> bool {
        ++ph;
        par ^= 1;
        bar_all(nthr, false);
        __threadfence();
        publish_value(0.0);
        __syncwarp();
        double dummy;
        const bool ok = wait(dummy);
        __threadfence();
        return bar_all(nthr, !ok);
    };

    bool stageB = false;
    int pm = MODE_NEW;      // mode of the phases run last
    long long iters = 0;
    for (;;) {
        bool bad = iters >= L.max_iters;
        bool again = false;     // another CG step, its state noted after the barrier
        double sum = 0.0;
        // Between the preconditioner's sub-steps there is no sum.
        const bool inner = CHEB && pm == MODE_PRE && (stageB || S.st.pre_j + 1 < cheb2);
        __syncwarp();
        if (!inner && pm != MODE_NEW) {
            const double ra = S.st.rr_alpha, inv = stageB ? 0.0 : reciprocal(ra);
            const double tolbb = S.tolbb, dmax = MIXED ? S.dmax : 0.0;
            const bool last = S.st.cg_steps + 1 >= Y.maxit || (MIXED && S.st.since_ru + 1 >= Y.stall_window);
            bool ok;
            if (CHEB && pm == MODE_PRE)
                ok = sum_slots<false>(my_slots + par * kOcMaxTiles, tiles, ph, ctl, sum);
            else
                ok = wait(sum);
            if (!ok) {
                bad = true;
            } else if (stageB) {
                const T a = quotient<T>(ra, sum);
                if (tid == 0) S.scal = a;
            } else {
                again = !CHEB && pm == MODE_CG && !last && finite_bits(sum) && greater_nonneg(sum, tolbb) &&
                        !(MIXED && greater_nonneg(dmax, sum));
                if (again) {
                    // The common case of decide(): beta = sum / ra, the quotient by
                    // 1 / ra with (FP64) one residual correction.
                    double beta = sum * inv;
                    if (!MIXED) beta = fma(fma(-beta, ra, sum), inv, beta);
                    if (tid == 0) {
                        S.scal = (T)beta;
                        S.restart = 0;
                        S.st.beta = beta;
                    }
                } else if (tid == 0) {
                    const EngState N = decide(Y, S.st, sum);
                    if (MIXED && N.prec == PREC_FP64 && N.mode != MODE_DONE) {
                        S.hand = 1;
                        if (tile == 0) hand_over(L, Y, sid, S.st, sum);
                    } else {
                        S.st = N;
                        S.scal = (T)N.beta;
                        S.restart = N.beta == 0.0;
                        S.tolbb = Y.tol2 * N.bb;
                        S.dmax = Y.delta2 * N.maxr2;
                    }
                }
            }
        } else if (tid == 0) {
            if (pm == MODE_NEW)
                S.st = decide(Y, S.st, 0.0);
            else if (!stageB)
                S.st.pre_j += 1;
        }
        if (bar_all(nthr, bad)) break;
        if (again && tid == 0) {
            S.st.cg_steps += 1;
            S.st.since_ru += 1;
            if (!MIXED) S.st.fp64_steps += 1;
            S.st.rr_last = sum;
            S.st.rr_alpha = sum;
            if (MIXED && sum > S.st.maxr2) {
                S.st.maxr2 = sum;
                S.dmax = Y.delta2 * sum;
            }
        }
        __syncwarp();
        if (stageB) {
            stageB = false;
            ++ph;
            if (CHEB && pm == MODE_PRE) {
                if (S.st.pre_j == cheb2 - 1) {
                    par ^= 1;
                    publish_signed();
                }
            } else {
                par ^= 1;
                publish();
            }
            continue;
        }
        if (S.hand) break;
        const int mode = S.st.mode;
        if (mode == MODE_DONE) break;
        ++iters;
        if (mode == MODE_INIT) {
            if (pm == MODE_INIT && tile_barrier()) break;
            ++ph;
            par ^= 1;
            publish();
        } else if (mode == MODE_RU) {
            if (tile_barrier() || tile_barrier()) break;
            ++ph;
            par ^= 1;
            publish();
        } else {
            ++ph;
            stageB = true;
            if (!CHEB || mode == MODE_CG) {
                par ^= 1;
                publish();
            }
        }
        pm = mode;
    }
    return ph - ph0;
}

// The compute warps: thread c of them owns the spatial site c of the tile's row.
// EX: the exact-block form of M to first order (link_order 1),
//   (M v)(tau) = v(tau) + (1 + h H) (L v)(tau - 1),  (M^T t)(tau) = t(tau) + L(tau) (1 + h H) t(tau + 1):
// the hops are on the slice before or after, so staged row k holds L v of slice
// k - 1, or t of slice k + 1, and the halo columns are those of these slices.
template <int D, typename T, int K, int SIDES, bool CHEB, bool EX>
__device__ __forceinline__ void compute_warps(const OcLaunch &L, ColShared<T> &S, unsigned char *smem, int sid, int tile)
{
    constexpr bool MIXED = sizeof(T) == 4;
    constexpr int RS = kColStride<D>;
    using PK = Packet<T>;
    using Raw = typename PK::Raw;
    const EngSystem &Y = S.sys;
    T *const Pb = (T *)smem;                        // p, o halo included: slice k at k RS
    T *const Tb = Pb + K * RS;                      // t
    T *const Wb = CHEB ? Tb + K * RS : Pb;          // preconditioner: M's input there (p stays in Pb)
    T *const Ph = EX ? Tb + K * RS : Pb;            // EX: p of the halo columns, and their links
    T *const Lh = EX ? Ph + K * RS : Pb;
    const int tid = (int)threadIdx.x, nthr = (int)blockDim.x, c = tid - 32;
    EngCtl *const ctl = L.ctl;

    // ---- the tile (as in hh_onchip.cu) and this thread's column ----
    const int no = Y.g.nx, ntau = Y.g.ntau, V = Y.g.V;
    const int nx = no, P = D == 3 ? no * no : 1;
    const int io = tile % L.go, it = tile / L.go;
    const int o0 = (int)((long long)io * no / L.go), so = (int)((long long)(io + 1) * no / L.go) - o0;
    const int t0 = (int)((long long)it * ntau / L.gt), st = (int)((long long)(it + 1) * ntau / L.gt) - t0;
    const int row = so * P;
    const bool active = c < row;
    const int ol = active ? c / P : 0, pos = active ? c - ol * P : 0;
    // This thread's halo columns: SIDES = 1: at most one, of its o edge; 2 (so = 1): both.
    const bool isL = active && ol == 0, side = active && (ol == 0 || ol == so - 1);
    int g0 = t0 * V + o0 * P + (active ? c : 0);                   // site of slice 0; + k V
    const int oL = (o0 == 0 ? no - 1 : o0 - 1) * P, oR = (o0 + so == no ? 0 : o0 + so) * P;
    int gs = t0 * V + (isL ? oL : oR) + pos;                       // halo site; + k V
    int gr = t0 * V + oR + pos;                                    // right one (SIDES = 2)
    int gp = (t0 == 0 ? ntau - 1 : t0 - 1) * V + o0 * P + (active ? c : 0);         // slice before the tile
    int gn = (t0 + st == ntau ? 0 : t0 + st) * V + o0 * P + (active ? c : 0);       // slice after it
    HH_CHECK(g0, 0, L.N - (st - 1) * V, BC_NEIGHBOUR);
    HH_CHECK(gs, 0, L.N - (st - 1) * V, BC_NEIGHBOUR);
    HH_CHECK(gr, 0, L.N - (st - 1) * V, BC_NEIGHBOUR);
    HH_CHECK(gp, 0, L.N, BC_NEIGHBOUR);
    HH_CHECK(gn, 0, L.N, BC_NEIGHBOUR);
    const int me = (active ? c : 0) + P;                           // staged index of the column
    const int hidx = isL ? pos : row + P + pos;                    // of its halo column
    int xr = me + 1, xl = me - 1, yp = 0, ym = 0;
    const int zp = me + P, zm = me - P;
    if (D == 3) {
        const int y = pos / nx, x = pos - y * nx;
        xr = x == nx - 1 ? me - (nx - 1) : me + 1;
        xl = x == 0 ? me + (nx - 1) : me - 1;
        yp = y == nx - 1 ? me - (nx - 1) * nx : me + nx;
        ym = y == 0 ? me + (nx - 1) * nx : me - nx;
    }
    // Packets: A (M's input) at these, B (t) L.N further on; slice k is k V further on.
    Raw *const pktA = (Raw *)L.pkt + (size_t)sid * 2 * L.N;
    Raw *p_own = pktA + g0, *p_side = pktA + gs, *p_right = pktA + gr;
    const int d_prev = gp - g0, d_next = gn - g0 + L.N;     // slice before (A) and after (B) from p_own
    // Halo packet of staged row u, from the halo column's slice 0.
    const int s_prev = gp - g0, s_next = gn - g0;           // (the same steps as in the own column)
    auto halo_step = [&](bool after, int u) -> int {
        if (!EX) return u * V;
        if (after) return u + 1 < st ? (u + 1) * V : s_next;
        return u == 0 ? s_prev : (u - 1) * V;
    };

    const T h = (T)Y.h;
    // The preconditioner's M input and z take the registers of p and x, which its
    // sub-steps do not touch: p is then read back from its staging (Pb), x from Xs.
    T r[K], t[K], lk[K], pw[K], xz[K];
    T *const Xs = CHEB ? Wb + K * RS + c : nullptr;     // + k (nthr - 32)
    T lkp = T(0), pp = T(0);    // link and p of the slice before the tile
    {
        const T *const src = MIXED ? (const T *)Y.L32 : (const T *)Y.L64;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            r[k] = t[k] = pw[k] = xz[k] = T(0);
            lk[k] = active && k < st ? __ldg(src + g0 + k * V) : T(0);
        }
        if (active) lkp = __ldg(src + gp);
        if (EX && side)
#pragma unroll
            for (int k = 0; k < SIDES * K; ++k) {
                const int u = k < K ? k : k - K;
                if (u < st) Lh[(k < K ? k * RS + hidx : u * RS + row + P + pos)] = __ldg(src + (k < K ? gs : gr) + halo_step(false, u));
            }
    }
    uint32_t ph = (uint32_t)L.seq[0];

    // This warp's part of the block's sum; warp 0 publishes it.
    auto give_sum = [&](auto v) {
        const ISum a = warp_isum(v);
        if ((tid & 31) == 0) S.red[(tid >> 5) - 1] = a;
        bar_arrive(kBarSum, nthr);
    };
    auto give_signed = [&](double v) {
        v = warp_sum(v);
        if ((tid & 31) == 0) S.redd[(tid >> 5) - 1] = v;
        bar_arrive(kBarSum, nthr);
    };
    auto tile_barrier = [&]() -> bool {
        ++ph;
        bar_all(nthr, false);
        return bar_all(nthr, false);
    };
    // The halo of the A (off = 0) or B (off = L.N) packets: this thread's halo
    // columns (hv) and the slice at p_own + d_time (tv).  The addresses are formed anew in
    // every phase (keep_base): kept, they would be dozens of registers.
    T hv[SIDES * K], tv = T(0);
    auto keep_base = [&]() {
        asm volatile("" : "+l"(p_own), "+l"(p_side));
        if (SIDES == 2) asm volatile("" : "+l"(p_right));
    };
    auto fetch_halo = [&](int off, int d_time) -> bool {
        constexpr int U = SIDES * K + 1;
        // At most B packets at a time: an FP64 one is four registers until it is ready.
        constexpr int B = MIXED || U <= 5 ? U : 5;
        keep_base();
        auto where = [&](int u) -> const Raw * {
            return u == U - 1 ? p_own + d_time
                   : u < K   ? p_side + off + halo_step(off != 0, u)
                             : p_right + off + halo_step(off != 0, u - K);
        };
        auto wanted = [&](int u) -> bool { return u == U - 1 ? active : side && (u < K ? u : u - K) < st; };
        SpinClock clk;
#pragma unroll
        for (int u0 = 0; u0 < U; u0 += B) {
            Raw raw[B];
            unsigned pend = 0;
#pragma unroll
            for (int i = 0; i < B; ++i)
                if (u0 + i < U && wanted(u0 + i)) raw[i] = PK::load(where(u0 + i));
#pragma unroll
            for (int i = 0; i < B; ++i)
                if (u0 + i < U && wanted(u0 + i) && !PK::ready(raw[i], ph)) pend |= 1u << i;
            while (pend) {
                if (!clk.tick(ctl)) return false;
#pragma unroll
                for (int i = 0; i < B; ++i)
                    if (u0 + i < U && (pend & (1u << i))) {
                        raw[i] = PK::load(where(u0 + i));
                        if (PK::ready(raw[i], ph)) pend &= ~(1u << i);
                    }
            }
#pragma unroll
            for (int i = 0; i < B; ++i)
                if (u0 + i < U) {
                    const T v = wanted(u0 + i) ? PK::value(raw[i]) : T(0);
                    if (u0 + i == U - 1)
                        tv = v;
                    else
                        hv[u0 + i < U - 1 ? u0 + i : 0] = v;
                }
        }
        return true;
    };
    // This thread's halo columns of a staged vector: the fetched values, or
    // (update) fetched + b times what is there.
    auto stage_halo = [&](T *v, bool update, T b) {
        if (side) {
#pragma unroll
            for (int k = 0; k < SIDES * K; ++k)
                if ((k < K ? k : k - K) < st) {
                    T *const cell = v + (k < K ? k * RS + hidx : (k - K) * RS + row + P + pos);
                    *cell = update ? fma(b, *cell, hv[k]) : hv[k];
                }
        }
    };
    auto hop = [&](const T *v) -> T {
        if (D == 1) return v[xr] + v[xl];
        return (v[xr] + v[xl]) + ((v[yp] + v[ym]) + (v[zp] + v[zm]));
    };
    auto publish_A = [&](int k, T v) {
        if (side || k == st - 1) PK::store(p_own + k * V, v, ph);
    };
    // (M^T t) at slice k.
    auto mt = [&](int k) -> T {
        const T nv = k + 1 < K && k + 1 < st ? t[k + 1 < K ? k + 1 : k] : tv;
        if (EX) return fma(lk[k], fma(h, hop(Tb + k * RS), nv), t[k]);
        return fma(lk[k], nv, fma(-h, hop(Tb + k * RS), t[k]));
    };

    bool stageB = false;
    int pm = MODE_NEW;      // mode of the phases run last
    int pj = 0;             // preconditioner sub-step (S.st.pre_j may already be the next)
    const int cheb2 = CHEB ? 2 * Y.cheb_n : 0;
    for (;;) {
        // ---- exchange: the halo, while warp 0 waits for the sum ----
        bool bad = false;
        if (pm != MODE_NEW) {
            bad = !fetch_halo(stageB ? L.N : 0, stageB ? d_next : d_prev);
            if (stageB) {
                stage_halo(Tb, false, T(0));
                if (EX && active) Tb[(st - 1) * RS + me] = tv;
            }
        }
        if (bar_all(nthr, bad)) break;

        if (stageB) {
            stageB = false;
            ++ph;
            keep_base();
            if (CHEB && pm == MODE_PRE) {
                // Factor update of a preconditioner sub-step.
                const int j = pj, kf = j >> 1;
                const bool last = j == cheb2 - 1;
                const T invlam = (T)__ldg(Y.cheb), a = (T)__ldg(Y.cheb + 2 + 3 * kf);
                const T b2 = (T)__ldg(Y.cheb + 3 + 3 * kf), invq = (T)__ldg(Y.cheb + 4 + 3 * kf);
                const T scale = last ? (T)__ldg(Y.cheb + 1) : T(1);
                double acc = 0.0;
                if (active) {
#pragma unroll
                    for (int k = 0; k < K; ++k)
                        if (k < st) {
                            const T y = mt(k), v = pw[k];
                            T u;
                            if ((j & 1) == 0) {
                                xz[k] = v;
                                u = fma(y, invlam, -a * v);
                            } else {
                                u = fma(y, invlam, fma(-a, v, b2 * xz[k])) * invq * scale;
                                if (last) acc = fma((double)r[k], (double)u, acc);
                            }
                            pw[k] = u;
                            publish_A(k, u);
                        }
                }
                if (last) give_signed(acc);
                continue;
            }
            // ---- r -= alpha M^T t, |r|^2; then x += alpha p while the sum travels ----
            const T alpha = S.scal;
            T acc = T(0);
            if (active) {
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (k < st) {
                        r[k] = fma(-alpha, mt(k), r[k]);
                        acc = fma(r[k], r[k], acc);
                        publish_A(k, r[k]);
                        if (CHEB) pw[k] = r[k];
                    }
            }
            give_sum(acc);
#pragma unroll
            for (int k = 0; k < K; ++k) {
                if (!CHEB)
                    xz[k] = fma(alpha, pw[k], xz[k]);
                else if (active && k < st)
                    Xs[k * (nthr - 32)] = fma(alpha, Pb[k * RS + me], Xs[k * (nthr - 32)]);
            }
            continue;
        }

        if (S.hand) break;
        const int mode = S.st.mode;
        if (mode == MODE_DONE) break;

        if (mode == MODE_INIT) {
            const bool zero = !(Y.x0_given && !S.st.no_guess);
            // A second INIT replaces the first one's packets: only once every
            // block has read them.
            if (pm == MODE_INIT && tile_barrier()) break;
            ++ph;
            keep_base();
            double acc = 0.0;
            if (active) {
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (k < st) {
                        const int g = g0 + k * V;
                        const double b = __ldg(Y.b + g);
                        acc = fma(b, b, acc);
                        r[k] = (T)b;
                        if (CHEB) pw[k] = (T)b;
                        publish_A(k, (T)b);
                        if (MIXED) {
                            if (zero) Y.x[g] = 0.0;
                            xz[k] = T(0);
                        } else {
                            const T x0 = zero ? T(0) : (T)Y.x[g];
                            if (CHEB)
                                Xs[k * (nthr - 32)] = x0;
                            else
                                xz[k] = x0;
                        }
                    }
            }
            give_sum(acc);
            pm = mode;
            continue;
        }

        if (mode == MODE_RU) {
            // x64 of the tile to memory (mixed: with the FP32 part added).
            if (active) {
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (k < st) {
                        const int g = g0 + k * V;
                        if (MIXED) {
                            Y.x[g] += (double)xz[k];
                            xz[k] = T(0);
                        } else {
                            Y.x[g] = (double)(CHEB ? Xs[k * (nthr - 32)] : xz[k]);
                        }
                    }
            }
            if (tile_barrier()) break;
            if (active)
#pragma unroll 1
                for (int k = 0; k < st; ++k) {
                    const int g = g0 + k * V;
                    Nbr nb;
                    neighbours(Y.g, g, nb);
                    Y.t[g] = EX ? stencil_M_ex<double>(Y.g, Y.h, Y.L64, Y.x, g, nb, 1)
                                : stencil_M<double>(Y.g, Y.h, Y.L64, Y.x, g, nb);
                }
            if (tile_barrier()) break;
            ++ph;
            keep_base();
            double acc = 0.0;
            if (active) {
#pragma unroll 1
                for (int k = 0; k < st; ++k) {
                    const int g = g0 + k * V;
                    Nbr nb;
                    neighbours(Y.g, g, nb);
                    const double res =
                        __ldg(Y.b + g) - (EX ? stencil_MT_ex<double>(Y.g, Y.h, Y.L64, Y.t, g, nb, 1)
                                             : stencil_MT<double>(Y.g, Y.h, Y.L64, Y.t, g, nb));
                    acc = fma(res, res, acc);
                    if (MIXED) Y.r[g] = res;
                    Tb[k * RS + me] = (T)res;     // to the registers below (staged t is not read any more)
                    publish_A(k, (T)res);
                }
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (k < st) {
                        r[k] = Tb[k * RS + me];
                        if (CHEB) pw[k] = r[k];
                    }
            }
            give_sum(acc);
            pm = mode;
            continue;
        }

        // ---- t = M v of a preconditioner sub-step (v in w) or, in a CG step, of
        // p = r + beta p (r: z with the preconditioner), formed on the tile and
        // its halo ----
        const bool cg = !CHEB || mode == MODE_CG;
        ++ph;
        stageB = true;
        pj = pm == MODE_PRE ? pj + 1 : 0;
        pm = mode;
        keep_base();
        T vp = tv;              // the slice before the tile
        T *const Sb = cg ? Pb : Wb;
        T pv[CHEB ? K : 1];     // p (preconditioner: pw holds z)
        if (cg) {
            const bool restart = S.restart != 0;
            const T beta = S.scal;
            if (CHEB) {
#pragma unroll
                for (int k = 0; k < K; ++k)
                    if (active && k < st)
                        pv[CHEB ? k : 0] = restart ? pw[k] : fma(beta, Pb[k * RS + me], pw[k]);
            } else {
#pragma unroll
                for (int k = 0; k < K; ++k) pw[k] = restart ? r[k] : fma(beta, pw[k], r[k]);
            }
            vp = pp = restart ? tv : fma(beta, pp, tv);
            // The halo of p is kept where it is staged (EX: L p is staged).
            stage_halo(EX ? Ph : Pb, !restart, beta);
            if (EX && side)
#pragma unroll
                for (int k = 0; k < SIDES * K; ++k) {
                    const int u = k < K ? k : k - K, cell = k < K ? k * RS + hidx : u * RS + row + P + pos;
                    if (u < st) Pb[cell] = Lh[cell] * Ph[cell];
                }
        } else {
            stage_halo(Wb, false, T(0));
        }
        auto v_of = [&](int k) -> T { return CHEB && cg ? pv[CHEB ? k : 0] : pw[k]; };
        if (active) {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < st) Sb[k * RS + me] = !EX ? v_of(k) : k == 0 ? lkp * vp : lk[k > 0 ? k - 1 : 0] * v_of(k > 0 ? k - 1 : 0);
        }
        bar_sync(kBarStage, nthr - 32);
        T acc = T(0);
        if (active) {
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (k < st) {
                    const T vm = k == 0 ? vp : v_of(k > 0 ? k - 1 : 0);
                    const T lm = k == 0 ? lkp : lk[k > 0 ? k - 1 : 0];
                    if (EX)
                        t[k] = v_of(k) + fma(h, hop(Sb + k * RS), lm * vm);
                    else
                        t[k] = fma(lm, vm, fma(-h, hop(Sb + k * RS), v_of(k)));
                    acc = fma(t[k], t[k], acc);
                    if (!EX)
                        Tb[k * RS + me] = t[k];
                    else if (k > 0)
                        Tb[(k - 1) * RS + me] = t[k];
                    if (side || k == 0) PK::store(p_own + L.N + k * V, t[k], ph);
                }
        }
        if (cg) give_sum(acc);
    }

    if (!MIXED && active && S.st.mode == MODE_DONE) {
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < st) Y.x[g0 + k * V] = (double)(CHEB ? Xs[k * (nthr - 32)] : xz[k]);
    }
}

template <int D, typename T, int K, int SIDES, bool CHEB, bool EX = false>
__global__ void __launch_bounds__(col_max_threads(sizeof(T), K), 1) k_onchip_cols(const OcLaunch L)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ ColShared<T> S;
    const int tid = (int)threadIdx.x, nthr = (int)blockDim.x;
    const int tiles = L.go * L.gt;
    const int sid = (int)blockIdx.x / tiles, tile = (int)blockIdx.x - sid * tiles;
    for (int j = tid; j < (int)(sizeof(EngSystem) / 4); j += nthr) ((int *)&S.sys)[j] = ((const int *)(L.sys + sid))[j];
    if (tid == 0) {
        S.st = L.state[0][sid];
        S.hand = 0;
        S.restart = 1;
        S.scal = T(0);
        S.tolbb = S.dmax = 0.0;
    }
    __syncthreads();
    if (tid >= 32) {
        compute_warps<D, T, K, SIDES, CHEB, EX>(L, S, smem, sid, tile);
        return;
    }
    const uint32_t phases = control_warp<T, CHEB>(L, S, sid, tile);
    __syncwarp();
    if (tid == 0) {
        if (tile == 0 && S.st.mode == MODE_DONE) {
            L.state[0][sid] = S.st;
            L.state[1][sid] = S.st;
        }
        atomicMax(L.seq + 1, L.seq[0] + (unsigned long long)phases + 1ull);
    }
}

template <int D, int SIDES>
const void *cols_kernel_d(bool mixed, bool cheb, bool ex, int K)
{
    if (ex) {
        if (mixed) return K <= 2 ? (const void *)k_onchip_cols<D, float, 2, SIDES, false, true>
                                 : (const void *)k_onchip_cols<D, float, 4, SIDES, false, true>;
        return K <= 2 ? (const void *)k_onchip_cols<D, double, 2, SIDES, false, true>
                      : (const void *)k_onchip_cols<D, double, 4, SIDES, false, true>;
    }
    if (mixed) {
        if (K <= 2) return (const void *)k_onchip_cols<D, float, 2, SIDES, false>;
        if (K <= 4) return (const void *)k_onchip_cols<D, float, 4, SIDES, false>;
        return (const void *)k_onchip_cols<D, float, 8, SIDES, false>;
    }
    if (cheb) {
        if (K <= 2) return (const void *)k_onchip_cols<D, double, 2, SIDES, true>;
        return (const void *)k_onchip_cols<D, double, 4, SIDES, true>;
    }
    if (K <= 2) return (const void *)k_onchip_cols<D, double, 2, SIDES, false>;
    if (K <= 4) return (const void *)k_onchip_cols<D, double, 4, SIDES, false>;
    return (const void *)k_onchip_cols<D, double, 8, SIDES, false>;
}

}  // namespace

const void *oc_cols_kernel(int d, bool mixed, bool cheb, bool ex, int K, int sides)
{
    if (d == 1) return cols_kernel_d<1, 1>(mixed, cheb, ex, K);
    return sides == 1 ? cols_kernel_d<3, 1>(mixed, cheb, ex, K) : cols_kernel_d<3, 2>(mixed, cheb, ex, K);
}

}  // namespace hh
