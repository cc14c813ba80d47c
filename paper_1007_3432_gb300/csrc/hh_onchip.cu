// On-chip CG engine (Sec. 4.1: CG on Q = M^T M, the vectors in shared memory).
//
// A CG iteration is two phases, t = M p with |t|^2 and the update with
// q = M^T t and |r|^2, each ending in a sum over all tiles of the system.
// On lattices of a few thousand to a million sites the phases of the grid
// engine (hh_engine.cu) take 4-6 us whatever the lattice, most of it one
// chain of memory round trips: release fence, signal, poll, acquire fence,
// reload of every vector from L2.  Here
//  * a block keeps r, p, t, x and the links of its tile in shared memory;
//  * the boundary sites of t and of r are written as packets {value, phase
//    number}, one 16-byte (FP64) or 8-byte (FP32) access each, and readers poll the
//    packets they need: the value is there when its phase number is, so no
//    fence orders it.  The search direction is not exchanged: a block keeps
//    p on its halo and updates it there, p = r + beta p, from the r packets,
//    which travel while |r|^2 is being summed;
//  * warp 0 polls the tiles' partial sums (packets too), decides, and hands
//    the scalar over at a block barrier, while the other warps fetch the halo.
// The preconditioner's sub-steps have no sums, so their phases wait for the
// neighbouring tiles only.
//
// Overwriting a packet needs no acknowledgement.  A site's r packet (phase n)
// is next written after its block has read the t packets (phase n + 1) of the
// sites around it, and those were published after their blocks had read the r
// packet; likewise for t, and for partial sums, whose two parities
// alternate.  (Where a phase ends in a sum, the sum alone orders them: every tile
// has read the packets of the phase before it gives its part.)  The reliable update exchanges x and t in global memory between
// barriers made of the same sums with fences around them.
//
// What bounds it: the chain exchange - barrier - phase - block sum, run by a few
// warps (FP64 from about 800 sites per SM: the FP64 pipe, 16 clocks per warp
// instruction).  Measured against the grid engine, us per iteration: d = 1
// 1024 x 128 FP64, 2 right-hand sides, 10.8 (15.6), 1024 x 512 29.3 (30.1), mixed 9.1
// (14.3), a degree-8 preconditioned step on 256 x 256 90 (197); d = 3 16^3 x 64
// mixed, one, 6.7 (15.1), two, 7.6 (16.5), 20^3 x 96 mixed, one, 10.4 (18.0).  It was
// faster on all of 800 lattices with 1 to 8 right-hand sides drawn among those that fit
// (4^3 to 24^3, chains of 16 to 2048 sites): by 1.1 at least (14^3 x 99 FP64, two:
// 29.8 against 32.8), at the median by 2.1 in FP64, 2.7 mixed, 3.2 preconditioned and
// 2.9 to 3.7 in the exact-block form; whole solves of the smallest (2 x 2 and up) by
// 1.6 to 3.8.  So a lattice that fits runs here.  Tiles whose column fits a
// thread's registers run in hh_onchip_cols.cu.
//
// Every wait is bounded (EngCtl::timeout_ns); on expiry the block records
// HH_ETIMEOUT, and all its threads leave at the next block barrier.
#include <atomic>

#include "hh_onchip_dev.cuh"
#include "hh_onchip_plan.cuh"

namespace hh {

namespace {

// ---------------------------------------------------------------------------
// The kernel.  D: lattice dimension; T: type of the CG steps (float: mixed
// precision, reliable updates in FP64); CHEB: Chebyshev-preconditioned (FP64).
// ---------------------------------------------------------------------------
template <int D, typename T, bool CHEB>
__global__ void __launch_bounds__(kOcMaxThreads, 1) k_onchip(const OcLaunch L)
{
    constexpr bool MIXED = sizeof(T) == 4;
    using PK = Packet<T>;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ EngSystem s_sys;
    __shared__ EngState s_st;
    __shared__ ISum s_red[kOcMaxThreads / 32];
    __shared__ double s_redd[kOcMaxThreads / 32];    // signed sums
    __shared__ T s_scal;            // beta or alpha of the phase about to run
    __shared__ int s_restart;       // beta = 0: p starts anew
    __shared__ double s_tolbb, s_dmax;   // tol^2 |b|^2 and delta^2 maxr2 of the fast decision
    __shared__ int s_hand;          // a mixed system leaves for FP64 steps in the grid engine

    const int tid = (int)threadIdx.x, nthr = (int)blockDim.x;
    const int tiles = L.go * L.gt;
    const int sid = (int)blockIdx.x / tiles, tile = (int)blockIdx.x - sid * tiles;
    EngCtl *const ctl = L.ctl;
    for (int j = tid; j < (int)(sizeof(EngSystem) / 4); j += nthr) ((int *)&s_sys)[j] = ((const int *)(L.sys + sid))[j];
    if (tid == 0) {
        s_st = L.state[0][sid];
        s_hand = 0;
    }
    __syncthreads();
    const EngSystem &Y = s_sys;

    // ---- the tile: o in [o0, o0 + so), tau in [t0, t0 + st), P sites each.
    // Compact index s = (tl so + ol) P + pos; extended index with one o column on
    // each side, e = (tl (so + 2) + ol + 1) P + pos.
    const int no = Y.g.nx, ntau = Y.g.ntau, V = Y.g.V;
    const int nx = no, P = D == 3 ? no * no : 1;
    const int io = tile % L.go, it = tile / L.go;
    const int o0 = (int)((long long)io * no / L.go), so = (int)((long long)(io + 1) * no / L.go) - o0;
    const int t0 = (int)((long long)it * ntau / L.gt), st = (int)((long long)(it + 1) * ntau / L.gt) - t0;
    const int row = so * P, RS = (so + 2) * P, C = st * row;
    const int gbase = t0 * V + o0 * P, gstep = V - row;     // site of s: gbase + s + tl gstep
    const int oL = (o0 == 0 ? no - 1 : o0 - 1) * P, oR = (o0 + so == no ? 0 : o0 + so) * P;
    const int tP = (t0 == 0 ? ntau - 1 : t0 - 1) * V + o0 * P;          // row before the tile
    const int tN = (t0 + st == ntau ? 0 : t0 + st) * V + o0 * P;        // row after it
    const FastDiv f_row = make_fastdiv((uint32_t)row), f_P = make_fastdiv((uint32_t)P);

    // ---- shared memory (sizes of the largest tile; see oc_smem) ----
    const int maxC = L.so * L.st * P, maxE = (L.so + 2) * (L.st + 1) * P, maxL = L.so * (L.st + 1) * P;
    T *const Pb = (T *)smem;            // p: rows -1 .. st - 1, extended
    T *const Tb = Pb + maxE;            // t: rows 0 .. st, extended
    T *const Sb = Tb + maxE;            // as p: r, or with the preconditioner M's input
    T *const Lb = Sb + maxE;            // links: rows -1 .. st - 1, compact
    T *q = Lb + maxL;
    T *const Xb = q;                    // x (x32), compact, unless it stays in global memory
    if (!L.x_global) q += maxC;
    T *const Rb = q;                    // preconditioner: r and z, compact
    T *const Zb = q + (CHEB ? maxC : 0);
    q += CHEB ? 2 * maxC : 0;
    unsigned char *const fl = (unsigned char *)q;    // d = 3: x-y edges of each spatial site of the row
    T *const Xg = MIXED ? (T *)Y.x32 : (T *)Y.x;

    unsigned char *const pktA = L.pkt + (size_t)sid * 2 * L.N * sizeof(typename PK::Raw);
    unsigned char *const pktB = pktA + (size_t)L.N * sizeof(typename PK::Raw);
    // Partial sums: kOcReplicas copies, each read by every kOcReplicas-th block.
    Raw16 *const slots = (Raw16 *)L.slots + (size_t)sid * 2 * kOcReplicas * kOcMaxTiles;
    const Raw16 *const my_slots = slots + (size_t)(tile % kOcReplicas) * 2 * kOcMaxTiles;

    const T h = (T)Y.h;
    if (D == 3)
        for (int s = tid; s < row; s += nthr) {
            const int pos = s - (int)fd_div((uint32_t)s, f_P) * P;
            const int y = pos / nx, x = pos - y * nx;
            fl[s] = (unsigned char)((x == 0) | (x == nx - 1) << 1 | (y == 0) << 2 | (y == nx - 1) << 3);
        }
    for (int j = tid; j < C + row; j += nthr) {
        // row -1 first, then the tile's rows
        const int s = j - row;
        int g = j < row ? tP + j : gbase + s + (int)fd_div((uint32_t)s, f_row) * gstep;
        HH_CHECK(g, 0, L.N, BC_NEIGHBOUR);
        Lb[j] = MIXED ? (T)__ldg(Y.L32 + g) : (T)__ldg(Y.L64 + g);
    }
    // The corners of the extended arrays are never read; p is updated over them too.
    for (int j = tid; j < maxE; j += nthr) Pb[j] = Sb[j] = T(0);

    // ---- phase counter, sums ----
    uint32_t ph = (uint32_t)L.seq[0];
    const uint32_t ph0 = ph;
    int par = 0;        // parity of the partial-sum packets
    const bool drop = L.drop != 0 && L.drop - 1 == tile && sid == 0;
    const int nwarp = nthr >> 5;

    // Publishes the block's sum of v under the current phase number (every thread
    // calls it; its barrier follows all of the block's writes of the phase).
    auto publish_value = [&](double v) {
        if (tid < kOcReplicas && !drop)
            st_raw(slots + (size_t)(2 * tid + par) * kOcMaxTiles + tile,
                   (unsigned long long)__double_as_longlong(v), ph);
    };
    auto publish = [&](auto v) {
        const ISum a = warp_isum(v);
        if ((tid & 31) == 0) s_red[tid >> 5] = a;
        __syncthreads();
        if (tid < 32) {
            ISum b = {0ull, 1};
            if (tid < nwarp) b = s_red[tid];
            publish_value(isum_value(warp_isum_parts(b)));
        }
    };
    // The same for a sum of either sign.
    auto publish_signed = [&](double v) {
        v = warp_sum(v);
        if ((tid & 31) == 0) s_redd[tid >> 5] = v;
        __syncthreads();
        if (tid < 32) {
            double w = tid < nwarp ? s_redd[tid] : 0.0;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
            publish_value(__shfl_sync(0xffffffffu, w, 0));
        }
    };
    // A barrier over the system's tiles that also orders plain global accesses.
    // Returns true when a wait ran out.
    auto tile_barrier = [&]() -> bool {
        ++ph;
        par ^= 1;
        __syncthreads();
        bool bad = false;
        if (tid < 32) {
            __threadfence();
            if (tid < kOcReplicas && !drop) st_raw(slots + (size_t)(2 * tid + par) * kOcMaxTiles + tile, 0ull, ph);
            __syncwarp();
            double dummy;
            bad = !sum_slots<true>(my_slots + par * kOcMaxTiles, tiles, ph, ctl, dummy);
            __threadfence();
        }
        return __syncthreads_or(bad ? 1 : 0) != 0;
    };

    const int H2 = 2 * st * P, HA = H2 + row;
    const FastDiv f_2P = make_fastdiv((uint32_t)(2 * P));
    // Halo threads: all but warp 0 (which waits for the sums) when there are others.
    const int hb = nwarp > 1 ? tid - 32 : tid, hn = nwarp > 1 ? nthr - 32 : nthr;
    // The halo of the packets in buf: o columns of the tile's rows into side (extended),
    // then the row at site grow into rdst.
    auto fetch_halo = [&](const unsigned char *buf, T *side, T *rdst, int grow) -> bool {
        constexpr int U = 4;
        bool ok = true;
        if (hb < 0) return ok;
        if constexpr (MIXED) {
            // Up to U slices of one column site at a time, then the row.
#pragma unroll 1
            for (int i = hb; i < 2 * P * ((st + U - 1) / U) && ok; i += hn) {
                const int q4 = (int)fd_div((uint32_t)i, f_2P), cs = i - q4 * 2 * P, k0 = q4 * U;
                int g = (t0 + k0) * V + (cs < P ? oL + cs : oR + cs - P);
                T *dst = side + k0 * RS + (cs < P ? cs : RS - 2 * P + cs);
                HH_CHECK(g, 0, L.N, BC_NEIGHBOUR);
                int hg[U];
                T v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) hg[u] = k0 + u < st ? g + u * V : -1;
                ok = fetch<T, U>(buf, hg, ph, v, ctl);
#pragma unroll
                for (int u = 0; u < U; ++u, dst += RS)
                    if (hg[u] >= 0) *dst = v[u];
            }
#pragma unroll 1
            for (int j = hb; j < row && ok; j += U * hn) {
                int g = grow + j;
                HH_CHECK(g, 0, L.N, BC_NEIGHBOUR);
                int hg[U];
                T v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) hg[u] = j + u * hn < row ? g + u * hn : -1;
                ok = fetch<T, U>(buf, hg, ph, v, ctl);
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (hg[u] >= 0) rdst[j + u * hn] = v[u];
            }
        } else {
#pragma unroll 1
            for (int j0 = hb; j0 < HA && ok; j0 += U * hn) {
                int hg[U];
                T *dst[U];
                T v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int j = j0 + u * hn;
                    hg[u] = -1;
                    if (j < H2) {
                        const int right = j >= st * P;
                        const int k = right ? j - st * P : j;
                        const int tl = D == 1 ? k : (int)fd_div((uint32_t)k, f_P);
                        const int pos = k - tl * P;
                        dst[u] = side + tl * RS + (right ? RS - P : 0) + pos;
                        hg[u] = (t0 + tl) * V + (right ? oR : oL) + pos;
                    } else if (j < HA) {
                        dst[u] = rdst + (j - H2);
                        hg[u] = grow + (j - H2);
                    }
                    if (hg[u] >= 0) HH_CHECK(hg[u], 0, L.N, BC_NEIGHBOUR);
                }
                ok = fetch<T, U>(buf, hg, ph, v, ctl);
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (hg[u] >= 0) *dst[u] = v[u];
            }
        }
        return ok;
    };

    // Hopping sum around extended index e of array v.
    auto hop = [&](const T *v, int e, int c) -> T {
        if (D == 1) return v[e + 1] + v[e - 1];
        const unsigned f = fl[c];
        const T xr = v[f & 2u ? e - (nx - 1) : e + 1], xl = v[f & 1u ? e + (nx - 1) : e - 1];
        const T yp = v[f & 8u ? e - (nx - 1) * nx : e + nx], ym = v[f & 4u ? e + (nx - 1) * nx : e - nx];
        return (xr + xl) + ((yp + ym) + (v[e + P] + v[e - P]));
    };
    // f<U>(s0): the sites s0 + u nthr, u < U, of a thread; U at a time so that
    // their loads and FP64 chains overlap, then one by one.
    auto sites = [&](auto &&f) {
        constexpr int UN = 4;
        int s = tid;
#pragma unroll 1
        for (; s + (UN - 1) * nthr < C; s += UN * nthr) f(s, std::integral_constant<int, UN>{});
#pragma unroll 1
        for (; s < C; s += nthr) f(s, std::integral_constant<int, 1>{});
    };

    // ---- FP32: work items of up to kSlices consecutive slices of one spatial site, so
    // that the index arithmetic is done once for them and the time neighbours of all but
    // the ends are in registers (16^3 x 64, one right-hand side: 8.2 -> 6.8 us per
    // iteration).  FP64 keeps the strided sites above, whose chains overlap better
    // (256 x 256 preconditioned: 91 us per step against 109) ----
    constexpr int kSlices = 4;
    const int nq = (st + kSlices - 1) / kSlices, items = row * nq;
    struct Item {
        int c, k0, n;           // row site, first slice, slices
        int e;                  // extended index (rows from 0) of slice k0
        int xr, xl, yp, ym;     // spatial neighbours from e
        bool edge;              // an o edge of the tile: its halo sites are read elsewhere
    };
    auto item = [&](int i) -> Item {
        Item w;
        const int q4 = (int)fd_div((uint32_t)i, f_row);
        w.c = i - q4 * row;
        w.k0 = q4 * kSlices;
        w.n = st - w.k0 < kSlices ? st - w.k0 : kSlices;
        w.e = w.k0 * RS + P + w.c;
        w.edge = w.c < P || w.c >= row - P;
        w.xr = 1;
        w.xl = -1;
        w.yp = w.ym = 0;
        if (D == 3) {
            const unsigned f = fl[w.c];
            w.xr = f & 2u ? -(nx - 1) : 1;
            w.xl = f & 1u ? nx - 1 : -1;
            w.yp = f & 8u ? -(nx - 1) * nx : nx;
            w.ym = f & 4u ? (nx - 1) * nx : -nx;
        }
        return w;
    };
    // Hopping sum around v (the item's site of one slice).
    auto item_hop = [&](const T *v, const Item &w) -> T {
        if (D == 1) return v[1] + v[-1];
        return (v[w.xr] + v[w.xl]) + ((v[w.yp] + v[w.ym]) + (v[P] + v[-P]));
    };

    bool bad = false;
    bool stageB = false;    // the next exchange brings t (and |t|^2), else M's input (and |r|^2)
    int pm = MODE_NEW;      // mode of the phases run last
    int pj = 0;             // preconditioner sub-step (s_st.pre_j may already be the next)
    long long iters = 0;
    __syncthreads();
    for (;;) {
        // ---- exchange: warp 0 waits for the sum of the last phase and turns it
        // into the next scalar (and mode), the other warps fetch the halo ----
        const int cheb2 = CHEB ? 2 * Y.cheb_n : 0;
        bool again = false;     // warp 0: another CG step, its state noted after the barrier
        double sum = 0.0;
        if (tid < 32) {
            // Between the preconditioner's sub-steps there is no sum.
            const bool inner = CHEB && pm == MODE_PRE && (stageB || s_st.pre_j + 1 < cheb2);
            __syncwarp();
            if (!inner && pm != MODE_NEW) {
                const double ra = s_st.rr_alpha, inv = stageB ? 0.0 : reciprocal(ra);
                const double tolbb = s_tolbb, dmax = MIXED ? s_dmax : 0.0;
                const bool last = s_st.cg_steps + 1 >= Y.maxit || (MIXED && s_st.since_ru + 1 >= Y.stall_window);
                const bool ok = CHEB && pm == MODE_PRE
                                    ? sum_slots<false>(my_slots + par * kOcMaxTiles, tiles, ph, ctl, sum)
                                    : sum_slots<true>(my_slots + par * kOcMaxTiles, tiles, ph, ctl, sum);
                if (!ok) {
                    bad = true;
                } else if (stageB) {
                    const T a = quotient<T>(ra, sum);
                    if (tid == 0) s_scal = a;
                } else {
                    again = !CHEB && pm == MODE_CG && !last && finite_bits(sum) && greater_nonneg(sum, tolbb) &&
                            !(MIXED && greater_nonneg(dmax, sum));
                    if (again) {
                        // The common case of decide(): beta = sum / ra, the quotient by
                        // 1 / ra with (FP64) one residual correction.
                        double beta = sum * inv;
                        if (!MIXED) beta = fma(fma(-beta, ra, sum), inv, beta);
                        if (tid == 0) {
                            s_scal = (T)beta;
                            s_restart = 0;
                            s_st.beta = beta;
                        }
                    } else if (tid == 0) {
                        const EngState S = decide(Y, s_st, sum);
                        if (MIXED && S.prec == PREC_FP64 && S.mode != MODE_DONE) {
                            // FP64 steps of a mixed system: the grid engine goes on from
                            // this reliable update (its state and |r|^2, x, r in memory).
                            s_hand = 1;
                            if (tile == 0) hand_over(L, Y, sid, s_st, sum);
                        } else {
                            s_st = S;
                            s_scal = (T)S.beta;
                            s_restart = S.beta == 0.0;
                            s_tolbb = Y.tol2 * S.bb;
                            s_dmax = Y.delta2 * S.maxr2;
                        }
                    }
                }
            } else if (tid == 0) {
                if (pm == MODE_NEW)
                    s_st = decide(Y, s_st, 0.0);
                else if (!stageB)
                    s_st.pre_j += 1;
            }
        }
        if (pm != MODE_NEW) {
            const bool ok = stageB ? fetch_halo(pktB, Tb, Tb + st * RS + P, tN)
                                   : fetch_halo(pktA, Sb + RS, Sb + P, tP);
            if (!ok) bad = true;
        }
        if (iters >= L.max_iters) bad = true;
        if (__syncthreads_or(bad ? 1 : 0)) break;
        if (again && tid == 0) {
            s_st.cg_steps += 1;
            s_st.since_ru += 1;
            if (!MIXED) s_st.fp64_steps += 1;
            s_st.rr_last = sum;
            s_st.rr_alpha = sum;
            if (MIXED && sum > s_st.maxr2) {
                s_st.maxr2 = sum;
                s_dmax = Y.delta2 * sum;
            }
        }

        if (stageB) {
            stageB = false;
            ++ph;
            if (CHEB && pm == MODE_PRE) {
                // Factor update of a preconditioner sub-step.
                const int j = pj, k = j >> 1;
                const bool last = j == cheb2 - 1;
                const T invlam = (T)__ldg(Y.cheb), a = (T)__ldg(Y.cheb + 2 + 3 * k);
                const T b2 = (T)__ldg(Y.cheb + 3 + 3 * k), invq = (T)__ldg(Y.cheb + 4 + 3 * k);
                const T scale = last ? (T)__ldg(Y.cheb + 1) : T(1);
                double acc = 0.0;
                sites([&](int s0, auto un) {
#pragma unroll
                    for (int u = 0; u < un.value; ++u) {
                        const int s = s0 + u * nthr;
                        const int tl = (int)fd_div((uint32_t)s, f_row), e = s + P + 2 * P * tl, r = s - tl * row;
                        const T y = fma(Lb[s + row], Tb[e + RS], fma(-h, hop(Tb, e, r), Tb[e])), v = Sb[RS + e];
                        T w;
                        if ((j & 1) == 0) {
                            Zb[s] = v;
                            w = fma(y, invlam, -a * v);
                        } else {
                            w = fma(y, invlam, fma(-a, v, b2 * Zb[s])) * invq * scale;
                            if (last) acc = fma((double)Rb[s], (double)w, acc);
                        }
                        Sb[RS + e] = w;
                        if (tl == st - 1 || r < P || r >= row - P) PK::store((typename PK::Raw *)pktA + gbase + s + tl * gstep, w, ph);
                    }
                });
                if (last) {
                    par ^= 1;
                    publish_signed(acc);
                }
                continue;
            }
            // ---- r -= alpha M^T t, |r|^2; then x += alpha p while the sum travels ----
            const T alpha = s_scal;
            T acc = T(0);
            par ^= 1;
            if constexpr (MIXED) {
#pragma unroll 1
                for (int i = tid; i < items; i += nthr) {
                    const Item w = item(i);
                    const T *tb = Tb + w.e;
                    T *sb = Sb + RS + w.e;
                    const T *lb = Lb + row + w.k0 * row + w.c;
                    typename PK::Raw *pa = (typename PK::Raw *)pktA + gbase + w.c + w.k0 * V;
                    T here = tb[0];
#pragma unroll
                    for (int u = 0; u < kSlices; ++u) {
                        if (u >= w.n) break;
                        const T next = tb[RS];
                        const T y = fma(*lb, next, fma(-h, item_hop(tb, w), here));
                        const T r = fma(-alpha, y, *sb);
                        *sb = r;
                        acc = fma(r, r, acc);
                        if (w.edge || w.k0 + u == st - 1) PK::store(pa, r, ph);
                        here = next;
                        tb += RS;
                        sb += RS;
                        lb += row;
                        pa += V;
                    }
                }
            } else {
                sites([&](int s0, auto un) {
#pragma unroll
                    for (int u = 0; u < un.value; ++u) {
                        const int s = s0 + u * nthr;
                        const int tl = (int)fd_div((uint32_t)s, f_row), e = s + P + 2 * P * tl, ro = s - tl * row;
                        const T y = fma(Lb[s + row], Tb[e + RS], fma(-h, hop(Tb, e, ro), Tb[e]));
                        const T r = fma(-alpha, y, CHEB ? Rb[s] : Sb[RS + e]);
                        Sb[RS + e] = r;
                        if (CHEB) Rb[s] = r;
                        acc = fma(r, r, acc);
                        if (tl == st - 1 || ro < P || ro >= row - P) PK::store((typename PK::Raw *)pktA + gbase + s + tl * gstep, r, ph);
                    }
                });
            }
            publish(acc);
            if constexpr (MIXED) {
#pragma unroll 1
                for (int i = tid; i < items; i += nthr) {
                    const int q4 = (int)fd_div((uint32_t)i, f_row), c = i - q4 * row, k0 = q4 * kSlices;
                    const T *pb = Pb + RS + k0 * RS + P + c;
                    const int step = L.x_global ? V : row;
                    T *xp = L.x_global ? Xg + gbase + c + k0 * V : Xb + k0 * row + c;
#pragma unroll
                    for (int u = 0; u < kSlices; ++u) {
                        if (k0 + u >= st) break;
                        *xp = fma(alpha, *pb, *xp);
                        pb += RS;
                        xp += step;
                    }
                }
            } else {
                sites([&](int s0, auto un) {
#pragma unroll
                    for (int u = 0; u < un.value; ++u) {
                        const int s = s0 + u * nthr;
                        const int tl = (int)fd_div((uint32_t)s, f_row), e = s + P + 2 * P * tl;
                        if (L.x_global) {
                            T *const xp = Xg + gbase + s + tl * gstep;
                            *xp = fma(alpha, Pb[RS + e], *xp);
                        } else {
                            Xb[s] = fma(alpha, Pb[RS + e], Xb[s]);
                        }
                    }
                });
            }
            continue;
        }

        if (s_hand) break;
        const int mode = s_st.mode;
        if (mode == MODE_DONE) break;
        ++iters;

        if (mode == MODE_INIT) {
            const bool zero = !(Y.x0_given && !s_st.no_guess);
            // A second INIT replaces the first one's packets: only once every
            // block has read them.
            if (pm == MODE_INIT && tile_barrier()) break;
            double acc = 0.0;
            ++ph;
            par ^= 1;
            for (int s = tid; s < C; s += nthr) {
                const int tl = (int)fd_div((uint32_t)s, f_row), g = gbase + s + tl * gstep, r = s - tl * row;
                const int e = s + P + 2 * P * tl;
                const double b = __ldg(Y.b + g);
                acc = fma(b, b, acc);
                Sb[RS + e] = (T)b;
                if (CHEB) Rb[s] = (T)b;
                if (tl == st - 1 || r < P || r >= row - P) PK::store((typename PK::Raw *)pktA + g, (T)b, ph);
                const double x = zero ? 0.0 : Y.x[g];
                if (MIXED) {
                    if (zero) Y.x[g] = 0.0;
                    if (L.x_global)
                        Xg[g] = T(0);
                    else
                        Xb[s] = T(0);
                } else if (!L.x_global) {
                    Xb[s] = (T)x;
                } else if (zero) {
                    Y.x[g] = 0.0;
                }
            }
            publish(acc);
            pm = mode;
            continue;
        }

        if (mode == MODE_RU) {
            // x64 of the tile to memory (mixed: with the FP32 part added).
            for (int s = tid; s < C; s += nthr) {
                const int g = gbase + s + (int)fd_div((uint32_t)s, f_row) * gstep;
                if (MIXED) {
                    Y.x[g] += (double)(L.x_global ? Xg[g] : Xb[s]);
                    if (L.x_global)
                        Xg[g] = T(0);
                    else
                        Xb[s] = T(0);
                } else if (!L.x_global) {
                    Y.x[g] = (double)Xb[s];
                }
            }
            if (tile_barrier()) break;
            for (int s = tid; s < C; s += nthr) {
                const int g = gbase + s + (int)fd_div((uint32_t)s, f_row) * gstep;
                Nbr nb;
                neighbours(Y.g, g, nb);
                Y.t[g] = stencil_M<double>(Y.g, Y.h, Y.L64, Y.x, g, nb);
            }
            if (tile_barrier()) break;
            double acc = 0.0;
            ++ph;
            par ^= 1;
            for (int s = tid; s < C; s += nthr) {
                const int tl = (int)fd_div((uint32_t)s, f_row), g = gbase + s + tl * gstep, r = s - tl * row;
                Nbr nb;
                neighbours(Y.g, g, nb);
                const double res = __ldg(Y.b + g) - stencil_MT<double>(Y.g, Y.h, Y.L64, Y.t, g, nb);
                acc = fma(res, res, acc);
                Sb[RS + s + P + 2 * P * tl] = (T)res;
                if (CHEB) Rb[s] = (T)res;
                if (MIXED) Y.r[g] = res;
                if (tl == st - 1 || r < P || r >= row - P) PK::store((typename PK::Raw *)pktA + g, (T)res, ph);
            }
            publish(acc);
            pm = mode;
            continue;
        }

        // ---- t = M v of a preconditioner sub-step or, in a CG step, of
        // p = r + beta p (r: z with the preconditioner), formed on the tile and
        // its halo ----
        const bool cg = !CHEB || mode == MODE_CG;
        if (cg) {
            const bool restart = s_restart != 0;
            const T beta = s_scal;
            const int E = (st + 1) * RS;
            int j = tid;
#pragma unroll 1
            for (; j + 3 * nthr < E; j += 4 * nthr) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const T v = Sb[j + u * nthr];
                    Pb[j + u * nthr] = restart ? v : fma(beta, Pb[j + u * nthr], v);
                }
            }
#pragma unroll 1
            for (; j < E; j += nthr) Pb[j] = restart ? Sb[j] : fma(beta, Pb[j], Sb[j]);
            __syncthreads();
        }
        const T *const v = cg ? Pb : Sb;
        T acc = T(0);
        ++ph;
        if constexpr (MIXED) {
#pragma unroll 1
            for (int i = tid; i < items; i += nthr) {
                const Item w = item(i);
                const T *vb = v + RS + w.e;
                T *tb = Tb + w.e;
                const T *lb = Lb + w.k0 * row + w.c;        // links of the slice before
                typename PK::Raw *pb = (typename PK::Raw *)pktB + gbase + w.c + w.k0 * V;
                T before = vb[-RS];
#pragma unroll
                for (int u = 0; u < kSlices; ++u) {
                    if (u >= w.n) break;
                    const T here = *vb;
                    const T y = fma(*lb, before, fma(-h, item_hop(vb, w), here));
                    *tb = y;
                    acc = fma(y, y, acc);
                    if (w.edge || w.k0 + u == 0) PK::store(pb, y, ph);
                    before = here;
                    vb += RS;
                    tb += RS;
                    lb += row;
                    pb += V;
                }
            }
        } else {
            sites([&](int s0, auto un) {
#pragma unroll
                for (int u = 0; u < un.value; ++u) {
                    const int s = s0 + u * nthr;
                    const int tl = (int)fd_div((uint32_t)s, f_row), r = s - tl * row;
                    const int e = s + P + 2 * P * tl;
                    const T y = fma(Lb[s], v[e], fma(-h, hop(v + RS, e, r), v[RS + e]));
                    Tb[e] = y;
                    if (cg) acc = fma(y, y, acc);
                    if (tl == 0 || r < P || r >= row - P) PK::store((typename PK::Raw *)pktB + gbase + s + tl * gstep, y, ph);
                }
            });
        }
        if (cg) {
            par ^= 1;
            publish(acc);
        }
        stageB = true;
        pj = pm == MODE_PRE ? pj + 1 : 0;
        pm = mode;
    }

    // ---- leave: x, the state, the last phase number ----
    __syncthreads();
    if (!MIXED && !L.x_global && s_st.mode == MODE_DONE)
        for (int s = tid; s < C; s += nthr) Y.x[gbase + s + (int)fd_div((uint32_t)s, f_row) * gstep] = (double)Xb[s];
    if (tid == 0) {
        if (tile == 0 && s_st.mode == MODE_DONE) {
            L.state[0][sid] = s_st;
            L.state[1][sid] = s_st;
        }
        atomicMax(L.seq + 1, L.seq[0] + (unsigned long long)(uint32_t)(ph - ph0) + 1ull);
    }
}

const void *oc_kernel(int d, bool mixed, bool cheb)
{
    if (d == 1)
        return mixed ? (const void *)k_onchip<1, float, false>
                     : cheb ? (const void *)k_onchip<1, double, true> : (const void *)k_onchip<1, double, false>;
    return mixed ? (const void *)k_onchip<3, float, false>
                 : cheb ? (const void *)k_onchip<3, double, true> : (const void *)k_onchip<3, double, false>;
}

}  // namespace

static const void *plan_kernel(const OcPlan &P, int d)
{
    if (P.cols) return oc_cols_kernel(d, P.mixed != 0, P.cheb != 0, P.ex != 0, P.cols, P.sides);
    return oc_kernel(d, P.mixed != 0, P.cheb != 0);
}

// Registers per thread of a layout's kernel, asked once per process.
static int kernel_regs(const OcPlan &P, int d)
{
    static std::atomic<int> known[2 * 2 * 2 * 2 * 3 * 9];
    std::atomic<int> &k =
        known[((((d == 3) * 2 + (P.mixed != 0)) * 2 + (P.cheb != 0)) * 2 + (P.ex != 0)) * 27 + P.sides * 9 + P.cols];
    int r = k.load(std::memory_order_relaxed);
    if (r == 0) {
        cudaFuncAttributes a;
        if (cudaFuncGetAttributes(&a, plan_kernel(P, d)) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        r = a.numRegs;
        k.store(r, std::memory_order_relaxed);
    }
    return r;
}

int oc_max_blocks(const OcPlan &P, int d)
{
    const void *fn = plan_kernel(P, d);
    int per = 0;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kOcMaxSmem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, P.threads, P.smem) != cudaSuccess)
        return 0;
    return per;
}

OcPlan oc_plan(int d, int nx, int ntau, int nsys, bool mixed, bool cheb, bool ex, int nsm, size_t smem_sm, size_t smem_blk,
               int forms)
{
    return oc_choose(
        d, nx, ntau, nsys, mixed, cheb, ex, nsm, smem_sm, smem_blk, forms,
        [d](const OcPlan &p) { return kernel_regs(p, d); },
        [=](const OcPlan &p) { return oc_max_blocks(p, d) * nsm >= p.go * p.gt * nsys; });
}

cudaError_t oc_launch(const OcLaunch &L, const OcPlan &P, int d, cudaStream_t st)
{
    if (P.threads % 32 != 0) return cudaErrorInvalidConfiguration;
    const void *fn = plan_kernel(P, d);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kOcMaxSmem);
    if (e != cudaSuccess) return e;
    OcLaunch arg = L;
    void *args[] = {(void *)&arg};
    return cudaLaunchCooperativeKernel(fn, dim3(P.go * P.gt * L.nsys), dim3(P.threads), args, P.smem, st);
}

}  // namespace hh
