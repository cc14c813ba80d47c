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
// alternate.  The reliable update exchanges x and t in global memory between
// barriers made of the same sums with fences around them.
//
// What bounds it: the chain exchange - barrier - phase - block sum, run by a few
// warps (FP64 from about 800 sites per SM: the FP64 pipe, 16 clocks per warp
// instruction).  Measured against the grid engine, us per iteration, 2
// right-hand sides: d = 1 32 x 64 FP64 5.9 (11.3), 1024 x 128 FP64 11.4 (15.4),
// mixed 7.3 (10.7); d = 3 8^3 x 40 FP64 7.7 (17.2), 12^3 x 64 mixed 7.9 (15.0),
// 16^3 x 64 mixed 9.7 (16.6); a degree-8 preconditioned step on 256 x 256 91 (199).
// It was faster wherever the vectors fit (20^3 x 64 mixed: 15.9 against 19.4).
//
// Every wait is bounded (EngCtl::timeout_ns); on expiry the block records
// HH_ETIMEOUT, and all its threads leave at the next block barrier.
#include <cstdlib>

#include "hh_engine_decide.cuh"
#include "hh_onchip.cuh"

namespace hh {

namespace {

// ---------------------------------------------------------------------------
// Packets.
// ---------------------------------------------------------------------------
struct Raw16 {
    unsigned long long v, seq;
};

__device__ __forceinline__ Raw16 ld_raw(const Raw16 *p)
{
    Raw16 r;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(r.v), "=l"(r.seq)
                 : "l"(p)
                 : "memory");
    return r;
}

__device__ __forceinline__ void st_raw(Raw16 *p, unsigned long long v, unsigned long long seq)
{
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
                 "l"(v), "l"(seq)
                 : "memory");
}

// One site's packet in a buffer of packets indexed by site.
template <typename T>
struct Packet;

template <>
struct Packet<double> {
    using Raw = Raw16;
    static __device__ __forceinline__ Raw load(const unsigned char *buf, int site)
    {
        return ld_raw((const Raw16 *)buf + site);
    }
    static __device__ __forceinline__ bool ready(const Raw &r, uint32_t seq) { return (uint32_t)r.seq == seq; }
    static __device__ __forceinline__ double value(const Raw &r) { return __longlong_as_double((long long)r.v); }
    static __device__ __forceinline__ void store(unsigned char *buf, int site, double v, uint32_t seq)
    {
        st_raw((Raw16 *)buf + site, (unsigned long long)__double_as_longlong(v), seq);
    }
};

template <>
struct Packet<float> {
    using Raw = unsigned long long;
    static __device__ __forceinline__ Raw load(const unsigned char *buf, int site)
    {
        return ld_relaxed_u64((const unsigned long long *)buf + site);
    }
    static __device__ __forceinline__ bool ready(const Raw &r, uint32_t seq) { return (uint32_t)(r >> 32) == seq; }
    static __device__ __forceinline__ float value(const Raw &r) { return __uint_as_float((uint32_t)r); }
    static __device__ __forceinline__ void store(unsigned char *buf, int site, float v, uint32_t seq)
    {
        const unsigned long long w = ((unsigned long long)seq << 32) | __float_as_uint(v);
        asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"((unsigned long long *)buf + site), "l"(w)
                     : "memory");
    }
};

// A bounded wait's clock: called once per failed poll; false when the budget
// is spent or another block has recorded an error.
struct SpinClock {
    unsigned spins = 0;
    uint64_t t0 = 0;
    __device__ __forceinline__ bool tick(EngCtl *ctl)
    {
        if ((++spins & 63u) != 0) return true;
        if (t0 == 0) t0 = global_ns();
        if (ld_volatile_i32(&ctl->error) != 0) return false;
        if ((long long)(global_ns() - t0) > ctl->timeout_ns) {
            atomicCAS(&ctl->error, 0, -6);
            return false;
        }
        return true;
    }
};

// U packets of a thread (site < 0: none): all loads in flight at once, then
// polled until each carries 'seq'.  False when the wait ran out.
template <typename T, int U>
__device__ __forceinline__ bool fetch(const unsigned char *buf, const int (&site)[U], uint32_t seq, T (&v)[U],
                                      EngCtl *ctl)
{
    typename Packet<T>::Raw raw[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (site[u] >= 0) raw[u] = Packet<T>::load(buf, site[u]);
    unsigned pend = 0;
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (site[u] >= 0) {
            v[u] = Packet<T>::value(raw[u]);
            if (!Packet<T>::ready(raw[u], seq)) pend |= 1u << u;
        }
    SpinClock clk;
    while (pend) {
        if (!clk.tick(ctl)) return false;
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (pend & (1u << u)) {
                const typename Packet<T>::Raw r = Packet<T>::load(buf, site[u]);
                if (Packet<T>::ready(r, seq)) {
                    v[u] = Packet<T>::value(r);
                    pend &= ~(1u << u);
                }
            }
    }
    return true;
}

// All 32 lanes of a warp: the sum of n partial-sum packets once each carries
// 'seq' (lane-strided sums in order, then a fixed tree; the same bits in every
// lane of every block).  False in every lane when the wait ran out.
__device__ __forceinline__ bool sum_slots(const Raw16 *slot, int n, uint32_t seq, EngCtl *ctl, double &sum)
{
    constexpr int U = 5;
    const int lane = (int)(threadIdx.x & 31u);
    double v = 0.0;
    bool ok = true;
    SpinClock clk;
#pragma unroll 1
    for (int j0 = 0; j0 < n && ok; j0 += 32 * U) {
        Raw16 a[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            a[u].v = 0;
            a[u].seq = seq;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (j0 + 32 * u + lane < n) a[u] = ld_raw(slot + j0 + 32 * u + lane);
        while (true) {
            bool ready = true;
#pragma unroll
            for (int u = 0; u < U; ++u) ready = ready && ((uint32_t)a[u].seq == seq);
            if (ready) break;
            if (!clk.tick(ctl)) {
                ok = false;
                break;
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if ((uint32_t)a[u].seq != seq) a[u] = ld_raw(slot + j0 + 32 * u + lane);
        }
        const double a01 = __longlong_as_double((long long)a[0].v) + __longlong_as_double((long long)a[1].v);
        const double a23 = __longlong_as_double((long long)a[2].v) + __longlong_as_double((long long)a[3].v);
        v += (a01 + a23) + __longlong_as_double((long long)a[4].v);
    }
    ok = __all_sync(0xffffffffu, ok);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    sum = v;
    return ok;
}

// Sum over a warp of non-negative values, in integers: each value's significand,
// shifted to the largest exponent of the warp, in three 27-bit parts that the
// integer warp reduction adds exactly (81 bits; what is shifted out is below
// 2^-80 of the largest value).  The same result in every lane; NaN if a value
// is not finite.  The shuffle tree of FP64 adds takes 5 x 16 cycles of the
// SM's FP64 pipe per warp, 1.4k cycles for 16 warps; this takes none of it.
struct SumParts {
    int e;                  // biased FP64 exponent
    unsigned long long m;   // significand, 53 bits
};

__device__ __forceinline__ SumParts sum_parts(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    SumParts p;
    p.e = (int)((b >> 52) & 0x7ffu);
    p.m = b & 0xfffffffffffffull;
    if (p.e)
        p.m |= 1ull << 52;
    else
        p.e = 1;
    return p;
}

__device__ __forceinline__ SumParts sum_parts(float v)
{
    const unsigned b = __float_as_uint(v);
    int e = (int)((b >> 23) & 0xffu);
    unsigned m = b & 0x7fffffu;
    if (e)
        m |= 1u << 23;
    else
        e = 1;
    SumParts p;
    p.e = e == 255 ? 0x7ff : e + (1023 - 127);
    p.m = (unsigned long long)m << 29;
    return p;
}

template <typename T>
__device__ __forceinline__ double warp_sum_nonneg(T v)
{
    const SumParts p = sum_parts(v);
    const int emax = (int)__reduce_max_sync(0xffffffffu, (unsigned)p.e);
    const int d = emax - p.e;
    // m 2^28 >> d as 81 bits: parts of bits [54, 81), [27, 54), [0, 27).
    unsigned a2 = 0, a1 = 0, a0 = 0;
    if (d <= 80) {
        const unsigned long long hi = d < 64 ? p.m >> d : 0ull;                       // bits from 28 up
        const unsigned long long lo = d == 0 ? 0ull : d < 64 ? p.m << (64 - d) : d == 64 ? p.m : p.m >> (d - 64);
        a2 = (unsigned)(hi >> 26);
        a1 = (unsigned)(hi << 1) & 0x7ffffffu;
        a1 |= (unsigned)(lo >> 63);
        a0 = (unsigned)(lo >> 36) & 0x7ffffffu;
    }
    const unsigned long long s2 = __reduce_add_sync(0xffffffffu, a2);
    const unsigned long long s1 = __reduce_add_sync(0xffffffffu, a1);
    const unsigned long long s0 = __reduce_add_sync(0xffffffffu, a0);
    if (emax == 0x7ff) return __longlong_as_double((long long)kSigNaN);
    // S = s2 2^54 + s1 2^27 + s0 in units of 2^(emax - 1023 - 80): its upper 64
    // bits (below them: a sticky bit) rounded to nearest even.
    const unsigned long long l = s0 + ((s1 & 0x1fffffffffull) << 27);   // < 2^60
    unsigned long long h = s2;                                          // units of 2^54
    const unsigned long long c = l >> 54;
    h += c;
    const unsigned long long rest = l & 0x3fffffffffffffull;            // 54 bits
    if (h == 0 && rest == 0) return 0.0;
    // h has up to 33 bits: with rest 87.  Normalise so that the top bit is bit 63.
    const int z = h ? __clzll((long long)h) : 0;
    unsigned long long t;
    int e;
    if (h) {
        t = (h << z) | (z ? ((rest << 10) >> (64 - z)) : 0ull);
        const unsigned long long low = z ? (rest << 10) << z : (rest << 10);
        t |= low != 0 ? 1ull : 0ull;
        e = 63 - z + 54;
    } else {
        const int zr = __clzll((long long)rest);
        t = rest << zr;
        e = 63 - zr;
    }
    // t in [2^63, 2^64), value t 2^(e - 63) units.
    unsigned long long m = t >> 11;
    const unsigned long long frac = t & 0x7ffull;
    m += (frac > 0x400ull || (frac == 0x400ull && (m & 1))) ? 1ull : 0ull;
    e += emax - 80;                     // biased exponent of the result
    if (e <= 0) return __longlong_as_double((long long)(m >> (e < -51 ? 53 : 1 - e)));
    if (e >= 0x7ff) return __longlong_as_double((long long)kSigNaN);
    return __longlong_as_double((long long)(((unsigned long long)(e - 1) << 52) + m));
}

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
    __shared__ double s_red[kOcMaxThreads / 32];
    __shared__ double s_scal;       // beta or alpha of the phase about to run
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
    unsigned char *const fl = (unsigned char *)q;    // d = 3: x-y edges of each compact site
    T *const Xg = MIXED ? (T *)Y.x32 : (T *)Y.x;

    unsigned char *const pktA = L.pkt + (size_t)sid * 2 * L.N * sizeof(typename PK::Raw);
    unsigned char *const pktB = pktA + (size_t)L.N * sizeof(typename PK::Raw);
    // Partial sums: kOcReplicas copies, each read by every kOcReplicas-th block.
    Raw16 *const slots = (Raw16 *)L.slots + (size_t)sid * 2 * kOcReplicas * kOcMaxTiles;
    const Raw16 *const my_slots = slots + (size_t)(tile % kOcReplicas) * 2 * kOcMaxTiles;

    const T h = (T)Y.h;
    if (D == 3)
        for (int s = tid; s < C; s += nthr) {
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
    const int wtop = nwarp <= 1 ? 0 : nwarp <= 2 ? 1 : nwarp <= 4 ? 2 : nwarp <= 8 ? 4 : 8;

    // Publishes the block's sum under the current phase number, from each
    // warp's sum (every thread calls it; its barrier follows all of the block's
    // writes of the phase).
    auto publish = [&](double wsum) {
        if ((tid & 31) == 0) s_red[tid >> 5] = wsum;
        __syncthreads();
        if (tid < 32) {
            double w = tid < nwarp ? s_red[tid] : 0.0;
            for (int o = wtop; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
            if (tid < kOcReplicas && !drop)
                st_raw(slots + (size_t)(2 * tid + par) * kOcMaxTiles + tile,
                       (unsigned long long)__double_as_longlong(__shfl_sync((1u << kOcReplicas) - 1u, w, 0)), ph);
        }
    };
    // Warp 0: waits for the sum published last.
    auto wait_sum = [&](double &sum) -> bool {
        return sum_slots(my_slots + par * kOcMaxTiles, tiles, ph, ctl, sum);
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
            bad = !wait_sum(dummy);
            __threadfence();
        }
        return __syncthreads_or(bad ? 1 : 0) != 0;
    };

    const int H2 = 2 * st * P, HA = H2 + row;
    // Halo threads: all but warp 0 (which waits for the sums) when there are others.
    const int hb = nwarp > 1 ? tid - 32 : tid, hn = nwarp > 1 ? nthr - 32 : nthr;
    // The halo of the packets in buf: o columns of the tile's rows into side (extended),
    // then the row at site grow into rdst.
    auto fetch_halo = [&](const unsigned char *buf, T *side, T *rdst, int grow) -> bool {
        constexpr int U = 4;
        bool ok = true;
        if (hb >= 0)
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
        return ok;
    };

    // Hopping sum around extended index e of array v.
    auto hop = [&](const T *v, int e, int s) -> T {
        if (D == 1) return v[e + 1] + v[e - 1];
        const unsigned f = fl[s];
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

    bool bad = false;
    bool stageB = false;    // the next exchange brings t (and |t|^2), else M's input (and |r|^2)
    int pm = s_st.mode;     // mode of the phases run last
    long long iters = 0;
    __syncthreads();
    for (;;) {
        // ---- exchange: warp 0 waits for the sum of the last phase and turns it
        // into the next scalar (and mode), the other warps fetch the halo ----
        const int cheb2 = CHEB ? 2 * Y.cheb_n : 0;
        if (tid < 32) {
            // Between the preconditioner's sub-steps there is no sum.
            const bool inner = CHEB && pm == MODE_PRE && (stageB || s_st.pre_j + 1 < cheb2);
            __syncwarp();
            if (!inner && pm != MODE_NEW) {
                const double ra = s_st.rr_alpha;
                double inv = 0.0, sum;
                if (!stageB) inv = 1.0 / ra;        // off the critical path: used when the sum arrives
                if (!wait_sum(sum)) {
                    bad = true;
                } else if (stageB) {
                    if (tid == 0) s_scal = ra / sum;
                } else {
                    const int steps = s_st.cg_steps + 1, since = s_st.since_ru + 1;
                    const bool stop = !(sum > s_tolbb) || (MIXED && sum < s_dmax) || !isfinite(sum) ||
                                      (MIXED && since >= Y.stall_window) || steps >= Y.maxit;
                    if (!CHEB && pm == MODE_CG && !stop) {
                        // The common case of decide(): another CG step, beta = sum / ra
                        // (the quotient by 1 / ra with one residual correction).
                        if (tid == 0) {
                            double beta = sum * inv;
                            beta = fma(fma(-beta, ra, sum), inv, beta);
                            s_scal = beta;
                            s_st.beta = beta;
                            s_st.cg_steps = steps;
                            s_st.since_ru = since;
                            if (!MIXED) s_st.fp64_steps += 1;
                            s_st.rr_last = sum;
                            s_st.rr_alpha = sum;
                            if (MIXED && sum > s_st.maxr2) {
                                s_st.maxr2 = sum;
                                s_dmax = Y.delta2 * sum;
                            }
                        }
                    } else if (tid == 0) {
                        const EngState S = decide(Y, s_st, sum);
                        if (MIXED && S.prec == PREC_FP64 && S.mode != MODE_DONE) {
                            // FP64 steps of a mixed system: the grid engine goes on from
                            // this reliable update (its state and |r|^2, x, r in memory).
                            s_hand = 1;
                            if (tile == 0) {
                                for (int j = 0; j < Y.ntiles; ++j)
                                    L.sig[(size_t)5 * L.sig_stride + Y.part0 + j] =
                                        (unsigned long long)__double_as_longlong(j == 0 ? sum : 0.0);
                                L.state[0][sid] = s_st;
                                L.state[1][sid] = s_st;
                            }
                        } else {
                            s_st = S;
                            s_scal = S.beta;
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

        if (stageB) {
            stageB = false;
            ++ph;
            if (CHEB && pm == MODE_PRE) {
                // Factor update of a preconditioner sub-step.
                const int j = s_st.pre_j, k = j >> 1;
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
                        const T y = fma(Lb[s + row], Tb[e + RS], fma(-h, hop(Tb, e, s), Tb[e])), v = Sb[RS + e];
                        T w;
                        if ((j & 1) == 0) {
                            Zb[s] = v;
                            w = fma(y, invlam, -a * v);
                        } else {
                            w = fma(y, invlam, fma(-a, v, b2 * Zb[s])) * invq * scale;
                            if (last) acc = fma((double)Rb[s], (double)w, acc);
                        }
                        Sb[RS + e] = w;
                        if (tl == st - 1 || r < P || r >= row - P) PK::store(pktA, gbase + s + tl * gstep, w, ph);
                    }
                });
                if (last) {
                    par ^= 1;
                    publish(warp_sum(acc));
                }
                continue;
            }
            // ---- r -= alpha M^T t, |r|^2; then x += alpha p while the sum travels ----
            const T alpha = (T)s_scal;
            T sum = T(0);
            par ^= 1;
            sites([&](int s0, auto un) {
#pragma unroll
                for (int u = 0; u < un.value; ++u) {
                    const int s = s0 + u * nthr;
                    const int tl = (int)fd_div((uint32_t)s, f_row), e = s + P + 2 * P * tl, ro = s - tl * row;
                    const T y = fma(Lb[s + row], Tb[e + RS], fma(-h, hop(Tb, e, s), Tb[e]));
                    const T r = fma(-alpha, y, CHEB ? Rb[s] : Sb[RS + e]);
                    Sb[RS + e] = r;
                    if (CHEB) Rb[s] = r;
                    sum = fma(r, r, sum);
                    if (tl == st - 1 || ro < P || ro >= row - P) PK::store(pktA, gbase + s + tl * gstep, r, ph);
                }
            });
            publish(warp_sum_nonneg(sum));
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
                if (tl == st - 1 || r < P || r >= row - P) PK::store(pktA, g, (T)b, ph);
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
            publish(warp_sum(acc));
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
                if (tl == st - 1 || r < P || r >= row - P) PK::store(pktA, g, (T)res, ph);
            }
            publish(warp_sum(acc));
            pm = mode;
            continue;
        }

        // ---- t = M v of a preconditioner sub-step or, in a CG step, of
        // p = r + beta p (r: z with the preconditioner), formed on the tile and
        // its halo ----
        const bool cg = !CHEB || mode == MODE_CG;
        if (cg) {
            const bool restart = s_st.beta == 0.0;
            const T beta = (T)s_scal;
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
        sites([&](int s0, auto un) {
#pragma unroll
            for (int u = 0; u < un.value; ++u) {
                const int s = s0 + u * nthr;
                const int tl = (int)fd_div((uint32_t)s, f_row), r = s - tl * row;
                const int e = s + P + 2 * P * tl;
                const T y = fma(Lb[s], v[e], fma(-h, hop(v + RS, e, s), v[RS + e]));
                Tb[e] = y;
                if (cg) acc = fma(y, y, acc);
                if (tl == 0 || r < P || r >= row - P) PK::store(pktB, gbase + s + tl * gstep, y, ph);
            }
        });
        if (cg) {
            par ^= 1;
            publish(warp_sum_nonneg(acc));
        }
        stageB = true;
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

// Dynamic shared memory a block may ask for: the 227 KB a block can have, less
// the kernels' static part.  The kernels' limit is set to it, whatever a
// launch uses, so that threads launching different layouts do not race on it.
constexpr int kOcStaticSmem = 2048;
constexpr int kOcMaxSmem = 227 * 1024 - kOcStaticSmem;

const void *oc_kernel(int d, bool mixed, bool cheb)
{
    if (d == 1)
        return mixed ? (const void *)k_onchip<1, float, false>
                     : cheb ? (const void *)k_onchip<1, double, true> : (const void *)k_onchip<1, double, false>;
    return mixed ? (const void *)k_onchip<3, float, false>
                 : cheb ? (const void *)k_onchip<3, double, true> : (const void *)k_onchip<3, double, false>;
}

// Dynamic shared memory of a block whose tile is at most so x st columns of P
// sites (the kernel's layout).
size_t oc_smem(int d, long long P, int so, int st, bool mixed, bool cheb, bool x_global)
{
    const long long C = P * so * st, E = P * (so + 2) * (st + 1), Lk = P * so * (st + 1);
    const long long vals = 3 * E + Lk + (x_global ? 0 : C) + (cheb ? 2 * C : 0);
    return (size_t)(vals * (mixed ? 4 : 8) + (d == 3 ? C : 0) + 16);
}

}  // namespace

OcPlan oc_plan(int d, int nx, int ntau, int nsys, bool mixed, bool cheb, int nsm, size_t smem_sm, size_t smem_blk)
{
    OcPlan best = {};
    const long long P = d == 3 ? (long long)nx * nx : 1;
    double best_cost = 0.0;
    constexpr size_t kStatic = kOcStaticSmem;    // static and reserved shared memory per block
    for (int m = 1; m <= 4; ++m) {
        const int G = (int)((long long)nsm * m / nsys) < kOcMaxTiles ? nsm * m / nsys : kOcMaxTiles;
        if (G < 1) continue;
        const int max_threads = kOcMaxThreads / m;
        // Tile extents that differ: so = ceil(nx / go), st = ceil(ntau / gt), with the fewest tiles each.
        for (int go = 1; go <= nx && go <= G; ++go) {
            const int so = (nx + go - 1) / go;
            if (go > 1 && (nx + go - 2) / (go - 1) == so) continue;
            for (int st = 1, gt; st <= ntau; st = gt == 1 ? ntau + 1 : (ntau + gt - 2) / (gt - 1)) {
                gt = (ntau + st - 1) / st;
                if ((long long)go * gt > G) continue;
                for (int xg = 0; xg < 2; ++xg) {
                    const size_t sm = oc_smem(d, P, so, st, mixed, cheb, xg != 0);
                    if (sm > kOcMaxSmem || sm + kStatic > smem_blk || (sm + kStatic) * m > smem_sm) continue;
                    const long long C = P * so * st, H = P * (2 * st + so);
                    // Clocks of one phase on an SM holding m tiles.
                    const double site = mixed ? 0.8 : 3.0;
                    const double cost = m * (C * (site + (xg ? 0.3 : 0.0)) + H * 1.0) + 10.0 * go * gt;
                    if (best.ok && cost >= best_cost) continue;
                    best_cost = cost;
                    best.ok = 1;
                    best.go = go;
                    best.gt = gt;
                    best.so = so;
                    best.st = st;
                    best.x_global = xg;
                    best.mixed = mixed;
                    best.cheb = cheb;
                    best.smem = sm;
                    // More than 8 warps only lengthen the block's barriers and sums while
                    // a thread has few sites.
                    int thr = (int)((C + 31) / 32 * 32);
                    if (thr > 256 && C <= 2048) thr = 256;
                    if (thr > max_threads) thr = max_threads;
                    if (thr < 64) thr = 64;
                    best.threads = thr;
                }
            }
        }
    }
    return best;
}

int oc_max_blocks(const OcPlan &P, int d)
{
    const void *fn = oc_kernel(d, P.mixed != 0, P.cheb != 0);
    int per = 0;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kOcMaxSmem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, P.threads, P.smem) != cudaSuccess)
        return 0;
    return per;
}

cudaError_t oc_launch(const OcLaunch &L, const OcPlan &P, int d, cudaStream_t st)
{
    const void *fn = oc_kernel(d, P.mixed != 0, P.cheb != 0);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kOcMaxSmem);
    if (e != cudaSuccess) return e;
    OcLaunch arg = L;
    void *args[] = {(void *)&arg};
    return cudaLaunchCooperativeKernel(fn, dim3(P.go * P.gt * L.nsys), dim3(P.threads), args, P.smem, st);
}

}  // namespace hh
