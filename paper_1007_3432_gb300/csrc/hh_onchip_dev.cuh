// Device helpers of the on-chip CG engine: packets (a value and the number of
// the phase it belongs to in one access), bounded polls, sums.
#pragma once

#include "hh_engine_decide.cuh"
#include "hh_onchip.cuh"

namespace hh {

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

// One site's packet.
template <typename T>
struct Packet;

template <>
struct Packet<double> {
    using Raw = Raw16;
    static __device__ __forceinline__ Raw load(const Raw *p) { return ld_raw(p); }
    static __device__ __forceinline__ bool ready(const Raw &r, uint32_t seq) { return (uint32_t)r.seq == seq; }
    static __device__ __forceinline__ double value(const Raw &r) { return __longlong_as_double((long long)r.v); }
    static __device__ __forceinline__ void store(Raw *p, double v, uint32_t seq)
    {
        st_raw(p, (unsigned long long)__double_as_longlong(v), seq);
    }
};

template <>
struct Packet<float> {
    using Raw = unsigned long long;
    static __device__ __forceinline__ Raw load(const Raw *p) { return ld_relaxed_u64(p); }
    static __device__ __forceinline__ bool ready(const Raw &r, uint32_t seq) { return (uint32_t)(r >> 32) == seq; }
    static __device__ __forceinline__ float value(const Raw &r) { return __uint_as_float((uint32_t)r); }
    static __device__ __forceinline__ void store(Raw *p, float v, uint32_t seq)
    {
        const unsigned long long w = ((unsigned long long)seq << 32) | __float_as_uint(v);
        asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
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
        if (site[u] >= 0) raw[u] = Packet<T>::load((const typename Packet<T>::Raw *)buf + site[u]);
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
                const typename Packet<T>::Raw r = Packet<T>::load((const typename Packet<T>::Raw *)buf + site[u]);
                if (Packet<T>::ready(r, seq)) {
                    v[u] = Packet<T>::value(r);
                    pend &= ~(1u << u);
                }
            }
    }
    return true;
}

// Sums of non-negative values in integers.  A shuffle tree of FP64 adds takes 80
// clocks a level and 16 clocks of the SM's FP64 pipe per warp and level (1.4k
// clocks for 16 warps); the integer warp reductions take 46 and none of it.
// Each significand gets kGuardWarp more bits, is shifted, rounding to nearest, to
// the largest exponent of the warp and added as 22-bit parts.  The largest value
// is then at least 2^57 units and a shifted one loses at most half a unit: 31 of
// them 31 2^-58, less than 2^-53 of the largest.  A block's warps are normalised to 55
// bits and added in two parts (15 2^-55 at most), and the total is rounded to a double
// (2^-53): less than 6 2^-53 of the sum, against the FP64 tree's 9 roundings of 2^-53
// (5 levels of a warp, 4 of 16 warps).
constexpr int kGuardWarp = 5;       // 32 values of 53 + 5 bits: 63 bits
constexpr int kGuardSlots = 8;      // 5 values of 53 + 8 bits per lane: 64 bits
constexpr int kNotFinite = 0x7fff;

struct Significand {
    int e;                  // biased FP64 exponent; kNotFinite: infinity or NaN
    unsigned long long m;   // 53 bits
};

__host__ __device__ __forceinline__ Significand significand_bits(unsigned long long b)
{
    Significand p;
    p.e = (int)((b >> 52) & 0x7ffu);
    p.m = b & 0xfffffffffffffull;
    if (p.e)
        p.m |= 1ull << 52;
    else
        p.e = 1;
    if (p.e == 0x7ff) p.e = kNotFinite;
    return p;
}

__host__ __device__ __forceinline__ Significand significand_bits32(unsigned b)
{
    int e = (int)((b >> 23) & 0xffu);
    unsigned m = b & 0x7fffffu;
    if (e)
        m |= 1u << 23;
    else
        e = 1;
    Significand p;
    p.e = e == 255 ? kNotFinite : e + (1023 - 127);
    p.m = (unsigned long long)m << 29;
    return p;
}

__device__ __forceinline__ Significand significand(double v)
{
    return significand_bits((unsigned long long)__double_as_longlong(v));
}

__device__ __forceinline__ Significand significand(float v)
{
    return significand_bits32(__float_as_uint(v));
}

// v / 2^d, rounded to nearest (d >= 0, v < 2^62).
__host__ __device__ __forceinline__ unsigned long long shift_round(unsigned long long v, int d)
{
    return d > 62 ? 0ull : (v + ((1ull << d) >> 1)) >> d;
}

// A sum s 2^(e - 1075 - kGuardWarp), s < 2^63; e >= kNotFinite: not finite.
struct ISum {
    unsigned long long s;
    int e;
};

// The total s2 2^44 + s1 2^22 + s0 of a warp's parts (s1, s0 < 2^27), divided by
// 2^shift and rounded to nearest.
__host__ __device__ __forceinline__ unsigned long long isum_join(unsigned long long s2, unsigned long long s1,
                                                                 unsigned long long s0, int shift)
{
    return (s2 << (44 - shift)) + (((s1 << 22) + s0 + ((1ull << shift) >> 1)) >> shift);
}

// Sum over the warp of one aligned term per lane, divided by 2^shift.
__device__ __forceinline__ unsigned long long warp_join(unsigned long long x, int shift)
{
    const unsigned s2 = __reduce_add_sync(0xffffffffu, (unsigned)(x >> 44));
    const unsigned s1 = __reduce_add_sync(0xffffffffu, (unsigned)(x >> 22) & 0x3fffffu);
    const unsigned s0 = __reduce_add_sync(0xffffffffu, (unsigned)x & 0x3fffffu);
    return isum_join(s2, s1, s0, shift);
}

// Sum over the warp, the same in every lane.
__device__ __forceinline__ ISum warp_isum(double v)
{
    const Significand p = significand(v);
    ISum r;
    r.e = (int)__reduce_max_sync(0xffffffffu, (unsigned)p.e);
    r.s = warp_join(shift_round(p.m << kGuardWarp, r.e - p.e), 0);
    return r;
}

// FP32 values: 24 bits in a window of 54, two parts of 27.  A value within 2^-30 of the
// largest is added exactly (an FP64 tree adds exactly within 2^-24); one below loses at
// most 2^-54 of the largest, 16 2^-53 of the sum for a whole warp, where each value
// carries an FP32 rounding of 2^-24 itself.
__device__ __forceinline__ ISum warp_isum(float v)
{
    const Significand p = significand(v);
    ISum r;
    r.e = (int)__reduce_max_sync(0xffffffffu, (unsigned)p.e);
    const unsigned long long x = shift_round(p.m << 1, r.e - p.e);
    const unsigned long long hi = __reduce_add_sync(0xffffffffu, (unsigned)(x >> 27));
    const unsigned long long lo = __reduce_add_sync(0xffffffffu, (unsigned)x & 0x7ffffffu);
    r.s = ((hi << 27) + lo) << (kGuardWarp - 1);
    return r;
}

// The value of s 2^(e - 1075 - guard).
__device__ __forceinline__ double isum_value(const ISum &a, int guard = kGuardWarp)
{
    if (a.e >= kNotFinite) return __longlong_as_double((long long)kSigNaN);
    const double v = __ull2double_rn(a.s);
    const int k = a.e - 1075 - guard, e = (int)((unsigned long long)__double_as_longlong(v) >> 52) + k;
    if (a.s == 0ull || e < 1 || e > 2046) return scalbn(v, k);
    return __longlong_as_double(__double_as_longlong(v) + ((long long)k << 52));
}

// A partial sum as 64 bits with the highest one set, and the exponent of that bit
// (in the units of e): s = 0 has exponent 0.
struct Normal {
    unsigned long long v;
    int e;
};

__host__ __device__ __forceinline__ Normal isum_normal(const ISum &a)
{
#ifdef __CUDA_ARCH__
    const int z = __clzll((long long)a.s);
#else
    const int z = a.s ? __builtin_clzll(a.s) : 64;
#endif
    Normal r;
    r.v = z < 64 ? a.s << z : 0ull;
    r.e = a.e >= kNotFinite ? 2 * kNotFinite : z < 64 ? a.e + 64 - z : 0;
    return r;
}

// Its 55 bits (56 when rounding carries) aligned to the largest exponent.
__host__ __device__ __forceinline__ unsigned long long normal_term(const Normal &a, int emax)
{
    const int d = 8 + emax - a.e;
    const unsigned long long w = d > 63 ? 0ull : a.v >> d;
    return (w >> 1) + (w & 1ull);
}

// Sum over the warp of one partial sum per lane (at most 16 of them not zero).
__device__ __forceinline__ ISum warp_isum_parts(const ISum &a)
{
    const Normal n = isum_normal(a);
    ISum r;
    r.e = (int)__reduce_max_sync(0xffffffffu, (unsigned)n.e);
    const unsigned long long x = normal_term(n, r.e);
    const unsigned hi = __reduce_add_sync(0xffffffffu, (unsigned)(x >> 28));
    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)x & 0xfffffffu);
    r.s = ((unsigned long long)hi << 28) + lo;
    r.e -= 55;
    return r;
}

// All 32 lanes of a warp: the sum of n partial-sum packets once each carries
// 'seq' (packet j in lane j % 32; the same bits in every lane of every
// block).  False in every lane when the wait ran out.  NONNEG: none of the
// values is negative, and they are added in integers.
template <bool NONNEG>
__device__ __forceinline__ bool sum_slots(const Raw16 *slot, int n, uint32_t seq, EngCtl *ctl, double &sum)
{
    constexpr int U = 5;
    const int lane = (int)(threadIdx.x & 31u);
    double v = 0.0;
    ISum acc = {0ull, 1};
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
        if (NONNEG && n <= 32 * U) {
            // One round: every value aligned to the largest exponent of all.
            Significand p[U];
            int em = 1;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                p[u] = significand(__longlong_as_double((long long)a[u].v));
                em = max(em, p[u].e);
            }
            acc.e = (int)__reduce_max_sync(0xffffffffu, (unsigned)em);
#pragma unroll
            for (int u = 0; u < U; ++u) acc.s += shift_round(p[u].m << kGuardSlots, acc.e - p[u].e);
        } else {
            const double a01 = __longlong_as_double((long long)a[0].v) + __longlong_as_double((long long)a[1].v);
            const double a23 = __longlong_as_double((long long)a[2].v) + __longlong_as_double((long long)a[3].v);
            v += (a01 + a23) + __longlong_as_double((long long)a[4].v);
        }
    }
    ok = __all_sync(0xffffffffu, ok);
    if (NONNEG && n <= 32 * U) {
        // 160 values of 61 bits: 159 2^-61 lost in the alignment, 2^-53 and less in the roundings.
        acc.s = warp_join(acc.s, 5);
        sum = isum_value(acc, kGuardSlots - 5);
    } else {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        sum = v;
    }
    return ok;
}

// Reciprocal and quotient of positive doubles: the hardware's seed of 1 / b,
// e = 1 - b y, y (1 + e + e^2) from the geometric series, and for the quotient a
// last correction by its residual (Markstein, IBM J. Res. Dev. 34 (1990) 111).
// Five dependent FP64 operations of 60 clocks; operands outside
// [2^-900, 2^900] go through the ordinary division.
__device__ __forceinline__ bool mid_range(double v)
{
    const unsigned e = (unsigned)(__double_as_longlong(v) >> 52);    // sign and exponent
    return e - (1023u - 900u) <= 1800u;
}

__device__ __forceinline__ double seed_reciprocal(double b)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
    return y;
}

__device__ __forceinline__ double reciprocal(double b)
{
    if (!mid_range(b)) return 1.0 / b;
    const double y = seed_reciprocal(b), e = fma(-b, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// T: the type the quotient is used in; for float one term of the series leaves
// 2^-40.
template <typename T>
__device__ __forceinline__ T quotient(double a, double b)
{
    if (!mid_range(a) || !mid_range(b)) return (T)(a / b);
    const double y = seed_reciprocal(b), e = fma(-b, y, 1.0), q0 = a * y;
    if (sizeof(T) == 4) return (T)fma(q0, e, q0);
    const double q = fma(q0, fma(e, e, e), q0);
    return (T)fma(fma(-q, b, a), y, q);
}

// a > b for non-negative a, b that are not NaN (integer compares: the FP64 pipe's
// take 79 clocks).
__device__ __forceinline__ bool greater_nonneg(double a, double b)
{
    return __double_as_longlong(a) > __double_as_longlong(b);
}

__device__ __forceinline__ bool finite_bits(double v)
{
    return ((unsigned long long)__double_as_longlong(v) >> 52 & 0x7ffu) != 0x7ffu;
}

// A mixed system leaves for FP64 steps in the grid engine: its state before the
// decision and the sum that the decision is taken on, as that engine expects
// them from its own reliable update (x, r in global memory, the signal slots of
// slot 3 at odd parity).  Called by one thread of the system's first tile.
__device__ inline void hand_over(const OcLaunch &L, const EngSystem &Y, int sid, const EngState &S, double sum)
{
    for (int j = 0; j < Y.ntiles; ++j)
        L.sig[(size_t)5 * L.sig_stride + Y.part0 + j] =
            (unsigned long long)__double_as_longlong(j == 0 ? sum : 0.0);
    L.state[0][sid] = S;
    L.state[1][sid] = S;
}

}  // namespace hh
