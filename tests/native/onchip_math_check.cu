// Checks of the on-chip engine's arithmetic helpers (hh_onchip_dev.cuh): the
// integer sums over a warp, a block of 16 warps and up to 160 partial-sum
// packets, and (with a GPU) the quotient and reciprocal.
//
//   onchip_math_check        the sums' integer arithmetic, emulated on the host,
//                            against exact sums: within the bounds stated beside it
//   onchip_math_check gpu    the device functions: sums bit for bit the emulated ones,
//                            quotients against the division
//
// Prints the largest errors and "ok", or the first failure and exits 1.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "../../paper_1007_3432_gb300/csrc/hh_onchip_dev.cuh"

using namespace hh;
typedef unsigned long long u64;

static Significand sig_of(double v)
{
    u64 b;
    std::memcpy(&b, &v, 8);
    return significand_bits(b);
}

static Significand sig_of(float v)
{
    unsigned b;
    std::memcpy(&b, &v, 4);
    return significand_bits32(b);
}

// What a warp's reductions give for one term per lane.
static u64 join_lanes(const u64 *x, int shift)
{
    unsigned s2 = 0, s1 = 0, s0 = 0;
    for (int i = 0; i < 32; ++i) {
        s2 += (unsigned)(x[i] >> 44);
        s1 += (unsigned)(x[i] >> 22) & 0x3fffffu;
        s0 += (unsigned)x[i] & 0x3fffffu;
    }
    return isum_join(s2, s1, s0, shift);
}

template <typename T>
static ISum emu_warp(const T *v)
{
    Significand p[32];
    ISum r = {0, 0};
    for (int i = 0; i < 32; ++i) {
        p[i] = sig_of(v[i]);
        if (p[i].e > r.e) r.e = p[i].e;
    }
    if constexpr (sizeof(T) == 4) {
        unsigned hi = 0, lo = 0;
        for (int i = 0; i < 32; ++i) {
            const u64 q = shift_round(p[i].m << 1, r.e - p[i].e);
            hi += (unsigned)(q >> 27);
            lo += (unsigned)q & 0x7ffffffu;
        }
        r.s = (((u64)hi << 27) + lo) << (kGuardWarp - 1);
    } else {
        u64 x[32];
        for (int i = 0; i < 32; ++i) x[i] = shift_round(p[i].m << kGuardWarp, r.e - p[i].e);
        r.s = join_lanes(x, 0);
    }
    return r;
}

static ISum emu_parts(const ISum *a, int n)
{
    ISum r = {0, 0};
    Normal q[16];
    for (int i = 0; i < n; ++i) {
        q[i] = isum_normal(a[i]);
        if (q[i].e > r.e) r.e = q[i].e;
    }
    unsigned hi = 0, lo = 0;
    for (int i = 0; i < n; ++i) {
        const u64 x = normal_term(q[i], r.e);
        hi += (unsigned)(x >> 28);
        lo += (unsigned)x & 0xfffffffu;
    }
    r.s = ((u64)hi << 28) + lo;
    r.e -= 55;
    return r;
}

static double value(const ISum &a, int guard)
{
    return a.e >= kNotFinite ? NAN : std::ldexp((double)a.s, a.e - 1075 - guard);
}

static double emu_slots(const double *v, int n)
{
    Significand p[160];
    ISum r = {0, 1};
    u64 x[32] = {};
    for (int i = 0; i < n; ++i) {
        p[i] = sig_of(v[i]);
        if (p[i].e > r.e) r.e = p[i].e;
    }
    for (int i = 0; i < n; ++i) x[i % 32] += shift_round(p[i].m << kGuardSlots, r.e - p[i].e);
    r.s = join_lanes(x, 5);
    return value(r, kGuardSlots - 5);
}

// Error of s against the exact sum of v, in units of 2^-53 of it.  The exact sum
// is formed in two doubles (two-sum); its own error is below 2^-100.
template <typename T>
static double error(double s, const T *v, int n)
{
    double hi = 0.0, lo = 0.0;
    for (int i = 0; i < n; ++i) {
        const double x = (double)v[i], t = hi + x, b = t - hi;
        lo += (hi - (t - b)) + (x - b);
        hi = t;
    }
    const double sum = hi + lo;
    if (sum == 0.0) return s == 0.0 ? 0.0 : INFINITY;
    return std::fabs((s - hi) - lo) / sum * 9007199254740992.0;
}

struct Draws {
    std::vector<double> v;  // 512 values a draw
    int n;
};

// Blocks of values: like sizes, sizes spread over many binades, zeros, and one
// large value beside many that all round the same way.
static Draws make_draws()
{
    Draws d;
    std::mt19937_64 g(17);
    auto unit = [&]() { return (double)(g() >> 11) * 0x1p-53; };
    d.n = 600;
    for (int k = 0; k < d.n; ++k) {
        const int spread = k % 6 == 0 ? 0 : (int)(g() % 90);
        for (int i = 0; i < 512; ++i) {
            double x = std::ldexp(0.5 + 0.5 * unit(), (int)(g() % (spread + 1)) - spread / 2);
            if (k % 6 == 1 && g() % 5 == 0) x = 0.0;
            if (k % 6 >= 4) {
                // one value of 1 per warp (or per block), the others just under or over
                // half a unit of 2^-53 .. 2^-60
                const bool big = k % 6 == 4 ? i % 32 == 0 : i == 0;
                const int q = 53 + (k / 6) % 9;
                x = big ? 1.0 : std::ldexp(k / 54 % 2 ? 1.0 - 0x1p-40 : 1.0 + 0x1p-40, -q);
            }
            if (k % 6 == 3) x = std::ldexp(x, -1040);       // denormal parts
            d.v.push_back(x);
        }
    }
    return d;
}

#define CUDA(e)                                                                     \
    do {                                                                            \
        cudaError_t r_ = (e);                                                       \
        if (r_ != cudaSuccess) {                                                    \
            std::printf("FAIL cuda: %s\n", cudaGetErrorString(r_));                 \
            return 1;                                                               \
        }                                                                           \
    } while (0)

// Block b: sums of its 512 values by warps (w64, w32), by the block (blk) and, of its
// first n values, as packets (slots).
__global__ void __launch_bounds__(512) k_sums(const double *v, Raw16 *pkt, EngCtl *ctl, double *w64, double *w32,
                                              double *blk, double *slots, int n)
{
    __shared__ ISum red[16];
    const int t = threadIdx.x, b = blockIdx.x;
    const double x = v[(size_t)b * 512 + t];
    const ISum a = warp_isum(x), f = warp_isum((float)x);
    if ((t & 31) == 0) {
        red[t >> 5] = a;
        w64[b * 16 + (t >> 5)] = isum_value(a);
        w32[b * 16 + (t >> 5)] = isum_value(f);
    }
    if (t < n) {
        pkt[(size_t)b * 160 + t].v = (u64)__double_as_longlong(x);
        pkt[(size_t)b * 160 + t].seq = 7;
    }
    __threadfence();
    __syncthreads();
    if (t < 32) {
        ISum p = {0ull, 1};
        if (t < 16) p = red[t];
        const double s = isum_value(warp_isum_parts(p));
        double q = 0.0;
        const bool ok = sum_slots<true>(pkt + (size_t)b * 160, n, 7, ctl, q);
        if (t == 0) {
            blk[b] = s;
            slots[b] = ok ? q : -1.0;
        }
    }
}

// Quotients and reciprocals of positive operands over many binades (the last
// eighth out of the fast range): counts of results that differ from the division, and
// the largest error of the reciprocal and of the FP32 quotient, in 2^-53 and 2^-24.
__global__ void k_quotients(const double *a, const double *b, int n, unsigned *differ, unsigned *rec53,
                            unsigned *f24)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double q = quotient<double>(a[i], b[i]), e = a[i] / b[i];
    if (__double_as_longlong(q) != __double_as_longlong(e)) atomicAdd(differ, 1u);
    const double r = reciprocal(b[i]);
    atomicMax(rec53, (unsigned)fmin(1e9, ceil(fabs(fma(r, b[i], -1.0)) * 0x1p53 * 16.0)));
    if (e < 1e38 && e > 1e-37) {
        const float f = quotient<float>(a[i], b[i]);
        atomicMax(f24, (unsigned)fmin(1e9, ceil(fabs((double)f / e - 1.0) * 0x1p24 * 4096.0)));
    }
}

int main(int argc, char **argv)
{
    const Draws d = make_draws();
    double worst_w = 0, worst_f = 0, worst_n = 0, worst_b = 0, worst_s = 0;
    const int counts[] = {160, 1, 37, 128};
    for (int k = 0; k < d.n; ++k) {
        const double *v = &d.v[(size_t)k * 512];
        ISum parts[16];
        for (int w = 0; w < 16; ++w) {
            parts[w] = emu_warp(v + 32 * w);
            worst_w = std::fmax(worst_w, error(value(parts[w], kGuardWarp), v + 32 * w, 32));
            float f[32];
            for (int i = 0; i < 32; ++i) f[i] = (float)v[32 * w + i];
            const double e = error(value(emu_warp(f), kGuardWarp), f, 32);
            worst_f = std::fmax(worst_f, e);
            float lo = INFINITY, hi = 0.0f;
            for (int i = 0; i < 32; ++i) {
                if (f[i] != 0.0f) lo = std::fmin(lo, f[i]);
                hi = std::fmax(hi, f[i]);
            }
            if (hi <= 0x1p29f * lo) worst_n = std::fmax(worst_n, e);
        }
        worst_b = std::fmax(worst_b, error(value(emu_parts(parts, 16), kGuardWarp), v, 512));
        for (int n : counts) worst_s = std::fmax(worst_s, error(emu_slots(v, n), v, n));
    }
    std::printf("errors in 2^-53 of the sum: warp %.2f, warp of floats %.2f (within 2^29: %.2f), block %.2f, "
                "packets %.2f\n", worst_w, worst_f, worst_n, worst_b, worst_s);
    // The bounds stated beside the sums.
    if (!(worst_w <= 2.0 && worst_f <= 17.0 && worst_n <= 1.0 && worst_b <= 6.0 && worst_s <= 2.0)) {
        std::printf("FAIL error of the sums\n");
        return 1;
    }
    for (double bad : {(double)INFINITY, (double)NAN}) {
        double v[32] = {};
        v[5] = bad;
        ISum p[16] = {};
        p[3] = emu_warp(v);
        if (p[3].e < kNotFinite || emu_parts(p, 16).e < kNotFinite || !std::isnan(emu_slots(v, 32))) {
            std::printf("FAIL not finite\n");
            return 1;
        }
    }
    if (argc < 2) {
        std::printf("ok\n");
        return 0;
    }

    // ---- device ----
    double *dv, *dw, *df, *db, *ds;
    Raw16 *dp;
    EngCtl *ctl;
    CUDA(cudaMalloc(&dv, d.v.size() * 8));
    CUDA(cudaMalloc(&dw, (size_t)d.n * 16 * 8));
    CUDA(cudaMalloc(&df, (size_t)d.n * 16 * 8));
    CUDA(cudaMalloc(&db, (size_t)d.n * 8));
    CUDA(cudaMalloc(&ds, (size_t)d.n * 8));
    CUDA(cudaMalloc(&dp, (size_t)d.n * 160 * sizeof(Raw16)));
    CUDA(cudaMalloc(&ctl, sizeof(EngCtl)));
    CUDA(cudaMemcpy(dv, d.v.data(), d.v.size() * 8, cudaMemcpyHostToDevice));
    EngCtl h = {};
    h.timeout_ns = 1000000000ll;
    CUDA(cudaMemcpy(ctl, &h, sizeof(h), cudaMemcpyHostToDevice));
    std::vector<double> w(d.n * 16), f(d.n * 16), b(d.n), s(d.n);
    for (int n : counts) {
        CUDA(cudaMemset(dp, 0, (size_t)d.n * 160 * sizeof(Raw16)));
        k_sums<<<d.n, 512>>>(dv, dp, ctl, dw, df, db, ds, n);
        CUDA(cudaGetLastError());
        CUDA(cudaMemcpy(w.data(), dw, w.size() * 8, cudaMemcpyDeviceToHost));
        CUDA(cudaMemcpy(f.data(), df, f.size() * 8, cudaMemcpyDeviceToHost));
        CUDA(cudaMemcpy(b.data(), db, b.size() * 8, cudaMemcpyDeviceToHost));
        CUDA(cudaMemcpy(s.data(), ds, s.size() * 8, cudaMemcpyDeviceToHost));
        for (int k = 0; k < d.n; ++k) {
            const double *v = &d.v[(size_t)k * 512];
            ISum parts[16];
            for (int q = 0; q < 16; ++q) {
                float x[32];
                for (int i = 0; i < 32; ++i) x[i] = (float)v[32 * q + i];
                parts[q] = emu_warp(v + 32 * q);
                if (w[k * 16 + q] != value(parts[q], kGuardWarp) || f[k * 16 + q] != value(emu_warp(x), kGuardWarp)) {
                    std::printf("FAIL device warp sum, draw %d warp %d\n", k, q);
                    return 1;
                }
            }
            if (b[k] != value(emu_parts(parts, 16), kGuardWarp) || s[k] != emu_slots(v, n)) {
                std::printf("FAIL device block or packet sum, draw %d, %d packets\n", k, n);
                return 1;
            }
        }
    }
    const int n = 640000;
    std::vector<double> qa(n), qb(n);
    std::mt19937_64 g(23);
    for (int i = 0; i < n; ++i) {
        const int sa = i % 8 == 7 ? 1000 : 400, sb = i % 8 == 7 ? 20 : 400;
        qa[i] = std::ldexp(1.0 + (double)(g() >> 12) * 0x1p-52, (int)(g() % (2 * sa)) - sa);
        qb[i] = std::ldexp(1.0 + (double)(g() >> 12) * 0x1p-52, (int)(g() % (2 * sb)) - sb);
    }
    double *ga, *gb;
    unsigned *cnt, out[3];
    CUDA(cudaMalloc(&ga, n * 8));
    CUDA(cudaMalloc(&gb, n * 8));
    CUDA(cudaMalloc(&cnt, 12));
    CUDA(cudaMemset(cnt, 0, 12));
    CUDA(cudaMemcpy(ga, qa.data(), n * 8, cudaMemcpyHostToDevice));
    CUDA(cudaMemcpy(gb, qb.data(), n * 8, cudaMemcpyHostToDevice));
    k_quotients<<<(n + 255) / 256, 256>>>(ga, gb, n, cnt, cnt + 1, cnt + 2);
    CUDA(cudaGetLastError());
    CUDA(cudaMemcpy(out, cnt, 12, cudaMemcpyDeviceToHost));
    std::printf("quotients that differ from the division %u of %d; reciprocal %.2f 2^-53; FP32 quotient %.4f 2^-24\n",
                out[0], n, out[1] / 16.0, out[2] / 4096.0);
    // Markstein's correction gives the rounded quotient when the reciprocal is within
    // half a unit; a last bit may differ where it is not.  The reciprocal: 2^-46 (e^3)
    // of series and two roundings.  FP32: half a unit and 2^-40.
    if (out[0] > (unsigned)n / 10000 || out[1] > 3 * 16 || out[2] > 4096 + 2) {
        std::printf("FAIL quotient\n");
        return 1;
    }
    std::printf("ok\n");
    return 0;
}
