// Host-only check of the on-chip engine's layout rule over lattices, numbers of
// systems, precisions and register counts (the rule must hold for kernels that
// compile to fewer registers than today's): blocks are whole warps, tiles cover
// the lattice within the extents the kernel sizes its arrays by, and the blocks
// of all systems fit on the chip at once.  Prints the first failure and exits 1.
#include <cstdio>

#include "../../paper_1007_3432_gb300/csrc/hh_onchip_plan.cuh"

static int fail(const char *what, int d, int nx, int ntau, int nsys, int regs, long long v)
{
    std::printf("FAIL %s: d %d nx %d ntau %d nsys %d regs %d: %lld\n", what, d, nx, ntau, nsys, regs, v);
    return 1;
}

int main()
{
    const int nsm = 152;
    const size_t smem_sm = 228 * 1024, smem_blk = 227 * 1024;
    long long layouts = 0;
    for (int d : {1, 3})
        for (int nx : {2, 3, 5, 8, 10, 13, 16, 17, 20, 22, 33, 96, 731, 1024, 2048}) {
            if (d == 3 && nx > 22) continue;
            for (int ntau : {2, 5, 17, 24, 33, 48, 84, 96, 128})
                for (int nsys : {1, 2, 3, 4, 5, 8, 64})
                    for (int kind = 0; kind < 5; ++kind)
                        for (int forms = 1; forms <= 3; ++forms)
                            for (int regs : {40, 64, 80, 128, 168}) {
                                const bool mixed = kind & 1, cheb = kind == 2, ex = kind >= 3;
                                const hh::OcPlan p =
                                    hh::oc_choose(d, nx, ntau, nsys, mixed, cheb, ex, nsm, smem_sm, smem_blk, forms,
                                                  [&](const hh::OcPlan &) { return regs; },
                                                  [](const hh::OcPlan &) { return true; });
                                if (!p.ok) continue;
                                ++layouts;
#define CHECK(cond, v) \
    if (!(cond)) return fail(#cond, d, nx, ntau, nsys, regs, (long long)(v))
                                CHECK(p.threads % 32 == 0, p.threads);
                                CHECK(p.threads >= 64 && p.threads <= hh::kOcMaxThreads, p.threads);
                                CHECK(p.go >= 1 && p.go <= nx && p.gt >= 1 && p.gt <= ntau, p.go * p.gt);
                                CHECK(p.go * p.gt <= hh::kOcMaxTiles, p.go * p.gt);
                                for (int i = 0; i < p.go; ++i) {
                                    const int so = (int)((long long)(i + 1) * nx / p.go - (long long)i * nx / p.go);
                                    CHECK(so >= 1 && so <= p.so, so);
                                    if (p.cols && p.sides == 1) CHECK(so >= 2, so);
                                }
                                for (int i = 0; i < p.gt; ++i) {
                                    const int st = (int)((long long)(i + 1) * ntau / p.gt - (long long)i * ntau / p.gt);
                                    CHECK(st >= 1 && st <= p.st, st);
                                    if (p.cols) CHECK(st <= p.cols, st);
                                }
                                const int P = d == 3 ? nx * nx : 1;
                                if (p.cols) CHECK(p.threads - 32 >= p.so * P, p.threads);
                                // Blocks one SM holds: shared memory, registers of a partition.
                                long long m = (long long)(smem_sm / (p.smem + 1024));
                                const long long parts = (p.threads / 32 + 3) / 4, rm = 16384 / (regs * 32) / parts;
                                if (rm < m) m = rm;
                                CHECK(p.smem + 1024 <= smem_blk, p.smem);
                                CHECK((long long)p.go * p.gt * nsys <= m * nsm, m);
                                // The exchange buffers are allocated for these many.
                                const long long N = (long long)P * nx * ntau;
                                CHECK(nsys <= hh::oc_most_systems(N, mixed, nsm, smem_sm), N);
                            }
        }
    // When the occupancy query refuses the best layout, the next one is taken: 32 x 64
    // in FP64 is best in the column form, and fits in the tile form too.
    for (bool refuse : {false, true}) {
        const hh::OcPlan p = hh::oc_choose(1, 32, 64, 2, false, false, false, nsm, smem_sm, smem_blk, 1,
                                           [](const hh::OcPlan &) { return 64; },
                                           [=](const hh::OcPlan &q) { return !refuse || q.cols == 0; });
        if (!p.ok || (p.cols == 0) != refuse) return fail("next layout", 1, 32, 64, 2, 64, p.cols);
    }
    const hh::OcPlan none = hh::oc_choose(1, 32, 64, 2, false, false, false, nsm, smem_sm, smem_blk, 1,
                                          [](const hh::OcPlan &) { return 64; },
                                          [](const hh::OcPlan &) { return false; });
    if (none.ok) return fail("all refused", 1, 32, 64, 2, 64, none.cols);
    // Phase numbers go up, and the 2^28 of a launch hold no multiple of 2^32.
    for (unsigned long long last : {0ull, 1ull, 0xeffffffeull, 0xefffffffull, 0xf0000000ull, 0xfffffffeull, 0xffffffffull,
                                    0x100000000ull, 0x5ffffffffull, 0x600000000ull}) {
        const unsigned long long first = hh::oc_first_phase(last), end = first + 0x0fffffffull;
        if (first <= last || (first & 0xffffffffull) == 0 || first >> 32 != end >> 32)
            return fail("phase number", 0, 0, 0, 0, (int)last, (long long)first);
    }
    if (layouts < 10000) return fail("layouts", 0, 0, 0, 0, 0, layouts);
    std::printf("ok\n");
    return 0;
}
