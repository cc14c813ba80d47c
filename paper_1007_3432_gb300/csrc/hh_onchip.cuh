// On-chip CG engine: host/device shared declarations.
//
// For lattices whose CG vectors fit in the shared memory of the GPU's SMs,
// one launch keeps them there for the whole solve.  Every right-hand side is
// a system of its own, cut into go x gt tiles over (o, tau), o being x for
// d = 1 and z for d = 3 (a d = 3 tile holds whole x-y planes); one block owns
// one tile.  What a block needs of its neighbours' tiles (two o columns and
// one row of slices) and the partial sums travel through global memory in
// packets that carry their own phase number: a reader polls the packet
// itself, so neither a fence nor a barrier stands between a value and its use.
#pragma once

#include "hh_engine.cuh"

namespace hh {

constexpr int kOcMaxThreads = 512;

// How a solve of nsys systems of one lattice is laid out on the chip.
struct OcPlan {
    int ok;             // 0: the systems do not fit; use the grid engine
    int go, gt;         // tiles over o and tau
    int so, st;         // extents of the largest tile
    int threads;
    int x_global;       // x stays in global memory (read and written by its owner only)
    int mixed, cheb;
    int ex;             // exact-block form of M, first order (column form only)
    int cols;           // column form (hh_onchip_cols.cu): slices per thread at most; 0: tile form
    int sides;          // its halo columns per thread: 2 when a tile can have one o position
    size_t smem;        // dynamic shared memory per block
};

struct OcLaunch {
    const EngSystem *sys;
    EngState *state[2];
    EngCtl *ctl;
    unsigned char *pkt;             // per system: N packets of the vector M reads, N of t = M v
    ulonglong2 *slots;              // per system, replica and parity: one partial-sum packet per tile
    unsigned long long *seq;        // [0] last phase number of the launches before this one,
                                    // [1] of this one (see k_engine_reset)
    unsigned long long *sig;        // the grid engine's signal slots (hand-over of a mixed system)
    int sig_stride;
    int nsys, N;
    int go, gt, so, st;
    int x_global;
    int drop;                       // fault injection: tile (drop - 1) of system 0 never publishes
                                    // its partial sums; 0: none
    long long max_iters;
};

// Column form: spatial sites of a tile (one per thread) and threads, at most.
constexpr int kColMaxRow = 480;
constexpr int kColMaxThreads = kColMaxRow + 32;
// Threads of a block of the kernel for K slices per thread: 8 FP64 slices take
// more than the 128 registers a block of 512 can have.
constexpr int col_max_threads(size_t elem, int K)
{
    return elem == 8 && K == 8 ? 288 : kColMaxThreads;
}
const void *oc_cols_kernel(int d, bool mixed, bool cheb, bool ex, int K, int sides);

// Row stride of the staged vectors, in elements: constant, so that the K rows of
// a neighbour are one address and immediate offsets.  d = 3: (so + 2) P sites,
// at most three times the row.
template <int D>
constexpr int kColStride = D == 1 ? kColMaxRow + 2 : 3 * kColMaxRow;

// Its dynamic shared memory per block.
inline size_t oc_cols_smem(int d, bool mixed, bool cheb, bool ex, int K, int threads)
{
    const size_t rs = d == 1 ? kColStride<1> : kColStride<3>;
    return K * ((cheb ? 3 : ex ? 4 : 2) * rs + (cheb ? (size_t)(threads - 32) : 0)) * (mixed ? 4 : 8);
}

// Packet bytes per site and vector, and partial-sum packets per system.
inline size_t oc_packet_bytes(bool mixed) { return mixed ? 8 : 16; }
constexpr int kOcMaxTiles = 608;
constexpr int kOcReplicas = 8;

// First phase number of a launch after 'last', the last of the launches before it.
// Packets compare its low 32 bits and cleared ones carry 0, so a launch that could
// reach a multiple of 2^32 (2^28 phases are minutes of one solve) starts behind it.
__host__ __device__ inline unsigned long long oc_first_phase(unsigned long long last)
{
    const unsigned long long first = last + 1, low = first & 0xffffffffull;
    if (low == 0) return first + 1;
    return low > 0xf0000000ull ? (((first >> 32) + 1) << 32) + 1 : first;
}

// Systems of N sites that can lie on the chip at most: the tile form keeps at least four
// vectors (links, p, t, r) in shared memory, the column form's registers hold fewer sites.
inline long long oc_most_systems(long long N, bool mixed, int nsm, size_t smem_sm)
{
    return (long long)nsm * (long long)(smem_sm / (4 * (mixed ? 4 : 8))) / N;
}

// Layout for nsys systems, on nsm SMs with smem_sm bytes of shared memory per
// SM and smem_blk at most per block.  forms: 1 the faster form, 2 the tile form,
// 3 the column form only.
OcPlan oc_plan(int d, int nx, int ntau, int nsys, bool mixed, bool cheb, bool ex, int nsm, size_t smem_sm, size_t smem_blk,
               int forms);

// Blocks of a layout's kernel that one SM holds at once.
int oc_max_blocks(const OcPlan &P, int d);

// Launches the solve (cooperative: its blocks wait on one another).
cudaError_t oc_launch(const OcLaunch &L, const OcPlan &P, int d, cudaStream_t st);

}  // namespace hh
