// Stable LSD radix sort of keys and their places inside one thread-block
// cluster.
//
// A few thousand to a few ten thousand keys are far too little work for a
// grid-wide sort: at 20,000 keys its 24 launches (histogram, copy, three scan
// launches and scatter per 8-bit digit) took 181 us for 240 KB of data, all
// of it launch and memory latency (31-bit keys, warm; here: 32 us; 2,000 keys
// 131 -> 18 us; 65,536 keys 186 -> 45 us).  Here the keys stay in the shared memory
// of up to 16 SMs for the whole sort, each packed with its first place into
// 8 bytes, and a pass costs two cluster barriers:
//  1. every warp ranks its keys by digit (ballots group equal digits, a
//     per-warp table counts them in order);
//  2. the block turns its warps' tables into offsets within the block and
//     publishes its digit totals; after a cluster barrier every block reads
//     all blocks' totals through distributed shared memory, which gives each
//     digit's first place in the cluster-wide order;
//  3. every key goes straight to its place in the shared memory of the block
//     that owns it, and a second barrier ends the pass.
// Block r of the cluster holds places [r * TILE, (r + 1) * TILE).
#pragma once

#include "common.cuh"
#include "perdevice.cuh"

namespace gcvo {
namespace csort {

constexpr int THREADS = 1024, WARPS = THREADS / 32, RADIX = 256;
constexpr int MAX_ITEMS = 4;      // keys per thread
constexpr int MAX_BLOCKS = 16;    // of a cluster (8 is the portable size)
constexpr int IDX_BITS = 16;      // of a place
constexpr int MAX_KEY_BITS = 64 - IDX_BITS;
constexpr int64_t MAX_N = (int64_t)MAX_BLOCKS * MAX_ITEMS * THREADS;
static_assert(MAX_N == (int64_t)1 << IDX_BITS, "a place fits in its bits");

template <int ITEMS>
struct Smem {
    static constexpr int TILE = THREADS * ITEMS;
    unsigned long long key[2][TILE];     // key << IDX_BITS | first place
    unsigned short hist[WARPS][RADIX];   // keys of a warp per digit, then their offset in the block
    int total[RADIX];                    // keys of the block per digit, read by the other blocks
    int base[RADIX];                     // place of the block's first key of each digit
    int wsum[RADIX / 32];
};
static_assert(sizeof(Smem<MAX_ITEMS>) <= 227 * 1024, "the largest tile fits in shared memory");

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_blocks() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// Barrier over the cluster (a hardware barrier: no block spins).
__device__ __forceinline__ void cluster_barrier(unsigned nblk) {
    if (nblk > 1)
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    else
        __syncthreads();
}
// The address in block `rank` of the cluster of a variable of this block's shared memory.
__device__ __forceinline__ uint32_t cluster_addr(const void *p, unsigned rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(a)
                 : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}

// The lanes with the same 8-bit digit d, among the lanes in `valid`: one
// ballot per bit.
__device__ __forceinline__ unsigned same_digit(int d, unsigned valid) {
    unsigned peers = valid;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const unsigned ones = __ballot_sync(0xffffffffu, (d >> b) & 1);
        peers &= (d >> b) & 1 ? ones : ~ones;
    }
    return peers;
}

// Sorts the n keys of the cluster by their low `bits` bits.  The block's
// keys are in S.key[0] (places [rank * TILE, ..)), packed with their places,
// and need not be visible to the other threads yet; returns the index of the
// buffer that holds its sorted ones.
template <int ITEMS>
__device__ int sort(Smem<ITEMS> &S, int n, int bits) {
    constexpr int TILE = Smem<ITEMS>::TILE;
    const unsigned rank = cluster_rank(), nblk = cluster_blocks();
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int mine = min(max(n - (int)rank * TILE, 0), TILE);
    const unsigned lt = (1u << lane) - 1u;
    int cur = 0;
    // every block has started before another writes to its buffers
    cluster_barrier(nblk);
    for (int pass = 0; 8 * pass < bits; ++pass, cur ^= 1) {
        unsigned *row = reinterpret_cast<unsigned *>(S.hist[w]);
#pragma unroll
        for (int k = 0; k < RADIX / 64; ++k) row[lane + 32 * k] = 0u;
        __syncwarp();
        unsigned long long key[ITEMS];
        int dig[ITEMS], off[ITEMS];
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int i = w * (32 * ITEMS) + 32 * k + lane;
            key[k] = S.key[cur][i];
            // byte IDX_BITS / 8 + pass of the packed key
            dig[k] = (int)(__byte_perm((unsigned)key[k], (unsigned)(key[k] >> 32), IDX_BITS / 8 + pass) & 255u);
            const unsigned peers = same_digit(dig[k], __ballot_sync(0xffffffffu, i < mine));
            const int before = __popc(peers & lt);
            int first = 0;
            if (i < mine) first = S.hist[w][dig[k]];
            __syncwarp();
            if (i < mine && before == 0) S.hist[w][dig[k]] = (unsigned short)(first + __popc(peers));
            __syncwarp();
            off[k] = first + before;
        }
        __syncthreads();
        {
            // 4 threads per digit, 8 warps each
            const int d = tid >> 2, part = tid & 3;
            int cnt[WARPS / 4], sum = 0;
#pragma unroll
            for (int q = 0; q < WARPS / 4; ++q) {
                cnt[q] = S.hist[part * (WARPS / 4) + q][d];
                sum += cnt[q];
            }
            int incl = sum;
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o, 4);
                if (part >= o) incl += v;
            }
            int at = incl - sum;
#pragma unroll
            for (int q = 0; q < WARPS / 4; ++q) {
                S.hist[part * (WARPS / 4) + q][d] = (unsigned short)at;
                at += cnt[q];
            }
            if (part == 3) S.total[d] = incl;
        }
        cluster_barrier(nblk);
        int before = 0;
        if (tid < RADIX) {
            int all = 0;
#pragma unroll 4
            for (unsigned q = 0; q < nblk; ++q) {
                int v;
                asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(cluster_addr(&S.total[tid], q)));
                if (q < rank) before += v;
                all += v;
            }
            int incl = all;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            if (lane == 31) S.wsum[w] = incl;
            before += incl - all;
        }
        __syncthreads();
        if (tid < RADIX) {
            for (int q = 0; q < w; ++q) before += S.wsum[q];
            S.base[tid] = before;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int i = w * (32 * ITEMS) + 32 * k + lane;
            if (i < mine) {
                const int g = S.base[dig[k]] + S.hist[w][dig[k]] + off[k];
                asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(
                                 cluster_addr(&S.key[cur ^ 1][g % TILE], (unsigned)(g / TILE))),
                             "l"(key[k])
                             : "memory");
            }
        }
        cluster_barrier(nblk);
    }
    return cur;
}

// Opens a kernel with an Smem<ITEMS> to all clusters on the current device and
// returns the sizes of which it can hold at least one (bit b: 2^b blocks).  A
// partition with few SMs to a GPC may not place 8 or 16 blocks of 1024 threads;
// the callers then take the grid-wide sort, and a single problem the batched
// preparation.
template <int ITEMS, class Kernel>
unsigned cluster_sizes(Kernel kernel) {
    unsigned sizes = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem<ITEMS>)) == cudaSuccess &&
        cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess)
        for (int b = 0; 1 << b <= MAX_BLOCKS; ++b) {
            cudaLaunchConfig_t cfg{};
            cfg.gridDim = dim3(1u << b);
            cfg.blockDim = dim3(THREADS);
            cfg.dynamicSmemBytes = sizeof(Smem<ITEMS>);
            cudaLaunchAttribute at{};
            at.id = cudaLaunchAttributeClusterDimension;
            at.val.clusterDim.x = 1u << b;
            at.val.clusterDim.y = at.val.clusterDim.z = 1;
            cfg.attrs = &at;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n > 0) sizes |= 1u << b;
        }
    cudaGetLastError();   // a size that does not fit is no error
    return sizes;
}

// The launch of a cluster of `blocks` blocks among those sizes.
inline bool placed(unsigned sizes, int blocks) {
    int b = 0;
    while (1 << b < blocks) ++b;
    return (sizes >> b & 1u) != 0;
}

// Keys per thread and blocks of a cluster for n keys (0 items: too many).
// Up to 2048 keys one block alone is fastest (2,000 keys of 31 bits: 18.0 us,
// two blocks 19.2, four 20.0: a cluster barrier costs more than a second key
// per thread); beyond that one key per thread over more blocks (4,096 keys:
// 20.4 us on four blocks, 24.6 on one), two and four only where 16 blocks
// are too few (20,000 keys: 31.6 us on 16 blocks of two, 36.7 on 8 of four).
inline void shape(int64_t n, int &items, int &blocks) {
    items = 0;
    blocks = 1;
    if (n > MAX_N) return;
    items = n <= THREADS ? 1 : n <= 2 * THREADS ? 2 : n <= MAX_BLOCKS * THREADS ? 1 : n <= 2 * MAX_BLOCKS * THREADS ? 2 : 4;
    while ((int64_t)blocks * items * THREADS < n) blocks *= 2;
}

}  // namespace csort
}  // namespace gcvo
