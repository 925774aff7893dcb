// The register loop of Algorithm 1 with the Gauss-Newton step (G-CVO-2) as one
// cooperative kernel: pair pass, finalize and transform of every iteration
// with grid-wide barriers between, until no problem is active.
//
// An iteration on clouds of a few thousand points is a chain of short kernels:
// pair pass, finalize and transform took 31 us at 2,000 points, of which about
// a third were launches and their ramps; the graph that replayed them was
// built anew for every call, and its eight iterations ran to the end after the
// last problem had stopped.  In one kernel the phases cost a barrier each.
//
// Measured: a registration of 22 iterations at 2,000 points 940 -> 685 us (31
// us an iteration; pair pass 12, its barrier 6, finalize 9 to 12, transform and
// barrier 3), the tracking of a LiDAR frame 1454 -> 1274 us.  Of this 108 and
// 47 us are the finalize's step in fewer FP64 instructions (fin.cuh).  On batches
// of 50,000 to 600,000 points, whose phases are long against the launches, the
// graphs are 1 to 5 % faster while most problems are active, and this kernel
// where few run on (128 pairs, one of them to 186 iterations: 94.9 -> 79.7 ms).
// The other orders, and a context that times its kernels, keep the graphs.
//
// The blocks of a cooperative launch are all resident, so the barrier's spin
// ends; it is bounded all the same.  They hold every SM, and the kernels of other
// streams wait, so a launch takes some iterations only (loop_iters, capi.cu).
#include <algorithm>

#include "common.cuh"
#include "fin.cuh"
#include "pair.cuh"
#include "perdevice.cuh"
#include "srcdev.cuh"
#include "tile.cuh"

namespace gcvo {
namespace {

static_assert(FIN_THREADS == PAIR_WARPS * 32, "one block shape for all phases");
// the finalize's shared memory lies over the first warp's staged points, below its barrier
static_assert(sizeof(FinShared) <= offsetof(Stage3, bar) && sizeof(FinShared) <= offsetof(Stage7, bar),
              "the finalize fits in a stage");

constexpr int LOOP_SPINS = 1 << 24;   // polls of a barrier, several seconds

// All blocks of the grid; `round` counts this block's barriers.  False when a
// block did not arrive in time.
__device__ bool grid_barrier(unsigned *bar, unsigned &round) {
    __shared__ int arrived;
    __syncthreads();
    ++round;
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(bar, 1u);
        const unsigned want = round * gridDim.x;
        int spins = 0;
        unsigned seen;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
        } while (seen < want && ++spins < LOOP_SPINS);
        __threadfence();
        arrived = seen >= want;
    }
    __syncthreads();
    return arrived != 0;
}

template <bool ISO, int FD, int SUB>
__global__ void __launch_bounds__(PAIR_WARPS * 32, 5) k_loop(LoopArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using Stage = StageT<PAIR_EVAL, FD>;
    Stage *stage = reinterpret_cast<Stage *>(smem_raw);
    FinShared &S = *reinterpret_cast<FinShared *>(smem_raw);
    tile_init(stage);
    unsigned parity = 0, round = 0;
    bool ok = true;
    // nothing to do, or a wait of an earlier launch ran out (both change only
    // behind a barrier that every block has to reach, or to give up on)
    if (a.resumed && (*(volatile int *)a.fin.n_active <= 0 || (*(volatile unsigned *)a.pair.status_word & DEV_ERR_TIMEOUT)))
        return;
    for (int it = 0; it < a.max_iters; ++it) {
        ok = tile_pass<PAIR_EVAL, ISO, FD, SUB>(a.pair, stage, parity);
        if (!__syncthreads_and(ok)) break;
        if (!(ok = grid_barrier(a.barrier, round))) break;
        fin_chunks(a.fin, S);
        if (!(ok = grid_barrier(a.barrier, round))) break;
        if (*(volatile int *)a.fin.n_active <= 0) break;
        transform_points(a.tr, blockIdx.x, gridDim.x);
        if (it + 1 < a.max_iters && !(ok = grid_barrier(a.barrier, round))) break;
    }
    if (!ok && threadIdx.x == 0) atomicOr(a.pair.status_word, DEV_ERR_TIMEOUT);
}

template <bool ISO, int FD, int SUB>
cudaError_t launch_t(const LoopArgs &a, int blocks, int sm_count, cudaStream_t s) {
    constexpr size_t smem = tile_smem_bytes<PAIR_EVAL, FD>();
    static PerDevice<std::pair<cudaError_t, int>> setup;
    const auto [err, per_sm] = setup.get([] {
        int n = 0;
        cudaError_t e = cudaFuncSetAttribute(k_loop<ISO, FD, SUB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_loop<ISO, FD, SUB>, PAIR_WARPS * 32, smem);
        return std::make_pair(e, n);
    });
    if (err != cudaSuccess) return err;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)std::max(1, std::min(blocks, std::max(1, per_sm) * sm_count)));
    cfg.blockDim = dim3(PAIR_WARPS * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_loop<ISO, FD, SUB>, a);
    if (e == cudaSuccess) count_launches(1);
    return e;
}

template <bool ISO, int FD>
cudaError_t launch_sub(const LoopArgs &a, int sub, int blocks, int sm_count, cudaStream_t s) {
    switch (pair_sub_for(PAIR_EVAL, sub)) {
        case 4: return launch_t<ISO, FD, 4>(a, blocks, sm_count, s);
        case 16: return launch_t<ISO, FD, 16>(a, blocks, sm_count, s);
        case 32: return launch_t<ISO, FD, 32>(a, blocks, sm_count, s);
        default: return launch_t<ISO, FD, 8>(a, blocks, sm_count, s);
    }
}

}  // namespace

cudaError_t launch_loop(const LoopArgs &a, bool iso, int fd, int sub, int blocks, int sm_count, cudaStream_t s) {
    if (iso)
        return fd <= 1 ? launch_sub<true, 1>(a, sub, blocks, sm_count, s)
               : fd <= 3 ? launch_sub<true, 3>(a, sub, blocks, sm_count, s)
                         : launch_sub<true, 7>(a, sub, blocks, sm_count, s);
    return fd <= 1 ? launch_sub<false, 1>(a, sub, blocks, sm_count, s)
           : fd <= 3 ? launch_sub<false, 3>(a, sub, blocks, sm_count, s)
                     : launch_sub<false, 7>(a, sub, blocks, sm_count, s);
}

}  // namespace gcvo
