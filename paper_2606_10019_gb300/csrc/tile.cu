// The pair pass as a kernel (tile.cuh) in all its passes and schedules, and the
// packing of the work items that its warps take.
#include "common.cuh"
#include "pair.cuh"
#include "perdevice.cuh"
#include "tile.cuh"

namespace gcvo {
namespace {

template <int MODE, bool ISO, int FD, int SUB, bool WIDE = false>
__global__ void __launch_bounds__(PAIR_WARPS * 32, MODE == PAIR_EVAL ? 5 : 4) k_tile(PairArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];   // PAIR_WARPS stages
    StageT<MODE, FD> *stage = reinterpret_cast<StageT<MODE, FD> *>(smem_raw);
    tile_init(stage);
    unsigned parity = 0;
    tile_pass<MODE, ISO, FD, SUB, WIDE>(a, stage, parity);
}

// Work-item packing over the sorted source points (keys: problem << 30 |
// Morton code of the fine voxels of edge rho / 4): one item per sub-tile.
// Start of each point's run of equal keys >> shift (input of a max-scan).
__global__ void k_seg_heads(const unsigned long long *keys, int64_t n, int shift, int *seg) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const bool head = i == 0 || (keys[i] >> shift) != (keys[i - 1] >> shift);
    seg[i] = head ? (int)i : 0;
}

// Sub-tile heads: every sub-th point of a run of one voxel.
__global__ void k_sub_heads(const int *seg2, int64_t n, int sub, int *sid) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    sid[i] = ((int)i - seg2[i]) % sub == 0 ? 1 : 0;
}

// Each sub-tile head writes its item word: first point << 6 | points.
__global__ void k_sub_count(const int *sid, int64_t n, int *cnt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    atomicAdd(cnt + sid[i] - 1, 1);
}

__global__ void k_fill_items(const unsigned long long *keys, const int *sid, const int *cnt, int64_t n, int *items,
                             int *item_prob) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (!(i == 0 || sid[i] != sid[i - 1])) return;
    const int it = sid[i] - 1;
    items[it] = (int)(((unsigned)i << 6) | (unsigned)cnt[it]);
    item_prob[it] = (int)(keys[i] >> 30);
}

// Item range of each problem: its points are [off, off + n).
__global__ void k_item_ranges(int np, const int64_t *point_off, const int *n_pts, const int *sid, ProbDev *probs) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    const int64_t f = point_off[p];
    probs[p].w0 = sid[f] - 1;
    probs[p].w1 = sid[f + n_pts[p] - 1];
}

// One block: each problem's finalize chunks (FIN_CHUNK of its work items
// each) get consecutive indices [c0, c1); *n_chunks receives the total.
constexpr int CHUNK_THREADS = 1024;
__global__ void __launch_bounds__(CHUNK_THREADS) k_chunk_ranges(int np, ProbDev *probs, int *n_chunks) {
    __shared__ int sc[CHUNK_THREADS];
    const int per = (np + CHUNK_THREADS - 1) / CHUNK_THREADS;
    const int p0 = threadIdx.x * per, p1 = min(np, p0 + per);
    int acc = 0;
    for (int p = p0; p < p1; ++p) acc += (probs[p].w1 - probs[p].w0 + FIN_CHUNK - 1) / FIN_CHUNK;
    sc[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 1; o < CHUNK_THREADS; o <<= 1) {
        const int v = threadIdx.x >= o ? sc[threadIdx.x - o] : 0;
        __syncthreads();
        sc[threadIdx.x] += v;
        __syncthreads();
    }
    int c = sc[threadIdx.x] - acc;
    for (int p = p0; p < p1; ++p) {
        probs[p].c0 = c;
        c += (probs[p].w1 - probs[p].w0 + FIN_CHUNK - 1) / FIN_CHUNK;
        probs[p].c1 = c;
    }
    if (threadIdx.x == CHUNK_THREADS - 1) *n_chunks = sc[threadIdx.x];
}

}  // namespace

// ---------------------------------------------------------------------------
// Host launchers.
// ---------------------------------------------------------------------------
// The opt-in above the 48 KB default, made once per kernel instance and device.
template <int MODE, bool ISO, int FD, int SUB, bool WIDE = false>
static cudaError_t tile_smem_optin() {
    static PerDevice<cudaError_t> once;
    return once.get([] {
        return cudaFuncSetAttribute(k_tile<MODE, ISO, FD, SUB, WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)tile_smem_bytes<MODE, FD>());
    });
}

template <int MODE, bool ISO, int FD, int SUB, bool WIDE = false>
static cudaError_t launch_tile_t(const PairArgs &a, int grid, cudaStream_t s) {
    const cudaError_t e = tile_smem_optin<MODE, ISO, FD, SUB, WIDE>();
    if (e != cudaSuccess) return e;
    k_tile<MODE, ISO, FD, SUB, WIDE><<<grid, PAIR_WARPS * 32, tile_smem_bytes<MODE, FD>(), s>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

template <int MODE, bool ISO, int FD, int SUB>
static int occupancy_t() {
    int nb = 0;
    if (tile_smem_optin<MODE, ISO, FD, SUB>() != cudaSuccess) return 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_tile<MODE, ISO, FD, SUB>, PAIR_WARPS * 32,
                                                  tile_smem_bytes<MODE, FD>());
    return nb;
}

// All three passes in all four schedules (the line-search pass of G-CVO-1
// and the G-CVO-E pass run over the same items as the evaluation pass).
#define PAIR_VARIANTS_U(X, M, U) \
    X(M, false, 1, U) X(M, false, 3, U) X(M, false, 7, U) X(M, true, 1, U) X(M, true, 3, U) X(M, true, 7, U)
#define PAIR_VARIANTS_M(X, M) \
    PAIR_VARIANTS_U(X, M, 4) PAIR_VARIANTS_U(X, M, 8) PAIR_VARIANTS_U(X, M, 16) PAIR_VARIANTS_U(X, M, 32)
#define PAIR_VARIANTS(X) \
    PAIR_VARIANTS_M(X, PAIR_EVAL) PAIR_VARIANTS_M(X, PAIR_LINESEARCH) PAIR_VARIANTS_M(X, PAIR_EXACT)

int pair_sub_for(int, int sub) { return sub == 4 || sub == 16 || sub == 32 ? sub : 8; }

// The kernel instance of a feature count: 1, up to 3, or up to 7 channels.
static int fd_class(int fd) { return fd <= 1 ? 1 : fd <= 3 ? 3 : 7; }

int pair_blocks_per_sm(int mode, bool iso, int fd, int sub) {
    sub = pair_sub_for(mode, sub);
#define OCC(M, I, F, U) \
    if (mode == M && iso == I && fd_class(fd) == F && sub == U) return occupancy_t<M, I, F, U>();
    PAIR_VARIANTS(OCC)
#undef OCC
    return 1;
}

cudaError_t launch_pair(const PairArgs &a, int mode, bool iso, int fd, int sub, int grid, cudaStream_t s) {
    sub = pair_sub_for(mode, sub);
#define L(M, I, F, U) \
    if (mode == M && iso == I && fd_class(fd) == F && sub == U) return launch_tile_t<M, I, F, U>(a, grid, s);
    PAIR_VARIANTS(L)
#undef L
    return cudaErrorInvalidValue;
}

cudaError_t launch_pair_unsorted(const PairArgs &a, bool iso, int fd, int grid, cudaStream_t s) {
    if (iso) return launch_pair(a, PAIR_EVAL, true, fd, 8, grid, s);   // one list anyway
    return fd <= 1 ? launch_tile_t<PAIR_EVAL, false, 1, 8, true>(a, grid, s)
                   : launch_tile_t<PAIR_EVAL, false, 3, 8, true>(a, grid, s);
}

gcvo_status pack_items(int np, const unsigned long long *keys, int64_t n, int sub, int level,
                       const int64_t *point_off, const int *n_pts, int *tmp, int *items, int *item_prob,
                       int *d_nitems, ProbDev *probs, int *n_chunks, void *scan_tmp, cudaStream_t s) {
    if (n >= (1LL << 26) || (sub != 4 && sub != 8 && sub != 16 && sub != 32) || level < 0 || level > 3)
        return GCVO_ERR_CAPACITY;
    const size_t stride = ((size_t)n + 63) / 64 * 64;
    int *seg2 = tmp, *sid = tmp + stride, *cnt = tmp + 2 * stride;
    const unsigned blocks = (unsigned)((n + 255) / 256);
    k_seg_heads<<<blocks, 256, 0, s>>>(keys, n, 3 * level, seg2);
    count_launches(1);
    GCVO_CUDA(cudaGetLastError());
    GCVO_TRY(scan_inclusive_max(seg2, n, scan_tmp, s));
    k_sub_heads<<<blocks, 256, 0, s>>>(seg2, n, sub, sid);
    count_launches(1);
    GCVO_CUDA(cudaGetLastError());
    GCVO_TRY(scan_inclusive_sum(sid, n, scan_tmp, s));
    GCVO_CUDA(cudaMemsetAsync(cnt, 0, (size_t)n * sizeof(int), s));
    k_sub_count<<<blocks, 256, 0, s>>>(sid, n, cnt);
    k_fill_items<<<blocks, 256, 0, s>>>(keys, sid, cnt, n, items, item_prob);
    k_item_ranges<<<(np + 127) / 128, 128, 0, s>>>(np, point_off, n_pts, sid, probs);
    k_chunk_ranges<<<1, CHUNK_THREADS, 0, s>>>(np, probs, n_chunks);
    count_launches(4);
    GCVO_CUDA(cudaGetLastError());
    GCVO_CUDA(cudaMemcpyAsync(d_nitems, sid + n - 1, sizeof(int), cudaMemcpyDeviceToDevice, s));
    return GCVO_OK;
}

}  // namespace gcvo
