// Per-point kNN covariances (gcvo_estimate_covariances, Eq. 7b and the
// eigenvalue bound that follows it) of a batch of clouds.
//
//  1. k_knn_sort: one thread-block cluster per cloud takes the cloud's box,
//     the Morton code of every point in it and sorts the points by it, all
//     in shared memory (csort.cuh).  Clouds of more points than a cluster
//     holds go through the grid-wide sort.
//  2. k_knn_search: one warp per point.  In Morton order the points of any
//     cell of any size 2^L voxels are one run, found by a binary search over
//     the codes, so one sorted array serves every search radius.  The warp
//     picks the smallest L at which the point's own cell holds about knn
//     points, and gathers the 2 x 2 x 2 cells of that size around the point
//     (16 lanes search the ends of their runs); every point nearer than the
//     block's nearest face has then been seen.  When the knn-th nearest is
//     farther than that, L grows.  The nearest points are kept sorted across
//     the lanes by (squared distance, index in the cloud), so the result
//     depends neither on the voxels nor on the other clouds of the batch.
//  3. k_knn_eig: the eigenvalue bound, one thread per point.
//
// The work is dependent loads and a selection, far from any bandwidth: with
// one thread per point the lanes of a warp walked neighbourhoods of different
// sizes (11 of 32 active) through a hash table rebuilt for three voxel sizes,
// with a read-back between, and 64-bit Jacobi sweeps on a GPU with 2 FP64
// results per SM and cycle.  Covariances of a 20,000-point LiDAR frame: 1824
// -> 164 us; of 32 clouds of 1,000 to 40,000 points: 3135 -> 866 us.
#include <algorithm>
#include <cstring>

#include "common.cuh"
#include "csort.cuh"

namespace gcvo {
namespace {

constexpr int KNN_AXIS_BITS = 16;       // voxels per axis: at most 2^16
constexpr int KNN_BOX = 7;              // ints per cloud: smallest xyz, smallest -xyz (ordered), bad
static_assert(3 * KNN_AXIS_BITS <= csort::MAX_KEY_BITS, "a Morton code fits in a sort key");

// One cloud of a batched covariance call (device copy).
struct KnnCloud {
    const float *xyz;     // 3 x n SoA
    float *cov;           // 6 x n SoA output
    int64_t n, off;       // points; index of the first one in the batch
    double eig_max, eig_ratio;
    double cell0;         // half the kernel range; 0: no eigenvalue bound
    int knn;
    int pad;
};

// Its voxels: 2^bits per axis, cubes of edge h from corner.
struct KnnGrid {
    float corner[3];
    float h, inv_h;
    int bits;
};

// The voxels of a box: edges of a quarter of half the kernel range, the scale
// of the neighbourhoods that the eigenvalue bound expects, or finer where n
// points on the box's largest face would lie closer; the search adapts from
// there, so the edge only has to be small enough.  Without a bound the finest.
__device__ KnnGrid knn_grid(const float mn[3], const float mx[3], int64_t n, double cell0) {
    KnnGrid g;
    double ext = 0.0;
    for (int a = 0; a < 3; ++a) {
        g.corner[a] = mn[a];
        ext = fmax(ext, (double)mx[a] - (double)mn[a]);
    }
    if (!(ext > 0.0) || !isfinite(ext)) {
        g.h = g.inv_h = 1.f;
        g.bits = 0;
        return g;
    }
    const double finest = ext / (double)((1 << KNN_AXIS_BITS) - 1);
    double h = finest;
    if (cell0 > 0.0) h = fmax(finest, fmin(0.25 * cell0, 0.5 * ext / sqrt((double)n)));
    g.h = (float)h;
    g.inv_h = (float)(1.0 / h);
    const int top = (int)fmin(floor(ext / h) + 1.0, (double)((1 << KNN_AXIS_BITS) - 1));
    g.bits = 32 - __clz(top);
    return g;
}

__device__ __forceinline__ unsigned long long spread3(unsigned v) {
    unsigned long long x = v & 0x1fffffu;
    x = (x | x << 32) & 0x1f00000000ffffull;
    x = (x | x << 16) & 0x1f0000ff0000ffull;
    x = (x | x << 8) & 0x100f00f00f00f00full;
    x = (x | x << 4) & 0x10c30c30c30c30c3ull;
    x = (x | x << 2) & 0x1249249249249249ull;
    return x;
}
__device__ __forceinline__ unsigned long long morton(int x, int y, int z) {
    return spread3((unsigned)x) | spread3((unsigned)y) << 1 | spread3((unsigned)z) << 2;
}

__device__ __forceinline__ int knn_voxel(float u, int bits) { return min(max((int)floorf(u), 0), (1 << bits) - 1); }

__device__ __forceinline__ unsigned long long knn_code(const KnnGrid &g, float x, float y, float z) {
    return morton(knn_voxel((x - g.corner[0]) * g.inv_h, g.bits), knn_voxel((y - g.corner[1]) * g.inv_h, g.bits),
                  knn_voxel((z - g.corner[2]) * g.inv_h, g.bits));
}

__device__ __forceinline__ int knn_enc(float f) {
    const int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float knn_dec(int k) { return __int_as_float(k >= 0 ? k : k ^ 0x7fffffff); }

// Box of the values that a block's threads hold: lowest of x, y, z, -x, -y,
// -z (ordered ints) and whether one is not finite, into out[KNN_BOX].
__device__ void knn_block_box(const float v[6], bool bad, int (*red)[KNN_BOX], int *out) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int e[KNN_BOX];
#pragma unroll
    for (int a = 0; a < 6; ++a) e[a] = __reduce_min_sync(0xffffffffu, knn_enc(v[a]));
    e[6] = __any_sync(0xffffffffu, bad) ? 0 : 1;
    if (lane == 0)
#pragma unroll
        for (int a = 0; a < KNN_BOX; ++a) red[w][a] = e[a];
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int a = 0; a < KNN_BOX; ++a) {
            const int m = __reduce_min_sync(0xffffffffu, lane < (int)(blockDim.x >> 5) ? red[lane][a] : 0x7fffffff);
            if (lane == 0) out[a] = m;
        }
    }
    __syncthreads();
}

// Cloud ids[c] of the launch in the cluster c: its grid, and its points in
// Morton order as (x, y, z, index in the cloud) with their codes.
template <int ITEMS>
__global__ void __launch_bounds__(csort::THREADS)
    k_knn_sort(const KnnCloud *cl, const int *ids, KnnGrid *grids, unsigned long long *code, float4 *pos, int *cloud,
               unsigned *status) {
    extern __shared__ __align__(16) unsigned char smem[];
    csort::Smem<ITEMS> &S = *reinterpret_cast<csort::Smem<ITEMS> *>(smem);
    __shared__ int red[csort::WARPS][KNN_BOX];
    __shared__ int box[KNN_BOX];
    __shared__ KnnGrid sg;
    constexpr int TILE = csort::Smem<ITEMS>::TILE;
    const unsigned rank = csort::cluster_rank(), nblk = csort::cluster_blocks();
    const int id = ids[blockIdx.x / nblk];
    const KnnCloud &c = cl[id];
    const int n = (int)c.n, first = (int)rank * TILE;
    const float *px = c.xyz, *py = px + n, *pz = py + n;
    float x[ITEMS], y[ITEMS], z[ITEMS];
    float v[6] = {INFINITY, INFINITY, INFINITY, INFINITY, INFINITY, INFINITY};
    bool bad = false;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const int i = first + k * csort::THREADS + (int)threadIdx.x;
        if (i < n) {
            x[k] = px[i];
            y[k] = py[i];
            z[k] = pz[i];
            bad |= !isfinite(x[k]) || !isfinite(y[k]) || !isfinite(z[k]);
            v[0] = fminf(v[0], x[k]);
            v[1] = fminf(v[1], y[k]);
            v[2] = fminf(v[2], z[k]);
            v[3] = fminf(v[3], -x[k]);
            v[4] = fminf(v[4], -y[k]);
            v[5] = fminf(v[5], -z[k]);
        }
    }
    knn_block_box(v, bad, red, box);
    csort::cluster_barrier(nblk);
    if (threadIdx.x < 32) {
        // lane q takes block q's box
        int e[KNN_BOX];
#pragma unroll
        for (int a = 0; a < KNN_BOX; ++a) {
            e[a] = 0x7fffffff;
            if (threadIdx.x < nblk)
                asm volatile("ld.shared::cluster.u32 %0, [%1];"
                             : "=r"(e[a])
                             : "r"(csort::cluster_addr(&box[a], threadIdx.x)));
            e[a] = __reduce_min_sync(0xffffffffu, e[a]);
        }
        if (threadIdx.x == 0) {
            const float mn[3] = {knn_dec(e[0]), knn_dec(e[1]), knn_dec(e[2])};
            const float mx[3] = {-knn_dec(e[3]), -knn_dec(e[4]), -knn_dec(e[5])};
            sg = knn_grid(mn, mx, n, c.cell0);
            if (rank == 0) {
                grids[id] = sg;
                if (e[6] == 0) atomicOr(status, DEV_ERR_NONFINITE);
            }
        }
    }
    __syncthreads();
    const KnnGrid g = sg;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const int i = k * csort::THREADS + (int)threadIdx.x;
        if (first + i < n)
            S.key[0][i] = knn_code(g, x[k], y[k], z[k]) << csort::IDX_BITS | (unsigned)(first + i);
    }
    const int b = csort::sort<ITEMS>(S, n, 3 * g.bits);
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const int i = k * csort::THREADS + (int)threadIdx.x;
        if (first + i < n) {
            const unsigned long long key = S.key[b][i];
            const int o = (int)(key & ((1u << csort::IDX_BITS) - 1u));
            const int64_t to = c.off + first + i;
            code[to] = key >> csort::IDX_BITS;
            pos[to] = make_float4(px[o], py[o], pz[o], __int_as_float(o));
            cloud[to] = id;
        }
    }
}

// The steps of k_knn_sort for a cloud that no cluster holds (or none that the
// device can place): its box, its
// codes, and after the grid-wide sort its points.
__global__ void __launch_bounds__(256) k_knn_box(const KnnCloud *cl, int id, int *box) {
    __shared__ int red[8][KNN_BOX];
    __shared__ int out[KNN_BOX];
    const KnnCloud &c = cl[id];
    float v[6] = {INFINITY, INFINITY, INFINITY, INFINITY, INFINITY, INFINITY};
    bool bad = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < c.n; i += (int64_t)gridDim.x * blockDim.x)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float p = c.xyz[a * c.n + i];
            bad |= !isfinite(p);
            v[a] = fminf(v[a], p);
            v[3 + a] = fminf(v[3 + a], -p);
        }
    knn_block_box(v, bad, red, out);
    if (threadIdx.x < KNN_BOX) atomicMin(box + threadIdx.x, out[threadIdx.x]);
}

__global__ void k_knn_codes(const KnnCloud *cl, int id, const int *box, KnnGrid *grids, unsigned long long *keys,
                            int *vals, unsigned *status) {
    const KnnCloud &c = cl[id];
    __shared__ KnnGrid sg;
    if (threadIdx.x == 0) {
        const float mn[3] = {knn_dec(box[0]), knn_dec(box[1]), knn_dec(box[2])};
        const float mx[3] = {-knn_dec(box[3]), -knn_dec(box[4]), -knn_dec(box[5])};
        sg = knn_grid(mn, mx, c.n, c.cell0);
        if (blockIdx.x == 0) {
            grids[id] = sg;
            if (box[6] == 0) atomicOr(status, DEV_ERR_NONFINITE);
        }
    }
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= c.n) return;
    keys[i] = knn_code(sg, c.xyz[i], c.xyz[c.n + i], c.xyz[2 * c.n + i]);
    vals[i] = (int)i;
}

__global__ void k_knn_place(const KnnCloud *cl, int id, const unsigned long long *keys, const int *vals,
                            unsigned long long *code, float4 *pos, int *cloud) {
    const KnnCloud &c = cl[id];
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= c.n) return;
    const int o = vals[i];
    code[c.off + i] = keys[i];
    pos[c.off + i] = make_float4(c.xyz[o], c.xyz[c.n + o], c.xyz[2 * c.n + o], __int_as_float(o));
    cloud[c.off + i] = id;
}

// First of the `n` ascending codes at `code` that is not below `key`.
__device__ __forceinline__ int lower_bound(const unsigned long long *code, int n, unsigned long long key) {
    int at = 0;
    for (int len = n; len > 0;) {
        const int half = len >> 1;
        if (__ldg(code + at + half) < key) {
            at += half + 1;
            len -= half + 1;
        } else {
            len = half;
        }
    }
    return at;
}

constexpr int KNN_WARPS = 8;
// Candidates above which a point's first block is tried smaller: 64 steps of a
// warp, against a binary search a level (1024: corner scenes 5 % faster still, but
// some LiDAR frames 183 -> 194 us; 4096: corner scenes 10 % slower).
constexpr int KNN_MANY = 2048;

// One entry of a warp's list of nearest points: the squared distance's bits
// above the index in the cloud (distances are not negative, so the order of
// the bits is the order of (distance, index)), and the point's sorted place.
struct KnnEntry {
    unsigned long long key;
    int at;
};

// Sum over the knn nearest points of (y - x)(y - x)^T / (knn - 1) for every
// point x of the batch, into the cloud's covariances.
__global__ void __launch_bounds__(KNN_WARPS * 32)
    k_knn_search(const KnnCloud *cl, const KnnGrid *grids, const unsigned long long *codes, const float4 *pos,
                 const int *cloud, int64_t N, const unsigned *status) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t t = (int64_t)blockIdx.x * KNN_WARPS + (threadIdx.x >> 5);
    if (t >= N || (*status & DEV_ERR_NONFINITE)) return;
    const int id = cloud[t];
    const KnnCloud &c = cl[id];
    const KnnGrid g = grids[id];
    const int n = (int)c.n, knn = c.knn;
    const unsigned long long *code = codes + c.off;
    const float4 *P = pos + c.off;
    const int me = (int)(t - c.off);
    const float4 q = P[me];
    const float u[3] = {(q.x - g.corner[0]) * g.inv_h, (q.y - g.corner[1]) * g.inv_h, (q.z - g.corner[2]) * g.inv_h};
    int vox[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) vox[a] = knn_voxel(u[a], g.bits);
    // the smallest cell of the point with two thirds of knn more points to
    // one side of it: on surfaces the block around it then holds 95 to 130
    // points, and 3 to 8 points in 100 need a larger one (knn points to one
    // side: 130 to 155 and 1 to 3; half of knn: 90 to 115 and 10 to 20)
    int L = max(g.bits, 1);
    {
        const unsigned long long k0 = code[me];
        const int away = (2 * knn + 2) / 3;
#pragma unroll
        for (int s = -1; s <= 1; s += 2) {
            const int o = me + s * away;
            if (o >= 0 && o < n) L = min(L, (66 - __clzll((long long)(k0 ^ code[o]))) / 3);
        }
        L = max(L, 1);
    }
    KnnEntry best{~0ull, 0};
    // A few points alone behind a boundary of large cells have their next ones in
    // the order far away, and a cell of that size may hold a third of the cloud:
    // smaller cells are tried first while the block around the point holds many.
    // The result is the same for any L.  One warp's 25,000 candidates were most of
    // the search of 66,000 points: covariances 1020 -> 401 us, of corner scenes of
    // 20,000 points 394 -> 134, of RGB-D frames up to 246 -> 145.
    bool down = true;
    for (;; ++L) {
        // lanes 0..7: first places of the 2 x 2 x 2 cells, the point's own
        // first (it holds the nearest points, and the list soon turns the
        // others' away); lanes 8..15: their ends
        const int cells = L >= g.bits ? 1 : 1 << (g.bits - L);
        int cell[3];
        float reach = INFINITY;
        bool inside = lane < 16;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int i0 = ((vox[a] >> (L - 1)) - 1) >> 1, own = (vox[a] >> L) - i0;
            if (i0 > 0) reach = fminf(reach, u[a] - (float)(i0 << L));
            if (i0 + 2 < cells) reach = fminf(reach, (float)((i0 + 2) << L) - u[a]);
            cell[a] = i0 + ((lane >> a & 1) ^ own);
            inside = inside && cell[a] >= 0 && cell[a] < cells;
        }
        int end = 0;
        if (inside) end = lower_bound(code, n, (morton(cell[0], cell[1], cell[2]) + (lane >> 3)) << (3 * L));
        const int last = __shfl_down_sync(FULL, end, 8);
        const int len = lane < 8 ? last - end : 0;
        // inclusive sums of the runs' lengths in lanes 0..7
        int incl = len;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const int v = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += v;
        }
        const int total = __shfl_sync(FULL, incl, 7);
        if (down && total > KNN_MANY && L > 1) {
            L -= 2;
            continue;
        }
        down = false;
        const bool all = L >= g.bits;
        if (total < knn && !all) continue;
        best.key = ~0ull;
        unsigned long long worst = ~0ull;   // the knn-th entry so far
        for (int base = 0; base < total; base += 32) {
            const int p = base + lane;
            // the run of place p: the first whose inclusive sum exceeds it
            int run = 0;
#pragma unroll
            for (int o = 4; o > 0; o >>= 1)
                if (__shfl_sync(FULL, incl, run + o - 1) <= p) run += o;
            const int before = __shfl_sync(FULL, incl - len, run & 7), start = __shfl_sync(FULL, end, run & 7);
            KnnEntry e{~0ull, 0};
            if (p < total) {
                e.at = start + (p - before);
                const float4 y = __ldg(P + e.at);
                const float ex = y.x - q.x, ey = y.y - q.y, ez = y.z - q.z;
                const float d2 = ex * ex + ey * ey + ez * ez;
                e.key = (unsigned long long)__float_as_uint(d2) << 32 | (unsigned)__float_as_int(y.w);
            }
            if (base == 0) {
                // bitonic sort of the first 32
#pragma unroll
                for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
                    for (int o = size >> 1; o > 0; o >>= 1) {
                        const unsigned long long ok = __shfl_xor_sync(FULL, e.key, o);
                        const int oa = __shfl_xor_sync(FULL, e.at, o);
                        const bool up = (lane & size) == 0 || size == 32;
                        const bool low = (lane & o) == 0;
                        if ((ok < e.key) == (low == up) && ok != e.key) {
                            e.key = ok;
                            e.at = oa;
                        }
                    }
                best = e;
                worst = __shfl_sync(FULL, best.key, knn - 1);
                continue;
            }
            unsigned todo = __ballot_sync(FULL, e.key < worst);
            while (todo) {
                const int from = __ffs(todo) - 1;
                const unsigned long long nk = __shfl_sync(FULL, e.key, from);
                const int na = __shfl_sync(FULL, e.at, from);
                const int rank = __popc(__ballot_sync(FULL, best.key < nk));
                const unsigned long long uk = __shfl_up_sync(FULL, best.key, 1);
                const int ua = __shfl_up_sync(FULL, best.at, 1);
                if (lane >= rank) {
                    best.key = lane == rank ? nk : uk;
                    best.at = lane == rank ? na : ua;
                }
                worst = __shfl_sync(FULL, best.key, knn - 1);
                todo &= __ballot_sync(FULL, e.key < worst) & ~(1u << from);
            }
        }
        if (all) break;
        // a voxel's float assignment may be off by a few rounding errors of u
        reach = (reach - 5e-7f * (float)(1 << g.bits)) * g.h * 0.9999f;
        const float far = __uint_as_float((unsigned)(worst >> 32));
        if (worst != ~0ull && reach > 0.f && far <= reach * reach) break;
    }
    // Sigma = 1/(n-1) sum (y - x)(y - x)^T, centred at the query point, in
    // ascending order of distance
    float d[3] = {0.f, 0.f, 0.f};
    if (lane < knn) {
        const float4 y = P[best.at];
        d[0] = y.x - q.x;
        d[1] = y.y - q.y;
        d[2] = y.z - q.z;
    }
    float S[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int m = 0; m < knn; ++m) {
        const float d0 = __shfl_sync(FULL, d[0], m), d1 = __shfl_sync(FULL, d[1], m), d2 = __shfl_sync(FULL, d[2], m);
        S[0] += d0 * d0;
        S[1] += d0 * d1;
        S[2] += d0 * d2;
        S[3] += d1 * d1;
        S[4] += d1 * d2;
        S[5] += d2 * d2;
    }
    float s = S[0];
#pragma unroll
    for (int k = 1; k < 6; ++k)
        if (lane == k) s = S[k];
    if (lane < 6) c.cov[(int64_t)lane * n + __float_as_int(q.w)] = s * (1.0f / (float)(knn - 1));
}

// Whether the entries of A' beside the diagonal d (e: 01, 02, 12) are small
// enough for the first-order clamp to [lo, hi]: E_pq^2 <= 2e-9 top |d_p - d_q|
// (the gaps less the rounding of d in FP32), top the largest clamped eigenvalue.
// Whatever the gap, an entry below 3e-9 top moves the result by no more, and
// between two eigenvalues on the same piece of the clamp (which meet on regular
// grids of points) the formula is exact but for the third: 1e-6 top will do.
// wide: the largest of d over top.
__device__ __forceinline__ bool eig_converged(const double (&d)[3], const double (&e)[3], float lo, float hi, float &wide) {
    const float x = (float)d[0], y = (float)d[1], z = (float)d[2], most = fmaxf(fmaxf(x, y), z);
    const float i = 1.0f / fmaxf(fminf(most, hi), lo), off = 2e-7f * most;
    wide = most * i;
    auto good = [&](float u, float v, double entry) {
        const float w = (float)entry * i;
        const bool same = (u <= lo) == (v <= lo) && (u >= hi) == (v >= hi);
        return w * w <= fmaxf(2e-9f * i * (fabsf(u - v) - off), same ? 1e-12f : 1e-17f);
    };
    return good(x, y, e[0]) && good(x, z, e[1]) && good(y, z, e[2]);
}

// Turns V until A' = V^T A V passes eig_converged, by sweeps of Jacobi's method
// in FP64; d and e: the diagonal of A' and its entries 01, 02, 12.  An angle is
// as good as FP32 makes it, which leaves 1e-7 of an entry, but its cosine and
// sine belong together to FP64 rounding (Newton steps), and V is made
// orthonormal again before every A'.
__device__ __noinline__ void eig_refine(const float *s, float lo, float hi, double (&V)[3][3], double (&d)[3], double (&e)[3]) {
    const double A[3][3] = {{s[0], s[1], s[2]}, {s[1], s[3], s[4]}, {s[2], s[4], s[5]}};
    for (int sweep = 0;; ++sweep) {
        double G[3][3], B[3][3], a[3][3];
        for (int p = 0; p < 3; ++p)
            for (int q = 0; q < 3; ++q)
                G[p][q] = (p == q ? 1.5 : 0.0) - 0.5 * (V[0][p] * V[0][q] + V[1][p] * V[1][q] + V[2][p] * V[2][q]);
        for (int r = 0; r < 3; ++r)
            for (int q = 0; q < 3; ++q) B[r][q] = V[r][0] * G[0][q] + V[r][1] * G[1][q] + V[r][2] * G[2][q];
        for (int r = 0; r < 3; ++r)
            for (int q = 0; q < 3; ++q) {
                V[r][q] = B[r][q];
                G[r][q] = A[r][0] * B[0][q] + A[r][1] * B[1][q] + A[r][2] * B[2][q];
            }
        for (int p = 0; p < 3; ++p)
            for (int q = p; q < 3; ++q) a[p][q] = a[q][p] = B[0][p] * G[0][q] + B[1][p] * G[1][q] + B[2][p] * G[2][q];
        for (int p = 0; p < 3; ++p) d[p] = a[p][p];
        e[0] = a[0][1];
        e[1] = a[0][2];
        e[2] = a[1][2];
        float wide;
        if (sweep == 8 || (sweep > 0 && eig_converged(d, e, lo, hi, wide))) return;
        for (int k = 0; k < 3; ++k) {
            const int p = k == 2 ? 1 : 0, q = k == 0 ? 1 : 2, r = 3 - p - q;
            const float den = 2.0f * (float)a[p][q];
            if (den == 0.f) continue;
            const float tau = (float)(a[q][q] - a[p][p]) / den;
            const double t = copysignf(1.0f, tau) / (fabsf(tau) + sqrtf(1.0f + tau * tau)), u = 1.0 + t * t;
            double c = rsqrtf((float)u);
            c = c * (1.5 - 0.5 * u * c * c);
            c = c * (1.5 - 0.5 * u * c * c);
            const double sn = t * c, app = a[p][p], aqq = a[q][q], apq = a[p][q], arp = a[r][p], arq = a[r][q];
            a[p][p] = c * c * app - 2.0 * c * sn * apq + sn * sn * aqq;
            a[q][q] = sn * sn * app + 2.0 * c * sn * apq + c * c * aqq;
            a[p][q] = a[q][p] = c * sn * (app - aqq) + (c * c - sn * sn) * apq;
            a[r][p] = a[p][r] = c * arp - sn * arq;
            a[r][q] = a[q][r] = sn * arp + c * arq;
            for (int m = 0; m < 3; ++m) {
                const double vp = V[m][p], vq = V[m][q];
                V[m][p] = c * vp - sn * vq;
                V[m][q] = sn * vp + c * vq;
            }
        }
    }
}

// Clamps the eigenvalues of every covariance to [eig_max / eig_ratio,
// eig_max].  FP64 sweeps of Jacobi's method would be most of the time
// (about 1500 FP64 operations per point, at 2 per SM and cycle), so the
// eigenvectors come from FP32 sweeps and FP64 only corrects them: with V the
// FP32 vectors made orthonormal to about 1e-13 by one Newton step, A' = V^T A V
// is diagonal up to E of about 1e-7 of the largest eigenvalue, and to first
// order in E (the Daleckii-Krein formula) the clamped matrix f(A') has f of
// the diagonal and E_pq (f(d_p) - f(d_q)) / (d_p - d_q) beside it: about 150
// FP64 operations.  The terms left out are E_pr E_rq times a second divided
// difference of f, which is at most the inverse of the largest gap among its
// three eigenvalues.  eig_converged keeps them below 4e-9 of the result's
// largest eigenvalue, a fifteenth of a float's rounding.  Points that miss it
// (elongated neighbourhoods: with the largest eigenvalue 1e4 times eig_max the
// formula alone was off by 4e-5) go through eig_refine; surfaces do not.
__global__ void __launch_bounds__(128) k_knn_eig(const KnnCloud *cl, const int *cloud, int64_t N, const unsigned *status) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= N || (*status & DEV_ERR_NONFINITE)) return;
    const KnnCloud &c = cl[cloud[t]];
    if (!(c.eig_max > 0.0)) return;
    const int64_t o = t - c.off;
    float s[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) s[k] = c.cov[k * c.n + o];
    // FP32 sweeps on the matrix scaled to a largest diagonal of about 1
    const float big = fmaxf(s[0], fmaxf(s[3], s[5]));
    const float sc = big > 1e-30f ? 1.0f / big : 1.0f;
    float a[3][3] = {{s[0] * sc, s[1] * sc, s[2] * sc}, {s[1] * sc, s[3] * sc, s[4] * sc}, {s[2] * sc, s[4] * sc, s[5] * sc}};
    float W[3][3] = {{1.f, 0.f, 0.f}, {0.f, 1.f, 0.f}, {0.f, 0.f, 1.f}};
    for (int sweep = 0; sweep < 8; ++sweep) {
        if (fabsf(a[0][1]) + fabsf(a[0][2]) + fabsf(a[1][2]) < 1e-8f) break;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int p = k == 2 ? 1 : 0, q = k == 0 ? 1 : 2;
            const float apq = a[p][q];
            if (apq == 0.f) continue;
            const float tau = (a[q][q] - a[p][p]) / (2.0f * apq);
            const float tn = copysignf(1.0f, tau) / (fabsf(tau) + sqrtf(1.0f + tau * tau));
            const float cs = rsqrtf(1.0f + tn * tn), sn = tn * cs;
            const int r = 3 - p - q;
            const float arp = a[r][p], arq = a[r][q];
            a[p][p] -= tn * apq;
            a[q][q] += tn * apq;
            a[p][q] = a[q][p] = 0.f;
            a[r][p] = a[p][r] = cs * arp - sn * arq;
            a[r][q] = a[q][r] = sn * arp + cs * arq;
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                const float vp = W[m][p], vq = W[m][q];
                W[m][p] = cs * vp - sn * vq;
                W[m][q] = sn * vp + cs * vq;
            }
        }
    }
    // V = W (3 I - W^T W) / 2
    double V[3][3];
    {
        double G[3][3];
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int q = p; q < 3; ++q)
                G[p][q] = G[q][p] = -0.5 * ((double)W[0][p] * W[0][q] + (double)W[1][p] * W[1][q] + (double)W[2][p] * W[2][q]);
#pragma unroll
        for (int p = 0; p < 3; ++p) G[p][p] += 1.5;
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int q = 0; q < 3; ++q) V[r][q] = W[r][0] * G[0][q] + W[r][1] * G[1][q] + W[r][2] * G[2][q];
    }
    const double A[3][3] = {{s[0], s[1], s[2]}, {s[1], s[3], s[4]}, {s[2], s[4], s[5]}};
    double F[3][3];   // f(A')
    {
        double AV[3][3], d[3], e[3], f[3];
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int q = 0; q < 3; ++q) AV[r][q] = A[r][0] * V[0][q] + A[r][1] * V[1][q] + A[r][2] * V[2][q];
        const double lo = c.eig_max / c.eig_ratio;
#pragma unroll
        for (int p = 0; p < 3; ++p) d[p] = V[0][p] * AV[0][p] + V[1][p] * AV[1][p] + V[2][p] * AV[2][p];
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int q = p + 1; q < 3; ++q)
                e[p + q - 1] = V[0][p] * AV[0][q] + V[1][p] * AV[1][q] + V[2][p] * AV[2][q];
        // V's own 1e-13 of the largest eigenvalue counts beyond 1e4 times the clamp
        float wide;
        if (!eig_converged(d, e, (float)lo, (float)c.eig_max, wide) || wide > 1e4f) {
            double Vr[3][3], dr[3], er[3];
#pragma unroll
            for (int r = 0; r < 9; ++r) Vr[r / 3][r % 3] = V[r / 3][r % 3];
            eig_refine(s, (float)lo, (float)c.eig_max, Vr, dr, er);
#pragma unroll
            for (int r = 0; r < 9; ++r) V[r / 3][r % 3] = Vr[r / 3][r % 3];
#pragma unroll
            for (int p = 0; p < 3; ++p) {
                d[p] = dr[p];
                e[p] = er[p];
            }
        }
#pragma unroll
        for (int p = 0; p < 3; ++p) F[p][p] = f[p] = fmin(fmax(d[p], lo), c.eig_max);
#pragma unroll
        for (int p = 0; p < 3; ++p)
#pragma unroll
            for (int q = p + 1; q < 3; ++q) {
                const float gap = (float)(d[p] - d[q]);
                const float slope = gap != 0.f ? (float)(f[p] - f[q]) / gap : (d[p] == f[p] ? 1.f : 0.f);
                F[p][q] = F[q][p] = e[p + q - 1] * (double)slope;
            }
    }
    double VF[3][3];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int q = 0; q < 3; ++q) VF[r][q] = V[r][0] * F[0][q] + V[r][1] * F[1][q] + V[r][2] * F[2][q];
    int k = 0;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int q = r; q < 3; ++q)
            c.cov[(int64_t)k++ * c.n + o] = (float)(VF[r][0] * V[q][0] + VF[r][1] * V[q][1] + VF[r][2] * V[q][2]);
}

size_t al256(size_t b) { return (b + 255) & ~size_t(255); }

template <int ITEMS>
bool knn_sort_fits(int blocks) {
    static PerDevice<unsigned> sizes;
    return csort::placed(sizes.get([] { return csort::cluster_sizes<ITEMS>(k_knn_sort<ITEMS>); }), blocks);
}

bool knn_sort_fits(int items, int blocks) {
    switch (items) {
        case 1: return knn_sort_fits<1>(blocks);
        case 2: return knn_sort_fits<2>(blocks);
        case 4: return knn_sort_fits<4>(blocks);
        default: return false;   // too many points
    }
}

template <int ITEMS>
gcvo_status launch_knn_sort(const KnnCloud *cl, const int *ids, int n_clouds, int blocks, KnnGrid *grids,
                            unsigned long long *code, float4 *pos, int *cloud, unsigned *status, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(blocks * n_clouds));
    cfg.blockDim = dim3(csort::THREADS);
    cfg.dynamicSmemBytes = sizeof(csort::Smem<ITEMS>);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)blocks;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    GCVO_CUDA(cudaLaunchKernelEx(&cfg, k_knn_sort<ITEMS>, cl, ids, grids, code, pos, cloud, status));
    count_launches(1);
    return GCVO_OK;
}

}  // namespace

size_t knn_meta_bytes(int n_clouds) {
    const size_t C = (size_t)std::max(n_clouds, 1);
    return al256(C * sizeof(KnnCloud)) + al256(C * sizeof(KnnGrid)) + al256(C * sizeof(int)) + al256(KNN_BOX * sizeof(int));
}

gcvo_status knn_covariances(gcvo_ctx *ctx, int n_clouds, const KnnJob *jobs) {
    if (n_clouds < 1 || !jobs) return GCVO_ERR_INVALID_ARG;
    cudaStream_t s = ctx->stream;
    const int C = n_clouds;
    std::vector<KnnCloud> cl(C);
    // clouds by the shape of their cluster (csort::shape); the last class has none
    constexpr int CLASSES = 9;
    int shape_items[CLASSES], shape_blocks[CLASSES], n_class = 0;
    std::vector<std::vector<int>> ids(CLASSES);
    std::vector<int> large;
    int64_t N = 0, n_large = 0;
    for (int c = 0; c < C; ++c) {
        const KnnJob &j = jobs[c];
        const gcvo_kernel_params &kp = *j.kp;
        if (j.n < kp.knn || j.n > ((int64_t)1 << 28)) return GCVO_ERR_INVALID_ARG;
        KnnCloud &k = cl[c];
        k.xyz = j.xyz;
        k.cov = j.cov;
        k.n = j.n;
        k.off = N;
        k.eig_max = kp.eig_max;
        k.eig_ratio = kp.eig_ratio;
        k.cell0 = kp.eig_max > 0 ? (kp.cutoff > 0 ? kp.cutoff : 3.0) * std::sqrt(2.0 * kp.eig_max) * 0.5 : 0.0;
        k.knn = kp.knn;
        k.pad = 0;
        N += j.n;
        int items, blocks;
        csort::shape(j.n, items, blocks);
        if (!knn_sort_fits(items, blocks)) {
            large.push_back(c);
            n_large = std::max(n_large, j.n);
            continue;
        }
        int q = 0;
        while (q < n_class && (shape_items[q] != items || shape_blocks[q] != blocks)) ++q;
        if (q == n_class) {
            shape_items[q] = items;
            shape_blocks[q] = blocks;
            ++n_class;
        }
        ids[q].push_back(c);
    }

    GCVO_TRY(ctx->knn_meta.ensure(knn_meta_bytes(C), s));
    char *m = static_cast<char *>(ctx->knn_meta.ptr);
    auto *d_cl = reinterpret_cast<KnnCloud *>(m);
    m += al256(C * sizeof(KnnCloud));
    auto *d_grid = reinterpret_cast<KnnGrid *>(m);
    m += al256(C * sizeof(KnnGrid));
    int *d_ids = reinterpret_cast<int *>(m);
    m += al256(C * sizeof(int));
    int *d_box = reinterpret_cast<int *>(m);
    GCVO_TRY(ctx->knn_code.ensure(N * sizeof(unsigned long long), s));
    GCVO_TRY(ctx->knn_pos.ensure(N * sizeof(float4), s));
    GCVO_TRY(ctx->knn_cloud.ensure(N * sizeof(int), s));
    GCVO_TRY(ctx->status_word.ensure(256, s));
    auto *code = ctx->knn_code.as<unsigned long long>();
    auto *pos = ctx->knn_pos.as<float4>();
    int *cloud = ctx->knn_cloud.as<int>();
    unsigned *stw = ctx->status_word.as<unsigned>();
    std::vector<int> flat;
    for (int q = 0; q < n_class; ++q) flat.insert(flat.end(), ids[q].begin(), ids[q].end());
    GCVO_CUDA(cudaMemcpyAsync(d_cl, cl.data(), C * sizeof(KnnCloud), cudaMemcpyHostToDevice, s));
    if (!flat.empty())
        GCVO_CUDA(cudaMemcpyAsync(d_ids, flat.data(), flat.size() * sizeof(int), cudaMemcpyHostToDevice, s));
    GCVO_CUDA(cudaMemsetAsync(stw, 0, sizeof(unsigned), s));

    const int *at = d_ids;
    for (int q = 0; q < n_class; ++q) {
        const int nq = (int)ids[q].size();
        switch (shape_items[q]) {
            case 1: GCVO_TRY(launch_knn_sort<1>(d_cl, at, nq, shape_blocks[q], d_grid, code, pos, cloud, stw, s)); break;
            case 2: GCVO_TRY(launch_knn_sort<2>(d_cl, at, nq, shape_blocks[q], d_grid, code, pos, cloud, stw, s)); break;
            default: GCVO_TRY(launch_knn_sort<4>(d_cl, at, nq, shape_blocks[q], d_grid, code, pos, cloud, stw, s));
        }
        at += nq;
    }
    if (n_large) {
        GCVO_TRY(ctx->sort_keys.ensure(n_large * sizeof(unsigned long long), s));
        GCVO_TRY(ctx->sort_vals.ensure(n_large * sizeof(int), s));
        GCVO_TRY(ctx->sort_tmp.ensure(radix_sort_scratch_bytes(n_large), s));
    }
    for (int c : large) {
        const unsigned blocks = (unsigned)((cl[c].n + 255) / 256);
        auto *keys = ctx->sort_keys.as<unsigned long long>();
        int *vals = ctx->sort_vals.as<int>();
        GCVO_CUDA(cudaMemsetAsync(d_box, 0x7f, KNN_BOX * sizeof(int), s));
        k_knn_box<<<std::min(blocks, (unsigned)std::max(1, ctx->sm_count) * 8), 256, 0, s>>>(d_cl, c, d_box);
        k_knn_codes<<<blocks, 256, 0, s>>>(d_cl, c, d_box, d_grid, keys, vals, stw);
        count_launches(2);
        GCVO_CUDA(cudaGetLastError());
        KnnGrid g;
        GCVO_CUDA(cudaMemcpyAsync(&g, d_grid + c, sizeof(g), cudaMemcpyDeviceToHost, s));
        GCVO_CUDA(cudaStreamSynchronize(s));   // the sort's key width
        GCVO_TRY(radix_sort_pairs(keys, vals, cl[c].n, 3 * g.bits, ctx->sort_tmp.ptr, ctx->sort_tmp.bytes, s));
        k_knn_place<<<blocks, 256, 0, s>>>(d_cl, c, keys, vals, code, pos, cloud);
        count_launches(1);
        GCVO_CUDA(cudaGetLastError());
    }
    k_knn_search<<<(unsigned)((N + KNN_WARPS - 1) / KNN_WARPS), KNN_WARPS * 32, 0, s>>>(d_cl, d_grid, code, pos, cloud, N,
                                                                                     stw);
    k_knn_eig<<<(unsigned)((N + 127) / 128), 128, 0, s>>>(d_cl, cloud, N, stw);
    count_launches(2);
    GCVO_CUDA(cudaGetLastError());
    unsigned hs = 0;
    GCVO_CUDA(cudaMemcpyAsync(&hs, stw, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
    GCVO_CUDA(cudaStreamSynchronize(s));
    return hs & DEV_ERR_NONFINITE ? GCVO_ERR_NONFINITE : GCVO_OK;
}

}  // namespace gcvo
