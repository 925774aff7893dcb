// The preparation of a single problem's source (an evaluation, a registration
// of one pair) in one launch of one thread-block cluster.
//
// Between the source arrays and the first pair pass lie the Morton codes, a
// sort, the packed records, the problem's state (with the Euclidean radius
// from the covariances' largest eigenvalue), the work items and the source at
// the initial pose.  As separate kernels for a batch (pair.cu, tile.cu) these
// are 15 launches and two host read-backs, which for one cloud of up to
// 65,536 points is nearly all waiting: an evaluation of a LiDAR frame spent
// 70 us of 225 in them beside the sort.  The cluster that sorts the codes
// (csort.cuh) also holds everything the other steps exchange, so they follow
// in the same launch with cluster barriers between, and the pose, the grid and
// the parameters arrive as kernel arguments instead of copies.  One evaluation
// of 400 points: 159 -> 68 us, of a LiDAR frame: 223 -> 117 us.
#include <algorithm>
#include <cstring>

#include "common.cuh"
#include "csort.cuh"
#include "pair.cuh"
#include "srcdev.cuh"

namespace gcvo {
namespace {

static_assert(SRC_ONE_MAX == csort::MAX_N, "a cluster holds the points of a single problem");

struct OneShared {
    int red[csort::WARPS][3];
    int ext[3];          // of the block: largest, smallest eigenvalue (ordered ints), 1 if a value is not finite
    int scan[csort::WARPS];
    int last_head;       // last start of a run of equal voxels in the block, -1: none
    int n_sub;           // sub-tiles that start in the block
    ProbDev prob;        // its split pose constants serve the transform
};

__device__ __forceinline__ int remote_int(const int *p, unsigned rank) {
    int v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(csort::cluster_addr(p, rank)) : "memory");
    return v;
}

// Inclusive scan over the block's threads (maximum or sum); `total` is the
// block's.
template <bool MAX>
__device__ __forceinline__ int one_scan(int v, int *warp_tot, int &total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    auto op = [](int a, int b) { return MAX ? max(a, b) : a + b; };
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v = op(v, u);
    }
    __syncthreads();
    if (lane == 31) warp_tot[w] = v;
    __syncthreads();
    int t = warp_tot[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, t, o);
        if (lane >= o) t = op(t, u);
    }
    total = __shfl_sync(0xffffffffu, t, 31);
    const int before = __shfl_sync(0xffffffffu, t, max(w - 1, 0));
    return w > 0 ? op(v, before) : v;
}

template <int ITEMS>
__global__ void __launch_bounds__(csort::THREADS) k_src_one(const SrcOneArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    csort::Smem<ITEMS> &S = *reinterpret_cast<csort::Smem<ITEMS> *>(smem);
    __shared__ OneShared O;
    constexpr int TILE = csort::Smem<ITEMS>::TILE;
    const unsigned rank = csort::cluster_rank(), nblk = csort::cluster_blocks();
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int n = a.n, first = (int)rank * TILE;
    if (rank == 0 && tid < 64) a.words[tid] = 0u;   // status, work counter, active problems, chunks

    // ---- codes, and the range of the covariances' eigenvalues
    int lmax = 0, lmin = 0x7f7f7f7f, bad = 0;
    const float org[3] = {a.xyz[0], a.xyz[n], a.xyz[2 * (size_t)n]};
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const int l = k * csort::THREADS + tid, i = first + l;
        if (i < n) {
            const float c[3] = {a.xyz[i], a.xyz[(size_t)n + i], a.xyz[2 * (size_t)n + i]};
            if (!isfinite(c[0]) || !isfinite(c[1]) || !isfinite(c[2])) bad = 1;
            if (!a.iso) {
                float s[6];
#pragma unroll
                for (int q = 0; q < 6; ++q) {
                    s[q] = a.cov[(size_t)q * n + i];
                    if (!isfinite(s[q])) bad = 1;
                }
                lmax = max(lmax, src_enc(sym3_max_eig(s[0], s[1], s[2], s[3], s[4], s[5])));
                lmin = min(lmin, src_enc(sym3_min_eig(s[0], s[1], s[2], s[3], s[4], s[5])));
            }
            S.key[0][l] = (unsigned long long)src_code(c, org, a.inv_hf) << csort::IDX_BITS | (unsigned)i;
        }
    }
    lmax = __reduce_max_sync(0xffffffffu, lmax);
    lmin = __reduce_min_sync(0xffffffffu, lmin);
    bad = __any_sync(0xffffffffu, bad);
    if (lane == 0) {
        O.red[w][0] = lmax;
        O.red[w][1] = lmin;
        O.red[w][2] = bad;
    }
    split_pose(a.T, a.grid.origin, &O.prob, tid);
    if (tid == 32) O.prob.sigma2 = (float)a.sigma2;
    __syncthreads();
    if (w == 0) {
        lmax = __reduce_max_sync(0xffffffffu, O.red[lane][0]);
        lmin = __reduce_min_sync(0xffffffffu, O.red[lane][1]);
        bad = __any_sync(0xffffffffu, O.red[lane][2]);
        if (lane == 0) {
            O.ext[0] = lmax;
            O.ext[1] = lmin;
            O.ext[2] = bad;
        }
    }
    csort::cluster_barrier(nblk);

    // ---- the problem's state
    if (rank == 0 && w == 0) {
        lmax = 0;
        lmin = 0x7f7f7f7f;
        bad = 0;
        if (lane < (int)nblk) {
            lmax = remote_int(&O.ext[0], lane);
            lmin = remote_int(&O.ext[1], lane);
            bad = remote_int(&O.ext[2], lane);
        }
        lmax = __reduce_max_sync(0xffffffffu, lmax);
        lmin = __reduce_min_sync(0xffffffffu, lmin);
        bad = __any_sync(0xffffffffu, bad);
        const int *gw = reinterpret_cast<const int *>(&a.grid);
        for (int k = lane; k < (int)(sizeof(GridDev) / sizeof(int)); k += 32) reinterpret_cast<int *>(a.grid_out)[k] = gw[k];
        if (lane < 12) {
            a.prob->T[lane] = a.T[lane];
            if (lane < 9) {
                a.prob->Rh[lane] = O.prob.Rh[lane];
                a.prob->Rl[lane] = O.prob.Rl[lane];
            } else {
                a.prob->ch[lane - 9] = O.prob.ch[lane - 9];
                a.prob->cl[lane - 9] = O.prob.cl[lane - 9];
            }
        }
        if (lane == 0) {
            const float lam = __int_as_float(lmax), lam_low = __int_as_float(lmin >= 0 ? lmin : lmin ^ 0x7fffffff);
            // as prepare() has them for a batch, operation by operation
            const double c2 = a.cutoff * a.cutoff;
            double r2;
            if (a.cutoff == 0) r2 = INFINITY;
            else if (a.iso) r2 = __dmul_rn(__dmul_rn(__dmul_rn(c2, a.iso_ell), a.iso_ell), 1.0 + 1e-5);
            else r2 = __dadd_rn(__dmul_rn(__dmul_rn(c2, __dadd_rn((double)a.grid.lam_max, (double)lam)), 1.0 + 2e-4), 1e-12);
            ProbDev *P = a.prob;
            P->status = bad ? -(int)GCVO_ERR_NONFINITE : 0;
            P->iter = 0;
            P->done = 0;
            P->rho2 = (float)r2;
            P->c2 = a.cutoff == 0 ? INFINITY : (float)c2;
            P->sigma2 = (float)a.sigma2;
            P->iso_inv = a.iso ? (float)(1.0 / (a.iso_ell * a.iso_ell)) : 0.f;
            // pair_needs_lo (capi.cu)
            const double s2 = a.iso ? a.iso_ell * a.iso_ell : (double)a.grid.lam_min + (double)fmaxf(0.0f, lam_low);
            P->lo = a.cutoff <= 0 || !isfinite(r2) || !(s2 > 0.0) ||
                    4.0 * a.cutoff * (a.half_diag + sqrt(r2)) * 5.9604644775390625e-08 / sqrt(s2) > 3e-4;
            P->tails = tail_slack(a.half_diag, r2, c2);
            a.words[SRC_WORD_ACTIVE] = bad ? 0u : 1u;
            if (bad) a.words[0] = DEV_ERR_NONFINITE;
        }
    }

    // ---- sort, packed records, the source at the initial pose
    const int b = csort::sort<ITEMS>(S, n, 30);
#pragma unroll 1
    for (int k = 0; k < ITEMS; ++k) {
        const int l = k * csort::THREADS + tid, i = first + l;
        if (i >= n) break;
        const unsigned long long key = S.key[b][l];
        const size_t o = key & ((1u << csort::IDX_BITS) - 1u), N = (size_t)n;
        float f[7] = {1.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, s[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (a.feat)
#pragma unroll
            for (int q = 0; q < 7; ++q)
                if (q < a.feat_dim) f[q] = a.feat[q * N + o];
        if (!a.iso)
#pragma unroll
            for (int q = 0; q < 6; ++q) s[q] = a.cov[q * N + o];
        const float4 z = make_float4(a.xyz[o], a.xyz[N + o], a.xyz[2 * N + o], f[0]);
        const float4 za = make_float4(s[0], s[1], s[2], s[3]), zb = make_float4(s[4], s[5], f[1], f[2]);
        float4 tp, tl, ta, tb;
        transform_point(&O.prob, z, za, zb, a.iso, tp, tl, ta, tb);
        a.spos[i] = z;
        a.sca[i] = za;
        a.scb[i] = zb;
        a.tpos[i] = tp;
        a.tlo[i] = tl;
        a.tca[i] = ta;
        a.tcb[i] = tb;
        if (a.sfx) {
            const float sg = O.prob.sigma2;
            a.sfx[i] = make_float4(f[3], f[4], f[5], f[6]);
            a.tfx[i] = make_float4(sg * f[3], sg * f[4], sg * f[5], sg * f[6]);
        }
        if (a.keys) a.keys[i] = key >> csort::IDX_BITS;
    }

    // ---- work items: sub-tiles of a.sub points inside one voxel of the level
    // (every a.sub-th point from the start of a run of equal voxels)
    const int shift = csort::IDX_BITS + 3 * a.level;
    unsigned heads = 0;
    int last = -1;
    {
        unsigned long long prev = 0;
        const int l0 = tid * ITEMS;
        if (l0 > 0) {
            prev = S.key[b][l0 - 1];
        } else if (rank > 0) {
            asm volatile("ld.shared::cluster.u64 %0, [%1];"
                         : "=l"(prev)
                         : "r"(csort::cluster_addr(&S.key[b][TILE - 1], rank - 1))
                         : "memory");
        }
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int i = first + l0 + k;
            if (i < n) {
                const unsigned long long key = S.key[b][l0 + k];
                if (i == 0 || key >> shift != prev >> shift) {
                    heads |= 1u << k;
                    last = i;
                }
                prev = key;
            }
        }
    }
    int total;
    const int incl = one_scan<true>(last, O.scan, total);
    int seg = __shfl_up_sync(0xffffffffu, incl, 1);   // last head before this thread's points, in the block
    __syncthreads();
    if (lane == 31) O.scan[w] = incl;
    if (tid == 0) O.last_head = total;
    __syncthreads();
    if (lane == 0) seg = w > 0 ? O.scan[w - 1] : -1;
    csort::cluster_barrier(nblk);
    for (unsigned q = 0; q < rank; ++q) seg = max(seg, remote_int(&O.last_head, q));
    unsigned subs = 0;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        const int i = first + tid * ITEMS + k;
        if (i < n) {
            if (heads >> k & 1u) seg = i;
            if (((i - seg) & (a.sub - 1)) == 0) subs |= 1u << k;
        }
    }
    const int mine = __popc(subs);
    int at = one_scan<false>(mine, O.scan, total) - mine;
    if (tid == 0) O.n_sub = total;
    csort::cluster_barrier(nblk);
    int n_items = 0;
    for (unsigned q = 0; q < nblk; ++q) {
        const int v = remote_int(&O.n_sub, q);
        if (q < rank) at += v;
        n_items += v;
    }
#pragma unroll
    for (int k = 0; k < ITEMS; ++k)
        if (subs >> k & 1u) a.tmp[at++] = first + tid * ITEMS + k;
    csort::cluster_barrier(nblk);   // the first points of all items
    for (int it = (int)rank * csort::THREADS + tid; it < n_items; it += (int)nblk * csort::THREADS) {
        const int f = __ldcg(a.tmp + it), next = it + 1 < n_items ? __ldcg(a.tmp + it + 1) : n;
        a.items[it] = (int)((unsigned)f << 6 | (unsigned)(next - f));
        a.item_prob[it] = 0;
    }
    if (rank == 0 && tid == 0) {
        const int chunks = (n_items + FIN_CHUNK - 1) / FIN_CHUNK;
        *a.n_items = n_items;
        a.prob->w0 = 0;
        a.prob->w1 = n_items;
        a.prob->c0 = 0;
        a.prob->c1 = chunks;
        a.words[SRC_WORD_CHUNKS] = (unsigned)chunks;
    }
}

template <int ITEMS>
bool fits_t(int blocks) {
    static PerDevice<unsigned> sizes;
    return csort::placed(sizes.get([] { return csort::cluster_sizes<ITEMS>(k_src_one<ITEMS>); }), blocks);
}

template <int ITEMS>
gcvo_status launch_t(const SrcOneArgs &a, int blocks, cudaStream_t s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(csort::THREADS);
    cfg.dynamicSmemBytes = sizeof(csort::Smem<ITEMS>);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)blocks;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    GCVO_CUDA(cudaLaunchKernelEx(&cfg, k_src_one<ITEMS>, a));
    count_launches(1);
    return GCVO_OK;
}

}  // namespace

bool src_one_fits(int64_t n) {
    int items, blocks;
    csort::shape(n, items, blocks);
    switch (items) {
        case 1: return fits_t<1>(blocks);
        case 2: return fits_t<2>(blocks);
        case 4: return fits_t<4>(blocks);
        default: return false;
    }
}

gcvo_status launch_src_one(const SrcOneArgs &a, cudaStream_t s) {
    int items, blocks;
    csort::shape(a.n, items, blocks);
    switch (items) {
        case 1: return launch_t<1>(a, blocks, s);
        case 2: return launch_t<2>(a, blocks, s);
        case 4: return launch_t<4>(a, blocks, s);
        default: return GCVO_ERR_CAPACITY;
    }
}

}  // namespace gcvo
