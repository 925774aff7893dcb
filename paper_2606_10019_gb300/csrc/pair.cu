// The FP64 side of the per-iteration hot path of Algorithm 1, the transform
// of the source points, and the source packing done once per call:
//   k_finalize  -- FP64 sums of the item partials over chunks of FIN_CHUNK
//                  work items of one problem (all SMs, whatever the batch);
//                  the block that adds a problem's last chunk takes its
//                  step: change of frame, connection term (Eq. 12), the
//                  6x6 solve of Eq. (13) (or the G-CVO-E Newton step with
//                  the exact Hessian), the update T <- T exp(xi) and the
//                  split pose constants the transform reads;
//   k_transform -- every source point of an active problem moved into the
//                  target grid's frame at the current pose (Algorithm 1,
//                  T^-1 z): p = R^T (z - t) - o in double-float arithmetic,
//                  stored as a float head and tail, and Sigma' = R^T Sigma R.
// Source packing sorts each source cloud by a Morton code of its own voxels
// and writes one float4 record triple per point in that order.
#include <algorithm>
#include <cstring>

#include "common.cuh"
#include "fin.cuh"
#include "pair.cuh"
#include "ptx.cuh"
#include "srcdev.cuh"

namespace gcvo {
namespace {

__global__ void __launch_bounds__(FIN_THREADS) k_finalize(FinalizeArgs a) {
    __shared__ FinShared S;
    fin_chunks(a, S);
}

// The transform constants of every problem's initial pose, one warp each.
__global__ void __launch_bounds__(32) k_fin_pose(FinalizeArgs a) {
    const int prob = blockIdx.x;
    const GridDev *G = a.grids + prob;
    split_pose(a.probs[prob].T, G->origin, a.probs + prob, threadIdx.x);
}

// ---------------------------------------------------------------------------
// Source grouping.
// ---------------------------------------------------------------------------
__global__ void k_src_keys(SrcArgs a) {
    const int p = blockIdx.y;
    const SrcDesc d = a.desc[p];
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= d.n) return;
    const int64_t gi = d.offset + i;
    float c[3], r[3];
    for (int k = 0; k < 3; ++k) {
        c[k] = d.xyz[k * d.n + i];
        r[k] = d.xyz[k * d.n];
    }
    a.keys[gi] = ((unsigned long long)p << 30) | src_code(c, r, d.inv_hf);
    a.vals[gi] = (int)gi;
    a.prob_of[gi] = p;
    a.local[gi] = (int)i;
    bool bad = false;
    for (int k = 0; k < 3; ++k) bad |= !isfinite(c[k]);
    if (!a.iso && d.cov) {
        float s[6];
        for (int k = 0; k < 6; ++k) {
            s[k] = d.cov[k * d.n + i];
            bad |= !isfinite(s[k]);
        }
        float l = sym3_max_eig(s[0], s[1], s[2], s[3], s[4], s[5]);
        atomicMax(a.lam_enc + p, src_enc(l));
        atomicMin(a.lam_min_enc + p, src_enc(sym3_min_eig(s[0], s[1], s[2], s[3], s[4], s[5])));
    }
    if (bad) atomicOr(a.status_word, DEV_ERR_NONFINITE);
}

// One packed record triple per sorted source point, and its problem.
__global__ void k_src_pack(SrcArgs a, const unsigned long long *keys, int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int src = a.vals[i];
    const SrcDesc d = a.desc[a.prob_of[src]];
    const int64_t li = a.local[src];
    const float x = d.xyz[li], y = d.xyz[d.n + li], z = d.xyz[2 * d.n + li];
    const float f0 = d.feat ? d.feat[li] : 1.f;
    const float f1 = (d.feat && a.feat_dim > 1) ? d.feat[d.n + li] : 0.f;
    const float f2 = (d.feat && a.feat_dim > 2) ? d.feat[2 * d.n + li] : 0.f;
    float s6[6] = {0, 0, 0, 0, 0, 0};
    if (!a.iso && d.cov)
        for (int k = 0; k < 6; ++k) s6[k] = d.cov[k * d.n + li];
    a.spos[i] = make_float4(x, y, z, f0);
    a.sca[i] = make_float4(s6[0], s6[1], s6[2], s6[3]);
    a.scb[i] = make_float4(s6[4], s6[5], f1, f2);
    if (a.sfx) {
        float fx[4] = {0.f, 0.f, 0.f, 0.f};
        for (int q = 3; q < a.feat_dim && q < 7; ++q) fx[q - 3] = d.feat[q * d.n + li];
        a.sfx[i] = make_float4(fx[0], fx[1], fx[2], fx[3]);
    }
    a.pprob[i] = (int)(keys[i] >> 30);
}

__global__ void __launch_bounds__(256) k_transform(TransformArgs a) { transform_points(a, blockIdx.x, gridDim.x); }

}  // namespace

// ---------------------------------------------------------------------------
// Host launchers.
// ---------------------------------------------------------------------------
cudaError_t launch_finalize(const FinalizeArgs &a, cudaStream_t s) {
    if (a.mode == FIN_POSE) k_fin_pose<<<(unsigned)a.n_problems, 32, 0, s>>>(a);
    else k_finalize<<<(unsigned)(a.reduce_blocks > 0 ? a.reduce_blocks : 1024), FIN_THREADS, 0, s>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_src_keys(const SrcArgs &a, int n_problems, int64_t max_n, cudaStream_t s) {
    dim3 grid((unsigned)((max_n + 255) / 256), (unsigned)n_problems);
    k_src_keys<<<grid, 256, 0, s>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_src_pack(const SrcArgs &a, const unsigned long long *keys, int64_t n, cudaStream_t s) {
    k_src_pack<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, keys, n);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_transform(const TransformArgs &a, cudaStream_t s) {
    if (a.n <= 0) return cudaSuccess;
    const int64_t blocks = std::min<int64_t>((a.n + 255) / 256, 1 << 20);
    k_transform<<<(unsigned)blocks, 256, 0, s>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace gcvo
