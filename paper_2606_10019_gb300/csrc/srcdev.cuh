// Device code of the source side shared by the batched kernels (pair.cu) and
// the one-cluster preparation of a single problem (srcone.cu): the Morton code
// of a source point, the split pose constants and the transform.
#pragma once

#include "common.cuh"
#include "pair.cuh"

namespace gcvo {

__device__ __forceinline__ unsigned src_spread3(unsigned v) {
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

// 30-bit Morton code of a point's fine voxel (edge 1 / inv_hf), counted from
// the cloud's first point.
__device__ __forceinline__ unsigned src_code(const float c[3], const float first[3], float inv_hf) {
    unsigned m = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int q = (int)floorf((c[k] - first[k]) * inv_hf) + 512;
        q = min(max(q, 0), 1023);
        m |= src_spread3((unsigned)q) << k;
    }
    return m;
}

__device__ __forceinline__ int src_enc(float f) {
    const int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7fffffff;
}

// The 12 split constants of the transform at the pose T: R as float head and
// tail, and c = R^T t + o (o the grid origin) likewise; lane k < 12 writes the
// k-th to P.
template <class Prob>
__device__ __forceinline__ void split_pose(const double *T, const double *o, Prob *P, int lane) {
    if (lane >= 12) return;
    double v;
    if (lane < 9) {
        v = T[lane];
    } else {
        const int k = lane - 9;
        v = T[k] * T[9] + T[3 + k] * T[10] + T[6 + k] * T[11] + o[k];
    }
    const float h = (float)v, l = (float)(v - (double)h);
    if (lane < 9) {
        P->Rh[lane] = h;
        P->Rl[lane] = l;
    } else {
        P->ch[lane - 9] = h;
        P->cl[lane - 9] = l;
    }
}

// ---------------------------------------------------------------------------
// The transform of Algorithm 1 (T^-1 z) of one point.  p = R^T z - c is formed
// in double-float arithmetic from the float head / tail splits of R and c:
// each head product R_h z is split exactly into a float and its rounding error
// with one FMA (the error-free product of Ogita, Rump and Oishi, "Accurate sum
// and dot product", SIAM J. Sci. Comput. 2005), the products are added with
// Knuth's TwoSum and the rounding errors, the tail products and c's tail are
// summed in a float alongside (their Sum2 / Dot2 scheme), and a final
// FastTwoSum gives p = p_hi + p_lo with an error near 2^-48 |R| |z|.
// Sigma' = R^T Sigma R is formed in float from the head of R.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// z = (x, y, z, l0), za = (Sxx, Sxy, Sxz, Syy), zb = (Syz, Szz, l1, l2).
template <class Prob>
__device__ __forceinline__ void transform_point(const Prob *P, float4 z, float4 za, float4 zb, bool iso, float4 &tpos,
                                                float4 &tlo, float4 &tca, float4 &tcb) {
    const float zz[3] = {z.x, z.y, z.z};
    float hi[3], lo[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float s = 0.f, err = 0.f;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float rh = P->Rh[3 * j + k];
            const float pr = __fmul_rn(rh, zz[j]);
            const float pe = __fmaf_rn(rh, zz[j], -pr);
            float e;
            two_sum(s, pr, s, e);
            err = __fadd_rn(err, __fadd_rn(__fadd_rn(e, pe), __fmul_rn(P->Rl[3 * j + k], zz[j])));
        }
        float e;
        two_sum(s, -P->ch[k], s, e);
        err = __fadd_rn(err, __fsub_rn(e, P->cl[k]));
        hi[k] = __fadd_rn(s, err);
        lo[k] = __fsub_rn(err, __fsub_rn(hi[k], s));
    }
    const float sg = P->sigma2;
    tpos = make_float4(hi[0], hi[1], hi[2], sg * z.w);
    tlo = make_float4(lo[0], lo[1], lo[2], 0.f);
    float q[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (!iso) {
        const float sm[9] = {za.x, za.y, za.z, za.y, za.w, zb.x, za.z, zb.x, zb.y};
        float Rf[9], T1[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) Rf[k] = P->Rh[k];
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int c = 0; c < 3; ++c)
                T1[3 * r + c] = sm[3 * r] * Rf[c] + sm[3 * r + 1] * Rf[3 + c] + sm[3 * r + 2] * Rf[6 + c];
        q[0] = Rf[0] * T1[0] + Rf[3] * T1[3] + Rf[6] * T1[6];
        q[1] = Rf[0] * T1[1] + Rf[3] * T1[4] + Rf[6] * T1[7];
        q[2] = Rf[0] * T1[2] + Rf[3] * T1[5] + Rf[6] * T1[8];
        q[3] = Rf[1] * T1[1] + Rf[4] * T1[4] + Rf[7] * T1[7];
        q[4] = Rf[1] * T1[2] + Rf[4] * T1[5] + Rf[7] * T1[8];
        q[5] = Rf[2] * T1[2] + Rf[5] * T1[5] + Rf[8] * T1[8];
    }
    tca = make_float4(q[0], q[1], q[2], q[3]);
    tcb = make_float4(q[4], q[5], sg * zb.z, sg * zb.w);
}

// The transform for every point of the active problems.
__device__ __forceinline__ void transform_points(const TransformArgs &a, int block, int blocks) {
    const int64_t stride = (int64_t)blocks * blockDim.x;
    for (int64_t i = (int64_t)block * blockDim.x + threadIdx.x; i < a.n; i += stride) {
        const ProbDev *P = a.probs + (a.pprob ? a.pprob[i] : 0);
        if (P->status != 0) continue;   // converged or failed: left as it was
        const float4 za = a.iso ? make_float4(0.f, 0.f, 0.f, 0.f) : a.sca[i];
        float4 tp, tl, ta, tb;
        transform_point(P, a.spos[i], za, a.scb[i], a.iso != 0, tp, tl, ta, tb);
        a.tpos[i] = tp;
        if (a.tlo) a.tlo[i] = tl;
        a.tca[i] = ta;
        a.tcb[i] = tb;
        if (a.tfx) {
            const float4 f = a.sfx[i];
            const float sg = P->sigma2;
            a.tfx[i] = make_float4(sg * f.x, sg * f.y, sg * f.z, sg * f.w);
        }
    }
}

}  // namespace gcvo
