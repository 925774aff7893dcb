// Learned initial-pose proposal: a point-set network that maps a (source,
// target) pair of clouds to a twist, so that Algorithm 1 can start closer to
// the optimum.  (The paper has no counterpart; it is the learned-proposal
// extension of the registration path.)
//
//   per point p = ((xyz - c) / s, l) with c, s the target's centroid and RMS
//   radius:  h1 = relu(W1 p + b1) (64), h2 = relu(W2 h1 + b2) (128),
//            h3 = W3 h2 + b3 (256);  cloud feature = max over points of h3
//   u = [feat_src, feat_tgt] (512): z1 = relu(H1 u + c1) (256),
//            z2 = relu(H2 z1 + c2) (128), out = H3 z2 + c3 (6)
//   out is the twist (omega, v / s) of S T S^-1 with S the shift by -c.
//
// Weights are BF16 copies of FP32 master weights (Adam); every product
// accumulates in FP32.  The per-point layers 2 and 3 (the dense part: 82 k
// flop per point) run on the tensor cores (tcgen05); the max-pool keeps the
// lowest point index on ties, so the argmax is deterministic.  Backward uses that only each channel's
// argmax point receives gradient from the max-pool.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "common.cuh"
#include "perdevice.cuh"
#include "ptx.cuh"

namespace gcvo {
namespace prop {

// parameter tensors, in the order of the flat parameter vector
enum { W1, B1, W2, B2, W3, B3, H1, C1, H2, C2, H3, C3, NT };
constexpr int ROWS[NT] = {64, 64, 128, 128, 256, 256, 256, 256, 128, 128, 6, 6};
constexpr int COLS[NT] = {4, 1, 64, 1, 128, 1, 512, 1, 256, 1, 128, 1};

struct Layout {
    int off[NT + 1];
    Layout() {
        off[0] = 0;
        for (int k = 0; k < NT; ++k) off[k + 1] = off[k] + ROWS[k] * COLS[k];
    }
    int n() const { return off[NT]; }
};

struct Net {
    const float *p;               // FP32 master (biases are read from here)
    const __nv_bfloat16 *w;       // BF16 copy, same layout
    int off[NT + 1];
};

// ---------------------------------------------------------------------------
// Normalisation: one block per pair.  Points of cloud 2b (source) and 2b+1
// (target) are written as float4 (x', y', z', l).
//
// Centroid and RMS radius are FP64 values; a thread's sums run in pairs of
// floats (TwoSum and exact products by FMA, about 2^-48 relative) and only the
// block's few partial sums in FP64, on one thread each: FP64 on every thread,
// at 2 results per SM and cycle, was most of this kernel (256 pairs of 4096
// points: 67 us, now about 27).
// ---------------------------------------------------------------------------
constexpr int PREP_THREADS = 512;

// (s, e) += v, s + e the sum to about twice float's precision.
__device__ __forceinline__ void acc2(float &s, float &e, float v) {
    const float t = __fadd_rn(s, v), bb = __fsub_rn(t, s);
    e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(v, bb)));
    s = t;
}

// The block's sum of every thread's (h, l) for K values, in FP64 to thread k.
template <int K>
__device__ double prep_block_sum(float (&h)[K], float (&l)[K], float2 (*red)[3]) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float hh = __shfl_xor_sync(0xffffffffu, h[k], o), ll = __shfl_xor_sync(0xffffffffu, l[k], o);
            acc2(h[k], l[k], hh);
            l[k] = __fadd_rn(l[k], ll);
        }
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) red[threadIdx.x >> 5][k] = make_float2(h[k], l[k]);
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x < K)
        for (int q = 0; q < PREP_THREADS / 32; ++q)
            s += (double)red[q][threadIdx.x].x + (double)red[q][threadIdx.x].y;
    return s;
}

// The block's sum of one double per thread, to every thread (only for values
// beyond float's range).
__device__ double prep_block_sum64(double v, double *red) {
    __syncthreads();
    if (threadIdx.x == 0) *red = 0.0;
    __syncthreads();
    atomicAdd(red, v);
    __syncthreads();
    return *red;
}

// log of a rigid transform: rotation vector from the skew part of R (with
// the symmetric part near pi), translation through the inverse V matrix.
__device__ void se3_log(const double T[16], double xi[6]) {
    const double R[9] = {T[0], T[1], T[2], T[4], T[5], T[6], T[8], T[9], T[10]};
    const double cth = fmin(1.0, fmax(-1.0, (R[0] + R[4] + R[8] - 1.0) / 2.0));
    double th = acos(cth);
    double w[3];
    if (th < 1e-6) {
        w[0] = (R[7] - R[5]) / 2;
        w[1] = (R[2] - R[6]) / 2;
        w[2] = (R[3] - R[1]) / 2;
    } else if (M_PI - th < 1e-4) {
        // axis from the diagonal of (R + I) / 2 = n n^T
        const double d[3] = {sqrt(fmax(0.0, (R[0] + 1) / 2)), sqrt(fmax(0.0, (R[4] + 1) / 2)),
                             sqrt(fmax(0.0, (R[8] + 1) / 2))};
        const int k = d[0] >= d[1] && d[0] >= d[2] ? 0 : (d[1] >= d[2] ? 1 : 2);
        double nrm[3];
        for (int j = 0; j < 3; ++j) nrm[j] = j == k ? d[k] : (R[3 * k + j] + R[3 * j + k]) / (4 * d[k]);
        const double s = 1.0 / sqrt(nrm[0] * nrm[0] + nrm[1] * nrm[1] + nrm[2] * nrm[2]);
        for (int j = 0; j < 3; ++j) w[j] = nrm[j] * s * th;
    } else {
        const double f = th / (2 * sin(th));
        w[0] = (R[7] - R[5]) * f;
        w[1] = (R[2] - R[6]) * f;
        w[2] = (R[3] - R[1]) * f;
    }
    // V^-1 t = (I - 1/2 W + (1/th^2)(1 - A / (2B)) W^2) t
    const double th2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
    th = sqrt(th2);
    double D;
    if (th < 1e-4) {
        D = 1.0 / 12 + th2 / 720;
    } else {
        double sn, cn;
        sincos(th, &sn, &cn);
        D = (1 - sn / th / (2 * ((1 - cn) / th2))) / th2;
    }
    // W t = w x t, W^2 t = w (w . t) - th^2 t
    const double t[3] = {T[3], T[7], T[11]};
    const double wt = w[0] * t[0] + w[1] * t[1] + w[2] * t[2];
    const double Wt[3] = {w[1] * t[2] - w[2] * t[1], w[2] * t[0] - w[0] * t[2], w[0] * t[1] - w[1] * t[0]};
    for (int k = 0; k < 3; ++k) {
        xi[k] = w[k];
        xi[3 + k] = t[k] - 0.5 * Wt[k] + D * (w[k] * wt - th2 * t[k]);
    }
}

// T_label, label: with labels (training), the twist of S T S^-1 (S the shift
// by -c), translation / s, of the pair's pose; one thread has it ready while
// the others write the points, and no host waits for c and s.
__global__ void __launch_bounds__(PREP_THREADS)
    k_prep(int n, const float *sx, const float *sf, int sf_stride, const float *tx, const float *tf, int tf_stride,
           float4 *pts, float *cs, const double *T_label, float *label) {
    __shared__ float2 red[PREP_THREADS / 32][3];
    __shared__ double c64[3], r64, wide;
    __shared__ float ch[3], cl[3], is;
    const int b = blockIdx.x;
    const float *t = tx + (size_t)b * 3 * n;
    const float *s = sx + (size_t)b * 3 * n;
    {
        float h[3] = {0.f, 0.f, 0.f}, l[3] = {0.f, 0.f, 0.f};
#pragma unroll 4
        for (int i = threadIdx.x; i < n; i += PREP_THREADS)
#pragma unroll
            for (int a = 0; a < 3; ++a) acc2(h[a], l[a], t[(size_t)a * n + i]);
        const double sum = prep_block_sum<3>(h, l, red);
        if (threadIdx.x < 3) c64[threadIdx.x] = sum / n;
        __syncthreads();
        for (int a = 0; a < 3; ++a)
            if (!isfinite(c64[a])) {
                double v = 0.0;
                for (int i = threadIdx.x; i < n; i += PREP_THREADS) v += t[(size_t)a * n + i];
                v = prep_block_sum64(v, &wide);
                if (threadIdx.x == 0) c64[a] = v / n;
                __syncthreads();
            }
        if (threadIdx.x < 3) {
            ch[threadIdx.x] = (float)c64[threadIdx.x];
            cl[threadIdx.x] = (float)(c64[threadIdx.x] - (double)ch[threadIdx.x]);
        }
        __syncthreads();
    }
    {
        float rh[1] = {0.f}, rl[1] = {0.f};
#pragma unroll 4
        for (int i = threadIdx.x; i < n; i += PREP_THREADS)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                // d + e = t - c, and its square (far from the origin e, with the centroid's tail in it, is
                // not small: 4 mm at 100 km)
                float d = t[(size_t)a * n + i], e = 0.f;
                acc2(d, e, -ch[a]);
                e = __fsub_rn(e, cl[a]);
                const float p = __fmul_rn(d, d);
                acc2(rh[0], rl[0], p);
                rl[0] = __fadd_rn(rl[0], __fmaf_rn(d, d, -p) + e * (2.f * d + e));
            }
        const double sum = prep_block_sum<1>(rh, rl, red);
        if (threadIdx.x == 0) r64 = sum;
        __syncthreads();
        if (!isfinite(r64)) {
            double v = 0.0;
            for (int i = threadIdx.x; i < n; i += PREP_THREADS)
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const double d = t[(size_t)a * n + i] - c64[a];
                    v += d * d;
                }
            v = prep_block_sum64(v, &wide);
            if (threadIdx.x == 0) r64 = v;
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            r64 = sqrt(r64 / n) + 1e-6;
            is = (float)(1.0 / r64);
        }
        __syncthreads();
    }
    const double sc = r64;
    if (threadIdx.x == PREP_THREADS - 1) {
        const float sf32 = (float)sc;
        cs[4 * b] = ch[0];
        cs[4 * b + 1] = ch[1];
        cs[4 * b + 2] = ch[2];
        cs[4 * b + 3] = sf32;
        if (T_label) {
            double Tc[16], xi[6];
            for (int k = 0; k < 16; ++k) Tc[k] = T_label[16 * (size_t)b + k];
            const double q[3] = {ch[0], ch[1], ch[2]};
            for (int r = 0; r < 3; ++r)
                Tc[4 * r + 3] += Tc[4 * r] * q[0] + Tc[4 * r + 1] * q[1] + Tc[4 * r + 2] * q[2] - q[r];
            se3_log(Tc, xi);
            for (int k = 0; k < 6; ++k) label[6 * (size_t)b + k] = (float)(k < 3 ? xi[k] : xi[k] / sf32);
        }
    }
#pragma unroll 2
    for (int i = threadIdx.x; i < n; i += PREP_THREADS) {
        pts[(size_t)(2 * b) * n + i] =
            make_float4((s[i] - ch[0]) * is, (s[(size_t)n + i] - ch[1]) * is, (s[2 * (size_t)n + i] - ch[2]) * is,
                        sf[(size_t)b * sf_stride + i]);
        pts[(size_t)(2 * b + 1) * n + i] =
            make_float4((t[i] - ch[0]) * is, (t[(size_t)n + i] - ch[1]) * is, (t[2 * (size_t)n + i] - ch[2]) * is,
                        tf[(size_t)b * tf_stride + i]);
    }
}

// ---------------------------------------------------------------------------
// Per-point MLP and max-pool on the tensor cores.
//
// A tile is 128 points of one cloud; a block (one per SM) walks a contiguous
// range of the batch's tiles.  Layer 1 (4 -> 64) is FP32; layer 2 is one
// 128 x 128 x 64 product (points x channels), layer 3 two 128 x 128 x 128
// products with the operands the other way round (128 channels x points), so
// that a lane of tensor memory holds one channel's value at every point and
// the max-pool needs no exchange between lanes.  Per tile the tensor cores
// need about 1280 cycles at their BF16 rate and the other pipes about 1100
// issue slots per scheduler, so the roles run side by side:
//   warps 0..7  in two groups, one for the even and one for the odd tiles:
//               layer 1 into shared memory, then layer 2's sums out of tensor
//               memory, bias, relu, BF16, back into shared memory;
//   warps 8..15 in two groups, one for each half of layer 3's channels: the
//               sums out of tensor memory, bias, the running maximum of every
//               channel and its point;
//   warp 16     one thread issues the MMAs.
// Each front group has its own buffers, each half of layer 3 its own sums: the
// next tile's first half runs while this one's second is read.  With one
// group of each kind, 2 warps per scheduler, the roles' dependent chains left
// two thirds of the issue slots empty (290 us; tensor pipe 26% busy).
// The sums have the bits of the mma.sync m16n8k16 chains that ran here before.
// 512 clouds of 4096 points: 1287 us with mma.sync (one block of 4 warps per
// cloud, B fragments from padded shared memory), about 215 us here.
// The maxima of a cloud that several blocks share meet in 64-bit atomics:
// (ordered value, inverted point index), so the lowest index wins a tie.
// ---------------------------------------------------------------------------
constexpr int PT_TILE = 128;
constexpr int PT_THREADS = 17 * 32;
constexpr uint32_t PT_COLS = 512;                 // tensor memory: 2 x 128 (layer 2), 2 x 128 (layer 3)
constexpr int PT_W2 = 0;                          // byte offsets in shared memory
constexpr int PT_W3 = PT_W2 + 128 * 128;          // [half][K block of 64][128 channels][128 bytes]
constexpr int PT_H1 = PT_W3 + 4 * 128 * 128;      // [buffer][128 points][128 bytes]
constexpr int PT_H2 = PT_H1 + 2 * 128 * 128;      // [buffer][K block][128 points][128 bytes]
constexpr int PT_W1 = PT_H2 + 4 * 128 * 128;      // [32 output pairs][12]: w0 w0' w1 w1' w2 w2' w3 w3' b b' - -
constexpr int PT_B2 = PT_W1 + 32 * 12 * 4;        // [128]
constexpr int PT_BAR = PT_B2 + 128 * 4;
constexpr int PT_SMEM = PT_BAR + 256;

struct PtBars {
    uint64_t h1_full[2], d2_full[2], h2_full[2], h2_free[2], d3_full[2], d3_free[2], drained;
    uint32_t tmem;
};
static_assert(sizeof(PtBars) <= 256, "the barriers fit");

// A float as an unsigned that orders like it, 0 below every float.
__device__ __forceinline__ unsigned pt_enc(float f) {
    const unsigned u = __float_as_uint(f);
    return u & 0x80000000u ? ~u : u | 0x80000000u;
}
__device__ __forceinline__ float pt_dec(unsigned u) {
    return __uint_as_float(u & 0x80000000u ? u & 0x7fffffffu : ~u);
}

// relu of two floats as packed BF16 (a NaN gives 0).
__device__ __forceinline__ uint32_t relu_bf16(uint64_t v) {
    float lo, hi;
    f2_unpack(v, lo, hi);
    const __nv_bfloat162 p = __hmax2(__floats2bfloat162_rn(lo, hi), __floats2bfloat162_rn(0.f, 0.f));
    return *reinterpret_cast<const uint32_t *>(&p);
}

__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Rows of a 128-row BF16 matrix (row-major in memory, ld values per row) into
// the swizzled layout, 64 columns from col0.
__device__ __forceinline__ void pt_stage(unsigned char *dst, const __nv_bfloat16 *src, int ld, int col0) {
    for (int i = threadIdx.x; i < 128 * 8; i += PT_THREADS) {
        const int r = i >> 3, c = i & 7;
        *reinterpret_cast<uint4 *>(dst + r * 128 + ((c ^ (r & 7)) << 4)) =
            *reinterpret_cast<const uint4 *>(src + (size_t)r * ld + col0 + 8 * c);
    }
}

// One output of layer 1 before its relu, for the point p = (x, y, z, l).  The
// forward pass (two outputs at a time, pt_layer1) and the backward pass sum in
// this order, so that they see the same activations: the last bits decide a
// BF16 rounding, and whether a relu near zero is open.
__device__ __forceinline__ float layer1_sum(float4 w, float bias, float4 p) {
    return __fadd_rn(__fmaf_rn(w.w, p.w, __fmaf_rn(w.z, p.z, __fmaf_rn(w.x, p.x, __fmul_rn(w.y, p.y)))), bias);
}

// Layer 1 of one point into row r of a tile.
__device__ __forceinline__ void pt_layer1(const float *w1, float4 p, unsigned char *h1, int r) {
    const uint64_t x = f2_pack(p.x, p.x), y = f2_pack(p.y, p.y), z = f2_pack(p.z, p.z), l = f2_pack(p.w, p.w);
#pragma unroll 4
    for (int c = 0; c < 8; ++c) {
        uint32_t h[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const ulonglong2 *w = reinterpret_cast<const ulonglong2 *>(w1 + 12 * (4 * c + k));
            const ulonglong2 a = w[0], b = w[1];
            const uint64_t bias = w[2].x;
            uint64_t s = f2_mul(a.y, y);
            s = f2_fma(a.x, x, s);
            s = f2_fma(b.x, z, s);
            s = f2_fma(b.y, l, s);
            h[k] = relu_bf16(f2_add(s, bias));
        }
        *reinterpret_cast<uint4 *>(h1 + r * 128 + ((c ^ (r & 7)) << 4)) = make_uint4(h[0], h[1], h[2], h[3]);
    }
}

__global__ void __launch_bounds__(PT_THREADS, 1)
    k_point_fwd(Net net, int n, int tiles_per_cloud, int64_t n_tiles, const float4 *pts, unsigned long long *top,
                unsigned *status) {
    extern __shared__ unsigned char pt_raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(pt_raw) + 1023) & ~(uintptr_t)1023);
    float *w1 = reinterpret_cast<float *>(sm + PT_W1);
    float *b2 = reinterpret_cast<float *>(sm + PT_B2);
    PtBars &B = *reinterpret_cast<PtBars *>(sm + PT_BAR);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t t0 = n_tiles * blockIdx.x / gridDim.x, t1 = n_tiles * (blockIdx.x + 1) / gridDim.x;
    const int nt = (int)(t1 - t0);

    pt_stage(sm + PT_W2, net.w + net.off[W2], 64, 0);
    for (int q = 0; q < 4; ++q)
        pt_stage(sm + PT_W3 + q * 128 * 128, net.w + net.off[W3] + (size_t)(q >> 1) * 128 * 128, 128, 64 * (q & 1));
    for (int i = tid; i < 64 * 4; i += PT_THREADS)
        w1[12 * (i >> 3) + 2 * (i & 3) + (i >> 2 & 1)] = __bfloat162float(net.w[net.off[W1] + i]);
    if (tid < 64) w1[12 * (tid >> 1) + 8 + (tid & 1)] = net.p[net.off[B1] + tid];
    if (tid < 128) b2[tid] = net.p[net.off[B2] + tid];
    if (warp == 16) tc5_alloc(&B.tmem, PT_COLS);
    if (tid == 0) {
        for (int k = 0; k < 2; ++k) {
            mbar_init(&B.h1_full[k], 128);
            mbar_init(&B.h2_full[k], 128);
            mbar_init(&B.d3_free[k], 128);
            mbar_init(&B.d2_full[k], 1);
            mbar_init(&B.h2_free[k], 1);
            mbar_init(&B.d3_full[k], 1);
        }
        mbar_init(&B.drained, 1);
    }
    fence_proxy_async_smem();
    tc5_fence_before();
    __syncthreads();
    tc5_fence_after();
    const uint32_t tmem = B.tmem;
    bool ok = true;   // every wait of this thread ended in time

    if (warp < 8) {
        const int r = tid & 127, b = warp >> 2;   // row of the tile, group
        auto point = [&](int i) {
            const int64_t t = t0 + i;
            const int64_t cloud = t / tiles_per_cloud;
            const int at = (int)(t - cloud * tiles_per_cloud) * PT_TILE + r;
            return pts[cloud * n + min(at, n - 1)];
        };
        unsigned char *h1 = sm + PT_H1 + b * 128 * 128, *h2 = sm + PT_H2 + b * 2 * 128 * 128;
        const uint32_t d2 = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)b * 128u;
        float4 p = point(min(b, nt - 1));
        for (int i = b; i < nt && ok; i += 2) {
            const unsigned ph = (unsigned)(i >> 1) & 1u;
            // h1's last reader, the group's last layer-2 product, is done: its sums were read below
            pt_layer1(w1, p, h1, r);
            fence_proxy_async_smem();
            mbar_arrive(&B.h1_full[b]);
            if (i + 2 < nt) p = point(i + 2);
            ok = mbar_wait(&B.d2_full[b], ph);
            if (i >= 2) ok = ok && mbar_wait(&B.h2_free[b], ph ^ 1u);
            if (!__all_sync(0xffffffffu, ok)) {
                ok = false;
                break;
            }
            tc5_fence_after();
#pragma unroll 1
            for (int q = 0; q < 4; ++q) {
                uint32_t v[32];
                tc5_ld32(d2 + 32 * q, v);
                tc5_wait_ld(v);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    uint32_t h[4];
#pragma unroll
                    for (int k = 0; k < 4; k += 2) {
                        const ulonglong2 bb = *reinterpret_cast<const ulonglong2 *>(b2 + 32 * q + 8 * c + 2 * k);
                        const int e = 8 * c + 2 * k;
                        h[k] = relu_bf16(f2_add(f2_pack(__uint_as_float(v[e]), __uint_as_float(v[e + 1])), bb.x));
                        h[k + 1] = relu_bf16(f2_add(f2_pack(__uint_as_float(v[e + 2]), __uint_as_float(v[e + 3])), bb.y));
                    }
                    const int cc = 4 * (q & 1) + c;
                    *reinterpret_cast<uint4 *>(h2 + (q >> 1) * 128 * 128 + r * 128 + ((cc ^ (r & 7)) << 4)) =
                        make_uint4(h[0], h[1], h[2], h[3]);
                }
            }
            tc5_fence_before();
            fence_proxy_async_smem();
            mbar_arrive(&B.h2_full[b]);
        }
    } else if (warp == 16) {
        if (lane == 0) {
            const uint32_t idesc = tc5_idesc(128, 128);
            const uint32_t w2a = smem_addr(sm + PT_W2), w3a = smem_addr(sm + PT_W3), h1a = smem_addr(sm + PT_H1),
                           h2a = smem_addr(sm + PT_H2);
            for (int i = -1; i < nt && ok; ++i) {
                if (i + 1 < nt) {   // layer 2 of tile i + 1
                    const int b = (i + 1) & 1;
                    ok = mbar_wait(&B.h1_full[b], (unsigned)((i + 1) >> 1) & 1u);
                    if (!ok) break;
                    tc5_fence_after();
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        tc5_mma(tmem + (uint32_t)b * 128u, tc5_desc(h1a + b * 128 * 128 + 32 * k), tc5_desc(w2a + 32 * k),
                                idesc, k);
                    tc5_commit(&B.d2_full[b]);
                }
                if (i < 0) continue;
                const int b = i & 1;
                ok = mbar_wait(&B.h2_full[b], (unsigned)(i >> 1) & 1u);
                for (int h = 0; h < 2 && ok; ++h) {   // layer 3 of tile i, channels 128 h ..
                    if (i > 0) ok = mbar_wait(&B.d3_free[h], (unsigned)(i - 1) & 1u);
                    if (!ok) break;
                    tc5_fence_after();
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        tc5_mma(tmem + 256u + 128u * (uint32_t)h, tc5_desc(w3a + (2 * h + (k >> 2)) * 128 * 128 + 32 * (k & 3)),
                                tc5_desc(h2a + (2 * b + (k >> 2)) * 128 * 128 + 32 * (k & 3)), idesc, k);
                    tc5_commit(&B.d3_full[h]);
                }
                if (ok) tc5_commit(&B.h2_free[b]);
            }
            // a wait may have run out with products in flight: they end before the tensor memory goes
            tc5_commit(&B.drained);
            ok = mbar_wait(&B.drained, 0) && ok;
        }
        ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
    } else {
        const int h = (warp >> 2) - 2, ch = tid - 256;   // half, channel
        const uint32_t d3 = tmem + ((uint32_t)((warp & 3) * 32) << 16) + 256u + 128u * (uint32_t)h;
        const float bias = net.p[net.off[B3] + ch];
        const uint64_t bb = f2_pack(bias, bias);
        float best = -INFINITY;
        int arg = 0;
        for (int i = 0; i < nt && ok; ++i) {
            const int64_t t = t0 + i, cloud = t / tiles_per_cloud;
            const int base = (int)(t - cloud * tiles_per_cloud) * PT_TILE;
            const int valid = n - base;   // points of the tile, if below 128
            ok = mbar_wait(&B.d3_full[h], (unsigned)i & 1u);
            if (!__all_sync(0xffffffffu, ok)) {
                ok = false;
                break;
            }
            tc5_fence_after();
#pragma unroll 1
            for (int q = 0; q < 4; ++q) {
                uint32_t v[32];
                tc5_ld32(d3 + 32 * q, v);
                tc5_wait_ld(v);
                if (q == 3) {
                    tc5_fence_before();
                    mbar_arrive(&B.d3_free[h]);
                }
                float x[32];
#pragma unroll
                for (int e = 0; e < 32; e += 2)
                    f2_unpack(f2_add(f2_pack(__uint_as_float(v[e]), __uint_as_float(v[e + 1])), bb), x[e], x[e + 1]);
                if (32 * q + 32 > valid)
#pragma unroll
                    for (int e = 0; e < 32; ++e)
                        if (32 * q + e >= valid) x[e] = -INFINITY;
                float m[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) m[e] = max3(x[e], x[e + 4], x[e + 8]);
#pragma unroll
                for (int e = 12; e < 28; e += 8)
#pragma unroll
                    for (int k = 0; k < 4; ++k) m[k] = max3(m[k], x[e + k], x[e + 4 + k]);
#pragma unroll
                for (int k = 0; k < 4; ++k) m[k] = fmaxf(m[k], x[28 + k]);
                const float top4 = max3(fmaxf(m[0], m[1]), m[2], m[3]);
                if (__any_sync(0xffffffffu, top4 > best)) {
                    int at = 31;
#pragma unroll
                    for (int e = 30; e >= 0; --e)
                        if (x[e] == top4) at = e;
                    if (top4 > best) {
                        best = top4;
                        arg = base + 32 * q + at;
                    }
                }
            }
            if (i + 1 == nt || (t + 1) % tiles_per_cloud == 0) {
                // + 0: the zeros compare equal
                const unsigned long long key = (unsigned long long)pt_enc(best + 0.f) << 32 | (0xffffffffu - (unsigned)arg);
                atomicMax(top + cloud * 256 + ch, key);
                best = -INFINITY;
                arg = 0;
            }
        }
    }
    if (!ok && lane == 0) atomicOr(status, DEV_ERR_TIMEOUT);
    tc5_fence_before();
    __syncthreads();
    tc5_fence_after();
    if (warp == 16) tc5_dealloc(tmem, PT_COLS);
}

size_t point_fwd_smem() { return PT_SMEM + 1024; }

// ---------------------------------------------------------------------------
// Head: one block per pair.  z1 = relu(H1 u + c1), z2 = relu(H2 z1 + c2),
// out = H3 z2 + c3; pre-activations y1, y2 kept for backward.  A row of
// weights is read by one warp, 16 (8) BF16 values per lane in 16-byte loads,
// and its sum taken across the lanes (256 pairs: 19 us); one thread per row
// read 4 bytes from each of 32 different lines at a time (89 us).
// ---------------------------------------------------------------------------
constexpr int HEAD_THREADS = 512;

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Dot product of 8 BF16 weights with 8 floats.
__device__ __forceinline__ float dot8(uint4 w, const float *u, float s) {
    const uint32_t q[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        s += __uint_as_float(q[k] << 16) * u[2 * k];
        s += __uint_as_float(q[k] & 0xffff0000u) * u[2 * k + 1];
    }
    return s;
}

__global__ void __launch_bounds__(HEAD_THREADS)
    k_head_fwd(Net net, const unsigned long long *top, float *feat, int *arg, float *y1, float *y2, float *out) {
    const int b = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    constexpr int NW = HEAD_THREADS / 32;
    __shared__ __align__(16) float u[512], z1[256], z2[128];
    {
        // the maxima of the pair's two clouds and their points
        const int i = threadIdx.x;
        const unsigned long long key = top[(size_t)b * 512 + i];
        u[i] = pt_dec((unsigned)(key >> 32));
        feat[(size_t)b * 512 + i] = u[i];
        arg[(size_t)b * 512 + i] = key ? (int)(0xffffffffu - (unsigned)key) : 0;   // 0: no block got to it
    }
    __syncthreads();
    {
        float x[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) x[k] = u[256 * (k >> 3) + 8 * lane + (k & 7)];
#pragma unroll 4
        for (int o = w; o < 256; o += NW) {
            const uint4 *row = reinterpret_cast<const uint4 *>(net.w + net.off[H1] + (size_t)o * 512);
            const float s = warp_sum(dot8(row[32 + lane], x + 8, dot8(row[lane], x, 0.f)));
            if (lane == 0) {
                const float y = s + net.p[net.off[C1] + o];
                y1[(size_t)b * 256 + o] = y;
                z1[o] = fmaxf(y, 0.f);
            }
        }
    }
    __syncthreads();
    {
        float x[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = z1[8 * lane + k];
#pragma unroll 4
        for (int o = w; o < 128; o += NW) {
            const uint4 *row = reinterpret_cast<const uint4 *>(net.w + net.off[H2] + (size_t)o * 256);
            const float s = warp_sum(dot8(row[lane], x, 0.f));
            if (lane == 0) {
                const float y = s + net.p[net.off[C2] + o];
                y2[(size_t)b * 128 + o] = y;
                z2[o] = fmaxf(y, 0.f);
            }
        }
    }
    __syncthreads();
    if (w < 6) {
        const __nv_bfloat16 *row = net.w + net.off[H3] + (size_t)w * 128;
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) s += __bfloat162float(row[lane + 32 * k]) * z2[lane + 32 * k];
        s = warp_sum(s);
        if (lane == 0) out[(size_t)b * 6 + w] = s + net.p[net.off[C3] + w];
    }
}

// Per-pair backward through the head: deltas of every layer, and d feat.  A
// thread sums a column (the loads of a warp are one line), two threads per
// column of H2, each half of its rows.
__global__ void __launch_bounds__(HEAD_THREADS)
    k_head_bwd(Net net, int B, const float *y1, const float *y2, const float *out, const float *label, float *d_out,
               float *d_y1, float *d_y2, float *d_feat, float *loss) {
    const int b = blockIdx.x, i = threadIdx.x;
    __shared__ float dy2[128], dy1[256], part[256], sd_out[6];
    if (i < 6) {
        const float d = out[(size_t)b * 6 + i] - label[(size_t)b * 6 + i];
        sd_out[i] = 2.0f * d / (float)B;
        d_out[(size_t)b * 6 + i] = 2.0f * d / (float)B;
        atomicAdd(loss, d * d / (float)B);
    }
    __syncthreads();
    if (i < 128) {
        float s = 0.f;
        for (int o = 0; o < 6; ++o) s += __bfloat162float(net.w[net.off[H3] + o * 128 + i]) * sd_out[o];
        const float d = y2[(size_t)b * 128 + i] > 0.f ? s : 0.f;
        dy2[i] = d;
        d_y2[(size_t)b * 128 + i] = d;
    }
    __syncthreads();
    {
        const int c = i & 255, o0 = (i >> 8) * 64;
        float s = 0.f;
#pragma unroll 16
        for (int o = o0; o < o0 + 64; ++o) s += __bfloat162float(net.w[net.off[H2] + o * 256 + c]) * dy2[o];
        if (i >= 256) part[c] = s;
        __syncthreads();
        if (i < 256) {
            const float d = y1[(size_t)b * 256 + c] > 0.f ? s + part[c] : 0.f;
            dy1[c] = d;
            d_y1[(size_t)b * 256 + c] = d;
        }
    }
    __syncthreads();
    float s = 0.f;
#pragma unroll 16
    for (int o = 0; o < 256; ++o) s += __bfloat162float(net.w[net.off[H1] + o * 512 + i]) * dy1[o];
    // d feat of cloud 2b (i < 256) or 2b+1
    d_feat[(size_t)b * 512 + i] = s;
}

// Head weight gradients, summed over the batch in order (deterministic):
// dW[o][i] += sum_b delta[b][o] * x[b][i], db[o] += sum_b delta[b][o], for the
// three layers in one launch.  A block takes 32 x 32 weights; the batch passes
// through shared memory 32 pairs at a time, so a delta or an input is read
// once per 32 weights and not once per weight (256 pairs: three launches of
// one thread per weight took 264 us, this one 21).
struct HeadLayer {
    const float *delta, *x;   // B x rows, B x cols
    float *dW, *db;
    int rows, cols, relu;     // relu: x holds pre-activations
};

__global__ void __launch_bounds__(256) k_head_grad(int B, HeadLayer L0, HeadLayer L1, HeadLayer L2) {
    __shared__ float sd[32][33], sx[32][33];
    int t = blockIdx.x;
    HeadLayer L = L0;
    for (int q = 0; q < 2; ++q) {
        const int tiles = (L.rows + 31) / 32 * (L.cols / 32);
        if (t < tiles) break;
        t -= tiles;
        L = q == 0 ? L1 : L2;
    }
    const int o0 = t / (L.cols / 32) * 32, i0 = t % (L.cols / 32) * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // input i0 + tx, outputs o0 + ty + 8 j
    float s[4] = {0.f, 0.f, 0.f, 0.f}, sb[4] = {0.f, 0.f, 0.f, 0.f};
    for (int b0 = 0; b0 < B; b0 += 32) {
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int b = b0 + ty + 8 * k;
            sd[ty + 8 * k][tx] = b < B && o0 + tx < L.rows ? L.delta[(size_t)b * L.rows + o0 + tx] : 0.f;
            float v = b < B ? L.x[(size_t)b * L.cols + i0 + tx] : 0.f;
            sx[ty + 8 * k][tx] = L.relu ? fmaxf(v, 0.f) : v;
        }
        __syncthreads();
#pragma unroll 8
        for (int b = 0; b < 32; ++b) {
            const float v = sx[b][tx];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float d = sd[b][ty + 8 * j];
                s[j] += d * v;
                sb[j] += d;
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int o = o0 + ty + 8 * j;
        if (o < L.rows) {
            L.dW[(size_t)o * L.cols + i0 + tx] += s[j];
            if (i0 == 0 && tx == 0) L.db[o] += sb[j];
        }
    }
}

// ---------------------------------------------------------------------------
// Per-point backward.  For every channel c of a cloud with gradient g_c, its
// argmax point p gets d h3[p][c] = g_c; h1 and h2 of p are recomputed as the
// forward did (BF16 inputs to layers 2 and 3), and dW3[c] += g_c h2, dW2 +=
// d2 h1^T with d2 = g_c W3[c] * relu'(a2), dW1 += d1 p^T with d1 =
// (W2^T d2) * relu'(a1) (and the biases).
//
// The channels are independent up to the sums, so they form matrices: a unit
// of work is BW_CH channels of one cloud, and its three products (a2 =
// H1 W2^T, dW2 = D2^T H1, d1 = D2 W2; 64 x 128 x 64 each) run from shared
// memory with 32, 32 and 16 sums per thread and 16-byte loads.  They stay in
// FP32 like the gradients (12.6 MFLOP per cloud, bound by the FP32 pipe and
// shared-memory loads), and a2 is summed input by input, the bias last, as
// its sign decides relu' and its rounding h2.  A block walks units with its sums of dW2,
// dW1, dB1 and dB2 in registers and adds them to the gradient once at the
// end; dW3's rows go out as they come.
// 512 clouds of 4096 points: about 0.17 ms; one block per cloud walking its
// 256 channels one after another, with a 64- or 128-long dependent sum per
// channel and thread, took 12.9 ms (training step 14.65 -> 1.91 ms).
// ---------------------------------------------------------------------------
constexpr int BW_CH = 64;          // channels of a unit
constexpr int BW_THREADS = 256;
constexpr int BW_LD1 = 64 + 4;     // padded rows: 16-byte loads of consecutive rows fall in different banks
constexpr int BW_LD2 = 128 + 4;
constexpr int BW_SMEM_FLOATS = 128 * BW_LD1 + BW_CH * BW_LD1 + BW_CH * BW_LD2 + BW_CH * 4 + BW_CH + 256 + 64 + 128 +
                               128 + 256 + 64;

__global__ void __launch_bounds__(BW_THREADS, 2) k_point_bwd(Net net, int n, int n_units, const float4 *pts,
                                                             const int *arg, const float *d_feat, float *grad) {
    extern __shared__ __align__(16) float bsm[];
    float *w2 = bsm;                       // [128][BW_LD1]
    float *h1 = w2 + 128 * BW_LD1;         // [BW_CH][BW_LD1]
    float *d2 = h1 + BW_CH * BW_LD1;       // [BW_CH][BW_LD2]
    float *pv = d2 + BW_CH * BW_LD2;       // [BW_CH][4]
    float *gs = pv + BW_CH * 4;            // [BW_CH]
    float *w1 = gs + BW_CH;                // [64][4]
    float *b1 = w1 + 256, *b2 = b1 + 64;
    float *sB2 = b2 + 128, *sW1 = sB2 + 128, *sB1 = sW1 + 256;
    const int tid = threadIdx.x;
    for (int i = tid; i < 128 * 64; i += BW_THREADS) w2[(i >> 6) * BW_LD1 + (i & 63)] = __bfloat162float(net.w[net.off[W2] + i]);
    for (int i = tid; i < 256; i += BW_THREADS) {
        w1[i] = __bfloat162float(net.w[net.off[W1] + i]);
        sW1[i] = 0.f;
    }
    if (tid < 128) {
        b2[tid] = net.p[net.off[B2] + tid];
        sB2[tid] = 0.f;
    }
    if (tid < 64) {
        b1[tid] = net.p[net.off[B1] + tid];
        sB1[tid] = 0.f;
    }
    // a2: channels 8 (tid / 32) .. + 7, outputs tid % 32 + 32 j
    const int c8 = (tid >> 5) * 8, ol = tid & 31;
    // dW2: outputs 8 (tid / 16) .. + 7, inputs 4 (tid % 16) .. + 3
    // d1: channels 4 (tid / 16) .. + 3, inputs 4 (tid % 16) .. + 3
    const int i4 = (tid & 15) * 4, o8 = (tid >> 4) * 8, c4 = (tid >> 4) * 4;
    float aW2[8][4], aW1[4][4], aB1[4], aB2[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        aB1[j] = aB2[j] = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) aW2[k][j] = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) aW1[j][k] = 0.f;
    }
    for (int u = blockIdx.x; u < n_units; u += gridDim.x) {
        const int cloud = u / (256 / BW_CH), ch0 = (u % (256 / BW_CH)) * BW_CH;
        __syncthreads();   // the last unit's reads (and the weights above)
        if (tid < BW_CH) {
            const size_t e = (size_t)cloud * 256 + ch0 + tid;
            const float g = d_feat[e];
            gs[tid] = g;
            // a channel without a gradient adds nothing; a cloud of NaN has no argmax
            const float4 q = g != 0.f ? pts[(size_t)cloud * n + min(max(arg[e], 0), n - 1)] : make_float4(0.f, 0.f, 0.f, 0.f);
            *reinterpret_cast<float4 *>(pv + 4 * tid) = q;
            if (g != 0.f) atomicAdd(grad + net.off[B3] + ch0 + tid, g);
        }
        __syncthreads();
        {
            const float4 q = *reinterpret_cast<const float4 *>(pv + 4 * (tid >> 2));
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const int o = (tid & 3) + 4 * k;
                const float4 w = *reinterpret_cast<const float4 *>(w1 + 4 * o);
                const float s = layer1_sum(w, b1[o], q);
                h1[(tid >> 2) * BW_LD1 + o] = __bfloat162float(__float2bfloat16_rn(fmaxf(s, 0.f)));
            }
        }
        __syncthreads();
        {
            float s[8][4];
#pragma unroll
            for (int k = 0; k < 8; ++k)
#pragma unroll
                for (int j = 0; j < 4; ++j) s[k][j] = 0.f;
#pragma unroll 2
            for (int i = 0; i < 64; i += 4) {
                float4 w[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) w[j] = *reinterpret_cast<const float4 *>(w2 + (ol + 32 * j) * BW_LD1 + i);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float4 h = *reinterpret_cast<const float4 *>(h1 + (c8 + k) * BW_LD1 + i);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        s[k][j] += w[j].x * h.x;
                        s[k][j] += w[j].y * h.y;
                        s[k][j] += w[j].z * h.z;
                        s[k][j] += w[j].w * h.w;
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float g = gs[c8 + k];
                const size_t row = (size_t)(ch0 + c8 + k) * 128;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int o = ol + 32 * j;
                    const float a = s[k][j] + b2[o];
                    float d = 0.f;
                    if (g != 0.f) {
                        const float h2 = __bfloat162float(__float2bfloat16_rn(fmaxf(a, 0.f)));
                        if (h2 != 0.f) atomicAdd(grad + net.off[W3] + row + o, g * h2);
                        if (a > 0.f) d = g * __bfloat162float(net.w[net.off[W3] + row + o]);
                    }
                    aB2[j] += d;
                    d2[(c8 + k) * BW_LD2 + o] = d;
                }
            }
        }
        __syncthreads();
#pragma unroll 4
        for (int c = 0; c < BW_CH; ++c) {
            const float4 h = *reinterpret_cast<const float4 *>(h1 + c * BW_LD1 + i4);
            const float4 da = *reinterpret_cast<const float4 *>(d2 + c * BW_LD2 + o8);
            const float4 db = *reinterpret_cast<const float4 *>(d2 + c * BW_LD2 + o8 + 4);
            const float d[8] = {da.x, da.y, da.z, da.w, db.x, db.y, db.z, db.w};
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                aW2[k][0] += d[k] * h.x;
                aW2[k][1] += d[k] * h.y;
                aW2[k][2] += d[k] * h.z;
                aW2[k][3] += d[k] * h.w;
            }
        }
        {
            float s[4][4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int j = 0; j < 4; ++j) s[k][j] = 0.f;
#pragma unroll 2
            for (int o = 0; o < 128; o += 4) {
                float4 w[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) w[j] = *reinterpret_cast<const float4 *>(w2 + (o + j) * BW_LD1 + i4);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float4 d = *reinterpret_cast<const float4 *>(d2 + (c4 + k) * BW_LD2 + o);
                    const float dd[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        s[k][0] += w[j].x * dd[j];
                        s[k][1] += w[j].y * dd[j];
                        s[k][2] += w[j].z * dd[j];
                        s[k][3] += w[j].w * dd[j];
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float4 q = *reinterpret_cast<const float4 *>(pv + 4 * (c4 + k));
                const float4 h = *reinterpret_cast<const float4 *>(h1 + (c4 + k) * BW_LD1 + i4);
                const float hh[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float d1 = hh[j] > 0.f ? s[k][j] : 0.f;
                    aB1[j] += d1;
                    aW1[j][0] += d1 * q.x;
                    aW1[j][1] += d1 * q.y;
                    aW1[j][2] += d1 * q.z;
                    aW1[j][3] += d1 * q.w;
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
        for (int j = 0; j < 4; ++j) atomicAdd(grad + net.off[W2] + (o8 + k) * 64 + i4 + j, aW2[k][j]);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        atomicAdd(sB2 + ol + 32 * j, aB2[j]);
        atomicAdd(sB1 + i4 + j, aB1[j]);
#pragma unroll
        for (int k = 0; k < 4; ++k) atomicAdd(sW1 + (i4 + j) * 4 + k, aW1[j][k]);
    }
    __syncthreads();
    if (tid < 128) atomicAdd(grad + net.off[B2] + tid, sB2[tid]);
    for (int i = tid; i < 256; i += BW_THREADS) atomicAdd(grad + net.off[W1] + i, sW1[i]);
    if (tid < 64) atomicAdd(grad + net.off[B1] + tid, sB1[tid]);
}

// Adam (Kingma & Ba) on the FP32 master weights; refreshes the BF16 copy.
// A forward pass that ran out of time (status) leaves the parameters alone.
__global__ void k_adam(int n, float *p, const float *g, float *m, float *v, __nv_bfloat16 *w, float lr, float b1,
                       float b2, float eps, float bc1, float bc2, const unsigned *status) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || *status) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
    p[i] = pi;
    w[i] = __float2bfloat16_rn(pi);
}

__global__ void k_to_bf16(int n, const float *p, __nv_bfloat16 *w) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) w[i] = __float2bfloat16_rn(p[i]);
}

}  // namespace prop
}  // namespace gcvo

// ---------------------------------------------------------------------------
// SE(3) exponential of a proposed twist (host, double).
// ---------------------------------------------------------------------------
namespace {

void se3_exp(const double xi[6], double T[16]) {
    const double *w = xi, *v = xi + 3;
    double th2 = w[0] * w[0] + w[1] * w[1] + w[2] * w[2], th = std::sqrt(th2);
    double A, B, C;
    if (th < 1e-4) {
        A = 1 - th2 / 6 + th2 * th2 / 120;
        B = 0.5 - th2 / 24 + th2 * th2 / 720;
        C = 1.0 / 6 - th2 / 120 + th2 * th2 / 5040;
    } else {
        A = std::sin(th) / th;
        B = (1 - std::cos(th)) / th2;
        C = (th - std::sin(th)) / (th2 * th);
    }
    double W[9] = {0, -w[2], w[1], w[2], 0, -w[0], -w[1], w[0], 0}, W2[9];
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) W2[3 * r + c] = W[3 * r] * W[c] + W[3 * r + 1] * W[3 + c] + W[3 * r + 2] * W[6 + c];
    for (int r = 0; r < 3; ++r) {
        double tr = 0;
        for (int c = 0; c < 3; ++c) {
            double I = r == c ? 1.0 : 0.0;
            T[4 * r + c] = I + A * W[3 * r + c] + B * W2[3 * r + c];
            tr += (I + B * W[3 * r + c] + C * W2[3 * r + c]) * v[c];
        }
        T[4 * r + 3] = tr;
    }
    T[12] = T[13] = T[14] = 0;
    T[15] = 1;
}

}  // namespace

using namespace gcvo;

struct gcvo_proposal {
    int device = 0;
    prop::Layout L;
    DevBuf p, g, m, v, w;                // master, grad, Adam moments, BF16 copy
    DevBuf pts, cs, top, feat, arg, y1, y2, out, label, pose, d_out, d_y1, d_y2, d_feat, loss;
    int step = 0;
    int cap_pairs = 0, cap_points = 0;
};

namespace {

prop::Net net_of(gcvo_proposal *P) {
    prop::Net n;
    n.p = P->p.as<float>();
    n.w = P->w.as<__nv_bfloat16>();
    for (int k = 0; k <= prop::NT; ++k) n.off[k] = P->L.off[k];
    return n;
}

// The status word of the forward pass (in the loss buffer, which holds 256 bytes).
unsigned *status_of(gcvo_proposal *P) { return P->loss.as<unsigned>() + 1; }

gcvo_status ensure_batch(gcvo_ctx *ctx, gcvo_proposal *P, int B, int n) {
    cudaStream_t s = ctx->stream;
    GCVO_TRY(P->pts.ensure((size_t)2 * B * n * sizeof(float4), s));
    GCVO_TRY(P->cs.ensure((size_t)B * 4 * sizeof(float), s));
    GCVO_TRY(P->top.ensure((size_t)2 * B * 256 * sizeof(unsigned long long), s));
    GCVO_TRY(P->feat.ensure((size_t)2 * B * 256 * sizeof(float), s));
    GCVO_TRY(P->arg.ensure((size_t)2 * B * 256 * sizeof(int), s));
    GCVO_TRY(P->y1.ensure((size_t)B * 256 * sizeof(float), s));
    GCVO_TRY(P->y2.ensure((size_t)B * 128 * sizeof(float), s));
    GCVO_TRY(P->out.ensure((size_t)B * 6 * sizeof(float), s));
    GCVO_TRY(P->label.ensure((size_t)B * 6 * sizeof(float), s));
    GCVO_TRY(P->pose.ensure((size_t)B * 16 * sizeof(double), s));
    GCVO_TRY(P->d_out.ensure((size_t)B * 6 * sizeof(float), s));
    GCVO_TRY(P->d_y1.ensure((size_t)B * 256 * sizeof(float), s));
    GCVO_TRY(P->d_y2.ensure((size_t)B * 128 * sizeof(float), s));
    GCVO_TRY(P->d_feat.ensure((size_t)2 * B * 256 * sizeof(float), s));
    GCVO_TRY(P->loss.ensure(256, s));
    return GCVO_OK;
}

// Normalisation and the forward pass of a batch; leaves out, feat, arg, y1,
// y2 on the device.
// With T_label (host, B x 16) the labels' twists too.
gcvo_status forward_batch(gcvo_ctx *ctx, gcvo_proposal *P, int B, int n, const float *sx, const float *sf, int sfs,
                          const float *tx, const float *tf, int tfs, const double *T_label) {
    cudaStream_t s = ctx->stream;
    GCVO_TRY(ensure_batch(ctx, P, B, n));
    const double *d_label = nullptr;
    if (T_label) {
        d_label = P->pose.as<double>();
        GCVO_CUDA(cudaMemcpyAsync(P->pose.ptr, T_label, (size_t)B * 16 * sizeof(double), cudaMemcpyHostToDevice, s));
    }
    prop::k_prep<<<B, prop::PREP_THREADS, 0, s>>>(n, sx, sf, sfs, tx, tf, tfs, P->pts.as<float4>(), P->cs.as<float>(),
                                                 d_label, P->label.as<float>());
    static PerDevice<cudaError_t> attr;
    GCVO_CUDA(attr.get([] {
        return cudaFuncSetAttribute(prop::k_point_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)prop::point_fwd_smem());
    }));
    prop::Net net = net_of(P);
    auto *top = P->top.as<unsigned long long>();
    const int tiles = (n + prop::PT_TILE - 1) / prop::PT_TILE;
    const int64_t n_tiles = (int64_t)2 * B * tiles;
    GCVO_CUDA(cudaMemsetAsync(top, 0, (size_t)2 * B * 256 * sizeof(*top), s));
    GCVO_CUDA(cudaMemsetAsync(P->loss.ptr, 0, 256, s));   // the loss, and the status word behind it
    prop::k_point_fwd<<<(unsigned)std::min<int64_t>(n_tiles, std::max(1, ctx->sm_count)), prop::PT_THREADS,
                        prop::point_fwd_smem(), s>>>(net, n, tiles, n_tiles, P->pts.as<float4>(), top, status_of(P));
    prop::k_head_fwd<<<B, prop::HEAD_THREADS, 0, s>>>(net, top, P->feat.as<float>(), P->arg.as<int>(), P->y1.as<float>(),
                                      P->y2.as<float>(), P->out.as<float>());
    count_launches(3);
    GCVO_CUDA(cudaGetLastError());
    return GCVO_OK;
}

bool valid_batch(int B, int n) { return B >= 1 && B <= 65535 && n >= 1 && n <= (1 << 24); }

}  // namespace

extern "C" {

gcvo_status gcvo_proposal_create(gcvo_ctx *ctx, gcvo_proposal **out) {
    if (!ctx || !out) return GCVO_ERR_INVALID_ARG;
    GCVO_CUDA(use_device(ctx->device));
    gcvo_proposal *P = new (std::nothrow) gcvo_proposal();
    if (!P) return GCVO_ERR_WORKSPACE;
    P->device = ctx->device;
    const size_t n = P->L.n();
    cudaStream_t s = ctx->stream;
    gcvo_status st = GCVO_OK;
    for (DevBuf *b : {&P->p, &P->g, &P->m, &P->v})
        if (st == GCVO_OK) st = b->ensure(n * sizeof(float), s);
    if (st == GCVO_OK) st = P->w.ensure(n * sizeof(__nv_bfloat16), s);
    if (st == GCVO_OK) {
        for (DevBuf *b : {&P->p, &P->g, &P->m, &P->v, &P->w})
            if (cudaMemsetAsync(b->ptr, 0, b->bytes, s) != cudaSuccess) st = GCVO_ERR_CUDA;
    }
    if (st != GCVO_OK) {
        gcvo_proposal_destroy(P);
        return st;
    }
    *out = P;
    return GCVO_OK;
}

gcvo_status gcvo_proposal_destroy(gcvo_proposal *P) {
    if (!P) return GCVO_ERR_INVALID_ARG;
    cudaSetDevice(P->device);
    for (DevBuf *b : {&P->p, &P->g, &P->m, &P->v, &P->w, &P->pts, &P->cs, &P->top, &P->feat, &P->arg, &P->y1, &P->y2,
                      &P->out, &P->label, &P->pose, &P->d_out, &P->d_y1, &P->d_y2, &P->d_feat, &P->loss})
        b->release();
    delete P;
    return GCVO_OK;
}

int64_t gcvo_proposal_n_params(void) { return prop::Layout().n(); }

gcvo_status gcvo_proposal_set_params(gcvo_ctx *ctx, gcvo_proposal *P, const float *params) {
    if (!ctx || !P || !params) return GCVO_ERR_INVALID_ARG;
    GCVO_CUDA(use_device(ctx->device));
    const int n = P->L.n();
    cudaStream_t s = ctx->stream;
    GCVO_CUDA(cudaMemcpyAsync(P->p.ptr, params, n * sizeof(float), cudaMemcpyDefault, s));
    GCVO_CUDA(cudaMemsetAsync(P->m.ptr, 0, n * sizeof(float), s));
    GCVO_CUDA(cudaMemsetAsync(P->v.ptr, 0, n * sizeof(float), s));
    prop::k_to_bf16<<<(n + 255) / 256, 256, 0, s>>>(n, P->p.as<float>(), P->w.as<__nv_bfloat16>());
    count_launches(1);
    GCVO_CUDA(cudaGetLastError());
    GCVO_CUDA(cudaStreamSynchronize(s));
    P->step = 0;
    return GCVO_OK;
}

gcvo_status gcvo_proposal_get_params(gcvo_ctx *ctx, const gcvo_proposal *P, float *params_out) {
    if (!ctx || !P || !params_out) return GCVO_ERR_INVALID_ARG;
    GCVO_CUDA(use_device(ctx->device));
    GCVO_CUDA(cudaMemcpyAsync(params_out, P->p.ptr, P->L.n() * sizeof(float), cudaMemcpyDefault, ctx->stream));
    GCVO_CUDA(cudaStreamSynchronize(ctx->stream));
    return GCVO_OK;
}

gcvo_status gcvo_proposal_get_state(gcvo_ctx *ctx, const gcvo_proposal *P, float *state_out, int64_t *step_out) {
    if (!ctx || !P || !state_out || !step_out) return GCVO_ERR_INVALID_ARG;
    GCVO_CUDA(use_device(ctx->device));
    const size_t n = (size_t)P->L.n();
    const DevBuf *parts[3] = {&P->p, &P->m, &P->v};
    for (int k = 0; k < 3; ++k)
        GCVO_CUDA(cudaMemcpyAsync(state_out + k * n, parts[k]->ptr, n * sizeof(float), cudaMemcpyDefault,
                                  ctx->stream));
    GCVO_CUDA(cudaStreamSynchronize(ctx->stream));
    *step_out = P->step;
    return GCVO_OK;
}

gcvo_status gcvo_proposal_set_state(gcvo_ctx *ctx, gcvo_proposal *P, const float *state, int64_t step) {
    if (!ctx || !P || !state || step < 0 || step > (int64_t)1 << 30) return GCVO_ERR_INVALID_ARG;
    GCVO_CUDA(use_device(ctx->device));
    const size_t n = (size_t)P->L.n();
    cudaStream_t s = ctx->stream;
    DevBuf *parts[3] = {&P->p, &P->m, &P->v};
    for (int k = 0; k < 3; ++k)
        GCVO_CUDA(cudaMemcpyAsync(parts[k]->ptr, state + k * n, n * sizeof(float), cudaMemcpyDefault, s));
    prop::k_to_bf16<<<(unsigned)((n + 255) / 256), 256, 0, s>>>((int)n, P->p.as<float>(), P->w.as<__nv_bfloat16>());
    count_launches(1);
    GCVO_CUDA(cudaGetLastError());
    GCVO_CUDA(cudaStreamSynchronize(s));
    P->step = (int)step;
    return GCVO_OK;
}

gcvo_status gcvo_proposal_infer(gcvo_ctx *ctx, gcvo_proposal *P, int B, int n, const float *src_xyz,
                                const float *src_feat, int src_feat_stride, const float *tgt_xyz,
                                const float *tgt_feat, int tgt_feat_stride, float *twist_out, double *T0_out) {
    if (!ctx || !P || !src_xyz || !src_feat || !tgt_xyz || !tgt_feat || !valid_batch(B, n)) return GCVO_ERR_INVALID_ARG;
    GCVO_CUDA(use_device(ctx->device));
    GCVO_TRY(forward_batch(ctx, P, B, n, src_xyz, src_feat, src_feat_stride, tgt_xyz, tgt_feat, tgt_feat_stride, nullptr));
    std::vector<float> out((size_t)B * 6), cs((size_t)B * 4);
    GCVO_CUDA(cudaMemcpyAsync(out.data(), P->out.ptr, out.size() * 4, cudaMemcpyDeviceToHost, ctx->stream));
    unsigned st = 0;
    GCVO_CUDA(cudaMemcpyAsync(cs.data(), P->cs.ptr, cs.size() * 4, cudaMemcpyDeviceToHost, ctx->stream));
    GCVO_CUDA(cudaMemcpyAsync(&st, status_of(P), sizeof(st), cudaMemcpyDeviceToHost, ctx->stream));
    GCVO_CUDA(cudaStreamSynchronize(ctx->stream));
    if (st & DEV_ERR_TIMEOUT) return GCVO_ERR_TIMEOUT;
    if (twist_out) memcpy(twist_out, out.data(), out.size() * 4);
    if (T0_out) {
        for (int b = 0; b < B; ++b) {
            // xi = (omega, v s) in the centred frame; T = S^-1 exp(xi) S
            double xi[6], Tc[16];
            const double sc = cs[4 * b + 3];
            for (int k = 0; k < 3; ++k) {
                xi[k] = out[6 * b + k];
                xi[3 + k] = out[6 * b + 3 + k] * sc;
            }
            se3_exp(xi, Tc);
            double *T = T0_out + 16 * b;
            memcpy(T, Tc, sizeof(Tc));
            const double c[3] = {cs[4 * b], cs[4 * b + 1], cs[4 * b + 2]};
            for (int r = 0; r < 3; ++r)
                T[4 * r + 3] = Tc[4 * r + 3] + c[r] - (Tc[4 * r] * c[0] + Tc[4 * r + 1] * c[1] + Tc[4 * r + 2] * c[2]);
        }
    }
    return GCVO_OK;
}

gcvo_status gcvo_proposal_train_step(gcvo_ctx *ctx, gcvo_proposal *P, int B, int n, const float *src_xyz,
                                     const float *src_feat, int src_feat_stride, const float *tgt_xyz,
                                     const float *tgt_feat, int tgt_feat_stride, const double *T_label, float lr,
                                     float *loss_out, float *grad_out) {
    if (!ctx || !P || !src_xyz || !src_feat || !tgt_xyz || !tgt_feat || !T_label || !valid_batch(B, n) ||
        !(lr >= 0.f))
        return GCVO_ERR_INVALID_ARG;
    GCVO_CUDA(use_device(ctx->device));
    cudaStream_t s = ctx->stream;
    GCVO_TRY(forward_batch(ctx, P, B, n, src_xyz, src_feat, src_feat_stride, tgt_xyz, tgt_feat, tgt_feat_stride,
                           T_label));
    const int np = P->L.n();
    GCVO_CUDA(cudaMemsetAsync(P->g.ptr, 0, np * sizeof(float), s));
    prop::Net net = net_of(P);
    prop::k_head_bwd<<<B, prop::HEAD_THREADS, 0, s>>>(net, B, P->y1.as<float>(), P->y2.as<float>(), P->out.as<float>(),
                                                     P->label.as<float>(), P->d_out.as<float>(), P->d_y1.as<float>(),
                                                     P->d_y2.as<float>(), P->d_feat.as<float>(), P->loss.as<float>());
    float *g = P->g.as<float>();
    const int *off = P->L.off;
    // dH1 = sum_b dy1 u^T (u = the pair's two features), dH2 = dy2 z1^T, dH3 = dout z2^T
    const prop::HeadLayer l1{P->d_y1.as<float>(), P->feat.as<float>(), g + off[prop::H1], g + off[prop::C1], 256, 512, 0};
    const prop::HeadLayer l2{P->d_y2.as<float>(), P->y1.as<float>(), g + off[prop::H2], g + off[prop::C2], 128, 256, 1};
    const prop::HeadLayer l3{P->d_out.as<float>(), P->y2.as<float>(), g + off[prop::H3], g + off[prop::C3], 6, 128, 1};
    prop::k_head_grad<<<8 * 16 + 4 * 8 + 4, 256, 0, s>>>(B, l1, l2, l3);
    // two blocks fit on an SM; fewer when there are not that many units
    static PerDevice<cudaError_t> bwd_attr;
    GCVO_CUDA(bwd_attr.get([] {
        return cudaFuncSetAttribute(prop::k_point_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    prop::BW_SMEM_FLOATS * (int)sizeof(float));
    }));
    const int units = 2 * B * (256 / prop::BW_CH);
    prop::k_point_bwd<<<std::min(units, 2 * std::max(1, ctx->sm_count)), prop::BW_THREADS,
                        prop::BW_SMEM_FLOATS * sizeof(float), s>>>(net, n, units, P->pts.as<float4>(), P->arg.as<int>(),
                                                                   P->d_feat.as<float>(), g);
    count_launches(3);
    GCVO_CUDA(cudaGetLastError());
    if (lr > 0.f) {
        P->step += 1;
        const float b1 = 0.9f, b2 = 0.999f;
        const float bc1 = 1.f - std::pow(b1, (float)P->step), bc2 = 1.f - std::pow(b2, (float)P->step);
        prop::k_adam<<<(np + 255) / 256, 256, 0, s>>>(np, P->p.as<float>(), g, P->m.as<float>(), P->v.as<float>(),
                                                     P->w.as<__nv_bfloat16>(), lr, b1, b2, 1e-8f, bc1, bc2, status_of(P));
        count_launches(1);
        GCVO_CUDA(cudaGetLastError());
    }
    float L[2] = {0.f, 0.f};   // the loss, the status word
    GCVO_CUDA(cudaMemcpyAsync(L, P->loss.ptr, sizeof(L), cudaMemcpyDeviceToHost, s));
    GCVO_CUDA(cudaStreamSynchronize(s));
    unsigned st;
    memcpy(&st, &L[1], sizeof(st));
    if (st) {
        if (lr > 0.f) P->step -= 1;
        return GCVO_ERR_TIMEOUT;
    }
    if (grad_out) {
        GCVO_CUDA(cudaMemcpyAsync(grad_out, g, np * sizeof(float), cudaMemcpyDeviceToHost, s));
        GCVO_CUDA(cudaStreamSynchronize(s));
    }
    if (loss_out) *loss_out = L[0];
    return GCVO_OK;
}

}  // extern "C"
