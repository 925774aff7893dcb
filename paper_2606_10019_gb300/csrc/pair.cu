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
#include "pair.cuh"
#include "ptx.cuh"
#include "srcdev.cuh"

namespace gcvo {
namespace {

// ---------------------------------------------------------------------------
// FP64 finalize: the per-problem step, on one warp.
//
// The step is a few hundred FP64 operations with little to share between
// problems, on a GPU that finishes 2 FP64 results per SM and cycle: a warp
// instruction costs the same for one lane as for 32, so what counts is the
// number of FP64 instructions in line.  One lane working through it alone
// took about 1300 of them, 43 us per iteration.  Here the lanes hold the
// entries of the matrices (a 6 x 6 entry, or a column in the solve), which
// leaves about 200; the exponential's coefficients are short series, one
// lane each.
// ---------------------------------------------------------------------------

// Entry (r, c) of w^.
__device__ __forceinline__ double hat_at(const double w[3], int r, int c) {
    const double v = r + c == 1 ? w[2] : r + c == 2 ? w[1] : w[0];
    return r == c ? 0.0 : ((c - r + 3) % 3 == 1 ? -v : v);
}

// Entry (r, c) of Gamma (Eq. 12), [[-1/2 g_w^, 0], [-g_v^, 0]].
__device__ __forceinline__ double gamma_at(const double g[6], int r, int c) {
    if (c > 2) return 0.0;
    return r < 3 ? -0.5 * hat_at(g, r, c) : -hat_at(g + 3, r - 3, c);
}

// out = B^T N B for B = [[I, 0], [-o^, I]] (6 x 6, row-major in shared
// memory; tmp is scratch): the change from the grid-origin frame to the
// caller's, with p = p_o + o and J = J_o B.  sym: N is symmetric, and the
// result is made so exactly.
__device__ void change_frame(const double *N, const double o[3], double *tmp, double *out, bool sym, int lane) {
    for (int e = lane; e < 36; e += 32) {
        const int r = e / 6, c = e % 6;
        double v = N[e];
        if (c < 3)
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if (k != c) v -= N[6 * r + 3 + k] * hat_at(o, k, c);
        tmp[e] = v;
    }
    __syncwarp();
    for (int e = lane; e < 36; e += 32) {
        int r = e / 6, c = e % 6;
        if (sym && r > c) {
            const int t = r;
            r = c;
            c = t;
        }
        double v = tmp[6 * r + c];
        if (r < 3)
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if (k != r) v += hat_at(o, r, k) * tmp[6 * (3 + k) + c];
        out[e] = v;
    }
    __syncwarp();
}

// Solves A x = b (A 6 x 6 row-major, b: shared memory) by Gauss-Jordan
// elimination with partial pivoting: lane j < 6 holds column j, lane 6 the
// right-hand side; x[k] ends in shared memory.  Returns 0, or 1 when a pivot
// is exactly zero (the same in every lane).
__device__ int solve6(const double *A, const double *b, double *x, int lane) {
    const unsigned FULL = 0xffffffffu;
    double col[6];
#pragma unroll
    for (int r = 0; r < 6; ++r) col[r] = lane < 6 ? A[6 * r + lane] : lane == 6 ? b[r] : 0.0;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        // the row of column k's largest entry, by its high word
        int piv = k, top = __double2hiint(col[k]) & 0x7fffffff;
#pragma unroll
        for (int r = k + 1; r < 6; ++r) {
            const int m = __double2hiint(col[r]) & 0x7fffffff;
            if (m > top) {
                top = m;
                piv = r;
            }
        }
        piv = __shfl_sync(FULL, piv, k);
#pragma unroll
        for (int r = k + 1; r < 6; ++r)
            if (r == piv) {
                const double t = col[k];
                col[k] = col[r];
                col[r] = t;
            }
        const double p = __shfl_sync(FULL, col[k], k);
        if (p == 0.0) return 1;
        double f[6];
#pragma unroll
        for (int r = 0; r < 6; ++r) f[r] = __shfl_sync(FULL, col[r], k);
        col[k] *= 1.0 / p;
#pragma unroll
        for (int r = 0; r < 6; ++r)
            if (r != k) col[r] -= f[r] * col[k];
    }
    if (lane == 6)
#pragma unroll
        for (int r = 0; r < 6; ++r) x[r] = col[r];
    __syncwarp();
    return 0;
}

// 1 / m! for m = 0 .. 23.
__constant__ double INV_FACT[24] = {1.0,
                                    1.0,
                                    1.0 / 2,
                                    1.0 / 6,
                                    1.0 / 24,
                                    1.0 / 120,
                                    1.0 / 720,
                                    1.0 / 5040,
                                    1.0 / 40320,
                                    1.0 / 362880,
                                    1.0 / 3628800,
                                    1.0 / 39916800,
                                    1.0 / 479001600,
                                    1.0 / 6227020800.0,
                                    1.0 / 87178291200.0,
                                    1.0 / 1307674368000.0,
                                    1.0 / 20922789888000.0,
                                    1.0 / 355687428096000.0,
                                    1.0 / 6402373705728000.0,
                                    1.0 / 121645100408832000.0,
                                    1.0 / 2432902008176640000.0,
                                    1.0 / 51090942171709440000.0,
                                    1.0 / 1124000727777607680000.0,
                                    1.0 / 25852016738884976640000.0};

// The coefficients of exp at the squared angle x = theta^2: lane 0 gets
// sin(theta) / theta, lane 1 (1 - cos(theta)) / theta^2, lane 2 (theta -
// sin(theta)) / theta^3: sum_k (-x)^k / (2 k + 1 + lane)!.  Up to a radian
// eleven terms leave less than 1e-19; larger steps take the closed forms.
__device__ double exp_coefficient(double x, int lane) {
    if (x <= 1.0) {
        const int m = 1 + min(lane, 2);
        double s = INV_FACT[20 + m];
#pragma unroll
        for (int k = 9; k >= 0; --k) s = INV_FACT[2 * k + m] - x * s;
        return s;
    }
    const double th = sqrt(x);
    double sn, cs;
    sincos(th, &sn, &cs);
    return lane == 0 ? sn / th : lane == 1 ? (1.0 - cs) / x : (th - sn) / (x * th);
}

// Smallest positive real root of the cubic d3 t^3 + d2 t^2 + d1 t + d0
// (G'(t) of Eq. 9), or -1 if none.  Closed forms (trigonometric / Cardano)
// for the cubic, then two Newton polishing steps per root.
__device__ double smallest_pos_root(double d3, double d2, double d1, double d0) {
    double roots[3];
    int nr = 0;
    double sc = fmax(fmax(fabs(d3), fabs(d2)), fmax(fabs(d1), fabs(d0)));
    if (sc == 0.0) return -1.0;
    if (fabs(d3) <= 1e-14 * sc) {
        if (fabs(d2) <= 1e-14 * sc) {
            if (d1 != 0.0) roots[nr++] = -d0 / d1;
        } else {
            double disc = d1 * d1 - 4.0 * d2 * d0;
            if (disc >= 0.0) {
                double sq = sqrt(disc);
                double qq = -0.5 * (d1 + copysign(sq, d1));
                if (qq != 0.0) roots[nr++] = d0 / qq;
                roots[nr++] = qq / d2;
            }
        }
    } else {
        double a = d2 / d3, b = d1 / d3, c = d0 / d3;
        double Q = (a * a - 3.0 * b) / 9.0;
        double Rr = (2.0 * a * a * a - 9.0 * a * b + 27.0 * c) / 54.0;
        double Q3 = Q * Q * Q;
        if (Rr * Rr < Q3) {
            double th = acos(fmin(fmax(Rr / sqrt(Q3), -1.0), 1.0));
            double m = -2.0 * sqrt(Q);
            roots[nr++] = m * cos(th / 3.0) - a / 3.0;
            roots[nr++] = m * cos((th + 2.0 * M_PI) / 3.0) - a / 3.0;
            roots[nr++] = m * cos((th - 2.0 * M_PI) / 3.0) - a / 3.0;
        } else {
            double A = -copysign(cbrt(fabs(Rr) + sqrt(Rr * Rr - Q3)), Rr);
            double B = A != 0.0 ? Q / A : 0.0;
            roots[nr++] = (A + B) - a / 3.0;
        }
    }
    double best = -1.0;
    for (int k = 0; k < nr; ++k) {
        double t = roots[k];
        for (int it = 0; it < 2; ++it) {
            double p = ((d3 * t + d2) * t + d1) * t + d0;
            double dp = (3.0 * d3 * t + 2.0 * d2) * t + d1;
            if (dp != 0.0) t -= p / dp;
        }
        if (t > 0.0 && (best < 0.0 || t < best)) best = t;
    }
    return best;
}

constexpr int FIN_THREADS = 256;   // 8 warps: item g of a chunk goes to warp g % 8

// Shared memory of one block of k_finalize.
struct FinShared {
    double red[FIN_THREADS / 32][64];
    long long cred[FIN_THREADS / 32][4];
    double tot[64];
    long long ctot[4];
    double N[36], tmp[36], M[36], D[36], A[36];
    double g[6], xi[6], T[12], dT[12];
    int last;
};

__device__ __forceinline__ void set_inactive(ProbDev *P, int st, int *n_active) {
    P->status = st;
    atomicSub(n_active, 1);
}

// T <- T exp(xi) with xi and T in S; the log row, the stop test, and the
// transform constants of a problem that stays active.
__device__ void apply_step(const FinalizeArgs &a, ProbDev *P, FinShared &S, const double *o, gcvo_iter_log *lg, int it,
                           int lane) {
    const unsigned FULL = 0xffffffffu;
    const double *w = S.xi, *v = S.xi + 3;
    const double x = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
    const double co = exp_coefficient(x, lane);
    const double A = __shfl_sync(FULL, co, 0), B = __shfl_sync(FULL, co, 1), C = __shfl_sync(FULL, co, 2);
    // w^ w^ = w w^T - x I
    if (lane < 9) {
        const int r = lane / 3, c = lane % 3;
        const double W2 = w[r] * w[c] - (r == c ? x : 0.0);
        S.dT[lane] = (r == c ? 1.0 : 0.0) + A * hat_at(w, r, c) + B * W2;
    } else if (lane < 12) {
        const int r = lane - 9, r1 = (r + 1) % 3, r2 = (r + 2) % 3;
        const double wv = w[0] * v[0] + w[1] * v[1] + w[2] * v[2];
        S.dT[lane] = v[r] + B * (w[r1] * v[r2] - w[r2] * v[r1]) + C * (w[r] * wv - x * v[r]);
    }
    __syncwarp();
    double tn = 0.0;
    if (lane < 9) {
        const int r = lane / 3, c = lane % 3;
        tn = S.T[3 * r] * S.dT[c] + S.T[3 * r + 1] * S.dT[3 + c] + S.T[3 * r + 2] * S.dT[6 + c];
    } else if (lane < 12) {
        const int r = lane - 9;
        tn = S.T[3 * r] * S.dT[9] + S.T[3 * r + 1] * S.dT[10] + S.T[3 * r + 2] * S.dT[11] + S.T[lane];
    }
    __syncwarp();
    if (lane < 12) {
        S.T[lane] = tn;
        P->T[lane] = tn;
    }
    __syncwarp();
    split_pose(S.T, o, P, lane);
    double l1 = 0.0;
#pragma unroll
    for (int k = 0; k < 6; ++k) l1 += fabs(S.xi[k]);
    if (lg && lane < 6) lg->xi[lane] = S.xi[lane];
    if (lane == 0) {
        if (lg) lg->xi_l1 = l1;
        P->iter = it + 1;
        if (!(l1 == l1)) set_inactive(P, -(int)GCVO_ERR_NONFINITE, a.n_active);
        else if (l1 < a.eps_tol) set_inactive(P, 1, a.n_active);
        else if (it + 1 >= a.k_max) set_inactive(P, 2, a.n_active);
    }
}

// The per-problem step of one warp from the slot sums S.tot and S.ctot.
__device__ void fin_step(const FinalizeArgs &a, int prob, ProbDev *P, FinShared &S, int lane) {
    const unsigned FULL = 0xffffffffu;
    const GridDev *G = a.grids + prob;
    const double o[3] = {G->origin[0], G->origin[1], G->origin[2]};
    const int it = P->iter;
    gcvo_iter_log *lg = a.logs ? a.logs + (size_t)prob * a.k_max + it : nullptr;
    const double *tot = S.tot;
    if (lane < 12) S.T[lane] = P->T[lane];
    __syncwarp();

    if (a.mode == FIN_LINESEARCH) {
        // G(t) ~ sum_k c_k t^k along xi = g (Eq. 9).  c_1 = dG/dt(0) = <g, g>
        // exactly; it is taken from the FP64 gradient rather than the FP32
        // pair sums, which cancel towards zero near the optimum.
        if (lane == 0) {
            double c1 = 0.0;
#pragma unroll
            for (int k = 0; k < 6; ++k) c1 += P->dir[k] * P->dir[k];
            const double ts = smallest_pos_root(4.0 * tot[4], 3.0 * tot[3], 2.0 * tot[2], c1);
            const double mu = ts > a.mu0 ? ts : a.mu0;
#pragma unroll
            for (int k = 0; k < 6; ++k) S.xi[k] = mu * P->dir[k];
        }
        __syncwarp();
        apply_step(a, P, S, G->origin, lg, it, lane);
        return;
    }

    // f, g and M (G-CVO-E: Q - M) in the grid-origin frame (p relative to
    // o), moved to the caller's: g = B^T g_o, M = B^T M_o B (change_frame)
    const double f = tot[0];
    for (int e = lane; e < 36; e += 32) {
        const int r = min(e / 6, e % 6), c = max(e / 6, e % 6);
        S.N[e] = tot[7 + r * 6 - r * (r - 1) / 2 + (c - r)];
    }
    if (lane < 6) {
        double v = tot[1 + lane];
        if (lane < 3)
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if (k != lane) v += hat_at(o, lane, k) * tot[4 + k];
        S.g[lane] = v;
    }
    __syncwarp();
    change_frame(S.N, o, S.tmp, S.M, true, lane);
    const bool exact = a.mode == FIN_EXACT || a.mode == FIN_EXACT_EVAL;
    if (exact) {
        // D(g) in the caller's frame from the grid-frame sums of the exact
        // pass.  Per source point, with y = Sigma_ij^-1 r summed over its
        // targets, S_y = sum w y, S_B = sum w (y u^T + K) and P = p^
        // (tile.cu, pair_exact), the pass leaves C = sum_points (-S_y^ P + P
        // S_B) in tot[28..36] and sum_points S_B in tot[37..45], row-major.
        // M holds B^T (Q - M)_o B; the rest is N_o = [[C, S_y^], [S_B, 0]] with
        // S_y summed over all points = -g_v, and D = M - B^T N_o B.
        const double sy[3] = {-tot[4], -tot[5], -tot[6]};
        for (int e = lane; e < 36; e += 32) {
            const int r = e / 6, c = e % 6;
            S.N[e] = c < 3 ? (r < 3 ? tot[28 + 3 * r + c] : tot[37 + 3 * (r - 3) + c]) : r < 3 ? hat_at(sy, r, c - 3) : 0.0;
        }
        __syncwarp();
        change_frame(S.N, o, S.tmp, S.D, false, lane);
        for (int e = lane; e < 36; e += 32) S.D[e] = S.M[e] - S.D[e];
        __syncwarp();
    }
    bool finite = isfinite(f) && (lane >= 6 || isfinite(S.g[lane]));
    for (int e = lane; e < 36; e += 32) finite = finite && isfinite(S.M[e]) && (!exact || isfinite(S.D[e]));
    finite = __all_sync(FULL, finite);

    if (lg) {
        if (lane < 6) lg->g[lane] = S.g[lane];
        if (lane < 16) lg->T[lane] = lane < 12 ? (lane % 4 < 3 ? S.T[3 * (lane / 4) + lane % 4] : S.T[9 + lane / 4]) : lane == 15 ? 1.0 : 0.0;
        if (lane == 0) {
            lg->f = f;
            lg->n_pairs = S.ctot[0];
            lg->n_kept = S.ctot[1];
        }
    }
    if (a.mode == FIN_EVAL || a.mode == FIN_EXACT_EVAL) {
        // H_GN = -M + Gamma (Eq. 12); G-CVO-E: H_E = D(g) + Gamma, M <- D(g)
        EvalOut *e = a.evalout + prob;
        if (lane < 6) e->g[lane] = S.g[lane];
        for (int k = lane; k < 36; k += 32) {
            const double m = exact ? S.D[k] : S.M[k];
            e->M[k] = m;
            e->H[k] = (exact ? m : -m) + gamma_at(S.g, k / 6, k % 6);
        }
        if (lane == 0) {
            e->f = f;
            e->n_pairs = S.ctot[0];
            e->n_kept = S.ctot[1];
            e->n_cand = S.ctot[2];
            e->rho2 = P->rho2;
        }
        return;
    }
    if (!finite) {
        if (lane == 0) set_inactive(P, -(int)GCVO_ERR_NONFINITE, a.n_active);
        return;
    }
    if (S.ctot[1] == 0 || !(f > 0.0)) {
        if (lane == 0) set_inactive(P, -(int)GCVO_ERR_NO_OVERLAP, a.n_active);
        return;
    }
    if (a.mode == FIN_GRAD) {
        // G-CVO-1: the line search runs along xi = g (Eq. 9); in the
        // grid-origin frame that direction has v' = omega x o + v.
        if (lane < 6) {
            P->dir[lane] = S.g[lane];
            double d = S.g[lane];
            if (lane > 2)
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    if (k != lane - 3) d -= hat_at(o, lane - 3, k) * S.g[k];   // omega x o = -o x omega
            P->dir32[lane] = (float)d;
        }
        return;
    }
    // G-CVO-2 step (M - Gamma) xi = g, Eq. (13); G-CVO-E: Newton step xi =
    // -H_E^-1 g, H_E = D(g) + Gamma (Eq. 12)
    for (int e = lane; e < 36; e += 32) {
        const double gm = gamma_at(S.g, e / 6, e % 6);
        S.A[e] = exact ? -(S.D[e] + gm) : S.M[e] - gm;
    }
    __syncwarp();
    if (solve6(S.A, S.g, S.xi, lane) != 0) {
        if (lane == 0) set_inactive(P, -(int)GCVO_ERR_SINGULAR, a.n_active);
        return;
    }
    apply_step(a, P, S, G->origin, lg, it, lane);
}

// The chunk rows: per chunk, per slot, a compensated FP32 sum of the (hi, lo)
// partials over each warp's items (8 loads in flight per warp), the warps
// added in FP64 in a fixed order; the pair counts likewise.  A persistent
// grid walks the chunks; the problem of chunk c is the last one with c0 <= c.
// The block that finishes a problem's last chunk adds its rows in chunk
// order and takes the step.  As two launches, the step on one lane, they
// were 22 + 46 us of the 85 us that an iteration took at 2,000 source points;
// a registration of 22 iterations went from 1989 to 1132 us.
__global__ void __launch_bounds__(FIN_THREADS) k_finalize(FinalizeArgs a) {
    __shared__ FinShared S;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // the G-CVO-E pass leaves slots 32..45 in a second partial row per item
    // (its slots 46..63 are never written, and their sums never read)
    const int rows = (a.mode == FIN_EXACT || a.mode == FIN_EXACT_EVAL) ? 2 : 1;
    const int nch = *a.n_chunks;
    // the pair pass is done with its work counter: ready for the next one
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.work = 0;
    for (int c = blockIdx.x; c < nch; c += gridDim.x) {
        int lo = 0, hi = a.n_problems - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.probs[mid].c0 <= c) lo = mid;
            else hi = mid - 1;
        }
        ProbDev *P = a.probs + lo;
        // the same for the whole block: the status only changes in the step
        // that follows the problem's last chunk
        if (P->status != 0) continue;
        const int c0 = P->c0, c1 = P->c1;
        const int i0 = P->w0 + (c - c0) * FIN_CHUNK, i1 = min(P->w1, i0 + FIN_CHUNK);
        for (int row = 0; row < rows; ++row) {
            const float *src = row == 0 ? a.part : a.part2;
            float H = 0.f, Lo = 0.f;
            long long cacc = 0;
#pragma unroll 8
            for (int g = i0 + w; g < i1; g += FIN_THREADS / 32) {
                const float *p = src + (size_t)g * 64;
                const float h = p[lane], l = p[32 + lane];
                const float sm = H + h;
                const float bp = sm - H;
                const float err = (H - (sm - bp)) + (h - bp);
                H = sm;
                Lo += l + err;
                if (row == 0 && lane < 3) cacc += a.counts[(size_t)g * 4 + lane];
            }
            S.red[w][32 * row + lane] = (double)H + (double)Lo;
            if (row == 0 && lane < 4) S.cred[w][lane] = cacc;
        }
        __syncthreads();
        if (threadIdx.x < 32 * rows) {
            double sm = 0.0;
#pragma unroll
            for (int q = 0; q < FIN_THREADS / 32; ++q) sm += S.red[q][threadIdx.x];
            S.tot[threadIdx.x] = sm;
            if (c1 - c0 > 1) a.chunk[(size_t)c * 64 + threadIdx.x] = sm;
        }
        if (threadIdx.x < 4) {
            long long cs = 0;
#pragma unroll
            for (int q = 0; q < FIN_THREADS / 32; ++q) cs += S.cred[q][threadIdx.x];
            S.ctot[threadIdx.x] = cs;
            if (c1 - c0 > 1) a.chunk_cnt[(size_t)c * 4 + threadIdx.x] = cs;
        }
        if (c1 - c0 > 1) {
            __threadfence();   // the row before the count of finished chunks
            __syncthreads();
            if (threadIdx.x == 0) {
                S.last = atomicAdd(&P->done, 1) == c1 - c0 - 1;
                if (S.last) P->done = 0;
            }
            __syncthreads();
            if (!S.last) continue;
            __threadfence();   // the other chunks' rows after the count
            // warp w takes every eighth row; the warps are added in order
            for (int row = 0; row < rows; ++row) {
                double sm = 0.0;
                for (int q = c0 + w; q < c1; q += FIN_THREADS / 32) sm += __ldcg(a.chunk + (size_t)q * 64 + 32 * row + lane);
                S.red[w][32 * row + lane] = sm;
            }
            if (lane < 4) {
                long long cs = 0;
                for (int q = c0 + w; q < c1; q += FIN_THREADS / 32) cs += __ldcg(a.chunk_cnt + (size_t)q * 4 + lane);
                S.cred[w][lane] = cs;
            }
            __syncthreads();
            if (threadIdx.x < 32 * rows) {
                double sm = 0.0;
#pragma unroll
                for (int q = 0; q < FIN_THREADS / 32; ++q) sm += S.red[q][threadIdx.x];
                S.tot[threadIdx.x] = sm;
            }
            if (threadIdx.x < 4) {
                long long cs = 0;
#pragma unroll
                for (int q = 0; q < FIN_THREADS / 32; ++q) cs += S.cred[q][threadIdx.x];
                S.ctot[threadIdx.x] = cs;
            }
        }
        __syncthreads();
        if (w == 0) fin_step(a, lo, P, S, lane);
        __syncthreads();
    }
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

// The transform of Algorithm 1 (T^-1 z, srcdev.cuh) for every point of an
// active problem.
__global__ void k_transform(TransformArgs a) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += stride) {
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
