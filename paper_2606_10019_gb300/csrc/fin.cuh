// The FP64 side of an iteration: sums of the work items' partials and the
// per-problem step (device code of k_finalize and of the register loop).
#pragma once

#include "common.cuh"
#include "pair.cuh"
#include "srcdev.cuh"

namespace gcvo {

// ---------------------------------------------------------------------------
// FP64 finalize: the per-problem step, on one warp.
//
// A GB300 SM finishes 2 FP64 results per cycle: an FP64 warp instruction keeps
// its scheduler's unit for 64 cycles, whether one lane needs it or 32, and a
// reciprocal costs 341.  What counts is therefore the number of FP64
// instructions of the warp, dependent or not.  One lane working through the
// step alone took about 1300 (43 us per iteration).  Here every lane holds one
// entry of the matrices, lanes that have the same kind of sum to do share its
// instructions, branches are replaced by selected operands, and tests use the
// values' bits: about 80 in all.
// ---------------------------------------------------------------------------

// Whether a double is finite, and whether a finite one is above zero, from its bits.
__device__ __forceinline__ bool finite64(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool positive64(double v) {
    return __double2hiint(v) >= 0 && (__double2hiint(v) | __double2loint(v)) != 0;
}

// Entry (r, c) of w^ (w in memory).
__device__ __forceinline__ double hat_at(const double *w, int r, int c) {
    const double v = w[r == c ? 0 : 3 - r - c];
    return r == c ? 0.0 : ((c - r + 3) % 3 == 1 ? -v : v);
}

// m + Gamma_rc, or m - Gamma_rc, for an entry of Gamma (Eq. 12) = [[-1/2 g_w^,
// 0], [-g_v^, 0]]: one FMA.
__device__ __forceinline__ double add_gamma(const double *g, int r, int c, double m, double sign) {
    const int q = r % 3;
    const double co = c > 2 || q == c ? 0.0 : ((c - q + 3) % 3 == 1 ? sign : -sign) * (r < 3 ? 0.5 : 1.0);
    return fma(co, g[(r < 3 ? 0 : 3) + (q == c || c > 2 ? 0 : 3 - q - c)], m);
}

// out = B^T N B for B = [[I, 0], [-o^, I]] (6 x 6, row-major; all in shared
// memory, tmp holds 18): the change from the grid-origin frame to the
// caller's, with p = p_o + o and J = J_o B.  sym: N is symmetric, and the
// result is made so exactly.
__device__ inline void change_frame(const double *N, const double *o, double *tmp, double *out, bool sym, int lane) {
    if (lane < 18) {   // columns 0..2 of N B
        const int r = lane / 3, c = lane % 3, k1 = (c + 1) % 3, k2 = (c + 2) % 3;
        tmp[lane] = fma(N[6 * r + 3 + k2], o[k1], fma(-N[6 * r + 3 + k1], o[k2], N[6 * r + c]));
    }
    __syncwarp();
    if (lane < 18) {   // rows 0..2 of B^T (N B), and the rest as it is
        const int r = lane / 6, c = lane % 6, k1 = (r + 1) % 3, k2 = (r + 2) % 3;
        const double *y = c < 3 ? tmp + c : N + c;
        const int ld = c < 3 ? 3 : 6;
        const double v = fma(o[k1], y[ld * (3 + k2)], fma(-o[k2], y[ld * (3 + k1)], y[ld * r]));
        if (!sym || r <= c) out[6 * r + c] = v;
        if (sym && r < c) out[6 * c + r] = v;
        if (c > 2) out[6 * (3 + r) + c] = N[6 * (3 + r) + c];
        else if (!sym) out[6 * (3 + r) + c] = tmp[3 * (3 + r) + c];
    }
    __syncwarp();
}

// Solves A x = b (A 6 x 6 row-major, b, x: shared memory) by Gauss-Jordan
// elimination with partial pivoting (by the entries' high words), the rows
// staying where they are.  Lane e < 30 holds the entry of row e % 6 in the
// right-hand side (column 6) and columns 5, 4, 3, 2; columns 1 and 0, which
// only the first step has to change, are a second entry of lanes 0..11.  A
// step is a reciprocal, a product and an FMA.  Returns 0, or 1 when a pivot
// is exactly zero (the same in every lane).
__device__ inline int solve6(const double *A, const double *b, double *x, int lane) {
    const unsigned FULL = 0xffffffffu;
    const int r = lane % 6, c = 6 - lane / 6;
    double v = lane < 6 ? b[lane] : lane < 30 ? A[6 * r + c] : 0.0;
    double v2 = lane < 12 ? A[6 * r + (lane < 6 ? 1 : 0)] : 0.0;
    unsigned used = 0;
    int singular = 0, perm[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const int first = k == 0 ? 6 : k == 1 ? 0 : 6 * (6 - k);   // lane of row 0 in column k
        const double pc = k < 2 ? v2 : v;
        const int row = lane - first;
        const bool open = row >= 0 && row < 6 && !(used >> row & 1u);
        const unsigned key = open ? 0x80000000u | ((unsigned)__double2hiint(pc) & 0x7ffffff8u) | (unsigned)row : 0u;
        const int pr = (int)(__reduce_max_sync(FULL, key) & 7u);
        double p = __shfl_sync(FULL, pc, first + pr);
        if (((__double2hiint(p) & 0x7fffffff) | __double2loint(p)) == 0) {
            singular = 1;
            p = 1.0;
        }
        const double inv = 1.0 / p;
        const double f = __shfl_sync(FULL, pc, first + r);
        const double scaled = __shfl_sync(FULL, v, lane - r + pr) * inv;   // of the pivot row, in this column
        v = r == pr ? scaled : fma(-f, scaled, v);
        if (k == 0) {
            const double s1 = __shfl_sync(FULL, v2, pr) * inv;
            v2 = lane >= 6 ? v2 : r == pr ? s1 : fma(-f, s1, v2);
        }
        used |= 1u << pr;
        perm[k] = pr;
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const double s = __shfl_sync(FULL, v, perm[k]);
        if (lane == k) x[k] = s;
    }
    __syncwarp();
    return singular;
}

// 1 / m! for m = 0 .. 23.
static __constant__ double INV_FACT[24] = {1.0,
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
// sin(theta)) / theta^3: sum_k (-x)^k / (2 k + 1 + lane)!, with as many terms
// as leave less than 1e-19 (eleven up to a radian, three below a
// milliradian).  Larger steps take the closed forms.
__device__ inline double exp_coefficient(double x, int lane) {
    const int hi = __double2hiint(x);
    if (hi < 0x3ff00000) {
        const int m = 1 + min(lane, 2), terms = hi < 0x3eb00000 ? 2 : hi < 0x3f500000 ? 4 : 10;
        double s = INV_FACT[2 * terms + m];
        for (int k = terms - 1; k >= 0; --k) s = fma(-x, s, INV_FACT[2 * k + m]);
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
__device__ inline double smallest_pos_root(double d3, double d2, double d1, double d0) {
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

constexpr int FIN_THREADS = 128;   // 4 warps: item g of a chunk goes to warp g % 4

// Shared memory of one block of the finalize.
struct FinShared {
    double red[FIN_THREADS / 32][64];
    long long cred[FIN_THREADS / 32][4];
    double tot[64];
    long long ctot[4];
    double N[36], tmp[18], M[36], D[36], A[36];
    double g[6], xi[6], o[3], T[12], Tn[12], E[18], y[3];
    int last;
};

__device__ __forceinline__ void set_inactive(ProbDev *P, int st, int *n_active) {
    P->status = st;
    atomicSub(n_active, 1);
}

// T <- T exp(xi) with xi and T in S; the log row, the stop test, and the
// transform constants of a problem that stays active.
__device__ inline void apply_step(const FinalizeArgs &a, ProbDev *P, FinShared &S, gcvo_iter_log *lg, int it, int lane) {
    const unsigned FULL = 0xffffffffu;
    const double *w = S.xi, *v = S.xi + 3;
    const double x = fma(w[2], w[2], fma(w[1], w[1], w[0] * w[0]));
    const double co = exp_coefficient(x, lane);
    const double A = __shfl_sync(FULL, co, 0), B = __shfl_sync(FULL, co, 1), C = __shfl_sync(FULL, co, 2);
    // exp's rotation I + A w^ + B w^2 in lanes 0..8, the matrix I + B w^ + C
    // w^2 of its translation in lanes 16..24; w^ w^ = w w^T - x I
    const int i = lane & 15, h = lane >> 4;
    if (i < 9) {
        const int r = i / 3, c = i % 3;
        const double W2 = fma(w[r], w[c], r == c ? -x : 0.0);
        S.E[9 * h + i] = fma(h ? C : B, W2, fma(h ? B : A, hat_at(w, r, c), r == c ? 1.0 : 0.0));
    }
    __syncwarp();
    // R dR in lanes 0..8, the translation V v in lanes 16..18
    if (i < (h ? 3 : 9)) {
        const double *p = h ? S.E + 9 + 3 * i : S.T + 3 * (i / 3), *q = h ? v : S.E + i % 3;
        const int ld = h ? 1 : 3;
        const double s = fma(p[2], q[2 * ld], fma(p[1], q[ld], p[0] * q[0]));
        (h ? S.y : S.Tn)[i] = s;
    }
    __syncwarp();
    if (lane < 3) S.Tn[9 + lane] = fma(S.T[3 * lane + 2], S.y[2], fma(S.T[3 * lane + 1], S.y[1], fma(S.T[3 * lane], S.y[0], S.T[9 + lane])));
    __syncwarp();
    if (lane < 12) P->T[lane] = S.Tn[lane];
    split_pose(S.Tn, S.o, P, lane);
    double l1 = lane < 6 ? fabs(S.xi[lane]) : 0.0;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) l1 += __shfl_xor_sync(FULL, l1, o);
    if (lg && lane < 6) lg->xi[lane] = S.xi[lane];
    if (lane == 0) {
        if (lg) lg->xi_l1 = l1;
        P->iter = it + 1;
        if ((__double2hiint(l1) & 0x7fffffff) > 0x7ff00000 || (__double2hiint(l1) == 0x7ff00000 && __double2loint(l1) != 0))
            set_inactive(P, -(int)GCVO_ERR_NONFINITE, a.n_active);
        else if (l1 < a.eps_tol) set_inactive(P, 1, a.n_active);
        else if (it + 1 >= a.k_max) set_inactive(P, 2, a.n_active);
    }
}

// The per-problem step of one warp from the slot sums S.tot and S.ctot.
__device__ inline void fin_step(const FinalizeArgs &a, int prob, ProbDev *P, FinShared &S, int lane) {
    const unsigned FULL = 0xffffffffu;
    const GridDev *G = a.grids + prob;
    const int it = P->iter;
    gcvo_iter_log *lg = a.logs ? a.logs + (size_t)prob * a.k_max + it : nullptr;
    const double *tot = S.tot;
    if (lane < 12) S.T[lane] = P->T[lane];
    if (lane < 3) S.o[lane] = G->origin[lane];

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
        apply_step(a, P, S, lg, it, lane);
        return;
    }

    // f, g and M (G-CVO-E: Q - M) in the grid-origin frame (p relative to
    // o), moved to the caller's: g = B^T g_o, M = B^T M_o B (change_frame)
    const double f = tot[0];
    for (int e = lane; e < 36; e += 32) {
        const int r = min(e / 6, e % 6), c = max(e / 6, e % 6);
        S.N[e] = tot[7 + r * 6 - r * (r - 1) / 2 + (c - r)];
    }
    __syncwarp();
    if (lane < 6) {   // g_w += o x g_v
        const int k = lane % 3, k1 = (k + 1) % 3, k2 = (k + 2) % 3;
        const double v = tot[1 + lane], m = fma(-S.o[k2], tot[4 + k1], fma(S.o[k1], tot[4 + k2], v));
        S.g[lane] = lane < 3 ? m : v;
    }
    change_frame(S.N, S.o, S.tmp, S.M, true, lane);
    const bool exact = a.mode == FIN_EXACT || a.mode == FIN_EXACT_EVAL;
    if (exact) {
        // D(g) in the caller's frame from the grid-frame sums of the exact
        // pass.  Per source point, with y = Sigma_ij^-1 r summed over its
        // targets, S_y = sum w y, S_B = sum w (y u^T + K) and P = p^
        // (tile.cuh, pair_exact), the pass leaves C = sum_points (-S_y^ P + P
        // S_B) in tot[28..36] and sum_points S_B in tot[37..45], row-major.
        // M holds B^T (Q - M)_o B; the rest is N_o = [[C, S_y^], [S_B, 0]] with
        // S_y summed over all points = -g_v, and D = M - B^T N_o B.
        for (int e = lane; e < 36; e += 32) {
            const int r = e / 6, c = e % 6;
            S.N[e] = c < 3 ? (r < 3 ? tot[28 + 3 * r + c] : tot[37 + 3 * (r - 3) + c]) : r < 3 ? -hat_at(tot + 4, r, c - 3) : 0.0;
        }
        __syncwarp();
        change_frame(S.N, S.o, S.tmp, S.D, false, lane);
        for (int e = lane; e < 36; e += 32) S.D[e] = S.M[e] - S.D[e];
        __syncwarp();
    }
    bool finite = finite64(f) && (lane >= 6 || finite64(S.g[lane]));
    for (int e = lane; e < 36; e += 32) finite = finite && finite64(S.M[e]) && (!exact || finite64(S.D[e]));
    finite = __all_sync(FULL, finite);

    if (lg) {
        if (lane < 6) lg->g[lane] = S.g[lane];
        if (lane < 16) lg->T[lane] = lane < 12 ? S.T[lane % 4 < 3 ? 3 * (lane / 4) + lane % 4 : 9 + lane / 4] : lane == 15 ? 1.0 : 0.0;
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
            e->H[k] = add_gamma(S.g, k / 6, k % 6, exact ? m : -m, 1.0);
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
    if (S.ctot[1] == 0 || !positive64(f)) {
        if (lane == 0) set_inactive(P, -(int)GCVO_ERR_NO_OVERLAP, a.n_active);
        return;
    }
    if (a.mode == FIN_GRAD) {
        // G-CVO-1: the line search runs along xi = g (Eq. 9); in the
        // grid-origin frame that direction has v' = omega x o + v.
        if (lane < 6) {
            const int k = lane % 3, k1 = (k + 1) % 3, k2 = (k + 2) % 3;
            const double d = S.g[lane], m = fma(-S.g[k2], S.o[k1], fma(S.g[k1], S.o[k2], d));
            P->dir[lane] = d;
            P->dir32[lane] = (float)(lane < 3 ? d : m);
        }
        return;
    }
    // G-CVO-2 step (M - Gamma) xi = g, Eq. (13); G-CVO-E: Newton step xi =
    // -H_E^-1 g, H_E = D(g) + Gamma (Eq. 12)
    for (int e = lane; e < 36; e += 32) S.A[e] = exact ? -S.D[e] : S.M[e];
    __syncwarp();
    if (lane < 18) {
        const int r = lane / 3, c = lane % 3;
        S.A[6 * r + c] = add_gamma(S.g, r, c, S.A[6 * r + c], -1.0);
    }
    __syncwarp();
    if (solve6(S.A, S.g, S.xi, lane) != 0) {
        if (lane == 0) set_inactive(P, -(int)GCVO_ERR_SINGULAR, a.n_active);
        return;
    }
    apply_step(a, P, S, lg, it, lane);
}

// The chunk rows: per chunk, per slot, a compensated FP32 sum of the (hi, lo)
// partials over each warp's items (all its loads in flight), the warps
// added in FP64 in a fixed order; the pair counts likewise.  A persistent
// grid walks the chunks; the problem of chunk c is the last one with c0 <= c.
// The block that finishes a problem's last chunk adds its rows in chunk
// order and takes the step.  As two launches, the step on one lane, they
// were 22 + 46 us of the 85 us that an iteration took at 2,000 source points;
// a registration of 22 iterations went from 1989 to 1132 us.
//
// Not inlined, so that the kernel of its own (pair.cu) and the register loop
// (loop.cu) run the same code: their results agree bit for bit.
static __device__ __noinline__ void fin_chunks(const FinalizeArgs &a, FinShared &S) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // the G-CVO-E pass leaves slots 32..45 in a second partial row per item
    // (its slots 46..63 are never written, and their sums never read)
    const int rows = (a.mode == FIN_EXACT || a.mode == FIN_EXACT_EVAL) ? 2 : 1;
    const int nch = *a.n_chunks;
    // the pair pass is done with its work counter: ready for the next one
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.work = 0;
    // with many chunks a block takes `run` consecutive ones and counts those of a
    // problem together: the count is a fence and an atomic's round trip (256
    // problems, 1.6 million points: 160 -> 97 us in sub-tiles of 8, 131 -> 72 in 16)
    const int lg = nch > 4 * (int)gridDim.x ? 2 : 0, run = 1 << lg;
    int counted = 0;   // chunks of this block that their problem's count lacks yet
    for (int i = 0, c; (c = (((i >> lg) * (int)gridDim.x + (int)blockIdx.x) << lg) + (i & (run - 1))) < nch; ++i) {
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
        constexpr int PER = FIN_CHUNK / (FIN_THREADS / 32);   // items of a warp, all in flight
        for (int row = 0; row < rows; ++row) {
            const float *src = (row == 0 ? a.part : a.part2) + (size_t)(i0 + w) * 64 + lane;
            float h[PER], l[PER];
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const bool in = i0 + w + k * (FIN_THREADS / 32) < i1;
                h[k] = in ? src[k * (FIN_THREADS / 32) * 64] : 0.f;
                l[k] = in ? src[k * (FIN_THREADS / 32) * 64 + 32] : 0.f;
            }
            float H = 0.f, Lo = 0.f;
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const float sm = H + h[k];
                const float bp = sm - H;
                const float err = (H - (sm - bp)) + (h[k] - bp);
                H = sm;
                Lo += l[k] + err;
            }
            S.red[w][32 * row + lane] = (double)H + (double)Lo;
        }
        {
            // counts: lanes 0..PER - 1 an item each
            long long c3[3] = {0, 0, 0};
            const int g = i0 + w + lane * (FIN_THREADS / 32);
            if (lane < PER && g < i1)
#pragma unroll
                for (int k = 0; k < 3; ++k) c3[k] = a.counts[(size_t)g * 4 + k];
#pragma unroll
            for (int o = PER / 2; o > 0; o >>= 1)
#pragma unroll
                for (int k = 0; k < 3; ++k) c3[k] += __shfl_xor_sync(0xffffffffu, c3[k], o);
            if (lane < 4) S.cred[w][lane] = lane == 0 ? c3[0] : lane == 1 ? c3[1] : lane == 2 ? c3[2] : 0;
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
            ++counted;
            if (((i + 1) & (run - 1)) != 0 && c + 1 < c1) {
                __syncthreads();   // the shared sums are read
                continue;
            }
            __threadfence();   // the rows before the count of finished chunks
            __syncthreads();
            if (threadIdx.x == 0) {
                S.last = atomicAdd(&P->done, counted) == c1 - c0 - counted;
                if (S.last) P->done = 0;
            }
            counted = 0;
            __syncthreads();
            if (!S.last) continue;
            __threadfence();   // the other chunks' rows after the count
            // warp w takes every fourth row; the warps are added in order
            for (int row = 0; row < rows; ++row) {
                double sm = 0.0;
#pragma unroll 8
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

}  // namespace gcvo
