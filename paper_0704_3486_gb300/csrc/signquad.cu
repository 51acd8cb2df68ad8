// K3, first column only: beta sgn(H_k) e_1 of the upper Hessenberg H_k
// (Sec. 5.3 step v) from the integral that Roberts' iterates discretise,
//
//   sgn(H) = (1/pi) int_{-inf}^{inf} (H - i t)^{-1} dt,
//
// by a quadrature whose every node is one Hessenberg solve with e_1. An
// iterate S^n of Roberts' iteration (Eq. Roberts) is exactly this integral
// with the 2^n nodes t = tan(pi (j + 1/2) / 2^n); here the nodes follow the
// substitution t = r b sc(v | 1 - r^2) (Hale, Higham and Trefethen, "Computing
// A^alpha, log(A) and related matrix functions by contour integrals", 2008),
// which spreads them evenly over |lambda| in [r b, b], so that 96 pairs +-t
// replace the 2^9 to 2^13 of Roberts' iterate. Cost: 192 solves of k^2/2
// complex multiply-adds, all independent, against ten inversions of k^3 with a
// chain of k pivots each.
//
// Solve (Hyman's method, as in Wilkinson, "The Algebraic Eigenvalue Problem",
// ch. 7): rows k-1 .. 1 of (H - i t) z = e_1 form an upper triangular system
// whose diagonal is the subdiagonal of H, so from z_{k-1} = 1 the recurrence
//   z_{l-1} = - (sum_{q >= l} (H - i t)_{lq} z_q) / h_{l,l-1}
// gives z up to a factor and row 0 gives that factor. Every row is satisfied
// to rounding relative to its own terms, so the solve is backward stable row
// by row; z is rescaled by powers of two where it grows.
//
// Accuracy: the rule f is the midpoint rule of an even periodic analytic
// function, so the nodes p = 1 (mod 3) are a rule f_A of a third of the pairs and
// the others a rule f_B: f = (f_A + 2 f_B)/3. A result is taken on two vectors,
//   d = (f - f_A)(H) e_1   and   r = (f_A f_B)(H) e_1 - e_1,
// where |d| and |r| together are at most the tolerance times |f(H) e_1|. With
// positive weights Re f_A > 0 where Re lambda > 0, and for every eigenvalue with
// sign s
//   |f_A - s| <= |f_A f_B - 1| + |f_B - f_A|,
// because f_A^2 - 1 = (f_A f_B - 1) - f_A (f_B - f_A) and |f_A + s| is at least 1
// and at least |f_A|. So the bound holds component by component: an eigenvalue that
// the window does not reach (f_A = f_B = 0 there, hence r = -1) or that the rule does
// not resolve cannot hide behind the others, however small its part of e_1, and one
// on the imaginary axis has |f_A f_B - 1| + |f_B - f_A| >= 1. Both vectors are of
// first order in the error of f_A; f is then far better. r needs no other solve: f_A f_B has simple
// poles, its residues at the nodes of f_A vanish, and at those of f_B the factor
// f_A(i t_p) is i tan(pi (p + 1/2) / 3) = +-i/sqrt(3) (to e^(-4 pi K n/K'), below
// 1e-16 from 16 pairs on), so
//   (f_A f_B)(H) = (sqrt(3)/2) i sum_{p = 0, 2 (mod 3)} +-w_p [(H - i t_p)^-1 - (H + i t_p)^-1],
// + for p = 0.
// Tolerance 1e-12 where H is of FP64 quality, 1e-8 where complex64 vectors made it
// (its rounding is 1e-7). Right-hand sides above it get a second rule (255 pairs over
// [1e-4 b, b]: spectra up to about 58 degrees off the real axis), then a third (4080
// pairs over the same: up to 88 degrees, and 4e-6 b on the real axis; the Ritz value near
// 0 that an odd k has, mu above 1), at orders above 320 a fourth (16320 pairs, up to 89.5
// degrees: Roberts' iteration runs on one block there, 1.6 s at 400; 4^4, mu = 2, eight
// right-hand sides: 303 ms), and those that fail these too (an eigenvalue closer to 0 or
// to the imaginary axis) Roberts' iteration itself (launch_newton), with its statuses.
// Measured over lattices 4^4 to 8^4, k 40 to 790, mu 0.05 to 0.3: |d| and |r| 5e-16 at the
// first rule, the first column within 5e-16 of Roberts' in the 2-norm. Whole applications,
// with Roberts' iteration (on 4 to 8 SMs per right-hand side, one block above k = 320)
// and with this: 6^4, 2 right-hand sides, k = 340: 1373 -> 547 ms; 8^4 mixed, one
// right-hand side, k = 200: 50.0 -> 23.1 ms; six fields of 4^4 to 8^4 with convergence
// checks up to k = 300, 54 right-hand sides: 921 -> 156 ms (with 48 pairs; see the
// pairs below for what they cost).
#include <algorithm>
#include <cmath>

#include "arnoldi_dev.cuh"
#include "common.cuh"
#include "kernels.h"

namespace ovs {

namespace {

constexpr double kTol64 = 1e-12, kTol32 = 1e-8;
// Pairs, multiples of 3: the third of the first rule reaches the tolerance on spectra
// up to 25 degrees off the real axis. Whole calls with 48 pairs, taken where f and f_A
// agreed to 3e-6 (which bounds nothing), and with these: 4^4 FP64, k = 100: 2.83 and 2.85
// ms; 3x5x7x9 FP64, k = 75, 60 fields: mean 5.08 and 5.08, median 4.48 and 4.57; the six
// fields above 127 and 132.
constexpr int kPairs64 = 96, kPairs32 = 66, kPairs2 = 255, kPairs3 = 4080, kPairs4 = 16320;
constexpr int kLastRule = 320;  // orders above take the fourth rule
constexpr double kWindow1 = 1e-3, kWindow2 = 1e-4;
constexpr int QS = 8;  // columns of H in flight per warp (cp.async stages)

// Node and weight / pi of the pairs, for b = 1: a table, or for more pairs than
// it holds (of which warp p takes p, p + kPairs2, ...) the constants of the rule.
struct QuadNodes {
    int pairs;
    double r, K, Kp, lq;
    double t[kPairs2], w[kPairs2];
};

double agm(double a, double b) {
    for (int i = 0; i < 60; ++i) {
        const double m = 0.5 * (a + b), g = std::sqrt(a * b);
        a = m;
        b = g;
    }
    return a;
}

// Midpoints v_j = (j + 1/2) K'/n of sc(v | 1 - r^2) on (0, K'): t_j = r sc(v_j)
// and w_j = (dt/dv)(v_j) K'/(n pi). The Fourier series of sn at imaginary
// argument converges fast on v <= K'/2; the other half is its mirror image
// t(K' - v) = r / t(v).
__host__ __device__ inline void quad_node(const QuadNodes& q, int j, double& t, double& w) {
    const double pi = 3.14159265358979323846;
    const int at = j < (q.pairs + 1) / 2 ? j : q.pairs - 1 - j;
    const double h = q.Kp / q.pairs, v = (at + 0.5) * h;
    double s = 0.0, d = 0.0;
    for (int i = 0; i < 8; ++i) {  // terms fall by e^(-pi Kp / 2K), 2e-3 at r = 1e-3 and 3e-7 at 1e-6
        const double o = 2 * i + 1, a = o * pi * v / (2 * q.K), c = 1.0 / (1.0 - exp(o * q.lq));
        const double ep = exp(o * q.lq / 2 + a), em = exp(o * q.lq / 2 - a);
        s += c * (ep - em) / 2;
        d += o * c * (ep + em) / 2;
    }
    s *= 2 * pi / q.K;
    d *= pi * pi / (q.K * q.K);
    t = at == j ? s : q.r / s;
    w = d * h / pi * (at == j ? 1.0 : q.r / (s * s));
}

QuadNodes make_nodes(int n, double r) {
    const double pi = 3.14159265358979323846;
    QuadNodes q{};
    q.pairs = n;
    q.r = r;
    q.K = pi / 2 / agm(1.0, std::sqrt(1.0 - r * r));
    q.Kp = pi / 2 / agm(1.0, r);
    q.lq = -pi * q.Kp / q.K;
    for (int j = 0; j < std::min(n, kPairs2); ++j) quad_node(q, j, q.t[j], q.w[j]);
    return q;
}

__device__ __forceinline__ double lane_d(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }

__device__ __forceinline__ void cp16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}

// order of the matrix of right-hand side r; -1 where it takes no part
__device__ __forceinline__ int quad_order(const int* k_used, int n_fixed, const int* due, const int* need, int level,
                                          int r) {
    if (due != nullptr && due[r] == 0) return -1;
    if (level > 1 && need[r] == 0) return -1;
    return n_fixed > 0 ? n_fixed : k_used[r];
}

// Largest column norm of H_r (as the bits of a non-negative double, for
// atomicMax) and the inverse subdiagonal: one warp per column. With Schur
// deflation the columns are those of [T X; 0 H_r].
__global__ void __launch_bounds__(256) k_quad_prep(const double2* __restrict__ H, long long h_rhs, int ldh,
                                                   const int* __restrict__ k_used, int n_fixed,
                                                   const int* __restrict__ due, unsigned long long* __restrict__ bmax,
                                                   double* __restrict__ isub, int kmax, int nb, SchurQuad sq) {
    const int r = blockIdx.y, lane = threadIdx.x & 31;
    const int j = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int n = quad_order(k_used, n_fixed, due, nullptr, 1, r);
    if (n < 0) return;
    if (j >= nb) {  // column j - nb of T
        if (j - nb >= sq.m) return;
        const double2* t = static_cast<const double2*>(sq.T) + (long long)(j - nb) * sq.m;
        double s = 0.0;
        for (int i = lane; i <= j - nb; i += 32) s += t[i].x * t[i].x + t[i].y * t[i].y;
        s = warp_sum(s);
        if (lane == 0) atomicMax(bmax + r, (unsigned long long)__double_as_longlong(sqrt(s)));
        return;
    }
    if (j >= n) return;
    const double2* c = H + r * h_rhs + (long long)j * ldh;
    const int rows = min(n, j + 2);
    double s = 0.0;
    for (int i = lane; i < rows; i += 32) s += c[i].x * c[i].x + c[i].y * c[i].y;
    if (sq.m > 0) {
        const double2* x = static_cast<const double2*>(sq.X) + r * sq.x_rhs + (long long)j * sq.m;
        for (int i = lane; i < sq.m; i += 32) s += x[i].x * x[i].x + x[i].y * x[i].y;
    }
    s = warp_sum(s);
    if (lane == 0) {
        atomicMax(bmax + r, (unsigned long long)__double_as_longlong(sqrt(s)));
        if (j + 1 < n) isub[(size_t)r * kmax + j + 1] = 1.0 / c[j + 1].x;
    }
}

// One node (one sign of t) per warp and pass: P[r][node][0..n) = (w/pi) (H - i t)^-1 e_1.
// Lane q of the warp owns rows q, q + 32, ...: s[j] sums row 32 j + q, and once
// row l has been used, its place keeps z_{l-1}. What bounds it: the FP64 units
// (two multiply-adds a clock and SM: 4 per complex term), for few right-hand
// sides the chain of k steps; the columns of H come from L2 through a ring of
// QS asynchronous copies, so their latency is off that chain. One warp per
// block: 96 nodes spread over as many SMs.
template <int KC>
__global__ void __launch_bounds__(32) k_quad_solve(const double2* __restrict__ H, long long h_rhs, int ldh,
                                                   const int* __restrict__ k_used, int n_fixed,
                                                   const int* __restrict__ due, const int* __restrict__ need, int level,
                                                   const unsigned long long* __restrict__ bmax,
                                                   const double* __restrict__ isub, int kmax, double2* __restrict__ P,
                                                   long long p_rhs, QuadNodes nodes) {
    extern __shared__ double2 ring[];  // [QS][32 KC]
    const int r = blockIdx.y, node = blockIdx.x, lane = threadIdx.x;
    const int n = quad_order(k_used, n_fixed, due, need, level, r);
    if (n <= 0) return;
    const double b = 2.0 * __longlong_as_double((long long)bmax[r]);
    const double2* Hr = H + r * h_rhs;
    const double* ib = isub + (size_t)r * kmax;
    // column c into its stage: rows 0 .. c
    auto fetch = [&](int c) {
        if (c >= 0) {
            const double2* src = Hr + (long long)c * ldh;
            double2* dst = ring + (size_t)(c % QS) * (32 * KC);
            for (int i = lane; i <= c; i += 32) cp16(dst + i, src + i);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    double2* out = P + r * p_rhs + (size_t)node * kmax;
    for (int pair = node >> 1; pair < nodes.pairs; pair += kPairs2) {
        double t, w;
        if (nodes.pairs <= kPairs2) {
            t = nodes.t[pair];
            w = nodes.w[pair];
        } else {
            quad_node(nodes, pair, t, w);
        }
        t = (node & 1) ? -t * b : t * b;
        w *= b;
        for (int c = n - 1; c > n - QS; --c) fetch(c);
        double sr[KC], si[KC];
#pragma unroll
        for (int j = 0; j < KC; ++j) sr[j] = si[j] = 0.0;
        double zr = 1.0, zi = 0.0, last = 1.0;  // z_l of the current column; z_{n-1}
#pragma unroll
        for (int sl = KC - 1; sl >= 0; --sl) {
            if (32 * sl >= n) continue;
            for (int q = min(31, n - 1 - 32 * sl); q >= 0; --q) {
                const int l = 32 * sl + q;
                __syncwarp();  // every lane has read the stage that is refilled here
                fetch(l - QS + 1);
                asm volatile("cp.async.wait_group %0;\n" ::"n"(QS - 1) : "memory");
                __syncwarp();
                const double ibl = l > 0 ? __ldg(ib + l) : 0.0;
                const double2* col = ring + (size_t)(l % QS) * (32 * KC);
                {  // slot sl first: z_{l-1} needs row l
                    double2 h = lane <= q ? col[32 * sl + lane] : make_double2(0.0, 0.0);
                    if (lane == q) h.y -= t;
                    sr[sl] = fma(h.x, zr, sr[sl]);
                    sr[sl] = fma(-h.y, zi, sr[sl]);
                    si[sl] = fma(h.x, zi, si[sl]);
                    si[sl] = fma(h.y, zr, si[sl]);
                }
                double nr = -lane_d(sr[sl], q) * ibl, ni = -lane_d(si[sl], q) * ibl;
                if (lane == q && l > 0) {
                    sr[sl] = nr;
                    si[sl] = ni;
                }
#pragma unroll
                for (int j = 0; j < sl; ++j) {
                    const double2 h = col[32 * j + lane];
                    sr[j] = fma(h.x, zr, sr[j]);
                    sr[j] = fma(-h.y, zi, sr[j]);
                    si[j] = fma(h.x, zi, si[j]);
                    si[j] = fma(h.y, zr, si[j]);
                }
                zr = nr;
                zi = ni;
                // exponent above 2^200: everything times 2^-200 (uniform over the warp)
                const int e = max((__double2hiint(zr) >> 20) & 0x7ff, (__double2hiint(zi) >> 20) & 0x7ff);
                if (e > 1023 + 200 && l > 0) {
                    const double f = 0x1p-200;
#pragma unroll
                    for (int j = 0; j < KC; ++j) {
                        sr[j] *= f;
                        si[j] *= f;
                    }
                    zr *= f;
                    zi *= f;
                    last *= f;
                }
            }
        }
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        const double gr = lane_d(sr[0], 0), gi = lane_d(si[0], 0);  // row 0: (H - i t)_0 z
        // w / gamma by a scaled division (gamma may be large)
        const double m = fmax(fabs(gr), fabs(gi));
        const double ar = gr / m, ai = gi / m, den = w / (m * (ar * ar + ai * ai));
        const double fr = ar * den, fi = -ai * den;
        const bool first = pair < kPairs2;
        auto put = [&](int l, double x, double y) {
            if (!first) {
                const double2 o = out[l];
                x += o.x;
                y += o.y;
            }
            out[l] = make_double2(x, y);
        };
#pragma unroll
        for (int j = 0; j < KC; ++j) {
            const int l = 32 * j + lane;  // this place holds z_{l-1}
            if (l >= 1 && l < n) put(l - 1, sr[j] * fr - si[j] * fi, sr[j] * fi + si[j] * fr);
        }
        if (lane == 0) put(n - 1, last * fr, last * fi);
        __syncwarp();
    }
}

// Schur part of a node: with w (H - i t)^-1 e_1 in P, the upper rows of
//   ([T X; 0 H] - i t)^-1 [c; beta e_1]
// are (T - i t)^-1 (c - beta X (H - i t)^-1 e_1); Q[r][node][0..m) = w times
// that. T is upper triangular, so a back substitution: one node per warp, lane
// q owns rows q, q + 32, ... The pair of sums over the nodes are the Schur and
// the Krylov coefficients of sgn of the composite matrix (Sec. 5.2, Eqs. newH,
// f_H): what App. A computes from sgn(T), sgn(H_k) and a Sylvester equation,
// without the recurrences that lose digits as k grows.
template <int MC>
__global__ void __launch_bounds__(32) k_quad_schur(const double2* __restrict__ P, long long p_rhs, int kmax,
                                                   const int* __restrict__ k_used, const int* __restrict__ need,
                                                   int level, const unsigned long long* __restrict__ bmax,
                                                   const double* __restrict__ beta, SchurQuad sq, QuadNodes nodes) {
    const int r = blockIdx.y, node = blockIdx.x, lane = threadIdx.x, m = sq.m;
    const int n = quad_order(k_used, 0, nullptr, need, level, r);
    if (n < 0) return;
    const double b = 2.0 * __longlong_as_double((long long)bmax[r]);
    const double t = (node & 1) ? -nodes.t[node >> 1] * b : nodes.t[node >> 1] * b;
    const double w = nodes.w[node >> 1] * b;
    const double2* T = static_cast<const double2*>(sq.T);
    const double2* X = static_cast<const double2*>(sq.X) + r * sq.x_rhs;
    const double2* c = static_cast<const double2*>(sq.c) + r * sq.c_rhs;
    const double2* z = P + r * p_rhs + (size_t)node * kmax;
    double vr[MC], vi[MC], dr[MC], di[MC];
#pragma unroll
    for (int j = 0; j < MC; ++j) {
        const int i = 32 * j + lane;
        vr[j] = vi[j] = dr[j] = di[j] = 0.0;
        if (i < m) {
            vr[j] = w * c[i].x;
            vi[j] = w * c[i].y;
            const double2 d = T[i + (long long)i * m];
            const double y = d.y - t, den = 1.0 / (d.x * d.x + y * y);
            dr[j] = d.x * den;
            di[j] = -y * den;
        }
    }
    const double bt = n > 0 ? beta[r] : 0.0;
#pragma unroll 4
    for (int l = 0; l < n; ++l) {
        const double2 zl = z[l];
        const double zr = -bt * zl.x, zi = -bt * zl.y;
#pragma unroll
        for (int j = 0; j < MC; ++j) {
            const int i = 32 * j + lane;
            const double2 x = i < m ? __ldg(X + (long long)l * m + i) : make_double2(0.0, 0.0);
            vr[j] = fma(x.x, zr, vr[j]);
            vr[j] = fma(-x.y, zi, vr[j]);
            vi[j] = fma(x.x, zi, vi[j]);
            vi[j] = fma(x.y, zr, vi[j]);
        }
    }
#pragma unroll
    for (int sl = MC - 1; sl >= 0; --sl) {
        for (int q = min(31, m - 1 - 32 * sl); q >= 0; --q) {  // not entered beyond m
            const int i = 32 * sl + q;
            const double yr = lane_d(vr[sl] * dr[sl] - vi[sl] * di[sl], q);
            const double yi = lane_d(vr[sl] * di[sl] + vi[sl] * dr[sl], q);
#pragma unroll
            for (int j = 0; j <= sl; ++j) {
                const int row = 32 * j + lane;
                const double2 x = row < i ? __ldg(T + (long long)i * m + row) : make_double2(0.0, 0.0);
                vr[j] = fma(-x.x, yr, vr[j]);
                vr[j] = fma(x.y, yi, vr[j]);
                vi[j] = fma(-x.x, yi, vi[j]);
                vi[j] = fma(-x.y, yr, vi[j]);
            }
            if (lane == q) {  // row i is done: it keeps its solution
                vr[sl] = yr;
                vi[sl] = yi;
            }
        }
    }
    double2* out = static_cast<double2*>(sq.Q) + r * sq.q_rhs + (size_t)node * m;
#pragma unroll
    for (int j = 0; j < MC; ++j)
        if (32 * j + lane < m) out[32 * j + lane] = make_double2(vr[j], vi[j]);
}

constexpr int RT = 512;

__device__ __forceinline__ double rsum(double v, double* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    for (int q = 0; q < RT / 32; ++q) s += sh[q];
    return s;
}

// Sum over the nodes, d and r (see the head of this file) and the verdict:
// need[r] = 0 where the result is accepted; only then it is written to coeff (and
// with Schur deflation to cS). One block per right-hand side; four groups of threads
// split the nodes.
__global__ void __launch_bounds__(RT) k_quad_sum(const double2* __restrict__ P, long long p_rhs, int pairs,
                                                 const int* __restrict__ k_used, int n_fixed,
                                                 const int* __restrict__ due, const double* __restrict__ beta,
                                                 int kmax, double2* __restrict__ coeff, long long coeff_stride,
                                                 int* __restrict__ need, int level, double tol, int iters_code,
                                                 int* __restrict__ iters, int* __restrict__ status, SchurQuad sq) {
    extern __shared__ double2 sum[];  // the result, n + m entries
    __shared__ double sh[RT / 32];
    __shared__ double2 part[3][RT];
    const int r = blockIdx.x, tid = threadIdx.x;
    const int n = quad_order(k_used, n_fixed, due, need, level, r);
    double2* cr = coeff + r * coeff_stride;
    if (n < 0) {
        if (level == 1 && tid == 0) need[r] = 0;
        return;
    }
    if (n == 0 && sq.m == 0) {  // an empty Krylov space: no coefficients
        for (int i = tid; i < kmax; i += RT) cr[i] = make_double2(0.0, 0.0);
        if (tid == 0) {
            need[r] = 0;
            iters[r] = 0;
            status[r] = 0;
        }
        return;
    }
    const double2* Pr = P + r * p_rhs;
    const double2* Qr = static_cast<const double2*>(sq.Q) + r * sq.q_rhs;
    const double2* sc = static_cast<const double2*>(sq.c) + r * sq.c_rhs;
    const int g = tid >> 7, i0 = tid & 127, all = n + sq.m;
    const double bt = n > 0 ? beta[r] : 0.0;
    double d2 = 0.0, r2 = 0.0, c2 = 0.0;
    for (int base = 0; base < all; base += 128) {
        const int i = base + i0;
        const double2* src = i < n ? Pr + i : Qr + (i - n);
        const int ld = i < n ? kmax : sq.m;
        double cx = 0.0, cy = 0.0, sx = 0.0, sy = 0.0, qx = 0.0, qy = 0.0;
        if (i < all) {
            for (int p = g; p < pairs; p += 4) {
                const double2 a = src[(size_t)(2 * p) * ld], c = src[(size_t)(2 * p + 1) * ld];
                const double x = a.x + c.x, y = a.y + c.y;
                cx += x;
                cy += y;
                const int third = p % 3;
                if (third == 1) {
                    sx += x;
                    sy += y;
                } else {
                    qx += third == 0 ? a.x - c.x : c.x - a.x;
                    qy += third == 0 ? a.y - c.y : c.y - a.y;
                }
            }
        }
        __syncthreads();
        part[0][tid] = make_double2(cx, cy);
        part[1][tid] = make_double2(sx, sy);
        part[2][tid] = make_double2(qx, qy);
        __syncthreads();
        if (g == 0 && i < all) {
            for (int q = 1; q < 4; ++q) {
                const double2 a = part[0][tid + 128 * q], c = part[1][tid + 128 * q], b = part[2][tid + 128 * q];
                cx += a.x;
                cy += a.y;
                sx += c.x;
                sy += c.y;
                qx += b.x;
                qy += b.y;
            }
            const double f = i < n ? bt : 1.0;  // the Schur rows have beta in them
            cx *= f;
            cy *= f;
            sx *= f;
            sy *= f;
            const double h = 0.86602540378443865 * f;
            const double2 e = i >= n ? sc[i - n] : make_double2(i == 0 ? bt : 0.0, 0.0);  // the vector that sgn acts on
            const double rx = -h * qy - e.x, ry = h * qx - e.y;
            d2 += (cx - 3.0 * sx) * (cx - 3.0 * sx) + (cy - 3.0 * sy) * (cy - 3.0 * sy);
            r2 += rx * rx + ry * ry;
            c2 += cx * cx + cy * cy;
            sum[i] = make_double2(cx, cy);
        }
    }
    d2 = rsum(d2, sh);
    r2 = rsum(r2, sh);
    c2 = rsum(c2, sh);
    const bool ok = sqrt(d2) + sqrt(r2) <= tol * sqrt(c2) && isfinite(c2);  // false for NaN
    if (ok) {
        for (int i = tid; i < kmax; i += RT) cr[i] = i < n ? sum[i] : make_double2(0.0, 0.0);
        for (int i = tid; i < sq.m; i += RT) static_cast<double2*>(sq.cS)[r * sq.cs_rhs + i] = sum[n + i];
    }
    if (tid == 0) {
        need[r] = ok ? 0 : 1;
        if (ok) {
            iters[r] = n > 0 ? iters_code : 0;
            status[r] = 0;
        }
    }
}

template <int KC>
cudaError_t solve(int pairs, int nrhs, cudaStream_t st, const void* H, long long h_rhs, int ldh, const int* k_used,
                  int n_fixed, const int* due, const int* need, int level, const unsigned long long* bmax,
                  const double* isub, int kmax, void* P, long long p_rhs, const QuadNodes& nodes) {
    const size_t smem = (size_t)QS * 32 * KC * sizeof(double2);
    const cudaError_t e = ensure_dyn_smem((const void*)k_quad_solve<KC>, smem);
    if (e != cudaSuccess) return e;
    k_quad_solve<KC><<<dim3(2 * pairs, nrhs), 32, smem, st>>>((const double2*)H, h_rhs, ldh, k_used, n_fixed, due,
                                                             need, level, bmax, isub, kmax, (double2*)P, p_rhs, nodes);
    return cudaGetLastError();
}

}  // namespace

// complex128 entries of work per right-hand side: the nodes' columns, the
// inverse subdiagonal and the norm
long long sign_quad_work(int kmax) { return (long long)(2 * kPairs2 + 1) * kmax + 2; }

cudaError_t launch_sign_quad(const void* H, long long h_rhs, int ldh, const int* k_used, const double* beta,
                             void* coeff, long long coeff_stride, void* work, long long work_rhs, int kmax,
                             int k_bound, int nrhs, int prec, int* iters, int* status, int* need, cudaStream_t st,
                             const int* due, int n_fixed, const SchurQuad& sq) {
    static const QuadNodes nodes64 = make_nodes(kPairs64, kWindow1), nodes32 = make_nodes(kPairs32, kWindow1),
                           nodes2 = make_nodes(kPairs2, kWindow2), nodes3 = make_nodes(kPairs3, kWindow2),
                           nodes4 = make_nodes(kPairs4, kWindow2);
    double2* P = (double2*)work;  // [nrhs][2 kPairs2][kmax], then bmax and isub of all right-hand sides
    if (work_rhs < sign_quad_work(kmax)) return cudaErrorInvalidValue;
    const long long p_rhs = 2LL * kPairs2 * kmax;
    unsigned long long* bmax = (unsigned long long*)(P + p_rhs * nrhs);
    double* isub = (double*)(bmax + 2 * nrhs);
    cudaError_t e = cudaMemsetAsync(bmax, 0, sizeof(*bmax) * nrhs, st);
    if (e != cudaSuccess) return e;
    const int nb = n_fixed > 0 ? n_fixed : k_bound;
    k_quad_prep<<<dim3((nb + sq.m + 7) / 8, nrhs), 256, 0, st>>>((const double2*)H, h_rhs, ldh, k_used, n_fixed, due,
                                                                 bmax, isub, kmax, nb, sq);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // (the Schur part needs every node's solution, which the third rule adds up)
    for (int level = 1; level <= (sq.m > 0 ? 2 : nb > kLastRule ? 4 : 3); ++level) {
        const QuadNodes& q = level == 2   ? nodes2
                             : level == 3 ? nodes3
                             : level == 4 ? nodes4
                             : prec == PREC_F64 ? nodes64 : nodes32;
        const int pairs = std::min(q.pairs, kPairs2);
        const int kc = (nb + 31) / 32;
#define OVS_QUAD(K)                                                                                               \
    e = solve<K>(pairs, nrhs, st, H, h_rhs, ldh, k_used, n_fixed, due, need, level, bmax, isub, kmax, P, p_rhs, q)
        if (kc <= 2) OVS_QUAD(2);
        else if (kc <= 4) OVS_QUAD(4);
        else if (kc <= 6) OVS_QUAD(6);
        else if (kc <= 8) OVS_QUAD(8);
        else if (kc <= 12) OVS_QUAD(12);
        else if (kc <= 16) OVS_QUAD(16);
        else if (kc <= 20) OVS_QUAD(20);
        else if (kc <= 25) OVS_QUAD(25);
        else return cudaErrorInvalidValue;
#undef OVS_QUAD
        if (e != cudaSuccess) return e;
        if (sq.m > 0) {
            const dim3 grid(2 * pairs, nrhs);
#define OVS_QSCHUR(M) \
    k_quad_schur<M><<<grid, 32, 0, st>>>(P, p_rhs, kmax, k_used, need, level, bmax, beta, sq, q)
            if (sq.m <= 32) OVS_QSCHUR(1);
            else if (sq.m <= 64) OVS_QSCHUR(2);
            else if (sq.m <= 128) OVS_QSCHUR(4);
            else if (sq.m <= 256) OVS_QSCHUR(8);
            else return cudaErrorInvalidValue;
#undef OVS_QSCHUR
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        int code = 0;  // the Roberts iterate of that degree: ceil(log2(2 pairs))
        while ((1 << code) < 2 * q.pairs) ++code;
        k_quad_sum<<<nrhs, RT, sizeof(double2) * (size_t)(nb + sq.m), st>>>(
            P, p_rhs, pairs, k_used, n_fixed, due, beta, kmax, (double2*)coeff, coeff_stride, need, level,
            prec == PREC_F64 ? kTol64 : kTol32, code, iters, status, sq);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace ovs
