// Device code of one Arnoldi step in the delayed-reorthogonalisation form of
// CGS2, shared by the kernels that run it as launches of its own (blas.cu) and by
// the sweeps (fine_sweeps.cu, pair_sweeps.cu).
#pragma once

#include "common.cuh"

namespace ovs {

template <typename R> __device__ __forceinline__ R warp_sum(R v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

constexpr double kBreakdownTol = 1e-12;  // relative to ||H_j||_F; rounding of an exactly
                                         // invariant space is ~100 eps at N ~ 1e5

__device__ __forceinline__ void block_sum3(double& a, double& b, double& c, double* sh) {
    a = warp_sum(a);
    b = warp_sum(b);
    c = warp_sum(c);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if (lane == 0) {
        sh[3 * w] = a;
        sh[3 * w + 1] = b;
        sh[3 * w + 2] = c;
    }
    __syncthreads();
    a = b = c = 0.0;
    for (int q = 0; q < nw; ++q) {
        a += sh[3 * q];
        b += sh[3 * q + 1];
        c += sh[3 * q + 2];
    }
    __syncthreads();
}

// Sums of four values over the block (at most 8 warps; sh: 32 doubles of shared
// memory; the threads from `used` on have nothing to add): true in warp 0, whose
// lanes then hold all four in v. A scheduler issues an FP64 operation of a warp
// every 64 clocks (66 to its result, 600 for a square root), so the four values
// are reduced together, in six additions per warp that has any.
__device__ __forceinline__ bool block_sum4(double (&v)[4], double* sh, int used) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = min((int)blockDim.x >> 5, (used + 31) >> 5);
    __syncthreads();
    if (warp < nw) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const bool up = (lane & 16) != 0;
            const double send = up ? v[k] : v[k + 2], keep = up ? v[k + 2] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
        }
        {
            const bool up = (lane & 8) != 0;
            const double send = up ? v[0] : v[1], keep = up ? v[1] : v[0];
            v[0] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
        }
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 4);
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
        // lane 8 q holds value q: 16 is bit 1 of its index, 8 bit 0
        if ((lane & 7) == 0) sh[4 * warp + (lane >> 3)] = v[0];
    }
    __syncthreads();
    if (warp != 0) return false;
    double a = lane < 4 * nw ? sh[lane] : 0.0;
    if (nw > 4) a += __shfl_xor_sync(0xffffffffu, a, 16);
    if (nw > 2) a += __shfl_xor_sync(0xffffffffu, a, 8);
    if (nw > 1) a += __shfl_xor_sync(0xffffffffu, a, 4);
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = __shfl_sync(0xffffffffu, a, k);
    return true;
}

// One Arnoldi step in the delayed-reorthogonalisation form of CGS2 (run by
// one block of at most 256
// threads per right-hand side, r active; sh: 32 doubles of shared memory).
// Input rr = red[r] = (s, t, u^H u, u^H z) from the
// sweep over V_0..V_{j-1} (s = V^H u, t = V^H z, z = A u), where u is the
// first-pass Gram-Schmidt residual of the previous step (x_ominus at j=0).
//  - beta = ||u - V s|| = sqrt(u^H u - ||s||^2) (V orthonormal);
//  - j > 0: column j-1 of H gets its second-pass correction s and
//    H[j][j-1] = beta; breakdown if beta <= 1e-12 ||H_j||_F (k_used = j);
//  - j = 0: beta is ||x_ominus|| (kept in beta0 for the result);
//  - column j, first pass: with g = Hbar_{j-1} s (Arnoldi relation
//    A V_{j-1} = V_j Hbar_{j-1}), H[i][j] = (t_i - g_i)/beta for i < j and
//    H[j][j] = (u^H z - s^H t)/beta^2 - g_j/beta (arnoldi_column, the
//    O(j^2) part, spread over many blocks);
//  - the update sweep then needs 1/beta and d = (u^H z - s^H t)/beta^2.
struct StepOut {  // per right-hand side
    double2* H;
    long long h_rhs;
    int ldh;
    double *beta0, *inv_beta;
    double2* dcoef;
    double* hnorm2;
    int *active, *k_used;
};
__device__ __forceinline__ void arnoldi_step(const double2* rr, int j, int r, const StepOut& o, double* sh) {
    const int tid = threadIdx.x, lane = tid & 31;
    double2* Hr = o.H + r * o.h_rhs;
    const int ldh = o.ldh;
    // ||s||^2, s^H t, ||column j-1||^2 after its second pass
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    for (int i = tid; i < j; i += blockDim.x) {
        const double2 si = rr[i], ti = rr[j + i];
        double2 h = Hr[i + (long long)(j - 1) * ldh];
        h = make_double2(h.x + si.x, h.y + si.y);
        Hr[i + (long long)(j - 1) * ldh] = h;
        v[0] += si.x * si.x + si.y * si.y;
        v[1] += si.x * ti.x + si.y * ti.y;
        v[2] += si.x * ti.y - si.y * ti.x;
        v[3] += h.x * h.x + h.y * h.y;
    }
    if (!block_sum4(v, sh, j)) return;  // warp 0 has the sums
    const double ss = v[0], shr = v[1], shi = v[2], c2 = v[3];
    if (lane != 0) return;
    const double b2 = rr[2 * j].x - ss;
    const double2 uz = rr[2 * j + 1];
    // a NaN (from a non-finite source) stays NaN, so that it is reported
    const double beta = (b2 > 0.0 || isnan(b2)) ? sqrt(b2) : 0.0;
    const double ib = b2 > 0.0 ? rsqrt(b2) : 0.0;  // beside the square root, not after it
    if (j == 0) {
        o.beta0[r] = beta;
        o.hnorm2[r] = 0.0;
        if (!(beta > 0.0) || !isfinite(beta)) {
            o.active[r] = 0;
            o.k_used[r] = 0;
            o.inv_beta[r] = 0.0;
            return;
        }
    } else {
        const double hn2 = o.hnorm2[r] + c2 + (b2 < 0.0 ? 0.0 : b2);
        const bool brk = !(b2 > kBreakdownTol * kBreakdownTol * hn2) || !isfinite(beta);  // beta > tol ||H_j||_F
        o.hnorm2[r] = hn2;
        Hr[j + (long long)(j - 1) * ldh] = make_double2(brk ? 0.0 : beta, 0.0);
        if (brk) {
            o.active[r] = 0;
            o.k_used[r] = j;
            o.inv_beta[r] = 0.0;
            return;
        }
    }
    o.inv_beta[r] = ib;
    o.dcoef[r] = make_double2((uz.x - shr) * ib * ib, (uz.y - shi) * ib * ib);
    o.k_used[r] = j + 1;
}

// Row l <= j of column j of H, first pass (after arnoldi_step of the same j): with
// g = Hbar_{j-1} s, H[l][j] = (t_l - g_l)/beta for l < j and
// H[j][j] = d - g_j/beta. One warp per row l: the lanes split the terms of
// g_l (H is upper Hessenberg, so i >= l - 1) and reduce with shuffles.
__device__ __forceinline__ void arnoldi_column(const double2* rr, int j, int l, double2* Hr, int ldh, double ib,
                                               double2 d) {
    const int lane = threadIdx.x & 31;
    double gr = 0.0, gi = 0.0;
    for (int i = (l > 0 ? l - 1 : 0) + lane; i < j; i += 32) {
        const double2 h = Hr[l + (long long)i * ldh];
        const double2 si = rr[i];
        gr += h.x * si.x - h.y * si.y;
        gi += h.x * si.y + h.y * si.x;
    }
    for (int off = 16; off > 0; off >>= 1) {
        gr += __shfl_xor_sync(0xffffffffu, gr, off);
        gi += __shfl_xor_sync(0xffffffffu, gi, off);
    }
    if (lane != 0) return;
    if (l < j) {
        const double2 ti = rr[j + l];
        Hr[l + (long long)j * ldh] = make_double2((ti.x - gr) * ib, (ti.y - gi) * ib);
    } else {
        Hr[j + (long long)j * ldh] = make_double2(d.x - gr * ib, d.y - gi * ib);
    }
}

}  // namespace ovs
