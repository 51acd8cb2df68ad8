// Shared by fine_sweeps.cu (complex64) and fix_sweeps.cu (complex128): the
// scalars and the column of an Arnoldi step inside its update kernel.
#pragma once

#include "arnoldi_dev.cuh"
#include "common.cuh"
#include "kernels.h"

namespace ovs {

constexpr int FT = 256, FW = FT / 32;  // threads and warps per block
constexpr int FU = 4;                  // units per lane of a tile of 32 FU
constexpr int FTILE = 32 * FU;
constexpr int FV = 4;  // basis vectors per pass of a warp

struct StepShared {  // of a block of the update
    double sh[4 * FW];
    double2 d;
    double ib, beta;
    int brk;
};

// Sum i of the chunks of right-hand side r.
__device__ __forceinline__ double2 chunk_sum(const double2* __restrict__ all, int S, int nchunk, int i) {
    double2 a = make_double2(0.0, 0.0);
#pragma unroll 12
    for (int b = 0; b < nchunk; ++b) {
        const double2 p = __ldg(all + (size_t)b * S + i);
        a.x += p.x;
        a.y += p.y;
    }
    return a;
}

// ||s||^2, s^H t, ||column J-1||^2 after its second pass (see arnoldi_step):
// true in warp 0, whose lanes hold the sums.
__device__ __forceinline__ bool step_sums(const double2* s, const double2* t, int J, int r, const FineStep& fs,
                                          StepShared& sm, double (&v)[4]) {
    const double2* fp = static_cast<const double2*>(fs.fp) + r * fs.fp_rhs;  // column J-1, first pass
    v[0] = v[1] = v[2] = v[3] = 0.0;
    for (int i = threadIdx.x; i < J; i += FT) {
        const double2 si = s[i], ti = t[i], f = fp[i];
        const double hx = f.x + si.x, hy = f.y + si.y;
        v[0] += si.x * si.x + si.y * si.y;
        v[1] += si.x * ti.x + si.y * ti.y;
        v[2] += si.x * ti.y - si.y * ti.x;
        v[3] += hx * hx + hy * hy;
    }
    return block_sum4(v, sm.sh, J);
}

// The scalars of the step, by one thread of the block; the first block of a
// right-hand side stores them.
__device__ __forceinline__ void step_scalars(const double (&v)[4], double uu, double2 uz, int J, int r, bool first,
                                             const FineStep& fs, StepShared& sm) {
    const double b2 = uu - v[0];
    // a NaN (from a non-finite source) stays NaN, so that it is reported
    const double beta = (b2 > 0.0 || isnan(b2)) ? sqrt(b2) : 0.0;
    const double hn2 = J == 0 ? 0.0 : fs.hnorm2[r] + v[3] + (b2 < 0.0 ? 0.0 : b2);
    const bool brk = !(b2 > kBreakdownTol * kBreakdownTol * hn2) || !isfinite(beta);
    const double ib = brk ? 0.0 : rsqrt(b2);  // beside the square root, not after it
    sm.beta = brk ? 0.0 : beta;
    sm.ib = ib;
    sm.d = make_double2((uz.x - v[1]) * ib * ib, (uz.y - v[2]) * ib * ib);
    sm.brk = brk ? 1 : 0;
    if (first) {
        if (J == 0) fs.beta0[r] = beta;
        fs.inv_beta[r] = ib;
        fs.hnorm2n[r] = hn2;
        fs.activen[r] = brk ? 0 : 1;
        fs.k_used[r] = brk ? J : J + 1;
    }
}

// Row l of column J-1 (complete) and J (first pass), by one warp.
__device__ __forceinline__ void step_column(const double2* s, const double2* t, int J, int l, int r,
                                            const FineStep& fs, const StepShared& sm) {
    if (l > J) return;
    const int lane = threadIdx.x & 31;
    const double2* fp = static_cast<const double2*>(fs.fp) + r * fs.fp_rhs;
    double2* Hr = static_cast<double2*>(fs.H) + r * fs.h_rhs;
    double gr = 0.0, gi = 0.0;
    for (int i = (l > 0 ? l - 1 : 0) + lane; i < J; i += 32) {
        double2 h;
        if (i < J - 1) {
            h = Hr[l + (long long)i * fs.ldh];
        } else {  // column J-1: its second pass is s
            h = l < J ? make_double2(fp[l].x + s[l].x, fp[l].y + s[l].y) : make_double2(sm.beta, 0.0);
            Hr[l + (long long)i * fs.ldh] = h;
        }
        const double2 si = s[i];
        gr += h.x * si.x - h.y * si.y;
        gi += h.x * si.y + h.y * si.x;
    }
    gr = warp_sum(gr);
    gi = warp_sum(gi);
    if (lane != 0 || sm.brk) return;
    double2* fpn = static_cast<double2*>(fs.fpn) + r * fs.fp_rhs;
    fpn[l] = l < J ? make_double2((t[l].x - gr) * sm.ib, (t[l].y - gi) * sm.ib)
                   : make_double2(sm.d.x - gr * sm.ib, sm.d.y - gi * sm.ib);
}

// Before a launch with `smem` bytes of dynamic shared memory: beyond 48 KB with the
// kernel's own (the updates for small fields have up to 17 KB) it has to be asked for;
// 8 KB at a time, as it grows with J.
inline cudaError_t allow_smem(const void* kernel, size_t smem) {
    return smem <= 16 * 1024 ? cudaSuccess : ensure_dyn_smem(kernel, (smem + 8191) / 8192 * 8192);
}

// complex128 forms (fix_sweeps.cu)
int fix_chunks(long long nunits, int J, int nrhs, int num_sms);
cudaError_t launch_fix_dots(int nw, const void* basis, long long basis_rhs, long long vec_stride, int J,
                            const int* vexp, long long vexp_rhs, int* uexp, const void* u, const void* z,
                            long long nunits, int nrhs, int num_sms, void* partial, const int* active,
                            cudaStream_t st);
cudaError_t launch_fix_update(void* basis, long long basis_rhs, long long vec_stride, int J, int* vexp,
                              long long vexp_rhs, const int* uexp, int* uexpn, const void* sums, long long s_rhs,
                              int nchunk, void* u, const void* z, long long nunits, int nrhs, int num_sms,
                              const FineStep& fs, cudaStream_t st);

}  // namespace ovs
