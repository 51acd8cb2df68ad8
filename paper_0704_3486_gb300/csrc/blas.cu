// K2 (classical Gram-Schmidt sweeps of the Arnoldi recurrence, Sec. 4
// Eq. Arnoldi), K4 (recombination y += V_k c, Eq. yproj3 / fAxLRArn) and
// K5 (LR projection c = L^+ x, x_ominus = x - R c, Sec. 5.3 Eq. xdec).
//
// A field is a flat array of 16-byte units (one complex128, or two
// complex64). Each right-hand side r owns its Krylov basis; in the register
// sweeps here a block of 256 threads covers one row block of one
// right-hand side and streams every basis vector through it, so the basis
// is read once per sweep with fully coalesced 16-byte loads. They serve the
// projections and the outer GMRES; the Arnoldi sweeps are in
// fix_sweeps.cu, fine_sweeps.cu, tma_sweeps.cu and pair_sweeps.cu.
// Also here: the shared-basis combination of the deflated part
// (k_shared_combine) and the small kernels of each Arnoldi step (partial
// sums, Hessenberg column, final pass).
//
// Precision: in the complex64 form the products and the partial sums of a
// thread (2*E terms) and of a warp (a 32-lane tree) are FP32; every warp
// partial is then added into FP64, so inner products, norms and Hessenberg
// entries are accumulated in FP64 over the rest of the vector.
#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

#include "arnoldi_dev.cuh"
#include "common.cuh"
#include "kernels.h"

namespace ovs {

constexpr int BT = 256;  // threads per block
constexpr int NWARP = BT / 32;

// ----------------------------------------------------------------- dots
// Warp transpose-reduction: every lane holds M values; after five halving
// exchanges lane l holds, in v[0 .. M/32), the warp sums of the values
// with index l*(M/32) + q. Each shuffle moves one useful value, so 32
// vectors cost 31 shuffles instead of 5 x 32.
template <int CUR, int O, typename R, int M>
__device__ __forceinline__ void tr_step(R (&v)[M], bool upper) {
#pragma unroll
    for (int i = 0; i < CUR / 2; ++i) {
        const R send = upper ? v[i] : v[i + CUR / 2];
        const R keep = upper ? v[i + CUR / 2] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
    }
}
template <typename R, int M> __device__ __forceinline__ void transpose_reduce(R (&v)[M], int lane) {
    static_assert(M % 32 == 0, "M must be a multiple of 32");
    tr_step<M, 16>(v, (lane & 16) != 0);
    tr_step<M / 2, 8>(v, (lane & 8) != 0);
    tr_step<M / 4, 4>(v, (lane & 4) != 0);
    tr_step<M / 8, 2>(v, (lane & 2) != 0);
    tr_step<M / 16, 1>(v, (lane & 1) != 0);
}

// Inner products of one basis sweep, per right-hand side r and row block b:
// s_i = V_i^H u (i < J), output partial[r][b][S], S = J + 2 (the last two
// entries are not written). Serves the projections, the set-up and the outer
// GMRES; the Arnoldi steps have their own sweeps.
// A lane keeps E 16-byte units of u in registers (a tile of 256*E units per
// block); G basis vectors are then streamed past them. Each lane accumulates
// its E*NC products per vector in FP32 (FP64 for complex128 fields), a warp
// transpose-reduction finishes the partial over the 32 lanes (at most
// 32*E*NC = 256 terms in FP32), and the warp partials are accumulated in FP64
// in shared memory.
template <typename R, int G, int E>
__global__ void __launch_bounds__(BT, sizeof(R) == 4 ? 2 : 1) k_gdots(const typename Unit<R>::vec* __restrict__ basis,
                                              long long basis_rhs_stride, long long vec_stride, int J,
                                              const typename Unit<R>::vec* __restrict__ u, long long u_rhs_stride,
                                              long long nunits, long long chunk, int nblk,
                                              double2* __restrict__ partial, const int* __restrict__ active) {
    using vec = typename Unit<R>::vec;
    constexpr int NC = Unit<R>::ncplx;
    constexpr int M = 2 * G;
    constexpr int PER = M / 32;
    extern __shared__ double2 sacc2[];  // [NWARP][S]
    double* sacc = reinterpret_cast<double*>(sacc2);
    const int r = blockIdx.x, b = blockIdx.y;
    if (active != nullptr && active[r] == 0) return;
    const int S = J + 2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < NWARP * S * 2; i += BT) sacc[i] = 0.0;
    __syncthreads();
    const vec* Vr = basis + r * basis_rhs_stride;
    const vec* ur = u + r * u_rhs_stride;
    double* myacc = sacc + (size_t)warp * S * 2;
    const long long u0 = (long long)b * chunk;
    const long long u1 = min(u0 + chunk, nunits);
    for (long long base = u0; base < u1; base += (long long)BT * E) {
        cplx<R> uc[E][NC];
        bool ok[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const long long q = base + tid + (long long)BT * e;
            ok[e] = q < u1;
#pragma unroll
            for (int c = 0; c < NC; ++c) uc[e][c] = {R(0), R(0)};
            if (ok[e]) Unit<R>::split(__ldg(ur + q), uc[e]);
        }
        for (int i0 = 0; i0 < J; i0 += G) {
            R v[M];
#pragma unroll
            for (int q = 0; q < M; ++q) v[q] = R(0);
#pragma unroll
            for (int gi = 0; gi < G; ++gi) {
                if (i0 + gi < J) {
                    const vec* vi = Vr + (long long)(i0 + gi) * vec_stride;
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        if (ok[e]) {
                            cplx<R> vc[NC];
                            Unit<R>::split(__ldcs(vi + base + tid + (long long)BT * e), vc);
#pragma unroll
                            for (int c = 0; c < NC; ++c) {
                                cplx<R> acc = {v[2 * gi], v[2 * gi + 1]};
                                cfmac(acc, vc[c], uc[e][c]);
                                v[2 * gi] = acc.re;
                                v[2 * gi + 1] = acc.im;
                            }
                        }
                    }
                }
            }
            transpose_reduce(v, lane);
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int idx = lane * PER + q;
                const int gi = idx >> 1, comp = idx & 1;
                if (i0 + gi < J) myacc[(i0 + gi) * 2 + comp] += double(v[q]);
            }
        }
    }
    __syncthreads();
    for (int i = tid; i < 2 * J; i += BT) {
        double sum = 0.0;
#pragma unroll
        for (int q = 0; q < NWARP; ++q) sum += sacc[(size_t)q * S * 2 + i];
        reinterpret_cast<double*>(partial + ((size_t)r * nblk + b) * S)[i] = sum;
    }
}

// --------------------------------------------------------------- update
// Out element type per basis unit: NC complex numbers of precision RO.
template <typename RO, int NC> struct OutIO;
template <> struct OutIO<double, 1> {
    __device__ __forceinline__ static void load(const void* p, long long u, cd* o) {
        double2 v = static_cast<const double2*>(p)[u];
        o[0] = {v.x, v.y};
    }
    __device__ __forceinline__ static void store(void* p, long long u, const cd* o) {
        static_cast<double2*>(p)[u] = make_double2(o[0].re, o[0].im);
    }
};
template <> struct OutIO<double, 2> {
    __device__ __forceinline__ static void load(const void* p, long long u, cd* o) {
        const double2* q = static_cast<const double2*>(p) + 2 * u;
        double2 a = q[0], b = q[1];
        o[0] = {a.x, a.y};
        o[1] = {b.x, b.y};
    }
    __device__ __forceinline__ static void store(void* p, long long u, const cd* o) {
        double2* q = static_cast<double2*>(p) + 2 * u;
        q[0] = make_double2(o[0].re, o[0].im);
        q[1] = make_double2(o[1].re, o[1].im);
    }
};
template <> struct OutIO<float, 2> {
    __device__ __forceinline__ static void load(const void* p, long long u, cf* o) {
        float4 v = static_cast<const float4*>(p)[u];
        o[0] = {v.x, v.y};
        o[1] = {v.z, v.w};
    }
    __device__ __forceinline__ static void store(void* p, long long u, const cf* o) {
        static_cast<float4*>(p)[u] = make_float4(o[0].re, o[0].im, o[1].re, o[1].im);
    }
};

// out_r = in_r + sum_{i<J} V_r,i * (alpha c_r,i). Strides of in/out are in
// complex numbers of precision RO; basis strides in units.
template <typename RV, typename RO, int E>
__global__ void __launch_bounds__(BT) k_update(const typename Unit<RV>::vec* __restrict__ basis,
                                               long long basis_rhs_stride, long long vec_stride, int J,
                                               const double2* __restrict__ coef,
                                               long long coef_stride, double alpha, const cplx<RO>* in,
                                               long long in_rhs_stride, cplx<RO>* out, long long out_rhs_stride,
                                               long long nunits, long long chunk, int nblk,
                                               double* __restrict__ norm_partial, const int* __restrict__ active) {
    using vec = typename Unit<RV>::vec;
    constexpr int NC = Unit<RV>::ncplx;
    extern __shared__ double2 scoef2[];
    cplx<RV>* scoef = reinterpret_cast<cplx<RV>*>(scoef2);  // alpha*c, converted once per block
    __shared__ double sred[NWARP];
    const int r = blockIdx.x, b = blockIdx.y;
    if (active != nullptr && active[r] == 0) return;
    const int tid = threadIdx.x;
    for (int i = tid; i < J; i += BT) {
        double2 c = coef[r * coef_stride + i];
        scoef[i] = {RV(alpha * c.x), RV(alpha * c.y)};
    }
    __syncthreads();
    const vec* Vr = basis + r * basis_rhs_stride;
    const cplx<RO>* inr = in ? in + r * in_rhs_stride : nullptr;
    cplx<RO>* outr = out + r * out_rhs_stride;
    const long long u0 = (long long)b * chunk;
    const long long u1 = min(u0 + chunk, nunits);
    double nrm = 0.0;
    for (long long base = u0; base < u1; base += (long long)BT * E) {
        cplx<RO> o[E][NC];
        cplx<RV> acc[E][NC];
        bool ok[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const long long u = base + tid + (long long)BT * e;
            ok[e] = u < u1;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                o[e][c] = {RO(0), RO(0)};
                acc[e][c] = {RV(0), RV(0)};
            }
            if (ok[e] && inr != nullptr) OutIO<RO, NC>::load(inr, u, o[e]);
        }
        int since_flush = 0;
        for (int i = 0; i < J; ++i) {
            const cplx<RV> ci = scoef[i];
            const vec* vi = Vr + (long long)i * vec_stride;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                if (ok[e]) {
                    cplx<RV> vc[NC];
                    Unit<RV>::split(__ldcs(vi + base + tid + (long long)BT * e), vc);
#pragma unroll
                    for (int c = 0; c < NC; ++c) cfma(acc[e][c], vc[c], ci);
                }
            }
            // Wider output than basis: flush the FP32 partial sums every 16 terms.
            if (sizeof(RO) > sizeof(RV) && ++since_flush == 16) {
                since_flush = 0;
#pragma unroll
                for (int e = 0; e < E; ++e)
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        o[e][c].re += RO(acc[e][c].re);
                        o[e][c].im += RO(acc[e][c].im);
                        acc[e][c] = {RV(0), RV(0)};
                    }
            }
        }
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (!ok[e]) continue;
            RV pn = RV(0);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                o[e][c].re += RO(acc[e][c].re);
                o[e][c].im += RO(acc[e][c].im);
                pn += RV(o[e][c].re) * RV(o[e][c].re) + RV(o[e][c].im) * RV(o[e][c].im);
            }
            nrm += double(pn);
            OutIO<RO, NC>::store(outr, base + tid + (long long)BT * e, o[e]);
        }
    }
    if (norm_partial != nullptr) {
        nrm = warp_sum(nrm);
        if ((tid & 31) == 0) sred[tid >> 5] = nrm;
        __syncthreads();
        if (tid == 0) {
            double s = 0.0;
#pragma unroll
            for (int q = 0; q < NWARP; ++q) s += sred[q];
            norm_partial[(size_t)r * nblk + b] = s;
        }
    }
}

// --------------------------------------------------------------- small ops
__global__ void k_reduce(const double2* __restrict__ partial, int nblk, int pstride, int J, int nrhs,
                         double2* __restrict__ out, long long out_stride, int accumulate,
                         const int* __restrict__ active) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= J * nrhs) return;
    const int r = idx / J, i = idx % J;
    if (active != nullptr && active[r] == 0) return;
    double sx = 0.0, sy = 0.0;
    for (int b = 0; b < nblk; ++b) {
        double2 p = partial[((size_t)r * nblk + b) * pstride + i];
        sx += p.x;
        sy += p.y;
    }
    double2* o = out + r * out_stride + i;
    if (accumulate) {
        double2 v = *o;
        *o = make_double2(v.x + sx, v.y + sy);
    } else {
        *o = make_double2(sx, sy);
    }
}

// The same for many blocks: a thread block takes 8 sums, every group of 8
// threads one 32nd of the blocks' parts, so that the loads of a sum run 32 deep and
// its additions spread over the FP64 units of many SMs (304 parts of 480 sums: 15
// blocks of 32 sums with 8 groups took 11.4 us, 60 of these take 5.8).
constexpr int RW = 8;         // sums per block
constexpr int RG = 256 / RW;  // groups
__global__ void __launch_bounds__(256) k_reduce_wide(const double2* __restrict__ partial, int nblk, int pstride, int J,
                                                     int nrhs, double2* __restrict__ out, long long out_stride,
                                                     int accumulate, const int* __restrict__ active) {
    __shared__ double2 sh[RG][RW];
    const int col = threadIdx.x % RW, g = threadIdx.x / RW;
    const int idx = blockIdx.x * RW + col;
    const bool live = idx < J * nrhs;
    const int r = live ? idx / J : 0, i = live ? idx - r * J : 0;
    const bool on = live && (active == nullptr || active[r] != 0);
    double2 s = make_double2(0.0, 0.0);
    if (on) {
#pragma unroll 4
        for (int b = g; b < nblk; b += RG) {
            const double2 p = partial[((size_t)r * nblk + b) * pstride + i];
            s.x += p.x;
            s.y += p.y;
        }
    }
    sh[g][col] = s;
#pragma unroll
    for (int half = RG / 2; half > 0; half /= 2) {
        __syncthreads();
        if (g < half) {
            s.x += sh[g + half][col].x;
            s.y += sh[g + half][col].y;
            sh[g][col] = s;
        }
    }
    if (g != 0 || !on) return;
    double2* o = out + r * out_stride + i;
    if (accumulate) {
        const double2 v = *o;
        s = make_double2(v.x + s.x, v.y + s.y);
    }
    *o = s;
}

// The step and the column of H as launches of their own (after the TMA
// sweeps): one block per right-hand side, and one warp per row with 8 rows per
// block and the right-hand side in y.
__global__ void __launch_bounds__(256) k_arnoldi_step(const double2* __restrict__ red, long long red_stride, int j,
                                                      StepOut o) {
    __shared__ double sh[32];
    const int r = blockIdx.x;
    if (o.active[r] == 0) return;
    arnoldi_step(red + r * red_stride, j, r, o, sh);
}
__global__ void __launch_bounds__(256) k_arnoldi_column(const double2* __restrict__ red, long long red_stride, int j,
                                                        double2* __restrict__ H, long long h_rhs, int ldh,
                                                        const double* __restrict__ inv_beta,
                                                        const double2* __restrict__ dcoef,
                                                        const int* __restrict__ active) {
    const int r = blockIdx.y;
    const int l = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (active[r] == 0 || l > j) return;  // stopped (breakdown, zero source) or past the column
    arnoldi_column(red + r * red_stride, j, l, H + r * h_rhs, ldh, inv_beta[r], dcoef[r]);
}

// Second Gram-Schmidt pass of the last column: red[r] holds s at [0, k) and
// u^H u at entry uu_at, from a sweep over V_0..V_{k-1};
// H[:k][k-1] += s (the first pass of the column is in fp, if not in H),
// H[k][k-1] = ||u - V s||.
__global__ void __launch_bounds__(256) k_arnoldi_final(const double2* __restrict__ red, long long red_stride, int k,
                                                       int uu_at, double2* __restrict__ H, long long h_rhs, int ldh,
                                                       const double2* __restrict__ fp, long long fp_rhs,
                                                       const int* __restrict__ active) {
    __shared__ double sh[3 * 8];
    const int r = blockIdx.x, tid = threadIdx.x;
    if (active[r] == 0) return;
    const double2* rr = red + r * red_stride;
    double2* Hr = H + r * h_rhs;
    double ss = 0.0, z1 = 0.0, z2 = 0.0;
    for (int i = tid; i < k; i += blockDim.x) {
        const double2 si = rr[i];
        const double2 h = fp != nullptr ? fp[r * fp_rhs + i] : Hr[i + (long long)(k - 1) * ldh];
        Hr[i + (long long)(k - 1) * ldh] = make_double2(h.x + si.x, h.y + si.y);
        ss += si.x * si.x + si.y * si.y;
    }
    block_sum3(ss, z1, z2, sh);
    if (tid == 0) {
        const double b2 = rr[uu_at].x - ss;
        Hr[k + (long long)(k - 1) * ldh] = make_double2(b2 > 0.0 ? sqrt(b2) : 0.0, 0.0);
    }
}

__global__ void k_sign_scale(const double2* __restrict__ c, const double* __restrict__ sgn, int m, int nrhs,
                             double2* __restrict__ out) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= m * nrhs) return;
    const int i = idx % m;
    double2 v = c[idx];
    out[idx] = make_double2(sgn[i] * v.x, sgn[i] * v.y);
}

// ------------------------------------------------------- shared-basis dots
// Inner products against a complex64 basis shared by all right-hand sides
// (the LR projection L^+ x, the Schur projections S^H z of every Arnoldi
// step): partial[(r*nblk + b)*pstride + i] = sum over the units of chunk b
// of S_i^H z_r, i < m, r < nrhs. A block takes one chunk of units and stages
// it KD units at a time, every S_i and every z_r, in shared memory by
// asynchronous 16-byte copies (cp.async), two stages deep: the copies of
// tile t+1 are in flight while tile t is multiplied, so a block keeps
// (m + nrhs) KD 16-byte units in flight without registers. Stage layout
// vector-major with a row pitch of KD+1 units: the copies write consecutive
// units, and the threads of a quarter warp, reading 8 consecutive vectors
// at one unit, fall on 8 distinct 4-bank groups. Each thread accumulates a
// tile of 4 basis vectors x 2 right-hand sides. Where these tiles need half of
// the threads or fewer, groups of threads share a staged tile's units (30 vectors
// and 16 right-hand sides: 64 threads per group, 4 groups; with two of eight warps
// at work a sweep at 8^4 took 20.6 us, now 14.5). A sum is FP32 over one staged tile
// (2 KD complex terms) and FP64 across tiles, each sum in one thread. Each element
// of the basis is read from memory once per call, not once per right-hand side.
constexpr int KD = 32;
constexpr int KP = KD + 1;  // row pitch of a staged vector, in units

__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int n = valid ? 16 : 0;  // 0: nothing is read, the 16 bytes are zero-filled
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

__global__ void __launch_bounds__(BT) k_shared_dots(const float4* __restrict__ S, long long svec, int m,
                                                    const float4* __restrict__ Z, long long zstride, int nrhs,
                                                    long long nunits, long long chunk, int nblk,
                                                    double2* __restrict__ partial, int pstride,
                                                    const int* __restrict__ active) {
    extern __shared__ float4 sd_smem[];
    const int rows = m + nrhs;  // staged vectors: S_0 .. S_(m-1), then z_0 .. z_(nrhs-1)
    const size_t stage = (size_t)rows * KP;
    const int b = blockIdx.x, tid = threadIdx.x;
    const long long u0 = (long long)b * chunk;
    const long long u1 = min(u0 + chunk, nunits);
    const int itiles = (m + 3) / 4, rtiles = (nrhs + 1) / 2;
    const int W = itiles * rtiles, G = BT / W;  // threads per group, groups
    const int g = tid / W, wt = tid - g * W, ti = wt % itiles, tr = wt / itiles;
    const bool work = g < G;
    float2* fs = reinterpret_cast<float2*>(sd_smem + 2 * stage);  // [8][G][W]: the groups' sums of a tile
    double2 acc[8];  // the thread's sums tid, tid + BT, ... of 8 W
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[q] = make_double2(0.0, 0.0);
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    // copies of the tile at unit t0 into stage buffer st (zero beyond u1)
    auto issue = [&](long long t0, int st) {
        float4* dst = sd_smem + st * stage;
        for (int idx = tid; idx < rows * KD; idx += BT) {
            const int row = idx / KD, u = idx - row * KD;
            const bool valid = t0 + u < u1;
            const float4* src = row < m ? S + (size_t)row * svec : Z + (size_t)(row - m) * zstride;
            cp_async16(dst + (size_t)row * KP + u, valid ? src + t0 + u : S, valid);
        }
        cp_async_commit();
    };
    const long long ntile = (u1 - u0 + KD - 1) / KD;
    if (ntile > 0) issue(u0, 0);
    for (long long t = 0; t < ntile; ++t) {
        if (t + 1 < ntile) {
            issue(u0 + (t + 1) * KD, (int)((t + 1) & 1));
            cp_async_wait<1>();  // tile t has landed (tile t+1 may still be in flight)
        } else {
            cp_async_wait<0>();
        }
        __syncthreads();
        const float4* sS = sd_smem + (t & 1) * stage;
        const float4* sZ = sS + (size_t)m * KP;
        const int cnt = (int)min((long long)KD, u1 - (u0 + t * KD));
        if (work) {
            float a32[4][2][2];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int c = 0; c < 2; ++c) a32[a][c][0] = a32[a][c][1] = 0.f;
            for (int u = g; u < cnt; u += G) {
                float4 sv[4], zv[2];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int i = ti + q * itiles;
                    sv[q] = (i < m) ? sS[(size_t)i * KP + u] : zero;
                }
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int r = tr + q * rtiles;
                    zv[q] = (r < nrhs) ? sZ[(size_t)r * KP + u] : zero;
                }
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int c = 0; c < 2; ++c) {  // conj(s) z for the two complex numbers of the unit
                        float re = a32[a][c][0], im = a32[a][c][1];
                        re = fmaf(sv[a].x, zv[c].x, re);
                        re = fmaf(sv[a].y, zv[c].y, re);
                        re = fmaf(sv[a].z, zv[c].z, re);
                        re = fmaf(sv[a].w, zv[c].w, re);
                        im = fmaf(sv[a].x, zv[c].y, im);
                        im = fmaf(-sv[a].y, zv[c].x, im);
                        im = fmaf(sv[a].z, zv[c].w, im);
                        im = fmaf(-sv[a].w, zv[c].z, im);
                        a32[a][c][0] = re;
                        a32[a][c][1] = im;
                    }
            }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int c = 0; c < 2; ++c)
                    fs[((a * 2 + c) * G + g) * W + wt] = make_float2(a32[a][c][0], a32[a][c][1]);
        }
        // the sums are there; stage (t & 1) is refilled by the copies issued in the next iteration
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int o = tid + q * BT;
            if (o >= 8 * W) break;
            const float2* p = fs + (size_t)(o / W) * G * W + o % W;
            float2 x = p[0];
            for (int k = 1; k < G; ++k) {
                x.x += p[(size_t)k * W].x;
                x.y += p[(size_t)k * W].y;
            }
            acc[q].x += (double)x.x;
            acc[q].y += (double)x.y;
        }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int o = tid + q * BT;
        if (o >= 8 * W) break;
        const int w = o % W, a = o / W >> 1, c = o / W & 1;
        const int i = w % itiles + a * itiles, r = w / itiles + c * rtiles;
        if (i >= m || r >= nrhs) continue;
        if (active != nullptr && active[r] == 0) continue;
        partial[((size_t)r * nblk + b) * pstride + i] = acc[q];
    }
}

static size_t shared_dots_smem(int m, int nrhs) {
    const int W = (m + 3) / 4 * ((nrhs + 1) / 2);
    return 2 * (size_t)(m + nrhs) * KP * sizeof(float4) + (size_t)8 * (BT / W) * W * sizeof(float2);
}

// Blocks of the shared-basis dots: as many per SM as their two stages fit, at most 2
// (every block is one more partial sum to add); 0 when the tile does not fit (the
// register sweep k_gdots serves then).
int shared_dots_blocks(int m, int nrhs, long long nunits, int num_sms) {
    const int itiles = (m + 3) / 4, rtiles = (nrhs + 1) / 2;
    if (m < 1 || nrhs < 1 || (long long)itiles * rtiles > BT) return 0;
    const size_t smem = shared_dots_smem(m, nrhs);
    if (smem > 216 * 1024) return 0;
    const long long per_sm = std::max<long long>(1, std::min<long long>(2, (long long)(220 * 1024) / (long long)smem));
    long long want = per_sm * num_sms;
    want = std::min<long long>(want, std::max<long long>(1, nunits / KD));
    return (int)want;
}

cudaError_t launch_shared_dots(const void* S, long long svec, int m, const void* Z, long long zstride, int nrhs,
                               long long nunits, int nblk, void* partial, int pstride, const int* active,
                               cudaStream_t st) {
    const size_t smem = shared_dots_smem(m, nrhs);
    cudaError_t e = ensure_dyn_smem((const void*)k_shared_dots, 216 * 1024);
    if (e != cudaSuccess) return e;
    long long chunk = (nunits + nblk - 1) / nblk;
    chunk = ((chunk + KD - 1) / KD) * KD;
    k_shared_dots<<<nblk, BT, smem, st>>>((const float4*)S, svec, m, (const float4*)Z, zstride, nrhs, nunits, chunk,
                                         nblk, (double2*)partial, pstride, active);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ launch
BlasPlan blas_plan(long long nunits, int nrhs, int num_sms) {
    BlasPlan p;
    long long want = std::max<long long>(1, (8LL * num_sms + nrhs - 1) / nrhs);
    long long chunk = (nunits + want - 1) / want;
    const long long tile = (long long)BT * 8;  // one inner-product tile of 8 units per thread
    chunk = ((chunk + tile - 1) / tile) * tile;
    p.chunk = chunk;
    p.nblk = (int)((nunits + chunk - 1) / chunk);
    return p;
}

cudaError_t ensure_dyn_smem(const void* kernel, size_t bytes) {
    static std::mutex mu;
    static std::map<std::pair<const void*, int>, size_t> granted;  // (kernel, device) -> bytes
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    size_t& cur = granted[std::make_pair(kernel, dev)];
    if (bytes <= cur) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) cur = bytes;
    return e;
}

// the register sweeps keep their reduction buffers (up to 200 KB) in
// dynamic shared memory
static void set_smem_attrs() {
    const size_t big = 200 * 1024;
    ensure_dyn_smem((const void*)k_gdots<double, 16, 4>, big);
    ensure_dyn_smem((const void*)k_gdots<float, 16, 4>, big);
    ensure_dyn_smem((const void*)k_update<double, double, 2>, big);
    ensure_dyn_smem((const void*)k_update<float, float, 2>, big);
    ensure_dyn_smem((const void*)k_update<float, double, 2>, big);
}

int gdots_stride(int nw, int J) { return nw * J + 2; }

cudaError_t launch_gdots(int prec, const void* basis, long long basis_rhs_stride, long long vec_stride, int J,
                         const void* u, long long u_rhs_stride, long long nunits, const BlasPlan& plan, int nrhs,
                         void* partial, const int* active, cudaStream_t st) {
    set_smem_attrs();
    dim3 grid(nrhs, plan.nblk);  // right-hand side fastest: a shared basis is re-read from L2
    const size_t smem = (size_t)NWARP * gdots_stride(1, J) * sizeof(double2);
    if (smem > 200 * 1024) return cudaErrorInvalidValue;
    if (prec == PREC_F64)
        k_gdots<double, 16, 4><<<grid, BT, smem, st>>>((const double2*)basis, basis_rhs_stride, vec_stride, J,
                                                       (const double2*)u, u_rhs_stride, nunits, plan.chunk, plan.nblk,
                                                       (double2*)partial, active);
    else
        k_gdots<float, 16, 4><<<grid, BT, smem, st>>>((const float4*)basis, basis_rhs_stride, vec_stride, J,
                                                      (const float4*)u, u_rhs_stride, nunits, plan.chunk, plan.nblk,
                                                      (double2*)partial, active);
    return cudaGetLastError();
}

cudaError_t launch_arnoldi_step(const void* red, long long red_stride, int j, void* H, long long h_rhs, int ldh,
                                double* beta0, double* inv_beta, void* dcoef, double* hnorm2, int* active,
                                int* k_used, int nrhs, cudaStream_t st) {
    const StepOut o{(double2*)H, h_rhs, ldh, beta0, inv_beta, (double2*)dcoef, hnorm2, active, k_used};
    k_arnoldi_step<<<nrhs, 256, 0, st>>>((const double2*)red, red_stride, j, o);
    return cudaGetLastError();
}

cudaError_t launch_arnoldi_column(const void* red, long long red_stride, int j, void* H, long long h_rhs, int ldh,
                                  const double* inv_beta, const void* dcoef, const int* active, int nrhs,
                                  cudaStream_t st) {
    const dim3 grid((j + 1 + 7) / 8, nrhs);
    k_arnoldi_column<<<grid, 256, 0, st>>>((const double2*)red, red_stride, j, (double2*)H, h_rhs, ldh, inv_beta,
                                           (const double2*)dcoef, active);
    return cudaGetLastError();
}

cudaError_t launch_arnoldi_final(const void* red, long long red_stride, int k, int uu_at, void* H, long long h_rhs,
                                 int ldh, const int* active, int nrhs, cudaStream_t st, const void* fp,
                                 long long fp_rhs) {
    k_arnoldi_final<<<nrhs, 256, 0, st>>>((const double2*)red, red_stride, k, uu_at, (double2*)H, h_rhs, ldh,
                                          (const double2*)fp, fp_rhs, active);
    return cudaGetLastError();
}

cudaError_t launch_update(int prec_v, int prec_out, const void* basis, long long basis_rhs_stride,
                          long long vec_stride, int J, const void* coef, long long coef_stride,
                          double alpha, const void* in, long long in_rhs_stride, void* out, long long out_rhs_stride,
                          long long nunits_v, const BlasPlan& plan, int nrhs, double* norm_partial,
                          const int* active, cudaStream_t st) {
    set_smem_attrs();
    dim3 grid(nrhs, plan.nblk);  // right-hand side fastest: a shared basis is re-read from L2
    size_t smem = (size_t)std::max(J, 1) * sizeof(double2);
    if (prec_v == PREC_F64 && prec_out == PREC_F64) {
        k_update<double, double, 2><<<grid, BT, smem, st>>>(
            (const double2*)basis, basis_rhs_stride, vec_stride, J, (const double2*)coef, coef_stride, alpha,
            (const cd*)in, in_rhs_stride, (cd*)out, out_rhs_stride, nunits_v, plan.chunk, plan.nblk, norm_partial,
            active);
    } else if (prec_v == PREC_F32 && prec_out == PREC_F32) {
        k_update<float, float, 2><<<grid, BT, smem, st>>>(
            (const float4*)basis, basis_rhs_stride, vec_stride, J, (const double2*)coef, coef_stride, alpha,
            (const cf*)in, in_rhs_stride, (cf*)out, out_rhs_stride, nunits_v, plan.chunk, plan.nblk, norm_partial,
            active);
    } else if (prec_v == PREC_F32 && prec_out == PREC_F64) {
        k_update<float, double, 2><<<grid, BT, smem, st>>>(
            (const float4*)basis, basis_rhs_stride, vec_stride, J, (const double2*)coef, coef_stride, alpha,
            (const cd*)in, in_rhs_stride, (cd*)out, out_rhs_stride, nunits_v, plan.chunk, plan.nblk, norm_partial,
            active);
    } else {
        return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// Shared-basis combination for all right-hand sides (the deflation part of
// Sec. 5.3: x - R c and R sgn(Lambda) c, with R the complex64 copy of the
// deflation basis): out_r = [in_r] + alpha * sum_{i < m} R_i c_{r,i}.
// A block takes a tile of BT*E units and a group of SG right-hand sides;
// blocks are numbered with the group fastest, so the SG-groups of a tile
// run together and R is read from DRAM once and from L2 by the other
// groups. The vector loop is unrolled by 4 (8 loads in flight per thread);
// products are FP32, and for a complex128 output the FP32 partial sums are
// added into FP64 accumulators every 16 vectors.
// E = 2 where that makes four blocks per SM, else 1: at 8^4 with 16
// right-hand sides 192 blocks of two units took 15.8 us, 384 of one take 11.4.
constexpr int SG = 4;
template <typename RO, int E>
__global__ void __launch_bounds__(BT) k_shared_combine(const float4* __restrict__ R, long long vec_stride, int m,
                                                       const double2* __restrict__ coef, long long coef_stride,
                                                       double alpha, const cplx<RO>* in, long long in_rhs_stride,
                                                       cplx<RO>* out, long long out_rhs_stride, long long nunits,
                                                       int nrhs, int ngroups) {
    extern __shared__ double2 smc[];
    cf* sc = reinterpret_cast<cf*>(smc);  // [SG][m] alpha * c
    const int grp = blockIdx.x % ngroups;
    const long long tile = blockIdx.x / ngroups;
    const int r0 = grp * SG;
    const int nr = min(SG, nrhs - r0);
    const int tid = threadIdx.x;
    for (int i = tid; i < SG * m; i += BT) {
        const int q = i / m, v = i - q * m;
        const double2 c = q < nr ? coef[(long long)(r0 + q) * coef_stride + v] : make_double2(0.0, 0.0);
        sc[i] = {float(alpha * c.x), float(alpha * c.y)};
    }
    __syncthreads();
    long long u[E];
    bool ok[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        u[e] = tile * (E * BT) + tid + (long long)BT * e;
        ok[e] = u[e] < nunits;
    }
    cplx<RO> o[SG][E][2];
    cf acc[SG][E][2];
#pragma unroll
    for (int q = 0; q < SG; ++q)
#pragma unroll
        for (int e = 0; e < E; ++e)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                o[q][e][c] = {RO(0), RO(0)};
                acc[q][e][c] = {0.f, 0.f};
            }
    auto flush = [&]() {
#pragma unroll
        for (int q = 0; q < SG; ++q)
#pragma unroll
            for (int e = 0; e < E; ++e)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    o[q][e][c].re += RO(acc[q][e][c].re);
                    o[q][e][c].im += RO(acc[q][e][c].im);
                    acc[q][e][c] = {0.f, 0.f};
                }
    };
    int i = 0;
    for (; i + 4 <= m; i += 4) {
        float4 v[4][E];
#pragma unroll
        for (int d = 0; d < 4; ++d)
#pragma unroll
            for (int e = 0; e < E; ++e)
                v[d][e] = ok[e] ? __ldg(R + (long long)(i + d) * vec_stride + u[e]) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int d = 0; d < 4; ++d)
#pragma unroll
            for (int e = 0; e < E; ++e) {
                cf vc[2];
                Unit<float>::split(v[d][e], vc);
#pragma unroll
                for (int q = 0; q < SG; ++q) {
                    const cf cq = sc[q * m + i + d];
#pragma unroll
                    for (int c = 0; c < 2; ++c) cfma(acc[q][e][c], vc[c], cq);
                }
            }
        if (sizeof(RO) > 4 && ((i + 4) & 15) == 0) flush();
    }
    for (; i < m; ++i) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const float4 v = ok[e] ? __ldg(R + (long long)i * vec_stride + u[e]) : make_float4(0.f, 0.f, 0.f, 0.f);
            cf vc[2];
            Unit<float>::split(v, vc);
#pragma unroll
            for (int q = 0; q < SG; ++q) {
                const cf cq = sc[q * m + i];
#pragma unroll
                for (int c = 0; c < 2; ++c) cfma(acc[q][e][c], vc[c], cq);
            }
        }
    }
    flush();
#pragma unroll
    for (int q = 0; q < SG; ++q) {
        if (q >= nr) break;
        const int r = r0 + q;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (!ok[e]) continue;
            cplx<RO> res[2];
            if (in != nullptr) OutIO<RO, 2>::load(in + (long long)r * in_rhs_stride, u[e], res);
            else res[0] = res[1] = {RO(0), RO(0)};
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                res[c].re += o[q][e][c].re;
                res[c].im += o[q][e][c].im;
            }
            OutIO<RO, 2>::store(out + (long long)r * out_rhs_stride, u[e], res);
        }
    }
}

cudaError_t launch_shared_combine(int prec_out, const void* R, long long vec_stride, int m, const void* coef,
                                  long long coef_stride, double alpha, const void* in, long long in_rhs_stride,
                                  void* out, long long out_rhs_stride, long long nunits, int nrhs, cudaStream_t st) {
    if (m < 1 || nrhs < 1) return cudaErrorInvalidValue;
    const int ngroups = (nrhs + SG - 1) / SG;
    const size_t smem = (size_t)SG * m * sizeof(cf);
    if (smem > 48 * 1024) return cudaErrorInvalidValue;
    auto blocks = [&](int E) { return (nunits + E * BT - 1) / (E * BT) * ngroups; };
    const int E = blocks(2) >= 4LL * device_sms() ? 2 : 1;
    if (blocks(E) > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    auto go = [&](auto kernel, const auto* x, auto* y) {
        kernel<<<(unsigned)blocks(E), BT, smem, st>>>((const float4*)R, vec_stride, m, (const double2*)coef, coef_stride,
                                                      alpha, x, in_rhs_stride, y, out_rhs_stride, nunits, nrhs, ngroups);
    };
    if (prec_out == PREC_F64)
        go(E == 2 ? k_shared_combine<double, 2> : k_shared_combine<double, 1>, (const cd*)in, (cd*)out);
    else
        go(E == 2 ? k_shared_combine<float, 2> : k_shared_combine<float, 1>, (const cf*)in, (cf*)out);
    return cudaGetLastError();
}

cudaError_t launch_reduce(const void* partial, int nblk, int pstride, int J, int nrhs, void* out,
                          long long out_stride, bool accumulate, const int* active, cudaStream_t st) {
    if (J <= 0) return cudaSuccess;
    const int n = J * nrhs;
    if (nblk >= 16) {  // below that a sum is one batch of loads
        k_reduce_wide<<<(n + RW - 1) / RW, 256, 0, st>>>((const double2*)partial, nblk, pstride, J, nrhs, (double2*)out,
                                                     out_stride, accumulate ? 1 : 0, active);
        return cudaGetLastError();
    }
    k_reduce<<<(n + 127) / 128, 128, 0, st>>>((const double2*)partial, nblk, pstride, J, nrhs, (double2*)out,
                                              out_stride, accumulate ? 1 : 0, active);
    return cudaGetLastError();
}

cudaError_t launch_sign_scale(const void* c, const double* sgn, int m, int nrhs, void* out, cudaStream_t st) {
    const int n = m * nrhs;
    if (n == 0) return cudaSuccess;
    k_sign_scale<<<(n + 127) / 128, 128, 0, st>>>((const double2*)c, sgn, m, nrhs, (double2*)out);
    return cudaGetLastError();
}

}  // namespace ovs
