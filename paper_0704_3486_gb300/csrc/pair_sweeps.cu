// Two Arnoldi steps per pass over the complex64 basis.
//
// The delayed-reorthogonalisation step (arnoldi_dev.cuh) reads the basis twice
// per step and is bound by that. Here a block step appends two vectors with the
// same two reads: from the first-pass residuals u1, u2 of the last block the
// stencil gives
//   x1 = A u2 - gamma u1,   x2 = A x1,
// one sweep gives the inner products of all four with V (second pass of u1, u2
// and first pass of x1, x2) and their Gram matrix, and one update writes
//   v_J = (u1 - V s1)/b1,   v_{J+1} = (u2 - V s2 - r12 v_J)/r22,
//   u1' = (x1 - V t1 - a1 v_J - c1 v_{J+1})/r22,
//   u2' = (x2 - V t2 - a2 v_J - c2 v_{J+1})/r22 - d u1'.
// With v_J, v_{J+1} the spans and the orthogonality are those of CGS2: every
// vector is projected against all earlier ones twice. The columns of H follow
// from the coefficients: A u2 = x1 + gamma u1 with u2 = V s2 + r12 v_J + r22
// v_{J+1} gives column J+1, and A x1 = x2 with x1 = r22 (V e + b1' v_J' + ...)
// gives column J of the next block (Eq. Arnoldi, solved for the one unknown
// column; A V_j is known from H).
//
// gamma = (||u2'||/||u1'||)^2 is the last subdiagonal squared, so x1 is close
// to orthogonal to u1, as in the three-term recurrence of a Hermitian operator
// (H_w(mu) is Hermitian at mu = 0): without it x2 loses digits to components
// along known vectors (in exact arithmetic any gamma gives the same V and H). The
// first block has no last subdiagonal: its gamma is the projection itself, for one
// more stencil and one more sweep over three vectors. With 0 there the second block's
// first column had twice the rounding of the others, where the weights are largest.
// Where a block is nevertheless badly conditioned (x1 loses more than half of
// its norm to V, or u2 most of it: a nearly invariant Krylov space), that
// right-hand side leaves with what is sound, one or two vectors and the
// residual u1, and takes single steps from there (pair_steps in api.cu).
//
// Measured, single steps and blocks: 12^4, 16 right-hand sides, k = 250: 323 ->
// 194 ms; 16^3 x 32, 8 right-hand sides, k = 200: 625 -> 377 ms (inner products
// 5.6 TB/s, update 6.7 TB/s); mean error against FP64 on the same sources at 12^4,
// k = 100: 1.28e-7 -> 1.23e-7 (1.37e-7 with gamma = 0 in the first block and the new
// vectors put together in five roundings).
#include <cuda_runtime.h>

#include <algorithm>

#include "arnoldi_dev.cuh"
#include "common.cuh"
#include "kernels.h"
#include "tma_dev.cuh"

namespace ovs {

namespace {

constexpr int PC = 1024;           // units per work item of the inner products, at most
constexpr int PNT = PC / DU;       // tiles of DU units
constexpr int PTHREADS = TB + 64;  // consumer warps, a producer and an accumulator warp
constexpr int NGRAM = 10;          // pairs p <= q of the four vectors
constexpr double kSlowRatio = 0.25;   // ||u1'||^2 / ||x1||^2 below this: single steps
constexpr double kNoiseRatio = 1e-8;  // ||u1'||^2 / ||gamma u1||^2 below this: x1 is half rounding, single steps
constexpr double kHalfRatio = 0.0625;  // ||u2 - V s2 - r12 v_J||^2 / ||u2||^2 below this: one vector only

__device__ __forceinline__ int gram_at(int p, int q) { return p * 4 - p * (p - 1) / 2 + (q - p); }

// warp sums of 64 values: lane l ends with values 2l and 2l + 1 in v[0], v[1]
template <int CUR, int O>
__device__ __forceinline__ void pstep(float (&v)[64], bool upper) {
#pragma unroll
    for (int i = 0; i < CUR / 2; ++i) {
        const float send = upper ? v[i] : v[i + CUR / 2];
        const float keep = upper ? v[i + CUR / 2] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
    }
}
// The same over 32 values, of which lane l ends with value l, with the rounding errors
// of the additions (Knuth's two-sum) beside the sums: v[i] + v[32 + i] is the warp's sum
// as FP64 would have it.
template <int CUR, int O>
__device__ __forceinline__ void pstep2(float (&v)[64], bool upper) {
#pragma unroll
    for (int i = 0; i < CUR / 2; ++i) {
        const float send = upper ? v[i] : v[i + CUR / 2], keep = upper ? v[i + CUR / 2] : v[i];
        const float got = __shfl_xor_sync(0xffffffffu, send, O);
        float low = 0.f;
        if (CUR < 32) {
            const float slow = upper ? v[32 + i] : v[32 + i + CUR / 2], klow = upper ? v[32 + i + CUR / 2] : v[32 + i];
            low = klow + __shfl_xor_sync(0xffffffffu, slow, O);
        }
        const float sum = keep + got, t = sum - keep;
        v[i] = sum;
        v[32 + i] = low + ((keep - (sum - t)) + (got - t));
    }
}
// named barriers over the consumers and the accumulator warp
constexpr int PSYNC = TB + 32;
__device__ __forceinline__ void named_sync(int id) { asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(PSYNC) : "memory"); }
__device__ __forceinline__ void named_arrive(int id) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(PSYNC) : "memory");
}
constexpr int kBarSeg = 1, kBarFull = 2, kBarFree = 4;  // + parity of the group

}  // namespace

// Inner products of V_0 .. V_{J-1} with four vectors w_p (u1, u2, x1, x2) and
// their Gram matrix: partial[r][slot][4J + 10] = V_i^H w_p at p J + i, then
// w_p^H w_q, p <= q. Persistent and warp-specialised like k_gdots2_ws, with
// work items of at most 1024 units (a thread holds 4 units of each vector) and a
// tenth warp that adds the eight consumer warps' sums of a group in FP64 into
// the block's accumulators. That is 32 operations of the FP64 pipe at 16 clocks
// each per group of 8 vectors; done by two of the consumer warps behind a
// barrier, as in k_gdots2_ws, it held all of them up twice as often as there
// and the sweep ran at 5.1 TB/s. The hand-over is a double buffer with named
// barriers on which the consumers only arrive. NS stages: 3, or 2 where the
// block's 4J + 10 accumulators leave no room.
//
// A wait that gives up raises `abort`; every warp then goes through its
// remaining groups without waiting for copies or computing, so that all named
// barriers stay paired, and the producer lets its copies land.
template <int NS>
__global__ void __launch_bounds__(PTHREADS, 1)
    k_pair_dots(const float4* __restrict__ basis, long long basis_rhs_stride, long long vec_stride, int J,
                const float4* __restrict__ w0, const float4* __restrict__ w1, const float4* __restrict__ w2,
                const float4* __restrict__ w3, long long nunits, int cu, int nrhs, int nslot,
                double2* __restrict__ partial, const int* __restrict__ active, int* __restrict__ err) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t full[NS];
    __shared__ __align__(8) uint64_t empty[NS];
    __shared__ float2 scratch[2][TW][32];
    __shared__ double gsum[TW][32];  // (component, pair) at 2 pair + component
    __shared__ int abort_flag;
    double* acc = reinterpret_cast<double*>(smem + NS * kDStage);  // [4J + 10][2]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int G = gridDim.x, q = blockIdx.x;
    const int S = 4 * J + NGRAM;
    const long long cpr = (nunits + cu - 1) / cu;
    const int nt = (cu + DU - 1) / DU;  // tiles per item
    const long long T = cpr * nrhs;
    const long long lo = range_lo(q, T, G), hi = range_lo(q + 1, T, G);
    const int ngroups = (J + TG - 1) / TG;
    volatile int* abort = &abort_flag;
    if (tid == 0) {
        for (int k = 0; k < NS; ++k) {
            mbar_init(&full[k], 1);
            mbar_init(&empty[k], TW);
        }
        abort_flag = 0;
        mbar_fence_init();
    }
    __syncthreads();

    if (warp == TW) {  // ---- producer warp: one lane issues every stage
        if (lane != 0 || ngroups == 0) return;
        int n = 0;
        bool ok = true;
        for (long long it = lo; it < hi && ok; ++it) {
            const long long r = it / cpr, c = it - r * cpr;
            if (active[r] == 0) continue;
            const long long u0 = c * cu;
            const int len = (int)min((long long)cu, nunits - u0);
            const float4* Vr = basis + r * basis_rhs_stride + u0;
            for (int g = 0; g < ngroups && ok; ++g) {
                const int nv = min(TG, J - g * TG);
                for (int t = 0; t < nt; ++t) {
                    const int s = n % NS;
                    if (n >= NS) {
                        if (!mbar_wait_or_abort(&empty[s], (uint32_t)((n / NS - 1) & 1), abort)) {
                            ok = false;
                            break;
                        }
                        fence_proxy_async_smem();
                    }
                    const int units = min(DU, len - t * DU);
                    if (units <= 0) {  // tile beyond a short item: complete the phase without bytes
                        mbar_expect_tx(&full[s], 0);
                    } else {
                        const uint32_t bytes = (uint32_t)units * 16u;
                        unsigned char* dst = smem + (size_t)s * kDStage;
                        mbar_expect_tx(&full[s], bytes * nv);
                        for (int v = 0; v < nv; ++v)
                            bulk_load(dst + (size_t)v * DU * 16, Vr + (long long)(g * TG + v) * vec_stride + t * DU,
                                      bytes, &full[s]);
                    }
                    ++n;
                }
            }
        }
        // the shared memory must outlive every copy (see k_gdots2_ws)
        for (int k = max(0, n - NS); k < n && ok; ++k)
            ok = mbar_wait_or_abort(&empty[k % NS], (uint32_t)((k / NS) & 1), abort);
        if (!ok) {
            atomicExch(err, OVS_ETIMEOUT_CODE);
            abort_flag = 1;
            for (int k = max(0, n - NS); k < n; ++k) mbar_wait_bounded(&full[k % NS], (uint32_t)((k / NS) & 1));
        }
        return;
    }

    int total = 0;  // groups of this block
    for (long long it = lo; it < hi; ++it)
        if (active[it / cpr] != 0) total += ngroups;

    if (warp == TW + 1) {  // ---- accumulator warp
        for (long long r = 0; r < nrhs; ++r) {  // unused slots of the right-hand sides that start here
            if (owner_of(r * cpr, T, G) != q) continue;
            const int used = owner_of((r + 1) * cpr - 1, T, G) - q + 1;
            double* base = reinterpret_cast<double*>(partial + ((size_t)r * nslot) * S);
            for (long long i = (long long)used * 2 * S + lane; i < (long long)nslot * 2 * S; i += 32) base[i] = 0.0;
        }
        long long seg_r = -1;
        int gg = 0;
        auto flush = [&](long long r) {
            named_sync(kBarSeg);  // the consumers' Gram sums are complete
            if (lane < 2 * NGRAM) {
                double s = 0.0;
                for (int w = 0; w < TW; ++w) s += gsum[w][lane];
                acc[8 * J + lane] = s;
            }
            named_sync(kBarSeg);  // they may be overwritten
            __syncwarp();
            const int slot = q - owner_of(r * cpr, T, G);
            double* out = reinterpret_cast<double*>(partial + ((size_t)r * nslot + slot) * S);
            for (int i = lane; i < 2 * S; i += 32) out[i] = acc[i];
            __syncwarp();
        };
        for (long long it = lo; it < hi; ++it) {
            const long long r = it / cpr;
            if (active[r] == 0) continue;
            if (r != seg_r) {
                if (seg_r >= 0) flush(seg_r);
                for (int i = lane; i < 2 * S; i += 32) acc[i] = 0.0;
                __syncwarp();
                seg_r = r;
            }
            for (int g = 0; g < ngroups; ++g, ++gg) {
                named_sync(kBarFull + (gg & 1));
                float2 p[TW];
#pragma unroll
                for (int w = 0; w < TW; ++w) p[w] = scratch[gg & 1][w][lane];
                if (gg + 2 < total) named_arrive(kBarFree + (gg & 1));
                double sx = 0.0, sy = 0.0;
#pragma unroll
                for (int w = 0; w < TW; ++w) {
                    sx += (double)p[w].x;
                    sy += (double)p[w].y;
                }
                const int gi = lane >> 2, k = lane & 3;  // item of the lane: vector gi of the group with w_k
                if (gi < J - g * TG) {
                    double* a = acc + (size_t)(k * J + g * TG + gi) * 2;
                    a[0] += sx;
                    a[1] += sy;
                }
            }
        }
        if (seg_r >= 0) flush(seg_r);
        return;
    }

    // ---- consumer warps
    int n = 0, gg = 0;
    long long seg_r = -1;
    bool bad = false;
    gsum[warp][lane] = 0.0;
    for (long long it = lo; it < hi; ++it) {
        const long long r = it / cpr, c = it - r * cpr;
        if (active[r] == 0) continue;
        if (r != seg_r) {
            if (seg_r >= 0) {
                named_sync(kBarSeg);
                named_sync(kBarSeg);
                gsum[warp][lane] = 0.0;
            }
            seg_r = r;
        }
        const long long u0 = c * cu;
        const int len = (int)min((long long)cu, nunits - u0);
        float4 w[4][PNT * DE];
        {
            const float4* src[4] = {w0 + r * nunits + u0, w1 + r * nunits + u0, w2 + r * nunits + u0,
                                    w3 + r * nunits + u0};
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int k = 0; k < PNT * DE; ++k) {
                    const int at = k * TB + tid;
                    w[p][k] = at < len ? __ldg(src[p] + at) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
        }
        {  // Gram matrix: FP32 over the 8 terms of a lane, FP64 beyond (over the lanes: two FP32)
            float v[64];
#pragma unroll
            for (int k = 2 * NGRAM; k < 32; ++k) v[k] = 0.f;
            int at = 0;
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int s = p; s < 4; ++s) {
                    cf a = {0.f, 0.f};
#pragma unroll
                    for (int k = 0; k < PNT * DE; ++k) {
                        cf x[2], y[2];
                        Unit<float>::split(w[p][k], x);
                        Unit<float>::split(w[s][k], y);
                        cfmac(a, x[0], y[0]);
                        cfmac(a, x[1], y[1]);
                    }
                    v[2 * at] = a.re;
                    v[2 * at + 1] = s != p ? a.im : 0.f;
                    ++at;
                }
            pstep2<32, 16>(v, (lane & 16) != 0);
            pstep2<16, 8>(v, (lane & 8) != 0);
            pstep2<8, 4>(v, (lane & 4) != 0);
            pstep2<4, 2>(v, (lane & 2) != 0);
            pstep2<2, 1>(v, (lane & 1) != 0);
            gsum[warp][lane] += (double)v[0] + (double)v[32];  // lane l: value l
        }
        for (int g = 0; g < ngroups; ++g) {
            float v[64];  // (vector gi, which p, component) at (gi 4 + p) 2 + comp
#pragma unroll
            for (int k = 0; k < 64; ++k) v[k] = 0.f;
            const int nv = min(TG, J - g * TG);
#pragma unroll
            for (int t = 0; t < PNT; ++t) {
                if (t >= nt) break;
                const int s = n % NS;
                const bool got = bad || mbar_wait_or_abort(&full[s], (uint32_t)((n / NS) & 1), abort);
                if (!__all_sync(0xffffffffu, got)) {  // keep `bad` uniform over the warp
                    if (lane == 0) {
                        atomicExch(err, OVS_ETIMEOUT_CODE);
                        abort_flag = 1;
                    }
                    bad = true;
                }
                if (!bad) {
                    const float4* st4 = reinterpret_cast<const float4*>(smem + (size_t)s * kDStage);
#pragma unroll
                    for (int e = 0; e < DE; ++e) {
                        const int k = t * DE + e;
                        if (k * TB + tid < len) {
#pragma unroll
                            for (int gi = 0; gi < TG; ++gi) {
                                if (gi < nv) {
                                    cf vc[2];
                                    Unit<float>::split(st4[gi * DU + e * TB + tid], vc);
#pragma unroll
                                    for (int p = 0; p < 4; ++p) {
                                        cf y[2];
                                        Unit<float>::split(w[p][k], y);
                                        cf a = {v[(gi * 4 + p) * 2], v[(gi * 4 + p) * 2 + 1]};
                                        cfmac(a, vc[0], y[0]);
                                        cfmac(a, vc[1], y[1]);
                                        v[(gi * 4 + p) * 2] = a.re;
                                        v[(gi * 4 + p) * 2 + 1] = a.im;
                                    }
                                }
                            }
                        }
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&empty[s]);
                }
                ++n;
            }
            // warp sums: lane l keeps both components of item l
            pstep<64, 16>(v, (lane & 16) != 0);
            pstep<32, 8>(v, (lane & 8) != 0);
            pstep<16, 4>(v, (lane & 4) != 0);
            pstep<8, 2>(v, (lane & 2) != 0);
            pstep<4, 1>(v, (lane & 1) != 0);
            if (gg >= 2) named_sync(kBarFree + (gg & 1));  // the accumulator has read group gg - 2
            scratch[gg & 1][warp][lane] = make_float2(v[0], v[1]);
            named_arrive(kBarFull + (gg & 1));
            ++gg;
        }
    }
    if (seg_r >= 0) {
        named_sync(kBarSeg);
        named_sync(kBarSeg);
    }
}

// gamma of the first block: Re <u1, A u2> / <u1, u1>, from the Gram matrix of (u1, u2,
// A u2, ...), which leaves x1 shortest. 0 where there is none (a zero or non-finite
// source).
__global__ void k_pair_start(const double2* __restrict__ red, long long red_stride, PairState* __restrict__ ps,
                             int nrhs) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= nrhs) return;
    const double2* g = red + r * red_stride;
    const double q = g[gram_at(0, 2)].x / g[gram_at(0, 0)].x;
    ps[r].gamma_next = isfinite(q) ? q : 0.0;
}

// Scalars of a block step (one block per right-hand side), from the reduced
// sums red[r] of k_pair_dots. See the head of this file; the breakdown rule is
// that of arnoldi_step. mode[r]: what the update writes (0 nothing).
__global__ void __launch_bounds__(256) k_pair_step(const double2* __restrict__ red, long long red_stride, int J,
                                                   int more, StepOut o, PairState* __restrict__ ps,
                                                   int* __restrict__ pact, int* __restrict__ mode,
                                                   int* __restrict__ jstart, int never) {
    __shared__ double sh[8][2 * NGRAM];
    __shared__ double sh3[24];
    const int r = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (pact[r] == 0) {
        if (tid == 0) mode[r] = 0;
        return;
    }
    const double2* rr = red + r * red_stride;
    double2* Hr = o.H + r * o.h_rhs;
    const int ldh = o.ldh;
    // G - C^H C
    double m[2 * NGRAM];
#pragma unroll
    for (int k = 0; k < 2 * NGRAM; ++k) m[k] = 0.0;
    for (int i = tid; i < J; i += 256) {
        double2 c[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) c[p] = rr[p * J + i];
        int at = 0;
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int s = p; s < 4; ++s) {
                m[2 * at] += c[p].x * c[s].x + c[p].y * c[s].y;
                m[2 * at + 1] += c[p].x * c[s].y - c[p].y * c[s].x;
                ++at;
            }
    }
#pragma unroll
    for (int k = 0; k < 2 * NGRAM; ++k) {
        const double s = warp_sum(m[k]);
        if (lane == 0) sh[warp][k] = s;
    }
    __syncthreads();
    if (tid < 2 * NGRAM) {
        double s = 0.0;
        for (int w = 0; w < 8; ++w) s += sh[w][tid];
        const double2 g = rr[4 * J + (tid >> 1)];
        sh[0][tid] = ((tid & 1) ? g.y : g.x) - s;
    }
    __syncthreads();
    auto gt = [&](int p, int q) { return cd{sh[0][2 * gram_at(p, q)], sh[0][2 * gram_at(p, q) + 1]}; };
    const double b2 = gt(0, 0).re;
    // a NaN (from a non-finite source) stays NaN, so that it is reported
    const double b1 = (b2 > 0.0 || isnan(b2)) ? sqrt(b2) : 0.0;
    if (J == 0) {
        if (tid == 0) {
            o.beta0[r] = b1;
            o.hnorm2[r] = 0.0;
        }
        if (!(b1 > 0.0) || !isfinite(b1)) {
            if (tid == 0) {
                o.active[r] = 0;
                pact[r] = 0;
                mode[r] = 0;
                o.k_used[r] = 0;
                jstart[r] = never;
            }
            return;
        }
    } else {  // column J-1: second pass; its norm and that of column J-2 join ||H||_F
        double c2 = 0.0, z1 = 0.0, z2 = 0.0;
        for (int i = tid; i < J; i += 256) {
            double2 h = Hr[i + (long long)(J - 1) * ldh];
            const double2 s = rr[i];
            h = make_double2(h.x + s.x, h.y + s.y);
            Hr[i + (long long)(J - 1) * ldh] = h;
            const double2 h2 = Hr[i + (long long)(J - 2) * ldh];
            c2 += h.x * h.x + h.y * h.y + h2.x * h2.x + h2.y * h2.y;
        }
        block_sum3(c2, z1, z2, sh3);
        const double hn2 = o.hnorm2[r] + c2 + b1 * b1;
        const bool brk = !(b1 > kBreakdownTol * sqrt(hn2)) || !isfinite(b1);
        if (tid == 0) {
            o.hnorm2[r] = hn2;
            Hr[J + (long long)(J - 1) * ldh] = make_double2(brk ? 0.0 : b1, 0.0);
            if (brk) {
                o.active[r] = 0;
                pact[r] = 0;
                mode[r] = 0;
                o.k_used[r] = J;
                jstart[r] = never;
            }
        }
        if (brk) return;
    }
    if (tid != 0) return;
    PairState s = ps[r];
    s.gamma_now = s.gamma_next;
    s.d_now = J == 0 ? make_double2(0.0, 0.0) : s.d_next;
    const double ib = 1.0 / b1;
    const cd r12 = gt(0, 1) * ib;
    const double g11 = rr[4 * J + gram_at(1, 1)].x;
    const double r22sq = gt(1, 1).re - (r12.re * r12.re + r12.im * r12.im);
    s.b1 = b1;
    s.r12 = make_double2(r12.re, r12.im);
    if (!(r22sq > kHalfRatio * g11)) {  // one vector; its residual goes on in single steps
        s.r22 = 0.0;
        mode[r] = 2;
        pact[r] = 0;
        jstart[r] = J + 1;
        o.k_used[r] = J + 1;
        o.inv_beta[r] = ib;
        ps[r] = s;
        return;
    }
    const double r22 = sqrt(r22sq), i2 = 1.0 / r22;
    s.r22 = r22;
    auto conjmul = [](cd a, cd b) { return cd{a.re * b.re + a.im * b.im, a.re * b.im - a.im * b.re}; };
    const cd a1 = gt(0, 2) * ib, a2 = gt(0, 3) * ib;
    const cd c1 = (gt(1, 2) - conjmul(r12, a1)) * i2, c2v = (gt(1, 3) - conjmul(r12, a2)) * i2;
    const double n1 = gt(2, 2).re - (a1.re * a1.re + a1.im * a1.im) - (c1.re * c1.re + c1.im * c1.im);
    cd d = (gt(2, 3) - conjmul(a1, a2) - conjmul(c1, c2v)) * (1.0 / n1);
    const double n2 = gt(3, 3).re - (a2.re * a2.re + a2.im * a2.im) - (c2v.re * c2v.re + c2v.im * c2v.im) -
                      (d.re * d.re + d.im * d.im) * n1;
    s.a1 = make_double2(a1.re, a1.im);
    s.a2 = make_double2(a2.re, a2.im);
    s.c1 = make_double2(c1.re, c1.im);
    s.c2 = make_double2(c2v.re, c2v.im);
    const bool sound = more && n1 > kSlowRatio * rr[4 * J + gram_at(2, 2)].x &&
                       n1 > kNoiseRatio * (s.gamma_now * b1) * (s.gamma_now * b1) && n2 > 0.0;
    s.d_next = sound ? make_double2(d.re, d.im) : make_double2(0.0, 0.0);
    s.gamma_next = sound ? n2 / n1 : 0.0;
    ps[r] = s;
    mode[r] = 1;
    o.k_used[r] = J + 2;
    jstart[r] = J + 2;
    if (!sound) pact[r] = 0;  // single steps from J + 2 on (none, if that is k)
}

// Columns J and J + 1 (first pass) of H, and the coefficients that the next
// block needs: one warp per row l <= J + 1. ec: [2][kmax] per right-hand side and
// parity (x1/r22 and x2/r22 in the basis); `ecn` is written for the next block.
__global__ void __launch_bounds__(256) k_pair_column(const double2* __restrict__ red, long long red_stride, int J,
                                                     double2* __restrict__ H, long long h_rhs, int ldh,
                                                     const PairState* __restrict__ ps, const int* __restrict__ mode,
                                                     const double2* __restrict__ ec, double2* __restrict__ ecn,
                                                     int kmax) {
    const int r = blockIdx.y, lane = threadIdx.x & 31;
    const int l = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int md = mode[r];
    if (md == 0 || l > J + 1 || (md == 2 && l > J)) return;
    const double2* rr = red + r * red_stride;
    const double2* e1 = ec + (size_t)r * 2 * kmax;
    const double2* e2 = e1 + kmax;
    double2* Hr = H + r * h_rhs;
    const PairState s = ps[r];
    double g1r = 0.0, g1i = 0.0, g2r = 0.0, g2i = 0.0;
    for (int i = (l > 0 ? l - 1 : 0) + lane; i < J; i += 32) {
        const double2 h = Hr[l + (long long)i * ldh];
        const double2 s1 = rr[i], s2 = rr[J + i], e = e1[i];
        const double ex = e.x + s1.x, ey = e.y + s1.y;
        g1r += h.x * ex - h.y * ey;
        g1i += h.x * ey + h.y * ex;
        g2r += h.x * s2.x - h.y * s2.y;
        g2i += h.x * s2.y + h.y * s2.x;
    }
    g1r = warp_sum(g1r);
    g1i = warp_sum(g1i);
    g2r = warp_sum(g2r);
    g2i = warp_sum(g2i);
    if (lane != 0) return;
    const double i1 = 1.0 / s.b1, i2 = md == 1 ? 1.0 / s.r22 : 0.0;
    double2 x, y;  // A (x1_prev / r22_prev) and x1 + gamma u1, row l
    if (l < J) {
        const double2 s1 = rr[l], s2 = rr[J + l], t1 = rr[2 * J + l], p2 = e2[l];
        x = make_double2(p2.x + s2.x + s.d_now.x * s1.x - s.d_now.y * s1.y,
                         p2.y + s2.y + s.d_now.x * s1.y + s.d_now.y * s1.x);
        y = make_double2(t1.x + s.gamma_now * s1.x, t1.y + s.gamma_now * s1.y);
    } else if (l == J) {
        x = make_double2(s.r12.x + s.d_now.x * s.b1, s.r12.y + s.d_now.y * s.b1);
        y = make_double2(s.a1.x + s.gamma_now * s.b1, s.a1.y);
    } else {
        x = make_double2(s.r22, 0.0);
        y = s.c1;
    }
    const cd cj = {(x.x - g1r) * i1, (x.y - g1i) * i1};
    Hr[l + (long long)J * ldh] = make_double2(cj.re, cj.im);
    if (md == 2) return;
    const cd rc = cmul(cd{s.r12.x, s.r12.y}, cj);
    Hr[l + (long long)(J + 1) * ldh] = make_double2((y.x - g2r - rc.re) * i2, (y.y - g2i - rc.im) * i2);
    double2* n1 = ecn + (size_t)r * 2 * kmax;
    const double2 p1 = l < J ? rr[2 * J + l] : (l == J ? s.a1 : s.c1);
    const double2 p2 = l < J ? rr[3 * J + l] : (l == J ? s.a2 : s.c2);
    n1[l] = make_double2(p1.x * i2, p1.y * i2);
    n1[kmax + l] = make_double2(p2.x * i2, p2.y * i2);
}

// w f - q in one rounding
__device__ __forceinline__ cf scale_less(cf w, float f, cf q) { return {fmaf(w.re, f, -q.re), fmaf(w.im, f, -q.im)}; }

// The update of a block step: writes v_J, v_{J+1}, u1', u2' (mode 1), or v_J
// and u1' = (u2 - V s2 - r12 v_J)/b1 (mode 2). Persistent and warp-specialised
// like k_arnoldi_update_ws, with four sums per unit. What is subtracted is small
// beside the scaled vector and is put together first, so that a vector has one
// rounding of its own size: x1 and x2 = A x1 are taken before u1' is rounded, so its
// rounding, unlike u's in single steps, is an error of the Arnoldi relation.
__global__ void __launch_bounds__(DTHREADS, 1)
    k_pair_update(float4* __restrict__ basis, long long basis_rhs_stride, long long vec_stride, int J,
                  const double2* __restrict__ red, long long red_stride, const PairState* __restrict__ ps,
                  const int* __restrict__ mode, float4* __restrict__ u1, float4* __restrict__ u2,
                  const float4* __restrict__ x1, const float4* __restrict__ x2, long long nunits, int tu, int nrhs,
                  int* __restrict__ err) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ __align__(8) uint64_t full[TNS];
    __shared__ __align__(8) uint64_t empty[TNS];
    __shared__ int abort_flag;
    float4* sc = reinterpret_cast<float4*>(smem + TNS * kStageBytes);  // (s1, s2), (t1, t2) of vector i at 2i
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int G = gridDim.x, q = blockIdx.x;
    const long long tpr = (nunits + tu - 1) / tu;
    const long long T = tpr * nrhs;
    const long long lo = range_lo(q, T, G), hi = range_lo(q + 1, T, G);
    const int ngroups = (J + TG - 1) / TG;
    volatile int* abort = &abort_flag;
    if (tid == 0) {
        for (int k = 0; k < TNS; ++k) {
            mbar_init(&full[k], 1);
            mbar_init(&empty[k], TW);
        }
        abort_flag = 0;
        mbar_fence_init();
    }
    __syncthreads();

    if (warp == TW) {  // ---- producer warp: one lane issues every stage
        if (lane != 0 || ngroups == 0) return;
        int n = 0;
        bool ok = true;
        for (long long it = lo; it < hi && ok; ++it) {
            const long long r = it / tpr, base = (it - r * tpr) * tu;
            if (mode[r] == 0) continue;
            const uint32_t bytes = (uint32_t)min((long long)tu, nunits - base) * 16u;
            const float4* Vr = basis + r * basis_rhs_stride + base;
            for (int g = 0; g < ngroups; ++g) {
                const int s = n % TNS;
                if (n >= TNS) {
                    if (!mbar_wait_or_abort(&empty[s], (uint32_t)((n / TNS - 1) & 1), abort)) {
                        ok = false;
                        break;
                    }
                    fence_proxy_async_smem();
                }
                const int nv = min(TG, J - g * TG);
                unsigned char* dst = smem + (size_t)s * kStageBytes;
                mbar_expect_tx(&full[s], bytes * nv);
                for (int v = 0; v < nv; ++v)
                    bulk_load(dst + (size_t)v * TU * 16, Vr + (long long)(g * TG + v) * vec_stride, bytes, &full[s]);
                ++n;
            }
        }
        for (int k = max(0, n - TNS); k < n && ok; ++k)
            ok = mbar_wait_or_abort(&empty[k % TNS], (uint32_t)((k / TNS) & 1), abort);
        if (!ok) {
            atomicExch(err, OVS_ETIMEOUT_CODE);
            abort_flag = 1;
            for (int k = max(0, n - TNS); k < n; ++k) mbar_wait_bounded(&full[k % TNS], (uint32_t)((k / TNS) & 1));
        }
        return;
    }

    // ---- consumer warps
    int n = 0, md = 0;
    long long seg_r = -1;
    bool bad = false;
    float ib = 0.f, i2 = 0.f;
    cf r12{}, a1{}, a2{}, c1{}, c2{}, d{};
    for (long long it = lo; it < hi; ++it) {
        const long long r = it / tpr, base = (it - r * tpr) * tu, end = min(base + tu, nunits);
        if (mode[r] == 0) continue;
        if (r != seg_r) {  // coefficients of the next right-hand side
            if (consumers_sync_or(bad)) return;
            const double2* rr = red + r * red_stride;
            for (int i = tid; i < J; i += TB) {
                const double2 p0 = rr[i], p1 = rr[J + i], p2 = rr[2 * J + i], p3 = rr[3 * J + i];
                sc[2 * i] = make_float4((float)p0.x, (float)p0.y, (float)p1.x, (float)p1.y);
                sc[2 * i + 1] = make_float4((float)p2.x, (float)p2.y, (float)p3.x, (float)p3.y);
            }
            if (consumers_sync_or(bad)) return;
            md = mode[r];
            const PairState s = ps[r];
            ib = (float)(1.0 / s.b1);
            const double j2 = md == 1 ? 1.0 / s.r22 : 0.0;
            i2 = (float)j2;
            r12 = {(float)s.r12.x, (float)s.r12.y};
            a1 = {(float)(s.a1.x * j2), (float)(s.a1.y * j2)};
            a2 = {(float)(s.a2.x * j2), (float)(s.a2.y * j2)};
            c1 = {(float)(s.c1.x * j2), (float)(s.c1.y * j2)};
            c2 = {(float)(s.c2.x * j2), (float)(s.c2.y * j2)};
            d = {(float)s.d_next.x, (float)s.d_next.y};
            seg_r = r;
        }
        float4* p1 = u1 + r * nunits;
        float4* p2 = u2 + r * nunits;
        const float4* q1 = x1 + r * nunits;
        const float4* q2 = x2 + r * nunits;
        float4 in[TE][4];
#pragma unroll
        for (int e = 0; e < TE; ++e) {
            const long long p = base + tid + (long long)TB * e;
            const bool live = p < end;
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
            in[e][0] = live ? p1[p] : zero;
            in[e][1] = live ? p2[p] : zero;
            in[e][2] = live ? __ldg(q1 + p) : zero;
            in[e][3] = live ? __ldg(q2 + p) : zero;
        }
        cf a[TE][4][2];
#pragma unroll
        for (int e = 0; e < TE; ++e)
#pragma unroll
            for (int p = 0; p < 4; ++p) a[e][p][0] = a[e][p][1] = {0.f, 0.f};
        for (int g = 0; g < ngroups; ++g) {
            const int s = n % TNS;
            const bool got = bad || mbar_wait_or_abort(&full[s], (uint32_t)((n / TNS) & 1), abort);
            if (!__all_sync(0xffffffffu, got)) {  // keep `bad` uniform over the warp
                if (lane == 0) {
                    atomicExch(err, OVS_ETIMEOUT_CODE);
                    abort_flag = 1;
                }
                bad = true;
            }
            if (!bad) {
                const float4* st4 = reinterpret_cast<const float4*>(smem + (size_t)s * kStageBytes);
                const int nv = min(TG, J - g * TG);
#pragma unroll
                for (int gi = 0; gi < TG; ++gi) {
                    if (gi < nv) {
                        const float4 k0 = sc[2 * (g * TG + gi)], k1 = sc[2 * (g * TG + gi) + 1];
                        const cf k[4] = {{k0.x, k0.y}, {k0.z, k0.w}, {k1.x, k1.y}, {k1.z, k1.w}};
#pragma unroll
                        for (int e = 0; e < TE; ++e) {
                            cf vc[2];
                            Unit<float>::split(st4[gi * TU + tid + TB * e], vc);
#pragma unroll
                            for (int p = 0; p < 4; ++p) {
                                cfma(a[e][p][0], vc[0], k[p]);
                                cfma(a[e][p][1], vc[1], k[p]);
                            }
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty[s]);
            }
            ++n;
        }
        if (bad) continue;
        float4* v0 = basis + r * basis_rhs_stride + (long long)J * vec_stride;
        float4* v1 = v0 + vec_stride;
#pragma unroll
        for (int e = 0; e < TE; ++e) {
            const long long p = base + tid + (long long)TB * e;
            if (p >= end) continue;
            cf w[4][2], o0[2], o1[2], n1[2], n2[2];
#pragma unroll
            for (int k = 0; k < 4; ++k) Unit<float>::split(in[e][k], w[k]);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                o0[c] = scale_less(w[0][c], ib, a[e][0][c] * ib);
                cf rest = a[e][1][c];
                cfma(rest, o0[c], r12);
                if (md == 1) {
                    o1[c] = scale_less(w[1][c], i2, rest * i2);
                    cf q1 = a[e][2][c] * i2, q2 = a[e][3][c] * i2;
                    cfma(q1, o0[c], a1);
                    cfma(q1, o1[c], c1);
                    n1[c] = scale_less(w[2][c], i2, q1);
                    cfma(q2, o0[c], a2);
                    cfma(q2, o1[c], c2);
                    cfma(q2, n1[c], d);
                    n2[c] = scale_less(w[3][c], i2, q2);
                } else {
                    n1[c] = scale_less(w[1][c], ib, rest * ib);
                }
            }
            v0[p] = Unit<float>::join(o0);
            p1[p] = Unit<float>::join(n1);
            if (md == 1) {
                v1[p] = Unit<float>::join(o1);
                p2[p] = Unit<float>::join(n2);
            }
        }
    }
}

// Single steps after the blocks: right-hand side r takes part in step j from
// jstart[r] on while it has not broken down (k_used[r] == j then).
__global__ void k_tail_mask(const int* __restrict__ jstart, const int* __restrict__ k_used, int j,
                            int* __restrict__ mask, int nrhs) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r < nrhs) mask[r] = (j >= jstart[r] && k_used[r] == j) ? 1 : 0;
}

static size_t pair_dots_smem(int J, int ns) { return ns * kDStage + (size_t)(4 * J + NGRAM) * 16; }
static Items pair_items(long long nunits, int nrhs, int num_sms) {
    return balanced_items(nunits, nrhs, num_sms, PC, 128);
}

int pair_stride(int J) { return 4 * J + NGRAM; }

int pair_slots(long long nunits, int nrhs, int num_sms) {
    const Items w = pair_items(nunits, nrhs, num_sms);
    const long long T = w.per_rhs * nrhs;
    int n = 1;
    for (long long r = 0; r < nrhs; ++r)
        n = std::max(n, owner_of((r + 1) * w.per_rhs - 1, T, w.grid) - owner_of(r * w.per_rhs, T, w.grid) + 1);
    return n;
}

cudaError_t launch_pair_dots(const void* basis, long long basis_rhs_stride, long long vec_stride, int J,
                             const void* u1, const void* u2, const void* x1, const void* x2, long long nunits,
                             int nrhs, int num_sms, int nslot, void* partial, const int* active, int* err,
                             cudaStream_t st) {
    const int ns = pair_dots_smem(J, 3) + 9 * 1024 <= 227 * 1024 ? 3 : 2;
    const size_t smem = pair_dots_smem(J, ns);
    const void* fn = ns == 3 ? (const void*)k_pair_dots<3> : (const void*)k_pair_dots<2>;
    const cudaError_t e = ensure_dyn_smem(fn, smem);
    if (e != cudaSuccess) return e;
    const Items w = pair_items(nunits, nrhs, num_sms);
    const int G = w.grid, cu = (int)w.chunk;
    const float4 *a = (const float4*)u1, *b = (const float4*)u2, *c = (const float4*)x1, *d = (const float4*)x2;
    if (ns == 3)
        k_pair_dots<3><<<G, PTHREADS, smem, st>>>((const float4*)basis, basis_rhs_stride, vec_stride, J, a, b, c, d,
                                                  nunits, cu, nrhs, nslot, (double2*)partial, active, err);
    else
        k_pair_dots<2><<<G, PTHREADS, smem, st>>>((const float4*)basis, basis_rhs_stride, vec_stride, J, a, b, c, d,
                                                  nunits, cu, nrhs, nslot, (double2*)partial, active, err);
    return cudaGetLastError();
}

cudaError_t launch_pair_start(const void* red, long long red_stride, PairState* ps, int nrhs, cudaStream_t st) {
    k_pair_start<<<(nrhs + 127) / 128, 128, 0, st>>>((const double2*)red, red_stride, ps, nrhs);
    return cudaGetLastError();
}

cudaError_t launch_pair_step(const void* red, long long red_stride, int J, bool more, void* H, long long h_rhs,
                             int ldh, double* beta0, double* inv_beta, void* dcoef, double* hnorm2, int* active,
                             int* k_used, PairState* ps, int* pact, int* mode, int* jstart, int never,
                             const void* ec, void* ecn, int kmax, int nrhs, cudaStream_t st) {
    const StepOut o{(double2*)H, h_rhs, ldh, beta0, inv_beta, (double2*)dcoef, hnorm2, active, k_used};
    k_pair_step<<<nrhs, 256, 0, st>>>((const double2*)red, red_stride, J, more ? 1 : 0, o, ps, pact, mode, jstart,
                                      never);
    k_pair_column<<<dim3((J + 2 + 7) / 8, nrhs), 256, 0, st>>>((const double2*)red, red_stride, J, (double2*)H, h_rhs,
                                                               ldh, ps, mode, (const double2*)ec, (double2*)ecn,
                                                               kmax);
    return cudaGetLastError();
}

cudaError_t launch_pair_update(void* basis, long long basis_rhs_stride, long long vec_stride, int J, const void* red,
                               long long red_stride, const PairState* ps, const int* mode, void* u1, void* u2,
                               const void* x1, const void* x2, long long nunits, int nrhs, int num_sms, int* err,
                               cudaStream_t st) {
    const size_t smem = TNS * kStageBytes + (size_t)std::max(J, 1) * 32;
    const cudaError_t e = ensure_dyn_smem((const void*)k_pair_update, smem);
    if (e != cudaSuccess) return e;
    const Items w = balanced_items(nunits, nrhs, num_sms, TU, 16);
    k_pair_update<<<w.grid, DTHREADS, smem, st>>>((float4*)basis, basis_rhs_stride, vec_stride, J, (const double2*)red,
                                             red_stride, ps, mode, (float4*)u1, (float4*)u2, (const float4*)x1,
                                             (const float4*)x2, nunits, (int)w.chunk, nrhs, err);
    return cudaGetLastError();
}

cudaError_t launch_tail_mask(const int* jstart, const int* k_used, int j, int* mask, int nrhs, cudaStream_t st) {
    k_tail_mask<<<(nrhs + 127) / 128, 128, 0, st>>>(jstart, k_used, j, mask, nrhs);
    return cudaGetLastError();
}

}  // namespace ovs
