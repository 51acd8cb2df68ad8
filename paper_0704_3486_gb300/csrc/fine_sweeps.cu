// K2 in two or three launches per Arnoldi step: the inner products, [their sums,]
// and the rest of the step. Here the complex64 form, where the lattice is too
// small for the TMA sweeps (tma_sweeps.cu) to give every SM a share of the basis;
// the complex128 form, on the same split, is fix_sweeps.cu.
//
// Split of the inner products: along the field (chunks of 128-unit tiles) and
// along the basis (sets of four vectors). Large problems: a block takes a chunk
// and a group of sets, a warp whole sets of the chunk. Small ones (SPREAD): a
// block takes one set of one chunk and its warps share the tiles (8^4, one
// right-hand side: 16.8 us; with one vector per warp 20).
//
// Nothing is done by one block between the two: every block of the update takes
// the step's scalars for itself, and where the partial sums are few (24 chunks
// and 102 sums at 4^4 and 50 vectors: 39 KB from L2) also adds the chunks; else
// k_reduce adds them in between. A last block doing both by a ticket took 14 us
// of a 27 us sweep at 4^4, a launch of one block per right-hand side 10 us of a
// step; programmatic dependent launch made 3x5x7x9 slower (7.5 ms against 5.9:
// waiting blocks hold the registers that the running sweep's next blocks need).
//
// Measured, against register sweeps of 2048-unit row blocks, a reduction, the
// scalars and the column in launches of their own (six per step): 8^4, one
// right-hand side, k = 200: 23.1 -> 7.8 ms.
#include <algorithm>

#include "fine_dev.cuh"

namespace ovs {

namespace {

using R = float;
using vec = Unit<R>::vec;
constexpr int NC = Unit<R>::ncplx;

// One halving exchange of the warp transpose-reduction over CUR values.
template <int CUR, int O, int M>
__device__ __forceinline__ void halve(R (&v)[M], bool upper) {
#pragma unroll
    for (int i = 0; i < CUR / 2; ++i) {
        const R send = upper ? v[i] : v[i + CUR / 2];
        const R keep = upper ? v[i + CUR / 2] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
    }
}

// partial[r][chunk]: s_i = V_i^H u and (NW = 2) t_i = V_i^H z for i < J, then
// (u^H u, 0) and u^H z.
// A warp takes four vectors at a time and streams its block's chunk of them,
// with u and z from L1, into 16 sums per lane over a tile (8 terms and 32 lanes)
// before they join FP64.
// What bounds it at these sizes: latency.
template <int NW, bool SPREAD>
__global__ void __launch_bounds__(FT, SPREAD ? 3 : 2)
    k_fine_dots(const vec* __restrict__ basis, long long basis_rhs, long long vec_stride, int J,
                const vec* __restrict__ u, const vec* __restrict__ z,
                long long nunits, int tiles, int nchunk, int vgroups, double2* __restrict__ partial,
                const int* __restrict__ active) {
    constexpr int M = FV * NW * 2;  // values of a pass: vector, which, component
    constexpr int SH = NW == 2 ? 1 : 2;  // 2^SH lanes end up with the same value
    __shared__ double ex[FW][3];
    __shared__ double wsum[SPREAD ? FW : 1][M];
    const int r = blockIdx.y;
    if (active != nullptr && active[r] == 0) return;
    const int chunk = blockIdx.x / vgroups, g = blockIdx.x - chunk * vgroups;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int S = NW * J + 2;
    const int nsets = (J + FV - 1) / FV;
    const vec* ur = u + r * nunits;
    const vec* zr = NW == 2 ? z + r * nunits : nullptr;
    double* part = reinterpret_cast<double*>(partial + ((size_t)r * nchunk + chunk) * S);
    const long long c0 = (long long)chunk * tiles * FTILE, c1 = min(c0 + (long long)tiles * FTILE, nunits);
    if (g == 0) {  // u^H u, u^H z of the chunk: FP32 over 8 terms, FP64 beyond
        double uu = 0.0, uzr = 0.0, uzi = 0.0;
        for (long long base = c0 + warp * FTILE + lane; base < c1; base += FW * FTILE) {
            cplx<R> a = {R(0), R(0)}, b = {R(0), R(0)};
#pragma unroll
            for (int e = 0; e < FU; ++e) {
                const long long p = base + 32 * e;
                if (p >= c1) break;
                cplx<R> uc[NC], zc[NC];
                Unit<R>::split(ur[p], uc);
                if (NW == 2) Unit<R>::split(zr[p], zc);
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    cfmac(a, uc[c], uc[c]);
                    if (NW == 2) cfmac(b, uc[c], zc[c]);
                }
            }
            uu += double(a.re);
            uzr += double(b.re);
            uzi += double(b.im);
        }
        uu = warp_sum(uu);
        uzr = warp_sum(uzr);
        uzi = warp_sum(uzi);
        if (lane == 0) {
            ex[warp][0] = uu;
            ex[warp][1] = uzr;
            ex[warp][2] = uzi;
        }
    }
    for (int q = SPREAD ? g : g + vgroups * warp; q < nsets; q += SPREAD ? nsets : vgroups * FW) {
        const int i0 = q * FV, nv = min(FV, J - i0);
        const vec* vb = basis + r * basis_rhs + (long long)i0 * vec_stride;
        R v[M];
        double kept = 0.0;
#pragma unroll
        for (int k = 0; k < M; ++k) v[k] = R(0);
        auto reduce = [&]() {
            halve<M, 16>(v, (lane & 16) != 0);
            halve<M / 2, 8>(v, (lane & 8) != 0);
            halve<M / 4, 4>(v, (lane & 4) != 0);
            if (NW == 2) halve<M / 8, 2>(v, (lane & 2) != 0);
            if (NW == 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
            kept += double(v[0]);
        };
        // one unit of u, z and the four vectors
        auto term = [&](const vec& uv, const vec& zv, const vec (&x)[FV]) {
            cplx<R> uc[NC], zc[NC];
            Unit<R>::split(uv, uc);
            Unit<R>::split(zv, zc);
#pragma unroll
            for (int gi = 0; gi < FV; ++gi) {
                cplx<R> vc[NC];
                Unit<R>::split(x[gi], vc);
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    cplx<R> a = {v[gi * NW * 2], v[gi * NW * 2 + 1]};
                    cfmac(a, vc[c], uc[c]);
                    v[gi * NW * 2] = a.re;
                    v[gi * NW * 2 + 1] = a.im;
                    if (NW == 2) {
                        cplx<R> b = {v[gi * 4 + 2], v[gi * 4 + 3]};
                        cfmac(b, vc[c], zc[c]);
                        v[gi * 4 + 2] = b.re;
                        v[gi * 4 + 3] = b.im;
                    }
                }
            }
        };
        for (long long base = c0 + lane + (SPREAD ? warp * FTILE : 0); base - lane < c1;
             base += SPREAD ? FW * FTILE : FTILE) {
            const bool whole = nv == FV && base - lane + FTILE <= c1;
            if (whole) {
#pragma unroll
                for (int e = 0; e < FU; e += 2) {  // 12 loads in flight, more where registers allow
                    vec x0[FV], x1[FV];
                    const long long p = base + 32 * e;
                    const vec u0 = ur[p], u1 = ur[p + 32];
                    const vec z0 = NW == 2 ? zr[p] : u0, z1 = NW == 2 ? zr[p + 32] : u1;
#pragma unroll
                    for (int gi = 0; gi < FV; ++gi) {
                        x0[gi] = vb[(long long)gi * vec_stride + p];
                        x1[gi] = vb[(long long)gi * vec_stride + p + 32];
                    }
                    term(u0, z0, x0);
                    term(u1, z1, x1);
                }
            } else {
                for (int e = 0; e < FU; ++e) {
                    const long long p = base + 32 * e;
                    if (p >= c1) break;
                    vec x[FV];
#pragma unroll
                    for (int gi = 0; gi < FV; ++gi)
                        x[gi] = gi < nv ? vb[(long long)gi * vec_stride + p] : vec{};
                    const vec uv = ur[p];
                    term(uv, NW == 2 ? zr[p] : uv, x);
                }
            }
            __syncwarp();
            reduce();
#pragma unroll
            for (int k = 0; k < M; ++k) v[k] = R(0);
        }
        const int k = lane >> SH;
        if (SPREAD) {
            if ((lane & ((1 << SH) - 1)) == 0) wsum[warp][k] = kept;
            __syncthreads();
            // the set's four vectors, over the warps that share its tiles
            const int gi = tid / (2 * NW), kk = tid % (2 * NW), which = kk >> 1;
            if (tid < FV * 2 * NW && q * FV + gi < J) {
                double a = 0.0;
#pragma unroll
                for (int w = 0; w < FW; ++w) a += wsum[w][gi * 2 * NW + kk];
                part[(size_t)(which * J + q * FV + gi) * 2 + (kk & 1)] = a;
            }
        } else {
            const int gi = k / (NW * 2), which = (k >> 1) & (NW - 1);
            if ((lane & ((1 << SH) - 1)) == 0 && gi < nv)
                part[(size_t)(which * J + i0 + gi) * 2 + (k & 1)] = kept;
        }
    }
    if (g == 0) {
        __syncthreads();
        if (tid < 4) {
            double a = 0.0;
            if (tid != 1)
                for (int w = 0; w < FW; ++w) a += ex[w][tid == 0 ? 0 : tid - 1];
            part[(size_t)(NW * J) * 2 + tid] = a;  // (u^H u, 0), u^H z
        }
    }
}

// The rest of step J (struct FineStep). The first nupd blocks of a right-hand
// side share its tiles, the others do 8 rows of the column each. Every block
// first adds the chunks' sums (nchunk = 1: they are added already) into shared
// memory; warp 0 then takes the scalars
// while the other warps are already at the basis (they are needed last).
// SPLIT = 1: a thread sums its E units over all J vectors. SPLIT = 8 (small
// fields): a block takes 32 E units, each warp every eighth vector, and the eight
// sums meet in shared memory.
template <int E, int SPLIT>
__global__ void __launch_bounds__(FT, 3)
    k_fine_update(vec* basis, long long basis_rhs, long long vec_stride, int J,
                  const double2* __restrict__ partial, long long p_rhs, int nchunk, vec* u,
                  const vec* __restrict__ z, long long nunits, int nupd, FineStep fs) {
    constexpr int T = SPLIT == 1 ? FT : 32;
    extern __shared__ double2 red[];  // [2J + 2]: s, t, (u^H u, 0), u^H z; then s and t in complex64
    __shared__ cplx<R> sum[SPLIT == 1 ? 1 : SPLIT][SPLIT == 1 ? 1 : 32 * E][NC][2];
    __shared__ StepShared sm;
    const int r = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool first = blockIdx.x == 0;
    if (fs.active[r] == 0) {
        if (first && tid == 0) fs.activen[r] = 0;
        return;
    }
    const int S = 2 * J + 2;
    cplx<R>* sc = reinterpret_cast<cplx<R>*>(red + S);
    for (int i = tid; i < S; i += FT) {
        const double2 a = chunk_sum(partial + r * p_rhs, S, nchunk, i);
        red[i] = a;
        if (i < 2 * J) sc[i] = {R(a.x), R(a.y)};
    }
    __syncthreads();
    double v[4];
    if (step_sums(red, red + J, J, r, fs, sm, v) && lane == 0)
        step_scalars(v, red[2 * J].x, red[2 * J + 1], J, r, first, fs, sm);
    if ((int)blockIdx.x >= nupd) {
        __syncthreads();
        step_column(red, red + J, J, ((int)blockIdx.x - nupd) * FW + warp, r, fs, sm);
        return;
    }
    vec* Vr = basis + r * basis_rhs;
    vec* vout = Vr + (long long)J * vec_stride;
    vec* ur = u + r * nunits;
    const vec* zr = z + r * nunits;
    auto finish = [&](long long p, const cplx<R> (&sa)[NC], const cplx<R> (&sb)[NC]) {
        const R ib = R(sm.ib);
        const cplx<R> d = {R(sm.d.x), R(sm.d.y)};
        cplx<R> uc[NC], zc[NC], vo[NC], un[NC];
        Unit<R>::split(ur[p], uc);
        Unit<R>::split(__ldg(zr + p), zc);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            vo[c] = {fmaf(uc[c].re, ib, -(sa[c].re * ib)), fmaf(uc[c].im, ib, -(sa[c].im * ib))};  // sa is small
            un[c] = (zc[c] - sb[c]) * ib - cmul(vo[c], d);
        }
        vout[p] = Unit<R>::join(vo);
        ur[p] = Unit<R>::join(un);
    };
    for (long long tile = blockIdx.x; tile * T * E < nunits; tile += nupd) {
        const long long base = tile * T * E + (SPLIT == 1 ? tid : lane);
        cplx<R> a[E][NC], b[E][NC];
        bool ok[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            ok[e] = base + (long long)T * e < nunits;
#pragma unroll
            for (int c = 0; c < NC; ++c) a[e][c] = b[e][c] = {R(0), R(0)};
        }
        auto add = [&](int i, const vec (&x)[E]) {
            const cplx<R> si = sc[i], ti = sc[J + i];
#pragma unroll
            for (int e = 0; e < E; ++e) {
                cplx<R> vc[NC];
                Unit<R>::split(x[e], vc);
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    cfma(a[e][c], vc[c], si);
                    cfma(b[e][c], vc[c], ti);
                }
            }
        };
        auto get = [&](int i, vec (&x)[E]) {
#pragma unroll
            for (int e = 0; e < E; ++e)
                x[e] = ok[e] ? __ldcs(Vr + (long long)i * vec_stride + base + (long long)T * e) : vec{};
        };
        int i = SPLIT == 1 ? 0 : warp;
        for (; i + 3 * SPLIT < J; i += 4 * SPLIT) {  // four vectors' loads in flight
            vec x0[E], x1[E], x2[E], x3[E];
            get(i, x0);
            get(i + SPLIT, x1);
            get(i + 2 * SPLIT, x2);
            get(i + 3 * SPLIT, x3);
            add(i, x0);
            add(i + SPLIT, x1);
            add(i + 2 * SPLIT, x2);
            add(i + 3 * SPLIT, x3);
        }
        for (; i < J; i += SPLIT) {
            vec x[E];
            get(i, x);
            add(i, x);
        }
        if (SPLIT > 1) {
#pragma unroll
            for (int e = 0; e < E; ++e)
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    sum[warp % SPLIT][SPLIT == 1 ? 0 : lane + 32 * e][c][0] = a[e][c];
                    sum[warp % SPLIT][SPLIT == 1 ? 0 : lane + 32 * e][c][1] = b[e][c];
                }
        }
        __syncthreads();  // the scalars are there (and the eight parts of the sums)
        if (sm.brk) return;  // uniform: a breakdown has no v_J
        if (SPLIT == 1) {
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (ok[e]) finish(base + (long long)T * e, a[e], b[e]);
        } else {
            // the eight parts, one real number per thread, then the two results. The part
            // with V_{J-1} comes last: it is the large one (a three-term recurrence has
            // little else), and every part added after it would round it once more.
            R* flat = reinterpret_cast<R*>(&sum[0][0][0][0]);
            constexpr int NV = SPLIT == 1 ? 1 : 32 * E * NC * 4;
            for (int k = tid; k < NV; k += FT) {
                R x = flat[J % SPLIT * NV + k];
#pragma unroll
                for (int w = 1; w < SPLIT; ++w) x += flat[(J + w) % SPLIT * NV + k];
                flat[k] = x;
            }
            __syncthreads();
            const long long p = tile * T * E + tid;
            if (tid < 32 * E && p < nunits) {
                cplx<R> sa[NC], sb[NC];
                const int at = SPLIT == 1 ? 0 : tid;
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    sa[c] = sum[0][at][c][0];
                    sb[c] = sum[0][at][c][1];
                }
                finish(p, sa, sb);
            }
            __syncthreads();  // the sums are overwritten by the next tile
        }
    }
}

// Split of a sweep over J vectors: chunks of `tiles` tiles and groups of the
// sets of four vectors. Below 64 (tile, set) pairs per SM the blocks take one
// set each, about two blocks per SM; every chunk more is one more partial sum to add.
struct FineSplit {
    int tiles, nchunk, vgroups;
    bool spread;
};
FineSplit fine_split(long long nunits, int J, int nrhs, int num_sms) {
    const long long all = (nunits + FTILE - 1) / FTILE;
    const int nsets = std::max(1, (J + FV - 1) / FV);
    FineSplit f;
    f.spread = all * nsets * nrhs < 64LL * num_sms;
    f.vgroups = f.spread ? nsets : std::max(1, nsets / 12);
    const long long want = std::max<long long>(1, 2LL * num_sms / ((long long)f.vgroups * nrhs));
    f.tiles = (int)std::max<long long>(1, (all + want - 1) / want);
    f.nchunk = (int)((all + f.tiles - 1) / f.tiles);
    return f;
}

template <int NW>
cudaError_t dots(const void* basis, long long basis_rhs, long long vec_stride, int J, const void* u, const void* z,
                 long long nunits, int nrhs, int num_sms, void* partial, const int* active, cudaStream_t st) {
    const FineSplit f = fine_split(nunits, J, nrhs, num_sms);
    const dim3 grid(f.nchunk * f.vgroups, nrhs);
    auto go = [&](auto kernel) {
        kernel<<<grid, FT, 0, st>>>((const vec*)basis, basis_rhs, vec_stride, J, (const vec*)u, (const vec*)z, nunits,
                                    f.tiles, f.nchunk, f.vgroups, (double2*)partial, active);
        return cudaGetLastError();
    };
    return f.spread ? go(k_fine_dots<NW, true>) : go(k_fine_dots<NW, false>);
}

template <int E, int SPLIT>
cudaError_t update_as(void* basis, long long basis_rhs, long long vec_stride, int J, const void* partial,
                      long long p_rhs, int nchunk, void* u, const void* z, long long nunits, int nrhs, int num_sms, const FineStep& fs,
                      cudaStream_t st) {
    const size_t smem = (size_t)(2 * J + 2) * sizeof(double2) + (size_t)2 * J * sizeof(cplx<R>);
    const cudaError_t e = allow_smem((const void*)k_fine_update<E, SPLIT>, smem);
    if (e != cudaSuccess) return e;
    const long long per = (long long)(SPLIT == 1 ? FT : 32) * E, tiles = (nunits + per - 1) / per;
    const int ncol = (J + 1 + FW - 1) / FW;
    // where every block adds the chunks: as many blocks as are resident
    const long long room = nchunk > 1 ? std::max<long long>(1, 3LL * num_sms / nrhs) : tiles;
    const long long each = (tiles + room - 1) / room;
    const int nupd = (int)((tiles + each - 1) / each);
    k_fine_update<E, SPLIT><<<dim3(nupd + ncol, nrhs), FT, smem, st>>>((vec*)basis, basis_rhs, vec_stride, J,
                                                                         (const double2*)partial, p_rhs, nchunk, (vec*)u,
                                                                         (const vec*)z, nunits, nupd, fs);
    return cudaGetLastError();
}

cudaError_t update(void* basis, long long basis_rhs, long long vec_stride, int J, const void* partial,
                   long long p_rhs, int nchunk, void* u, const void* z, long long nunits, int nrhs, int num_sms,
                   const FineStep& fs, cudaStream_t st) {
    const long long wide = (nunits + FT - 1) / FT * nrhs;  // blocks of one unit per thread
#define OVS_UPD(E, SPLIT)                                                                                              \
    update_as<E, SPLIT>(basis, basis_rhs, vec_stride, J, partial, p_rhs, nchunk, u, z, nunits, nrhs, num_sms, fs, st)
    if (wide >= 8LL * num_sms) return OVS_UPD(2, 1);
    if (wide >= 2LL * num_sms) return OVS_UPD(1, 1);
    if (wide * 8 > 3LL * num_sms) return OVS_UPD(2, 8);
    return OVS_UPD(1, 8);
#undef OVS_UPD
}

}  // namespace

int fine_chunks(int prec, long long nunits, int J, int nrhs, int num_sms) {
    return prec == PREC_F64 ? fix_chunks(nunits, J, nrhs, num_sms) : fine_split(nunits, J, nrhs, num_sms).nchunk;
}

int fine_chunks_max(int nrhs, int num_sms) { return 2 * num_sms + nrhs; }

cudaError_t launch_fine_dots(int prec, int nw, const void* basis, long long basis_rhs, long long vec_stride, int J,
                             const FixScales& fx, const void* u, const void* z, long long nunits, int nrhs,
                             int num_sms, void* partial, const int* active, cudaStream_t st) {
    if (prec == PREC_F64)
        return launch_fix_dots(nw, basis, basis_rhs, vec_stride, J, fx.vexp, fx.vexp_rhs, fx.uexp, u, z, nunits, nrhs,
                               num_sms, partial, active, st);
    return nw == 1 ? dots<1>(basis, basis_rhs, vec_stride, J, u, z, nunits, nrhs, num_sms, partial, active, st)
                   : dots<2>(basis, basis_rhs, vec_stride, J, u, z, nunits, nrhs, num_sms, partial, active, st);
}

bool fine_sums_in_update(int chunks, int J) { return (long long)chunks * (2 * J + 2) <= 4096; }

cudaError_t launch_fine_update(int prec, void* basis, long long basis_rhs, long long vec_stride, int J,
                               const FixScales& fx, const void* sums, long long s_rhs, int nchunk, void* u,
                               const void* z, long long nunits, int nrhs, int num_sms, const FineStep& fs,
                               cudaStream_t st) {
    if (prec == PREC_F64)
        return launch_fix_update(basis, basis_rhs, vec_stride, J, fx.vexp, fx.vexp_rhs, fx.uexp, fx.uexpn, sums, s_rhs,
                                 nchunk, u, z, nunits, nrhs, num_sms, fs, st);
    return update(basis, basis_rhs, vec_stride, J, sums, s_rhs, nchunk, u, z, nunits, nrhs, num_sms, fs, st);
}

}  // namespace ovs
