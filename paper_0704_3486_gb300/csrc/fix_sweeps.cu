// K2, complex128: the inner products, the update and the recombination over the
// Krylov basis, on the integer multipliers.
//
// The chip has 2 FP64 multiply-adds per clock and SM; at 8^4 with four sources
// they made the sweeps seven times slower than reading the basis. A 32 x 32 + 64
// bit multiply-add runs at about 50 per clock. So the operands of a sum are
// fixed-point numbers of 58 bits, scaled by a power of two over the largest
// element (of a basis vector; of u and z: per 1024 units; of the coefficients:
// per sweep), in two signed limbs
//     x = hi 2^30 + lo,  |hi| <= 2^28,  |lo| <= 2^29,
// and a product takes three of the four limb products, summed exactly in 64
// bits: hi hi (at most 64 products of a lane: 2^62) and hi lo + lo hi (32
// products: 2^62, then carried). What is dropped is lo lo, at most 2^-58 of the
// product of the two scales and of random sign (in u^H u a square: of 1024 units' sum
// at most 2^-47 of the largest element's square), and the rounding of the operands
// to a unit, 2^-58 of the scale (which is one to two times the largest element, of a
// basis vector up to four times), within three quarters; zeros stay zeros. An FP64 sum rounds
// each partial sum by 2^-54. The results' error against 64 bits is smaller than that
// of the FP64 sweeps on Gaussian sources (4^4 5.0e-16 for 7.2e-16, 8^4 8.0e-16 for
// 1.1e-15, 6^4 with k = 340 4.5e-16 for 1.1e-15) and like it on point sources (k = 40,
// restated on the CPU against long double: 8^4 7.0e-16 for 9.1e-16, 12^4 4.0e-16 for
// 3.7e-16; with the last bit set instead of a rounding, zeros included, 2.8e-15 and
// 5.5e-15).
//
// The basis is kept in limbs, 16 bytes per element: converting its elements in
// every sweep took 30 of 90 instructions each (8^4: 58 ms, now 50). The scale of
// v_J is known before it is computed, from max |u| (found by the inner products)
// and ||s||. u, z, H and the results are complex128.
//
// Conversion: the mantissa shifted by the difference of the exponents to two bits more
// than a number has, negated for a negative value, plus half a unit; the two bits go.
// An exponent of 0 (a zero; a subnormal is far below any scale in use) gives 0.
//
// Measured, against the same split in FP64: 8^4, 4 right-hand sides, k = 200:
// 136 -> 50 ms; 6^4, 2, k = 340: 75.9 -> 35.6 ms; 3x5x7x9, 3, k = 75: 5.98 -> 4.88
// ms; 4^4, 1, k = 100: 3.26 -> 2.83 ms. Tried without gain: the conversion of one
// component by the FP64 unit, three or four resident blocks, four vectors per warp
// (spills).
#include <algorithm>

#include "fine_dev.cuh"

namespace ovs {

namespace {

constexpr int SUB = 8 * FTILE;  // units with one scale of u and z: 32 per lane
constexpr int kSet = 2;  // vectors per warp of the inner products
constexpr int kNonFinite = 1 << 20;

struct Fix {
    int hi, lo;
};
// v 2^(1022 - e) 2^58 to a whole number, within 3/4, for a biased exponent e not below
// v's own
__device__ __forceinline__ Fix to_fix(double v, int e) {
    const int h = __double2hiint(v);
    const unsigned l = (unsigned)__double2loint(v);
    const int ev = (h >> 20) & 0x7ff, d = e - ev;
    const unsigned mh = (__funnelshift_l(l, (unsigned)h, 7) & 0x07ffffffu) | 0x08000000u;
    unsigned long long m = ev != 0 ? ((unsigned long long)mh << 32) | (l << 7) : 0ull;
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(d));  // shifts above 64 give 0
    const long long y = (h < 0 ? -(long long)m : (long long)m) + 2;
    const unsigned yl = (unsigned)y;
    return {(int)(y >> 32) + (int)(yl >> 31), (int)yl >> 2};
}
__device__ __forceinline__ unsigned abs_hi(double2 v) {
    return max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu);
}
__device__ __forceinline__ int exponent(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
__device__ __forceinline__ double nan64() { return __longlong_as_double(0x7ff8000000000000ll); }

// back to FP64: pow is 2^(e - 1022 - 58)
__device__ __forceinline__ double from_fix(Fix x, double pow) { return fma((double)x.hi, 1073741824.0, (double)x.lo) * pow; }

struct Acc {  // sum = hh 2^60 + hl 2^30
    long long hh, hl;
};
__device__ __forceinline__ void mul_add(Acc& a, Fix x, Fix y) {
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a.hh) : "r"(x.hi), "r"(y.hi));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a.hl) : "r"(x.hi), "r"(y.lo));
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a.hl) : "r"(x.lo), "r"(y.hi));
}
__device__ __forceinline__ void carry(Acc& a) {
    a.hh += a.hl >> 30;
    a.hl &= (1ll << 30) - 1;
}
__device__ __forceinline__ Fix neg(Fix x) { return {-x.hi, -x.lo}; }
// a complex pair in 16 bytes: re.lo, re.hi, im.lo, im.hi
__device__ __forceinline__ int4 pack(Fix re, Fix im) { return make_int4(re.lo, re.hi, im.lo, im.hi); }
__device__ __forceinline__ Fix re_of(int4 q) { return {q.y, q.x}; }
__device__ __forceinline__ Fix im_of(int4 q) { return {q.w, q.z}; }

// One halving exchange of the warp transpose-reduction over CUR sums of three
// limbs of 24 bits.
template <int CUR, int O, int M>
__device__ __forceinline__ void halve(int (&v)[M][3], bool upper) {
#pragma unroll
    for (int i = 0; i < CUR / 2; ++i)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int send = upper ? v[i][b] : v[i + CUR / 2][b];
            const int keep = upper ? v[i + CUR / 2][b] : v[i][b];
            v[i][b] = keep + __shfl_xor_sync(0xffffffffu, send, O);
        }
}

// partial[r][chunk]: s_i = V_i^H u and (NW = 2) t_i = V_i^H z for i < J, then
// u^H u and u^H z, for which u counts as vector J.
// A block takes a chunk and eight sets of two vectors, a warp one of the sets
// (SPREAD, small problems: four vectors, a warp one of them and every other tile),
// with u and z of 1024 units at a time as limbs in shared memory.
// What bounds it: issue. Per element of the basis 24 multiply-adds, 28 integer
// operations of the conversion and 8 of the carries; 16 B from memory.
template <int NW, bool SPREAD>
__global__ void __launch_bounds__(FT, 2)
    k_fix_dots(const int4* __restrict__ basis, long long basis_rhs, long long vec_stride, int J,
               const int* __restrict__ vexp, long long vexp_rhs, int* uexp, const double2* __restrict__ u,
               const double2* __restrict__ z, long long nunits, int tiles, int nchunk, int vgroups,
               double2* __restrict__ partial, const int* __restrict__ active) {
    constexpr int VS = SPREAD ? FV : kSet;  // vectors of a set
    constexpr int VW = SPREAD ? 1 : VS;  // vectors of a warp
    constexpr int EB = FU / 2;           // units of a lane in flight, twice
    constexpr int M = VW * NW * 2;       // sums: vector, which, component
    constexpr int SH = M == 16 ? 1 : M == 8 ? 2 : M == 4 ? 3 : 4;  // 2^SH lanes end up with the same sum
    __shared__ int4 fu[SUB], fz[NW == 2 ? SUB : 1];
    __shared__ unsigned wmax[FW][2];
    __shared__ double wsum[FW][M];
    const int r = blockIdx.y;
    if (active != nullptr && active[r] == 0) return;
    const int chunk = blockIdx.x / vgroups, g = blockIdx.x - chunk * vgroups;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double2* ur = u + r * nunits;
    const double2* zr = NW == 2 ? z + r * nunits : nullptr;
    const int* ve = vexp + r * vexp_rhs;
    const int nsets = (J + 1 + VS - 1) / VS;
    const int q = SPREAD ? g : (int)((long long)nsets * g / vgroups) + warp;
    const int qend = SPREAD ? g + 1 : (int)((long long)nsets * (g + 1) / vgroups);
    const int i0 = q * VS + (SPREAD ? warp % FV : 0);
    const int nv = q < qend ? max(0, min(VW, J + 1 - i0)) : 0;
    const int4* vb[VW];
    int ev[VW];
#pragma unroll
    for (int gi = 0; gi < VW; ++gi) {
        const bool own = gi < nv && i0 + gi < J;
        vb[gi] = own ? basis + r * basis_rhs + (long long)(i0 + gi) * vec_stride : nullptr;
        ev[gi] = own ? __ldg(ve + i0 + gi) : 0;
    }
    const long long c0 = (long long)chunk * tiles * FTILE, c1 = min(c0 + (long long)tiles * FTILE, nunits);
    double total = 0.0;
    for (long long b0 = c0; b0 < c1; b0 += SUB) {
        const int n = (int)min((long long)SUB, c1 - b0);
        int eu, ez = 0;
        {
            double2 a[SUB / FT], b[SUB / FT];
            unsigned mu = 0, mz = 0;
#pragma unroll
            for (int e = 0; e < SUB / FT; ++e) {
                const int p = tid + FT * e;
                a[e] = p < n ? ur[b0 + p] : make_double2(0.0, 0.0);
                b[e] = NW == 2 && p < n ? zr[b0 + p] : make_double2(0.0, 0.0);
                mu = max(mu, abs_hi(a[e]));
                mz = max(mz, abs_hi(b[e]));
            }
            mu = __reduce_max_sync(0xffffffffu, mu);
            mz = __reduce_max_sync(0xffffffffu, mz);
            if (lane == 0) {
                wmax[warp][0] = mu;
                wmax[warp][1] = mz;
            }
            __syncthreads();  // and nobody reads the last limbs any more
#pragma unroll
            for (int w = 0; w < FW; ++w) {
                mu = max(mu, wmax[w][0]);
                mz = max(mz, wmax[w][1]);
            }
            eu = (int)(mu >> 20);
            ez = (int)(mz >> 20);
            if (uexp != nullptr && g == 0 && tid == 0) atomicMax(uexp + r, eu);
#pragma unroll
            for (int e = 0; e < SUB / FT; ++e) {
                const int p = tid + FT * e;
                if (p >= (n + FTILE - 1) / FTILE * FTILE) break;
                const bool in = p < n;  // the rest of the last tile: zeros
                fu[p] = in ? pack(to_fix(a[e].x, eu), to_fix(a[e].y, eu)) : make_int4(0, 0, 0, 0);
                if (NW == 2) fz[p] = in ? pack(to_fix(b[e].x, ez), to_fix(b[e].y, ez)) : make_int4(0, 0, 0, 0);
            }
            __syncthreads();
        }
        if (nv == 0) continue;
        Acc acc[M];
#pragma unroll
        for (int k = 0; k < M; ++k) acc[k] = {0, 0};
        int es[VW];
#pragma unroll
        for (int gi = 0; gi < VW; ++gi) es[gi] = i0 + gi < J ? ev[gi] : eu;
        auto fetch = [&](int p0, int4 (&x)[EB][VW]) {
#pragma unroll
            for (int e = 0; e < EB; ++e)
#pragma unroll
                for (int gi = 0; gi < VW; ++gi)
                    x[e][gi] = vb[gi] != nullptr ? __ldg(vb[gi] + b0 + min(p0 + 32 * e, n - 1)) : fu[p0 + 32 * e];
        };
        auto add = [&](int p0, const int4 (&x)[EB][VW]) {
#pragma unroll
            for (int e = 0; e < EB; ++e) {
                const int4 uq = fu[p0 + 32 * e], zq = NW == 2 ? fz[p0 + 32 * e] : uq;
#pragma unroll
                for (int gi = 0; gi < VW; ++gi) {
                    const Fix vr = re_of(x[e][gi]), vi = im_of(x[e][gi]), ni = neg(vi);
#pragma unroll
                    for (int w = 0; w < NW; ++w) {
                        const int4 o = w == 0 ? uq : zq;
                        Acc& re = acc[(gi * NW + w) * 2];
                        Acc& im = acc[(gi * NW + w) * 2 + 1];
                        mul_add(re, vr, re_of(o));
                        mul_add(re, vi, im_of(o));
                        mul_add(im, vr, im_of(o));
                        mul_add(im, ni, re_of(o));
                    }
                }
            }
        };
        constexpr int TS = SPREAD ? FW / FV : 1;
        const int nt = (n + FTILE - 1) / FTILE;
        int t = SPREAD ? warp / FV : 0;
        int4 x[EB][VW], y[EB][VW];
        if (t < nt) fetch(t * FTILE + lane, x);
        for (; t < nt; t += TS) {
            const int p0 = t * FTILE + lane;
            fetch(p0 + 32 * EB, y);
            add(p0, x);
            if (t + TS < nt) fetch(p0 + TS * FTILE, x);
            add(p0 + 32 * EB, y);
            if (SPREAD || (t & 1)) {
#pragma unroll
                for (int k = 0; k < M; ++k) carry(acc[k]);
            }
        }
        int v[M][3];  // the sums times 2^10 in limbs of 24 bits
#pragma unroll
        for (int k = 0; k < M; ++k) {
            carry(acc[k]);
            v[k][2] = (int)(acc[k].hh >> 38);
            v[k][1] = (int)(acc[k].hh >> 14) & 0xffffff;
            v[k][0] = ((int)acc[k].hh & 0x3fff) << 10 | (int)(acc[k].hl >> 20);
        }
        if (M >= 2) halve<M, 16>(v, (lane & 16) != 0);
        if (M >= 4) halve<M / 2, 8>(v, (lane & 8) != 0);
        if (M >= 8) halve<M / 4, 4>(v, (lane & 4) != 0);
        if (M >= 16) halve<M / 8, 2>(v, (lane & 2) != 0);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            int x = v[0][b];
            if (M < 4) x += __shfl_xor_sync(0xffffffffu, x, 8);
            if (M < 8) x += __shfl_xor_sync(0xffffffffu, x, 4);
            if (M < 16) x += __shfl_xor_sync(0xffffffffu, x, 2);
            v[0][b] = x + __shfl_xor_sync(0xffffffffu, x, 1);
        }
        const int k = lane >> SH, gi = k / (NW * 2), which = (k >> 1) & (NW - 1);
        int ek = 0;
#pragma unroll
        for (int i = 0; i < VW; ++i) ek = i == gi ? es[i] : ek;
        const int eo = which == 0 ? eu : ez;
        const double sum = fma((double)v[0][2], 281474976710656.0, (double)(((long long)v[0][1] << 24) + v[0][0]));
        total += ek == 2047 || eo == 2047 ? nan64() : scalbn(sum, ek + eo - 2044 - 66);
    }
    const int S = NW * J + 2;
    double* part = reinterpret_cast<double*>(partial + ((size_t)r * nchunk + chunk) * S);
    if (SPREAD) {
        if ((lane & ((1 << SH) - 1)) == 0) wsum[warp][lane >> SH] = total;
        __syncthreads();
        const int gi = tid / M, kk = tid % M, which = kk >> 1, i = q * VS + gi;
        if (tid < FV * M && i <= J)
            part[(size_t)(i < J ? which * J + i : NW * J + which) * 2 + (kk & 1)] = wsum[gi][kk] + wsum[gi + FV][kk];
    } else {
        const int k = lane >> SH, gi = k / (NW * 2), which = (k >> 1) & (NW - 1), i = i0 + gi;
        if ((lane & ((1 << SH) - 1)) == 0 && gi < nv)
            part[(size_t)(i < J ? which * J + i : NW * J + which) * 2 + (k & 1)] = total;
    }
}

// Coefficients as limbs in place (each thread those it has read), with the
// scales of the basis vectors in them: x_i 2^(vexp_i - 1022) relative to the
// largest, whose exponent (or kNonFinite) is returned in every thread. m holds
// the thread's largest; red: FW ints of shared memory.
__device__ __forceinline__ int coef_exponent(double2 c, int ev) {
    const int e = (int)(abs_hi(c) >> 20);
    return e == 2047 ? kNonFinite : e == 0 ? -kNonFinite : e + ev - 1022;
}
__device__ __forceinline__ double2 coef_limbs(double2 c, int ev, int ref) {
    const int e = ref - ev + 1022;
    const Fix re = to_fix(c.x, e), im = to_fix(c.y, e);
    return make_double2(__hiloint2double(re.hi, re.lo), __hiloint2double(im.hi, im.lo));
}
// a unit of an accumulated sum (2^60 of the limbs' product)
__device__ __forceinline__ double coef_scale(int ref) {
    return ref >= kNonFinite / 2 ? nan64() : ref <= -kNonFinite / 2 ? 0.0 : scalbn(1.0, ref - 1022 - 56);
}

// out[w] = sum over the vectors first, first + SPLIT, ... of V_i[at] c_w,i in
// units of coef_scale. JP: J rounded up to 4 SPLIT, with zero coefficients.
// hh takes 32 vectors and hl 8 before they are carried on.
template <int NW, int E, int SPLIT>
__device__ __forceinline__ void fix_sum(const int4* __restrict__ V, long long vec_stride, int J, int JP,
                                        const int4* c, int first, const long long (&at)[E],
                                        double (&out)[E][NW][2]) {
#pragma unroll
    for (int e = 0; e < E; ++e)
#pragma unroll
        for (int w = 0; w < NW; ++w) out[e][w][0] = out[e][w][1] = 0.0;
    for (int i = first; i < JP;) {
        Acc a[E][NW][2];
#pragma unroll
        for (int e = 0; e < E; ++e)
#pragma unroll
            for (int w = 0; w < NW; ++w) a[e][w][0] = a[e][w][1] = {0, 0};
#pragma unroll 2
        for (int b = 0; b < 8 && i < JP; ++b, i += 4 * SPLIT) {
            int4 x[4][E];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int iv = min(i + k * SPLIT, J - 1);
#pragma unroll
                for (int e = 0; e < E; ++e) x[k][e] = __ldcs(V + (long long)iv * vec_stride + at[e]);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const Fix vr = re_of(x[k][e]), vi = im_of(x[k][e]), ni = neg(vi);
#pragma unroll
                    for (int w = 0; w < NW; ++w) {
                        const int4 o = c[w * JP + i + k * SPLIT];
                        mul_add(a[e][w][0], vr, re_of(o));
                        mul_add(a[e][w][0], ni, im_of(o));
                        mul_add(a[e][w][1], vr, im_of(o));
                        mul_add(a[e][w][1], vi, re_of(o));
                    }
                }
            }
            if (b & 1) {
#pragma unroll
                for (int e = 0; e < E; ++e)
#pragma unroll
                    for (int w = 0; w < NW; ++w) {
                        carry(a[e][w][0]);
                        carry(a[e][w][1]);
                    }
            }
        }
#pragma unroll
        for (int e = 0; e < E; ++e)
#pragma unroll
            for (int w = 0; w < NW; ++w)
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    out[e][w][q] += fma((double)a[e][w][q].hl, 9.31322574615478515625e-10, (double)a[e][w][q].hh);
    }
}

// The rest of step J (struct FineStep): v_J = (u - V s)/beta, u <- (z - V t)/beta
// - v_J d, the scalars in every block, the column of H in the blocks after the
// first nupd of a right-hand side (8 rows each), and vexp_J.
// SPLIT = 1: a thread sums its E units over all J vectors. SPLIT = 8 (small
// fields): a block takes 32 E units, each warp every eighth vector, and the eight
// sums meet in shared memory.
template <int E, int SPLIT>
__global__ void __launch_bounds__(FT, E == 1 ? 3 : 2)
    k_fix_update(int4* basis, long long basis_rhs, long long vec_stride, int J, int* vexp, long long vexp_rhs,
                 const int* __restrict__ uexp, int* uexpn, const double2* __restrict__ partial, long long p_rhs, int nchunk, double2* u,
                 const double2* __restrict__ z, long long nunits, int nupd, FineStep fs) {
    constexpr int T = SPLIT == 1 ? FT : 32;
    extern __shared__ double2 red[];  // s [JP], t [JP], u^H u, u^H z; s and t then become limbs
    __shared__ double sum[SPLIT == 1 ? 1 : SPLIT][SPLIT == 1 ? 1 : 32 * E][4];
    __shared__ StepShared sm;
    __shared__ int wmax[FW][2], s_ev;
    const int r = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool first = blockIdx.x == 0;
    if (first && tid == 0) uexpn[r] = 0;
    if (fs.active[r] == 0) {
        if (first && tid == 0) fs.activen[r] = 0;
        return;
    }
    const int S = 2 * J + 2, JP = (J + 4 * SPLIT - 1) / (4 * SPLIT) * (4 * SPLIT);
    int* ve = vexp + r * vexp_rhs;
    for (int i = tid; i < S; i += FT)
        red[i < J ? i : i < 2 * J ? JP + i - J : 2 * JP + i - 2 * J] = chunk_sum(partial + r * p_rhs, S, nchunk, i);
    __syncthreads();
    double v[4];
    const bool w0 = step_sums(red, red + JP, J, r, fs, sm, v);
    if ((int)blockIdx.x >= nupd) {
        if (w0 && lane == 0) step_scalars(v, red[2 * JP].x, red[2 * JP + 1], J, r, false, fs, sm);
        __syncthreads();
        step_column(red, red + JP, J, ((int)blockIdx.x - nupd) * FW + warp, r, fs, sm);
        return;
    }
    int es = -kNonFinite, et = -kNonFinite;
    for (int i = tid; i < J; i += FT) {
        const int ev = ve[i];
        es = max(es, coef_exponent(red[i], ev));
        et = max(et, coef_exponent(red[JP + i], ev));
    }
    es = __reduce_max_sync(0xffffffffu, es);
    et = __reduce_max_sync(0xffffffffu, et);
    if (lane == 0) {
        wmax[warp][0] = es;
        wmax[warp][1] = et;
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < FW; ++w) {
        es = max(es, wmax[w][0]);
        et = max(et, wmax[w][1]);
    }
    for (int i = tid; i < JP; i += FT) {
        const int ev = i < J ? ve[i] : 0;
        red[i] = i < J ? coef_limbs(red[i], ev, es) : make_double2(0.0, 0.0);
        red[JP + i] = i < J ? coef_limbs(red[JP + i], ev, et) : make_double2(0.0, 0.0);
    }
    __syncthreads();
    // the scalars while the other warps are at the basis: they are needed last
    if (w0 && lane == 0) {
        step_scalars(v, red[2 * JP].x, red[2 * JP + 1], J, r, first, fs, sm);
        // |v_J| < (max |u| + ||s||) / beta, the rows of V being at most 1 long
        s_ev = exponent((scalbn(1.0, uexp[r] - 1022) + 2.0 * sqrt(v[0])) * sm.ib * 1.0000001);
        if (first && !sm.brk) atomicMax(ve + J, s_ev);
    }
    const double ss = coef_scale(es), st = coef_scale(et);
    int4* Vr = basis + r * basis_rhs;
    int4* vout = Vr + (long long)J * vec_stride;
    double2* ur = u + r * nunits;
    const double2* zr = z + r * nunits;
    auto finish = [&](long long p, double ax, double ay, double bx, double by) {
        const double2 uc = ur[p], zc = __ldg(zr + p);
        const double ib = sm.ib;
        const double2 d = sm.d;
        const double2 vo = make_double2((uc.x - ss * ax) * ib, (uc.y - ss * ay) * ib);
        const int ev = s_ev;
        if ((int)(abs_hi(vo) >> 20) > ev) atomicMax(ve + J, 2047);  // bound broken: reported as a NaN
        vout[p] = pack(to_fix(vo.x, ev), to_fix(vo.y, ev));
        ur[p] = make_double2((zc.x - st * bx) * ib - (vo.x * d.x - vo.y * d.y),
                             (zc.y - st * by) * ib - (vo.x * d.y + vo.y * d.x));
    };
    const int4* c = reinterpret_cast<const int4*>(red);
    for (long long tile = blockIdx.x; tile * T * E < nunits; tile += nupd) {
        const long long base = tile * T * E + (SPLIT == 1 ? tid : lane);
        long long at[E];
#pragma unroll
        for (int e = 0; e < E; ++e) at[e] = min(base + (long long)T * e, nunits - 1);
        double a[E][2][2];
        fix_sum<2, E, SPLIT>(Vr, vec_stride, J, JP, c, SPLIT == 1 ? 0 : warp, at, a);
        if (SPLIT > 1) {
#pragma unroll
            for (int e = 0; e < E; ++e)
#pragma unroll
                for (int q = 0; q < 4; ++q) sum[warp % SPLIT][SPLIT == 1 ? 0 : lane + 32 * e][q] = a[e][q >> 1][q & 1];
        }
        __syncthreads();  // the scalars are there (and the eight parts of the sums)
        if (sm.brk) return;  // uniform: a breakdown has no v_J
        if (SPLIT == 1) {
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (base + (long long)T * e < nunits)
                    finish(base + (long long)T * e, a[e][0][0], a[e][0][1], a[e][1][0], a[e][1][1]);
        } else {
            // the eight parts, one real number per thread, then the two results
            double* flat = &sum[0][0][0];
            constexpr int NV = SPLIT == 1 ? 1 : 32 * E * 4;
            for (int k = tid; k < NV; k += FT) {
                double x = flat[k];
#pragma unroll
                for (int w = 1; w < SPLIT; ++w) x += flat[w * NV + k];
                flat[k] = x;
            }
            __syncthreads();
            const long long p = tile * T * E + tid;
            const double* q = sum[0][SPLIT == 1 ? 0 : tid % (32 * E)];
            if (tid < 32 * E && p < nunits) finish(p, q[0], q[1], q[2], q[3]);
            __syncthreads();  // the sums are overwritten by the next tile
        }
    }
}

// y += alpha sum_{i < min(J, Jdev[r])} V_i c_i: the recombination, on the same
// split as the update.
template <int SPLIT>
__global__ void __launch_bounds__(FT, 3)
    k_fix_combine(const int4* __restrict__ basis, long long basis_rhs, long long vec_stride, int Jmax,
                  const int* __restrict__ Jdev, const int* __restrict__ vexp, long long vexp_rhs,
                  const double2* __restrict__ coef, long long coef_stride, double alpha, double2* y,
                  long long nunits) {
    constexpr int T = SPLIT == 1 ? FT : 32;
    extern __shared__ double2 red[];  // c as limbs
    __shared__ double sum[SPLIT == 1 ? 1 : SPLIT][SPLIT == 1 ? 1 : 32][2];
    __shared__ int wmax[FW];
    const int r = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int J = Jdev != nullptr ? min(Jmax, Jdev[r]) : Jmax;
    if (J <= 0) return;
    const int JP = (J + 4 * SPLIT - 1) / (4 * SPLIT) * (4 * SPLIT);
    const int* ve = vexp + r * vexp_rhs;
    const double2* cr = coef + r * coef_stride;
    int ec = -kNonFinite;
    for (int i = tid; i < J; i += FT) ec = max(ec, coef_exponent(cr[i], ve[i]));
    ec = __reduce_max_sync(0xffffffffu, ec);
    if (lane == 0) wmax[warp] = ec;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < FW; ++w) ec = max(ec, wmax[w]);
    for (int i = tid; i < JP; i += FT) red[i] = i < J ? coef_limbs(cr[i], ve[i], ec) : make_double2(0.0, 0.0);
    __syncthreads();
    const double sc = alpha * coef_scale(ec);
    const long long p = (long long)blockIdx.x * T + (SPLIT == 1 ? tid : lane);
    const long long at[1] = {min(p, nunits - 1)};
    double a[1][1][2];
    fix_sum<1, 1, SPLIT>(basis + r * basis_rhs, vec_stride, J, JP, reinterpret_cast<const int4*>(red),
                         SPLIT == 1 ? 0 : warp, at, a);
    if (SPLIT > 1) {
        sum[warp % SPLIT][SPLIT == 1 ? 0 : lane][0] = a[0][0][0];
        sum[warp % SPLIT][SPLIT == 1 ? 0 : lane][1] = a[0][0][1];
        __syncthreads();
        if (tid >= 32) return;
#pragma unroll
        for (int w = 1; w < SPLIT; ++w) {
            a[0][0][0] += sum[w][SPLIT == 1 ? 0 : lane][0];
            a[0][0][1] += sum[w][SPLIT == 1 ? 0 : lane][1];
        }
    }
    if (p >= nunits) return;
    double2 o = y[r * nunits + p];
    o.x = fma(sc, a[0][0][0], o.x);
    o.y = fma(sc, a[0][0][1], o.y);
    y[r * nunits + p] = o;
}

// A vector of the basis in FP64.
__global__ void __launch_bounds__(FT) k_fix_expand(const int4* __restrict__ v, const int* __restrict__ vexp,
                                                   double2* __restrict__ out, long long nunits) {
    const long long p = (long long)blockIdx.x * FT + threadIdx.x;
    if (p >= nunits) return;
    const int i = blockIdx.y;
    const int4 q = v[i * nunits + p];
    const double pow = scalbn(1.0, vexp[i] - 1022 - 58);
    out[i * nunits + p] = make_double2(from_fix(re_of(q), pow), from_fix(im_of(q), pow));
}

struct FixSplit {
    int tiles, nchunk, vgroups;
    bool spread;
};
FixSplit fix_split(long long nunits, int J, int nrhs, int num_sms) {
    const long long all = (nunits + FTILE - 1) / FTILE;
    FixSplit f;
    f.spread = all * (J + 1) * nrhs < 128LL * num_sms;
    f.vgroups = f.spread ? J / FV + 1 : J / (kSet * FW) + 1;
    const long long want = std::max<long long>(1, 2LL * num_sms / ((long long)f.vgroups * nrhs));
    f.tiles = (int)std::max<long long>(1, (all + want - 1) / want);
    f.nchunk = (int)((all + f.tiles - 1) / f.tiles);
    return f;
}

}  // namespace

int fix_chunks(long long nunits, int J, int nrhs, int num_sms) { return fix_split(nunits, J, nrhs, num_sms).nchunk; }

cudaError_t launch_fix_dots(int nw, const void* basis, long long basis_rhs, long long vec_stride, int J,
                            const int* vexp, long long vexp_rhs, int* uexp, const void* u, const void* z,
                            long long nunits, int nrhs, int num_sms, void* partial, const int* active,
                            cudaStream_t st) {
    const FixSplit f = fix_split(nunits, J, nrhs, num_sms);
    auto go = [&](auto kernel) {
        kernel<<<dim3(f.nchunk * f.vgroups, nrhs), FT, 0, st>>>((const int4*)basis, basis_rhs, vec_stride, J, vexp,
                                                                vexp_rhs, uexp, (const double2*)u, (const double2*)z, nunits,
                                                                f.tiles, f.nchunk, f.vgroups, (double2*)partial, active);
        return cudaGetLastError();
    };
    if (nw == 1) return f.spread ? go(k_fix_dots<1, true>) : go(k_fix_dots<1, false>);
    return f.spread ? go(k_fix_dots<2, true>) : go(k_fix_dots<2, false>);
}

cudaError_t launch_fix_update(void* basis, long long basis_rhs, long long vec_stride, int J, int* vexp,
                              long long vexp_rhs, const int* uexp, int* uexpn, const void* sums, long long s_rhs,
                              int nchunk, void* u, const void* z, long long nunits, int nrhs, int num_sms, const FineStep& fs,
                              cudaStream_t st) {
    const long long wide = (nunits + FT - 1) / FT * nrhs;  // blocks of one unit per thread
    auto go = [&](auto kernel, int E, int SPLIT) -> cudaError_t {
        const size_t smem = (size_t)(2 * ((J + 4 * SPLIT - 1) / (4 * SPLIT) * (4 * SPLIT)) + 2) * sizeof(double2);
        const cudaError_t e = allow_smem((const void*)kernel, smem);
        if (e != cudaSuccess) return e;
        const long long per = (long long)(SPLIT == 1 ? FT : 32) * E, tiles = (nunits + per - 1) / per;
        const int ncol = (J + 1 + FW - 1) / FW;
        // where every block adds the chunks: as many blocks as are resident
        const long long room = nchunk > 1 ? std::max<long long>(1, 3LL * num_sms / nrhs) : tiles;
        const long long each = (tiles + room - 1) / room;
        const int nupd = (int)((tiles + each - 1) / each);
        kernel<<<dim3(nupd + ncol, nrhs), FT, smem, st>>>((int4*)basis, basis_rhs, vec_stride, J, vexp, vexp_rhs, uexp,
                                                          uexpn, (const double2*)sums, s_rhs, nchunk, (double2*)u,
                                                          (const double2*)z, nunits, nupd, fs);
        return cudaGetLastError();
    };
    if (wide >= 2LL * num_sms) return go(k_fix_update<1, 1>, 1, 1);
    if (wide * 8 > 3LL * num_sms) return go(k_fix_update<2, 8>, 2, 8);
    return go(k_fix_update<1, 8>, 1, 8);
}

cudaError_t launch_fine_combine(const void* basis, long long basis_rhs, long long vec_stride, int J, const int* Jdev,
                                const int* vexp, long long vexp_rhs, const void* coef, long long coef_stride,
                                double alpha, void* y, long long nunits, int nrhs, int num_sms, cudaStream_t st) {
    auto go = [&](auto kernel, int SPLIT) -> cudaError_t {
        const size_t smem = (size_t)((J + 4 * SPLIT - 1) / (4 * SPLIT) * (4 * SPLIT)) * sizeof(double2);
        const cudaError_t e = allow_smem((const void*)kernel, smem);
        if (e != cudaSuccess) return e;
        const int per = SPLIT == 1 ? FT : 32;
        kernel<<<dim3((unsigned)((nunits + per - 1) / per), nrhs), FT, smem, st>>>(
            (const int4*)basis, basis_rhs, vec_stride, J, Jdev, vexp, vexp_rhs, (const double2*)coef, coef_stride,
            alpha, (double2*)y, nunits);
        return cudaGetLastError();
    };
    if ((nunits + FT - 1) / FT * nrhs >= 2LL * num_sms) return go(k_fix_combine<1>, 1);
    return go(k_fix_combine<8>, 8);
}

cudaError_t launch_fix_expand(const void* v, const int* vexp, int n, void* out, long long nunits, cudaStream_t st) {
    k_fix_expand<<<dim3((unsigned)((nunits + FT - 1) / FT), n), FT, 0, st>>>((const int4*)v, vexp, (double2*)out, nunits);
    return cudaGetLastError();
}

}  // namespace ovs
