// K1: the Wilson-Dirac stencil at chemical potential, H_w(mu) = gamma5 D_w(mu)
// (Sec. 2, Eqs. Dov and Dw), and K7: field layout conversions.
//
// A thread block is a tile of sites (threadIdx.x) times a tile of
// right-hand sides (threadIdx.y): the warps of one block work on the same
// sites for different right-hand sides, so a link reaches shared L1 once per
// block and not once per right-hand side. A thread may in addition take RT
// right-hand sides (RT = 1 or 2), loading each link once for them. Each of
// the eight hops projects
// the neighbour's 4-spinor onto the rank-2 subspace of (1 -/+ gamma_nu)
// (a 2 x 3 half spinor), multiplies the two colour vectors by U (forward)
// or U^+ (backward), scales by kappa-independent factors (e^{+/-mu} on
// temporal hops, -1 on hops that wrap in t) and adds the reconstructed
// 4-spinor. The diagonal term and gamma5 are applied in the store.
//
// Chiral basis: gamma_k = [[0, -i s_k], [i s_k, 0]], gamma_4 = [[0,1],[1,0]],
// so with upper = spins (0,1) and lower = spins (2,3):
//   (1 - gamma_k) psi = [h; -i s_k h],   h = psi_up + i s_k psi_dn
//   (1 + gamma_k) psi = [h;  i s_k h],   h = psi_up - i s_k psi_dn
//   (1 - gamma_4) psi = [h; -h],         h = psi_up - psi_dn
//   (1 + gamma_4) psi = [h;  h],         h = psi_up + psi_dn
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace ovs {

// ------------------------------------------------------------- field access
template <typename R> struct Field;
template <> struct Field<double> {
    __device__ __forceinline__ static void load(const void* f, int V, int s, cd (&p)[12]) {
        const double2* d = static_cast<const double2*>(f);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const double2* u = d + 2 * ((size_t)q * V + s);
            double2 a = __ldg(u), b = __ldg(u + 1);
            p[2 * q] = {a.x, a.y};
            p[2 * q + 1] = {b.x, b.y};
        }
    }
    __device__ __forceinline__ static void store(void* f, int V, int s, const cd (&p)[12]) {
        double2* d = static_cast<double2*>(f);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            double2* u = d + 2 * ((size_t)q * V + s);
            u[0] = make_double2(p[2 * q].re, p[2 * q].im);
            u[1] = make_double2(p[2 * q + 1].re, p[2 * q + 1].im);
        }
    }
    // row a of U (fwd) or column a of U
    __device__ __forceinline__ static void row(const void* u, int V, int nu, int s, int a, bool fwd, cd (&m)[3]) {
        const double2* d = static_cast<const double2*>(u) + (size_t)nu * 9 * V;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const double2 v = __ldg(d + (size_t)(fwd ? 3 * a + b : 3 * b + a) * V + s);
            m[b] = {v.x, v.y};
        }
    }
    __device__ __forceinline__ static void link(const void* u, int V, int nu, int s, cd (&m)[9]) {
        const double2* d = static_cast<const double2*>(u) + (size_t)nu * 9 * V;
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            double2 v = __ldg(d + (size_t)e * V + s);
            m[e] = {v.x, v.y};
        }
    }
};
template <> struct Field<float> {
    __device__ __forceinline__ static void load(const void* f, int V, int s, cf (&p)[12]) {
        const float4* d = static_cast<const float4*>(f);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            float4 v = __ldg(d + (size_t)q * V + s);
            p[2 * q] = {v.x, v.y};
            p[2 * q + 1] = {v.z, v.w};
        }
    }
    __device__ __forceinline__ static void store(void* f, int V, int s, const cf (&p)[12]) {
        float4* d = static_cast<float4*>(f);
#pragma unroll
        for (int q = 0; q < 6; ++q)
            d[(size_t)q * V + s] = make_float4(p[2 * q].re, p[2 * q].im, p[2 * q + 1].re, p[2 * q + 1].im);
    }
    // complex64 links: per direction four float4 planes holding the entries
    // (0,1) (2,3) (4,5) (6,7) of U (row-major 3x3), at float4 plane 4 nu + q;
    // the ninth entry of every direction in float2 planes after those 16
    // planes (float2 plane 32 + nu). Five loads per link instead of nine.
    __device__ __forceinline__ static void row(const void* u, int V, int nu, int s, int a, bool fwd, cf (&m)[3]) {
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int e = fwd ? 3 * a + b : 3 * b + a;
            const size_t at = e < 8 ? 2 * ((size_t)(nu * 4 + e / 2) * V + s) + (e & 1) : (size_t)(32 + nu) * V + s;
            const float2 v = __ldg(static_cast<const float2*>(u) + at);
            m[b] = {v.x, v.y};
        }
    }
    __device__ __forceinline__ static void link(const void* u, int V, int nu, int s, cf (&m)[9]) {
        const float4* d = static_cast<const float4*>(u) + (size_t)nu * 4 * V;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 v = __ldg(d + (size_t)q * V + s);
            m[2 * q] = {v.x, v.y};
            m[2 * q + 1] = {v.z, v.w};
        }
        const float2 w = __ldg(static_cast<const float2*>(u) + (size_t)(32 + nu) * V + s);
        m[8] = {w.x, w.y};
    }
};

// --------------------------------------------------------------------- hops
// Forward hop: acc += (1 - gamma_NU) * fac * U * psi
template <int NU, typename R>
__device__ __forceinline__ void hop_fwd(const cplx<R> (&p)[12], const cplx<R> (&U)[9], R fac, cplx<R> (&acc)[12]) {
    cplx<R> h0[3], h1[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const cplx<R> a0 = p[c], a1 = p[3 + c], a2 = p[6 + c], a3 = p[9 + c];
        if (NU == 0) { h0[c] = a0 + ti(a3); h1[c] = a1 + ti(a2); }
        if (NU == 1) { h0[c] = a0 + a3;     h1[c] = a1 - a2; }
        if (NU == 2) { h0[c] = a0 + ti(a2); h1[c] = a1 - ti(a3); }
        if (NU == 3) { h0[c] = a0 - a2;     h1[c] = a1 - a3; }
        if (NU == 3) {  // fac is 1 on spatial hops
            h0[c] = h0[c] * fac;
            h1[c] = h1[c] * fac;
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        cplx<R> u0 = {R(0), R(0)}, u1 = {R(0), R(0)};
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            cfma(u0, U[3 * a + b], h0[b]);
            cfma(u1, U[3 * a + b], h1[b]);
        }
        acc[a] = acc[a] + u0;
        acc[3 + a] = acc[3 + a] + u1;
        if (NU == 0) { acc[6 + a] = acc[6 + a] + tmi(u1); acc[9 + a] = acc[9 + a] + tmi(u0); }
        if (NU == 1) { acc[6 + a] = acc[6 + a] - u1;      acc[9 + a] = acc[9 + a] + u0; }
        if (NU == 2) { acc[6 + a] = acc[6 + a] + tmi(u0); acc[9 + a] = acc[9 + a] + ti(u1); }
        if (NU == 3) { acc[6 + a] = acc[6 + a] - u0;      acc[9 + a] = acc[9 + a] - u1; }
    }
}

// Backward hop: acc += (1 + gamma_NU) * fac * U^+ * psi, U the link of the
// backward neighbour in direction NU.
template <int NU, typename R>
__device__ __forceinline__ void hop_bwd(const cplx<R> (&p)[12], const cplx<R> (&U)[9], R fac, cplx<R> (&acc)[12]) {
    cplx<R> h0[3], h1[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const cplx<R> a0 = p[c], a1 = p[3 + c], a2 = p[6 + c], a3 = p[9 + c];
        if (NU == 0) { h0[c] = a0 + tmi(a3); h1[c] = a1 + tmi(a2); }
        if (NU == 1) { h0[c] = a0 - a3;      h1[c] = a1 + a2; }
        if (NU == 2) { h0[c] = a0 + tmi(a2); h1[c] = a1 + ti(a3); }
        if (NU == 3) { h0[c] = a0 + a2;      h1[c] = a1 + a3; }
        if (NU == 3) {  // fac is 1 on spatial hops
            h0[c] = h0[c] * fac;
            h1[c] = h1[c] * fac;
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        cplx<R> u0 = {R(0), R(0)}, u1 = {R(0), R(0)};
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            cfmac(u0, U[3 * b + a], h0[b]);
            cfmac(u1, U[3 * b + a], h1[b]);
        }
        acc[a] = acc[a] + u0;
        acc[3 + a] = acc[3 + a] + u1;
        if (NU == 0) { acc[6 + a] = acc[6 + a] + ti(u1); acc[9 + a] = acc[9 + a] + ti(u0); }
        if (NU == 1) { acc[6 + a] = acc[6 + a] + u1;     acc[9 + a] = acc[9 + a] - u0; }
        if (NU == 2) { acc[6 + a] = acc[6 + a] + ti(u0); acc[9 + a] = acc[9 + a] + tmi(u1); }
        if (NU == 3) { acc[6 + a] = acc[6 + a] + u0;     acc[9 + a] = acc[9 + a] + u1; }
    }
}

// Operands of one hop: the link and the neighbour spinors of the tile.
template <typename R, int RT> struct HopData {
    cplx<R> U[9];
    cplx<R> p[RT][12];
    R fac;
};

// Load the operands of the forward (FWD) or backward hop in direction NU:
// U_NU(s) and psi(s + NU), or U_NU(s - NU) and psi(s - NU); the factor is
// e^{+mu} / e^{-mu} on temporal hops (efwd / ebwd) and -1 on hops that
// wrap in time (antiperiodic).
template <int NU, bool FWD, typename R, int RT>
__device__ __forceinline__ void hop_load(const void* links, const char* in, size_t in_stride, int r0,
                                         const bool (&live)[RT], const Geom& g, int s, int coord, R efwd, R ebwd,
                                         HopData<R, RT>& d) {
    const int L = g.L[NU], st = g.stride[NU];
    int sn;
    if (FWD) {
        sn = (coord == L - 1) ? s - (L - 1) * st : s + st;
        d.fac = (NU == 3 && coord == L - 1) ? -efwd : efwd;
        Field<R>::link(links, g.V, NU, s, d.U);
    } else {
        sn = (coord == 0) ? s + (L - 1) * st : s - st;
        d.fac = (NU == 3 && coord == 0) ? -ebwd : ebwd;
        Field<R>::link(links, g.V, NU, sn, d.U);
    }
#pragma unroll
    for (int i = 0; i < RT; ++i)
        if (live[i]) Field<R>::load(in + (size_t)(r0 + i) * in_stride, g.V, sn, d.p[i]);
}

template <int NU, bool FWD, typename R, int RT>
__device__ __forceinline__ void hop_apply(const HopData<R, RT>& d, const bool (&live)[RT], cplx<R> (&acc)[RT][12]) {
#pragma unroll
    for (int i = 0; i < RT; ++i) {
        if (!live[i]) continue;
        if (FWD)
            hop_fwd<NU>(d.p[i], d.U, d.fac, acc[i]);
        else
            hop_bwd<NU>(d.p[i], d.U, d.fac, acc[i]);
    }
}

// Optional epilogues of the stencil: out = ah * (stencil result) + bx * X + by * Y
// (AX = 1: the Chebyshev filter of the eigensolver set-up), or (stencil
// result) - ps[r].gamma_next X (AX = 2: the block steps of pair_sweeps.cu).
struct Axpy {
    const char* X;
    size_t xs;
    double bx;
    const char* Y;
    size_t ys;
    double by;
    double ah;
    const PairState* ps = nullptr;
};

// out_r = [gamma5] (in_r - kappa * hops(in_r)) for the right-hand sides r
// of the thread. in/out strides are in bytes between right-hand sides.
// Blocks are numbered with the right-hand-side tile fastest, so the blocks
// of all tiles that share a tile of sites (and of links) run back to back.
template <typename R, bool G5, int RT, int AX = 0>
__global__ void __launch_bounds__(256) k_wilson(const void* __restrict__ links, const char* __restrict__ in,
                                                char* out, size_t in_stride, size_t out_stride, Geom g,
                                                R kappa, R emu, R emmu, int nrhs, int ntiles,
                                                const int* __restrict__ active, Axpy ax = Axpy{}) {
    const int tile = blockIdx.x % ntiles;
    const int s = (blockIdx.x / ntiles) * blockDim.x + threadIdx.x;
    const int r0 = (tile * blockDim.y + threadIdx.y) * RT;
    if (s >= g.V || r0 >= nrhs) return;
    bool live[RT];
    bool any = false;
#pragma unroll
    for (int i = 0; i < RT; ++i) {
        live[i] = (r0 + i < nrhs) && (active == nullptr || active[r0 + i] != 0);
        any = any || live[i];
    }
    if (!any) return;
    int c = s;
    const int x = c % g.L[0]; c /= g.L[0];
    const int y = c % g.L[1]; c /= g.L[1];
    const int z = c % g.L[2];
    const int t = c / g.L[2];
    cplx<R> acc[RT][12];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int q = 0; q < 12; ++q) acc[i][q] = {R(0), R(0)};
    // the eight hops in a two-deep pipeline (RT = 1): the operands of the next
    // hop are loaded before the current one is computed
    HopData<R, RT> A, B;
    const R one = R(1);
    if (RT > 1) {  // registers of two RT-tiles in flight would spill: one hop at a time
        hop_load<0, true>(links, in, in_stride, r0, live, g, s, x, one, one, A);
        hop_apply<0, true>(A, live, acc);
        hop_load<0, false>(links, in, in_stride, r0, live, g, s, x, one, one, A);
        hop_apply<0, false>(A, live, acc);
        hop_load<1, true>(links, in, in_stride, r0, live, g, s, y, one, one, A);
        hop_apply<1, true>(A, live, acc);
        hop_load<1, false>(links, in, in_stride, r0, live, g, s, y, one, one, A);
        hop_apply<1, false>(A, live, acc);
        hop_load<2, true>(links, in, in_stride, r0, live, g, s, z, one, one, A);
        hop_apply<2, true>(A, live, acc);
        hop_load<2, false>(links, in, in_stride, r0, live, g, s, z, one, one, A);
        hop_apply<2, false>(A, live, acc);
        hop_load<3, true>(links, in, in_stride, r0, live, g, s, t, emu, emmu, A);
        hop_apply<3, true>(A, live, acc);
        hop_load<3, false>(links, in, in_stride, r0, live, g, s, t, emu, emmu, A);
        hop_apply<3, false>(A, live, acc);
    } else {
    hop_load<0, true>(links, in, in_stride, r0, live, g, s, x, one, one, A);
    hop_load<0, false>(links, in, in_stride, r0, live, g, s, x, one, one, B);
    hop_apply<0, true>(A, live, acc);
    hop_load<1, true>(links, in, in_stride, r0, live, g, s, y, one, one, A);
    hop_apply<0, false>(B, live, acc);
    hop_load<1, false>(links, in, in_stride, r0, live, g, s, y, one, one, B);
    hop_apply<1, true>(A, live, acc);
    hop_load<2, true>(links, in, in_stride, r0, live, g, s, z, one, one, A);
    hop_apply<1, false>(B, live, acc);
    hop_load<2, false>(links, in, in_stride, r0, live, g, s, z, one, one, B);
    hop_apply<2, true>(A, live, acc);
    hop_load<3, true>(links, in, in_stride, r0, live, g, s, t, emu, emmu, A);
    hop_apply<2, false>(B, live, acc);
    hop_load<3, false>(links, in, in_stride, r0, live, g, s, t, emu, emmu, B);
    hop_apply<3, true>(A, live, acc);
    hop_apply<3, false>(B, live, acc);
    }
#pragma unroll
    for (int i = 0; i < RT; ++i) {
        if (!live[i]) continue;
        const int r = r0 + i;
        cplx<R> p[12];
        Field<R>::load(in + (size_t)r * in_stride, g.V, s, p);
#pragma unroll
        for (int q = 0; q < 12; ++q) {
            cplx<R> v = p[q] - acc[i][q] * kappa;
            if (G5 && q >= 6) v = -v;
            p[q] = v;
        }
        if (AX == 2) {
            cplx<R> xv[12];
            Field<R>::load(ax.X + (size_t)r * ax.xs, g.V, s, xv);
            const R gm = R(ax.ps[r].gamma_next);
#pragma unroll
            for (int q = 0; q < 12; ++q) p[q] = p[q] - xv[q] * gm;
        }
        if (AX == 1) {
            cplx<R> xv[12], yv[12];
            Field<R>::load(ax.X + (size_t)r * ax.xs, g.V, s, xv);
            Field<R>::load(ax.Y + (size_t)r * ax.ys, g.V, s, yv);
            const R ah = R(ax.ah), bx = R(ax.bx), by = R(ax.by);
#pragma unroll
            for (int q = 0; q < 12; ++q) p[q] = p[q] * ah + xv[q] * bx + yv[q] * by;
        }
        Field<R>::store(out + (size_t)r * out_stride, g.V, s, p);
    }
}

// The stencil on small fields: a cluster of eight blocks takes 32 sites of one
// right-hand side, one hop each, a warp per colour row of the link, and the
// blocks then add the eight contributions, 48 of the 384 entries each, from each
// other's shared memory. A thread of k_wilson does 1,392 flops in a row, so 4^4
// in FP64 sat on 8 SMs' FP64 units (36 us); here it is spread over 64, and a
// warp, alone on its scheduler at some 20 clocks an instruction, has a
// twentieth of the instructions. The sums run in the order of k_wilson (x+, x-,
// y+, ...; within a hop as there), so the results are the same bit for bit.
// CIN, COUT: in, out are canonical complex128 vectors, so that an operator on
// small fields is one launch without layout passes.
template <int HOP, typename R, bool CIN>
__device__ __forceinline__ void one_hop(const void* links, const char* in, size_t in_stride, int r, const Geom& g,
                                        int s, int coord, R efwd, R ebwd, int a, cplx<R> (&out)[4]) {
    constexpr int NU = HOP / 2;
    constexpr bool FWD = HOP % 2 == 0;
    const int L = g.L[NU], st = g.stride[NU];
    int sn;
    R fac;
    if (FWD) {
        sn = (coord == L - 1) ? s - (L - 1) * st : s + st;
        fac = (NU == 3 && coord == L - 1) ? -efwd : efwd;
    } else {
        sn = (coord == 0) ? s + (L - 1) * st : s - st;
        fac = (NU == 3 && coord == 0) ? -ebwd : ebwd;
    }
    cplx<R> U[3], p[12];
    Field<R>::row(links, g.V, NU, FWD ? s : sn, a, FWD, U);
    if (CIN) {
        const double2* x = reinterpret_cast<const double2*>(in + (size_t)r * in_stride) + (size_t)sn * 12;
#pragma unroll
        for (int q = 0; q < 12; ++q) {
            const double2 v = __ldg(x + q);
            p[q] = {R(v.x), R(v.y)};
        }
    } else {
        Field<R>::load(in + (size_t)r * in_stride, g.V, sn, p);
    }
    cplx<R> u0 = {R(0), R(0)}, u1 = {R(0), R(0)};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const cplx<R> a0 = p[c], a1 = p[3 + c], a2 = p[6 + c], a3 = p[9 + c];
        cplx<R> h0, h1;
        if (FWD) {
            if (NU == 0) { h0 = a0 + ti(a3); h1 = a1 + ti(a2); }
            if (NU == 1) { h0 = a0 + a3;     h1 = a1 - a2; }
            if (NU == 2) { h0 = a0 + ti(a2); h1 = a1 - ti(a3); }
            if (NU == 3) { h0 = a0 - a2;     h1 = a1 - a3; }
            if (NU == 3) {
                h0 = h0 * fac;
                h1 = h1 * fac;
            }
            cfma(u0, U[c], h0);
            cfma(u1, U[c], h1);
        } else {
            if (NU == 0) { h0 = a0 + tmi(a3); h1 = a1 + tmi(a2); }
            if (NU == 1) { h0 = a0 - a3;      h1 = a1 + a2; }
            if (NU == 2) { h0 = a0 + tmi(a2); h1 = a1 + ti(a3); }
            if (NU == 3) { h0 = a0 + a2;      h1 = a1 + a3; }
            if (NU == 3) {
                h0 = h0 * fac;
                h1 = h1 * fac;
            }
            cfmac(u0, U[c], h0);
            cfmac(u1, U[c], h1);
        }
    }
    out[0] = u0;
    out[1] = u1;
    if (NU == 0) { out[2] = FWD ? tmi(u1) : ti(u1); out[3] = FWD ? tmi(u0) : ti(u0); }
    if (NU == 1) { out[2] = FWD ? -u1 : u1;         out[3] = FWD ? u0 : -u0; }
    if (NU == 2) { out[2] = FWD ? tmi(u0) : ti(u0); out[3] = FWD ? ti(u1) : tmi(u1); }
    if (NU == 3) { out[2] = FWD ? -u0 : u0;         out[3] = FWD ? -u1 : u1; }
}

template <typename R, bool G5, int AX, bool CIN, bool COUT>
__global__ void __cluster_dims__(8, 1, 1) __launch_bounds__(96)
    k_wilson_split(const void* __restrict__ links, const char* __restrict__ in, char* out, size_t in_stride,
                   size_t out_stride, Geom g, R kappa, R emu, R emmu, const int* __restrict__ active, Axpy ax) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ cplx<R> part[12][32];
    const int r = blockIdx.y, hop = (int)cl.block_rank(), lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    if (active != nullptr && active[r] == 0) return;  // uniform over the cluster
    const int s0 = (int)(blockIdx.x / 8) * 32;
    const int s = min(s0 + lane, g.V - 1);
    int c = s;
    const int x = c % g.L[0]; c /= g.L[0];
    const int y = c % g.L[1]; c /= g.L[1];
    const int z = c % g.L[2];
    const int t = c / g.L[2];
    cplx<R> o[4];
    const R one = R(1);
    switch (hop) {
        case 0: one_hop<0, R, CIN>(links, in, in_stride, r, g, s, x, one, one, row, o); break;
        case 1: one_hop<1, R, CIN>(links, in, in_stride, r, g, s, x, one, one, row, o); break;
        case 2: one_hop<2, R, CIN>(links, in, in_stride, r, g, s, y, one, one, row, o); break;
        case 3: one_hop<3, R, CIN>(links, in, in_stride, r, g, s, y, one, one, row, o); break;
        case 4: one_hop<4, R, CIN>(links, in, in_stride, r, g, s, z, one, one, row, o); break;
        case 5: one_hop<5, R, CIN>(links, in, in_stride, r, g, s, z, one, one, row, o); break;
        case 6: one_hop<6, R, CIN>(links, in, in_stride, r, g, s, t, emu, emmu, row, o); break;
        default: one_hop<7, R, CIN>(links, in, in_stride, r, g, s, t, emu, emmu, row, o); break;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) part[3 * q + row][lane] = o[q];
    cl.sync();
    const cplx<R>* src = reinterpret_cast<const cplx<R>*>(in + (size_t)r * in_stride);
    cplx<R>* dst = reinterpret_cast<cplx<R>*>(out + (size_t)r * out_stride);
    const int idx = hop * 48 + (int)threadIdx.x;  // this block adds 48 of the 384 entries
    const int q = idx >> 5, at = idx & 31;
    if (threadIdx.x < 48 && s0 + at < g.V) {
        cplx<R> a = {R(0), R(0)};
#pragma unroll
        for (int h = 0; h < 8; ++h) a = a + cl.map_shared_rank(&part[0][0], h)[q * 32 + at];
        const size_t e = 2 * ((size_t)(q >> 1) * g.V + s0 + at) + (q & 1);  // entry q of the site
        const size_t ec = (size_t)(s0 + at) * 12 + q;                     // and in a canonical vector
        cplx<R> own;
        if (CIN) {
            const double2 x0 = reinterpret_cast<const double2*>(in + (size_t)r * in_stride)[ec];
            own = {R(x0.x), R(x0.y)};
        } else {
            own = src[e];
        }
        cplx<R> v = own - a * kappa;
        if (G5 && q >= 6) v = -v;
        if (AX == 2) v = v - reinterpret_cast<const cplx<R>*>(ax.X + (size_t)r * ax.xs)[e] * R(ax.ps[r].gamma_next);
        if (AX == 1) {
            const cplx<R> xv = reinterpret_cast<const cplx<R>*>(ax.X + (size_t)r * ax.xs)[e];
            const cplx<R> yv = reinterpret_cast<const cplx<R>*>(ax.Y + (size_t)r * ax.ys)[e];
            v = v * R(ax.ah) + xv * R(ax.bx) + yv * R(ax.by);
        }
        if (COUT) reinterpret_cast<double2*>(out + (size_t)r * out_stride)[ec] = make_double2(double(v.re), double(v.im));
        else dst[e] = v;
    }
    cl.sync();  // no block leaves while another reads its part
}

// Flat precision conversion of internal fields (the two layouts pair up).
__global__ void k_f64_to_f32(const double2* __restrict__ a, float2* __restrict__ b, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double2 v = a[i];
        b[i] = make_float2(float(v.x), float(v.y));
    }
}
__global__ void k_f32_to_f64(const float2* __restrict__ a, double2* __restrict__ b, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float2 v = a[i];
        b[i] = make_double2(double(v.x), double(v.y));
    }
}

// Uniform (-1, 1) real and imaginary parts from a 64-bit mixing hash of
// (seed, index) (splitmix64 finaliser); used for random starting blocks.
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}
__global__ void k_random_fill(double2* __restrict__ q, long long n, uint64_t seed) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const uint64_t a = mix64(seed * 0x9E3779B97F4A7C15ULL + 2 * (uint64_t)i + 1);
        const uint64_t b = mix64(a + 0x632BE59BD9B4E019ULL);
        q[i] = make_double2(((a >> 11) + 0.5) * 0x1p-52 - 1.0, ((b >> 11) + 0.5) * 0x1p-52 - 1.0);
    }
}

// ------------------------------------------------------------ layouts (K7)
// A block takes LT sites. The canonical side is read and written in its own
// order, 16 bytes per lane in a row, and the sites' twelve entries meet in shared
// memory at a pitch of 13 (8 lanes then fall on 8 different 16-byte groups of
// banks). Read site by site instead, a warp's load touched 32 lines for 512
// bytes: 3.3 TB/s over the two passes of a 16-source operator at 16^3 x 32.
constexpr int LT = 128;

// canonical complex128 [nrhs][V][12]  ->  internal planes of precision R
template <typename R>
__global__ void __launch_bounds__(LT) k_to_internal(const double2* __restrict__ canon, size_t canon_stride,
                                                    char* __restrict__ out, size_t out_stride, int V) {
    __shared__ cplx<R> sm[LT * 13];
    const int s0 = blockIdx.x * LT, r = blockIdx.y, tid = threadIdx.x;
    const int n = min(LT, V - s0) * 12;
    const double2* src = canon + r * canon_stride + (size_t)s0 * 12;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const int i = k * LT + tid;
        if (i < n) {
            const double2 v = __ldcs(src + i);
            sm[i / 12 * 13 + i % 12] = {R(v.x), R(v.y)};
        }
    }
    __syncthreads();
    if (s0 + tid >= V) return;
    cplx<R> p[12];
#pragma unroll
    for (int q = 0; q < 12; ++q) p[q] = sm[tid * 13 + q];
    Field<R>::store(out + r * out_stride, V, s0 + tid, p);
}

// internal planes of precision R -> canonical complex128; OV (R = double): D_ov(mu)
// y = x + gamma5 sgn(H_w) x (Sec. 2, Eq. Dov) fused into this last pass, with x
// the canonical source: gamma5 = diag(1, 1, -1, -1) flips the entries of spin 2
// and 3 (spin*3 + colour >= 6).
template <typename R, bool OV>
__global__ void __launch_bounds__(LT) k_to_canonical(const char* __restrict__ in, size_t in_stride,
                                                     const double2* __restrict__ x, size_t x_stride,
                                                     double2* __restrict__ canon, size_t canon_stride, int V) {
    __shared__ cplx<R> sm[LT * 13];
    const int s0 = blockIdx.x * LT, r = blockIdx.y, tid = threadIdx.x;
    if (s0 + tid < V) {
        cplx<R> p[12];
        Field<R>::load(in + r * in_stride, V, s0 + tid, p);
#pragma unroll
        for (int q = 0; q < 12; ++q) sm[tid * 13 + q] = p[q];
    }
    __syncthreads();
    const int n = min(LT, V - s0) * 12;
    double2* dst = canon + r * canon_stride + (size_t)s0 * 12;
    const double2* xs = OV ? x + r * x_stride + (size_t)s0 * 12 : nullptr;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const int i = k * LT + tid;
        if (i < n) {
            const cplx<R> p = sm[i / 12 * 13 + i % 12];
            if (OV) {
                const double2 xv = xs[i];
                const double g = i % 12 < 6 ? 1.0 : -1.0;
                dst[i] = make_double2(fma(g, double(p.re), xv.x), fma(g, double(p.im), xv.y));
            } else {
                dst[i] = make_double2(double(p.re), double(p.im));
            }
        }
    }
}

// canonical links complex128 [V][4][3][3] -> planes [nu][e][V] (complex128 and,
// if u32 != nullptr, complex64)
__global__ void k_links_to_internal(const double2* __restrict__ canon, double2* __restrict__ u64,
                                    float2* __restrict__ u32, int V) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
#pragma unroll
    for (int nu = 0; nu < 4; ++nu)
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            double2 v = canon[((size_t)s * 4 + nu) * 9 + e];
            u64[((size_t)nu * 9 + e) * V + s] = v;
            if (u32 != nullptr) {  // complex64 layout of Field<float>::link
                const size_t i = e < 8 ? ((size_t)(nu * 4 + e / 2) * V + s) * 2 + (e & 1) : (size_t)(32 + nu) * V + s;
                u32[i] = make_float2(float(v.x), float(v.y));
            }
        }
}

__global__ void k_links_to_canonical(const double2* __restrict__ u64, double2* __restrict__ canon, int V) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
#pragma unroll
    for (int nu = 0; nu < 4; ++nu)
#pragma unroll
        for (int e = 0; e < 9; ++e) canon[((size_t)s * 4 + nu) * 9 + e] = u64[((size_t)nu * 9 + e) * V + s];
}

// ------------------------------------------------------------- host launch
// The complex128 stencil by two threads per site. A scheduler takes an FP64
// operation of a warp every 64 clocks, so the 936 operations of a site in one
// thread are 31 us however small the field, and a field that fills the chip
// unevenly pays a whole such wave for the rest. Thread `half` takes component
// half of the half-spinor of every hop: one spin and its partner of the neighbour,
// one upper spin of the sum, and the lower spin that this component goes to in x
// and y; for z and t it is the other thread's, so the two exchange their lower
// sums between y and z. Every entry is summed in the order of k_wilson (the same
// bits). The two halves are warps of a block (no divergence).
// Measured, k_wilson and this: see the rule in wilson_dispatch.
template <int NU, bool FWD, int HALF>
__device__ __forceinline__ void half_hop(const void* links, const char* in, const Geom& g, int s, int coord,
                                         double efwd, double ebwd, cd (&up)[3], cd (&lo)[3]) {
    const int L = g.L[NU], st = g.stride[NU];
    int sn;
    double fac;
    cd U[9];
    if (FWD) {
        sn = (coord == L - 1) ? s - (L - 1) * st : s + st;
        fac = (NU == 3 && coord == L - 1) ? -efwd : efwd;
        Field<double>::link(links, g.V, NU, s, U);
    } else {
        sn = (coord == 0) ? s + (L - 1) * st : s - st;
        fac = (NU == 3 && coord == 0) ? -ebwd : ebwd;
        Field<double>::link(links, g.V, NU, sn, U);
    }
    constexpr int P = NU < 2 ? 3 - HALF : 2 + HALF;  // the partner spin
    const double2* d = reinterpret_cast<const double2*>(in);
    cd h[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int e = 3 * HALF + c, q = 3 * P + c;
        const double2 av = __ldg(d + 2 * ((size_t)(e >> 1) * g.V + sn) + (e & 1));
        const double2 bv = __ldg(d + 2 * ((size_t)(q >> 1) * g.V + sn) + (q & 1));
        const cd a = {av.x, av.y}, b = {bv.x, bv.y};
        if (NU == 0) h[c] = FWD ? a + ti(b) : a + tmi(b);
        if (NU == 1) h[c] = FWD == (HALF == 0) ? a + b : a - b;
        if (NU == 2) h[c] = FWD == (HALF == 0) ? a + ti(b) : a + tmi(b);
        if (NU == 3) h[c] = FWD ? a - b : a + b;
        if (NU == 3) h[c] = h[c] * fac;  // 1 on spatial hops
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        cd u = {0.0, 0.0};
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            if (FWD)
                cfma(u, U[3 * a + b], h[b]);
            else
                cfmac(u, U[3 * b + a], h[b]);
        }
        up[a] = up[a] + u;
        if (NU == 0) lo[a] = FWD ? lo[a] + tmi(u) : lo[a] + ti(u);
        if (NU == 1) lo[a] = FWD == (HALF == 0) ? lo[a] + u : lo[a] - u;
        if (NU == 2) lo[a] = FWD == (HALF == 0) ? lo[a] + tmi(u) : lo[a] + ti(u);
        if (NU == 3) lo[a] = FWD ? lo[a] - u : lo[a] + u;
    }
}

template <bool G5>
__global__ void __launch_bounds__(512) k_wilson_half(const void* __restrict__ links, const char* __restrict__ in,
                                                     char* out, size_t in_stride, size_t out_stride, Geom g,
                                                     double kappa, double emu, double emmu, int nrhs, int ntiles,
                                                     const int* __restrict__ active) {
    __shared__ cd swap[2][3][256];
    const int tile = blockIdx.x % ntiles, sites = 16 * blockDim.y;
    const int half = threadIdx.y & 1, slot = (threadIdx.y >> 1) * 32 + threadIdx.x;
    const int s0 = (blockIdx.x / ntiles) * sites + slot, s = min(s0, g.V - 1);
    const int r = tile * blockDim.z + threadIdx.z, sl = threadIdx.z * sites + slot;
    const bool live = r < nrhs && (active == nullptr || active[r] != 0);
    const char* ir = in + (size_t)min(r, nrhs - 1) * in_stride;
    int c = s;
    const int x = c % g.L[0]; c /= g.L[0];
    const int y = c % g.L[1]; c /= g.L[1];
    const int z = c % g.L[2];
    const int t = c / g.L[2];
    cd up[3], lo[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) up[a] = lo[a] = {0.0, 0.0};
    auto xy = [&](auto h) {
        constexpr int H = decltype(h)::value;
        half_hop<0, true, H>(links, ir, g, s, x, 1.0, 1.0, up, lo);
        half_hop<0, false, H>(links, ir, g, s, x, 1.0, 1.0, up, lo);
        half_hop<1, true, H>(links, ir, g, s, y, 1.0, 1.0, up, lo);
        half_hop<1, false, H>(links, ir, g, s, y, 1.0, 1.0, up, lo);
    };
    auto zt = [&](auto h) {
        constexpr int H = decltype(h)::value;
        half_hop<2, true, H>(links, ir, g, s, z, 1.0, 1.0, up, lo);
        half_hop<2, false, H>(links, ir, g, s, z, 1.0, 1.0, up, lo);
        half_hop<3, true, H>(links, ir, g, s, t, emu, emmu, up, lo);
        half_hop<3, false, H>(links, ir, g, s, t, emu, emmu, up, lo);
        // own entries: spin H and, after the exchange, spin 2 + H
        if (s0 >= g.V) return;
        const double2* d = reinterpret_cast<const double2*>(ir);
        double2* o = reinterpret_cast<double2*>(out + (size_t)r * out_stride);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const int e = k < 3 ? 3 * H + k : 6 + 3 * H + k - 3;
            const size_t at = 2 * ((size_t)(e >> 1) * g.V + s) + (e & 1);
            const double2 pv = __ldg(d + at);
            cd v = cd{pv.x, pv.y} - (k < 3 ? up[k % 3] : lo[k % 3]) * kappa;
            if (G5 && e >= 6) v = -v;
            o[at] = make_double2(v.re, v.im);
        }
    };
    if (live) {
        if (half == 0)
            xy(std::integral_constant<int, 0>{});
        else
            xy(std::integral_constant<int, 1>{});
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) swap[half][a][sl] = lo[a];
    __syncthreads();
    if (!live) return;
#pragma unroll
    for (int a = 0; a < 3; ++a) lo[a] = swap[1 - half][a][sl];
    if (half == 0)
        zt(std::integral_constant<int, 0>{});
    else
        zt(std::integral_constant<int, 1>{});
}

static inline dim3 site_grid(int V, int nrhs, int threads) { return dim3((V + threads - 1) / threads, nrhs); }

// Groups of 32 sites and right-hand sides up to which the stencil is spread
// over the hops as well (k_wilson_split). Measured, k_wilson and split: FP64
// 8 groups 36 and 14 us, 90 37 and 16, 512 39 and 56; complex64 128 groups 9.2
// and 9.5 us.
template <typename R> constexpr long long kSplitGroups = sizeof(R) == 8 ? 256 : 96;
// The same where it also replaces the two layout passes (canonical vectors on both
// sides). Measured, three launches and one: complex64 128 groups 14.4 and 10.4 us,
// 164 14.4 and 14.4 (H_w^2 20.6 and 24.7); FP64 384 groups 43.1 and 41.1 us (77.9
// and 82.1), 512 44.9 and 51.4.
template <typename R> constexpr long long kSplitCanonical = sizeof(R) == 8 ? 256 : 144;

// Where the complex128 stencil takes two threads per site (k_wilson_half): the
// warps of 32 sites fill the FP64 schedulers (four per SM, 608 here) less than once, or
// half warps fill them in fewer half waves. Measured per H_w with both layout passes,
// k_wilson and half: 384 warps 44.6 and 37.0 us, 512 45.2 and 43.2, 640 61.5 and
// 54.5, 1280 98.5 and 90.2, 2592 178.9 and 164.0; where the half waves are as many
// (1024) 71.8 and 75.3, (16384) 926.7 and 928.5.
static bool two_threads_per_site(long long warps) {
    const long long n = 4LL * device_sms();
    return warps <= n || (2 * warps + n - 1) / n < 2 * ((warps + n - 1) / n);
}

static bool valid_shape(const StencilShape& sh) {
    for (int i = 0; i < kNumStencilShapes; ++i)
        if (kStencilShapes[i].rt == sh.rt && kStencilShapes[i].sites == sh.sites && kStencilShapes[i].rb == sh.rb)
            return true;
    return false;
}

template <typename R, bool G5, int AX>
static void wilson_dispatch(const StencilShape& sh, unsigned blocks, int ntiles, cudaStream_t st, const void* links,
                            const void* in, size_t in_stride, void* out, size_t out_stride, const Geom& g,
                            double kappa, double emu, double emmu, int nrhs, const int* active, const Axpy& ax) {
    const R k = (R)kappa, e1 = (R)emu, e2 = (R)emmu;
    const char* i = (const char*)in;
    char* o = (char*)out;
    const long long groups = (g.V + 31) / 32;
    if (groups * nrhs <= kSplitGroups<R> && nrhs <= 65535) {
        k_wilson_split<R, G5, AX, false, false><<<dim3((unsigned)(8 * groups), nrhs), 96, 0, st>>>(links, i, o, in_stride, out_stride,
                                                                                    g, k, e1, e2, active, ax);
        return;
    }
    if constexpr (sizeof(R) == 8 && AX == 0) {
        if (sh.rt == 1 && two_threads_per_site(groups * nrhs)) {
            k_wilson_half<G5><<<blocks, dim3(32, sh.sites / 16, sh.rb), 0, st>>>(links, i, o, in_stride, out_stride, g,
                                                                               kappa, emu, emmu, nrhs, ntiles, active);
            return;
        }
    }
    const dim3 block(sh.sites, sh.rb);
    if (sh.rt == 1)
        k_wilson<R, G5, 1, AX><<<blocks, block, 0, st>>>(links, i, o, in_stride, out_stride, g, k, e1, e2, nrhs, ntiles,
                                                           active, ax);
    else
        k_wilson<R, G5, 2, AX><<<blocks, block, 0, st>>>(links, i, o, in_stride, out_stride, g, k, e1, e2, nrhs, ntiles,
                                                           active, ax);
}

cudaError_t launch_wilson(int prec, bool gamma5, const void* links, const void* in, size_t in_stride, void* out,
                          size_t out_stride, const Geom& g, int nrhs, double kappa, double mu, const int* active,
                          cudaStream_t st, StencilShape sh) {
    if (!valid_shape(sh)) return cudaErrorInvalidValue;
    const int ntiles = (nrhs + sh.rt * sh.rb - 1) / (sh.rt * sh.rb);
    const long long blocks = (long long)ntiles * ((g.V + sh.sites - 1) / sh.sites);
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    const double emu = exp(mu), emmu = exp(-mu);
    const Axpy ax{};
    if (prec == PREC_F64) {
        if (gamma5)
            wilson_dispatch<double, true, 0>(sh, (unsigned)blocks, ntiles, st, links, in, in_stride, out,
                                                 out_stride, g, kappa, emu, emmu, nrhs, active, ax);
        else
            wilson_dispatch<double, false, 0>(sh, (unsigned)blocks, ntiles, st, links, in, in_stride, out,
                                                  out_stride, g, kappa, emu, emmu, nrhs, active, ax);
    } else {
        if (gamma5)
            wilson_dispatch<float, true, 0>(sh, (unsigned)blocks, ntiles, st, links, in, in_stride, out,
                                                out_stride, g, kappa, emu, emmu, nrhs, active, ax);
        else
            wilson_dispatch<float, false, 0>(sh, (unsigned)blocks, ntiles, st, links, in, in_stride, out,
                                                 out_stride, g, kappa, emu, emmu, nrhs, active, ax);
    }
    return cudaGetLastError();
}

cudaError_t launch_wilson_axpy(int prec, const void* links, const void* in, size_t in_stride, void* out,
                               size_t out_stride, const void* X, size_t xs, double bx, const void* Y, size_t ys,
                               double by, double ah, const Geom& g, int nrhs, double kappa, double mu,
                               cudaStream_t st, StencilShape sh) {
    if (!valid_shape(sh)) return cudaErrorInvalidValue;
    const int ntiles = (nrhs + sh.rt * sh.rb - 1) / (sh.rt * sh.rb);
    const long long blocks = (long long)ntiles * ((g.V + sh.sites - 1) / sh.sites);
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    const double emu = exp(mu), emmu = exp(-mu);
    const Axpy ax{(const char*)X, xs, bx, (const char*)Y, ys, by, ah};
    if (prec == PREC_F64)
        wilson_dispatch<double, true, 1>(sh, (unsigned)blocks, ntiles, st, links, in, in_stride, out, out_stride,
                                            g, kappa, emu, emmu, nrhs, nullptr, ax);
    else
        wilson_dispatch<float, true, 1>(sh, (unsigned)blocks, ntiles, st, links, in, in_stride, out, out_stride,
                                           g, kappa, emu, emmu, nrhs, nullptr, ax);
    return cudaGetLastError();
}

bool wilson_spread(int prec, const Geom& g, int nrhs) {
    return (long long)((g.V + 31) / 32) * nrhs <= (prec == PREC_F64 ? kSplitCanonical<double> : kSplitCanonical<float>);
}

cudaError_t launch_wilson_canonical(int prec, bool gamma5, const void* links, const void* in, size_t in_stride,
                                    bool in_canon, void* out, size_t out_stride, bool out_canon, const Geom& g,
                                    int nrhs, double kappa, double mu, cudaStream_t st) {
    const dim3 grid(8 * ((g.V + 31) / 32), nrhs);
    const double ep = exp(mu), em = exp(-mu);
#define OVS_CANON(R, G5, CI, CO)                                                                                   \
    k_wilson_split<R, G5, 0, CI, CO><<<grid, 96, 0, st>>>(links, (const char*)in, (char*)out, in_stride, out_stride, \
                                                          g, (R)kappa, (R)ep, (R)em, nullptr, Axpy{})
#define OVS_CANON_G5(R, CI, CO)                 \
    do {                                        \
        if (gamma5) OVS_CANON(R, true, CI, CO); \
        else OVS_CANON(R, false, CI, CO);       \
    } while (0)
#define OVS_CANON_R(R)                                        \
    do {                                                      \
        if (in_canon && out_canon) OVS_CANON_G5(R, true, true); \
        else if (in_canon) OVS_CANON_G5(R, true, false);        \
        else OVS_CANON_G5(R, false, true);                      \
    } while (0)
    if (!wilson_spread(prec, g, nrhs) || nrhs > 65535 || !(in_canon || out_canon)) return cudaErrorInvalidValue;
    if (prec == PREC_F64) OVS_CANON_R(double);
    else OVS_CANON_R(float);
#undef OVS_CANON_R
#undef OVS_CANON_G5
#undef OVS_CANON
    return cudaGetLastError();
}

cudaError_t launch_wilson_pair(const void* links, const void* in, size_t in_stride, void* out, size_t out_stride,
                               const void* X, size_t xs, const PairState* ps, const Geom& g, int nrhs, double kappa,
                               double mu, const int* active, cudaStream_t st, StencilShape sh) {
    if (!valid_shape(sh)) return cudaErrorInvalidValue;
    const int ntiles = (nrhs + sh.rt * sh.rb - 1) / (sh.rt * sh.rb);
    const long long blocks = (long long)ntiles * ((g.V + sh.sites - 1) / sh.sites);
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    Axpy ax{};
    ax.X = (const char*)X;
    ax.xs = xs;
    ax.ps = ps;
    wilson_dispatch<float, true, 2>(sh, (unsigned)blocks, ntiles, st, links, in, in_stride, out, out_stride, g, kappa,
                                    exp(mu), exp(-mu), nrhs, active, ax);
    return cudaGetLastError();
}

cudaError_t launch_convert(int to_prec, const void* in, void* out, long long ncplx, cudaStream_t st) {
    const int blocks = (int)std::min<long long>((ncplx + 255) / 256, 8192);
    if (to_prec == PREC_F32)
        k_f64_to_f32<<<blocks, 256, 0, st>>>((const double2*)in, (float2*)out, ncplx);
    else
        k_f32_to_f64<<<blocks, 256, 0, st>>>((const float2*)in, (double2*)out, ncplx);
    return cudaGetLastError();
}

cudaError_t launch_random_fill(void* q, long long ncplx, uint64_t seed, cudaStream_t st) {
    const int blocks = (int)std::min<long long>((ncplx + 255) / 256, 8192);
    k_random_fill<<<blocks, 256, 0, st>>>((double2*)q, ncplx, seed);
    return cudaGetLastError();
}

cudaError_t launch_to_internal(int prec, const void* canon, size_t canon_stride_cplx, void* out, size_t out_stride,
                               int V, int nrhs, cudaStream_t st) {
    const dim3 grid = site_grid(V, nrhs, LT);
    if (prec == PREC_F64)
        k_to_internal<double><<<grid, LT, 0, st>>>((const double2*)canon, canon_stride_cplx, (char*)out, out_stride, V);
    else
        k_to_internal<float><<<grid, LT, 0, st>>>((const double2*)canon, canon_stride_cplx, (char*)out, out_stride, V);
    return cudaGetLastError();
}

cudaError_t launch_to_canonical(int prec, const void* in, size_t in_stride, void* canon, size_t canon_stride_cplx,
                                int V, int nrhs, cudaStream_t st) {
    const dim3 grid = site_grid(V, nrhs, LT);
    if (prec == PREC_F64)
        k_to_canonical<double, false><<<grid, LT, 0, st>>>((const char*)in, in_stride, nullptr, 0, (double2*)canon,
                                                           canon_stride_cplx, V);
    else
        k_to_canonical<float, false><<<grid, LT, 0, st>>>((const char*)in, in_stride, nullptr, 0, (double2*)canon,
                                                          canon_stride_cplx, V);
    return cudaGetLastError();
}

cudaError_t launch_to_canonical_overlap(const void* in, size_t in_stride, const void* x, size_t x_stride_cplx,
                                        void* canon, size_t canon_stride_cplx, int V, int nrhs, cudaStream_t st) {
    k_to_canonical<double, true><<<site_grid(V, nrhs, LT), LT, 0, st>>>(
        (const char*)in, in_stride, (const double2*)x, x_stride_cplx, (double2*)canon, canon_stride_cplx, V);
    return cudaGetLastError();
}

cudaError_t launch_links_to_internal(const void* canon, void* u64, void* u32, int V, cudaStream_t st) {
    k_links_to_internal<<<(V + 127) / 128, 128, 0, st>>>((const double2*)canon, (double2*)u64, (float2*)u32, V);
    return cudaGetLastError();
}

cudaError_t launch_links_to_canonical(const void* u64, void* canon, int V, cudaStream_t st) {
    k_links_to_canonical<<<(V + 127) / 128, 128, 0, st>>>((const double2*)u64, (double2*)canon, V);
    return cudaGetLastError();
}

}  // namespace ovs
