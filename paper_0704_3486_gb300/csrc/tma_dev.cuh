// Device code shared by the TMA sweeps (tma_sweeps.cu, pair_sweeps.cu): bounded
// mbarrier waits, bulk copies, the consumers' barriers and the split of the
// work items.
#pragma once

#include <algorithm>

#include "common.cuh"

namespace ovs {
namespace {

constexpr int TB = 256;       // threads per block
constexpr int TW = TB / 32;   // warps
constexpr int TG = 8;         // basis vectors per stage
// update sweep: 2 units per thread per tile, 3 stages of 64 KB
constexpr int TE = 2;
constexpr int TU = TB * TE;
constexpr int TNS = 3;
constexpr size_t kStageBytes = (size_t)TG * TU * 16;
constexpr unsigned long long kWaitNs = 1000000000ull;  // a wait gives up after 1 s
constexpr int OVS_ETIMEOUT_CODE = -7;        // OVS_ETIMEOUT

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// try_wait until the phase completes or kWaitNs have passed (the clock is
// read only once the first try has failed)
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if (global_ns() - t0 > kWaitNs) return false;
    }
}
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }


constexpr int CU = 2048;                     // units per row chunk
constexpr int DU = 512;                      // units per tile
constexpr int DE = DU / TB;                  // units per consumer thread per tile
constexpr int DNT = CU / DU;                 // tiles per chunk
constexpr int DS = 3;                        // stages
constexpr int DTHREADS = TB + 32;            // consumer warps + producer warp
constexpr size_t kDStage = (size_t)TG * DU * 16;

__device__ __forceinline__ double wsum_d(double v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
// named barrier 1 over the TB consumer threads; the OR of `p` over them
__device__ __forceinline__ bool consumers_sync_or(bool p) {
    uint32_t r;
    asm volatile(
        "{\n .reg .pred a, b;\n setp.ne.u32 a, %1, 0;\n bar.red.or.pred b, 1, %2, a;\n selp.u32 %0, 1, 0, b;\n}"
        : "=r"(r)
        : "r"((uint32_t)p), "n"(TB)
        : "memory");
    return r != 0;
}
__device__ __forceinline__ void consumers_sync() { asm volatile("bar.sync 1, %0;" ::"n"(TB) : "memory"); }
// bounded wait that also gives up once another thread has raised `abort`
__device__ __forceinline__ bool mbar_wait_or_abort(uint64_t* bar, uint32_t parity, volatile int* abort) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if (*abort || global_ns() - t0 > kWaitNs) return false;
    }
}
// block that owns flattened item i under the contiguous split of T items
// over G blocks (block q owns [floor(qT/G), floor((q+1)T/G)))
__host__ __device__ inline int owner_of(long long i, long long T, int G) {
    return (int)(((i + 1) * G - 1) / T);
}
// Work items of a sweep: pieces of `chunk` units of every right-hand side, at
// most `most`, the largest share of a block as close to the mean as pieces of
// a multiple of 32 units allow (156 pieces of 2048 units on 152 blocks took
// twice the time of 152). `piece` is the cost of an item beyond its units, in
// units.
struct Items {
    long long chunk, per_rhs;
    int grid;
};
inline Items balanced_items(long long nunits, int nrhs, int num_sms, int most, int piece) {
    Items best{most, (nunits + most - 1) / most, 0};
    double cost = -1.0;
    for (int m = 1; m <= 64; ++m) {  // items per block
        const long long per = (long long)num_sms * m / nrhs;
        if (per < 1) continue;
        const long long c = ((nunits + per - 1) / per + 31) / 32 * 32;
        if (c > most) continue;
        const double t = (double)m * (double)(c + piece);
        if (cost < 0.0 || t < cost) {
            cost = t;
            best.chunk = c;
            best.per_rhs = (nunits + c - 1) / c;
        }
    }
    best.grid = (int)std::max<long long>(1, std::min<long long>(num_sms, best.per_rhs * nrhs));
    return best;
}
__host__ __device__ inline long long range_lo(int q, long long T, int G) { return (long long)q * T / G; }
}  // namespace
}  // namespace ovs
