// Device helpers shared by the tensor-core kernels: mbarrier waits with a
// cycle limit, TMA tile loads, tcgen05 descriptors / MMA / tensor-memory
// loads and stores, and the exact integer requantization and Sylvester
// butterflies of the epilogues. Every wait that can spin is bounded.
#pragma once

#include <cuda.h>
#include <cstdint>

#include "hatq_internal.h"

namespace hatq {
namespace tc {

constexpr int kBlockK = 64;            // fp16 elements per 128-byte swizzle row
constexpr int kTileM = 128;
constexpr long long kWaitLimitCycles = 4000000000LL;   // about 2 s at 2 GHz

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait. Returns false when the CTA aborts (this wait expired, or
// another role raised the abort flag, or the device error word is set).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *err,
                                          long long limit = kWaitLimitCycles) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    for (uint32_t spin = 1;; ++spin) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((spin & 63) == 0) {
            if (*abort_flag) return false;
            if (*reinterpret_cast<volatile int *>(err) != 0) { *abort_flag = 1; return false; }
            if (clock64() - t0 > limit) {
                *abort_flag = 1;
                atomicExch(err, kErrWaitTimeout);
                return false;
            }
        }
    }
}


// Forms for the converged issuing warps: the instruction is predicated on the
// elected lane instead of branched around, so that the code stays uniform and
// its operands in uniform registers.
__device__ __forceinline__ void mbar_expect_tx_if(uint32_t pr, uint32_t bar, uint32_t bytes) {
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %2, 0;\n @q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n}\n" ::"r"(bar),
        "r"(bytes), "r"(pr)
        : "memory");
}
__device__ __forceinline__ void tma_load_2d_if(uint32_t pr, uint32_t dst, const CUtensorMap *tm, uint32_t bar, int x, int y) {
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %5, 0;\n"
        " @q cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n}\n" ::"r"(dst),
        "l"(tm), "r"(bar), "r"(x), "r"(y), "r"(pr)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d_if(uint32_t pr, uint32_t dst, const CUtensorMap *tm, uint32_t bar, int c0, int c1,
                                               int c2, int c3) {
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %7, 0;\n"
        " @q cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];\n}\n" ::"r"(dst),
        "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(pr)
        : "memory");
}
// ------------------------------------------------------------------ CTA pairs
// Two CTAs of a cluster on neighbouring SMs, the even one the leader: its MMA warp
// issues for both (cta_group::2), barriers it waits on are reached from the other
// CTA by their cluster addresses.
// the address of this CTA's shared-memory location in the leader CTA
__device__ __forceinline__ uint32_t leader_addr(uint32_t addr) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
    return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
// The CTA group's barrier over all threads: the pair's, or the CTA's own.
template <bool PAIR>
__device__ __forceinline__ void group_sync() {
    if constexpr (PAIR) cluster_sync();
    else asm volatile("barrier.sync 0;" ::: "memory");
}
// Tensor memory: all 512 columns, by one warp (of each CTA of a pair).
template <bool PAIR>
__device__ __forceinline__ void tmem_alloc512(uint32_t holder) {
    if constexpr (PAIR) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(holder), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(holder), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
}
template <bool PAIR>
__device__ __forceinline__ void tmem_dealloc512(uint32_t tmem) {
    if constexpr (PAIR)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    else
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}
// The end of an issuing warp after a failure, away from its loops: gives this
// CTA's copies and MMAs in flight `limit` cycles to land, meets the other warps of
// the CTA group at the kernel's last barrier, frees the tensor memory if asked to
// and exits.
template <bool PAIR>
__device__ __noinline__ __attribute__((noreturn)) inline void issue_unwind(uint32_t tmem, bool dealloc, long long limit) {
    const long long t0 = clock64();
    while (clock64() - t0 < limit) {
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    group_sync<PAIR>();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (dealloc) tmem_dealloc512<PAIR>(tmem);
    asm volatile("exit;");
    __builtin_unreachable();
}
constexpr long long kUnwindCycles = 20000000LL;        // about 10 ms: far beyond any copy or MMA of a CTA
// A converged warp's bounded wait without a result: a failure leaves through
// issue_unwind, so the caller's loops keep uniform trip counts (and their
// counters, addresses and descriptors uniform registers). In a pair the barrier
// may be reached from both CTAs.
template <bool PAIR>
__device__ __forceinline__ void mbar_wait_issue(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *err,
                                                uint32_t tmem, bool dealloc) {
    auto done = [&]() { return PAIR ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity); };
    if (__all_sync(0xffffffffu, done())) return;
    const long long t0 = clock64();
    for (uint32_t spin = 1;; ++spin) {
        if (__all_sync(0xffffffffu, done())) return;
        if ((spin & 63) == 0) {
            const bool other = *abort_flag != 0 || *reinterpret_cast<volatile int *>(err) != 0;
            const bool late = clock64() - t0 > kWaitLimitCycles;
            if (__any_sync(0xffffffffu, other || late)) {
                *abort_flag = 1;
                if (__all_sync(0xffffffffu, !other)) atomicExch(err, kErrWaitTimeout);
                issue_unwind<PAIR>(tmem, dealloc, kUnwindCycles);
            }
        }
    }
}
// The pair's copies: the bytes count on the leader's barrier (cluster address).
__device__ __forceinline__ void tma_load_2d_pair_if(uint32_t pr, uint32_t dst, const CUtensorMap *tm, uint32_t leader_bar, int x,
                                                    int y) {
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %5, 0;\n"
        " @q cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n}\n" ::"r"(dst),
        "l"(tm), "r"(leader_bar), "r"(x), "r"(y), "r"(pr)
        : "memory");
}

// Programmatic dependent launch, before anything else in the kernel: the stream's next
// kernel may place its CTAs as this grid's leave (a CTA takes all of an SM's registers, so
// none runs beside one of these), and this one waits until every earlier kernel has
// finished and its writes are visible.
// Convolutions one after the other: 1080p synthesis 376 -> 352 us, three 256-channel
// layers 43.1 -> 41.0, 33 small layers 460 -> 411. Not in the GDN kernel: launched early
// behind its convolution, the pair took 2641 us instead of 2580.
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// One lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ void fence_barrier_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *tm, uint32_t bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
        "l"(tm), "r"(bar), "r"(x), "r"(y)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *tm, uint32_t bar, int c0, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(dst),
        "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *tm, uint32_t bar, int c0, int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
        "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
        : "memory");
}

// Box of a 4-D tensor written from shared memory (parts outside the tensor are
// dropped). Commit, then wait until at most N of this thread's latest groups
// still read shared memory (or, with bulk_wait_all, until all are written).
__device__ __forceinline__ void tma_store_4d(uint32_t src, const CUtensorMap *tm, int c0, int c1, int c2, int c3) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%1, {%2, %3, %4, %5}], [%0];" ::"r"(src),
                 "l"(tm), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async_shared() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// tcgen05 shared-memory matrix descriptor: K-major operand, 128-byte swizzle,
// 8-row groups 1024 bytes apart (stride byte offset), version field = 1.
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)1 << 16;                 // leading byte offset (unused for this layout)
    d |= (uint64_t)(1024 >> 4) << 32;       // stride byte offset
    d |= (uint64_t)1 << 46;                 // descriptor version
    d |= (uint64_t)2 << 61;                 // 128-byte swizzle
    return d;
}

// Instruction descriptor, kind::f16: D = f32, A = B = f16, both K-major, M = 128 (256 for a CTA pair).
__device__ __forceinline__ uint32_t idesc_f16(int n, int m = kTileM) {
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// D (+)= A * B^T with the A operand in TMEM (lane = row, two fp16 per 32-bit
// column, K ascending) and B described in shared memory.
__device__ __forceinline__ void umma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
// D (+)= A * B^T with both operands described in shared memory.
__device__ __forceinline__ void umma_f16_ss(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
// Both operands in shared memory, for a CTA or a pair (M = 256: 128 rows in each
// CTA, N / 2 columns of B in each), predicated, with the descriptors as 32-bit
// halves: only the low words (start addresses) change between instructions.
template <bool PAIR>
__device__ __forceinline__ void umma_f16_ss_if(uint32_t pr, uint32_t d_tmem, uint32_t alo, uint32_t ahi, uint32_t blo,
                                                    uint32_t bhi, uint32_t idesc, uint32_t acc) {
    if constexpr (PAIR)
        asm volatile(
            "{\n .reg .pred p, q;\n .reg .b64 da, db;\n mov.b64 da, {%1, %2};\n mov.b64 db, {%3, %4};\n setp.ne.b32 p, %6, 0;\n"
            " setp.ne.b32 q, %7, 0;\n @q tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %5, p;\n}\n" ::"r"(d_tmem),
            "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(acc), "r"(pr)
            : "memory");
    else
        asm volatile(
            "{\n .reg .pred p, q;\n .reg .b64 da, db;\n mov.b64 da, {%1, %2};\n mov.b64 db, {%3, %4};\n setp.ne.b32 p, %6, 0;\n"
            " setp.ne.b32 q, %7, 0;\n @q tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n}\n" ::"r"(d_tmem),
            "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(acc), "r"(pr)
            : "memory");
}
// one arrival on the barrier (at this offset in both CTAs of a pair)
template <bool PAIR>
__device__ __forceinline__ void umma_commit_if(uint32_t pr, uint32_t bar) {
    if constexpr (!PAIR)
        asm volatile(
            "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
            " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(bar),
            "r"(pr)
            : "memory");
    else
        asm volatile(
        "{\n .reg .pred q;\n .reg .b16 m;\n setp.ne.b32 q, %1, 0;\n mov.b16 m, 3;\n"
        " @q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], m;\n}\n" ::"r"(bar),
        "r"(pr)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// 32 consecutive TMEM columns of this thread's lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld1(uint32_t taddr, uint32_t &r) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]),
        "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]),
        "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// ------------------------------------------------------------------ epilogue math

__device__ __forceinline__ int requant8(long long v, int n) {
    // round(v / 2^n) half to even, clamped to [-127, 127]: v + 2^(n-1) - 1 + bit_n(v), then >> n.
    int q;
    if (n >= 32) {
        // |v| < 2^62, so the shifted value fits in 32 bits.
        const long long u = v + ((1LL << (n - 1)) - 1) + ((int)((unsigned long long)v >> n) & 1);
        q = (int)(u >> n);
    } else if (n > 0) {
        const long long u = v + ((1LL << (n - 1)) - 1) + ((v >> n) & 1);
        const long long w = u >> n;
        q = w < -127 ? -127 : (w > 127 ? 127 : (int)w);
    } else {
        q = v < -127 ? -127 : (v > 127 ? 127 : (int)v);
    }
    return q < -127 ? -127 : (q > 127 ? 127 : q);
}

// The same rounding for 33 <= n <= 62 on the 32-bit halves of v (s = n - 32,
// kh = 2^(s-1) - 1): v + 2^(n-1) - 1 + bit_n(v) has the high word
// hi + kh + c, where c is the carry out of the low word, lo + (2^32 - 1) + bit,
// i.e. c = [lo or bit nonzero]; its shift by n is that high word shifted by s.
__device__ __forceinline__ int requant8_hi(long long v, int s, int kh) {
    const uint32_t lo = (uint32_t)v;
    const int hi = (int)((unsigned long long)v >> 32);
    const uint32_t bit = (uint32_t)(hi >> s) & 1u;
    const int c = (int)min(lo | bit, 1u);
    return min(max((hi + kh + c) >> s, -127), 127);
}
// n = 32: v + 2^31 - 1 + bit_32(v) carries out of the low word iff lo + bit > 2^31.
__device__ __forceinline__ int requant8_32(long long v) {
    const uint32_t lo = (uint32_t)v;
    const int hi = (int)((unsigned long long)v >> 32);
    const int c = (lo > 0x80000000u || (lo == 0x80000000u && (hi & 1))) ? 1 : 0;
    return min(max(hi + c, -127), 127);
}
// The same rounding for 32 <= n <= 62 with only the lower clamp (the
// saturating pack below does the upper one): the 64-bit sum
// v + (2^(n-1) - 1) + bit_n(v) (kadd = 2^(n-1) - 1, s = n - 32; no overflow for
// |v| < 2^62) shifted by n is its high word shifted by s.
__device__ __forceinline__ int requant8_lo(long long v, long long kadd, int s) {
    const int bit = ((int)((unsigned long long)v >> 32) >> s) & 1;
    const unsigned long long u = (unsigned long long)(v + kadd) + (unsigned long long)bit;
    return max((int)(u >> 32) >> s, -127);
}
// bytes (q0, q1, q2, q3) of a word, each q saturated to [-128, 127]
__device__ __forceinline__ uint32_t pack4_sat(int q0, int q1, int q2, int q3) {
    uint32_t hi, d;
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(hi) : "r"(q3), "r"(q2), "r"(0u));
    asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(q1), "r"(q0), "r"(hi));
    return d;
}
// requant8 with the 32-bit-piece paths for shifts >= 32 (n is uniform).
__device__ __forceinline__ int requant8_any(long long v, int n) {
    if (n > 32) return requant8_hi(v, n - 32, (1 << (n - 33)) - 1);
    return n == 32 ? requant8_32(v) : requant8(v, n);
}

// Low bytes of four codes in [-127, 127] packed into one word.
__device__ __forceinline__ uint32_t pack4(int q0, int q1, int q2, int q3) {
    return __byte_perm(__byte_perm((uint32_t)q0, (uint32_t)q1, 0x0040), __byte_perm((uint32_t)q2, (uint32_t)q3, 0x0040),
                       0x5410);
}

// max(v, 0) with the two products on the multiply-add pipe: the sign mask m is
// 0 or -1 and x + m x is x or 0. (A compare and two selects are three
// operations on the integer pipe, which bounds the 64-bit transitions.)
__device__ __forceinline__ long long relu_mad(long long v) {
    const int lo = (int)(uint32_t)v, hi = (int)((unsigned long long)v >> 32), m = hi >> 31;
    int l, h;
    asm("mad.lo.s32 %0, %1, %2, %1;" : "=r"(l) : "r"(lo), "r"(m));
    asm("mad.lo.s32 %0, %1, %2, %1;" : "=r"(h) : "r"(hi), "r"(m));
    return (long long)(((unsigned long long)(uint32_t)h << 32) | (uint32_t)l);
}

template <int G, int HB, typename T>
__device__ __forceinline__ void fwht_fixed(T (&t)[G]) {
#pragma unroll
    for (int h = 1; h < HB; h <<= 1) {
#pragma unroll
        for (int i = 0; i < G; ++i) {
            if (i & h) continue;
            const T a = t[i], b = t[i + h];
            t[i] = a + b;
            t[i + h] = a - b;
        }
    }
}

// Unnormalized Sylvester transform of every hb-block inside t[0..G).
template <int G, typename T>
__device__ __forceinline__ void fwht(T (&t)[G], int hb) {
    switch (hb) {
        case 2: fwht_fixed<G, 2>(t); break;
        case 4: fwht_fixed<G, 4>(t); break;
        case 8: fwht_fixed<G, 8>(t); break;
        case 16: fwht_fixed<G, 16>(t); break;
        case 32: if (G >= 32) fwht_fixed<G, (G >= 32 ? 32 : 2)>(t); break;
        case 64: if (G >= 64) fwht_fixed<G, (G >= 64 ? 64 : 2)>(t); break;
        default: break;
    }
}

// The same transform as one sequence of stages: whole groups (hb = G, the
// usual case) run straight through, smaller blocks stop after log2(hb) stages.
template <int G, typename T>
__device__ __forceinline__ void fwht_stages(T (&t)[G], int hb) {
    if (hb == G) {
        fwht_fixed<G, G>(t);
        return;
    }
#pragma unroll
    for (int h = 1; h < G / 2; h <<= 1) {
        if (h >= hb) break;
#pragma unroll
        for (int i = 0; i < G; ++i) {
            if (i & h) continue;
            const T a = t[i], b = t[i + h];
            t[i] = a + b;
            t[i + h] = a - b;
        }
    }
}

}  // namespace tc
}  // namespace hatq
