// tcgen05 / TMA / mbarrier building blocks shared by the tensor-core kernels of libcsr
// (the matching-pursuit encoder and the Gram products of the dictionary training step):
// single-instruction inline-PTX wrappers, the shared-memory matrix descriptor of a K-major
// 128-byte-swizzled bf16 tile, and the bounded waits every hand-off goes through.
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace csr {
namespace tc {

// ---------------------------------------------------------------------------------------
// PTX wrappers
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// The same with a hint of how long the hardware may keep the thread suspended (nanoseconds)
// before the instruction returns false: a thread that polls with a long hint leaves the issue
// slots of its scheduler to the other warps.
__device__ __forceinline__ bool mbar_try_wait_hint(uint64_t* bar, uint32_t parity, uint32_t suspend_ns) {
    uint32_t ok;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(suspend_ns)
        : "memory");
    return ok != 0;
}
// One look at the barrier without suspending the thread.
__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void fence_barrier_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// ---- thread-block cluster: peers' shared memory and barriers ----
__device__ __forceinline__ uint32_t map_to_cta(uint32_t saddr, uint32_t cta_rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(cta_rank));
    return r;
}
// Eight bytes into a peer's shared memory; the peer's barrier is credited with them when they
// have landed, so the reader needs nothing but to wait for its barrier.
__device__ __forceinline__ void st_async_u64(uint32_t raddr, unsigned long long v, uint32_t rbar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(raddr), "l"(v),
                 "r"(rbar)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Every thread of every CTA of the cluster (a lone CTA is a cluster of one).
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int c0, int c1, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]^T for one 64-channel block of both operands (bf16 or fp16, `idesc` says which; fp32 accumulate):
// four MMAs, 32 bytes apart in the swizzled rows, then a commit (umma_commit) to each barrier given.  The whole warp
// calls, converged, with the same arguments, and one elected lane issues: in code that only lane 0 runs, every MMA first has
// to move its descriptors to the uniform registers the instruction takes, 116 cycles a piece, 168
// when the other warps are busy too, more than the 128 x 256 x 16 MMA itself takes.  Measured, 128
// MMAs in a row per SM with eight warps reading tensor memory: 178 cycles per MMA from lane 0,
// 139 with the election (128 is the tensor core's own rate).  One election for a block instead of one for each MMA and commit
// shortens the issuing warp's chain per row tile (615 cycles in a copy with clocks, while a d = 64 tile's MMAs take 512): 262144 rows,
// N = 4096, s = 8: 1798 -> 1748 us; 100003 rows, N = 5001, d = 64, s = 6: 428 -> 424; exact mode, 100000 rows, N = 4096, s = 8: 1278 -> 1256.
// (An issuing warp per accumulator: 2154 and 477 us.  The tensor core takes the MMAs of two warps in turn, so that both accumulators
// complete, and are drained, at the same time.)
__device__ __forceinline__ void umma_f16_block(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p, e, t;\n"
        "setp.ne.b32 p, %10, 0;\n"
        "setp.eq.b32 t, 0, 0;\n"
        "elect.sync _|e, 0xffffffff;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %5, %9, p;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %2, %6, %9, t;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %3, %7, %9, t;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %4, %8, %9, t;\n"
        "}\n" ::"r"(d_tmem), "l"(a), "l"(a + 2), "l"(a + 4), "l"(a + 6), "l"(b), "l"(b + 2), "l"(b + 4), "l"(b + 6), "r"(idesc),
        "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void umma_f16_block(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate, uint64_t* bar0) {
    asm volatile(
        "{\n"
        ".reg .pred p, e, t;\n"
        "setp.ne.b32 p, %10, 0;\n"
        "setp.eq.b32 t, 0, 0;\n"
        "elect.sync _|e, 0xffffffff;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %5, %9, p;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %2, %6, %9, t;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %3, %7, %9, t;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %4, %8, %9, t;\n"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%11];\n"
        "}\n" ::"r"(d_tmem), "l"(a), "l"(a + 2), "l"(a + 4), "l"(a + 6), "l"(b), "l"(b + 2), "l"(b + 4), "l"(b + 6), "r"(idesc),
        "r"(accumulate), "r"(smem_u32(bar0))
        : "memory");
}
__device__ __forceinline__ void umma_f16_block(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate, uint64_t* bar0, uint64_t* bar1) {
    asm volatile(
        "{\n"
        ".reg .pred p, e, t;\n"
        "setp.ne.b32 p, %10, 0;\n"
        "setp.eq.b32 t, 0, 0;\n"
        "elect.sync _|e, 0xffffffff;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %5, %9, p;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %2, %6, %9, t;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %3, %7, %9, t;\n"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %4, %8, %9, t;\n"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%11];\n"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%12];\n"
        "}\n" ::"r"(d_tmem), "l"(a), "l"(a + 2), "l"(a + 4), "l"(a + 6), "l"(b), "l"(b + 2), "l"(b + 4), "l"(b + 6), "r"(idesc),
        "r"(accumulate), "r"(smem_u32(bar0)), "r"(smem_u32(bar1))
        : "memory");
}
// The mbarrier gets one arrival once every tcgen05.mma issued so far by the elected lane is done (the
// whole warp calls, as above).
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile(
        "{\n"
        ".reg .pred e;\n"
        "elect.sync _|e, 0xffffffff;\n"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
        "}\n" ::"r"(smem_u32(bar))
        : "memory");
}
// Waits for this thread's outstanding tcgen05.ld.  The registers are passed through the
// statement so that no use of them can be scheduled ahead of the wait.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&v)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]), "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]), "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]), "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31])
                 :
                 : "memory");
}

// Orders later uses of the registers after the preceding tcgen05.wait::ld without emitting
// an instruction (the asynchronous load that fills them is invisible to the compiler).
__device__ __forceinline__ void reg_fence(uint32_t (&v)[32]) {
    asm volatile(""
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]), "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]), "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]), "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31])
                 :
                 : "memory");
}

// 32 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
          "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr)
        : "memory");
}

// Shared-memory matrix descriptor of a K-major bf16 tile stored as rows of 128 bytes with
// the 128-byte swizzle: 8-row groups are 1024 bytes apart.
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t saddr) {
    uint64_t desc = 0;
    desc |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);   // start address, 16-byte units
    desc |= static_cast<uint64_t>(1) << 16;                  // leading byte offset (unused with swizzle)
    desc |= static_cast<uint64_t>(1024 >> 4) << 32;          // stride byte offset between 8-row groups
    desc |= static_cast<uint64_t>(1) << 46;                  // descriptor version of sm_100
    desc |= static_cast<uint64_t>(2) << 61;                  // 128-byte swizzle
    return desc;
}

// Instruction descriptors of tcgen05.mma kind::f16: fp32 accumulator, A and B both bf16 or both fp16, both K-major.
__host__ __device__ constexpr uint32_t instr_desc_f16(int m, int n) {
    return (1u << 4) | (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(m >> 4) << 24);
}
__host__ __device__ constexpr uint32_t instr_desc_bf16(int m, int n) {
    return instr_desc_f16(m, n) | (1u << 7) | (1u << 10);
}

struct WaitCtx {
    volatile uint32_t* abort;
    uint32_t* status;
    unsigned long long limit_ns;
};

// Waits for the phase with the given parity; gives up after w.limit_ns (wall clock) or when
// another thread of the CTA has given up.  A limit of zero allows one look at the barrier
// that does not suspend the thread: whatever is not complete by then counts as expired.
__device__ __forceinline__ bool wait_bounded(uint64_t* bar, uint32_t parity, const WaitCtx& w) {
    if (w.limit_ns != 0) {
        if (mbar_try_wait(bar, parity)) return true;
        const unsigned long long t0 = globaltimer_ns();
        for (uint32_t it = 1; it < (1u << 28); ++it) {
            if (mbar_try_wait(bar, parity)) return true;
            if ((it & 63u) == 0) {
                if (*w.abort) return false;
                if (globaltimer_ns() - t0 > w.limit_ns) break;
            }
        }
    } else if (mbar_test_wait(bar, parity)) {
        return true;
    }
    *w.abort = 1;
    atomicOr(w.status, kStatusTimeout);
    return false;
}

// The same wait for hand-offs that take long (a whole pick, a whole sweep): every poll lets the
// hardware suspend the thread for up to `suspend_ns`.
__device__ __forceinline__ bool wait_bounded_suspended(uint64_t* bar, uint32_t parity, const WaitCtx& w, uint32_t suspend_ns) {
    if (w.limit_ns != 0) {
        if (mbar_try_wait(bar, parity)) return true;
        const unsigned long long t0 = globaltimer_ns();
        for (uint32_t it = 1; it < (1u << 28); ++it) {
            if (mbar_try_wait_hint(bar, parity, suspend_ns)) return true;
            if ((it & 7u) == 0) {
                if (*w.abort) return false;
                if (globaltimer_ns() - t0 > w.limit_ns) break;
            }
        }
    } else if (mbar_test_wait(bar, parity)) {
        return true;
    }
    *w.abort = 1;
    atomicOr(w.status, kStatusTimeout);
    return false;
}

// The waits of a warp that stays converged (every lane polls; the answer is the same for all).
__device__ __forceinline__ bool warp_wait_bounded(uint64_t* bar, uint32_t parity, const WaitCtx& w) {
    return __all_sync(0xffffffffu, wait_bounded(bar, parity, w));
}
__device__ __forceinline__ bool warp_wait_bounded_suspended(uint64_t* bar, uint32_t parity, const WaitCtx& w, uint32_t suspend_ns) {
    return __all_sync(0xffffffffu, wait_bounded_suspended(bar, parity, w, suspend_ns));
}
// A value every lane of the warp holds, as one the compiler knows to be uniform.
__device__ __forceinline__ uint32_t warp_uniform(uint32_t v) { return __shfl_sync(0xffffffffu, v, 0); }

// The same wait on a barrier that other CTAs of the cluster arrive on.
__device__ __forceinline__ bool wait_bounded_cluster(uint64_t* bar, uint32_t parity, const WaitCtx& w) {
    if (w.limit_ns != 0) {
        if (mbar_try_wait_cluster(bar, parity)) return true;
        const unsigned long long t0 = globaltimer_ns();
        for (uint32_t it = 1; it < (1u << 28); ++it) {
            if (mbar_try_wait_cluster(bar, parity)) return true;
            if ((it & 63u) == 0) {
                if (*w.abort) return false;
                if (globaltimer_ns() - t0 > w.limit_ns) break;
            }
        }
    } else if (mbar_test_wait(bar, parity)) {
        return true;
    }
    *w.abort = 1;
    atomicOr(w.status, kStatusTimeout);
    return false;
}

// A CTA that has given up must stay until what its peers have sent it has landed: the cluster barrier does
// not wait for st.async.  One thread calls this after the cluster barrier that every CTA passes when it
// sends no more; `phase`: the barrier's first phase not waited out, `bytes` its transaction count.  A
// peer can be one phase ahead, no further (it would need this CTA's words).  A phase that some peer
// never sent for does not complete: what was sent for it has 20 ms to land.
__device__ __forceinline__ void let_words_land(uint64_t* bar, uint32_t phase, uint32_t bytes) {
    const unsigned long long t0 = globaltimer_ns();
    for (int k = 0; k < 2; ++k, ++phase) {
        for (uint32_t it = 0; !mbar_try_wait_cluster(bar, phase & 1); ++it)
            if (globaltimer_ns() - t0 > 20000000ull || it >= (1u << 28)) return;
        if (k == 0) mbar_expect_tx(bar, bytes);
    }
}

}  // namespace tc
}  // namespace csr
