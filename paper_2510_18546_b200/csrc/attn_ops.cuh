// PTX wrappers of the tcgen05 kernels: waits, pairs of CTAs, MMA issue, packed arithmetic, descriptors.
#pragma once
#include "ptx_ops.cuh"

namespace enl {
namespace {

constexpr uint32_t kFull = 0xffffffffu;

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// A test that never suspends (about 35 cycles until its result can be used, half of a poll with a suspend hint).
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// The same poll with acquire semantics at cluster scope: data another CTA of the cluster wrote before its
// release.cluster arrival is visible afterwards.  No suspend hint: a thread suspended with the long hint was seen
// to sleep through an arrival that came from the other CTA.
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Distributed shared memory of a two-CTA cluster: stores to the peer's, and arrivals on its barriers.
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// 16-byte store into the peer's shared memory whose completion is counted (in bytes) on a barrier of the peer: the
// sender needs no release fence, which would also wait for its earlier global stores
__device__ __forceinline__ void peer_push4(uint32_t addr, float a, float b, float c, float d, uint32_t bar_peer)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d), "r"(bar_peer) : "memory");
}
// an arrival that publishes nothing (a plain "go ahead")
__device__ __forceinline__ void peer_arrive_relaxed(uint32_t bar)
{
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void peer_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// bulk copy from this CTA's shared memory into the peer's; the bytes are counted on a barrier of the peer
__device__ __forceinline__ void peer_bulk_copy(uint32_t dst_peer, uint32_t src_local, uint32_t bytes, uint32_t bar_peer)
{
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst_peer), "r"(src_local), "r"(bytes), "r"(bar_peer) : "memory");
}
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Bounded wait: gives up about kWaitLimitNs after its 16th failed poll, or when another role has raised the abort flag.
// The result is made warp-uniform so that warp-collective tcgen05 instructions stay converged.
template <bool kCluster = false>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag,
                                          int32_t *status)
{
    auto poll = [&]() { return kCluster ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity); };
    bool ok = kCluster ? poll() : mbar_test(bar, parity);       // the common case: already complete
    if (!ok) {
        // the clock is read only every 16 failed polls (the first reading starts the limit): a poll already
        // sleeps inside the instruction
        unsigned long long t0 = 0;
        uint32_t spins = 0;
        while (!(ok = poll())) {
            if ((++spins & 15u) == 0u) {
                if (*abort_flag) break;
                const unsigned long long now = global_ns();
                if (t0 == 0) {
                    t0 = now;
                } else if (now - t0 > kWaitLimitNs) {
                    *abort_flag = 1;
                    atomicExch(status, 1);
                    break;
                }
            }
        }
    }
    return __all_sync(kFull, ok);
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after()  { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// One lane of the converged warp, chosen by elect.sync.  The choice has to come from that instruction and right where a
// tcgen05 instruction is issued: the compiler then knows that exactly one thread issues and keeps the operands in uniform
// registers.  With a predicate of our own (lane == 0) an MMA took 87 cycles to issue and a commit 100, with elect.sync
// the issue keeps up with the pipe (64): the loop without any softmax work went from 3389 to 2662 cycles per key tile.
__device__ __forceinline__ bool elect_one()
{
    uint32_t r;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(r));
    return r != 0;
}
// D[tmem] (+)= A[smem] * B[smem] and D[tmem] (+)= A[tmem] * B[smem], called by the whole warp.  The shared-memory
// descriptors are given as (low word, high word): the high word is constant and the low word (the start address field)
// moves by a small constant from one MMA to the next.
__device__ __forceinline__ void mma_ss2(uint32_t d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                        uint32_t idesc, uint32_t acc)
{
    if (elect_one())
        asm volatile(
            "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
            "mov.b64 da, {%1, %2};\n\tmov.b64 db, {%3, %4};\n\tsetp.ne.b32 p, %6, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}"
            ::"r"(d), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void mma_ts2(uint32_t d, uint32_t a, uint32_t b_lo, uint32_t b_hi, uint32_t idesc, uint32_t acc)
{
    if (elect_one())
        asm volatile(
            "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\t"
            "mov.b64 db, {%2, %3};\n\tsetp.ne.b32 p, %5, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n\t}"
            ::"r"(d), "r"(a), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    if (elect_one())
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// 3-input max and packed 2 x fp32 arithmetic (one issue slot for two lanes of work)
__device__ __forceinline__ float fmax3(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ uint64_t pack2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// Shared-memory matrix descriptor, 128-byte swizzle, rows of 128 B, 8-row groups 1024 B apart unless given.
// K-major operand (the contraction dimension is contiguous): LBO unused.
// MN-major operand: LBO = distance between 64-element column blocks.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t group_bytes = 1024u)
{
    uint64_t d = 0;
    d |= static_cast<uint64_t>((addr & 0x3FFFFu) >> 4);               // start address
    d |= static_cast<uint64_t>((lbo_bytes >> 4) & 0x3FFFu) << 16;      // leading byte offset
    d |= static_cast<uint64_t>(group_bytes >> 4) << 32;                     // stride byte offset
    d |= static_cast<uint64_t>(1) << 46;                               // descriptor version (sm_100)
    d |= static_cast<uint64_t>(2) << 61;                               // 128-byte swizzle
    return d;
}
// K-major operand of one K step without a swizzle, of which only channel 0 counts: a row is 16 bytes (channels 0..7, and at
// offset 0 again as 8..15), groups of 8 rows are group_bytes apart (0: every group reads the same rows).
__device__ __forceinline__ uint64_t smem_desc_plain(uint32_t addr, uint32_t group_bytes)
{
    return (static_cast<uint64_t>(1) << 46) | (static_cast<uint64_t>(group_bytes >> 4) << 32) | ((addr & 0x3FFFFu) >> 4);
}
// Instruction descriptor, kind::f16: bf16 x bf16 -> fp32, M = 128.
__host__ __device__ constexpr uint32_t make_idesc(int n, bool b_mn_major)
{
    return (1u << 4)                              // D format fp32
         | (1u << 7) | (1u << 10)                 // A, B format bf16
         | ((b_mn_major ? 1u : 0u) << 16)         // B major
         | (static_cast<uint32_t>(n >> 3) << 17)  // N
         | (static_cast<uint32_t>(128 >> 4) << 24);  // M
}


}  // namespace
}  // namespace enl
