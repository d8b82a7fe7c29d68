// PTX wrappers of the mma.sync kernels (one-token steps, short calls).
#pragma once
#include "ptx_ops.cuh"

namespace enl {
namespace {

// Bounded wait, warp-uniform result.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int32_t *status)
{
    bool ok = mbar_try_wait(bar, parity);
    if (!ok) {
        // the clock is read only every 16 failed polls (the first reading starts the limit): a poll already
        // sleeps inside the instruction
        unsigned long long t0 = 0;
        uint32_t spins = 0;
        while (!(ok = mbar_try_wait(bar, parity))) {
            if ((++spins & 15u) == 0u) {
                if (*abort_flag) break;
                const unsigned long long now = global_ns();
                if (t0 == 0) {
                    t0 = now;
                } else if (now - t0 > kWaitLimitNs) {
                    *abort_flag = 1;
                    atomicExch(status, 2);
                    break;
                }
            }
        }
    }
    return __all_sync(0xffffffffu, ok);
}
// The K/V stream is read once: its lines are marked evict-first so that what is reused from launch to launch
// (code, plan, partial results) stays in L2.
__device__ __forceinline__ uint64_t policy_evict_first()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
// Where the 16-byte chunk ch of row `row` of a page lies: two groups of 8 rows, a group being one swizzled 8 x 128-byte block per
// 64 channels (the layout of the boxes that fetch a page).
template <int D>
__device__ __forceinline__ uint32_t page_chunk(uint32_t base, int row, int ch)
{
    return base + static_cast<uint32_t>((row >> 3) * (D * 16) + (ch >> 3) * 1024 + (row & 7) * 128 + (((ch & 7) ^ (row & 7)) << 4));
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
// D (fp32, m16n8) += A (bf16, m16k16, row) * B (bf16, k16n8, col)
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float rcp(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

}  // namespace
}  // namespace enl
