// Attention of short calls, sm_100a: a few dozen query rows over a few hundred keys (a new object against its group, a short
// instruction), one launch of latency.
//
// Same computation and row layout as enl_attn_sm100.cu.  There such a call took 11 us for two key tiles: 3 us a tile through
// a chain of roles (loader, MMA issuer, softmax warps, accumulator in TMEM) whose unrolled code is fetched anew by every
// launch, and 2 us of epilogue.  The tensor work is nothing here (0.1 us of the pipe), so this kernel has no roles and little
// code: a CTA takes 16, 32 or 64 query rows of one kv head, loads every page of K and V the rows can see at once (they fit
// shared memory: up to kSmallMaxPages pages), and its 12 warps are 1, 2 or 4 row groups x 12, 6 or 3 key ranges, each walking
// its pages with everything in registers (the fewest rows with which all the CTAs run at once: a page costs a warp 0.5 us):
//   S = Q K^T      mma.sync m16n8k16, A = 16 query rows, B = the K page (ldmatrix)
//   p = exp2(S-m)  running maximum per row kept by the warp, O and the sums rescaled when it grows
//   O += P V       A = P straight from the S accumulators, B = the V page (ldmatrix.trans)
// then the ranges are merged through shared memory (their outputs lie where the pages lay).  A range's pages are in
// stream order, so a row has one open slot; its log2-sum is parked when it ends.
// When neither plan nor pool have been written since the last attention launch the cached pages are fetched before the wait
// for the previous kernel.
// Measured per launch in a chain of 20 layers (32 q / 8 kv heads, large kernel -> this one), one group, no masses: D 128, 41 rows
// over 121 keys 9.5 -> 5.5 us, 61 over 301 11.1 -> 7.4, 128 over 308 12.4 -> 8.4, 256 over 276 12.5 -> 10.6; four groups with
// masses 9.5 -> 7.1, 11.3 -> 8.3, 12.1 -> 9.4, 12.6 -> 11.7.  D 64, four groups with masses: 8.5 -> 5.4, 9.7 -> 6.2, 10.8 -> 6.9,
// 10.7 -> 8.6.
#include <cuda_bf16.h>

#include "decode_ops.cuh"
#include "enl_internal.h"

namespace enl {
namespace {

constexpr int kWarps     = 12;
constexpr int kThreads   = kWarps * 32;
constexpr float kRescaleThreshold = 8.0f;                 // log2 units

// Shared memory: pages [K, V] (later the ranges' outputs) | barriers | page list | per range and row (m, l) | row log-sum-exp |
// parked log-sums [range][slot][row]
// kRowGroups: groups of 16 query rows per CTA
template <int D, int kRowGroups>
struct Cfg {
    static constexpr int kKeyRanges  = kWarps / kRowGroups;
    static constexpr int kRows       = kRowGroups * 16;
    static constexpr int kStageBytes = D * kPageTokens * 2;            // one page of one head
    static constexpr int kORow       = D + 8;                          // row of a range's output: no two rows of a store share banks
    static constexpr int kOutBytes   = kKeyRanges * kRows * kORow * 4;
    static __host__ __device__ constexpr int pages_bytes(int pages)
    {
        return pages * 2 * kStageBytes > kOutBytes ? pages * 2 * kStageBytes : kOutBytes;
    }
    // slots of a range: at most one per page
    static __host__ __device__ constexpr int range_slots(int pages) { return (pages + kKeyRanges - 1) / kKeyRanges; }
    static constexpr int smem_bytes(int pages)
    {
        return pages_bytes(pages) + kSmallMaxPages * 16 + (2 * kKeyRanges + 1) * kRows * 4 + 16 +
               kKeyRanges * range_slots(pages) * kRows * 4 + 1024;     // + alignment slack
    }
};

template <int D, int kRowGroups>
__global__ void __launch_bounds__(kThreads, 1) small_kernel(const __grid_constant__ SmallParams p)
{
    using C = Cfg<D, kRowGroups>;
    constexpr int kKeyRanges = C::kKeyRanges, kRows = C::kRows;
    constexpr int kSteps  = D / 16;                       // k16 steps of Q K^T
    constexpr int kNB     = D / 8;                        // 8-channel blocks of O
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t sbase = (raw + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (sbase - raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, tq = lane & 3;               // MMA row group and thread-in-group
    const int rg = warp % kRowGroups, kr = warp / kRowGroups;
    const int after = C::pages_bytes(p.list_pages);
    const uint32_t bar0 = sbase + static_cast<uint32_t>(after);               // [page]
    int2 *pg_list = reinterpret_cast<int2 *>(smem + after + kSmallMaxPages * 8);
    float *wm = reinterpret_cast<float *>(smem + after + kSmallMaxPages * 16);      // [range][row]: reference, then weight
    float *wl = wm + kKeyRanges * kRows;
    float *lse = wl + kKeyRanges * kRows;                                     // [row]
    volatile int *abort_flag = reinterpret_cast<volatile int *>(lse + kRows);
    float *parked = lse + kRows + 4;                                          // [range][slot][row]
    const int range_slots = C::range_slots(p.list_pages);

    if (threadIdx.x == 0) {
        *abort_flag = 0;
        asm volatile("prefetch.tensormap [%0];" ::"l"(&p.tm_kpool) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&p.tm_vpool) : "memory");
    }
    if (static_cast<int>(threadIdx.x) < kSmallMaxPages) mbar_init(bar0 + 8u * threadIdx.x, 1);
    // The plan or the pool has been written since the last attention launch: nothing of them may be read before the
    // kernel before has ended, and the next launch may start only then (it relies on both).  grid = (row blocks, kv heads,
    // episodes); a single episode travels in the parameters, its pages included: it needs no launch that writes the plan (with
    // one a store and a lone call, 64 rows over 4 groups, took 14.5 us instead of 11.6) and waits for the pool only.
    EpInfo ep;
    if (gridDim.z == 1) {
        ep = p.ep0;
    } else {
        if (p.wait_first) pdl_wait();
        const int4 *src = reinterpret_cast<const int4 *>(p.eps + blockIdx.z);
        const int4 e0 = __ldg(src), e1 = __ldg(src + 1);
        ep.stream_off = e0.x; ep.n_ctiles = e0.y; ep.n_slots = e0.z; ep.q_off = e0.w;
        ep.n_q = e1.x; ep.new_off = e1.y; ep.n_new = e1.z; ep.n_entries = e1.w;
    }
    const int kvh = blockIdx.y, rep = p.rep, G = ep.n_slots;
    const int tokens = kRows / rep, t0 = blockIdx.x * tokens;                 // first query token (episode-relative)
    const int n_tok = min(tokens, ep.n_q - t0);
    const int n_rows = n_tok * rep;                                           // <= 0: nothing here
    const int c0 = ep.n_new - ep.n_q + t0;                                    // last new key that the first token sees
    const int n_cached = ep.n_entries;                                        // cached stream entries without the null ones at the end
    int n_c = 0;                                                              // cached pages
    if (n_rows > 0) {
        // (page id, or -1 - first row of the new keys; slot << 8 | valid keys)
        for (int i = threadIdx.x; i < n_cached; i += kThreads)
            pg_list[i] = gridDim.z == 1 ? p.list[i] : make_int2(__ldg(p.stream_page + ep.stream_off + i), __ldg(p.stream_meta + ep.stream_off + i));
        n_c = n_cached;
    }
    const int n_newp = n_rows > 0 ? (c0 + n_tok - 1) / kPageTokens + 1 : 0;   // pages of new keys that the block's last token sees
    const int total = n_c + n_newp;                                           // <= p.list_pages <= kSmallMaxPages (host guarantees)
    for (int i = threadIdx.x; i < n_newp; i += kThreads)
        pg_list[n_c + i] = make_int2(-1 - i * kPageTokens, (G << 8) | min(kPageTokens, ep.n_new - i * kPageTokens));
    if (threadIdx.x == 0) {
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    if (p.wait_first && gridDim.z == 1) pdl_wait();
    pdl_trigger();
    auto issue = [&](int i, int pg) {
        const uint32_t full = bar0 + 8u * i, dst = sbase + static_cast<uint32_t>(i * 2 * C::kStageBytes);
        mbar_expect_tx(full, 2u * C::kStageBytes);
        // (no evict-first hint: the row blocks of a kv head share its pages)
        if (pg >= 0) {
            tma_load_4d(dst, &p.tm_kpool, 0, 0, 0, (pg * p.Hkv + kvh) * kPageGroups<D>, full);
            tma_load_4d(dst + C::kStageBytes, &p.tm_vpool, 0, 0, 0, (pg * p.Hkv + kvh) * kPageGroups<D>, full);
        } else {
#pragma unroll
            for (int x = 0; x < 2 * kPageGroups<D>; ++x)                      // a group of rows of K or V
                tma_load_4d(dst + static_cast<uint32_t>(x * (C::kStageBytes / kPageGroups<D>)), x < kPageGroups<D> ? &p.tm_knew : &p.tm_vnew, 0,
                            ep.new_off + (-1 - pg) + x % kPageGroups<D> * kBoxRows<D>, 0, kvh, full);
        }
    };
    // page i is fetched by lane 0 of warp i % kWarps: the cached ones while the previous kernel still runs
    if (lane == 0)
        for (int i = warp; i < n_c; i += kWarps) issue(i, pg_list[i].x);
    pdl_wait();
    if (lane == 0)
        for (int i = n_c + (warp + kWarps - n_c % kWarps) % kWarps; i < total; i += kWarps) issue(i, pg_list[i].x);
    if (n_rows <= 0) return;

    // rows g and g + 8 of the warp's 16: the query rows as the A operand
    const int r0 = rg * 16 + g, r1 = r0 + 8;
    uint32_t qa[kSteps][4];
    {
        auto row_ptr = [&](int r) {
            return static_cast<const __nv_bfloat16 *>(p.q) +
                   (static_cast<long long>(ep.q_off + t0 + r / rep) * p.Hq + kvh * rep + r % rep) * D + 2 * tq;
        };
        const __nv_bfloat16 *a = row_ptr(r0), *b = row_ptr(r1);
        const bool on0 = r0 < n_rows, on1 = r1 < n_rows;
#pragma unroll
        for (int ks = 0; ks < kSteps; ++ks) {
            qa[ks][0] = on0 ? *reinterpret_cast<const uint32_t *>(a + ks * 16) : 0u;
            qa[ks][1] = on1 ? *reinterpret_cast<const uint32_t *>(b + ks * 16) : 0u;
            qa[ks][2] = on0 ? *reinterpret_cast<const uint32_t *>(a + ks * 16 + 8) : 0u;
            qa[ks][3] = on1 ? *reinterpret_cast<const uint32_t *>(b + ks * 16 + 8) : 0u;
        }
    }
    const int vis0 = c0 + r0 / rep + 1, vis1 = c0 + r1 / rep + 1;             // new keys that the two rows see
    const float scale = p.scale_log2;
    float o[kNB][4];
#pragma unroll
    for (int nb = 0; nb < kNB; ++nb) { o[nb][0] = o[nb][1] = o[nb][2] = o[nb][3] = 0.f; }
    float m[2] = {kNegInf, kNegInf};                                          // references of the two rows (the same in a quad)
    float l[2] = {0.f, 0.f}, acc[2] = {0.f, 0.f};                             // lane-local parts of the row sums and of the open slot's
    const int n_ranges = min(total, kKeyRanges);                              // no range without a page
    const int pg_beg = kr < n_ranges ? total * kr / n_ranges : total, pg_end = kr < n_ranges ? total * (kr + 1) / n_ranges : total;
    const int slot_first = pg_end > pg_beg ? pg_list[pg_beg].y >> 8 : 0;
    int cur_slot = slot_first;
    bool ok = true;
    auto quad_sum = [](float x) {
        x += __shfl_xor_sync(0xffffffffu, x, 1);
        return x + __shfl_xor_sync(0xffffffffu, x, 2);
    };
    auto park = [&]() {                                                       // the slot that ends
        const float a0 = quad_sum(acc[0]), a1 = quad_sum(acc[1]);
        if (tq == 0) {
            float *d = parked + (kr * range_slots + cur_slot - slot_first) * kRows;
            d[r0] = (a0 > 0.f) ? lg2(a0) + m[0] : kNegInf;
            d[r1] = (a1 > 0.f) ? lg2(a1) + m[1] : kNegInf;
        }
        acc[0] = acc[1] = 0.f;
    };
#pragma unroll 1
    for (int i = pg_beg; i < pg_end; ++i) {
        const int2 e = pg_list[i];
        ok = mbar_wait(bar0 + 8u * i, 0, abort_flag, p.status);
        if (!ok) break;
        const uint32_t base = sbase + static_cast<uint32_t>(i * 2 * C::kStageBytes);
        // S: keys 0..7 and 8..15 of the page, two chains each
        float c[2][4] = {}, c2[2][4] = {};
#pragma unroll
        for (int kq = 0; kq < kSteps / 2; ++kq)                               // four 8-channel chunks = two k16 steps
#pragma unroll
            for (int nb = 0; nb < 2; ++nb) {
                const int row = nb * 8 + (lane & 7), ch = kq * 4 + (lane >> 3);
                uint32_t b[4];
                ldsm_x4(page_chunk<D>(base, row, ch), b);
                mma_bf16(c[nb], qa[2 * kq], b[0], b[1]);
                mma_bf16(c2[nb], qa[2 * kq + 1], b[2], b[3]);
            }
        // visible keys of the page: padding, and the causal limit of either row
        int n0 = e.y & 0xff, n1 = n0;
        if (e.x < 0) {
            n0 = min(n0, vis0 - (-1 - e.x));
            n1 = min(n1, vis1 - (-1 - e.x));
        }
        float s[2][4];                                                        // [row][key 2 tq, 2 tq + 1, 8 + 2 tq, 9 + 2 tq]
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int key = (x >> 1) * 8 + 2 * tq + (x & 1);
            s[0][x] = key < n0 ? (c[x >> 1][x & 1] + c2[x >> 1][x & 1]) * scale : kNegInf;
            s[1][x] = key < n1 ? (c[x >> 1][2 + (x & 1)] + c2[x >> 1][2 + (x & 1)]) * scale : kNegInf;
        }
        const int slot = e.y >> 8;
        while (cur_slot < slot) { park(); ++cur_slot; }
        float mx[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            mx[x] = fmaxf(fmaxf(s[x][0], s[x][1]), fmaxf(s[x][2], s[x][3]));
            mx[x] = fmaxf(mx[x], __shfl_xor_sync(0xffffffffu, mx[x], 1));
            mx[x] = fmaxf(mx[x], __shfl_xor_sync(0xffffffffu, mx[x], 2));
        }
        if (__any_sync(0xffffffffu, mx[0] > m[0] + kRescaleThreshold || mx[1] > m[1] + kRescaleThreshold)) {   // also when m is still -inf
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                const float m_new = fmaxf(m[x], mx[x]);
                const float alpha = (m_new == m[x]) ? 1.f : ex2(m[x] - m_new);
                l[x] *= alpha;
                acc[x] *= alpha;
#pragma unroll
                for (int nb = 0; nb < kNB; ++nb) { o[nb][2 * x] *= alpha; o[nb][2 * x + 1] *= alpha; }
                m[x] = m_new;
            }
        }
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const float m_use = (m[x] == kNegInf) ? 0.f : m[x];
#pragma unroll
            for (int y = 0; y < 4; ++y) s[x][y] = ex2(s[x][y] - m_use);
            const float t = (s[x][0] + s[x][1]) + (s[x][2] + s[x][3]);
            l[x] += t;
            acc[x] += t;
        }
        const uint32_t pa[4] = {pack_bf16(s[0][0], s[0][1]), pack_bf16(s[1][0], s[1][1]), pack_bf16(s[0][2], s[0][3]), pack_bf16(s[1][2], s[1][3])};
        const int row = ((lane >> 3) & 1) * 8 + (lane & 7);                   // token addressed by this lane
        const uint32_t vbase = base + C::kStageBytes;
#pragma unroll
        for (int nq = 0; nq < kNB / 2; ++nq) {                                // two 8-channel blocks per ldmatrix
            const int ch = nq * 2 + (lane >> 4);
            uint32_t b[4];
            ldsm_x4_trans(page_chunk<D>(vbase, row, ch), b);
            mma_bf16(o[2 * nq], pa, b[0], b[1]);
            mma_bf16(o[2 * nq + 1], pa, b[2], b[3]);
        }
    }
    if (pg_end > pg_beg) park();
    // error path only: give the copies in flight time to land before the CTA retires
    if (!ok) {
        const unsigned long long t = global_ns();
        while (global_ns() - t < 50000ull) { }
    }
    l[0] = quad_sum(l[0]);
    l[1] = quad_sum(l[1]);
    if (tq == 0) {
        wm[kr * kRows + r0] = m[0];
        wm[kr * kRows + r1] = m[1];
        wl[kr * kRows + r0] = l[0];
        wl[kr * kRows + r1] = l[1];
    }
    __syncthreads();                                                          // every page has been read: the outputs may go there
    if (*abort_flag) return;
    float *obuf = reinterpret_cast<float *>(smem);                            // [range][row][kORow]
    if (kr < n_ranges) {
#pragma unroll
        for (int nb = 0; nb < kNB; ++nb) {
            *reinterpret_cast<float2 *>(obuf + (kr * kRows + r0) * C::kORow + nb * 8 + 2 * tq) = make_float2(o[nb][0], o[nb][1]);
            *reinterpret_cast<float2 *>(obuf + (kr * kRows + r1) * C::kORow + nb * 8 + 2 * tq) = make_float2(o[nb][2], o[nb][3]);
        }
    }
    // weights of the ranges (exp2(m - lse): they take the unnormalised outputs straight to the result)
    constexpr int kLanes = kKeyRanges > 8 ? 16 : kKeyRanges > 4 ? 8 : 4;      // lanes per row, one range each
    {
        const int r = threadIdx.x / kLanes, k = lane % kLanes;                // kRows * kLanes = 256
        const bool on = r < kRows && k < n_ranges;
        const float mk = on ? wm[k * kRows + r] : kNegInf;
        float M = mk;
#pragma unroll
        for (int of = kLanes / 2; of > 0; of >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, of));
        const float f = (mk == kNegInf) ? 0.f : ex2(mk - M);
        float L = on ? f * wl[k * kRows + r] : 0.f;
#pragma unroll
        for (int of = kLanes / 2; of > 0; of >>= 1) L += __shfl_xor_sync(0xffffffffu, L, of);
        if (on) wm[k * kRows + r] = (L > 0.f) ? f / L : 0.f;
        if (on && k == 0) lse[r] = (L > 0.f) ? M + lg2(L) : kNegInf;
    }
    __syncthreads();
    const long long row_h0 = static_cast<long long>(ep.q_off + t0) * p.Hq + kvh * rep;        // + (r / rep) * Hq + r % rep
#pragma unroll 2
    for (int idx = threadIdx.x; idx < n_rows * (D / 8); idx += kThreads) {    // eight channels of a row
        const int r = idx / (D / 8), c8 = idx % (D / 8);
        float a[8] = {};
#pragma unroll
        for (int k = 0; k < kKeyRanges; ++k) {
            if (k >= n_ranges) break;
            const float w = wm[k * kRows + r];
            const float4 *src = reinterpret_cast<const float4 *>(obuf + (k * kRows + r) * C::kORow + c8 * 8);
            const float4 x = src[0], y = src[1];
            a[0] += w * x.x; a[1] += w * x.y; a[2] += w * x.z; a[3] += w * x.w;
            a[4] += w * y.x; a[5] += w * y.y; a[6] += w * y.z; a[7] += w * y.w;
        }
        *reinterpret_cast<uint4 *>(static_cast<__nv_bfloat16 *>(p.out) + (row_h0 + static_cast<long long>(r / rep) * p.Hq + r % rep) * D + c8 * 8) =
            make_uint4(pack_bf16(a[0], a[1]), pack_bf16(a[2], a[3]), pack_bf16(a[4], a[5]), pack_bf16(a[6], a[7]));
    }
    if (!p.mass) return;
    // masses: the ranges' shares of a slot added up
    for (int idx = threadIdx.x; idx < n_rows * (G + 1); idx += kThreads) {
        const int r = idx / (G + 1), s = idx % (G + 1);
        float w = 0.f;
        for (int k = 0; k < n_ranges; ++k) {
            const int b = total * k / n_ranges, e = total * (k + 1) / n_ranges;
            const int first = pg_list[b].y >> 8, last = pg_list[e - 1].y >> 8;
            if (s >= first && s <= last) w += ex2(parked[(k * range_slots + s - first) * kRows + r] - lse[r]);
        }
        p.mass[(row_h0 + static_cast<long long>(r / rep) * p.Hq + r % rep) * p.mass_stride + s] = w;
    }
}

}  // namespace

namespace {
template <int D>
cudaError_t opt_in()
{
    cudaError_t e = cudaFuncSetAttribute(small_kernel<D, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<D, 1>::smem_bytes(kSmallMaxPages));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(small_kernel<D, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<D, 2>::smem_bytes(kSmallMaxPages));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(small_kernel<D, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<D, 4>::smem_bytes(kSmallMaxPages));
    return e;
}
template <int D>
cudaError_t launch(const SmallParams &p, int row_groups, dim3 grid, cudaStream_t st)
{
    if (row_groups == 1) return launch_pdl(small_kernel<D, 1>, grid, dim3(kThreads), Cfg<D, 1>::smem_bytes(p.list_pages), st, p);
    if (row_groups == 2) return launch_pdl(small_kernel<D, 2>, grid, dim3(kThreads), Cfg<D, 2>::smem_bytes(p.list_pages), st, p);
    return launch_pdl(small_kernel<D, 4>, grid, dim3(kThreads), Cfg<D, 4>::smem_bytes(p.list_pages), st, p);
}
}  // namespace

cudaError_t prepare_small(int head_dim)
{
    if (head_dim == 128) return opt_in<128>();
    if (head_dim == 64) return opt_in<64>();
    return cudaErrorInvalidValue;
}

cudaError_t launch_small(const SmallParams &p, int head_dim, int row_groups, int row_blocks, int batch, cudaStream_t st)
{
    if (batch <= 0 || row_blocks <= 0) return cudaSuccess;
    if (p.list_pages > kSmallMaxPages || (batch == 1 && (p.n_list != p.ep0.n_entries || p.n_list > kSmallMaxPages)) || (16 * row_groups) % p.rep || (row_groups != 1 && row_groups != 2 && row_groups != 4))
        return cudaErrorInvalidValue;
    const dim3 grid(row_blocks, p.Hkv, batch);
    cudaError_t e;
    if (head_dim == 128) e = launch<128>(p, row_groups, grid, st);
    else if (head_dim == 64) e = launch<64>(p, row_groups, grid, st);
    else return cudaErrorInvalidValue;
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace enl
