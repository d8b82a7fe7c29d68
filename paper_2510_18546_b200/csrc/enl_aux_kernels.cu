// Small kernels around the attention: scatter of a group's K/V rows into pool pages (the store of
// Sec. 3.2 "Discrete Memory Caching") and the merge of KV splits (log-sum-exp weighted average of the
// partial outputs, sum of the partial per-slot masses).
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>
#include <cstring>

#include "enl_internal.h"

namespace enl {
namespace {

// k, v: [n_tokens][Hkv][D] bf16 -> pool layer [page][Hkv][16][D]; 16-byte chunks, one per thread-iteration.
// The `zero_rows` rows behind the last token (the padding of the group's last page) are cleared: the attention
// kernels give padded keys probability 0, and 0 times whatever an earlier, longer version of the group left
// there must stay 0 (a stale non-finite value would not).
__device__ __forceinline__ void scatter_rows(uint4 *__restrict__ kpool, uint4 *__restrict__ vpool, const uint4 *__restrict__ k,
                                             const uint4 *__restrict__ v, const PageRun &run, int first_pos, int n_tokens,
                                             int zero_rows, int Hkv, int chunks_per_row)
{
    const long long total = static_cast<long long>(n_tokens + zero_rows) * Hkv * chunks_per_row;
    const long long n_src = static_cast<long long>(n_tokens) * Hkv * chunks_per_row;
    for (long long id = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; id < total;
         id += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int ch = static_cast<int>(id % chunks_per_row);
        const long long th = id / chunks_per_row;
        const int head = static_cast<int>(th % Hkv);
        const int tok = static_cast<int>(th / Hkv);
        const int pos = first_pos + tok;
        const int page = run.ids[pos / kPageTokens - run.first_page];
        const long long dst = ((static_cast<long long>(page) * Hkv + head) * kPageTokens + pos % kPageTokens) *
                                  chunks_per_row + ch;
        const bool real = id < n_src;
        kpool[dst] = real ? k[id] : make_uint4(0u, 0u, 0u, 0u);
        vpool[dst] = real ? v[id] : make_uint4(0u, 0u, 0u, 0u);
    }
}
__global__ void page_scatter_kernel(uint4 *__restrict__ kpool, uint4 *__restrict__ vpool,
                                    const uint4 *__restrict__ k, const uint4 *__restrict__ v,
                                    const __grid_constant__ PageRun run, int first_pos, int n_tokens, int zero_rows,
                                    int Hkv, int chunks_per_row)
{
    pdl_trigger();
    pdl_wait();                                             // an attention kernel may still be reading these pages
    scatter_rows(kpool, vpool, k, v, run, first_pos, n_tokens, zero_rows, Hkv, chunks_per_row);
}

// grid (blocks, layers): the same scatter for several layers of one group at once
__global__ void page_scatter_layers_kernel(uint4 *__restrict__ kpool, uint4 *__restrict__ vpool, long long layer_chunks,
                                           const __grid_constant__ LayerSrc src, long long src_chunk_off,
                                           const __grid_constant__ PageRun run, int first_pos, int n_tokens,
                                           int zero_rows, int Hkv, int chunks_per_row)
{
    const uint4 *k = static_cast<const uint4 *>(src.k[blockIdx.y]) + src_chunk_off;
    const uint4 *v = static_cast<const uint4 *>(src.v[blockIdx.y]) + src_chunk_off;
    uint4 *kp = kpool + layer_chunks * blockIdx.y, *vp = vpool + layer_chunks * blockIdx.y;
    pdl_trigger();
    pdl_wait();                                             // an attention kernel may still be reading these pages
    scatter_rows(kp, vp, k, v, run, first_pos, n_tokens, zero_rows, Hkv, chunks_per_row);
}

__device__ __forceinline__ float ex2f(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// One warp per (query row, q head): lane l merges channels 4l..4l+3 (D = 128) or 2l, 2l+1 (D = 64), and slot l, l + 32, ...
// Splits are taken kBatch at a time, their partial outputs and the log-sums of 32 slots on the way together, the first ones with
// the log-sum-exps: up to eight splits cost one memory round trip (four or fewer are not charged for eight).
template <int D, int kBatch>
__global__ void __launch_bounds__(256) combine_kernel(const CombineParams p)
{
    constexpr int V = D / 32;                               // channels per lane
    const int lane = threadIdx.x & 31;
    const long long rh = blockIdx.x * static_cast<long long>(blockDim.x >> 5) + (threadIdx.x >> 5);
    const long long split_stride = static_cast<long long>(p.n_q_total) * p.Hq;
    pdl_trigger();
    pdl_wait();                                             // the partial results come from the previous kernel
    if (rh >= split_stride) return;
    const float ninf = -__builtin_huge_valf();
    const int row = static_cast<int>(rh / p.Hq);
    const int G = p.mass ? p.row_slots[row] : -1;
    const int G0 = p.part_rng ? -1 : G;                     // slots whose log-sums come along with the outputs
    const float *o0 = p.part_o + rh * D + lane * V;
    const float *s0 = p.part_slot ? p.part_slot + rh * p.slot_stride + lane : nullptr;
    float ov[kBatch][V], sv[kBatch];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const int k = k0 + j < p.n_splits ? k0 + j : 0; // (a split beyond the last has weight 0)
            if constexpr (V == 4) {
                const float4 t = __ldcg(reinterpret_cast<const float4 *>(o0 + k * split_stride * D));
                ov[j][0] = t.x; ov[j][1] = t.y; ov[j][2] = t.z; ov[j][3] = t.w;
            } else {
                const float2 t = __ldcg(reinterpret_cast<const float2 *>(o0 + k * split_stride * D));
                ov[j][0] = t.x; ov[j][1] = t.y;
            }
            sv[j] = (lane <= G0 && k0 + j < p.n_splits) ? __ldcg(s0 + k * split_stride * p.slot_stride) : ninf;
        }
    };
    fetch(0);
    // every lane needs every split's log-sum-exp: lane k loads split k (and k + 32), then shuffles
    const float my0 = lane < p.n_splits ? __ldcg(p.part_lse + lane * split_stride + rh) : ninf;
    const float my1 = lane + 32 < p.n_splits ? __ldcg(p.part_lse + (lane + 32) * split_stride + rh) : ninf;
    int2 r0 = make_int2(0, -1), r1 = r0;                    // slots that the splits have written of this row
    if (p.part_rng) {
        if (lane < p.n_splits) r0 = __ldcg(p.part_rng + static_cast<long long>(lane) * p.n_q_total + row);
        if (lane + 32 < p.n_splits) r1 = __ldcg(p.part_rng + static_cast<long long>(lane + 32) * p.n_q_total + row);
    }
    float mx = fmaxf(my0, my1);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float sum = (my0 != ninf ? ex2f(my0 - mx) : 0.f) + (my1 != ninf ? ex2f(my1 - mx) : 0.f);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const float lse = mx + log2f(sum);
    const float lse_s = (lse > ninf) ? lse : 0.f;
    const float w0 = my0 != ninf ? ex2f(my0 - lse) : 0.f;
    const float w1 = my1 != ninf ? ex2f(my1 - lse) : 0.f;

    float acc[V], mass = 0.f;
#pragma unroll
    for (int x = 0; x < V; ++x) acc[x] = 0.f;
    for (int k0 = 0; k0 < p.n_splits; k0 += kBatch) {
        if (k0 > 0) fetch(k0);
#pragma unroll
        for (int j = 0; j < kBatch; ++j) {
            const int k = k0 + j;
            // a split that saw no key has weight 0 and never wrote its partial output: what sits there is stale
            const float w = __shfl_sync(0xffffffffu, k < 32 ? w0 : w1, k & 31);
            if (w != 0.f && k < p.n_splits) {
#pragma unroll
                for (int x = 0; x < V; ++x) acc[x] = fmaf(w, ov[j][x], acc[x]);
            }
            mass += ex2f(sv[j] - lse_s);                    // exp2(-inf) = 0: absent slots drop out
        }
    }
    __nv_bfloat16 *dst = static_cast<__nv_bfloat16 *>(p.out) + rh * D + lane * V;
#pragma unroll
    for (int x = 0; x < V; x += 2)
        *reinterpret_cast<__nv_bfloat162 *>(dst + x) = __floats2bfloat162_rn(acc[x], acc[x + 1]);
    if (!p.mass) return;
    float *masses = p.mass + rh * p.mass_stride;
    if (p.part_rng) {
        // Many slots, most of them in one split only: of every 64 slots (two a lane), the splits whose ranges reach into them, four at a time.
        // (All splits of every slot, which the attention kernel then has to clear: 17 rows over 400 groups in 60 splits, 4 heads, 66 us and not 28.)
        for (int s = 0; s <= G; s += 64) {                  // warp-uniform
            uint32_t m0 = __ballot_sync(0xffffffffu, r0.x <= s + 63 && r0.y >= s), m1 = __ballot_sync(0xffffffffu, r1.x <= s + 63 && r1.y >= s);
            const int s_lo = s + lane, s_hi = s_lo + 32;
            float mass_lo = 0.f, mass_hi = 0.f;
            while ((m0 | m1) != 0u) {
                float lo[4], hi[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int k = m0 ? __ffs(m0) - 1 : m1 ? __ffs(m1) + 31 : -1;
                    const int first = __shfl_sync(0xffffffffu, k < 32 ? r0.x : r1.x, k & 31), last = __shfl_sync(0xffffffffu, k < 32 ? r0.y : r1.y, k & 31);
                    const float *sk = s0 + s + k * split_stride * p.slot_stride;
                    lo[u] = (k >= 0 && s_lo >= first && s_lo <= last) ? __ldcg(sk) : ninf;
                    hi[u] = (k >= 0 && s_hi >= first && s_hi <= last) ? __ldcg(sk + 32) : ninf;
                    if (m0) m0 &= m0 - 1u;
                    else m1 &= m1 - 1u;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    mass_lo += ex2f(lo[u] - lse_s);
                    mass_hi += ex2f(hi[u] - lse_s);
                }
            }
            if (s_lo <= G) masses[s_lo] = mass_lo;
            if (s_hi <= G) masses[s_hi] = mass_hi;
        }
        return;
    }
    if (lane <= G) masses[lane] = mass;
    for (int s = 32; s <= G; s += 32) {                     // warp-uniform
        mass = 0.f;
        for (int k0 = 0; k0 < p.n_splits; k0 += kBatch) {
#pragma unroll
            for (int j = 0; j < kBatch; ++j)
                sv[j] = (s + lane <= G && k0 + j < p.n_splits) ? __ldcg(s0 + s + (k0 + j) * split_stride * p.slot_stride) : ninf;
#pragma unroll
            for (int j = 0; j < kBatch; ++j) mass += ex2f(sv[j] - lse_s);
        }
        if (s + lane <= G) masses[s + lane] = mass;
    }
}

// Masses of the attention kernel's calls with many slots, of scoring passes and of per-object sums: the attention kernel has
// left every slot's log2-sum in the mass buffer and every row's log2-sum-exp beside it.  One warp per 32 (row, head) pairs and
// 32 slots, lanes over the slots: every access is a coalesced line, kLoads pairs' lines in flight.  Bandwidth-bound: reads and
// writes every mass once.  Four layers of 1024 rows x 32 heads over 1000 groups (131 MB of masses each): 9.4 -> 8.5 ms against
// finishing them inside the attention kernel.
// With mass_sum the masses of one object's rows are added up on the way and leave as one atomic add per warp, object and slot
// (Sec. 3.3 consumes only averages over an object's tokens and the q heads).
template <bool kSplits, bool kSums, int kLoads>
__global__ void __launch_bounds__(256) mass_finish_kernel(const FinishParams p)
{
    const int lane = threadIdx.x & 31;
    const long long n_pairs = static_cast<long long>(p.n_q_total) * p.Hq;
    const long long first = (static_cast<long long>(blockIdx.x) * 8 + (threadIdx.x >> 5)) * 32;
    const int s = blockIdx.y * 32 + lane;
    const float ninf = -__builtin_huge_valf();
    pdl_trigger();
    const long long mine = first + lane;
    int G = -1, obj = -1;
    if (mine < n_pairs) {
        const int row = static_cast<int>(mine / p.Hq);
        G = p.row_slots ? __ldg(p.row_slots + row) : p.max_slots;   // of the gather plan: the attention kernel has waited for it
        if (kSums) obj = __ldg(p.row_obj + row);
    }
    pdl_wait();
    // lane x holds pair x: the row's log-sum-exp over the splits, the splits' parts of slots they share with the one before
    float lse = ninf;
    float2 bnd[kSplits ? kFinishSplits : 1];
    if (kSplits) {
#pragma unroll
        for (int k = 0; k < kFinishSplits; ++k) bnd[k] = make_float2(0.f, __int_as_float(-1));
    }
    if (mine < n_pairs) {
        if constexpr (kSplits) {
            float v[kFinishSplits], mx = ninf, sum = 0.f;
#pragma unroll
            for (int k = 0; k < kFinishSplits; ++k) {
                v[k] = k < p.n_splits ? __ldcg(p.lse + k * n_pairs + mine) : ninf;
                if (k > 0 && k < p.n_splits) bnd[k] = __ldcg(p.bnd + k * n_pairs + mine);
                mx = fmaxf(mx, v[k]);
            }
#pragma unroll
            for (int k = 0; k < kFinishSplits; ++k) sum += v[k] != ninf ? ex2f(v[k] - mx) : 0.f;
            lse = mx != ninf ? mx + log2f(sum) : ninf;
#pragma unroll
            for (int k = 1; k < kFinishSplits; ++k) bnd[k].x = (lse != ninf && k < p.n_splits) ? ex2f(bnd[k].x - lse) : 0.f;
        } else {
            lse = __ldcg(p.lse + mine);
        }
    }
    const int n_here = static_cast<int>(max(0ll, min(32ll, n_pairs - first)));
    // splits (bit k) that share a slot of this warp's with the one before: seldom any
    uint32_t shared = 0;
    if constexpr (kSplits) {
#pragma unroll
        for (int k = 1; k < kFinishSplits; ++k)
            if (__any_sync(0xffffffffu, (__float_as_int(bnd[k].y) >> 5) == static_cast<int>(blockIdx.y))) shared |= 1u << k;
    }
    float run = 0.f;                                        // this slot's sum over the rows of the current object
    int run_obj = -1;
    float *const col = p.mass + first * p.mass_stride + s;
    auto turn = [&](auto one_row) {
        constexpr bool kOneRow = decltype(one_row)::value;  // the pairs have one slot count and one object
        if (kOneRow) run_obj = obj;
        for (int x0 = 0; x0 < n_here; x0 += kLoads) {
            float v[kLoads];
#pragma unroll
            for (int u = 0; u < kLoads; ++u) {
                const int g = kOneRow ? G : __shfl_sync(0xffffffffu, G, x0 + u);
                v[u] = s <= g ? __ldcg(col + static_cast<long long>(x0 + u) * p.mass_stride) : ninf;
            }
#pragma unroll
            for (int u = 0; u < kLoads; ++u) {
                const int x = x0 + u, g = kOneRow ? G : __shfl_sync(0xffffffffu, G, x);
                const float ref = __shfl_sync(0xffffffffu, lse, x);
                float w = (ref != ninf) ? ex2f(v[u] - ref) : 0.f;
                if constexpr (kSplits) {
                    if (shared) {
#pragma unroll
                        for (int k = 1; k < kFinishSplits; ++k) {
                            if (!((shared >> k) & 1u)) continue;
                            const float b = __shfl_sync(0xffffffffu, bnd[k].x, x);
                            const int bs = __shfl_sync(0xffffffffu, __float_as_int(bnd[k].y), x);
                            if (s == bs) w += b;
                        }
                    }
                }
                if (s <= g) col[static_cast<long long>(x) * p.mass_stride] = w;
                if constexpr (kSums) {
                    if (!kOneRow) {
                        const int o = __shfl_sync(0xffffffffu, obj, x);
                        if (o != run_obj) {                 // the same in every lane
                            if (run_obj >= 0 && run != 0.f) atomicAdd(p.mass_sum + static_cast<long long>(run_obj) * p.sum_stride + s, run);
                            run = 0.f;
                            run_obj = o;
                        }
                    }
                    if (s <= g) run += w;
                }
            }
        }
    };
    // A row's 32 q heads are one warp's pairs in many models; then nothing has to be looked up pair by pair (four layers of 512 rows over 200 groups 526 -> 513 us in all).
    const int G0 = __shfl_sync(0xffffffffu, G, 0), obj0 = __shfl_sync(0xffffffffu, obj, 0);
    if (n_here == 32 && __all_sync(0xffffffffu, G == G0 && obj == obj0)) turn(std::true_type{});
    else turn(std::false_type{});
    if constexpr (kSums)
        if (run_obj >= 0 && run != 0.f) atomicAdd(p.mass_sum + static_cast<long long>(run_obj) * p.sum_stride + s, run);
}

// Pages between the pool and the pinned host pool: pairs (from, to) of layers layer0 .. layer0 + n_layers - 1, K and V, 2 KB per
// warp and trip.  Bound by the host link, whose latency 64 warps with 2 KB in flight each cover (32: 34 GB/s, 64: 50.5, more: 51).
constexpr int kCopyThreads = 256;
constexpr int kPieceChunks = 128;                           // a page is a multiple of 2 KB
__global__ void __launch_bounds__(kCopyThreads) page_copy_kernel(const uint4 *src_k, const uint4 *src_v, uint4 *dst_k, uint4 *dst_v, size_t src_layer,
                                                                 size_t dst_layer, const int2 *pairs, int n_pairs, int layer0, long long total, int pieces)
{
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (long long i = blockIdx.x * (kCopyThreads / 32) + (threadIdx.x >> 5); i < total; i += gridDim.x * (kCopyThreads / 32)) {
        const int page = static_cast<int>(i / pieces), piece = static_cast<int>(i - static_cast<long long>(page) * pieces);
        const int layer = layer0 + (page >> 1) / n_pairs;                // K and V of a page follow one another
        const int2 pr = pairs[(page >> 1) % n_pairs];
        const size_t off = static_cast<size_t>(piece) * kPieceChunks + lane;
        const uint4 *s = ((page & 1) ? src_v : src_k) + src_layer * layer + static_cast<size_t>(pr.x) * pieces * kPieceChunks + off;
        uint4 *d = ((page & 1) ? dst_v : dst_k) + dst_layer * layer + static_cast<size_t>(pr.y) * pieces * kPieceChunks + off;
        uint4 v[kPieceChunks / 32];
#pragma unroll
        for (int u = 0; u < kPieceChunks / 32; ++u) v[u] = s[u * 32];
#pragma unroll
        for (int u = 0; u < kPieceChunks / 32; ++u) d[u * 32] = v[u];
    }
}

// The gather plan as kernel parameters -> device memory.  It waits for the kernel before (which may read the previous plan
// in the same place) and does not let its successor start early: the successor reads the plan in its set-up.
template <int kBytes>
struct PlanBlob {
    uint4 *dst;
    int32_t n;                                              // 16-byte words
    int32_t pad;
    uint4 data[kBytes / 16];
};
template <int kBytes>
__global__ void __launch_bounds__(128) plan_write_kernel(const __grid_constant__ PlanBlob<kBytes> p)
{
    const int i = blockIdx.x * 128 + threadIdx.x;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (i < p.n) v = p.data[i];
    pdl_wait();
    if (i < p.n) p.dst[i] = v;
}

template <int kBytes>
cudaError_t plan_write(void *dst, const void *src, size_t bytes, cudaStream_t st)
{
    static thread_local PlanBlob<kBytes> blob;              // too large for the stack of every caller
    blob.dst = static_cast<uint4 *>(dst);
    blob.n = static_cast<int32_t>((bytes + 15) / 16);
    std::memcpy(blob.data, src, bytes);
    return launch_pdl(plan_write_kernel<kBytes>, dim3((blob.n + 127) / 128), dim3(128), 0, st, blob);
}

}  // namespace

// Three sizes: what a launch costs grows with the parameters it carries.
cudaError_t launch_plan_write(void *dst, const void *src, size_t bytes, cudaStream_t st)
{
    if (bytes == 0) return cudaSuccess;
    if (bytes > kPlanParamBytes) return cudaErrorInvalidValue;
    const cudaError_t e = bytes <= 2048   ? plan_write<2048>(dst, src, bytes, st)
                          : bytes <= 8192 ? plan_write<8192>(dst, src, bytes, st)
                                          : plan_write<kPlanParamBytes>(dst, src, bytes, st);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_page_copy(const uint8_t *src_k, const uint8_t *src_v, uint8_t *dst_k, uint8_t *dst_v,
                             size_t src_layer_bytes, size_t dst_layer_bytes, const int2 *pairs, int n_pairs, int layer0,
                             int n_layers, int page_bytes, int ctas, cudaStream_t st)
{
    if (n_pairs <= 0 || n_layers <= 0) return cudaSuccess;
    const int pieces = page_bytes / (16 * kPieceChunks);
    const long long total = 2ll * n_pairs * n_layers * pieces;
    const long long need = (total + kCopyThreads / 32 - 1) / (kCopyThreads / 32);
    // an ordinary launch: the CTAs of dependent ones would take their places early and keep attention CTAs out
    page_copy_kernel<<<static_cast<unsigned>(std::min<long long>(ctas, need)), kCopyThreads, 0, st>>>(
        reinterpret_cast<const uint4 *>(src_k), reinterpret_cast<const uint4 *>(src_v), reinterpret_cast<uint4 *>(dst_k),
        reinterpret_cast<uint4 *>(dst_v), src_layer_bytes / 16, dst_layer_bytes / 16, pairs, n_pairs, layer0, total, pieces);
    return cudaGetLastError();
}

cudaError_t launch_page_scatter(void *kpool_layer, void *vpool_layer, const void *k, const void *v,
                                const PageRun &run, int first_pos, int n_tokens, int zero_rows, int Hkv, int D,
                                int n_sm, cudaStream_t st)
{
    if (n_tokens <= 0) return cudaSuccess;
    const int cpr = D * 2 / 16;
    const long long total = static_cast<long long>(n_tokens + zero_rows) * Hkv * cpr;
    const int threads = 256;
    long long blocks = (total + threads - 1) / threads;
    if (blocks > n_sm * 8) blocks = n_sm * 8;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(blocks));
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, page_scatter_kernel, static_cast<uint4 *>(kpool_layer),
                                             static_cast<uint4 *>(vpool_layer), static_cast<const uint4 *>(k),
                                             static_cast<const uint4 *>(v), run, first_pos, n_tokens, zero_rows, Hkv, cpr);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_page_scatter_layers(void *kpool, void *vpool, size_t layer_bytes, int layer0, int n_layers,
                                       const LayerSrc &src, size_t src_off, const PageRun &run, int first_pos,
                                       int n_tokens, int zero_rows, int Hkv, int D, int n_sm, cudaStream_t st)
{
    if (n_tokens <= 0 || n_layers <= 0) return cudaSuccess;
    if (n_layers > kScatterLayers) return cudaErrorInvalidValue;
    const int cpr = D * 2 / 16;
    const long long total = static_cast<long long>(n_tokens + zero_rows) * Hkv * cpr;
    const int threads = 256;
    long long blocks = (total + threads - 1) / threads;
    const long long cap = std::max(1, n_sm * 8 / n_layers);
    if (blocks > cap) blocks = cap;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(blocks), static_cast<unsigned>(n_layers));
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    uint4 *kp = reinterpret_cast<uint4 *>(static_cast<uint8_t *>(kpool) + layer_bytes * layer0);
    uint4 *vp = reinterpret_cast<uint4 *>(static_cast<uint8_t *>(vpool) + layer_bytes * layer0);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, page_scatter_layers_kernel, kp, vp,
                                             static_cast<long long>(layer_bytes / 16), src,
                                             static_cast<long long>(src_off / 16), run, first_pos, n_tokens, zero_rows, Hkv, cpr);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_mass_finish(const FinishParams &p, int n_sm, cudaStream_t st)
{
    const long long pairs = static_cast<long long>(p.n_q_total) * p.Hq;
    if (pairs <= 0) return cudaSuccess;
    if (p.n_splits > kFinishSplits) return cudaErrorInvalidValue;
    const dim3 grid(static_cast<unsigned>((pairs + 255) / 256), static_cast<unsigned>(p.max_slots / 32 + 1));
    // Loads in flight per warp: sixteen where a multiprocessor has few warps to hide a round trip with (up to four CTAs each), eight where
    // the grid fills it.  148 multiprocessors:
    // Four layers with outputs, 8 -> 16 loads: 448 CTAs (512 rows over 200 groups) 467 -> 440 us, 896 CTAs (1024 rows) 799 -> 805,
    // 1280 CTAs 1132 -> 1177, 4096 CTAs (1000 groups) 3735 -> 3817; averages only, 896 CTAs 597 -> 602.
    const bool few = static_cast<long long>(grid.x) * grid.y <= 4ll * n_sm;
    auto launch = [&](auto loads) {
        constexpr int kLoads = decltype(loads)::value;
        if (p.n_splits > 1)
            return p.mass_sum ? launch_pdl(mass_finish_kernel<true, true, kLoads>, grid, dim3(256), 0, st, p)
                              : launch_pdl(mass_finish_kernel<true, false, kLoads>, grid, dim3(256), 0, st, p);
        return p.mass_sum ? launch_pdl(mass_finish_kernel<false, true, kLoads>, grid, dim3(256), 0, st, p)
                          : launch_pdl(mass_finish_kernel<false, false, kLoads>, grid, dim3(256), 0, st, p);
    };
    const cudaError_t e = few ? launch(std::integral_constant<int, 16>{}) : launch(std::integral_constant<int, 8>{});
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_combine(const CombineParams &p, cudaStream_t st)
{
    const long long pairs = static_cast<long long>(p.n_q_total) * p.Hq;
    if (pairs <= 0) return cudaSuccess;
    const int warps = 8;
    const int blocks = static_cast<int>((pairs + warps - 1) / warps);
    cudaError_t e;
    if (p.n_splits <= 4)
        e = p.D == 128 ? launch_pdl(combine_kernel<128, 4>, dim3(blocks), dim3(warps * 32), 0, st, p)
                       : launch_pdl(combine_kernel<64, 4>, dim3(blocks), dim3(warps * 32), 0, st, p);
    else
        e = p.D == 128 ? launch_pdl(combine_kernel<128, 8>, dim3(blocks), dim3(warps * 32), 0, st, p)
                       : launch_pdl(combine_kernel<64, 8>, dim3(blocks), dim3(warps * 32), 0, st, p);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace enl
