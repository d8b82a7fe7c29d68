// Attention of one-token steps whose key stream is short: splits merged through distributed shared memory, sm_100a.
//
// What it computes is what enl_decode_sm100.cu computes: for every episode and kv head, the attention of the rep q heads that
// read this kv head over the selected groups' pages and the new-token keys, with the probability mass of every slot.
//
// The time of such a call is latency, not bandwidth: with 2600 keys all the CTAs' loads are in flight at once and the
// streaming kernel spends 6 of its 8.6 us on merging -- partial results to memory, a fence, a counter, and the last CTA
// reading them back (0.9 + 1.9 us), while the next launch cannot even start.  Here the splits of one (episode, kv head) are
// the CTAs of one thread-block cluster: each merges its warps in its own shared memory and pushes what the others need of
// the result into theirs, with st.async, whose bytes the receiver's barrier counts: the receiver adds up its share of the output as soon
// as it is there, nobody fences and nobody waits for a second cluster barrier (its release waits for every earlier store, ~0.5 us).
// And two CTAs fit an SM (12 warps of 80 registers, ~110 KB), so the next launch is resident while this
// one runs: its set-up and its first pages (from the pool, which only this library writes) are done before its wait for the
// previous kernel ends.  Where its last clusters have to wait for an SM (sixteens of eight kv heads), the set-up itself counts: each warp
// asks for its first page before anything else, and prefetches are dealt to the warps (start to wait 2.7 -> 1.8 us).
// Measured per launch in a chain of 20 layers (32 q / 8 kv heads, 24 groups; streaming kernel, this one with cluster barriers, now):
// D 128 with masses, 640 keys 9.2, 6.0, 5.4 us, 2560 keys 10.2, 8.3, 6.9; without, 640 keys 5.0, 4.6, 2560 keys 6.7, 5.9; D 64 with
// masses, 640 keys 8.6, 5.6, 4.7, 2560 keys 9.1, 7.3, 5.7; contiguous keys (the entry point that allocates nothing), 2500 keys 91, 10.2, 8.9.
//
// Per page, all in registers of one warp:
//   S^T = K Q^T        mma.sync m16n8k16, A = the 16 keys (ldmatrix), B = the rep query rows padded to 8
//   p   = exp2(S - m)  running maximum per head kept by the warp, O and the sums rescaled when it grows
//   O^T += V^T P^T     A = V^T (ldmatrix.trans), B = P^T out of the S accumulators (one 8 x 8 transpose per 8 keys)
// With the keys as the rows of the product nothing of a 16-row MMA is padding: half the MMAs of the other way round, and no
// accumulators of unused rows.
// The entry point that allocates nothing uses the same kernel over contiguous keys (kStatic): a page is then up to 16 keys of
// one segment, fetched from any row by the tensor maps of the caller's K and V, and P goes into the product as three bf16
// terms whose sum is the fp32 value: that path promises fp32 probabilities.
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "decode_ops.cuh"
#include "enl_internal.h"

namespace enl {
namespace {

constexpr int kWarps   = 12;                              // two CTAs of 12 warps per SM: 80 registers a thread
constexpr int kThreads = kWarps * 32;
constexpr int kStages  = 2;                               // per warp: K and V of one page
constexpr int kMaxRep  = 8;                               // q heads per kv head (columns of the MMA)
constexpr int kPrefetchPages = 24;                        // pages per CTA asked into the L2 before the previous kernel has ended
constexpr float kRescaleThreshold = 8.0f;                 // log2 units

// Stores into a peer's shared memory whose completion is counted (in bytes) on a barrier of the peer: neither side needs a
// fence or a round trip.  Not for a cluster of one: that is launched without clusters, where these instructions are illegal.
__device__ __forceinline__ void peer_push(uint32_t addr, float v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(addr), "f"(v), "r"(bar) : "memory");
}
__device__ __forceinline__ void peer_push4(uint32_t addr, float4 v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar) : "memory");
}
// Waits for what the peers push.  No CTA may leave before it has arrived, so a wait of its own that ran out does not cut this one short:
// its limit covers that of the peers' waits, after which they push whatever they have.
__device__ __forceinline__ void wait_for_peers(uint32_t bar, int32_t *status)
{
    unsigned long long t0 = 0;
    for (uint32_t spins = 1;; ++spins) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done) : "r"(bar) : "memory");
        if (__all_sync(0xffffffffu, done != 0u)) return;
        if ((spins & 15u) == 0u) {
            const unsigned long long now = global_ns();
            if (t0 == 0) t0 = now;
            if (__any_sync(0xffffffffu, now - t0 > 4 * kWaitLimitNs)) { atomicExch(status, 2); return; }
        }
    }
}
// (nothing to publish but barriers, which fence.mbarrier_init has: no wait for earlier stores)
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// the 8 x 8 matrix of 16-bit values that the warp holds, transposed
__device__ __forceinline__ uint32_t transpose8x8(uint32_t x)
{
    uint32_t y;
    asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}

// Shared memory: ring [warp][stage][D*32 B] | barriers | slot ranges | merge words | query fragments | rows sent by the
// cluster | parked slot sums | page list | slot table.  The lists are sized by the launch (two CTAs have to fit an SM).
template <int D>
struct Cfg {
    static constexpr int kStageBytes = D * kPageTokens * 2;            // one page of one head: 4 KB (D=128) / 2 KB
    static constexpr int kRingBytes  = kWarps * kStages * kStageBytes;
    static constexpr int kORow       = D + 4;                          // row of a warp's output: no two rows of a store share banks
    static_assert(kWarps * kMaxRep * kORow * 4 <= kRingBytes, "the warps' outputs fit the idle ring");
    static constexpr int kBarOff     = kRingBytes;                     // [warp][stage]
    static constexpr int kInBarOff   = kBarOff + kWarps * kStages * 8; // what the cluster sends has arrived: outputs, shares of a slot
    static constexpr int kRngOff     = kInBarOff + 16;                 // [kMaxCluster] (first slot, slots)
    static constexpr int kMiscOff    = kRngOff + kMaxCluster * 8;
    // wm[warp][rep], wl[warp][rep], cm[rep], cl[rep], warp weights[rep][kMaxCluster], log2-sum-exps (then weights) of the
    // cluster's CTAs[rep][kMaxCluster], ctrs[2], flags[2]
    static constexpr int kMiscBytes  = (2 * kWarps * kMaxRep + 2 * kMaxRep + 2 * kMaxRep * kMaxCluster + 4) * 4;
    static constexpr int kQOff       = kMiscOff + kMiscBytes;          // [D / 16][32 lanes] B fragments of the query rows
    static constexpr int kShareOff   = kQOff + D / 16 * 32 * 8;        // [kMaxCluster][kMaxRep]: the cluster's shares of this CTA's last slot
    static constexpr int kInOff      = kShareOff + kMaxCluster * kMaxRep * 4;        // [CTA][float4]: what the cluster's CTAs send for this CTA's share of the output
    static_assert(kInOff % 16 == 0, "alignment");
    // parked slot sums: a warp's pages come in stream order, so it parks each slot it meets once
    static __host__ __device__ constexpr int ent_cap(int pages, int slots)
    {
        return pages + kWarps < kWarps * slots ? pages + kWarps : kWarps * slots;
    }
    static constexpr int smem_bytes(int pages, int slots, int rep)
    {
        return kInOff + rep * D * 4 + ent_cap(pages, slots) * (((rep + 1) & ~1) + 1) * 4 + 8 + pages * 8 + slots * kMaxRep * 4 + 1024;   // + alignment slack
    }
};
static_assert(kWarps <= kMaxCluster, "the two weight tables have one row length");

__device__ __forceinline__ const ClusterDecodeParams &common(const ClusterDecodeParams &p) { return p; }
__device__ __forceinline__ const ClusterDecodeParams &common(const StaticDecodeParams &p) { return p.d; }

template <int D, bool kStatic>
__global__ void __launch_bounds__(kThreads, 2)
    decode_cluster_kernel(const __grid_constant__ std::conditional_t<kStatic, StaticDecodeParams, ClusterDecodeParams> prm)
{
    using C = Cfg<D>;
    constexpr int kMB     = D / 16;                       // 16-channel blocks of O^T
    const ClusterDecodeParams &p = common(prm);
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t sbase = (raw + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (sbase - raw);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, tq = lane & 3;               // MMA row group and thread-in-group
    int2 *rng_tab = reinterpret_cast<int2 *>(smem + C::kRngOff);              // [CTA of the cluster]: first slot and slots of its page range
    float *wm = reinterpret_cast<float *>(smem + C::kMiscOff);                // [warp][kMaxRep]
    float *wl = wm + kWarps * kMaxRep;
    float *cm = wl + kWarps * kMaxRep;                                        // log2-sum-exp of the CTA's range
    float *cl = cm + kMaxRep;
    float *ww = cl + kMaxRep;                                                 // [kMaxRep][kMaxCluster]: weights of the warps
    float *cw = ww + kMaxRep * kMaxCluster;                                   // [kMaxRep][kMaxCluster]: log2-sum-exps of the cluster's CTAs
    int *ctrs = reinterpret_cast<int *>(cw + kMaxRep * kMaxCluster);          // [0] next page to hand out, [1] parked entries, [3] see `owner`
    volatile int *abort_flag = ctrs + 2;
    const int rep = p.rep, rep2 = (rep + 1) & ~1;
    const int n_ent_cap = C::ent_cap(p.list_pages, p.list_slots);
    float *ent_val = reinterpret_cast<float *>(smem + C::kInOff) + rep * D;   // [n_ent_cap][rep2]: parked log2 slot sums
    int *ent_slot = reinterpret_cast<int *>(ent_val + n_ent_cap * rep2);      // [n_ent_cap]: their slots
    int2 *pg_list = reinterpret_cast<int2 *>(ent_slot + ((n_ent_cap + 1) & ~1));   // the CTA's pages in stream order
    float *cslot = reinterpret_cast<float *>(pg_list + p.list_pages);         // [slot][kMaxRep]: shares of the range's sum
    const uint32_t bar0 = sbase + C::kBarOff;
    const uint32_t bar_in = sbase + C::kInBarOff, bar_share = bar_in + 8;
    const float *share_in = reinterpret_cast<const float *>(smem + C::kShareOff);
    auto bar_full = [&](int s) { return bar0 + 8u * (warp * kStages + s); };
    auto stage_addr = [&](int s) { return sbase + static_cast<uint32_t>((warp * kStages + s) * C::kStageBytes); };

    if (threadIdx.x == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(kStatic ? &p.tm_knew : &p.tm_kpool) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(kStatic ? &p.tm_vnew : &p.tm_vpool) : "memory");
    }
    // The plan or the pool has been written since the last attention launch: nothing of them may be read before the
    // kernel before has ended, and the next launch may start only then (it relies on both).
    if (p.wait_first) pdl_wait();
    // grid = (CTAs of the cluster, kv heads, episodes); a single episode travels in the parameters
    const int split = blockIdx.x, n_splits = gridDim.x, kvh = blockIdx.y;
    const int ls = 31 - __clz(n_splits), lr = 31 - __clz(rep);                // both are powers of two
    EpInfo ep;
    if (gridDim.z == 1) {
        ep = p.ep0;
    } else {
        const int4 *src = reinterpret_cast<const int4 *>(p.eps + blockIdx.z);
        const int4 e0 = __ldg(src), e1 = __ldg(src + 1);
        ep.stream_off = e0.x; ep.n_ctiles = e0.y; ep.n_slots = e0.z; ep.q_off = e0.w;
        ep.n_q = e1.x; ep.new_off = e1.y; ep.n_new = e1.z; ep.n_entries = e1.w;
    }
    const int G = ep.n_slots;
    const int n_cached = kStatic ? 0 : ep.n_ctiles * kPagesPerTile;           // cached stream entries (padded)
    int total;
    if constexpr (kStatic) total = prm.page_off[G + 1];
    else total = n_cached + (ep.n_new + kPageTokens - 1) / kPageTokens;
    const int pg_beg = total * split >> ls, pg_end = total * (split + 1) >> ls;   // (at most kMaxCluster * kClusterMaxPages pages)
    const int n_cta = pg_end - pg_beg;                                        // <= p.list_pages (host guarantees)

    // page e of the stream: (page id, or -1 - first row of the caller's keys; slot << 8 | valid keys)
    auto entry = [&](int e) -> int2 {
        if constexpr (kStatic) {
            int lo = 0, hi = G;                                              // the last slot that starts at or before page e
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (prm.page_off[mid] <= e) lo = mid; else hi = mid - 1;
            }
            const int r = prm.seg_off[lo] + (e - prm.page_off[lo]) * kPageTokens;
            return make_int2(-1 - r, (lo << 8) | min(kPageTokens, prm.seg_off[lo + 1] - r));
        } else {
            if (e < n_cached) return make_int2(__ldg(p.stream_page + ep.stream_off + e), __ldg(p.stream_meta + ep.stream_off + e));
            const int r = (e - n_cached) * kPageTokens;
            return make_int2(-1 - r, (G << 8) | min(kPageTokens, ep.n_new - r));
        }
    };

    const uint64_t pol = policy_evict_first();
    // K or V of one page into this warp's ring
    auto issue = [&](bool is_v, int page) {
        const int st = is_v ? 1 : 0;
        const uint32_t full = bar_full(st), dst = stage_addr(st);
        mbar_expect_tx(full, static_cast<uint32_t>(C::kStageBytes));
        if (!kStatic && page >= 0) {
            const CUtensorMap *tm = is_v ? &p.tm_vpool : &p.tm_kpool;
            tma_load_4d(dst, tm, 0, 0, 0, (page * p.Hkv + kvh) * kPageGroups<D>, full, pol);
        } else {
            const CUtensorMap *tm = is_v ? &p.tm_vnew : &p.tm_knew;
            const int krow = ep.new_off + (-1 - page);                       // rows past the tensor's end read as zero
            tma_load_4d(dst, tm, 0, krow, 0, kvh, full, pol);
            if constexpr (kPageGroups<D> == 2) tma_load_4d(dst + C::kStageBytes / 2, tm, 0, krow + kBoxRows<D>, 0, kvh, full, pol);
        }
    };
    // While the previous kernel of the stream still runs: the pool is written by launches of this library only, and none has
    // come in between, so the first cached page of every warp is fetched for good; what else comes first is asked into the L2
    // (which observes nothing: the L2 is the point of coherence).  The first round is handed out statically.
    int cur = warp;
    const int2 first = cur < n_cta ? entry(pg_beg + cur) : make_int2(-1, 0);
    const int pg0 = first.x;
    if (lane == 0) {
        for (int s = 0; s < kStages; ++s) mbar_init(bar_full(s), 1);
        if (warp == 0) {
            mbar_init(bar_in, 1);
            mbar_init(bar_share, 1);
            mbar_expect_tx(bar_in, static_cast<uint32_t>(rep * (D + n_splits) * 4));
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (pg0 >= 0) { issue(false, pg0); issue(true, pg0); }
    }
    if (threadIdx.x == 0) { *abort_flag = 0; ctrs[0] = kWarps; ctrs[1] = 0; }
    // The slot range of every CTA of the cluster (the same arithmetic as that CTA uses): the merge looks up whose table holds a slot.
    if (static_cast<int>(threadIdx.x) < n_splits) {
        const int k = threadIdx.x;
        const int b0 = total * k >> ls, b1 = total * (k + 1) >> ls;
        int2 r = make_int2(0, 0);
        if (b1 > b0) {
            const int s0 = entry(b0).y >> 8;
            r = make_int2(s0, (entry(b1 - 1).y >> 8) - s0 + 1);
        }
        rng_tab[k] = r;
    }
    for (int i = threadIdx.x; i < n_cta; i += kThreads) pg_list[i] = entry(pg_beg + i);
    __syncthreads();
    cluster_arrive_relaxed();                                                // every CTA of the cluster has started (waited for before the first store to a peer)
    pdl_trigger();
    int slot_first = 0, n_local = 0;                                         // slots the CTA's range touches
    if (n_cta > 0) {
        slot_first = pg_list[0].y >> 8;
        n_local = (pg_list[n_cta - 1].y >> 8) - slot_first + 1;
    }
    // The CTA in whose range a slot begins writes its mass; the CTAs behind whose ranges the slot reaches into send their shares.  Which
    // CTA wants this one's share of its first slot (-1: this one does), and how many send theirs of its last?
    if (p.mass && warp == kWarps - 1) {
        const int2 r = lane < n_splits ? rng_tab[lane] : make_int2(0, 0);
        const int last = r.x + r.y - 1;
        const uint32_t into = __ballot_sync(0xffffffffu, lane < split && r.y > 0 && last == slot_first);
        const uint32_t after = __ballot_sync(0xffffffffu, lane > split && r.y > 0 && r.x == slot_first + n_local - 1);
        if (lane == 0) {
            ctrs[3] = n_cta > 0 ? __ffs(into) - 1 : -1;
            const bool wanted = n_local > 1 || (n_local == 1 && into == 0u);
            mbar_expect_tx(bar_share, wanted ? static_cast<uint32_t>(__popc(after) * rep * 4) : 0u);
        }
    }
    // (a warp takes a page: a box costs the warp that asks for it some 50 cycles)
    for (int i = warp; i < min(n_cta, kPrefetchPages); i += kWarps) {
        const int pg = pg_list[i].x;
        if (pg < 0) {
            if (lane < 2 * kPageGroups<D>)
                tma_prefetch_4d((lane & 1) ? &p.tm_vnew : &p.tm_knew, 0, ep.new_off + (-1 - pg) + (lane >> 1) * kBoxRows<D>, 0, kvh);
        } else if (i >= kWarps && lane < 2) {
            tma_prefetch_4d((lane & 1) ? &p.tm_vpool : &p.tm_kpool, 0, 0, 0, (pg * p.Hkv + kvh) * kPageGroups<D>);
        }
    }
    const uint8_t *q_rows = static_cast<const uint8_t *>(p.q) + (static_cast<long long>(ep.q_off) * p.Hq + kvh * rep) * D * 2;
    if (static_cast<int>(threadIdx.x) * 128 < rep * D * 2)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(q_rows + threadIdx.x * 128) : "memory");

    // so far only shared memory, the gather plan and the pool were touched; the caller's tensors come next
    pdl_wait();
    if (lane == 0 && cur < n_cta && pg0 < 0) { issue(false, pg0); issue(true, pg0); }
    // the next page of the CTA that nobody has taken yet (CTA-relative index; >= n_cta: none left)
    auto claim = [&]() -> int {
        int v = 0;
        if (lane == 0) v = atomicAdd(&ctrs[0], 1);
        return __shfl_sync(0xffffffffu, v, 0);
    };
    // The query rows of this kv head as the B operand of S^T = K Q^T (heads >= rep are zero), in the order the lanes read them
    uint2 *qfrag = reinterpret_cast<uint2 *>(smem + C::kQOff);
    for (int ks = warp; ks < D / 16; ks += kWarps) {
        const uint8_t *qrow = q_rows + (g * D + ks * 16 + 2 * tq) * 2;
        uint2 v = make_uint2(0u, 0u);
        if (g < rep) v = make_uint2(*reinterpret_cast<const uint32_t *>(qrow), *reinterpret_cast<const uint32_t *>(qrow + 16));
        qfrag[ks * 32 + lane] = v;
    }
    __syncthreads();
    // read now, while the first pages are on their way, what is otherwise first read from the parameters after the stream
    asm volatile("" ::"l"(p.out), "l"(p.mass), "r"(p.mass_stride), "r"(p.Hq));
    const float scale = p.scale_log2;
    bool ok = true;
    int n_done = 0;                                                          // pages this warp has worked through

    // A thread's columns are the heads 2 tq and 2 tq + 1 throughout (index 0, 1 of what follows).
    float o[kMB][4];                        // O^T: channels 16 mb + g (first two) and 16 mb + g + 8
#pragma unroll
    for (int mb = 0; mb < kMB; ++mb) { o[mb][0] = o[mb][1] = o[mb][2] = o[mb][3] = 0.f; }
    float m[2] = {kNegInf, kNegInf};        // running reference maxima (the same in all lanes of equal tq)
    float lsum[2] = {0.f, 0.f}, acc[2] = {0.f, 0.f};       // lane-local parts of the heads' sums and of the current slot's
    int cur_slot = -1;
    auto over_keys = [](float x) {          // sum over the lanes of equal tq
        x += __shfl_xor_sync(0xffffffffu, x, 4);
        x += __shfl_xor_sync(0xffffffffu, x, 8);
        return x + __shfl_xor_sync(0xffffffffu, x, 16);
    };
    auto park = [&]() {                      // the slot that ends: its id and the log2 of its sums (absolute) join the CTA's list
        if (cur_slot >= 0) {
            const float a0 = over_keys(acc[0]), a1 = over_keys(acc[1]);
            int e = 0;
            if (lane == 0) { e = atomicAdd(&ctrs[1], 1); ent_slot[e] = cur_slot; }
            e = __shfl_sync(0xffffffffu, e, 0);
            if (g == 0 && 2 * tq < rep2)
                *reinterpret_cast<float2 *>(ent_val + e * rep2 + 2 * tq) =
                    make_float2((a0 > 0.f) ? lg2(a0) + m[0] : kNegInf, (a1 > 0.f) ? lg2(a1) + m[1] : kNegInf);
        }
        acc[0] = acc[1] = 0.f;
    };

    for (; cur < n_cta && ok; ++n_done) {
        const uint32_t par = static_cast<uint32_t>(n_done & 1);
        const int nn = claim();                                              // the page that follows
        const int nn_page = nn < n_cta ? pg_list[nn].x : 0;
        const int meta = pg_list[cur].y;
        // ---- S = Q K^T ----
        ok = mbar_wait(bar_full(0), par, abort_flag, p.status);
        if (!ok) break;
        uint32_t base = stage_addr(0);
        // two chains of products: those of one chain wait for one another
        float c[4] = {0.f, 0.f, 0.f, 0.f}, c2[4] = {0.f, 0.f, 0.f, 0.f};
        {
            const int row = ((lane >> 3) & 1) * 8 + (lane & 7);              // token whose 16-byte chunks this lane addresses
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
                const int ch = 2 * ks + (lane >> 4);
                uint32_t a[4];
                ldsm_x4(page_chunk<D>(base, row, ch), a);
                const uint2 qv = qfrag[ks * 32 + lane];
                mma_bf16((ks & 1) ? c2 : c, a, qv.x, qv.y);
            }
        }
        const int nv = meta & 0xff, slot = meta >> 8;
        float s[4];                                                          // keys g (first two) and g + 8
#pragma unroll
        for (int x = 0; x < 4; ++x) s[x] = (g + (x >> 1) * 8 < nv) ? (c[x] + c2[x]) * scale : kNegInf;
        // the ring slot is read out: the page after the next one
        auto refill = [&](bool is_v) {
            __syncwarp();                                                    // orders the warp's reads before the copy
            if (lane == 0 && nn < n_cta) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                issue(is_v, nn_page);
            }
        };
        refill(false);

        // ---- p = exp2(S - m), sums ----
        float mx[2] = {fmaxf(s[0], s[2]), fmaxf(s[1], s[3])};
#pragma unroll
        for (int of = 4; of <= 16; of *= 2) {
            mx[0] = fmaxf(mx[0], __shfl_xor_sync(0xffffffffu, mx[0], of));
            mx[1] = fmaxf(mx[1], __shfl_xor_sync(0xffffffffu, mx[1], of));
        }
        if (slot != cur_slot) { park(); cur_slot = slot; }
        if (__any_sync(0xffffffffu, mx[0] > m[0] + kRescaleThreshold || mx[1] > m[1] + kRescaleThreshold)) {   // also when m is still -inf
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                const float m_new = fmaxf(m[x], mx[x]);
                const float alpha = (m_new == m[x]) ? 1.f : ex2(m[x] - m_new);   // 0 when nothing has been accumulated yet
                lsum[x] *= alpha;
                acc[x] *= alpha;
#pragma unroll
                for (int mb = 0; mb < kMB; ++mb) { o[mb][x] *= alpha; o[mb][2 + x] *= alpha; }
                m[x] = m_new;
            }
        }
        float pr[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) pr[x] = ex2(s[x] - ((m[x & 1] == kNegInf) ? 0.f : m[x & 1]));
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const float ps = pr[x] + pr[2 + x];
            acc[x] += ps;
            lsum[x] += ps;
        }
        // P^T as the B operand of O^T += V^T P^T: keys along the contraction, heads along the columns
        constexpr int kTerms = kStatic ? 3 : 1;                              // bf16 terms of a probability
        uint32_t b0[kTerms], b1[kTerms];
#pragma unroll
        for (int t = 0; t < kTerms; ++t) {
            b0[t] = transpose8x8(pack_bf16(pr[0], pr[1]));
            b1[t] = transpose8x8(pack_bf16(pr[2], pr[3]));
            if (t + 1 < kTerms) {
#pragma unroll
                for (int x = 0; x < 4; ++x) pr[x] -= __bfloat162float(__float2bfloat16_rn(pr[x]));   // exact: what the terms so far leave
            }
        }

        // ---- O += P V ----
        ok = mbar_wait(bar_full(1), par, abort_flag, p.status);
        if (!ok) break;
        base = stage_addr(1);
        const int row = (lane >> 4) * 8 + (lane & 7);                        // token addressed by this lane
#pragma unroll
        for (int mb = 0; mb < kMB; ++mb) {
            const int ch = 2 * mb + ((lane >> 3) & 1);
            uint32_t a[4];
            ldsm_x4_trans(page_chunk<D>(base, row, ch), a);
#pragma unroll
            for (int t = 0; t < kTerms; ++t) mma_bf16(o[mb], a, b0[t], b1[t]);
        }
        refill(true);
        cur = nn;
    }
    park();

    // error path only: give this warp's copies in flight (at most two pages) time to land before the CTA retires
    if (!ok && warp < n_cta) {
        const unsigned long long t0 = global_ns();
        while (global_ns() - t0 < 50000ull) { }
    }
    lsum[0] = over_keys(lsum[0]);
    lsum[1] = over_keys(lsum[1]);
    if (g == 0) {
        *reinterpret_cast<float2 *>(wm + warp * kMaxRep + 2 * tq) = make_float2(m[0], m[1]);
        *reinterpret_cast<float2 *>(wl + warp * kMaxRep + 2 * tq) = make_float2(lsum[0], lsum[1]);
    }
    // the table of the CTA's slots cleared for the merge of the parked sums
    for (int idx = threadIdx.x; idx < n_local * kMaxRep; idx += kThreads) cslot[idx] = 0.f;
    __syncthreads();                                                         // every stage consumed: the ring is free
    // (after an expired wait the CTA goes on with whatever it has: its peers wait for it at the cluster's barriers)

    // ---- merge the warps of the CTA ----
    float *obuf = reinterpret_cast<float *>(smem);                           // [warp][kMaxRep][kORow]
    {
        float *h0 = obuf + (warp * kMaxRep + 2 * tq) * C::kORow + g;
        if (2 * tq < rep) {
#pragma unroll
            for (int mb = 0; mb < kMB; ++mb) { h0[mb * 16] = o[mb][0]; h0[mb * 16 + 8] = o[mb][2]; }
        }
        if (2 * tq + 1 < rep) {
#pragma unroll
            for (int mb = 0; mb < kMB; ++mb) { h0[C::kORow + mb * 16] = o[mb][1]; h0[C::kORow + mb * 16 + 8] = o[mb][3]; }
        }
    }
    if (warp < rep) {                                                        // warp h takes head h: lane w holds warp w's (m, l)
        const int h = warp;
        const float mw = lane < kWarps ? wm[lane * kMaxRep + h] : kNegInf;
        float M = mw;
#pragma unroll
        for (int of = 8; of > 0; of >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, of));
        const float f = (mw == kNegInf) ? 0.f : ex2(mw - M);
        float Lh = lane < kWarps ? wl[lane * kMaxRep + h] * f : 0.f;
#pragma unroll
        for (int of = 8; of > 0; of >>= 1) Lh += __shfl_xor_sync(0xffffffffu, Lh, of);
        if (lane < kWarps) ww[h * kMaxCluster + lane] = f;
        if (lane == 0) {
            cm[h] = (Lh > 0.f) ? M + lg2(Lh) : kNegInf;                      // log2-sum-exp of the CTA's range
            cl[h] = (Lh > 0.f) ? rcp(Lh) : 0.f;
        }
    }
    __syncthreads();
    // What the other CTAs of the cluster need of this one goes straight into their shared memory: its log2-sum-exps to all of
    // them, its output rows (relative to its own sum) to the one that writes them out.
    cluster_wait();                                                          // they have all started
    if (static_cast<int>(threadIdx.x) < (rep << ls)) {
        const int h = threadIdx.x >> ls, k = threadIdx.x & (n_splits - 1);
        if (n_splits == 1) cw[h * kMaxCluster] = cm[h];
        else peer_push(peer_addr(smem_u32(cw + h * kMaxCluster + split), k), cm[h], peer_addr(bar_in, k));
    }
    const int n_f4 = rep * (D / 4);                                          // the rep output rows as float4 (16 .. 256)
    const int lf = 31 - __clz(n_f4) - ls;                                    // log2 of a CTA's share of them
    if (static_cast<int>(threadIdx.x) < n_f4) {
        const int ff = threadIdx.x, h = ff / (D / 4);
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const float4 v = *reinterpret_cast<const float4 *>(obuf + (w * kMaxRep + h) * C::kORow + (ff % (D / 4)) * 4);
            const float f = ww[h * kMaxCluster + w];
            a.x += f * v.x; a.y += f * v.y; a.z += f * v.z; a.w += f * v.w;
        }
        const float inv = cl[h];
        a.x *= inv; a.y *= inv; a.z *= inv; a.w *= inv;
        const int owner = ff >> lf, at = (split << lf) + (ff & ((1 << lf) - 1));
        if (n_splits == 1) *reinterpret_cast<float4 *>(smem + C::kInOff + at * 16) = a;
        else peer_push4(peer_addr(sbase + C::kInOff + at * 16, owner), a, peer_addr(bar_in, owner));
    }
    // parked sums -> shares of the range's sum.  No slot's sum exceeds it, so the shares are at most 1 and add up without a
    // maximum pass (a share below 2^-126 counts as nothing).
    if (p.mass) {
        const int n_ent = ctrs[1];
        for (int idx = threadIdx.x; idx < n_ent << lr; idx += kThreads) {
            const int e = idx >> lr, h = idx & (rep - 1);
            const float v = ent_val[e * rep2 + h];
            if (v != kNegInf) atomicAdd(&cslot[(ent_slot[e] - slot_first) * kMaxRep + h], ex2(v - cm[h]));
        }
    }
    if (p.mass) {
        __syncthreads();                                                     // the shares are complete
        const int owner = ctrs[3];
        if (owner >= 0 && static_cast<int>(threadIdx.x) < rep)
            peer_push(peer_addr(sbase + C::kShareOff + (split * kMaxRep + threadIdx.x) * 4, owner), cslot[threadIdx.x], peer_addr(bar_share, owner));
    }
    if (n_splits == 1) __syncthreads();
    else wait_for_peers(bar_in, p.status);

    // ---- merge the CTAs of the cluster: every CTA takes its share of the rows, thread (float4, CTA) ----
    const long long row_h0 = static_cast<long long>(ep.q_off) * p.Hq + kvh * rep;             // + h: (row, head) index
    auto weight_of = [&](int h, int k) -> float {                            // of CTA k in head h; by whole groups of n_splits lanes
        const float x = cw[h * kMaxCluster + k];
        float mxv = x;
        for (int of = n_splits >> 1; of > 0; of >>= 1) mxv = fmaxf(mxv, __shfl_xor_sync(0xffffffffu, mxv, of));
        const float e = (x != kNegInf) ? ex2(x - mxv) : 0.f;
        float sum = e;
        for (int of = n_splits >> 1; of > 0; of >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, of);
        return (sum > 0.f) ? e / sum : 0.f;
    };
    if (static_cast<int>(threadIdx.x) < ((n_f4 + 31) & ~31)) {
        const bool mine = static_cast<int>(threadIdx.x) < n_f4;
        const int fl = threadIdx.x >> ls, k = threadIdx.x & (n_splits - 1), f4 = (split << lf) + fl;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (mine) v = *reinterpret_cast<const float4 *>(smem + C::kInOff + ((k << lf) + fl) * 16);
        const float w = weight_of(mine ? f4 / (D / 4) : 0, k);
        v.x *= w; v.y *= w; v.z *= w; v.w *= w;
        for (int of = n_splits >> 1; of > 0; of >>= 1) {
            v.x += __shfl_xor_sync(0xffffffffu, v.x, of);
            v.y += __shfl_xor_sync(0xffffffffu, v.y, of);
            v.z += __shfl_xor_sync(0xffffffffu, v.z, of);
            v.w += __shfl_xor_sync(0xffffffffu, v.w, of);
        }
        if (mine && k == 0) {
            uint2 o2;
            o2.x = pack_bf16(v.x, v.y);
            o2.y = pack_bf16(v.z, v.w);
            *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(p.out) + row_h0 * D + f4 * 4) = o2;
        }
    }
    if (!p.mass) return;
    // Masses: every CTA writes the slots whose pages begin in its range (and the empty ones behind them), its last slot with
    // what the CTAs behind have sent.
    float *wt = wm;                                                          // [kMaxRep][kMaxCluster] (the warps' words are spent)
    static_assert(kMaxRep * kMaxCluster <= 2 * kWarps * kMaxRep && kMaxRep * kMaxCluster <= 128 && kThreads >= 256 + 128, "weights");
    if (threadIdx.x >= 256) {                                                // the warps that have no output to write
        const int t = threadIdx.x - 256, h = t >> ls, k = t & (n_splits - 1);
        const float w = weight_of(h < rep ? h : 0, k);
        if (h < rep) wt[h * kMaxCluster + k] = w;
    }
    __syncthreads();
    if (n_splits > 1) wait_for_peers(bar_share, p.status);
    if (n_cta > 0) {
        int s0 = slot_first, s1 = G + 1;                                     // this CTA's slots
        if (split == 0) s0 = 0;
        for (int k = split - 1; k >= 0; --k)
            if (rng_tab[k].y > 0) {
                if (rng_tab[k].x + rng_tab[k].y - 1 == slot_first) ++s0;     // begins in a range before
                break;
            }
        for (int k = split + 1; k < n_splits; ++k)
            if (rng_tab[k].y > 0) {
                s1 = max(rng_tab[k].x, slot_first + n_local);
                break;
            }
        for (int idx = threadIdx.x; idx < (s1 - s0) << lr; idx += kThreads) {
            const int h = idx & (rep - 1), s = s0 + (idx >> lr);
            const float *w = wt + h * kMaxCluster;
            float sum = 0.f;
            if (s >= slot_first && s < slot_first + n_local) {
                sum = w[split] * cslot[(s - slot_first) * kMaxRep + h];
                if (s == slot_first + n_local - 1)
                    for (int k = split + 1; k < n_splits && rng_tab[k].x <= s; ++k)
                        if (rng_tab[k].y > 0 && rng_tab[k].x == s) sum += w[k] * share_in[k * kMaxRep + h];
            }
            p.mass[(row_h0 + h) * p.mass_stride + s] = sum;
        }
    }
}

template <int D, bool kStatic, typename P>
cudaError_t launch(const P &p, const ClusterDecodeParams &d, int batch, int cluster, cudaStream_t st)
{
    if (batch <= 0) return cudaSuccess;
    if (cluster < 1 || cluster > kMaxCluster || (cluster & (cluster - 1)) || d.list_pages > kClusterMaxPages) return cudaErrorInvalidValue;
    const cudaError_t e = launch_pdl(decode_cluster_kernel<D, kStatic>, dim3(cluster, d.Hkv, batch), dim3(kThreads),
                                     Cfg<D>::smem_bytes(d.list_pages, d.list_slots, d.rep), st, p, cluster);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <int D, bool kStatic>
cudaError_t prepare(ClusterCaps *caps)
{
    const auto kernel = decode_cluster_kernel<D, kStatic>;
    const int most = Cfg<D>::smem_bytes(kClusterMaxPages, kClusterMaxPages, kMaxRep);
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e != cudaSuccess) return e;
    const bool wide = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    // A device's answers are asked for once: ten occupancy queries per kernel are most of what making a small cache takes.  They
    // are kept without the heap or a lock, since the entry point that promises to do without comes here, too (callers that race
    // store the same values).
    static ClusterCaps known[kMaxDevices];
    static int ready[kMaxDevices];
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    const bool keep = dev >= 0 && dev < kMaxDevices;
    if (keep && __atomic_load_n(&ready[dev], __ATOMIC_ACQUIRE)) {
        *caps = known[dev];
        cudaGetLastError();
        return cudaSuccess;
    }
    for (int i = 0; i < 5; ++i)
        for (int two = 0; two < 2; ++two) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(1 << i);
            cfg.blockDim = dim3(kThreads);
            cfg.dynamicSmemBytes = two ? std::min(kClusterPairSmem, most) : most;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = 1 << i;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int n = 0;
            if ((i == 4 && !wide) || cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) n = 0;
            (two ? caps->two : caps->one)[i] = n;
        }
    if (keep) {
        known[dev] = *caps;
        __atomic_store_n(&ready[dev], 1, __ATOMIC_RELEASE);
    }
    cudaGetLastError();
    return cudaSuccess;
}

}  // namespace

int decode_cluster_smem(int head_dim, int list_pages, int list_slots, int rep)
{
    return head_dim == 128 ? Cfg<128>::smem_bytes(list_pages, list_slots, rep) : Cfg<64>::smem_bytes(list_pages, list_slots, rep);
}

cudaError_t prepare_decode_cluster(int head_dim, ClusterCaps *caps)
{
    if (head_dim == 128) return prepare<128, false>(caps);
    if (head_dim == 64) return prepare<64, false>(caps);
    return cudaErrorInvalidValue;
}

cudaError_t prepare_decode_static(int head_dim, ClusterCaps *caps)
{
    if (head_dim == 128) return prepare<128, true>(caps);
    if (head_dim == 64) return prepare<64, true>(caps);
    return cudaErrorInvalidValue;
}

cudaError_t launch_decode_cluster(const ClusterDecodeParams &p, int head_dim, int batch, int cluster, cudaStream_t st)
{
    if (head_dim == 128) return launch<128, false>(p, p, batch, cluster, st);
    if (head_dim == 64) return launch<64, false>(p, p, batch, cluster, st);
    return cudaErrorInvalidValue;
}

cudaError_t launch_decode_static(const StaticDecodeParams &p, int head_dim, int cluster, cudaStream_t st)
{
    if (head_dim == 128) return launch<128, true>(p, p.d, 1, cluster, st);
    if (head_dim == 64) return launch<64, true>(p, p.d, 1, cluster, st);
    return cudaErrorInvalidValue;
}

}  // namespace enl
