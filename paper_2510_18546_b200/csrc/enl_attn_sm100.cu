// Selective-KV flash attention with fused per-group mass, sm_100a (tcgen05 + TMEM + TMA).
//
// What it computes (paper, App. A: softmax(Q K^T / sqrt(D)) V; App. C: the prompt is the selected
// groups followed by the new tokens; Sec. 3.3: attention between new tokens and a group):
// one CTA takes two Q tiles of 128 rows each -- (128/rep) consecutive query tokens x the rep q heads
// that read one kv head -- and walks the key stream of its episode in steps of 64 keys: the selected groups' pages in
// list order (four 16-token pages a step, fetched as separate TMA boxes from wherever the pages lie in the pool), then the
// new-token keys up to the causal limit.  Per step:
//   S_i = Q_i K^T            tcgen05.mma, operands in shared memory, accumulator in TMEM
//                            (after an MMA of one K step that puts -inf under page padding, where there is any)
//   p   = exp2(S * c - m)    one thread per row, fp32; causally hidden columns -> 0
//   O_i += P_i V             tcgen05.mma, P (bf16) read from TMEM, V from shared memory
// The row sum of p is split by the slot (selected group, or the new tokens) each 16-key page belongs
// to; when a slot ends its log2-sum-exp is parked: in shared memory for calls with few slots, whose values are turned into
// probabilities after the last step, else in the mass buffer, where mass_finish_kernel does.  With KV splits every split writes partial results that a
// second kernel merges, or (two splits, head_dim 128) the two CTAs of a cluster merge in place.
//
// Roles (12 warps): warps 0-3 are the softmax warpgroup of Q tile 0, warps 4-7 that of Q tile 1: one
// thread per query row holds the row's 64 scores of a step in registers, so the row maximum, the
// exponentials and the four page sums need no exchange between threads.  Warps 8 and 10 fetch K and V, warps 9 and 11 issue the
// MMAs of tile 0 and tile 1 (9 owns the TMEM).  A softmax warpgroup and its issuer are a walker.
//
// What bounds it, and why it is split like this (all cycles per 128 keys and pair of Q tiles, 64 groups, 1024 rows; the tensor pipe
// needs 2176, the special-function unit 2048):
//  * S is double-buffered: Q K^T of step j + 2 is issued behind P V of step j, so a softmax warp finds its next scores waiting.  Tiles of
//    128 keys leave no TMEM for that; their chain scores -> softmax -> P V -> Q K^T took 3640.
//  * The issuers: issuing an MMA costs its scheduler about 13 issue slots, a wait its warp 100 cycles and more.  One warp that
//    alternated between the tiles was what both waited for (4700 with these steps); one warp for Q K^T and one for P V slowed the
//    two softmax warps of the former's scheduler to 4300.  An issuer per tile, on different schedulers, waits for nothing but its own tile.
//  * The producers: a TMA box costs its warp 50 cycles and a fetch some 200 to 350 more.  One producer with two boxes of half a page
//    per page needed 3800.
//  * Turns: the warps of the two tiles that share a scheduler take their exponentials one after the other (a named barrier).  Left alone
//    the tiles fall into step, both wanting the special-function unit and then both not: 4150 against 3500.
// Together: long calls 251 -> 238 thousand cycles a launch (then at the power cap), the planner's 512 rows over 24 groups 33.5 -> 31.0 us
// (29.9 to 30.3 with the early pages and a start that takes no division).
// Not kept: exponentials on the FMA pipe, a quarter of them 270 thousand cycles (the warps have issue slots, but a step is one chain);
// the maximum beside the exponentials, with the reference a step behind: 6700 against 5860 us a pass; tiles of 128 keys with all of the
// above: the same on long calls, 8 % slower on the planner's, whose ends waste half a tile.
//
// Calls with few CTAs run the second form (kHalves): a CTA has one Q tile, its two walkers take the first and the second half of its steps
// and put outputs and slots together at the end, in TMEM lanes that both read: twice as many CTAs, or half as many splits to merge through
// memory, and no walker idle where a call has fewer rows than two tiles.  With masses, 2560 keys: 41 rows 16.6 -> 15.4 us, 128 rows
// 22.6 -> 19.1, 256 rows 28.3 -> 26.2; 512 rows at head_dim 64, which has no pairs of CTAs, 39.0 -> 34.1.
//
// TMEM columns: S0 [0,128) S1 [128,256), two buffers of 64 columns each, O0 [256,384) O1 [384,512); P_i (bf16 pairs) overwrites the
// first 32 columns of the buffer that held its scores once these are in registers.
#include <cuda_bf16.h>

#include "attn_ops.cuh"
#include "enl_internal.h"
#include "tmem_ops.cuh"

namespace enl {
namespace {

constexpr int kThreads      = 384;
constexpr int kSoftmaxWarps = 8;
constexpr int kRegsSoftmax  = 184;            // 256 x 184 + 128 x 128 <= 384 x 168, what the launch allocates
constexpr int kRegsOther    = 128;
constexpr int kKWarp        = 8;              // fetches K
constexpr int kVWarp        = 10;             // fetches V
constexpr int kMmaWarp      = 9;              // issues the MMAs of Q tile 0 (and owns the TMEM); those of tile 1 two warps on
constexpr uint32_t kTmemCols = 512;
constexpr int kParkSlots = 25;                // calls with up to this many mass slots park their slot sums in shared memory
constexpr int kStepPages = kStepKeys / kPageTokens;
constexpr float kRescaleThreshold = 8.0f;     // log2 units: p stays below 2^8 between updates of the reference

template <int D>
struct Cfg {
    static constexpr int kBlocks    = D / 64;             // 64-channel (128-byte) column blocks
    static constexpr int kBlockBytes = 128 * 128;          // Q tile: 128 rows x 128 B
    static constexpr int kTileBytes = kBlocks * kBlockBytes;
    // K or V of a step: eight groups of 8 rows, a group being one 8 x 128-byte block per 64 channels
    static constexpr int kGroupBytes = kBlocks * 1024;
    static constexpr int kStepBytes = kStepKeys / 8 * kGroupBytes;
    static constexpr int kRing      = 4;                  // steps whose K (and whose V) are in shared memory at once
    static constexpr int kRingOff   = kQTiles * kTileBytes;
    static constexpr int kBarOff    = kRingOff + 2 * kRing * kStepBytes;
    // the operands of the MMA that hides page padding, 16 bytes per row: 1 for 8 queries (behind the barriers; every group of
    // 8 rows reads them), 0 or -inf for every key of a step in the ring; and a word per step: has it padding at all?
    static constexpr int kHideFlagOff = kBarOff + 352;
    static constexpr int kOnesOff   = kBarOff + 384;
    // pair merge: what the other CTA of the cluster knows about this CTA's rows, [tile][128] x (m, l, shared-slot log-sum, -)
    static constexpr int kXpeerOff  = kBarOff + 512;
    static constexpr int kHideOff   = kXpeerOff + kQTiles * 128 * 16;
    static constexpr int kHideBytes = kStepKeys * 16;
    // slot log-sums of calls with at most kParkSlots slots, [tile][slot][128 rows] fp32 (what is left of the 227 KB)
    static constexpr int kParkOff   = kHideOff + kRing * kHideBytes;
    static constexpr int kSmemBytes = kParkOff + kQTiles * kParkSlots * 128 * 4 + 1024;   // + alignment slack
    static_assert(8 * 33 + 8 <= 352 && kSmemBytes <= 232448, "shared memory");
};

// ---- the kernel ----------------------------------------------------------------------------
template <int D, bool kHalves>
__global__ void __launch_bounds__(kThreads, 1) attn_kernel(const __grid_constant__ AttnParams p)
{
    using C = Cfg<D>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t sbase = (raw + 1023u) & ~1023u;               // 1024-B aligned (swizzle atoms)
    uint8_t *smem = smem_raw + (sbase - raw);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // shared-memory map
    auto q_addr     = [&](int i) { return sbase + static_cast<uint32_t>(i * C::kTileBytes); };
    auto k_addr = [&](int x) { return sbase + static_cast<uint32_t>(C::kRingOff + 2 * x * C::kStepBytes); };
    auto v_addr = [&](int x) { return k_addr(x) + static_cast<uint32_t>(C::kStepBytes); };
    const uint32_t bar0 = sbase + C::kBarOff;
    const uint32_t bar_q_full = bar0;
    auto bar_k_full  = [&](int x) { return bar0 + 8u * (1 + x); };             // x: place in the ring
    auto bar_k_empty = [&](int x) { return bar0 + 8u * (5 + x); };
    auto bar_v_full  = [&](int x) { return bar0 + 8u * (9 + x); };
    auto bar_v_empty = [&](int x) { return bar0 + 8u * (13 + x); };
    auto bar_s_full  = [&](int i, int b) { return bar0 + 8u * (17 + 2 * i + b); };   // b: step & 1
    auto bar_p_full  = [&](int i, int b) { return bar0 + 8u * (21 + 2 * i + b); };
    auto bar_pv_done = [&](int i) { return bar0 + 8u * (25 + i); };            // P_i V of a step
    auto bar_o_done  = [&](int i) { return bar0 + 8u * (27 + i); };            // of the last step
    // pair merge (cluster of two): the peer's row sums have arrived / the peer's partial output has arrived /
    // the peer's K/V ring is idle and may be written / the peer has received what this CTA staged for it
    const uint32_t bar_peer_ml = bar0 + 8u * 29;
    const uint32_t bar_peer_o = bar0 + 8u * 30;
    const uint32_t bar_peer_free = bar0 + 8u * 31;
    const uint32_t bar_peer_ack = bar0 + 8u * 32;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + C::kBarOff + 8 * 33);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    volatile uint32_t *hide_flag = reinterpret_cast<volatile uint32_t *>(smem + C::kHideFlagOff);

    if (p.wait_first) pdl_wait();
    // work item
    const Item it = p.items[blockIdx.x];
    const EpInfo ep = p.eps[it.ep];
    const int rep = p.rep;
    const int lr = 31 - __clz(rep);                                      // a power of two
    const int tile_tokens = kTileRows >> lr;
    // Calls with few CTAs (kHalves): one Q tile per CTA, and the two walkers (softmax warpgroup + issuer) take half of its steps each
    // and put their results together at the end.  Else a walker has a Q tile of its own and walks all the steps.
    const int t_hi = min(it.t0 + (kHalves ? 1 : kQTiles) * tile_tokens, ep.n_q);    // exclusive
    const int n_qt = (t_hi - it.t0 > tile_tokens) ? 2 : 1;
    const int c_max = ep.n_new - ep.n_q + t_hi - 1;                      // last new key any row sees
    const int n_csteps = (ep.n_entries + kStepPages - 1) / kStepPages;  // steps over cached pages
    const int total_steps = n_csteps + c_max / kStepKeys + 1;
    const int j_beg = static_cast<int>(static_cast<long long>(total_steps) * it.split / p.n_splits);
    const int j_end = static_cast<int>(static_cast<long long>(total_steps) * (it.split + 1) / p.n_splits);
    const int n_steps = j_end - j_beg;
    const int n_walk = kHalves ? min(2, n_steps) : n_qt;                  // walkers with work
    // walker i: its steps and the first of them; in the order in which K and V are fetched, its step jj is number place_of(i, jj), and
    // number v is step step_of(v) of the stream
    auto count_of = [&](int i) { return kHalves ? (n_steps + 1 - i) >> 1 : n_steps; };
    auto first_of = [&](int i) { return kHalves && i ? j_beg + ((n_steps + 1) >> 1) : j_beg; };
    auto place_of = [&](int i, int jj) { return kHalves ? 2 * jj + i : jj; };
    auto step_of = [&](int v) { return kHalves ? first_of(v & 1) + (v >> 1) : j_beg + v; };

    // ---- set-up ----
    if (threadIdx.x == 0) {
        *abort_flag = 0;
        mbar_init(bar_q_full, 1);
        for (int x = 0; x < C::kRing; ++x) {
            mbar_init(bar_k_full(x), 1); mbar_init(bar_k_empty(x), kHalves ? 1 : n_qt);
            mbar_init(bar_v_full(x), 1); mbar_init(bar_v_empty(x), kHalves ? 1 : n_qt);
        }
        for (int i = 0; i < kQTiles; ++i) {
            for (int b = 0; b < 2; ++b) {
                mbar_init(bar_s_full(i, b), 1);
                mbar_init(bar_p_full(i, b), 4);       // one arrival per softmax warp of the tile
            }
            mbar_init(bar_pv_done(i), 1);
            mbar_init(bar_o_done(i), 1);
        }
        mbar_init(bar_peer_ml, 1);                                   // this thread's arrival below + 16 bytes per row from the peer
        mbar_init(bar_peer_o, 1);                                    // this thread's arrival below + 64 KB from the peer
        mbar_init(bar_peer_free, 1);
        mbar_init(bar_peer_ack, 1);
        if (p.pair_merge) {
            mbar_expect_tx(bar_peer_ml, static_cast<uint32_t>(n_qt * 128 * 16));
            mbar_expect_tx(bar_peer_o, 4u * 16384u);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x < 8) {
        *reinterpret_cast<uint4 *>(smem + C::kOnesOff + threadIdx.x * 16) = make_uint4(0x3f80u, 0u, 0u, 0u);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const bool pair = !kHalves && p.pair_merge != 0;
    if (pair) cluster_sync_all();                // the peer's barriers exist before anything is sent to them
    // Everything above touched only shared memory, TMEM and the gather plan.  From here on the pool is read, which the previous kernel of
    // the stream leaves alone (wait_first), and the caller's tensors and the scratch are, for which it must have finished.
    pdl_trigger();
    // While the previous kernel drains, the producers (which wait for it later) fetch the cached pages of the first steps: the pool is
    // written by launches of this library only, and none has come in between.  What else comes first is asked into the L2: the Q tiles and
    // new tokens.  (Only CTAs of the first wave wait for the previous kernel; for the others this would be loads issued twice.)
    // How many steps: with none a launch took 2.4 us from the wait to its first scores (the page words' round trip and then the pages').
    // With two steps the planner's layer took 29.3 us where none took 30.5 and four 29.7; where the kernel before is the one that merges the splits,
    // whose reads more loads hold up, one: 128 rows over 2560 keys 19.0 -> 18.35 us, with two steps 18.6, with four 19.3.
    const bool producer = warp == kKWarp || warp == kVWarp;
    if (producer && n_steps > 0 && static_cast<int>(blockIdx.x) < p.first_wave) {
        if (warp == kKWarp && lane < n_qt * C::kBlocks)
            tma_prefetch_3d(&p.tm_q, (lane % C::kBlocks) * 64, it.kvh * rep, ep.q_off + it.t0 + (lane / C::kBlocks) * tile_tokens);
        constexpr int kBoxes = kStepKeys / kBoxRows<D>;              // of a step
        const int vn = lane / kBoxes, jn = step_of(vn);
        if (vn < min(C::kRing, n_steps) && jn >= n_csteps)
            tma_prefetch_4d(warp == kKWarp ? &p.tm_knew : &p.tm_vnew, 0, ep.new_off + (jn - n_csteps) * kStepKeys + lane % kBoxes * kBoxRows<D>, 0, it.kvh);
    }
    if (!producer) pdl_wait();
    // Beyond kParkSlots the kernel that merges splits is told which slots a split writes of a row, and the others are left as they were:
    // clearing them took 30 us of the 81 that the masses of 128 rows over 400 groups in 17 splits (8 heads) did a thread per row, and
    // reading them as long again.  (Here, by a warp that would only wait now: the softmax warps have no registers to spare; from their
    // epilogue a layer of the planner's took 0.8 % longer, from the producers' end the loop 3 to 8 %.)
    if (warp == kMmaWarp + 2 && it.kvh == 0 && p.part_rng && n_steps > 0) {
        const int first = j_beg < n_csteps ? __ldg(p.stream_meta + ep.stream_off + j_beg * kStepPages) >> 8 : ep.n_slots;
        const int last = j_end > n_csteps ? ep.n_slots : __ldg(p.stream_meta + ep.stream_off + j_end * kStepPages - 1) >> 8;
        for (int t = it.t0 + lane; t < t_hi; t += 32)
            p.part_rng[static_cast<long long>(it.split) * p.n_q_total + ep.q_off + t] = make_int2(first, last);
    }

    bool ok = true;

    if (warp >= kSoftmaxWarps) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsOther));
      if (warp == kKWarp || warp == kVWarp) {
        // ================= TMA producers =================
        // K and V have a warp each, and a box is a whole page of a kv head: eight lanes with half a page each took 767 cycles per 16 KB,
        // four with a page take 562 (the wait for the ring's place included).
        const bool is_k = warp == kKWarp;
        const CUtensorMap *tm_pool = is_k ? &p.tm_kpool : &p.tm_vpool, *tm_new = is_k ? &p.tm_knew : &p.tm_vnew;
        const uint32_t ring = is_k ? k_addr(0) : v_addr(0), full0 = is_k ? bar_k_full(0) : bar_v_full(0),
                       empty0 = is_k ? bar_k_empty(0) : bar_v_empty(0);
        if (n_steps > 0) {
            // before anything of the caller's: the wait for the previous kernel, and then the Q tiles first
            const int early = p.wait_first || static_cast<int>(blockIdx.x) >= p.first_wave ? 0 : p.n_splits > 1 && !pair ? 1 : 2;   // nothing to wait for: Q first
            bool waited = false;
            auto wait_previous = [&]() {
                pdl_wait();
                waited = true;
                if (is_k && lane == 0) {
                    mbar_expect_tx(bar_q_full, static_cast<uint32_t>(n_qt * C::kTileBytes));
                    for (int i = 0; i < n_qt; ++i)
                        for (int b = 0; b < C::kBlocks; ++b)
                            tma_load_3d(q_addr(i) + b * C::kBlockBytes, &p.tm_q, b * 64, it.kvh * rep,
                                        ep.q_off + it.t0 + i * tile_tokens, bar_q_full);
                }
                __syncwarp();
            };
            // Page words (id; slot << 8 | valid keys) of 32 pages at a time, one per lane, fetched eight steps ahead (of either walker): a
            // load in every step kept the ring waiting for the L2.
            constexpr int kBatch = 32 / kStepPages;
            struct Words { int id, meta; };
            auto words = [&](int j) {
                const int e = j * kStepPages + lane;
                Words w = {kZeroPage, kPageTokens};
                if (e < n_csteps * kStepPages) {
                    w.id = __ldg(p.stream_page + ep.stream_off + e);
                    w.meta = __ldg(p.stream_meta + ep.stream_off + e);
                }
                return w;
            };
            Words cur0 = {0, 0}, cur1 = {0, 0}, next0 = words(first_of(0)), next1 = kHalves ? words(first_of(1)) : cur1;
            int fetched = 0;
            for (int v = 0; v < n_steps; ++v) {
                const int i = kHalves ? v & 1 : 0, jj = kHalves ? v >> 1 : v, j = step_of(v), x = v % C::kRing;
                if (jj % kBatch == 0) {
                    if (i == 0) { cur0 = next0; next0 = words(j + kBatch); }
                    else { cur1 = next1; next1 = words(j + kBatch); }
                }
                if (!waited && (v >= early || j >= n_csteps)) wait_previous();
                const int pg = lane % kStepPages, at = jj % kBatch * kStepPages;
                const int group = (__shfl_sync(kFull, i ? cur1.id : cur0.id, at + pg) * p.Hkv + it.kvh) * kPageGroups<D>;
                const int valid = __shfl_sync(kFull, i ? cur1.meta : cur0.meta, at + pg) & 0xff;
                if (v >= C::kRing) ok = mbar_wait(empty0 + 8u * x, static_cast<uint32_t>((v / C::kRing - 1) & 1), abort_flag, p.status);
                if (!ok) break;
                const uint32_t dst = ring + static_cast<uint32_t>(2 * x * C::kStepBytes), full = full0 + 8u * x;
                if (is_k) {
                    const bool padded = __any_sync(kFull, valid < kPageTokens);
                    if (lane == 0) hide_flag[x] = padded ? 1u : 0u;
                    if (padded) {                                    // what hides the padding of these keys: see issue_qk
                        uint4 *hide = reinterpret_cast<uint4 *>(smem + C::kHideOff + x * C::kHideBytes);
#pragma unroll
                        for (int y = 0; y < kStepKeys / 32; ++y) {
                            const int n = __shfl_sync(kFull, valid, 2 * y + (lane >> 4));
                            hide[y * 32 + lane] = make_uint4((lane & 15) < n ? 0u : 0xff80u, 0u, 0u, 0u);
                        }
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    }
                    __syncwarp();
                }
                if (lane == 0) mbar_expect_tx(full, static_cast<uint32_t>(C::kStepBytes));
                if (j < n_csteps) {
                    if (lane < kStepPages) tma_load_4d(dst + static_cast<uint32_t>(lane * 2 * C::kGroupBytes), tm_pool, 0, 0, 0, group, full);
                } else if (lane < kStepKeys / kBoxRows<D>) {
                    tma_load_4d(dst + static_cast<uint32_t>(lane * (kBoxRows<D> * D * 2)), tm_new, 0,
                                ep.new_off + (j - n_csteps) * kStepKeys + lane * kBoxRows<D>, 0, it.kvh, full);
                }
                ++fetched;
            }
            if (!waited) wait_previous();
            // error path only: let the copies already in flight land before the CTA retires
            if (!ok) {
                for (int f = max(0, fetched - C::kRing); f < fetched; ++f) {
                    const unsigned long long t0 = global_ns();
                    while (!mbar_try_wait(full0 + 8u * (f % C::kRing), static_cast<uint32_t>((f / C::kRing) & 1)) &&
                           global_ns() - t0 < 2000000ull) { }
                }
            }
        }
      } else {
        // ================= MMA issuer of a walker =================
        const int i = warp == kMmaWarp ? 0 : 1;
        const int n_mine = count_of(i);
        if (n_mine > 0 && i < n_walk) {
            constexpr uint32_t idesc_qk = make_idesc(kStepKeys, false), idesc_pv = make_idesc(D, true);
            // descriptor words: place x of the ring starts 2 * kStepUnits x address units behind place 0
            constexpr uint32_t kStepUnits = C::kStepBytes >> 4, kGroupUnits = C::kGroupBytes >> 4;
            const uint64_t dq0 = smem_desc(q_addr(kHalves ? 0 : i), 16), dk0 = smem_desc(k_addr(0), 16, C::kGroupBytes), dv0 = smem_desc(v_addr(0), 1024, C::kGroupBytes);
            const uint32_t dq_lo = static_cast<uint32_t>(dq0), dq_hi = static_cast<uint32_t>(dq0 >> 32);
            const uint32_t dk_lo = static_cast<uint32_t>(dk0), dk_hi = static_cast<uint32_t>(dk0 >> 32);
            const uint32_t dv_lo = static_cast<uint32_t>(dv0), dv_hi = static_cast<uint32_t>(dv0 >> 32);
            const uint64_t d_ones = smem_desc_plain(sbase + C::kOnesOff, 0u), d_hide = smem_desc_plain(sbase + C::kHideOff, 128u);
            const uint32_t t_si = tmem_base + static_cast<uint32_t>(i * 128), t_oi = tmem_base + static_cast<uint32_t>(256 + i * 128);
            // S_i = Q_i K^T into buffer b; where a page is padded (`hide`) an MMA of one K step before it puts -inf under the padding
            // keys and 0 under the others.  It costs the pipe 1/8 of the step's Q K^T and takes the compares and selects of
            // ragged pages out of the softmax warps (in the tiles of 128 keys: 4374 -> 3999 cycles).
            auto issue_qk = [&](int x, int b, bool hide) {
                const uint32_t ka = dk_lo + static_cast<uint32_t>(x) * (2u * kStepUnits), d = t_si + static_cast<uint32_t>(b * kStepKeys);
                if (hide)
                    mma_ss2(d, static_cast<uint32_t>(d_ones), static_cast<uint32_t>(d_ones >> 32),
                            static_cast<uint32_t>(d_hide) + static_cast<uint32_t>(x) * (C::kHideBytes >> 4),
                            static_cast<uint32_t>(d_hide >> 32), idesc_qk, 0u);
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk) {
                    const uint32_t in_row = static_cast<uint32_t>((kk & 3) * 2);                       // 32 bytes per 16 channels
                    mma_ss2(d, dq_lo + static_cast<uint32_t>((kk >> 2) * (C::kBlockBytes >> 4)) + in_row, dq_hi,
                            ka + static_cast<uint32_t>((kk >> 2) * (1024 >> 4)) + in_row, dk_hi, idesc_qk, kk > 0 || hide ? 1u : 0u);
                }
                tc_commit(bar_s_full(i, b));
                tc_commit(bar_k_empty(x));
            };
            // O_i (+)= P_i V; P of keys 2c, 2c+1 sits in column c of the buffer that held their scores
            auto issue_pv = [&](int x, int b, bool first) {
                const uint32_t va = dv_lo + static_cast<uint32_t>(x) * (2u * kStepUnits), a = t_si + static_cast<uint32_t>(b * kStepKeys);
#pragma unroll
                for (int k4 = 0; k4 < kStepPages; ++k4)                  // 16 keys = two groups of 8 rows, 8 columns of P
                    mma_ts2(t_oi, a + static_cast<uint32_t>(k4 * 8), va + static_cast<uint32_t>(k4 * 2) * kGroupUnits, dv_hi, idesc_pv,
                            (first && k4 == 0) ? 0u : 1u);
                tc_commit(bar_pv_done(i));
                tc_commit(bar_v_empty(x));
            };
            auto wait_k = [&](int v) { return mbar_wait(bar_k_full(v % C::kRing), static_cast<uint32_t>((v / C::kRing) & 1), abort_flag, p.status); };
            ok = mbar_wait(bar_q_full, 0, abort_flag, p.status);
            for (int jj = 0; jj < min(2, n_mine) && ok; ++jj) {
                const int v = place_of(i, jj);
                ok = wait_k(v);
                if (!ok) break;
                tc_fence_after();
                issue_qk(v, jj, hide_flag[v] != 0u);
            }
            for (int jj = 0; jj < n_mine && ok; ++jj) {
                const int v = place_of(i, jj), v2 = place_of(i, jj + 2), b = jj & 1;
                const bool more = jj + 2 < n_mine;
                // P comes last: nothing but the MMAs themselves stands between its arrival and the next scores
                ok = mbar_wait(bar_v_full(v % C::kRing), static_cast<uint32_t>((v / C::kRing) & 1), abort_flag, p.status);
                if (ok && more) ok = wait_k(v2);
                const bool hide = more && hide_flag[v2 % C::kRing] != 0u;
                if (ok) ok = mbar_wait(bar_p_full(i, b), static_cast<uint32_t>((jj >> 1) & 1), abort_flag, p.status);
                if (!ok) break;
                tc_fence_after();
                issue_pv(v % C::kRing, b, jj == 0);
                if (more) issue_qk(v2 % C::kRing, b, hide);
                else if (jj + 1 == n_mine) tc_commit(bar_o_done(i));
            }
            // pair merge: once every MMA of this CTA has completed, its K/V ring is idle and the peer may write
            // into it (only a CTA that finishes a Q tile receives anything)
            if (ok && pair && i == 0 && it.split < n_qt) {
                for (int t = 0; t < n_qt && ok; ++t) ok = mbar_wait(bar_o_done(t), 0, abort_flag, p.status);
                if (ok && lane == 0) peer_arrive(peer_addr(bar_peer_free, cluster_rank() ^ 1u));
            }
        }
      }
    } else {
      asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
      if ((warp >> 2) < n_walk) {
        // ================= softmax / epilogue: one thread per query row =================
        const int i = warp >> 2;                                   // walker
        const int tile_t0 = it.t0 + (kHalves ? 0 : i * tile_tokens);  // first token of its Q tile
        const int j0 = first_of(i), n_mine = count_of(i);          // its steps
        const int q4 = warp & 3;                                   // TMEM lane quadrant
        const int r = q4 * 32 + lane;
        const int t = tile_t0 + (r >> lr);           // episode-relative query token
        const int h = it.kvh * rep + (r & (rep - 1));
        const bool row_valid = t < ep.n_q;
        const int c = min(ep.n_new - ep.n_q + t, ep.n_new - 1);    // last visible new key
        const int c_lo = ep.n_new - ep.n_q + tile_t0;   // the same for the tile's first row: every row sees at least this far
        const int G = ep.n_slots;
        const uint32_t lane_sel = static_cast<uint32_t>(q4 * 32) << 16;
        const uint32_t t_s = tmem_base + lane_sel + static_cast<uint32_t>(i * 128);
        const uint32_t t_o = tmem_base + lane_sel + static_cast<uint32_t>(256 + i * 128);
        const bool split_mode = p.n_splits > 1 && !pair;
        // Where this row's slot log-sums are parked until the row's total is known: shared memory when the call has few
        // slots (one store per slot end, no round trip to the L2 at the end), else the buffer that takes the result.
        float *const slot_rows = split_mode ? p.part_slot : p.mass;
        const bool park_smem = p.park_smem != 0, want_slots = slot_rows != nullptr;
        float *slot_global = nullptr;
        if (row_valid && want_slots && !park_smem)
            slot_global = slot_rows + (static_cast<long long>((split_mode ? it.split * p.n_q_total : 0) + ep.q_off + t) * p.Hq + h) * p.mass_stride;
        float *park_row = reinterpret_cast<float *>(smem + C::kParkOff) + i * (kParkSlots * 128) + r;   // + slot * 128; (each walker its own slots)
        const float scale = p.scale_log2;

        // Where two split the steps between them (the CTAs of a pair, the walkers of a CTA) the slot in which they meet is walked by both.
        // The first writes it (adding what the second sends); the second keeps its part in `bnd` instead of storing it.
        int shared_slot = -1, skip_slot = -1;
        float bnd = kNegInf;
        const bool two_halves = kHalves && n_walk == 2;
        if (pair || two_halves) {
            const int jb = two_halves ? first_of(1) : (it.split == 0) ? j_end : j_beg;       // first step of the second
            const int last0 = (jb > n_csteps) ? G : (__ldg(p.stream_meta + ep.stream_off + jb * kStepPages - 1) >> 8);
            const int first1 = (jb < n_csteps) ? (__ldg(p.stream_meta + ep.stream_off + jb * kStepPages) >> 8) : G;
            if (last0 == first1) { shared_slot = last0; if ((two_halves ? i : it.split) == 1) skip_slot = last0; }
        }
        float m = kNegInf, l = 0.f, acc = 0.f;                     // reference (log2 units), row sum, sum of the current slot
        int cur_slot = 0;
        // The slot that ends (if `ends`, the same for the whole warp) parks its log2-sum-exp; the one behind it is the next in the list, since
        // every slot has a page.  Predicated stores and no shuffle: what comes back through the queue of the special-function unit, which the
        // other tile's warp keeps full, costs a hundred cycles and more.  (Branches with a shuffle and a logarithm per slot: 310 cycles of a
        // step of 1950, groups of two pages; 600 rows over 400 such groups 282 -> 256 us.  Slots staged in shared memory and written out a row
        // at a time: 330.  Without masses nothing is parked: 266 -> 237.)
        auto park = [&](bool ends, float v) {
            const bool mine = ends && cur_slot != skip_slot;
            if (mine && park_smem) park_row[cur_slot * 128] = v;
            if (mine && slot_global) slot_global[cur_slot] = v;
            bnd = ends && !mine ? v : bnd;
            cur_slot += ends ? 1 : 0;
        };

        // Slots of 32 pages at a time, one per lane, fetched eight steps ahead, and a warp-uniform mask of those pages whose slot differs
        // from the page before.  The pages of a new-token step are one slot (G).
        constexpr int kBatch = 32 / kStepPages;
        auto load_slots = [&](int jj) -> int {
            const int e = (j0 + jj) * kStepPages + lane;
            return e < n_csteps * kStepPages ? __ldg(p.stream_meta + ep.stream_off + e) >> 8 : G;
        };
        int slots_next = load_slots(0), slots = __shfl_sync(kFull, slots_next, 0);
        cur_slot = slots;
        uint32_t changes = 0;
        // The two warps that share a scheduler (one of each tile) take their exponentials in turns: both at once leave its special-function
        // unit idle while both do the rest.  (Named barriers 1..8: (tile, quadrant) may begin.)
        auto await_turn = [&](int jj) {
            if (n_walk == 2 && (i == 1 || jj > 0)) asm volatile("bar.sync %0, 64;" ::"r"(1 + q4 + 4 * i) : "memory");
        };
        auto pass_turn = [&](int jj) {
            if (n_walk == 2 && (i == 0 ? !kHalves || jj < count_of(1) : jj + 1 < count_of(0))) asm volatile("bar.arrive %0, 64;" ::"r"(1 + q4 + 4 * (i ^ 1)) : "memory");
        };

        int jj = 0;
        for (; jj < n_mine; ++jj) {
            const int j = j0 + jj;
            if (jj % kBatch == 0) {
                const int last = __shfl_sync(kFull, slots, 31);
                slots = slots_next;
                slots_next = load_slots(jj + kBatch);
                int prev = __shfl_up_sync(kFull, slots, 1);
                if (lane == 0) prev = last;
                changes = want_slots ? __ballot_sync(kFull, slots != prev) : 0u;
            }
            const uint32_t chg_mask = (changes >> (jj % kBatch * kStepPages)) & ((1u << kStepPages) - 1u);

            const uint32_t t_sb = t_s + static_cast<uint32_t>((jj & 1) * kStepKeys);
            ok = mbar_wait(bar_s_full(i, jj & 1), static_cast<uint32_t>((jj >> 1) & 1), abort_flag, p.status);
            if (!ok) break;
            tc_fence_after();

            // the row's 64 scores
            uint32_t su[kStepKeys];
#pragma unroll
            for (int k = 0; k < kStepKeys / 32; ++k)
                tmem_ld32_issue(t_sb + static_cast<uint32_t>(k * 32), reinterpret_cast<uint32_t(&)[32]>(su[k * 32]));
            tmem_ld_wait();
#pragma unroll
            for (int k = 0; k < kStepKeys / 32; ++k) tmem_ld32_arrived(reinterpret_cast<uint32_t(&)[32]>(su[k * 32]));
            float s[kStepKeys];
#pragma unroll
            for (int x = 0; x < kStepKeys; ++x) s[x] = __uint_as_float(su[x]);

            // hide keys after the causal limit (page padding is hidden in S already)
            if (j >= n_csteps) {
                const int kbase = (j - n_csteps) * kStepKeys;
                const int vis = c - kbase + 1;                      // visible keys of this row
                const int vis_lo = c_lo - kbase + 1;                // <= vis of every row of the tile
                if (vis_lo < kStepKeys) {
#pragma unroll
                    for (int x = 0; x < kStepKeys; ++x)
                        if (x >= vis) s[x] = kNegInf;
                }
            }

            // row maximum: four independent chains
            float mx4[kStepPages];
#pragma unroll
            for (int k = 0; k < kStepPages; ++k) {
                float a = fmax3(s[k * 16], s[k * 16 + 1], s[k * 16 + 2]);
#pragma unroll
                for (int x = 3; x < 15; x += 2) a = fmax3(a, s[k * 16 + x], s[k * 16 + x + 1]);
                mx4[k] = fmaxf(a, s[k * 16 + 15]);
            }
            const float m_cand = fmaxf(fmax3(mx4[0], mx4[1], mx4[2]), mx4[3]) * scale;

            // The reference moves only when the row maximum has grown by more than the threshold (probabilities
            // stay below 2^threshold meanwhile); then the sums and the accumulator O_i are rescaled.  S_i of this
            // step may have been made before P_i V of the previous one, so that one is waited for first: seldom.
            const bool need = m_cand > m + kRescaleThreshold;       // also true when m == -inf < m_cand
            if (__any_sync(kFull, need)) {
                const float m_new = fmaxf(m, m_cand);
                const float alpha = (m_new == kNegInf) ? 1.f : ex2(m - m_new);
                l *= alpha;
                acc *= alpha;
                m = m_new;
                if (jj > 0) {
                    ok = mbar_wait(bar_pv_done(i), static_cast<uint32_t>((jj - 1) & 1), abort_flag, p.status);
                    if (!ok) break;
                    tc_fence_after();
#pragma unroll 1
                    for (int k = 0; k < D / 32; ++k) {
                        uint32_t o[32];
                        tmem_ld32_wait(t_o + static_cast<uint32_t>(k * 32), o);
#pragma unroll
                        for (int x = 0; x < 32; ++x) o[x] = __float_as_uint(__uint_as_float(o[x]) * alpha);
                        tmem_st32(t_o + static_cast<uint32_t>(k * 32), o);
                    }
                }
            }
            const float m_use = (m == kNegInf) ? 0.f : m;

            // p = exp2(s * scale - m) in fp32; bf16 pairs (even key in the low half) into P_i, 32 keys per store, handed
            // to the issuer once a step.  The page sums (of the fp32 values) are taken along the way: their adds
            // fill issue slots that the exponentials leave free.
            await_turn(jj);
            const uint64_t sc2 = pack2(scale, scale), nm2 = pack2(-m_use, -m_use);
            uint64_t ps2[kStepPages];
#pragma unroll
            for (int ch = 0; ch < kStepKeys / 32; ++ch) {
                uint32_t pk[16];
#pragma unroll
                for (int x = 0; x < 16; ++x) {
                    const int e = ch * 2 + (x >> 3);
                    float a0, a1;
                    unpack2(fma2(pack2(s[ch * 32 + 2 * x], s[ch * 32 + 2 * x + 1]), sc2, nm2), a0, a1);
                    a0 = ex2(a0);
                    a1 = ex2(a1);
                    const uint64_t p2 = pack2(a0, a1);
                    pk[x] = pack_bf16(a0, a1);
                    ps2[e] = (x & 7) ? add2(ps2[e], p2) : p2;
                }
                tmem_st16(t_sb + static_cast<uint32_t>(ch * 16), pk);
            }
            pass_turn(jj);
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_p_full(i, jj & 1));

            // under the MMAs: row sum, slots
            float ps[kStepPages];
#pragma unroll
            for (int e = 0; e < kStepPages; ++e) {
                float lo, hi;
                unpack2(ps2[e], lo, hi);
                ps[e] = lo + hi;
            }
            const float tot = (ps[0] + ps[1]) + (ps[2] + ps[3]);
            l += tot;
            if (chg_mask == 0u) {
                acc += tot;
            } else {
#pragma unroll
                for (int e = 0; e < kStepPages; ++e) {
                    const bool ends = (chg_mask >> e) & 1u;
                    park(ends, lg2(acc) + m_use);
                    acc = (ends ? 0.f : acc) + ps[e];
                }
            }
        }

        for (; jj < n_mine; ++jj) { await_turn(jj); pass_turn(jj); }      // error path only: the other tile's warp may be waiting

        // ---- per-row results ----
        const float m_use = (m == kNegInf) ? 0.f : m;
        const float lse = (l > 0.f) ? m_use + lg2(l) : kNegInf;
        // (row, head) index of row rr of this warp, or -1 beyond the episode's queries
        auto row_index = [&](int rr) -> int {
            const int r2 = q4 * 32 + rr;
            const int t2 = tile_t0 + (r2 >> lr);
            if (t2 >= ep.n_q) return -1;
            const int g2 = ep.q_off + t2;
            return (split_mode ? it.split * p.n_q_total + g2 : g2) * p.Hq + it.kvh * rep + (r2 & (rep - 1));
        };
        // The warp's 32 rows x 128 bytes leave through the (idle) shared memory of the Q tile: row-per-thread
        // stores would touch 32 different rows per instruction.  Each thread stages its own 128 bytes, 16-byte
        // chunks swizzled by row, and the warp writes four whole row pieces per instruction.
        int ridx8[8];
#pragma unroll
        for (int itr = 0; itr < 8; ++itr) ridx8[itr] = row_index(itr * 4 + (lane >> 3));
        uint8_t *stg = smem + i * C::kTileBytes + q4 * 4096;
        auto flush_piece = [&](const uint32_t (&w)[32], uint8_t *gbase, long long row_pitch, int piece) {
#pragma unroll
            for (int cch = 0; cch < 8; ++cch)
                *reinterpret_cast<uint4 *>(stg + lane * 128 + ((cch ^ (lane & 7)) << 4)) =
                    make_uint4(w[4 * cch], w[4 * cch + 1], w[4 * cch + 2], w[4 * cch + 3]);
            __syncwarp();
#pragma unroll
            for (int itr = 0; itr < 8; ++itr) {
                const int rr = itr * 4 + (lane >> 3), cch = lane & 7;
                const uint4 v = *reinterpret_cast<const uint4 *>(stg + rr * 128 + ((cch ^ (rr & 7)) << 4));
                if (ridx8[itr] >= 0)
                    *reinterpret_cast<uint4 *>(gbase + ridx8[itr] * row_pitch + piece * 128 + cch * 16) = v;
            }
            __syncwarp();
        };
        // Masses out of shared memory: shares of the row's total, ref / extra being the log-sum-exp of the whole row and, in a
        // pair, the other split's part of the slot in which the splits meet.  (Log-sums parked in the mass buffer are left to
        // mass_finish_kernel: it reads and writes them at memory speed, while here every 32 slots of a warp cost a memory round trip with
        // the tensor pipe idle: 245 of 2300 us of a scoring pass over 1000 groups.)
        const int my_ridx = row_index(lane);
        const long long rh = my_ridx;
        float *const slot_out = my_ridx >= 0 && slot_rows ? slot_rows + rh * p.mass_stride : nullptr;
        auto finish_masses = [&](float ref, float extra, int first, int last) {
            if (my_ridx < 0) return;
            float *slots = p.mass + static_cast<long long>(my_ridx) * p.mass_stride;
#pragma unroll 4
            for (int sl = first; sl <= last; ++sl) {
                if (sl == skip_slot) continue;
                float w = (ref != kNegInf) ? ex2(park_row[sl * 128] - ref) : 0.f;
                if (sl == shared_slot && ref != kNegInf) w += ex2(extra - ref);
                slots[sl] = w;
            }
        };
        // slots this walker walked (all of them where nothing is split)
        int first_slot = 0, last_slot = G;
        if (p.n_splits > 1 || two_halves) {
            first_slot = G + 1;
            last_slot = -1;
            if (n_mine > 0) {
                const int je = j0 + n_mine;
                first_slot = (j0 < n_csteps) ? (__ldg(p.stream_meta + ep.stream_off + j0 * kStepPages) >> 8) : G;
                last_slot = (je > n_csteps) ? G : (__ldg(p.stream_meta + ep.stream_off + je * kStepPages - 1) >> 8);
            }
        }
        // The merged row: what a walker or a CTA of a pair makes of its own (m_use, l) and the other's (x, y of pe)
        float row_lse = lse, other_bnd = kNegInf, w_own = 0.f, w_other = 0.f;
        auto merge_rows = [&](const float4 &pe) {
            const bool va = l > 0.f, vb = pe.y > 0.f;
            const float M = fmaxf(va ? m_use : kNegInf, vb ? pe.x : kNegInf);
            const float fa = va ? ex2(m_use - M) : 0.f;
            const float fb = vb ? ex2(pe.x - M) : 0.f;
            const float L = (va ? l * fa : 0.f) + (vb ? pe.y * fb : 0.f);
            row_lse = (L > 0.f) ? M + lg2(L) : kNegInf;
            other_bnd = pe.z;
            w_own = (L > 0.f) ? fa / L : 0.f;
            w_other = (L > 0.f) ? fb / L : 0.f;
        };
        // log-sum of the slot in which two meet, from the open sum of the first and what the second sent
        auto shared_log = [&]() {
            const float own = lg2(acc) + m_use, mx = fmaxf(own, other_bnd);
            return (mx != kNegInf) ? mx + lg2(ex2(own - mx) + ex2(other_bnd - mx)) : kNegInf;
        };

        if (two_halves) {
            // ---- the walkers tell each other (reference, sum, part of the slot in which they meet) of every row; each goes on with its
            // own slots and half of the channels, whose accumulators both lie in the TMEM lanes it reads ----
            if (ok) park(true, lg2(acc) + m_use);
            float4 *rows = reinterpret_cast<float4 *>(smem + C::kXpeerOff);
            rows[i * 128 + r] = make_float4(m_use, ok ? l : 0.f, bnd, 0.f);
            asm volatile("bar.sync 9, 256;" ::: "memory");           // reached whatever happened (the waits are bounded)
            merge_rows(rows[(i ^ 1) * 128 + r]);
            if (split_mode) {
                if (i == 0 && my_ridx >= 0) p.part_lse[rh] = row_lse;
                if (slot_out) {
                    if (park_smem) {                                 // slots that this split did not walk contribute nothing
                        for (int sl = i == 0 ? 0 : first_slot; sl <= (i == 0 ? last_slot : G); ++sl)
                            if (sl != skip_slot)
                                slot_out[sl] = (sl < first_slot || sl > last_slot) ? kNegInf : sl == shared_slot ? shared_log() : park_row[sl * 128];
                    } else if (i == 0 && shared_slot >= 0) {
                        slot_out[shared_slot] = shared_log();
                    }
                }
            } else if (p.mass) {
                if (park_smem) {
                    finish_masses(row_lse, other_bnd, first_slot, last_slot);
                } else if (my_ridx >= 0 && i == 0) {
                    p.lse_out[rh] = row_lse;
                    if (shared_slot >= 0) slot_out[shared_slot] = shared_log();
                }
            }
            for (int t = 0; t < 2 && ok; ++t) ok = mbar_wait(bar_o_done(t), 0, abort_flag, p.status);
            if (ok) {
                tc_fence_after();
                const float w0 = i == 0 ? w_own : w_other, w1 = i == 0 ? w_other : w_own;
                const uint32_t t_o0 = tmem_base + lane_sel + 256u, t_o1 = t_o0 + 128u;
                // 32 channels of the merged row
                auto merged = [&](int col, float (&x)[32]) {
                    uint32_t a[32], b[32];
                    tmem_ld32_issue(t_o0 + static_cast<uint32_t>(col), a);
                    tmem_ld32_issue(t_o1 + static_cast<uint32_t>(col), b);
                    tmem_ld_wait();
                    tmem_ld32_arrived(a);
                    tmem_ld32_arrived(b);
#pragma unroll
                    for (int y = 0; y < 32; ++y) x[y] = fmaf(__uint_as_float(a[y]), w0, __uint_as_float(b[y]) * w1);
                };
                if (split_mode) {
#pragma unroll 1
                    for (int pc = i; pc < D / 32; pc += 2) {         // 32 fp32 channels = 128 bytes per row and piece
                        float x[32];
                        uint32_t w[32];
                        merged(pc * 32, x);
#pragma unroll
                        for (int y = 0; y < 32; ++y) w[y] = __float_as_uint(x[y]);
                        flush_piece(w, reinterpret_cast<uint8_t *>(p.part_o), D * 4, pc);
                    }
                } else {
#pragma unroll 1
                    for (int pc = i; pc < D / 64; pc += 2) {         // 64 bf16 channels = 128 bytes per row and piece
                        float x[32];
                        uint32_t w[32];
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            merged(pc * 64 + k * 32, x);
#pragma unroll
                            for (int y = 0; y < 16; ++y) w[k * 16 + y] = pack_bf16(x[2 * y], x[2 * y + 1]);
                        }
                        flush_piece(w, static_cast<uint8_t *>(p.out), D * 2, pc);
                    }
                }
            }
        }
        bool exported = false;
        if (ok && !two_halves) {
            park(n_mine > 0, lg2(acc) + m_use);
            if (!pair && !split_mode) {
                // ---- the whole key stream was this CTA's: output and masses ----
                if (p.mass) {
                    if (park_smem) finish_masses(lse, kNegInf, 0, G);
                    else if (my_ridx >= 0) p.lse_out[rh] = lse;
                }
                if (n_steps > 0) {
                    const float inv = (l > 0.f) ? 1.f / l : 0.f;
                    ok = mbar_wait(bar_o_done(i), 0, abort_flag, p.status);
                    if (ok) {
                        tc_fence_after();
#pragma unroll 1
                        for (int pc = 0; pc < D / 64; ++pc) {        // 64 bf16 channels = 128 bytes per row and piece
                            uint32_t o[32], w[32];
#pragma unroll
                            for (int k = 0; k < 2; ++k) {
                                tmem_ld32_wait(t_o + static_cast<uint32_t>(pc * 64 + k * 32), o);
#pragma unroll
                                for (int x = 0; x < 16; ++x)
                                    w[k * 16 + x] = pack_bf16(__uint_as_float(o[2 * x]) * inv, __uint_as_float(o[2 * x + 1]) * inv);
                            }
                            flush_piece(w, static_cast<uint8_t *>(p.out), D * 2, pc);
                        }
                    }
                }
            } else if (split_mode) {
                // ---- partial results for the merge kernel: O / l in fp32, the row's log-sum-exp, raw slot log-sums ----
                if (my_ridx >= 0) p.part_lse[rh] = lse;
                if (slot_out) {
                    if (park_smem)                                   // slots that this split did not walk contribute nothing
                        for (int sl = 0; sl <= G; ++sl)
                            slot_out[sl] = (sl < first_slot || sl > last_slot) ? kNegInf : park_row[sl * 128];
                }
                if (n_steps > 0) {
                    const float inv = (l > 0.f) ? 1.f / l : 0.f;
                    ok = mbar_wait(bar_o_done(i), 0, abort_flag, p.status);
                    if (ok) {
                        tc_fence_after();
#pragma unroll 1
                        for (int pc = 0; pc < D / 32; ++pc) {        // 32 fp32 channels = 128 bytes per row and piece
                            uint32_t o[32];
                            tmem_ld32_wait(t_o + static_cast<uint32_t>(pc * 32), o);
#pragma unroll
                            for (int x = 0; x < 32; ++x) o[x] = __float_as_uint(__uint_as_float(o[x]) * inv);
                            flush_piece(o, reinterpret_cast<uint8_t *>(p.part_o), D * 4, pc);
                        }
                    }
                }
            } else {
              if constexpr (D == 128 && !kHalves) {
                // ---- pair merge: the two CTAs of the cluster hold the two halves of the key stream ----
                const uint32_t peer = cluster_rank() ^ 1u;
                // they tell each other (reference, sum, shared-slot part) of every row
                {
                    const uint32_t mine = sbase + static_cast<uint32_t>(C::kXpeerOff + (i * 128 + r) * 16);
                    peer_push4(peer_addr(mine, peer), m_use, l, bnd, 0.f, peer_addr(bar_peer_ml, peer));
                }
                constexpr uint32_t kRingOff = C::kRingOff;
                constexpr uint32_t kExportStageOff = 65536;         // upper half of the ring (4 stages x 32 KB)
                const uint32_t warp_off = kRingOff + static_cast<uint32_t>(q4 * 16384);
                if (i != it.split && n_steps > 0) {
                    // This CTA finishes Q tile `it.split`; the accumulator of the other tile goes to the peer, which
                    // finishes that one.  It goes as it is (relative to this CTA's own reference; the peer learns the
                    // weight from the row sums above), so that nothing but the last MMA stands before it: staged
                    // row-per-thread in the upper half of this CTA's ring (idle once both tiles' MMAs are done; 16 KB
                    // per warp, 16-byte chunks swizzled by row), then one bulk copy per warp into the lower half of
                    // the peer's ring, counted in bytes on the peer's barrier.
                    ok = mbar_wait(bar_o_done(i), 0, abort_flag, p.status);
                    if (ok && n_qt == 2) ok = mbar_wait(bar_o_done(i ^ 1), 0, abort_flag, p.status);
                    if (ok) {
                        tc_fence_after();
                        uint8_t *stage = smem + warp_off + kExportStageOff + lane * 512;
#pragma unroll 1
                        for (int k = 0; k < 4; ++k) {
                            uint32_t o[32];
                            tmem_ld32_wait(t_o + static_cast<uint32_t>(k * 32), o);
#pragma unroll
                            for (int cch = 0; cch < 8; ++cch)
                                *reinterpret_cast<uint4 *>(stage + (((k * 8 + cch) ^ (lane & 7)) << 4)) =
                                    make_uint4(o[4 * cch], o[4 * cch + 1], o[4 * cch + 2], o[4 * cch + 3]);
                        }
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                        ok = mbar_wait<true>(bar_peer_free, 0, abort_flag, p.status);
                        if (ok && lane == 0)
                            peer_bulk_copy(peer_addr(sbase + warp_off, peer), sbase + warp_off + kExportStageOff, 16384,
                                           peer_addr(bar_peer_o, peer));
                        exported = ok;
                    }
                }
                if (ok) ok = mbar_wait<true>(bar_peer_ml, 0, abort_flag, p.status);
                if (ok) merge_rows(*reinterpret_cast<const float4 *>(smem + C::kXpeerOff + (i * 128 + r) * 16));
                // each CTA writes the slots it walked against the merged log-sum-exp; the slot both walked is
                // written by split 0, which adds the part split 1 sent.  (Before the output: the peer's accumulator is
                // still on its way.)
                if (ok && p.mass) {
                    if (park_smem) {
                        finish_masses(row_lse, other_bnd, first_slot, last_slot);
                    } else if (my_ridx >= 0 && it.split == 0) {
                        p.lse_out[rh] = row_lse;
                        if (shared_slot >= 0) slot_out[shared_slot] = shared_log();      // the slot parked last: its own part is still in acc
                    }
                }
                if (ok && i == it.split && n_steps > 0) {
                    // this CTA finishes the tile: its own accumulator and what the peer sent, each with its weight;
                    // thread (warp, lane) reads what thread (warp, lane) of the peer wrote
                    ok = mbar_wait(bar_o_done(i), 0, abort_flag, p.status);
                    if (ok) {
                        tc_fence_after();
                        ok = mbar_wait<true>(bar_peer_o, 0, abort_flag, p.status);
                        // the peer may retire once its staging area has been read out: tell it
                        if (ok && q4 == 0 && lane == 0) peer_arrive_relaxed(peer_addr(bar_peer_ack, peer));
                    }
                    if (ok) {
                        const uint8_t *theirs = smem + warp_off + lane * 512;
#pragma unroll 1
                        for (int pc = 0; pc < 2; ++pc) {
                            uint32_t o[32], w[32];
#pragma unroll
                            for (int k = 0; k < 2; ++k) {
                                tmem_ld32_wait(t_o + static_cast<uint32_t>(pc * 64 + k * 32), o);
#pragma unroll
                                for (int cch = 0; cch < 8; ++cch) {
                                    const float4 a = *reinterpret_cast<const float4 *>(
                                        theirs + ((((pc * 2 + k) * 8 + cch) ^ (lane & 7)) << 4));
                                    auto mix = [&](uint32_t own, float th) { return fmaf(__uint_as_float(own), w_own, th * w_other); };
                                    w[k * 16 + 2 * cch] = pack_bf16(mix(o[4 * cch], a.x), mix(o[4 * cch + 1], a.y));
                                    w[k * 16 + 2 * cch + 1] = pack_bf16(mix(o[4 * cch + 2], a.z), mix(o[4 * cch + 3], a.w));
                                }
                            }
                            flush_piece(w, static_cast<uint8_t *>(p.out), D * 2, pc);
                        }
                    }
                }
                // what this CTA staged for its peer must have been fetched before the CTA may retire
                if (exported) ok = mbar_wait<true>(bar_peer_ack, 0, abort_flag, p.status);
              }
            }
        }
      }
    }

    // ---- teardown ----
    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
    }
}

}  // namespace

int attention_park_slots() { return kParkSlots; }

template <int D>
static cudaError_t prepare()
{
    cudaError_t e = cudaFuncSetAttribute(attn_kernel<D, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<D>::kSmemBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(attn_kernel<D, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<D>::kSmemBytes);
    return e;
}

cudaError_t prepare_attention(int head_dim)
{
    return head_dim == 128 ? prepare<128>() : head_dim == 64 ? prepare<64>() : cudaErrorInvalidValue;
}

bool attention_pairs_supported()
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = Cfg<128>::kSmemBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, attn_kernel<128, false>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n > 0;
}

cudaError_t launch_attention(const AttnParams &p, int head_dim, int n_items, cudaStream_t st)
{
    if (n_items <= 0) return cudaSuccess;
    if (p.pair_merge && (head_dim != 128 || p.n_splits != 2 || p.halves || (n_items & 1))) return cudaErrorInvalidValue;
    if (head_dim != 128 && head_dim != 64) return cudaErrorInvalidValue;
    const auto kernel = head_dim == 128 ? (p.halves ? attn_kernel<128, true> : attn_kernel<128, false>)
                                        : (p.halves ? attn_kernel<64, true> : attn_kernel<64, false>);
    const int smem = head_dim == 128 ? Cfg<128>::kSmemBytes : Cfg<64>::kSmemBytes;
    const cudaError_t e = launch_pdl(kernel, dim3(n_items), dim3(kThreads), smem, st, p, p.pair_merge ? 2u : 1u);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace enl
