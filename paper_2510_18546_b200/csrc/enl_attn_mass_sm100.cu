// Group masses without outputs (the scoring pass), sm_100a (tcgen05 + TMEM + TMA).
//
// Sec. 3.3 consumes only the attention between new tokens and groups: of softmax(Q K^T / sqrt(D)) the sums per slot, no V, no
// output.  Half the tensor work of enl_attn_sm100.cu and none of what P V brings with it (P, its way to the MMA issuer, the
// accumulator and its rescaling) is left, so the split of the work is another one:
//   - S of both Q tiles is double-buffered in TMEM (4 x 128 columns): the next Q K^T runs under a tile's softmax;
//   - page padding is hidden by an MMA of one K step that S starts from (see enl_attn_sm100.cu; added in the softmax warps, the
//     same took 130 of 3080 cycles per tile);
//   - two threads per query row take 64 keys each, sixteen softmax warps in all, and share nothing: with no accumulator there is no need
//     for a common reference.  A thread takes its exponentials against the reference of the tiles before and finds the tile's
//     maximum beside them; any reference is exact as long as nothing overflows, so only scores more than 64 (log2) above it
//     make the warp start the tile over;
//   - the page sums go to a slot warp per Q tile (four rows per lane) that adds them to the open slot and parks the log2-sum
//     of a slot that ends in the mass buffer.  The stream is in slot order, so a row has one open slot;
//   - key ranges may be split over CTAs: a slot that two splits share is written by the earlier one, the later one's part and
//     every split's log2-sum-exp go to mass_finish_kernel, which turns log-sums into masses.
// Bound by the exponentials and the issue slots around them, not by the tensor pipe.  Measured against the general kernel
// that skipped its output: 512 rows x 32 heads over 200 groups (16 000 keys) 375 -> 122 us a layer, mass_finish_kernel included
// (this kernel alone 117 in a serialised capture), of which the two-way split of the keys is half; per key tile and pair of Q tiles
// 4400 -> 2940 cycles.
#include <cuda_bf16.h>

#include "attn_ops.cuh"
#include "enl_internal.h"
#include "tmem_ops.cuh"

namespace enl {
namespace {

constexpr int kSoftmaxWarps = 16;             // two warpgroups per Q tile: keys 0..63 and 64..127 of every key tile
constexpr int kProducerWarp = 16;
constexpr int kMmaWarp      = 17;
constexpr int kSlotWarp     = 18;             // + Q tile
constexpr int kThreads      = 20 * 32;        // 96 registers a thread, for all roles: the slot warps use them, too (with 64 they took 1.2 of a softmax warp's time)
constexpr uint32_t kTmemCols = 512;
constexpr float kRescaleThreshold = 8.0f;     // log2 units: a reference that lags the maximum by more moves before the next tile
constexpr float kJumpThreshold = 64.0f;       // log2 units: scores further above the reference make the tile start over
constexpr int kHalfKeys  = kTileKeys / 2;
constexpr int kHalfPages = kPagesPerTile / 2;

template <int D>
struct Cfg {
    static constexpr int kHalves    = D / 64;             // 64-channel (128-byte) column blocks
    static constexpr int kHalfBytes = 128 * 128;          // 128 rows x 128 B
    static constexpr int kTileBytes = kHalves * kHalfBytes;
    static constexpr int kGroupBytes = kHalves * 1024;     // K: eight rows, one 8 x 128-byte block per 64 channels
    static constexpr int kStages    = 4;
    static constexpr int kBarOff    = (kQTiles + kStages) * kTileBytes;
    // operands of the MMA that hides page padding, 16 bytes per row: 1 for 8 queries, 0 or -inf for every key of a stage
    static constexpr int kOnesOff   = kBarOff + 256;
    static constexpr int kHideOff   = kBarOff + 512;
    static constexpr int kHideBytes = kTileKeys * 16;
    // what the softmax threads leave for the slot warps: [buffer][tile][half][128] page sums x 4, and their references
    static constexpr int kSumOff    = kHideOff + kStages * kHideBytes;
    static constexpr int kSumBytes  = kQTiles * 2 * 128 * 16;
    static constexpr int kRefOff    = kSumOff + 2 * kSumBytes;
    static constexpr int kLseOff    = kRefOff + 2 * kSumBytes / 4;     // [tile][128] log2-sum-exps of the second half
    static constexpr int kSmemBytes = kLseOff + kQTiles * 128 * 4 + 1024;   // + alignment slack
    static_assert(kSmemBytes <= 232448 && kSumOff % 16 == 0, "shared memory");
};

template <int D>
__global__ void __launch_bounds__(kThreads, 1) mass_kernel(const __grid_constant__ MassParams p)
{
    using C = Cfg<D>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t sbase = (raw + 1023u) & ~1023u;               // 1024-B aligned (swizzle atoms)
    uint8_t *smem = smem_raw + (sbase - raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    auto q_addr     = [&](int i) { return sbase + static_cast<uint32_t>(i * C::kTileBytes); };
    auto stage_addr = [&](int s) { return sbase + static_cast<uint32_t>((kQTiles + s) * C::kTileBytes); };
    const uint32_t bar0 = sbase + C::kBarOff;
    const uint32_t bar_q_full = bar0;
    auto bar_k_full  = [&](int s) { return bar0 + 8u * (1 + s); };
    auto bar_k_empty = [&](int s) { return bar0 + 8u * (1 + C::kStages + s); };
    constexpr int kBar1 = 1 + 2 * C::kStages;
    auto bar_s_full  = [&](int i, int b) { return bar0 + 8u * (kBar1 + 2 * i + b); };
    auto bar_s_free  = [&](int i, int b) { return bar0 + 8u * (kBar1 + 4 + 2 * i + b); };       // S buffer read out
    auto bar_sums    = [&](int i, int b) { return bar0 + 8u * (kBar1 + 8 + 2 * i + b); };       // page sums of a tile are there
    auto bar_taken   = [&](int i, int b) { return bar0 + 8u * (kBar1 + 12 + 2 * i + b); };      // ... have been taken
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + C::kBarOff + 8 * (kBar1 + 16));
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    // ---- set-up ----
    if (threadIdx.x == 0) {
        *abort_flag = 0;
        mbar_init(bar_q_full, 1);
        for (int s = 0; s < C::kStages; ++s) { mbar_init(bar_k_full(s), 1); mbar_init(bar_k_empty(s), 1); }
        for (int i = 0; i < kQTiles; ++i)
            for (int b = 0; b < 2; ++b) {
                mbar_init(bar_s_full(i, b), 1);
                mbar_init(bar_s_free(i, b), kSoftmaxWarps / kQTiles);    // one arrival per softmax warp of the tile
                mbar_init(bar_sums(i, b), kSoftmaxWarps / kQTiles);
                mbar_init(bar_taken(i, b), 1);
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
    // The plan or the pool has been written since the last attention launch: nothing of them may be read before the
    // kernel before has ended, and the next launch may start only then (it relies on both).
    if (p.wait_first) pdl_wait();

    const Item it = p.items[blockIdx.x];
    const EpInfo ep = p.eps[it.ep];
    const int rep = p.rep;
    const int tile_tokens = kTileRows / rep;
    const int t_hi = min(it.t0 + kQTiles * tile_tokens, ep.n_q);        // exclusive
    const int n_qt = (t_hi - it.t0 > tile_tokens) ? 2 : 1;
    const int total_tiles = ep.n_ctiles + (ep.n_new - ep.n_q + t_hi - 1) / kTileKeys + 1;    // up to the last new key any row sees
    const int j_beg = static_cast<int>(static_cast<long long>(total_tiles) * it.split / p.n_splits);
    const int j_end = static_cast<int>(static_cast<long long>(total_tiles) * (it.split + 1) / p.n_splits);
    const int n_tiles = j_end - j_beg;                                   // at least one (host guarantees)
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    pdl_trigger();
    pdl_wait();                                  // the caller's tensors and the mass buffer come next
    bool ok = true;

    if (warp >= kSoftmaxWarps) {
      if (warp == kProducerWarp) {
        // ================= TMA producer =================
        if (lane == 0) {
            mbar_expect_tx(bar_q_full, static_cast<uint32_t>(n_qt * C::kTileBytes));
            for (int i = 0; i < n_qt; ++i)
                for (int hf = 0; hf < C::kHalves; ++hf)
                    tma_load_3d(q_addr(i) + hf * C::kHalfBytes, &p.tm_q, hf * 64, it.kvh * rep,
                                ep.q_off + it.t0 + i * tile_tokens, bar_q_full);
        }
        // page words (id; slot << 8 | valid keys) of 32 pages at a time, one per lane, fetched four tiles ahead
        constexpr int kBatch = 32 / kPagesPerTile;
        auto words = [&](int t, int &id, int &meta) {
            const int e = (j_beg + t) * kPagesPerTile + lane;
            id = kZeroPage;
            meta = kPageTokens;
            if (e < ep.n_ctiles * kPagesPerTile) {
                id = __ldg(p.stream_page + ep.stream_off + e);
                meta = __ldg(p.stream_meta + ep.stream_off + e);
            }
        };
        int id_cur = 0, meta_cur = 0, id_next, meta_next;
        words(0, id_next, meta_next);
        int jj = 0;
        for (; jj < n_tiles && ok; ++jj) {
            const int j = j_beg + jj, st = jj % C::kStages;
            const bool cached = j < ep.n_ctiles;
            if (jj % kBatch == 0) {
                id_cur = id_next;
                meta_cur = meta_next;
                words(jj + kBatch, id_next, meta_next);
            }
            const int at = jj % kBatch * kPagesPerTile + lane % kPagesPerTile;
            const int group = (__shfl_sync(kFull, id_cur, at) * p.Hkv + it.kvh) * kPageGroups<D>, valid = __shfl_sync(kFull, meta_cur, at) & 0xff;
            if (jj >= C::kStages) {
                ok = mbar_wait(bar_k_empty(st), static_cast<uint32_t>((jj / C::kStages - 1) & 1), abort_flag, p.status);
                if (!ok) break;
            }
            if (cached) {                                            // what hides the padding of these keys
                uint4 *hide = reinterpret_cast<uint4 *>(smem + C::kHideOff + st * C::kHideBytes);
#pragma unroll
                for (int x = 0; x < kTileKeys / 32; ++x) {
                    const int n = __shfl_sync(kFull, valid, 2 * x + (lane >> 4));
                    hide[x * 32 + lane] = make_uint4((lane & 15) < n ? 0u : 0xff80u, 0u, 0u, 0u);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
            }
            if (lane == 0) mbar_expect_tx(bar_k_full(st), static_cast<uint32_t>(C::kTileBytes));
            __syncwarp();
            if (cached) {
                if (lane < kPagesPerTile)
                    tma_load_4d(stage_addr(st) + static_cast<uint32_t>(lane * 2 * C::kGroupBytes), &p.tm_kpool, 0, 0, 0, group, bar_k_full(st));
            } else if (lane < kTileKeys / kBoxRows<D>) {
                tma_load_4d(stage_addr(st) + static_cast<uint32_t>(lane * (kBoxRows<D> * D * 2)), &p.tm_knew, 0,
                            ep.new_off + (j - ep.n_ctiles) * kTileKeys + lane * kBoxRows<D>, 0, it.kvh, bar_k_full(st));
            }
        }
        // error path only: let the copies already in flight land before the CTA retires
        for (int f = max(0, jj - C::kStages); f < jj && !ok; ++f) {
            const unsigned long long t0 = global_ns();
            while (!mbar_try_wait(bar_k_full(f % C::kStages), static_cast<uint32_t>((f / C::kStages) & 1)) &&
                   global_ns() - t0 < 2000000ull) { }
        }
      } else if (warp == kMmaWarp) {
        // ================= MMA issuer =================
        constexpr uint32_t idesc_qk = make_idesc(kTileKeys, false);
        constexpr uint32_t kTileUnits = C::kTileBytes >> 4;
        const uint64_t dq0 = smem_desc(q_addr(0), 16), dk0 = smem_desc(stage_addr(0), 16, C::kGroupBytes);
        const uint32_t dq_lo = static_cast<uint32_t>(dq0), dq_hi = static_cast<uint32_t>(dq0 >> 32);
        const uint32_t dk_lo = static_cast<uint32_t>(dk0), dk_hi = static_cast<uint32_t>(dk0 >> 32);
        const uint64_t d_ones = smem_desc_plain(sbase + C::kOnesOff, 0u), d_hide = smem_desc_plain(sbase + C::kHideOff, 128u);
        ok = mbar_wait(bar_q_full, 0, abort_flag, p.status);
        for (int jj = 0; jj < n_tiles && ok; ++jj) {
            const int st = jj % C::kStages, buf = jj & 1;
            ok = mbar_wait(bar_k_full(st), static_cast<uint32_t>((jj / C::kStages) & 1), abort_flag, p.status);
            for (int i = 0; i < n_qt && ok; ++i) {
                if (jj >= 2) ok = mbar_wait(bar_s_free(i, buf), static_cast<uint32_t>((jj / 2 - 1) & 1), abort_flag, p.status);
                if (!ok) break;
                tc_fence_after();
                const bool hide = j_beg + jj < ep.n_ctiles;
                if (hide)
                    mma_ss2(tmem_base + static_cast<uint32_t>((2 * buf + i) * 128), static_cast<uint32_t>(d_ones),
                            static_cast<uint32_t>(d_ones >> 32), static_cast<uint32_t>(d_hide) + static_cast<uint32_t>(st) * (C::kHideBytes >> 4),
                            static_cast<uint32_t>(d_hide >> 32), idesc_qk, 0u);
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk) {
                    const uint32_t in_row = static_cast<uint32_t>((kk & 3) * 2);                       // 32 bytes per 16 channels
                    mma_ss2(tmem_base + static_cast<uint32_t>((2 * buf + i) * 128),
                            dq_lo + static_cast<uint32_t>(i) * kTileUnits + static_cast<uint32_t>((kk >> 2) * (C::kHalfBytes >> 4)) + in_row, dq_hi,
                            dk_lo + static_cast<uint32_t>(st) * kTileUnits + static_cast<uint32_t>((kk >> 2) * (1024 >> 4)) + in_row, dk_hi,
                            idesc_qk, kk > 0 || hide ? 1u : 0u);
                }
                tc_commit(bar_s_full(i, buf));
            }
            if (ok) tc_commit(bar_k_empty(st));
        }
        // nothing may still be under way when the CTA gives up its barriers: the last commit
        if (ok) ok = mbar_wait(bar_k_empty((n_tiles - 1) % C::kStages), static_cast<uint32_t>(((n_tiles - 1) / C::kStages) & 1),
                               abort_flag, p.status);
      } else if (warp - kSlotWarp < n_qt) {
        // ================= slot book-keeping: four rows per lane =================
        const int i = warp - kSlotWarp;
        float m_half[4][2], f_half[4][2];                              // the halves' references, what their sums are scaled by
        float acc[4], m_acc[4], bnd[4];                                // open slot's sum, its reference; log-sum of the slot shared with the split before
        int idx[4];                                                    // (row, head) index, -1 beyond the episode's queries
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            acc[q] = 0.f;
            m_acc[q] = m_half[q][0] = m_half[q][1] = kNegInf;
            f_half[q][0] = f_half[q][1] = 1.f;
            bnd[q] = kNegInf;
            const int r = q * 32 + lane, t = it.t0 + i * tile_tokens + r / rep;
            idx[q] = t < ep.n_q ? (ep.q_off + t) * p.Hq + it.kvh * rep + r % rep : -1;
        }
        const int32_t *meta = p.stream_meta + ep.stream_off;
        int slot = j_beg < ep.n_ctiles ? __ldg(meta + j_beg * kPagesPerTile) >> 8 : ep.n_slots;
        int apart = -1;                                                // the slot that the split before has begun
        if (it.split > 0) {
            const int before = j_beg > ep.n_ctiles ? ep.n_slots : __ldg(meta + j_beg * kPagesPerTile - 1) >> 8;
            if (before == slot) apart = slot;
        }
        auto park = [&]() {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float v = acc[q] > 0.f ? lg2(acc[q]) + m_acc[q] : kNegInf;
                acc[q] = 0.f;
                if (slot == apart) bnd[q] = v;
                else if (idx[q] >= 0) p.mass[static_cast<long long>(idx[q]) * p.mass_stride + slot] = v;
            }
            ++slot;
        };
        auto load_chg = [&](int j) -> uint32_t {
            return j < ep.n_ctiles ? __ldg(p.tile_chg + ep.stream_off / kPagesPerTile + j) : (j == ep.n_ctiles ? 1u : 0u);
        };
        uint32_t chg_next = load_chg(j_beg) & ~1u;                     // the first page opens its slot
        for (int jj = 0; jj < n_tiles; ++jj) {
            const int buf = jj & 1;
            const uint32_t chg = chg_next;
            chg_next = load_chg(j_beg + jj + 1);
            ok = mbar_wait(bar_sums(i, buf), static_cast<uint32_t>((jj >> 1) & 1), abort_flag, p.status);
            if (!ok) break;
            float ps[4][kPagesPerTile], ma[4], mb[4];
            bool moved = false;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 *sums = reinterpret_cast<const float4 *>(smem + C::kSumOff + buf * C::kSumBytes) + i * 256 + q * 32 + lane;
                const float *refs = reinterpret_cast<const float *>(smem + C::kRefOff + buf * (C::kSumBytes / 4)) + i * 256 + q * 32 + lane;
                ma[q] = refs[0];
                mb[q] = refs[128];
                const float4 a = sums[0], b = sums[128];
                moved = moved || ma[q] != m_half[q][0] || mb[q] != m_half[q][1];
                ps[q][0] = a.x; ps[q][1] = a.y; ps[q][2] = a.z; ps[q][3] = a.w;
                ps[q][4] = b.x; ps[q][5] = b.y; ps[q][6] = b.z; ps[q][7] = b.w;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_taken(i, buf));
            // Everything is relative to the larger of the two halves' references (a half that has seen nothing yet has sums of
            // 0).  They seldom move.
            if (__any_sync(kFull, moved)) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float m = fmaxf(ma[q], mb[q]);
                    m_half[q][0] = ma[q];
                    m_half[q][1] = mb[q];
                    f_half[q][0] = (ma[q] == m) ? 1.f : ex2(ma[q] - m);
                    f_half[q][1] = (mb[q] == m) ? 1.f : ex2(mb[q] - m);
                    if (m != m_acc[q]) acc[q] = acc[q] > 0.f ? acc[q] * ex2(m_acc[q] - m) : 0.f;
                    m_acc[q] = m;
                }
            }
#pragma unroll
            for (int e = 0; e < kPagesPerTile; ++e) {
                if ((chg >> e) & 1u) park();                           // the same in every lane
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[q] = fmaf(ps[q][e], f_half[q][e / kHalfPages], acc[q]);
            }
        }
        if (ok) {
            park();
            if (p.n_splits > 1) {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (idx[q] >= 0)
                        p.bnd_out[static_cast<long long>(it.split) * p.n_q_total * p.Hq + idx[q]] = make_float2(bnd[q], __int_as_float(apart));
            }
        }
      }
    } else {
      if ((warp >> 3) < n_qt) {
        // ================= softmax: two threads per query row, 64 keys of every tile each =================
        const int i = warp >> 3;                                   // Q tile
        const int half = (warp >> 2) & 1;                          // keys 64 * half .. of a tile
        const int q4 = warp & 3;                                   // TMEM lane quadrant
        const int r = q4 * 32 + lane;
        const int t = it.t0 + i * tile_tokens + r / rep;           // episode-relative query token
        const int c = min(ep.n_new - ep.n_q + t, ep.n_new - 1);    // last visible new key
        const uint32_t t_s0 = tmem_base + (static_cast<uint32_t>(q4 * 32) << 16) + static_cast<uint32_t>(i * 128 + half * kHalfKeys);
        const float scale = p.scale_log2;
        const uint64_t sc2 = pack2(scale, scale);
        float m = kNegInf, m_run = kNegInf;                        // reference and maximum so far (log2 units)
        float l = 0.f;                                             // sum, relative to m
        for (int jj = 0; jj < n_tiles; ++jj) {
            const int j = j_beg + jj, buf = jj & 1;
            const uint32_t t_s = t_s0 + static_cast<uint32_t>(buf * 256);
            const uint32_t par = static_cast<uint32_t>((jj >> 1) & 1);
            auto move_reference = [&](float to) {
                const float m_new = fmaxf(m, to);
                l *= (m_new == kNegInf) ? 1.f : ex2(m - m_new);
                m = m_new;
            };
            if (m_run > m + kRescaleThreshold) move_reference(m_run);
            ok = mbar_wait(bar_s_full(i, buf), par, abort_flag, p.status);
            if (!ok) break;
            tc_fence_after();

            float s[kHalfKeys];
            float m_goal;
            uint64_t ps2[kHalfPages];
            auto exps_of_tile = [&]() {
                tmem_ld32_issue(t_s, *reinterpret_cast<uint32_t(*)[32]>(&s[0]));
                tmem_ld32_issue(t_s + 32u, *reinterpret_cast<uint32_t(*)[32]>(&s[32]));
                tmem_ld_wait();
                tmem_ld32_arrived(*reinterpret_cast<uint32_t(*)[32]>(&s[0]));
                tmem_ld32_arrived(*reinterpret_cast<uint32_t(*)[32]>(&s[32]));
                // hide keys after the causal limit (page padding is hidden in S already)
                if (j >= ep.n_ctiles) {
                    const int vis = c - (j - ep.n_ctiles) * kTileKeys + 1 - half * kHalfKeys;
#pragma unroll
                    for (int x = 0; x < kHalfKeys; ++x)
                        if (x >= vis) s[x] = kNegInf;
                }
                const float m_use = (m == kNegInf) ? 0.f : m;
                const uint64_t nm2 = pack2(-m_use, -m_use);
                float mx[kHalfPages];
#pragma unroll
                for (int e = 0; e < kHalfPages; ++e) {
                    mx[e] = fmaxf(s[e * 16], s[e * 16 + 1]);
#pragma unroll
                    for (int x = 0; x < 8; ++x) {
                        const float s0 = s[e * 16 + 2 * x], s1 = s[e * 16 + 2 * x + 1];
                        if (x) mx[e] = fmax3(mx[e], s0, s1);
                        float a0, a1;
                        unpack2(fma2(pack2(s0, s1), sc2, nm2), a0, a1);
                        const uint64_t p2 = pack2(ex2(a0), ex2(a1));
                        ps2[e] = x ? add2(ps2[e], p2) : p2;
                    }
                }
                m_goal = fmaxf(fmax3(mx[0], mx[1], mx[2]), mx[3]) * scale;
            };
            exps_of_tile();
            if (__any_sync(kFull, m_goal > m + kJumpThreshold)) {  // also when m == -inf < m_goal
                if (m_goal > m + kJumpThreshold) move_reference(m_goal);
                exps_of_tile();
            }
            m_run = fmaxf(m_run, m_goal);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_s_free(i, buf));
            float ps[kHalfPages];
#pragma unroll
            for (int e = 0; e < kHalfPages; ++e) {
                float lo, hi;
                unpack2(ps2[e], lo, hi);
                ps[e] = lo + hi;
            }
            l += (ps[0] + ps[1]) + (ps[2] + ps[3]);
            if (jj >= 2) {
                ok = mbar_wait(bar_taken(i, buf), par ^ 1u, abort_flag, p.status);
                if (!ok) break;
            }
            reinterpret_cast<float4 *>(smem + C::kSumOff + buf * C::kSumBytes)[i * 256 + half * 128 + r] = make_float4(ps[0], ps[1], ps[2], ps[3]);
            reinterpret_cast<float *>(smem + C::kRefOff + buf * (C::kSumBytes / 4))[i * 256 + half * 128 + r] = m;
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_sums(i, buf));
        }

        // ---- the row's log2-sum-exp out of both halves' ----
        float *lses = reinterpret_cast<float *>(smem + C::kLseOff) + i * 128;
        const float lse = (l > 0.f) ? m + lg2(l) : kNegInf;
        if (half == 1) lses[r] = lse;
        asm volatile("bar.sync %0, 256;" ::"r"(1 + i) : "memory");
        if (ok && half == 0 && t < ep.n_q) {
            const float other = lses[r], mx = fmaxf(lse, other);
            const float both = (mx == kNegInf) ? kNegInf : mx + lg2(ex2(lse - mx) + ex2(other - mx));
            const long long rh = static_cast<long long>(ep.q_off + t) * p.Hq + it.kvh * rep + r % rep;
            p.lse_out[static_cast<long long>(it.split) * p.n_q_total * p.Hq + rh] = both;
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

cudaError_t prepare_mass(int head_dim)
{
    if (head_dim == 128) return cudaFuncSetAttribute(mass_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<128>::kSmemBytes);
    if (head_dim == 64) return cudaFuncSetAttribute(mass_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<64>::kSmemBytes);
    return cudaErrorInvalidValue;
}

cudaError_t launch_mass(const MassParams &p, int head_dim, int n_items, cudaStream_t st)
{
    if (n_items <= 0) return cudaSuccess;
    cudaError_t e;
    if (head_dim == 128) e = launch_pdl(mass_kernel<128>, dim3(n_items), dim3(kThreads), Cfg<128>::kSmemBytes, st, p);
    else if (head_dim == 64) e = launch_pdl(mass_kernel<64>, dim3(n_items), dim3(kThreads), Cfg<64>::kSmemBytes, st, p);
    else return cudaErrorInvalidValue;
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace enl
