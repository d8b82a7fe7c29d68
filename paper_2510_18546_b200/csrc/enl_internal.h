// Internal declarations shared by the host side and the kernels of the library.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace enl {

constexpr int kPageTokens = 16;     // tokens per page: one TMA box per kv head (see below)
constexpr int kTileKeys   = 128;    // keys per KV tile (8 pages)
constexpr int kPagesPerTile = kTileKeys / kPageTokens;
constexpr int kStepKeys   = 64;     // keys that attn_kernel takes at once
constexpr int kTileRows   = 128;    // query rows per Q tile = (128 / rep) tokens x rep q heads of one kv head
constexpr int kQTiles     = 2;      // Q tiles per CTA (they share every K/V tile the CTA loads)
constexpr int kZeroPage   = 0;      // page 0 is never handed out: all zeros, target of null stream entries

// One episode of an attend call.
struct EpInfo {
    int32_t stream_off;     // first KV-stream entry (multiple of kPagesPerTile)
    int32_t n_ctiles;       // cached tiles (128 keys each, last one padded with null entries)
    int32_t n_slots;        // selected groups G_b; mass slot G_b = new tokens
    int32_t q_off, n_q;     // first query row (global) and count
    int32_t new_off, n_new; // first new-token key (global) and count
    int32_t n_entries;      // stream entries without the null ones that fill the last tile
};

// One CTA of the attention launch.
struct Item {
    int32_t ep;             // episode
    int32_t kvh;            // kv head
    int32_t t0;             // first query token (episode-relative) of the CTA's Q tiles
    int32_t split;          // KV split index in [0, n_splits)
};

// How keys and values are fetched: by boxes that leave one swizzled block of 8 rows x 128 bytes per 64 channels, and then the next 8 rows.
// With R = kBoxRows, the rows of 64 channels that lie behind one another in such a box (8, at head_dim 64 all 16 of a page):
//   pool (a layer), dims {64 channels, R rows, D/64 blocks, groups of R rows}, box {64, R, D/64, 16/R}: a page of a kv head, 16 D contiguous
//     values, in one box; its last coordinate is (page * Hkv + head) * kPageGroups
//   a caller's [n][Hkv][D], dims {64 channels, n rows, D/64 blocks, Hkv heads}, box {64, R, D/64, 1}: R rows of a head
// A box costs the warp that asks for it some 50 cycles, so a box of half as much (64 channels of a page, as a two-dimensional map gives
// them) had every producer take twice as long.  (Groups of eight at head_dim 64, too, are up to 4 % slower: one token over two streams of
// 16000 keys, 8 kv heads, 19.0 against 19.7 us.)
constexpr int box_rows(int D) { return 1024 / D; }
template <int D> constexpr int kBoxRows = box_rows(D);
template <int D> constexpr int kPageGroups = kPageTokens / kBoxRows<D>;

// Kernel parameters (passed by value as a __grid_constant__).
struct AttnParams {
    CUtensorMap tm_q;       // [n_q][Hq][D]      box {64, rep, 128/rep}
    CUtensorMap tm_knew;    // [n_new][Hkv][D]: rows of a head (see above)
    CUtensorMap tm_vnew;
    CUtensorMap tm_kpool;   // one layer: a page of a head
    CUtensorMap tm_vpool;
    const Item   *items;
    const EpInfo *eps;
    const int32_t *stream_page;   // KV stream: page id of every entry
    const int32_t *stream_meta;   // KV stream: slot << 8 | valid tokens
    void   *out;            // bf16 [n_q][Hq][D]
    float  *mass;           // fp32 or null
    float  *part_o;         // split mode: [split][row][Hq][D] fp32 (normalised by the split's own sum)
    float  *part_lse;       // split mode: [split][row][Hq] log2-sum-exp of the split
    float  *part_slot;      // split mode: [split][row][Hq][mass_stride] per-slot log2-sum-exp (with part_rng only of the slots that the split has walked)
    int2   *part_rng;       // split mode, log-sums not parked in shared memory: [split][row] first and last of them (the same for all heads)
    int32_t *status;        // device word: nonzero = a bounded wait expired
    int32_t n_q_total;      // rows over the batch
    int32_t Hq, Hkv, rep;   // rep = Hq / Hkv
    int32_t mass_stride;
    int32_t n_splits;
    int32_t pair_merge;     // 1: two splits, launched as clusters of two CTAs that merge through distributed shared memory
    int32_t halves;         // 1: items are Q tiles of 128 rows, whose steps the two walkers of a CTA share (see the kernel)
    float   scale_log2;     // log2(e) / sqrt(D)
    int32_t park_smem;      // 1: the call has at most attention_park_slots() slots: the kernel turns their log-sums into masses itself;
                            // 0: log-sums go to mass, log-sum-exps to lse_out, and mass_finish_kernel does
    float  *lse_out;        // [n_q_total][Hq] log2-sum-exp of every row
    int32_t wait_first;     // 1: the plan or the pool has been written since the last attention launch: wait for the kernel before
                            // at the very start; 0: both may be read while it still runs
    int32_t first_wave;     // CTAs that start while the previous kernel of the stream may still run (the number of SMs)
};

// Masses without outputs (see enl_attn_mass_sm100.cu)
struct MassParams {
    CUtensorMap tm_q;       // [n_q][Hq][D]      box {64, rep, 128/rep}
    CUtensorMap tm_knew;    // as in AttnParams
    CUtensorMap tm_kpool;
    const Item   *items;
    const EpInfo *eps;
    const int32_t *stream_page;
    const int32_t *stream_meta;
    const uint8_t *tile_chg; // per cached tile: pages whose slot is not that of the page before (a bit each)
    float  *mass;           // log2-sums of the slots, for mass_finish_kernel
    float  *lse_out;        // [split][n_q_total][Hq] log2-sum-exp of every row
    float2 *bnd_out;        // with splits: [split][n_q_total][Hq] the split's part of the slot it shares with the split before it
                            // (log2), and that slot (or -1)
    int32_t *status;
    int32_t n_q_total;
    int32_t Hq, Hkv, rep;
    int32_t mass_stride;
    int32_t n_splits;
    int32_t wait_first;     // as in AttnParams
    float   scale_log2;
};

// Decode (one query token per episode): pages of the key stream one CTA may cover, and the most splits
// the merge kernel takes.
constexpr int kDecodeMaxPages = 256;
constexpr int kMaxSplits      = 64;

struct DecodeParams {
    CUtensorMap tm_knew;    // as in AttnParams
    CUtensorMap tm_vnew;
    CUtensorMap tm_kpool;
    CUtensorMap tm_vpool;
    EpInfo ep0;             // episode 0 (used when the call has one episode; grid = splits x kv heads x episodes)
    const EpInfo *eps;
    const int32_t *stream_page;
    const int32_t *stream_meta;
    const void *q;          // bf16 [n_q][Hq][D], one row per episode
    void   *out;            // bf16 [n_q][Hq][D]
    float  *mass;           // fp32 or null
    float  *part_o, *part_lse, *part_slot;      // as in AttnParams; part_slot is null when mass is
    int2   *part_rng;       // [split][episode][kv head]: first slot and number of slots the split's range touched
    int32_t *counters;      // [episode][kv head], zero between launches: splits that have finished
    int32_t *status;
    int32_t n_q_total;
    int32_t Hq, Hkv, rep;
    int32_t slot_stride;    // row stride of part_slot
    int32_t mass_stride;    // row stride of mass
    int32_t n_splits;
    int32_t wait_first;     // as in AttnParams
    float   scale_log2;
};

// The same for calls whose splits fit a thread-block cluster (see enl_decode_cluster_sm100.cu): no partial results in memory.
struct ClusterDecodeParams {
    CUtensorMap tm_knew;    // as in AttnParams
    CUtensorMap tm_vnew;
    CUtensorMap tm_kpool;
    CUtensorMap tm_vpool;
    EpInfo ep0;             // episode 0 (used when the call has one episode; grid = cluster x kv heads x episodes)
    const EpInfo *eps;
    const int32_t *stream_page;
    const int32_t *stream_meta;
    const void *q;          // bf16 [n_q][Hq][D], one row per episode
    void   *out;            // bf16 [n_q][Hq][D]
    float  *mass;           // fp32 or null
    int32_t *status;
    int32_t Hq, Hkv, rep;
    int32_t mass_stride;
    // (the small kernel takes these parameters too; its list is every page that a CTA's rows see)
    int32_t list_pages;     // most pages a CTA of this launch covers, and most slots they can touch (sizes of its lists)
    int32_t list_slots;
    int32_t wait_first;     // as in AttnParams
    float   scale_log2;
};
constexpr int kSmallMaxPages = 24;
struct SmallParams : ClusterDecodeParams {
    int32_t n_list;             // the cached pages of a single episode travel here (else 0: they are in the gather plan)
    int2    list[kSmallMaxPages];   // page id, slot << 8 | valid keys
};
constexpr int kMaxCluster = 16;
constexpr int kMaxDevices = 64;     // devices whose properties are kept in fixed arrays
// Contiguous keys in segments instead of pool pages (the entry point that allocates nothing).
constexpr int kStaticMaxSeg = 255;
struct StaticDecodeParams {
    ClusterDecodeParams d;                  // tm_knew / tm_vnew cover the whole stream, ep0.n_slots = segments
    int32_t seg_off[kStaticMaxSeg + 2];     // first key of every slot (slot n_seg = the new keys), then the total
    int32_t page_off[kStaticMaxSeg + 2];    // the same in pages (16 keys of one slot, the last one of a slot partly filled)
};

struct CombineParams {
    const float *part_o, *part_lse, *part_slot;
    const int2 *part_rng;       // [split][row]: first and last slot that the split has written, or null: all are
    void  *out;
    float *mass;
    const int32_t *row_slots;   // [n_q_total]: G_b of the row's episode
    int32_t n_q_total, Hq, D;
    int32_t slot_stride;        // row stride of part_slot
    int32_t mass_stride;        // row stride of mass
    int32_t n_splits;
};

// Programmatic dependent launch: a kernel launched this way may start (set-up only) while the previous kernel
// of the stream is still draining; it must execute pdl_wait() before it touches anything a predecessor may have
// written, and pdl_trigger() as early as it likes so that its own successor can be set up the same way.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename Kernel, typename Params>
inline cudaError_t launch_pdl(Kernel kernel, dim3 grid, dim3 block, size_t smem, cudaStream_t st, const Params &prm,
                              unsigned cluster_x = 1)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cluster_x > 1) {                                     // grid.x must be a multiple of cluster_x
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = cluster_x;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
    }
    void *args[1] = {const_cast<Params *>(&prm)};           // not the typed form: that copies the parameters once more
    return cudaLaunchKernelExC(&cfg, reinterpret_cast<const void *>(kernel), args);
}
// the same for kernels that take several plain arguments
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_n(void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
#endif

// Parked log-sums -> masses, and their sums per object (see mass_finish_kernel)
struct FinishParams {
    float *mass;                // [n_q_total][Hq][mass_stride]: log2-sums of the slots, replaced by shares of the row's total
    const float *lse;           // [split][n_q_total][Hq]
    const float2 *bnd;          // [split][n_q_total][Hq] (only with splits)
    const int32_t *row_slots;   // [n_q_total]: G_b of the row's episode, or null: max_slots
    const int32_t *row_obj;     // [n_q_total]: object of every query row, -1 = none (only with mass_sum)
    float *mass_sum;            // fp32 [n_obj][sum_stride] or null: added to
    int32_t n_q_total, Hq, mass_stride, sum_stride, n_splits, max_slots;
};
constexpr int kFinishSplits = 8;
// n_sm: multiprocessors of the device
cudaError_t launch_mass_finish(const FinishParams &p, int n_sm, cudaStream_t st);

// Tensor map of a caller's [n][Hkv][D] bf16 keys or values with boxes of box_rows(D) rows of a head (in enl_host.cu)
bool encode_key_map(CUtensorMap *tm, const void *base, int D, int Hkv, int n);

// launchers (defined in the .cu files of the kernels)
cudaError_t launch_attention(const AttnParams &p, int head_dim, int n_items, cudaStream_t st);
cudaError_t launch_combine(const CombineParams &p, cudaStream_t st);
cudaError_t launch_decode(const DecodeParams &p, int head_dim, int batch, cudaStream_t st);
cudaError_t prepare_decode(int head_dim);
// cluster: CTAs per (episode, kv head), 1, 2, 4, 8 or 16
cudaError_t launch_decode_cluster(const ClusterDecodeParams &p, int head_dim, int batch, int cluster, cudaStream_t st);
cudaError_t launch_decode_static(const StaticDecodeParams &p, int head_dim, int cluster, cudaStream_t st);
constexpr int kClusterMaxPages = 288;         // pages of a CTA of these kernels
// Short calls (see enl_attn_small_sm100.cu): every page a CTA sees in shared memory at once.
cudaError_t prepare_small(int head_dim);
// row_groups: 1, 2 or 4 groups of 16 query rows (tokens x q heads of a kv head) per CTA
cudaError_t launch_small(const SmallParams &p, int head_dim, int row_groups, int row_blocks, int batch, cudaStream_t st);
int decode_cluster_smem(int head_dim, int list_pages, int list_slots, int rep);
constexpr int kClusterPairSmem = 115712;      // two CTAs of up to this much fit an SM (228 KB, of which a CTA takes 1 KB for itself)
// How many clusters of 2^i CTAs the current device runs at once: with two CTAs per SM, and with one (larger lists).
struct ClusterCaps {
    int two[5], one[5];
    int get(int i, int smem) const { return smem <= kClusterPairSmem ? two[i] : one[i]; }
};
// log2 of the widest cluster worth having for `heads` (kv heads x episodes) streams of up to `pages` pages.  Sixteen CTAs read a
// stream fastest, but from eight streams on they leave the next launch room for six of its eight clusters only, and clusters of eight
// merge faster.  Measured (one token, 24 groups, sixteens against eights, us; without masses, with masses):
//   8 kv heads, D 128, 640 keys (a page a warp) 5.05 / 4.59, 5.81 / 5.43; 1280 keys (two pages) 5.33 / 6.14, 6.19 / 6.81; 2560 keys
//     5.88 / 6.92, 6.85 / 7.83;  D 64, the same sizes: 4.37 / 3.93, 5.06 / 4.69; 4.51 / 4.95, 5.30 / 5.66; 4.81 / 5.60, 5.73 / 6.53
//   6 kv heads, D 128, 640 keys 4.70 / 5.01, 5.51 / 5.51; 2560 keys 5.77 / 7.27, 6.75 / 8.10;  5 kv heads 4.61 / 4.78, 5.39 / 5.53;
//     5.51 / 7.19, 6.48 / 8.02
// Contiguous keys (24 segments and new keys), with masses: 8 kv heads, D 128, 75 pages 7.07 / 6.66, 92 pages 7.22 /
//     6.84, 108 pages 7.45 / 8.36, 176 pages 9.27 / 9.75, 261 pages 11.28 / 11.85; D 64, 86 pages 6.31 / 5.86, 106 pages 6.44 / 6.69, 188 pages
//     7.02 / 7.53; one q head per kv head, D 128, 73 pages 6.68 / 6.52, 108 pages 7.05 / 8.10; eight, 79 pages 7.55 / 7.16, 106 pages 7.93 / 8.66
inline int widest_cluster_log(int heads, int pages) { return heads >= 8 && pages <= 8 * 12 ? 3 : 4; }
// Opt the kernel for pool pages, and the one for contiguous keys, in on the current device and ask for its capacities there.
cudaError_t prepare_decode_cluster(int head_dim, ClusterCaps *caps);
cudaError_t prepare_decode_static(int head_dim, ClusterCaps *caps);
// Page ids of (part of) one group, passed by value to the scatter kernel.
constexpr int kScatterPages = 64;
struct PageRun {
    int32_t ids[kScatterPages];   // ids[i] = page holding group positions (first_page + i)*16 ..
    int32_t first_page;           // index within the group of ids[0]
};
// zero_rows: rows behind the last token of the run's last page that are cleared (the group ends there)
cudaError_t launch_page_scatter(void *kpool_layer, void *vpool_layer, const void *k, const void *v,
                                const PageRun &run, int first_pos, int n_tokens, int zero_rows,
                                int Hkv, int D, int n_sm, cudaStream_t st);
// The same for up to kScatterLayers layers in one launch: layer l reads k[l] + src_off, v[l] + src_off (bytes)
// and writes the pool of layer layer0 + l.
constexpr int kScatterLayers = 64;
struct LayerSrc {
    const void *k[kScatterLayers];
    const void *v[kScatterLayers];
};
cudaError_t launch_page_scatter_layers(void *kpool, void *vpool, size_t layer_bytes, int layer0, int n_layers,
                                       const LayerSrc &src, size_t src_off, const PageRun &run, int first_pos,
                                       int n_tokens, int zero_rows, int Hkv, int D, int n_sm, cudaStream_t st);
// Copies whole pages (all kv heads) between two pools of the page format, every layer, K and V: pairs[i] =
// {source page, destination page}; the pools may be device memory or pinned host memory.
cudaError_t launch_page_copy(const uint8_t *src_k, const uint8_t *src_v, uint8_t *dst_k, uint8_t *dst_v,
                             size_t src_layer_bytes, size_t dst_layer_bytes, const int2 *pairs, int n_pairs, int layer0,
                             int n_layers, int page_bytes, int ctas, cudaStream_t st);
// Writes a gather plan of up to kPlanParamBytes to device memory out of the kernel's own parameters: no staging buffer
// that the host would have to wait for, and (unlike a copy) it chains to its neighbours by programmatic dependent launch.
constexpr int kPlanParamBytes = 28672;        // of the 32764 that a launch may carry
cudaError_t launch_plan_write(void *dst, const void *src, size_t bytes, cudaStream_t st);
int attention_park_slots();
cudaError_t launch_mass(const MassParams &p, int head_dim, int n_items, cudaStream_t st);
cudaError_t prepare_mass(int head_dim);
// Opts the attention kernel into its dynamic shared memory size on the current device.
cudaError_t prepare_attention(int head_dim);
// can the device run the head_dim-128 kernel as clusters of two CTAs (the in-kernel merge of two KV splits)?
bool attention_pairs_supported();

}  // namespace enl
