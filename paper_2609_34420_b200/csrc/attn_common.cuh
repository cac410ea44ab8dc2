// Host-side pieces shared by the attention entry points: TMA descriptor encoding for the
// packed [T, H, d] bf16 tensors and argument validation.
#pragma once

#include <cuda.h>

#include "gt_common.cuh"

namespace gt {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

// 3-D tensor map over a bf16 [T, H, d] tensor; one box = 128 consecutive rows of one head
// (d x 1 x 128 elements), written to shared memory as 128 rows of 2d bytes with the
// swizzle mode that matches the row length (128B for d=64, 64B for d=32, 32B for d=16).
gt_status encode_thd_map(CUtensorMap* map, const void* base, int32_t n_total, int32_t n_heads, int32_t head_dim);

// 2-D tensor map over the uint8 SPD matrix of a single graph (n rows of pitch round_up(n,16));
// one box = box_rows rows x 128 key columns, written with the 128-byte swizzle (16-byte chunk c
// of row r lands at chunk c ^ (r & 7)); out-of-range rows / columns are zero-filled.
gt_status encode_spd_map(CUtensorMap* map, const uint8_t* spd, int32_t n, int32_t box_rows);

// 2-D tensor map over the fp32 dQ accumulator [T, H*d]; one box = 128 rows x 32 floats of one
// head, 128-byte swizzle (target of the backward kernel's TMA reduce-add).
gt_status encode_dq_map(CUtensorMap* map, const float* dq_acc, int32_t n_total, int32_t n_heads, int32_t head_dim);

// Tensor maps of the SPD blocks of a packed batch, whose sizes and offsets are known on the device only: map g is `model` (a map
// of any size, from encode_spd_map) with graph g's base, dimensions and pitch put in.  One thread per graph; the reader of a
// map acquires it with acquire_tensor_map before its first use.
__device__ __forceinline__ void make_spd_map(uint8_t* map, const CUtensorMap& model, const uint8_t* block, int32_t n)
{
    const uint32_t ld = (uint32_t)((n + 15) & ~15);
#pragma unroll
    for (int i = 0; i < 8; ++i) ((uint4*)map)[i] = ((const uint4*)&model)[i];
    asm volatile("tensormap.replace.tile.global_address.global.b1024.b64 [%0], %1;" ::"l"(map), "l"(block) : "memory");
    asm volatile("tensormap.replace.tile.global_dim.global.b1024.b32 [%0], 0, %1;" ::"l"(map), "r"(ld) : "memory");
    asm volatile("tensormap.replace.tile.global_dim.global.b1024.b32 [%0], 1, %1;" ::"l"(map), "r"(n) : "memory");
    asm volatile("tensormap.replace.tile.global_stride.global.b1024.b64 [%0], 0, %1;" ::"l"(map), "l"((uint64_t)ld) : "memory");
    asm volatile("fence.proxy.tensormap::generic.release.gpu;" ::: "memory");
}
__device__ __forceinline__ void acquire_tensor_map(const void* map)
{
    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(map) : "memory");
}
constexpr size_t kMapBytes = 128;
// Their place in a workspace whose address is a multiple of 16; none for a single graph.
inline size_t maps_bytes(int32_t n_graphs) { return n_graphs > 1 ? align_up((size_t)n_graphs * kMapBytes, 256) + kMapBytes : 0; }
inline uint8_t* maps_at(uint8_t* region) { return (uint8_t*)align_up(reinterpret_cast<uintptr_t>(region), kMapBytes); }

// Work list of a packed batch, whose sizes are on the device only: entry i = {graph, block of `rows` rows of it, the graph's first
// row, its rows}; graph -1: unused.  A grid of (largest graph) x (graphs) launches a third to a half of its blocks for nothing where
// sizes vary a lot, and those hold up the others (30 graphs of 128 to 4 096 nodes: forward 520 -> 504 us, backward 1 332 -> 1 275;
// 64 of 512 to 2 048: 949 -> 945, 2 565 -> 2 518).  Up to kListSorted graphs come by falling size: the blocks that take longest start
// first, which a few large graphs need (in batch order 510 and 1 303 us).  More graphs stay in the batch's order: the tail is short
// anyway, and blocks of different lengths side by side hide each other's fill and drain (200 graphs of 64 to 1 000 nodes: 436 us in
// order, 443 sorted).  A warp per graph writes its graph's entries and the unused ones behind them, with nothing to wait for.
constexpr int kListSorted = 64;
inline size_t list_entries(const gt_batch* b, int32_t rows) { return (size_t)(b->n_total / rows) + (size_t)b->n_graphs; }
inline size_t list_bytes(const gt_batch* b, int32_t rows) { return b->n_graphs > 1 ? align_up(list_entries(b, rows) * sizeof(int4), 256) : 0; }
// The grid without the list has more than `blocks` blocks more than the one with it (many graphs of one size need no list).
inline bool list_saves(const gt_batch* b, int32_t rows, int32_t n_heads, size_t blocks)
{
    return (size_t)((b->max_seqlen + rows - 1) / rows) * (size_t)b->n_graphs * (size_t)n_heads > list_entries(b, rows) * (size_t)n_heads + blocks;
}
template <int kRows>
__device__ __forceinline__ void write_work_list(int4* list, int32_t entries, const int32_t* __restrict__ cu_seqlens, int32_t n_graphs, int32_t g)
{
    const int lane = threadIdx.x & 31;
    const int32_t c0 = cu_seqlens[g], n = cu_seqlens[g + 1] - c0, blocks = (n + kRows - 1) / kRows;
    int32_t first = c0 / kRows + g, end = (c0 + n) / kRows + g + 1;      // in batch order: the next graph's first entry
    if (n_graphs <= kListSorted) {
        int32_t before = 0, all = 0;
        for (int j = lane; j < n_graphs; j += 32) {
            const int32_t other = cu_seqlens[j + 1] - cu_seqlens[j], b = (other + kRows - 1) / kRows;
            before += other > n || (other == n && j < g) ? b : 0;
            all += b;
        }
        first = __reduce_add_sync(0xffffffffu, before);
        end = first + blocks == __reduce_add_sync(0xffffffffu, all) ? entries : first + blocks;
    }
    for (int32_t i = first + lane; i < end && i < entries; i += 32)
        list[i] = i < first + blocks ? make_int4(g, i - first, c0, n) : make_int4(-1, 0, 0, 0);
}

// The graph that entry `entry` belongs to in the batch's order, where graph g's entries begin at cu_seqlens[g] / kRows + g; by whole warps.
template <int kRows>
__device__ __forceinline__ int32_t graph_of_entry(const int32_t* __restrict__ cu_seqlens, int32_t n_graphs, int32_t entry)
{
    const int lane = threadIdx.x & 31;
    int32_t lo = 0, n = n_graphs;                          // it is one of [lo, lo + n)
    while (n > 1) {
        const int32_t step = (n + 31) / 32, x = lane * step;
        const bool begins = x < n && cu_seqlens[lo + x] / kRows + lo + x <= entry;
        const int32_t last = __popc(__ballot_sync(0xffffffffu, begins)) - 1;       // (lane 0's begins)
        lo += last * step;
        n = min(step, n - last * step);
    }
    return lo;
}

// Clusters of `split` blocks that the device holds at a time (a cluster's blocks lie in one group of SMs), -1: none.
constexpr int kMaxSplit = 4;
struct ClusterFit { std::atomic<int32_t> n[kMaxSplit + 1] = {}; };       // by size; 0: not asked yet
template <typename Kernel>
int32_t clusters_at_a_time(Kernel kern, int threads, size_t smem, ClusterFit& fits, int32_t split)
{
    if (split == 1) return sm_count();                     // (whatever the shared memory, these kernels' blocks have an SM each)
    int32_t fit = fits.n[split].load(std::memory_order_relaxed);
    if (fit != 0) return fit;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)split;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)split);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    fit = n > 0 ? n : -1;
    fits.n[split].store(fit, std::memory_order_relaxed);
    return fit;
}

// Blocks of a cluster that share the work of one: where `blocks` of `tiles` tiles each end soonest, taking a tile as the unit of time,
// `fixed` for a block's fill and drain and `shared` for what a cluster costs on top.  The grid runs in waves, so that a last wave
// of few blocks may end sooner in shares, too.  Sharing has to promise 5 %.
template <typename Kernel>
int32_t cluster_split(Kernel kern, int threads, size_t smem, ClusterFit& fits, int64_t blocks, int32_t tiles, float fixed, float shared)
{
    int32_t best = 1;
    float least = 0.95f * (float)((blocks + sm_count() - 1) / sm_count()) * ((float)tiles + fixed);
    for (int32_t split = 2; split <= kMaxSplit && split <= tiles; ++split) {
        const int32_t fit = clusters_at_a_time(kern, threads, smem, fits, split);
        if (fit <= 0) continue;
        const float time = (float)((blocks + fit - 1) / fit) * ((float)((tiles + split - 1) / split) + fixed + shared);
        if (time < least) {
            least = time;
            best = split;
        }
    }
    return best;
}

struct AttnArgsCheck {
    const void* ptrs[12];
    int n_ptrs;
};

inline gt_status validate_attn_common(const gt_batch* batch, int32_t n_heads, int32_t head_dim, int32_t max_dist,
                                      const int64_t* spd_offsets)
{
    gt_status st = validate_batch(batch);
    if (st != GT_OK) return st;
    if (n_heads < 1 || max_dist < 1 || max_dist > 254) return GT_ERR_INVALID_ARG;
    if (head_dim != 32 && head_dim != 64) return GT_ERR_UNSUPPORTED;
    if (batch->n_graphs > 1 && spd_offsets == nullptr) return GT_ERR_INVALID_ARG;
    return GT_OK;
}

}  // namespace gt
