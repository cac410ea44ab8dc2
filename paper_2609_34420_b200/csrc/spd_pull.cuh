// Bit rows of the distance build's pull kernels (spd_pull.cu, spd_pull_large.cu), and their plans.
#pragma once

#include "gt_common.cuh"

namespace gt {

struct PullPlan {
    bool fits;                // false: the batch has a graph that does not fit; another build is used
    int targets;              // target columns of a thread block: 32, 64 or 128
    int threads;
    unsigned blocks;
    size_t smem_bytes;
};

PullPlan spd_pull_plan(const gt_batch* batch, int64_t nnz, int32_t max_dist);

gt_status spd_pull_launch(const PullPlan& plan, const int32_t* row_ptr, const int32_t* col_idx,
                          const int32_t* cu_seqlens, const int64_t* spd_offsets, const gt_batch* batch,
                          int32_t max_dist, uint8_t* spd, cudaStream_t stream);

// The variant for one graph whose edge list does not fit shared memory: lists and code planes in the workspace.
struct PullLargePlan {
    bool fits;
    int threads;
    unsigned blocks;
    size_t smem_bytes;
    size_t order_off, info_off, hub_off, list_off, plane_off, total_bytes;
    int32_t n_pad;            // pitch of a code plane, in words
};

PullLargePlan spd_pull_large_plan(const gt_batch* batch, int64_t nnz, int32_t max_dist);

gt_status spd_pull_large_launch(const PullLargePlan& plan, const int32_t* row_ptr, const int32_t* col_idx, int64_t nnz,
                                const gt_batch* batch, int32_t max_dist, uint8_t* spd, void* workspace, cudaStream_t stream);

constexpr size_t kPullSmemLimit = 226 * 1024;      // and under 1 KB of static arrays

__host__ __device__ constexpr size_t pull_align(size_t x) { return (x + 15) & ~(size_t)15; }

inline int pull_planes(int32_t max_dist)           // bits of the largest code, max_dist + 1
{
    int planes = 1;
    while (((max_dist + 1) >> planes) != 0) ++planes;
    return planes;
}

constexpr int kLeaders = 1;

template <int kT>
struct Rows {
    static constexpr int kWords = kT / 32;
    static constexpr int kBytes = kT / 8;
    // Bit of target t of the block.  Within a word of 32 targets, target 4k+j sits at bit 8j+k: the byte lanes of
    // (word >> k) & 0x01010101 are then four neighbouring output bytes.
    static __device__ __forceinline__ int bit(int t) { return (t & 3) * 8 + ((t >> 2) & 7); }
    static __device__ __forceinline__ void load(const uint8_t* base, int i, uint32_t (&w)[kWords])
    {
        if constexpr (kT == 32) w[0] = ((const uint32_t*)base)[i];
        else if constexpr (kT == 64) { const uint2 x = ((const uint2*)base)[i]; w[0] = x.x; w[1] = x.y; }
        else { const uint4 x = ((const uint4*)base)[i]; w[0] = x.x; w[1] = x.y; w[2] = x.z; w[3] = x.w; }
    }
    static __device__ __forceinline__ void store(uint8_t* base, int i, const uint32_t (&w)[kWords])
    {
        if constexpr (kT == 32) ((uint32_t*)base)[i] = w[0];
        else if constexpr (kT == 64) ((uint2*)base)[i] = make_uint2(w[0], w[1]);
        else ((uint4*)base)[i] = make_uint4(w[0], w[1], w[2], w[3]);
    }
    // the bit of target t, as a row (t outside the block: empty)
    static __device__ __forceinline__ void add_target(int t, int nt, uint32_t (&w)[kWords])
    {
        const bool in = (unsigned)t < (unsigned)nt;
        const uint32_t m = 1u << bit(t & (kT - 1));
#pragma unroll
        for (int k = 0; k < kWords; ++k) w[k] |= in && (t >> 5) == k ? m : 0u;
    }
};

// Four bit planes of 32 targets -> eight words of four bytes: bit 8 l + j of plane b becomes bit b (kHigh: 4 + b) of byte l of
// o[j].  Pairs of planes are merged into 2-bit fields, these into nibbles, and the nibbles taken apart.
template <bool kHigh>
__device__ __forceinline__ void nibbles(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t* o)
{
    const uint32_t e0 = (c0 & 0x55555555u) | ((c1 & 0x55555555u) << 1), e1 = ((c0 >> 1) & 0x55555555u) | (c1 & 0xAAAAAAAAu);
    const uint32_t f0 = (c2 & 0x55555555u) | ((c3 & 0x55555555u) << 1), f1 = ((c2 >> 1) & 0x55555555u) | (c3 & 0xAAAAAAAAu);
    const uint32_t n[4] = {(e0 & 0x33333333u) | ((f0 & 0x33333333u) << 2), (e1 & 0x33333333u) | ((f1 & 0x33333333u) << 2),
                           ((e0 >> 2) & 0x33333333u) | (f0 & 0xCCCCCCCCu), ((e1 >> 2) & 0x33333333u) | (f1 & 0xCCCCCCCCu)};
#pragma unroll
    for (int j = 0; j < 4; ++j) {           // n[j]: nibbles j (low) and j + 4 (high) of every byte lane
        if (kHigh) {
            o[j] |= (n[j] << 4) & 0xF0F0F0F0u;
            o[j + 4] |= n[j] & 0xF0F0F0F0u;
        } else {
            o[j] = n[j] & 0x0F0F0F0Fu;
            o[j + 4] = (n[j] >> 4) & 0x0F0F0F0Fu;
        }
    }
}

// inclusive sum over the lanes of a warp
__device__ __forceinline__ int warp_scan(int x, int lane)
{
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, x, off);
        if (lane >= off) x += up;
    }
    return x;
}

// Close the targets' rows under each other, a strongly connected set at a time.  With a leader a, C = all that its row
// leads to and B = all targets whose rows lead to a; every target of both has exactly the row C.  One warp holds the
// rows; a few leaders are enough (the passes below finish what is left).
template <int kT>
__device__ __forceinline__ void close_targets(uint8_t* cur, const uint16_t* tpos, int nt, const uint32_t (&full)[Rows<kT>::kWords], int lane)
{
    using R = Rows<kT>;
    constexpr int W = R::kWords;
    constexpr int kPer = kT / 32;                  // targets per lane
    uint32_t row[kPer][W], todo[W];
    int bits[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int t = lane + 32 * j;
        bits[j] = t < nt ? R::bit(t & (kT - 1)) : 32;
#pragma unroll
        for (int k = 0; k < W; ++k) row[j][k] = 0u;
        if (t < nt) R::load(cur, tpos[t], row[j]);
    }
#pragma unroll
    for (int k = 0; k < W; ++k) todo[k] = full[k];
    for (int leader = 0; leader < kLeaders; ++leader) {
        unsigned best = 0u;                                      // the longest row that is left: size << 7 | target
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const uint32_t m = bits[j] < 32 ? 1u << bits[j] : 0u;
            int size = 0;
#pragma unroll
            for (int k = 0; k < W; ++k) size += __popc(row[j][k]);
            if (todo[j] & m) best = max(best, (unsigned)size << 7 | (unsigned)(lane + 32 * j));
        }
        best = __reduce_max_sync(0xffffffffu, best);
        if (best == 0u) break;
        const int lead = (int)(best & 127u);
        uint32_t c[W], back[W];
#pragma unroll
        for (int k = 0; k < W; ++k) c[k] = back[k] = (lead >> 5) == k ? 1u << R::bit(lead & (kT - 1)) : 0u;
        for (bool grew = true; grew;) {
            uint32_t x[W], y[W], fresh = 0u;
#pragma unroll
            for (int k = 0; k < W; ++k) x[k] = y[k] = 0u;
#pragma unroll
            for (int j = 0; j < kPer; ++j) {                     // target lane + 32 j sits in word j
                const uint32_t m = bits[j] < 32 ? 1u << bits[j] : 0u;
                uint32_t leads = 0u;
#pragma unroll
                for (int k = 0; k < W; ++k) {
                    if (c[j] & m) x[k] |= row[j][k];
                    leads |= row[j][k] & back[k];
                }
                if (leads) y[j] |= m;
            }
#pragma unroll
            for (int k = 0; k < W; ++k) {
                x[k] = __reduce_or_sync(0xffffffffu, x[k]) | c[k];
                y[k] = __reduce_or_sync(0xffffffffu, y[k]) | back[k];
                fresh |= (x[k] ^ c[k]) | (y[k] ^ back[k]);
                c[k] = x[k]; back[k] = y[k];
            }
            grew = fresh != 0u;
        }
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const uint32_t m = bits[j] < 32 ? 1u << bits[j] : 0u;
            if (c[j] & back[j] & m) {
#pragma unroll
                for (int k = 0; k < W; ++k) row[j][k] = c[k];
                R::store(cur, tpos[lane + 32 * j], c);
            }
        }
#pragma unroll
        for (int k = 0; k < W; ++k) todo[k] &= ~(c[k] & back[k]);
    }
}

// Row i inherits the rows of the targets it reaches (tpos: where the targets' rows are).
template <int kT>
__device__ __forceinline__ void inherit(uint8_t* cur, int i, const uint16_t* tpos)
{
    using R = Rows<kT>;
    constexpr int W = R::kWords;
    uint32_t row[W], rem[W];
    R::load(cur, i, row);
#pragma unroll
    for (int k = 0; k < W; ++k) rem[k] = row[k];
    bool grew = false;
    for (;;) {
        int word = -1;
#pragma unroll
        for (int k = W - 1; k >= 0; --k) word = rem[k] ? k : word;
        if (word < 0) break;
        uint32_t rw = 0u;
#pragma unroll
        for (int k = 0; k < W; ++k) rw = word == k ? rem[k] : rw;
        const int bit = __ffs((int)rw) - 1;
        const int t = word * 32 + (bit & 7) * 4 + (bit >> 3);
        uint32_t x[W];
        R::load(cur, tpos[t], x);
#pragma unroll
        for (int k = 0; k < W; ++k) {
            grew |= (x[k] & ~row[k]) != 0u;
            row[k] |= x[k];
            rem[k] &= ~x[k];            // target t is in its own row
        }
    }
    if (grew) R::store(cur, i, row);
}

// 32 output bytes of which the row's pitch (a multiple of 16) has room for `room`: a whole sector where it is aligned.
__device__ __forceinline__ void store_row_piece(uint8_t* at, const uint32_t (&o)[8], int room)
{
    if (room >= 32 && ((uintptr_t)at & 31u) == 0) {
        asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(at), "r"(o[0]), "r"(o[1]), "r"(o[2]),
                     "r"(o[3]), "r"(o[4]), "r"(o[5]), "r"(o[6]), "r"(o[7])
                     : "memory");
    } else {
        *(uint4*)at = make_uint4(o[0], o[1], o[2], o[3]);
        if (room > 16) *(uint4*)(at + 16) = make_uint4(o[4], o[5], o[6], o[7]);
    }
}

// One word of a row's code planes -> 32 output bytes at `row`, columns `col` and up of a block of nt valid targets and `cols`
// columns inside the row pitch; columns past the last target are row padding.
__device__ __forceinline__ void emit_word(const uint32_t (&c)[8], int n_planes, uint8_t* row, int col, int nt, int cols)
{
    uint32_t o[8];
    nibbles<false>(c[0], c[1], c[2], c[3], o);
    if (n_planes > 4) nibbles<true>(c[4], c[5], c[6], c[7], o);
    if (col + 32 > nt) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int past = col + 4 * j + 4 - nt;       // bytes of this word past the last node
            if (past > 0) o[j] |= past >= 4 ? 0xffffffffu : 0xffffffffu << (8 * (4 - past));
        }
    }
    store_row_piece(row, o, cols - col);
}

}  // namespace gt
