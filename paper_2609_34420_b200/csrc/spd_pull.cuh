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
    size_t order_off, info_off, hub_off, list_off, component_off, plane_off, total_bytes;
    int32_t n_pad;            // pitch of a code plane, in words
};

constexpr int32_t kDenseMinNodes = 14500;          // a single graph from here on that is not pulled takes the bit matrices

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

// Close the targets' rows under each other around the target a with the longest row.  C = all that its row leads to, B = all
// targets whose rows lead to a; every target of both, a strongly connected set, has exactly the row C.  One warp holds the rows; the
// passes finish what is left (eight such sets at a time took longer).
template <int kT>
__device__ __forceinline__ void close_targets(uint8_t* cur, const uint16_t* tpos, int nt, const uint32_t (&full)[Rows<kT>::kWords], int lane)
{
    using R = Rows<kT>;
    constexpr int W = R::kWords;
    constexpr int kPer = kT / 32;                  // targets per lane
    uint32_t row[kPer][W];
    int bits[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int t = lane + 32 * j;
        bits[j] = t < nt ? R::bit(t & (kT - 1)) : 32;
#pragma unroll
        for (int k = 0; k < W; ++k) row[j][k] = 0u;
        if (t < nt) R::load(cur, tpos[t], row[j]);
    }
    unsigned best = 0u;                                      // the longest row: size << 7 | target
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const uint32_t m = bits[j] < 32 ? 1u << bits[j] : 0u;
        int size = 0;
#pragma unroll
        for (int k = 0; k < W; ++k) size += __popc(row[j][k]);
        if (full[j] & m) best = max(best, (unsigned)size << 7 | (unsigned)(lane + 32 * j));
    }
    best = __reduce_max_sync(0xffffffffu, best);
    if (best == 0u) return;
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
        if (c[j] & back[j] & m) R::store(cur, tpos[lane + 32 * j], c);
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

// ---- reachability over long ways ----
// A pass brings a row one edge nearer to its targets, and a row from which no target of the block has been reached yet inherits
// nothing, so by the kernels' passes alone a ring of 9 000 nodes takes 4 500 of them.  A kernel gives up after a number of rounds, and
// finish_far takes the rows from its output, finishes them in the caller's edge list and mends the output, with two shortcuts
// before its passes, both exact for any directed graph:
//   jump        a vertex reaches what a vertex that it reaches does: row |= row[jump], jump = jump[jump], which doubles the way at
//               every round, from one of the out-neighbours on; 16 rounds (n < 2^16), and again with another one 64 rounds later
//   components  vertices joined by edges that have a reverse reach each other, so all rows of such a component become their union,
//               and an undirected graph is finished
// It stands at the kernels' very end: the same rounds inside their loops cost graphs that never come here 4 to 8 % (64 directed
// graphs of 512 to 2 048 nodes: 244 -> 255 us, here 249; power law, 9 000 nodes: 234 -> 254, here 234).
constexpr int kJumpRounds = 16, kJumpEvery = 64, kMergeEvery = 16;
constexpr int kMaxSearch = 64;           // longest edge list that is searched for an edge's reverse

// Out-neighbour number `which` of every vertex (itself, if it has none).
__device__ __forceinline__ void start_jumps(uint16_t* jump, const int32_t* __restrict__ rows, const int32_t* __restrict__ cols, int node0, int n, int which)
{
    for (int v = threadIdx.x; v < n; v += blockDim.x) {
        const int e0 = rows[v], deg = rows[v + 1] - e0;
        jump[v] = (uint16_t)(deg > 0 ? cols[e0 + which % deg] - node0 : v);
    }
    __syncthreads();
}

// f(v, u, v has more than kMaxSearch out-edges) for every edge v -> u: a warp takes the edges of 32 vertices, one after the other, by its lanes.
template <class F>
__device__ __forceinline__ void for_edges(const int32_t* __restrict__ rows, const int32_t* __restrict__ cols, int node0, int n, F f)
{
    const int lane = threadIdx.x & 31;
    for (int v0 = (threadIdx.x >> 5) * 32; v0 < n; v0 += blockDim.x) {
        const int e0 = rows[min(v0 + lane, n)], e1 = rows[min(v0 + lane + 1, n)];
        const int last = __shfl_sync(0xffffffffu, e1, 31);
        int e = __shfl_sync(0xffffffffu, e0, 0) + lane, next = e < last ? cols[e] : 0;
        for (; __any_sync(0xffffffffu, e < last); e += 32) {
            const int u = next - node0;
            if (e + 32 < last) next = cols[e + 32];
            int src = 0;                                   // vertices whose edges end at or before e
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (__shfl_sync(0xffffffffu, e1, src + step - 1) <= e) src += step;
            const bool hub = __shfl_sync(0xffffffffu, e1 - e0, src & 31) > kMaxSearch;
            if (e < last) f(v0 + src, u, hub);
            __syncwarp();
        }
    }
}

// A component's vertices point to its root, the one that comes last in this order: with neighbours numbered one after the other, as
// in a mesh, hooks by number would make one long chain.
__device__ __forceinline__ uint32_t component_order(int v) { return ((uint32_t)v * 40503u) & 0xffffu; }

__device__ __forceinline__ int root_of(volatile uint16_t* up, int x)
{
    for (;;) {
        const int parent = up[x];
        if (parent == x) return x;
        const int above = up[parent];
        if (above != parent) up[x] = (uint16_t)above;      // x is no root and stays none, so no hook is lost
        x = parent;
    }
}

// Roots are hooked under later ones only, by compare and swap.  An edge between two vertices of more than kMaxSearch out-edges is
// taken for one without a reverse.
__device__ __forceinline__ void find_components(uint16_t* up, const int32_t* __restrict__ rows, const int32_t* __restrict__ cols, int node0, int n)
{
    for (int v = threadIdx.x; v < n; v += blockDim.x) up[v] = (uint16_t)v;
    __syncthreads();
    for_edges(rows, cols, node0, n, [&](int v, int u, bool hub) {
        if (u == v || (u > v && !hub)) return;
        int a = root_of(up, v), b = root_of(up, u);
        if (a == b) return;
        const int e0 = rows[u], e1 = rows[u + 1];
        if (e1 - e0 > kMaxSearch) return;
        bool both = false;
        for (int e = e0; e < e1 && !both; e += 4) {
#pragma unroll
            for (int k = 0; k < 4; ++k) both |= cols[min(e + k, e1 - 1)] - node0 == v;
        }
        while (both && a != b) {
            const bool swap = component_order(a) > component_order(b);
            const int low = swap ? b : a, high = swap ? a : b;
            if (atomicCAS(&up[low], (unsigned short)low, (unsigned short)high) == low) break;
            a = root_of(up, a);
            b = root_of(up, b);
        }
    });
    for (int moved = 1; __syncthreads_or(moved);) {        // everyone's root; a vertex' owner is the only one to write here
        moved = 0;
        for (int v = threadIdx.x; v < n; v += blockDim.x) {
            const int parent = ((volatile uint16_t*)up)[v], above = ((volatile uint16_t*)up)[parent];
            if (above != parent) { ((volatile uint16_t*)up)[v] = (uint16_t)above; moved = 1; }
        }
    }
}

// One round of the shortcuts; `up` and `jump`: nullptr for a round without.
template <int kT>
__device__ __forceinline__ void shortcuts(uint8_t* cur, const uint16_t* up, volatile uint16_t* jump, int n)
{
    using R = Rows<kT>;
    constexpr int W = R::kWords;
    if (up != nullptr) {
        for (int v = threadIdx.x; v < n; v += blockDim.x) {
            const int r = up[v];
            if (r == v) continue;
            uint32_t mine[W], all[W];
            R::load(cur, v, mine);
            R::load(cur, r, all);
#pragma unroll
            for (int k = 0; k < W; ++k)
                if (mine[k] & ~all[k]) atomicOr((uint32_t*)cur + r * W + k, mine[k]);
        }
        __syncthreads();
        for (int v = threadIdx.x; v < n; v += blockDim.x) {
            uint32_t all[W];
            R::load(cur, up[v], all);
            R::store(cur, v, all);
        }
        __syncthreads();
    }
    if (jump != nullptr) {
        for (int v = threadIdx.x; v < n; v += blockDim.x) {
            uint32_t mine[W], other[W];
            const int to = jump[v], next = jump[to];
            __threadfence_block();                         // a row that is read here covers the way up to a jump that was read before it
            R::load(cur, v, mine);
            R::load(cur, to, other);
#pragma unroll
            for (int k = 0; k < W; ++k) mine[k] |= other[k];
            R::store(cur, v, mine);
            __threadfence_block();
            jump[v] = (uint16_t)next;
        }
        __syncthreads();
    }
}

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p)
{
    uint32_t x;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(p) : "memory");
    return x;
}
__device__ __forceinline__ void st_release(uint32_t* p, uint32_t x) { asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(x) : "memory"); }

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
// The same in a matrix that begins anywhere (gt_spd_validate takes one).  Unrolled: an index into o would put it in local memory, which
// slows all of a kernel down by 8 %.
__device__ __forceinline__ void store_row_piece_anywhere(uint8_t* at, const uint32_t (&o)[8], int room)
{
    if (((uintptr_t)at & 15u) == 0) {
        store_row_piece(at, o, room);
        return;
    }
#pragma unroll
    for (int j = 0; j < 32; ++j)
        if (j < 16 || room > 16) at[j] = (uint8_t)(o[j / 4] >> (8 * (j % 4)));
}

struct FarState {
    uint8_t* out;                 // column t0 of row 0
    int64_t ld;
    const int32_t* rows;          // the graph's part of the caller's edge list
    const int32_t* cols;
    uint32_t* found;              // word that says whether `component` is there (for blocks of one graph that follow); nullptr: not kept
    uint16_t* component;
    int node0, n, t0, nt;
    uint32_t none_code;           // far_code + 1
    int components;               // rounds without them
};

// Pairs that are written as unreachable although there is a long way -> far; by the whole block.  `smem`: rows in the vertices' order,
// 4 n bytes behind them.
template <int kT>
__device__ __forceinline__ void finish_far(uint8_t* smem, const FarState& p)
{
    using R = Rows<kT>;
    constexpr int W = R::kWords;
    __shared__ uint32_t s_found;
    __shared__ uint16_t s_to[kT];
    const int n = p.n;
    uint8_t* const cur = smem;
    uint16_t *const up = (uint16_t*)(smem + pull_align((size_t)n * R::kBytes)), *const jump = up + n;
    const uint32_t none4 = p.none_code * 0x01010101u;
    uint32_t full[W];
#pragma unroll
    for (int k = 0; k < W; ++k) full[k] = 0u;
    for (int t = 0; t < p.nt; ++t) R::add_target(t, p.nt, full);
    for (int t = threadIdx.x; t < p.nt; t += blockDim.x) s_to[t] = (uint16_t)(p.t0 + t);
    // A word of a row is 32 bytes of the output, of which the row's pitch has room for 16 or 32.
    auto bytes_of = [&](int at, uint32_t (&o)[8]) {
        const uint8_t* piece = p.out + (int64_t)(at / W) * p.ld + 32 * (at % W);
        const bool first = 32 * (at % W) < p.nt, second = 32 * (at % W) + 16 < p.nt;
        if (((uintptr_t)piece & 15u) != 0) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                o[j] = 0u;
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if (j < 4 ? first : second) o[j] |= (uint32_t)piece[4 * j + b] << (8 * b);
            }
            return;
        }
        const uint4 a = first ? *(const uint4*)piece : make_uint4(0u, 0u, 0u, 0u), b = second ? *(const uint4*)(piece + 16) : make_uint4(0u, 0u, 0u, 0u);
        o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w;
        o[4] = b.x; o[5] = b.y; o[6] = b.z; o[7] = b.w;
    };
    for (int at = threadIdx.x; at < n * W; at += 4 * blockDim.x) {
        uint32_t o[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i) bytes_of(min(at + i * (int)blockDim.x, n * W - 1), o[i]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint32_t w = 0u;
#pragma unroll
            for (int b = 0; b < 8; ++b) w |= (~__vcmpeq4(o[i][b], none4) & 0x01010101u) << b;
            if (at + i * (int)blockDim.x < n * W) ((uint32_t*)cur)[at + i * (int)blockDim.x] = w;
        }
    }
    __syncthreads();
    for (int v = threadIdx.x; p.nt < kT && v < n; v += blockDim.x) {              // not the padding behind the last target
        uint32_t w[W];
        R::load(cur, v, w);
#pragma unroll
        for (int k = 0; k < W; ++k) w[k] &= full[k];
        R::store(cur, v, w);
    }
    for (int round = 0;; ++round) {
        if (round % kJumpEvery == 0) start_jumps(jump, p.rows, p.cols, p.node0, n, round / kJumpEvery);
        if (round == p.components) {
            if (threadIdx.x == 0) s_found = p.found ? ld_acquire(p.found) : 0u;
            __syncthreads();
            if (s_found) {
                for (int v = threadIdx.x; v < n; v += blockDim.x) up[v] = __ldcg(&p.component[v]);
                __syncthreads();
            } else {
                find_components(up, p.rows, p.cols, p.node0, n);
                if (p.found) {                             // (several blocks may leave the same numbers)
                    for (int v = threadIdx.x; v < n; v += blockDim.x) __stcg(&p.component[v], up[v]);
                    __threadfence();
                    __syncthreads();
                    if (threadIdx.x == 0) st_release(p.found, 1u);
                }
            }
        }
        shortcuts<kT>(cur, round >= p.components && (round - p.components) % kMergeEvery == 0 ? up : nullptr, round % kJumpEvery < kJumpRounds ? jump : nullptr, n);
        if (threadIdx.x < 32) close_targets<kT>(cur, s_to, p.nt, full, (int)threadIdx.x);
        __syncthreads();
        for (int v = threadIdx.x; v < n; v += blockDim.x)
            if ((unsigned)(v - p.t0) >= (unsigned)p.nt) inherit<kT>(cur, v, s_to);
        __syncthreads();
        uint32_t gained = 0u;
        for_edges(p.rows, p.cols, p.node0, n, [&](int v, int u, bool) {
            uint32_t mine[W], other[W];
            R::load(cur, v, mine);
            R::load(cur, u, other);
#pragma unroll
            for (int k = 0; k < W; ++k) {
                if (other[k] & ~mine[k]) atomicOr((uint32_t*)cur + v * W + k, other[k]);
                gained |= other[k] & ~mine[k];
            }
        });
        if (!__syncthreads_or(gained != 0u)) break;
    }
    for (int at = threadIdx.x; at < n * W; at += blockDim.x) {
        const uint32_t w = ((const uint32_t*)cur)[at];
        uint32_t o[8], any = 0u;
        bytes_of(at, o);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const uint32_t far = __vcmpeq4(o[b], none4) & ((w >> b) & 0x01010101u);
            o[b] -= far;
            any |= far;
        }
        if (any) store_row_piece_anywhere(p.out + (int64_t)(at / W) * p.ld + 32 * (at % W), o, (int)min(p.ld - p.t0 - 32 * (at % W), (int64_t)32));
    }
    __syncthreads();
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
    store_row_piece_anywhere(row, o, cols - col);
}

}  // namespace gt
