// gt_spd_build for graphs of up to about 5 000 nodes: reachability rows in shared memory, pulled along out-edges.
//
// A thread block owns kT target columns [t0, t0+kT) of one graph.  Row v is a bit set: which of those targets vertex v
// reaches within l hops.  One level is
//     V_{l+1}[v] = V_l[v] | OR over out-neighbours u of v of V_l[u]
// with the two states in shared memory and a thread per vertex (a warp per vertex with many out-edges): plain loads and
// ORs, no atomics, one barrier per level, and no output traffic until the end.  The level at which a bit appears goes
// into bit-sliced code planes (plane b holds bit b of the distance), also in shared memory; when the search ends a thread
// turns a vertex' planes into kT output bytes and writes them as whole 32-byte sectors of row v.  Directed graphs need
// no transposed edge list, because the block owns columns.
//
// Pairs at max_dist or farther share one code, so exact levels stop at max_dist - 1 and only reachability is left.  It is
// completed by in-place passes over the rows, sped up by closing the block's targets under each other: target t's own row
// says which targets follow from t, so after a transitive closure of those kT rows every vertex inherits the closed row of
// each target it reaches.  That only adds what is reachable, and the passes run until one changes nothing, so it is exact
// for any directed graph.  What is still open after kPlainRounds of them (graphs hundreds of edges across) is left to finish_far.
//
// What bounds it: the shared-memory pipe in the level passes (a gathered row costs the bank conflicts of 32 random rows:
// 3.5 wavefronts for 32 lanes of 4 bytes, 6.2 of 8, 10.6 of 16: wider rows cost less per target), and the pipe of logic and
// shifts, which has half the rate, in the edge lists' making and in the output.  One graph of 4 096 nodes, clocks of a block:
// order and lists 19k, state 4k, five passes 39k, output 13k of 79k.  The lists' offsets by all warps, groups of vertices in turns that
// go back and forth (they come by falling degree), lanes of finished vertices left out, and no work on planes and codes that a graph
// does not have: 41.1 -> 38.4 us, a packed batch of 64 graphs of 512 to 2 048 nodes 291 -> 278 us.
#include "spd_pull.cuh"

namespace gt {
namespace {

constexpr int kSorted = 256;           // batches of up to this many graphs are worked on by falling size
constexpr int kBins = 66;              // hubs, then degrees 64 .. 0
constexpr uint16_t kListed = 0x8000;   // vertices are numbered below this
// Vertices with more out-edges than this are pulled by a whole warp: some 150 instructions each, where 32 of them side by side
// in one group cost 100 and 8 per pair of edges (a limit of 32: 11.4k clocks a level at 4 096 nodes, issue bound).
constexpr int kHubDegree = 64;

// Rounds of the search for what is farther than max_dist, after which finish_far takes over, and its rounds before it asks for the components.
constexpr int kPlainRounds = 40, kFarComponents = 8;

struct PullParams {
    const int32_t* row_ptr;
    const int32_t* col_idx;
    const int32_t* cu_seqlens;         // nullptr: single graph
    const int64_t* spd_offsets;        // nullptr: single graph at offset 0
    uint8_t* spd;
    int32_t n_total;
    int32_t n_graphs;
    int32_t max_dist;
    int32_t n_planes;                  // bits of the largest code, max_dist + 1
    uint32_t smem_bytes;
};

template <int kT>
__global__ void __launch_bounds__(1024, 1) spd_pull_kernel(PullParams p)
{
    using R = Rows<kT>;
    constexpr int W = R::kWords;
    // Rows of one word stay in the vertices' order: a vertex' own row is then read out of order, which costs less than looking
    // up every edge's position.  Wider rows lie by position (their out-of-order accesses cost 6 or 11 wavefronts, not 3.5).
    constexpr bool kByPosition = W > 1;
    extern __shared__ __align__(16) uint8_t pull_smem[];
    __shared__ int s_graph, s_node0, s_n, s_first, s_list_words, s_bin[kBins];
    int* s_cu = (int*)pull_smem;             // before the rows
    __shared__ uint32_t s_live[3];
    __shared__ uint16_t s_tpos[kT];          // position of target t
    __shared__ int s_words[33];              // list words of the hubs, then of every warp's groups

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    grid_wait();
    grid_release();
    // Which targets of which graph?  In a batch of up to kSorted graphs the larger graphs come first (their blocks take
    // longer, and the last wave is short then): a graph's first block is the number of blocks of all graphs before it in
    // that order.  In a batch of more, graph g owns the blocks from cu[g]/kT + g up to the next graph's first, at least
    // ceil(n_g/kT) of them.  Either way nothing has to be computed beforehand; a block past the last target has no work.
    int32_t node0 = 0, n = p.n_total;
    int g = 0, t0 = (int)blockIdx.x * kT;
    if (p.cu_seqlens) {
        const int me = (int)blockIdx.x;
        if (threadIdx.x == 0) { s_graph = 0; s_node0 = 0; s_n = 0; s_first = 0; }
        if (p.n_graphs <= kSorted) {
            for (int i = threadIdx.x; i <= p.n_graphs; i += blockDim.x) s_cu[i] = p.cu_seqlens[i];
            __syncthreads();
            for (int i = warp; i < p.n_graphs; i += n_warps) {           // a warp per graph
                const int size = s_cu[i + 1] - s_cu[i], blocks = (size + kT - 1) / kT;
                int first = 0;
                for (int j = lane; j < p.n_graphs; j += 32) {
                    const int other = s_cu[j + 1] - s_cu[j];
                    first += other > size || (other == size && j < i) ? (other + kT - 1) / kT : 0;
                }
                first = __reduce_add_sync(0xffffffffu, first);
                if (me >= first && me < first + blocks && lane == 0) { s_graph = i; s_n = size; s_first = first; s_node0 = s_cu[i]; }
            }
        } else {
            __syncthreads();
            for (int i = threadIdx.x; i < p.n_graphs; i += blockDim.x) {
                const int32_t c0 = p.cu_seqlens[i], c1 = p.cu_seqlens[i + 1];
                if (me >= c0 / kT + i && me < c1 / kT + i + 1) { s_graph = i; s_node0 = c0; s_n = c1 - c0; s_first = c0 / kT + i; }
            }
        }
        __syncthreads();
        g = s_graph; node0 = s_node0; n = s_n;
        t0 = (me - s_first) * kT;
    }
    if (t0 >= n) return;
    const int nt = min(kT, n - t0);
    const int32_t* __restrict__ grp = p.row_ptr + node0;
    const int32_t e_base = grp[0];
    const int nnz = grp[n] - e_base;

    const uint32_t row_bytes = (uint32_t)pull_align((size_t)n * R::kBytes);
    uint8_t* cur = pull_smem;
    uint8_t* nxt = cur + row_bytes;
    uint8_t* planes = nxt + row_bytes;
    uint16_t* order = (uint16_t*)(planes + (size_t)p.n_planes * row_bytes);          // vertex at position i (and kListed)
    uint32_t* ginfo = (uint32_t*)((uint8_t*)order + pull_align(2 * (size_t)n));       // per group of 32 positions: list << 6 | pairs
    uint32_t* hub_at = ginfo + pull_align(4 * (size_t)(n / 32 + 1)) / 4;               // staged: word at which a hub's list starts; else: the hubs
    const uint32_t used = (uint32_t)((uint8_t*)hub_at - pull_smem);
    // The edge list with 16-bit positions goes to shared memory where it fits behind the state; while it is laid out, the
    // columns and the row offsets are staged in the space of the second state and the planes.
    const uint32_t spare = (uint32_t)(1 + p.n_planes) * row_bytes;
    bool staged = nnz < 65536 && used + 2u * (uint32_t)nnz <= p.smem_bytes && 4u * (uint32_t)n + 2u * (uint32_t)nnz + 64u <= spare;

    uint32_t full[W];
#pragma unroll
    for (int k = 0; k < W; ++k) full[k] = nt == kT ? 0xffffffffu : 0u;
    for (int t = 0; t < nt && nt < kT; ++t) R::add_target(t, nt, full);

    if (threadIdx.x < kBins) s_bin[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_live[0] = 0u;
    __syncthreads();
    int n_hubs = 0;
    uint32_t* list = hub_at;                           // edge lists, behind hub_at
    uint16_t* pos = (uint16_t*)nxt;                    // position of vertex v (kByPosition)
    uint16_t* eoff = pos + (kByPosition ? (n + 7) & ~7 : 0);             // first edge of vertex v
    const int skew = (int)(((uintptr_t)(p.col_idx + e_base) >> 2) & 3u);
    uint16_t* raw = eoff + ((n + 8) & ~7) + skew;      // columns (original ids), placed as the caller's list is in its vectors
    if (staged) {
        // ---- positions by falling degree: the 32 vertices of a group have (nearly) the same number of edges ----
        uint32_t* key = (uint32_t*)cur;                // dead before the rows are written
        {
            const int32_t* cols = p.col_idx + e_base;
            const int n_vec = nnz > 0 ? (skew + nnz + 3) / 4 : 0;     // aligned 16-byte vectors; ragged ends one by one
            for (int v0 = threadIdx.x; v0 <= n; v0 += 4 * blockDim.x) {
                int32_t e[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) e[i] = grp[min(v0 + i * (int)blockDim.x, n)];
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (v0 + i * (int)blockDim.x <= n) eoff[v0 + i * (int)blockDim.x] = (uint16_t)(e[i] - e_base);
            }
            for (int j0 = threadIdx.x; j0 < n_vec; j0 += 4 * blockDim.x) {
                int4 c[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int e = 4 * (j0 + i * (int)blockDim.x) - skew;
                    c[i] = make_int4(node0, node0, node0, node0);
                    if (e >= 0 && e + 4 <= nnz) c[i] = *(const int4*)(cols + e);
                    else {
                        if (e >= 0 && e < nnz) c[i].x = cols[e];
                        if (e + 1 >= 0 && e + 1 < nnz) c[i].y = cols[e + 1];
                        if (e + 2 >= 0 && e + 2 < nnz) c[i].z = cols[e + 2];
                        if (e + 3 >= 0 && e + 3 < nnz) c[i].w = cols[e + 3];
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int j = j0 + i * (int)blockDim.x;
                    if (j < n_vec)
                        ((uint2*)(raw - skew))[j] = make_uint2((uint32_t)(c[i].x - node0) | (uint32_t)(c[i].y - node0) << 16,
                                                               (uint32_t)(c[i].z - node0) | (uint32_t)(c[i].w - node0) << 16);
                }
            }
        }
        __syncthreads();
        for (int v0 = warp * 32; v0 < n; v0 += blockDim.x) {
            const int v = v0 + lane;
            const int deg = v < n ? (int)eoff[v + 1] - (int)eoff[v] : 0;
            const int bin = v < n ? (deg > kHubDegree ? 0 : 1 + kHubDegree - deg) : kBins;
            const uint32_t peers = __match_any_sync(0xffffffffu, bin);
            const int leader = __ffs((int)peers) - 1;
            int rank = 0;
            if (lane == leader && v < n) rank = atomicAdd(&s_bin[bin], __popc(peers));
            rank = __shfl_sync(0xffffffffu, rank, leader) + __popc(peers & ((1u << lane) - 1u));
            if (v < n) key[v] = (uint32_t)bin << 16 | (uint32_t)rank;
        }
        __syncthreads();
        if (warp == 0) {                              // exclusive scan of the bins
            int carry = 0;
            for (int b = 0; b < kBins; b += 32) {
                const int cnt = b + lane < kBins ? s_bin[b + lane] : 0;
                const int x = warp_scan(cnt, lane);
                if (b + lane < kBins) s_bin[b + lane] = carry + x - cnt;
                carry += __shfl_sync(0xffffffffu, x, 31);
            }
        }
        __syncthreads();
        n_hubs = s_bin[1];
        list = hub_at + ((n_hubs + 4) & ~3);
        for (int v = threadIdx.x; v < n; v += blockDim.x) {
            const uint32_t k = key[v];
            const int i = s_bin[k >> 16] + (int)(k & 0xffffu);
            if (kByPosition) pos[v] = (uint16_t)i;
            order[i] = (uint16_t)v;
        }
        __syncthreads();
        // ---- edge lists: hubs first (contiguous), then groups of 32 vertices with edge pair j of lane l at word 32 j + l ----
        const int groups = (n - n_hubs + 31) / 32;
        // A warp adds up the words of its 32 groups; beyond 32 groups everyone then adds what comes before, the hubs' words first.
        const int gq = 32 * warp + lane, gi = n_hubs + 32 * gq;
        const int gv = gi < n ? order[gi] : 0;
        const int pairs = gi < n ? ((int)eoff[gv + 1] - (int)eoff[gv] + 1) / 2 : 0;
        const int through = warp_scan(32 * pairs, lane);
        int before = through - 32 * pairs;
        if (warp == 0) {
            int at = 0;                                // in words
            for (int h = 0; h < n_hubs; h += 32) {
                const int v = h + lane < n_hubs ? order[h + lane] : 0;
                const int words = h + lane < n_hubs ? ((int)eoff[v + 1] - (int)eoff[v] + 1) / 2 : 0;
                const int x = warp_scan(words, lane);
                if (h + lane < n_hubs) hub_at[h + lane] = (uint32_t)(at + x - words);
                at += __shfl_sync(0xffffffffu, x, 31);
            }
            if (lane == 0) { hub_at[n_hubs] = (uint32_t)at; s_words[0] = at; }
            if (groups <= 32) {
                before += at;
                if (lane == 31) s_list_words = at + through;
            }
        }
        if (groups > 32) {
            if (lane == 31) s_words[warp + 1] = through;
            __syncthreads();
            const int others = lane <= n_warps ? s_words[lane] : 0;
            before += __reduce_add_sync(0xffffffffu, lane <= warp ? others : 0);
            if (threadIdx.x < 32) {
                const int all = __reduce_add_sync(0xffffffffu, others) + (n_warps == 32 ? s_words[32] : 0);
                if (lane == 0) s_list_words = all;
            }
        }
        if (gi < n) ginfo[gq] = (uint32_t)before << 6 | (uint32_t)pairs;
        __syncthreads();
        staged = used + 4u * (uint32_t)(((n_hubs + 4) & ~3) + s_list_words) <= p.smem_bytes;
    }
    if (staged) {
        // Fill them from the staged columns; a vertex' own position fills up.  The columns are still original ids here, so
        // the state after the first level comes with it.
        for (int h = warp; h < n_hubs; h += n_warps) {
            const int v = order[h];
            const int e0 = eoff[v], deg = (int)eoff[v + 1] - e0;
            uint16_t* dst = (uint16_t*)(list + hub_at[h]);
            uint32_t w[W];
#pragma unroll
            for (int k = 0; k < W; ++k) w[k] = 0u;
            for (int i = lane; i < ((deg + 1) & ~1); i += 32) {
                const int u = i < deg ? raw[e0 + i] : v;
                dst[i] = kByPosition ? pos[u] : (uint16_t)u;
                R::add_target(u - t0, nt, w);
            }
            R::add_target(v - t0, nt, w);
#pragma unroll
            for (int k = 0; k < W; ++k) w[k] = __reduce_or_sync(0xffffffffu, w[k]);
            if (lane == 0) R::store(cur, kByPosition ? h : v, w);
        }
        // (Groups come by falling degree: the warps take them in turns that go back and forth.)
        for (int q = warp, step = 2 * (n_warps - warp) - 1; n_hubs + 32 * q < n; q += step, step = 2 * n_warps - step) {
            const int i = n_hubs + 32 * q + lane;
            const int v = order[min(i, n - 1)];
            const int e0 = eoff[v], deg = i < n ? (int)eoff[v + 1] - e0 : 0;
            const uint32_t info = ginfo[q];
            uint32_t* dst = list + (info >> 6) + lane;
            uint32_t w[W];
#pragma unroll
            for (int k = 0; k < W; ++k) w[k] = 0u;
            R::add_target(v - t0, nt, w);
            for (int j = 0; j < (int)(info & 63u); ++j) {
                const int u0 = 2 * j < deg ? raw[e0 + 2 * j] : v, u1 = 2 * j + 1 < deg ? raw[e0 + 2 * j + 1] : v;
                dst[32 * j] = kByPosition ? (uint32_t)pos[u0] | (uint32_t)pos[u1] << 16 : (uint32_t)u0 | (uint32_t)u1 << 16;
                R::add_target(u0 - t0, nt, w);
                R::add_target(u1 - t0, nt, w);
            }
            if (i < n) R::store(cur, kByPosition ? i : v, w);
        }
        for (int t = threadIdx.x; t < nt; t += blockDim.x) s_tpos[t] = kByPosition ? pos[t0 + t] : (uint16_t)(t0 + t);
        __syncthreads();
    } else {                                           // the caller's list in place, vertices in their own order
        const int hub_cap = (int)((p.smem_bytes - used) / 4u);
        __syncthreads();
        if (threadIdx.x == 0) s_bin[0] = 0;
        __syncthreads();
        for (int v = threadIdx.x; v < n; v += blockDim.x) {
            uint32_t w[W];
#pragma unroll
            for (int k = 0; k < W; ++k) w[k] = 0u;
            R::add_target(v - t0, nt, w);
            R::store(cur, v, w);
            uint16_t mark = 0;
            if (grp[v + 1] - grp[v] > kHubDegree) {    // a hub for a warp, if there is room to list it
                const int at = atomicAdd(&s_bin[0], 1);
                if (at < hub_cap) { hub_at[at] = (uint32_t)v; mark = kListed; }
            }
            order[v] = (uint16_t)v | mark;
        }
        for (int t = threadIdx.x; t < nt; t += blockDim.x) s_tpos[t] = (uint16_t)(t0 + t);
        __syncthreads();
        n_hubs = min(s_bin[0], hub_cap);
    }
    const int group0 = staged ? n_hubs : 0;            // first position that belongs to a group
    const int n_groups = (n - group0 + 31) / 32;
    for (uint32_t i = threadIdx.x; i < (uint32_t)p.n_planes * row_bytes / 16; i += blockDim.x) ((uint4*)planes)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (staged) {                                      // plane 0 holds the pairs at distance 1
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            uint32_t w[W], self[W];
            R::load(cur, kByPosition ? i : (int)order[i], w);
#pragma unroll
            for (int k = 0; k < W; ++k) self[k] = 0u;
            R::add_target((int)order[i] - t0, nt, self);
#pragma unroll
            for (int k = 0; k < W; ++k) w[k] &= ~self[k];
            R::store(planes, i, w);
        }
    }
    __syncthreads();

    auto row_of = [&](int i) -> int { return kByPosition ? i : order[i] & (kListed - 1); };        // of position i
    // bits that position i gained at level `code`: into the code planes
    auto note = [&](int i, const uint32_t (&old)[W], const uint32_t (&acc)[W], int code) {
        uint32_t fresh[W], any = 0u;
#pragma unroll
        for (int k = 0; k < W; ++k) { fresh[k] = acc[k] & ~old[k]; any |= fresh[k]; }
        if (any == 0u) return;
        for (int b = 0; (code >> b) != 0; ++b) {
            if (!((code >> b) & 1)) continue;
            uint32_t c[W];
            uint8_t* plane = planes + (size_t)b * row_bytes;
            R::load(plane, i, c);
#pragma unroll
            for (int k = 0; k < W; ++k) c[k] |= fresh[k];
            R::store(plane, i, c);
        }
    };
    // One pass from `src` to `dst` (the same rows: a pass of the reachability phase, code 0).  With one word per row it leaves
    // in `live` the targets that some row has gained: where none has, that target's search is over, so rows that miss only
    // such targets are done (targets in small components would otherwise keep every row open to the last level).  The wider
    // rows are used on batches of small graphs, where that gains less than the registers for it cost.
    uint32_t live[W];
#pragma unroll
    for (int k = 0; k < W; ++k) live[k] = full[k];
    int turn = 0;
    auto pass = [&](const uint8_t* src, uint8_t* dst, int code) {
        uint32_t gained = 0u;
        for (int h = warp; h < n_hubs; h += n_warps) {
            const int i = staged ? h : (int)hub_at[h];
            const int own_row = row_of(i);
            uint32_t old[W], acc[W];
            R::load(src, own_row, old);
            uint32_t miss = 0u;
#pragma unroll
            for (int k = 0; k < W; ++k) { acc[k] = old[k]; miss |= live[k] & ~old[k]; }
            if (miss != 0u) {
                const uint16_t* mine = (const uint16_t*)(list + (staged ? hub_at[h] : 0));
                const int e0 = staged ? 0 : grp[i], len = staged ? 2 * (int)(hub_at[h + 1] - hub_at[h]) : grp[i + 1] - e0;
                for (int e = lane; e < len; e += 32) {
                    const int u = staged ? (int)mine[e] : p.col_idx[e0 + e] - node0;
                    uint32_t x[W];
                    R::load(src, u, x);
#pragma unroll
                    for (int k = 0; k < W; ++k) acc[k] |= x[k];
                }
#pragma unroll
                for (int k = 0; k < W; ++k) acc[k] = __reduce_or_sync(0xffffffffu, acc[k]);
            }
            if (lane == 0) {
                note(i, old, acc, code);
#pragma unroll
                for (int k = 0; k < W; ++k) gained |= acc[k] & ~old[k];
                R::store(dst, own_row, acc);
            }
        }
        for (int q = warp, step = 2 * (n_warps - warp) - 1; q < n_groups; q += step, step = 2 * n_warps - step) {
            const int i = group0 + 32 * q + lane;
            uint32_t old[W], acc[W];
            const int own_row = row_of(min(i, n - 1));
            R::load(src, own_row, old);
            uint32_t miss = 0u;
#pragma unroll
            for (int k = 0; k < W; ++k) { acc[k] = old[k]; miss |= live[k] & ~old[k]; }
            bool own = i < n;
            if (staged) {
                if (miss != 0u && own) {
                    const uint32_t info = ginfo[q];
                    const uint32_t* mine = list + (info >> 6) + lane;
                    constexpr int kPairs = W == 4 ? 2 : 4;         // 4 or 8 rows in flight
                    int left = (int)(info & 63u);
                    for (; left >= kPairs; left -= kPairs, mine += 32 * kPairs) {
                        uint32_t u[kPairs], x[2 * kPairs][W];
#pragma unroll
                        for (int j = 0; j < kPairs; ++j) u[j] = mine[32 * j];
#pragma unroll
                        for (int j = 0; j < kPairs; ++j) { R::load(src, (int)(u[j] & 0xffffu), x[2 * j]); R::load(src, (int)(u[j] >> 16), x[2 * j + 1]); }
#pragma unroll
                        for (int j = 0; j < 2 * kPairs; ++j)
#pragma unroll
                            for (int k = 0; k < W; ++k) acc[k] |= x[j][k];
                    }
                    for (; left > 0; --left, mine += 32) {
                        const uint32_t u = mine[0];
                        uint32_t x[W], y[W];
                        R::load(src, (int)(u & 0xffffu), x);
                        R::load(src, (int)(u >> 16), y);
#pragma unroll
                        for (int k = 0; k < W; ++k) acc[k] |= x[k] | y[k];
                    }
                }
            } else if (own) {
                const int e1 = grp[i + 1];
                int e = grp[i];
                own = !(order[i] & kListed);                       // listed hubs: above
                if (own && miss != 0u) {
                    for (; e + 4 <= e1; e += 4) {
                        int u[4];
                        uint32_t x[4][W];
#pragma unroll
                        for (int j = 0; j < 4; ++j) u[j] = p.col_idx[e + j] - node0;
#pragma unroll
                        for (int j = 0; j < 4; ++j) R::load(src, u[j], x[j]);
#pragma unroll
                        for (int k = 0; k < W; ++k) acc[k] |= x[0][k] | x[1][k] | x[2][k] | x[3][k];
                    }
                    for (; e < e1; ++e) {
                        uint32_t x[W];
                        R::load(src, p.col_idx[e] - node0, x);
#pragma unroll
                        for (int k = 0; k < W; ++k) acc[k] |= x[k];
                    }
                }
            }
            if (own) {
                note(i, old, acc, code);
#pragma unroll
                for (int k = 0; k < W; ++k) gained |= acc[k] & ~old[k];
                R::store(dst, own_row, acc);
            }
        }
        if constexpr (W == 1) {
            if (threadIdx.x == 0) s_live[(turn + 1) % 3] = 0u;               // for the next pass; last read two passes ago
            gained = __reduce_or_sync(0xffffffffu, gained);
            if (lane == 0 && gained) atomicOr(&s_live[turn], gained);
            __syncthreads();
            live[0] = s_live[turn];
            turn = (turn + 1) % 3;
            return live[0] != 0u;
        } else {
            return __syncthreads_or(gained != 0u) != 0;
        }
    };

    bool open = true;                       // some row may still grow
    for (int level = staged ? 2 : 1; level < p.max_dist && open; ++level) {
        open = pass(cur, nxt, level);
        uint8_t* t = cur; cur = nxt; nxt = t;
    }
    for (int round = 0; round < kPlainRounds && open; ++round) {
        if (warp == 0) close_targets<kT>(cur, s_tpos, nt, full, lane);
        __syncthreads();
        // every vertex inherits the rows of the targets it reaches; a closed row covers all targets inside it
        for (int v = threadIdx.x; v < n; v += blockDim.x)
            if ((unsigned)((kByPosition ? order[v] & (kListed - 1) : v) - t0) >= (unsigned)nt) inherit<kT>(cur, v, s_tpos);
        __syncthreads();
        open = pass(cur, cur, 0);
    }

    // ---- output: the planes and the final rows as bytes ----
    const int64_t ld = (int64_t)((n + 15) & ~15);
    uint8_t* out = p.spd + (p.spd_offsets ? p.spd_offsets[g] : 0) + t0;
    const uint32_t far_code = (uint32_t)p.max_dist, none_code = (uint32_t)p.max_dist + 1u;
    const int cols = (int)min((int64_t)kT, ld - t0);             // columns of this block inside the pitch
    // A thread turns one word of a row (32 targets) into 32 bytes; the W words of a row go to neighbouring lanes, so that a
    // warp's store covers whole pieces of 32 W bytes.
    for (int at = threadIdx.x; at < n * W; at += blockDim.x) {
        const int i = at / W, k = at % W;
        const int v = order[i] & (kListed - 1);
        const int col = 32 * k;
        if (col >= cols) continue;
        uint8_t* row = out + (int64_t)v * ld + col;
        const int self = v - t0 - col;
        auto word = [&](const uint8_t* rows) -> uint32_t { return ((const uint32_t*)rows)[at]; };
        const uint32_t reach = kByPosition ? word(cur) : ((const uint32_t*)cur)[v];
        uint32_t seen = (unsigned)self < 32u ? 1u << R::bit(self) : 0u;
        uint32_t c[8];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            c[b] = b < p.n_planes ? word(planes + (size_t)b * row_bytes) : 0u;
            seen |= c[b];
            c[b + 4] = 0u;
        }
        if (p.n_planes > 4) {
#pragma unroll
            for (int b = 4; b < 8; ++b) {
                c[b] = b < p.n_planes ? word(planes + (size_t)b * row_bytes) : 0u;
                seen |= c[b];
            }
        }
        const uint32_t far = reach & ~seen, none = ~reach;
        if (far | none) {
#pragma unroll
            for (int b = 0; b < 8; ++b)
                if (b < 4 || p.n_planes > 4) c[b] |= (far & (0u - ((far_code >> b) & 1u))) | (none & (0u - ((none_code >> b) & 1u)));
        }
        emit_word(c, (c[4] | c[5] | c[6] | c[7]) != 0u ? 8 : 4, row, col, nt, cols);
    }
    if (open) {
        __shared__ FarState s_far;
        __syncthreads();
        if (threadIdx.x == 0) s_far = {out, ld, grp, p.col_idx, nullptr, nullptr, node0, n, t0, nt, none_code, kFarComponents};
        __syncthreads();
        finish_far<kT>(pull_smem, s_far);
    }
}

size_t pull_state_bytes(int targets, int32_t n, int planes)
{
    return pull_align((size_t)n * targets / 8) * (size_t)(2 + planes) + pull_align(2 * (size_t)n) + pull_align(4 * (size_t)(n / 32 + 1)) + 64;
}

template <int kT>
gt_status launch(const PullParams& p, const PullPlan& pl, cudaStream_t s)
{
    static std::atomic<uint64_t> granted{0};
    const gt_status st = grant_smem(spd_pull_kernel<kT>, granted, kPullSmemLimit);
    if (st != GT_OK) return st;
    return launch_overlapped(spd_pull_kernel<kT>, dim3(pl.blocks), (unsigned)pl.threads, pl.smem_bytes, s, p);
}

}  // namespace

PullPlan spd_pull_plan(const gt_batch* b, int64_t nnz, int32_t max_dist)
{
    PullPlan pl{};
    const int32_t n = b->max_seqlen;
    if (n >= kListed) return pl;
    const int planes = pull_planes(max_dist);
    // Edges of the largest graph: known for a single graph, else taken from the batch's average degree (a graph whose list
    // turns out not to fit is read in place).
    const int64_t edges = b->n_graphs == 1 ? nnz : (int64_t)((double)nnz / b->n_total * n * 1.02) + 1;
    const int64_t hubs = edges / (kHubDegree + 1) < n ? edges / (kHubDegree + 1) : n;
    const size_t list = 4 * (size_t)(hubs + 4) + 2 * ((size_t)edges + (b->n_graphs == 1 ? (size_t)n + 2112 : (size_t)n / 2 + 448));
    // Wider rows cost less per target (wavefronts above), narrower ones give more thread blocks: 128 and 64 targets are taken
    // while they leave two blocks per SM.
    for (int t = 128; t >= 32 && !pl.fits; t >>= 1) {
        const size_t state = pull_state_bytes(t, n, planes);
        if (state + list > kPullSmemLimit || (t > 32 && b->n_total / t < 2 * sm_count())) continue;
        pl.fits = true;
        pl.targets = t;
        pl.threads = n <= 256 ? 256 : (n <= 1024 ? 512 : 1024);
        pl.blocks = b->n_graphs == 1 ? (unsigned)((n + t - 1) / t) : (unsigned)(b->n_total / t + b->n_graphs);
        pl.smem_bytes = state + list < 2048 ? 2048 : state + list;       // (up to kSorted graphs are sorted by size there)
    }
    return pl;
}

gt_status spd_pull_launch(const PullPlan& pl, const int32_t* row_ptr, const int32_t* col_idx, const int32_t* cu_seqlens,
                          const int64_t* spd_offsets, const gt_batch* batch, int32_t max_dist, uint8_t* spd, cudaStream_t s)
{
    PullParams p{};
    p.row_ptr = row_ptr;
    p.col_idx = col_idx;
    p.cu_seqlens = cu_seqlens;
    p.spd_offsets = spd_offsets;
    p.spd = spd;
    p.n_total = batch->n_total;
    p.n_graphs = batch->n_graphs;
    p.max_dist = max_dist;
    p.n_planes = pull_planes(max_dist);
    p.smem_bytes = (uint32_t)pl.smem_bytes;
    switch (pl.targets) {
        case 128: return launch<128>(p, pl, s);
        case 64: return launch<64>(p, pl, s);
        default: return launch<32>(p, pl, s);
    }
}

}  // namespace gt
