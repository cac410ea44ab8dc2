// gt_spd_build for a single graph whose reachability rows fit shared memory but whose edge list does not (about 5 000 to
// 19 000 nodes): the pull of spd_pull.cu with the edge list and the code planes in the workspace.
//
// Two small kernels sort the vertices by degree and lay the edge list out once for all thread blocks: groups of 32 vertices
// of (nearly) equal degree with their edges interleaved, 16-bit vertex numbers in pairs, so that a warp reads 128 coalesced
// bytes for 64 edges; vertices with many edges follow one after the other and are pulled by a whole warp.  Then a thread
// block per 32 target columns (persistent, two blocks per SM where the rows leave room) runs the levels.  Level 1 needs no
// rows: an edge whose head lies in the block is the pair.  The code planes are read and written where they are first needed
// only (level 1, 2, 4, .. open a plane) and by the lane that owns the vertex, coalesced, from L2.
//
// What bounds it: the issue slots (some hundred instructions per group of 32 vertices besides those of its edges), then the
// bank conflicts of the row gathers, 3.5 wavefronts for 32 edges (spd_pull.cu).  Power-law
// graphs of degree 12 against the frontier push that served them before: 12 000 nodes 915 -> 417 us, 14 400 nodes 1 395 ->
// 632 us; against the bit-matrix build 16 384 nodes 920 -> 738 us; a graph of degree 10 and 8 192 nodes 374 -> 163 us.
#include <type_traits>

#include "spd_pull.cuh"

namespace gt {
namespace {

constexpr int kLargeHubDegree = 126;
constexpr int kLargeBins = 128;            // hubs, then degrees 126 .. 0
constexpr size_t kLargeSmemLimit = 222 * 1024;      // and 3 KB of static arrays
constexpr int kTargets = 32;
// Beyond this the bit-matrix build is the faster one (power law, degree 12: 18 000 nodes 0.85 against 0.91 ms, 20 000 nodes
// 1.13 against 1.04 ms; from 592 blocks of targets on there is a fifth round); the row sets would fit up to 28 000 nodes.
constexpr int32_t kLargeMaxNodes = 18944;
// Many edges per vertex: beyond kDenseDegree the bit matrices are the faster ones where they are the alternative (Erdos-Renyi / power law:
// 16 000 nodes, degree 25 687 against 778 us / 804 against 710, degree 50 974 against 822 / 1 140 against 680; 18 900 nodes, degree
// 50 1 223 against 1 282 / 1 370 against 976); where the push is, beyond kLargeHubDegree, when every vertex is pulled by a warp (9 000
// nodes, degree 100 400 against 933 us, degree 200 1 767 against 1 267).
constexpr int kDenseDegree = 32;
constexpr int kCachedHubs = 400;           // hubs whose numbers and lists' places are kept in shared memory

constexpr int kPlainRounds = 3, kFarComponents = 1;         // as in spd_pull.cu; a round takes 6 to 25 us here

struct LargeParams {
    const int32_t* row_ptr;
    const int32_t* col_idx;
    uint16_t* order;          // [n] vertex at position i (by falling degree)
    uint32_t* info;           // [n/32 + 1] per group: first word of its list << 6 | pairs of edges
    uint32_t* hub_at;         // first word of a hub's list, and one past the last hub's
    uint32_t* list;
    uint32_t* planes;         // [grid][n_planes][n_pad]
    uint32_t* counts;         // [0] hubs, [1] `component` is there
    uint16_t* component;      // [n] root of a vertex' component (finish_far), once a block has needed it
    uint8_t* spd;
    int32_t n;
    int32_t n_pad;
    int32_t max_dist;
    int32_t n_planes;
};

// Positions by falling degree, and where every list starts.  One block.
__global__ void __launch_bounds__(1024, 1) spd_large_order_kernel(LargeParams p)
{
    extern __shared__ __align__(16) uint8_t large_smem[];
    __shared__ int s_bin[kLargeBins];
    const int n = p.n, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* key = (uint32_t*)large_smem;
    uint16_t* degree = (uint16_t*)(key + n);           // of a vertex
    uint16_t* sorted = degree + n;                     // by position
    if (threadIdx.x < kLargeBins) s_bin[threadIdx.x] = 0;
    grid_wait();
    grid_release();
    for (int v0 = threadIdx.x; v0 < n; v0 += 8 * blockDim.x) {
        int32_t e0[8], e1[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int v = min(v0 + i * (int)blockDim.x, n - 1);
            e0[i] = p.row_ptr[v];
            e1[i] = p.row_ptr[v + 1];
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (v0 + i * (int)blockDim.x < n) degree[v0 + i * (int)blockDim.x] = (uint16_t)min(e1[i] - e0[i], 65535);
    }
    __syncthreads();
    for (int v0 = warp * 32; v0 < n; v0 += blockDim.x) {
        const int v = v0 + lane;
        const int deg = v < n ? degree[v] : 0;
        const int bin = v < n ? (deg > kLargeHubDegree ? 0 : 1 + kLargeHubDegree - deg) : kLargeBins;
        const uint32_t peers = __match_any_sync(0xffffffffu, bin);
        const int leader = __ffs((int)peers) - 1;
        int rank = 0;
        if (lane == leader && v < n) rank = atomicAdd(&s_bin[bin], __popc(peers));
        rank = __shfl_sync(0xffffffffu, rank, leader) + __popc(peers & ((1u << lane) - 1u));
        if (v < n) key[v] = (uint32_t)bin << 16 | (uint32_t)rank;
    }
    __syncthreads();
    if (warp == 0) {
        int carry = 0;
        for (int b = 0; b < kLargeBins; b += 32) {
            const int cnt = s_bin[b + lane], x = warp_scan(cnt, lane);
            s_bin[b + lane] = carry + x - cnt;
            carry += __shfl_sync(0xffffffffu, x, 31);
        }
    }
    __syncthreads();
    const int n_hubs = s_bin[1];
    for (int v = threadIdx.x; v < n; v += blockDim.x) {
        const uint32_t k = key[v];
        const int i = s_bin[k >> 16] + (int)(k & 0xffffu);
        p.order[i] = (uint16_t)v;
        sorted[i] = degree[v];
        if (i < n_hubs) p.hub_at[i] = (uint32_t)(p.row_ptr[v + 1] - p.row_ptr[v] + 1) / 2;      // words, for now
    }
    __syncthreads();
    if (warp == 0) {
        int at = 0;
        for (int h = 0; h < n_hubs; h += 32) {
            const int words = h + lane < n_hubs ? (int)p.hub_at[h + lane] : 0, x = warp_scan(words, lane);
            if (h + lane < n_hubs) p.hub_at[h + lane] = (uint32_t)(at + x - words);
            at += __shfl_sync(0xffffffffu, x, 31);
        }
        if (lane == 0) { p.hub_at[n_hubs] = (uint32_t)at; p.counts[0] = (uint32_t)n_hubs; p.counts[1] = 0u; }
        for (int g0 = 0; n_hubs + 32 * g0 < n; g0 += 32) {
            const int i = n_hubs + 32 * (g0 + lane);
            const int pairs = i < n ? (sorted[i] + 1) / 2 : 0, x = warp_scan(32 * pairs, lane);
            if (i < n) p.info[g0 + lane] = (uint32_t)(at + x - 32 * pairs) << 6 | (uint32_t)pairs;
            at += __shfl_sync(0xffffffffu, x, 31);
        }
    }
}

// The lists; a thread block per hub or group, so that no warp walks along many edges.  A vertex' own number fills up.
__global__ void __launch_bounds__(256) spd_large_lists_kernel(LargeParams p)
{
    grid_wait();
    grid_release();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n_hubs = (int)p.counts[0];
    int task = (int)blockIdx.x;
    if (task < n_hubs) {
        const int v = p.order[task];
        const int e0 = p.row_ptr[v], deg = p.row_ptr[v + 1] - e0;
        uint32_t* dst = p.list + p.hub_at[task];
        for (int w = threadIdx.x; 2 * w < deg; w += blockDim.x) {
            const uint32_t a = (uint32_t)p.col_idx[e0 + 2 * w], b = 2 * w + 1 < deg ? (uint32_t)p.col_idx[e0 + 2 * w + 1] : (uint32_t)v;
            dst[w] = a | b << 16;
        }
        return;
    }
    task -= n_hubs;
    const int i = n_hubs + 32 * task + lane;
    if (n_hubs + 32 * task >= p.n) return;
    const int v = p.order[min(i, p.n - 1)];
    const uint32_t info = p.info[task];
    const int e0 = p.row_ptr[v], deg = i < p.n ? p.row_ptr[v + 1] - e0 : 0;
    uint32_t* dst = p.list + (info >> 6) + lane;
    const int pairs = (int)(info & 63u);
    for (int j = warp; j < pairs; j += 8) {
        const uint32_t a = 2 * j < deg ? (uint32_t)p.col_idx[e0 + 2 * j] : (uint32_t)v;
        const uint32_t b = 2 * j + 1 < deg ? (uint32_t)p.col_idx[e0 + 2 * j + 1] : (uint32_t)v;
        dst[32 * j] = a | b << 16;
    }
}

__global__ void __launch_bounds__(1024, 1) spd_large_pull_kernel(LargeParams p)
{
    using R = Rows<kTargets>;
    extern __shared__ __align__(16) uint8_t large_smem[];
    __shared__ uint32_t s_live[3], s_hub_at[kCachedHubs + 1], s_unfinished[(kLargeMaxNodes / kTargets + 31) / 32];      // a bit per turn of the block
    __shared__ uint16_t s_tpos[kTargets], s_hub[kCachedHubs];
    grid_wait();
    grid_release();
    const int n = p.n, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const uint32_t row_words = (uint32_t)pull_align(4 * (size_t)n) / 4;
    uint32_t* const rows0 = (uint32_t*)large_smem;
    uint32_t* const rows1 = rows0 + row_words;
    uint32_t* __restrict__ planes = p.planes + (size_t)blockIdx.x * p.n_planes * p.n_pad;
    const uint16_t* __restrict__ order = p.order;
    const uint32_t* __restrict__ list = p.list;
    const int n_hubs = (int)p.counts[0];
    const int n_groups = (n - n_hubs + 31) / 32;
    const int64_t ld = (int64_t)((n + 15) & ~15);
    const uint32_t far_code = (uint32_t)p.max_dist, none_code = (uint32_t)p.max_dist + 1u;
    if (threadIdx.x < 3) s_live[threadIdx.x] = 0u;
    if (threadIdx.x < sizeof(s_unfinished) / 4) s_unfinished[threadIdx.x] = 0u;
    for (int h = threadIdx.x; h <= min(n_hubs, kCachedHubs); h += blockDim.x) {
        s_hub_at[h] = p.hub_at[h];
        if (h < min(n_hubs, kCachedHubs)) s_hub[h] = order[h];
    }
    int turn = 0;

    for (int t0 = (int)blockIdx.x * kTargets; t0 < n; t0 += (int)gridDim.x * kTargets) {
        const int nt = min(kTargets, n - t0);
        uint32_t full[1] = {0xffffffffu};
        if (nt < kTargets) {
            full[0] = 0u;
            for (int t = 0; t < nt; ++t) R::add_target(t, nt, full);
        }
        uint32_t *cur = rows0, *nxt = rows1, live = full[0];
        if (threadIdx.x < nt) s_tpos[threadIdx.x] = (uint16_t)(t0 + threadIdx.x);
        __syncthreads();                                   // the last block's rows have been written out

        // What position i gained at level `code` goes into the code planes, coalesced.  A plane is opened by the level that is
        // its bit: that level writes every position, later ones add to it with a reduction, which nothing waits for.
        auto note = [&](int i, uint32_t fresh, int code) {
            for (int b = 0; (code >> b) != 0; ++b) {
                if (!((code >> b) & 1)) continue;
                uint32_t* c = planes + (size_t)b * p.n_pad + i;
                if (code == (1 << b)) __stcg(c, fresh);
                else if (fresh) asm volatile("red.global.or.b32 [%0], %1;" ::"l"(c), "r"(fresh) : "memory");
            }
        };
        // One pass from `src` to `dst`; level 1 (code 1) goes by vertex numbers and reads no rows; code 0: reachability only.
        // Leaves in `live` the targets that some row has gained; a target without any is finished.
        auto pass = [&](auto first_level, const uint32_t* src, uint32_t* dst, int code) -> bool {
            constexpr bool by_id = decltype(first_level)::value;
            uint32_t gained = 0u;
            const bool opens = code != 0 && (code & (code - 1)) == 0;
            auto own_bit = [&](uint32_t v) -> uint32_t {
                const uint32_t t = v - (uint32_t)t0;
                return t < (uint32_t)nt ? 1u << R::bit((int)(t & 31u)) : 0u;
            };
            auto both = [&](uint32_t u) -> uint32_t {                      // the rows of a pair of edges
                if constexpr (by_id) return own_bit(u & 0xffffu) | own_bit(u >> 16);
                else return src[u & 0xffffu] | src[u >> 16];
            };
            auto own_row = [&](int v) -> uint32_t {
                if constexpr (by_id) return own_bit((uint32_t)v);
                else return src[v];
            };
            for (int h = warp; h < n_hubs; h += n_warps) {
                const bool cached = h < kCachedHubs;
                const int v = cached ? s_hub[h] : order[h];
                const uint32_t old = own_row(v);
                uint32_t acc = old;
                if (live & ~old) {
                    const int w0 = (int)(cached ? s_hub_at[h] : p.hub_at[h]), w1 = (int)(cached ? s_hub_at[h + 1] : p.hub_at[h + 1]);
                    for (int w = w0 + lane; w < w1; w += 128) {
                        uint32_t u[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) u[j] = list[min(w + 32 * j, w1 - 1)];
#pragma unroll
                        for (int j = 0; j < 4; ++j) acc |= both(u[j]);
                    }
                    acc = __reduce_or_sync(0xffffffffu, acc);
                }
                if (lane == 0) {
                    gained |= acc & ~old;
                    note(h, acc & ~old, code);
                    dst[v] = acc;
                }
            }
            // Groups, with their loads from L2 ahead of their use: vertex numbers and the list's place two groups ahead, the
            // own row (which says whether the list is wanted) and the first words of the list one group ahead, further words
            // one step ahead.
            // Groups come by falling degree: the warps take them in turns that go back and forth, beginning with the warps that have one hub
            // less.  Lanes of finished vertices read no rows (power law, degree 12, 16 384 nodes 724 -> 710 us; 8 192 of degree 10 156 -> 154).
            constexpr int kWords = 6;                                      // per step: 12 rows
            int q = n_warps - 1 - warp, step = 2 * warp + 1, v1 = 0, v2 = 0;
            uint32_t info1 = 0u, info2 = 0u, old1 = 0u, u1[kWords];
            bool want1 = false;
            auto place = [&](int qq, int& v, uint32_t& info) {
                if (qq < n_groups) { v = order[min(n_hubs + 32 * qq + lane, n - 1)]; info = p.info[qq]; }
            };
            auto first_words = [&](int qq) {
                if (qq >= n_groups) return;
                old1 = own_row(v1);
                want1 = (live & ~old1) != 0u && n_hubs + 32 * qq + lane < n;
                if (want1) {
                    const uint32_t* mine = list + (info1 >> 6) + lane;
                    const int left = (int)(info1 & 63u);
#pragma unroll
                    for (int j = 0; j < kWords; ++j)
                        if (j < left) u1[j] = mine[32 * j];
                }
            };
            place(q, v1, info1);
            place(q + step, v2, info2);
            first_words(q);
            for (; q < n_groups; q += step, step = 2 * n_warps - step) {
                const int i = n_hubs + 32 * q + lane, v = v1;
                const uint32_t old = old1;
                const bool want = want1;
                uint32_t acc = old, u[kWords];
                const uint32_t* mine = list + (info1 >> 6) + lane;
                int left = (int)(info1 & 63u);
#pragma unroll
                for (int j = 0; j < kWords; ++j) u[j] = u1[j];
                v1 = v2; info1 = info2;
                place(q + 2 * n_warps, v2, info2);
                if (want) {
                    while (left > kWords) {
                        mine += 32 * kWords;
#pragma unroll
                        for (int j = 0; j < kWords; ++j)
                            if (j < left - kWords) u1[j] = mine[32 * j];
#pragma unroll
                        for (int j = 0; j < kWords; ++j) acc |= both(u[j]);
                        left -= kWords;
#pragma unroll
                        for (int j = 0; j < kWords; ++j) u[j] = u1[j];
                    }
                }
                first_words(q + step);
                if (want) {
#pragma unroll
                    for (int j = 0; j < kWords; ++j)
                        if (j < left) acc |= both(u[j]);
                }
                if (i < n) {
                    const uint32_t fresh = acc & ~old;
                    gained |= fresh;
                    if (want || opens) note(i, fresh, code);
                    dst[v] = acc;
                }
            }
            if (threadIdx.x == 0) s_live[(turn + 1) % 3] = 0u;             // for the next pass; last read two passes ago
            gained = __reduce_or_sync(0xffffffffu, gained);
            if (lane == 0 && gained) atomicOr(&s_live[turn], gained);
            __syncthreads();
            live = s_live[turn];
            turn = (turn + 1) % 3;
            return live != 0u;
        };

        bool open = pass(std::true_type{}, nullptr, cur, 1);
        int last = 1;
        for (int level = 2; level < p.max_dist && open; ++level) {
            open = pass(std::false_type{}, cur, nxt, level);
            uint32_t* t = cur; cur = nxt; nxt = t;
            last = level;
        }
        for (int round = 0; round < kPlainRounds && open; ++round) {
            if (warp == 0) close_targets<kTargets>((uint8_t*)cur, s_tpos, nt, full, lane);
            __syncthreads();
            for (int v = threadIdx.x; v < n; v += blockDim.x)
                if ((unsigned)(v - t0) >= (unsigned)nt) inherit<kTargets>((uint8_t*)cur, v, s_tpos);
            __syncthreads();
            open = pass(std::false_type{}, cur, cur, 0);
        }
        if (open && threadIdx.x == 0) s_unfinished[t0 / kTargets / (int)gridDim.x / 32] |= 1u << (t0 / kTargets / (int)gridDim.x % 32);

        __threadfence();                                   // the reductions on the planes, before they are read
        __syncthreads();
        uint8_t* out = p.spd + t0;
        const int cols = (int)min((int64_t)kTargets, ld - t0);
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const int v = order[i];
            uint32_t c[8], seen = (unsigned)(v - t0) < (unsigned)nt ? 1u << R::bit((v - t0) & 31) : 0u;
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                c[b] = (1 << b) <= last ? __ldcg(&planes[(size_t)b * p.n_pad + i]) : 0u;
                seen |= c[b];
            }
            const uint32_t reach = cur[v], far = reach & ~seen, none = ~reach;
            if (far | none) {
#pragma unroll
                for (int b = 0; b < 8; ++b) c[b] |= (far & (0u - ((far_code >> b) & 1u))) | (none & (0u - ((none_code >> b) & 1u)));
            }
            emit_word(c, (c[4] | c[5] | c[6] | c[7]) != 0u ? 8 : 4, out + (int64_t)v * ld, 0, nt, cols);
        }
    }
    __syncthreads();
    for (int turns = 0, t0 = (int)blockIdx.x * kTargets; t0 < p.n; ++turns, t0 += (int)gridDim.x * kTargets) {
        if (!((s_unfinished[turns / 32] >> (turns % 32)) & 1u)) continue;
        __shared__ FarState s_far;
        __syncthreads();
        if (threadIdx.x == 0)
            s_far = {p.spd + t0, (int64_t)((p.n + 15) & ~15), p.row_ptr, p.col_idx, &p.counts[1], p.component, 0, p.n, t0, min(kTargets, p.n - t0),
                     (uint32_t)p.max_dist + 1u, kFarComponents};
        __syncthreads();
        finish_far<kTargets>(large_smem, s_far);
    }
}

size_t static_smem()
{
    static const size_t bytes = [] {
        cudaFuncAttributes a{};
        if (cudaFuncGetAttributes(&a, spd_large_pull_kernel) == cudaSuccess) return a.sharedSizeBytes;
        cudaGetLastError();
        return (size_t)4096;
    }();
    return bytes;
}

}  // namespace

PullLargePlan spd_pull_large_plan(const gt_batch* b, int64_t nnz, int32_t max_dist)
{
    PullLargePlan pl{};
    const size_t n = (size_t)b->n_total;
    const size_t rows = 2 * pull_align(4 * n);
    if (b->n_graphs != 1 || b->n_total > kLargeMaxNodes || nnz >= (1 << 26) || nnz > (int64_t)b->n_total * (b->n_total < kDenseMinNodes ? kLargeHubDegree : kDenseDegree)) return pl;
    pl.fits = true;
    // Two blocks of 512 threads per SM, whose phases overlap, where two pairs of row sets fit (up to 14 126 nodes), with the static
    // arrays and the 1 KB that the device keeps of a block's shared memory; else one of 1 024 (14 160 nodes, degree 12: 709 us with one
    // of 512, 555 with one of 1 024; 14 140 nodes 607 and 491).
    const bool two = 2 * (rows + static_smem() + 1024) <= 228 * 1024;
    pl.threads = two ? 512 : 1024;
    const size_t want = (size_t)sm_count() * (two ? 2 : 1), have = (n + kTargets - 1) / kTargets;
    pl.blocks = (unsigned)(have < want ? have : want);
    pl.smem_bytes = rows;
    pl.n_pad = (int32_t)align_up(n, 32);
    size_t off = kHeaderBytes;
    pl.order_off = off; off += align_up(2 * n, 256);
    pl.info_off = off; off += align_up(4 * (n / 32 + 2), 256);
    pl.hub_off = off; off += align_up(4 * ((size_t)nnz / (kLargeHubDegree + 1) + 2), 256);
    pl.list_off = off; off += align_up(2 * ((size_t)nnz + n + 32 * (kLargeHubDegree + 2)) + 256, 256);
    pl.component_off = off; off += align_up(2 * n, 256);
    pl.plane_off = off; off += 4 * (size_t)pl.blocks * (size_t)pull_planes(max_dist) * (size_t)pl.n_pad;
    pl.total_bytes = off;
    return pl;
}

gt_status spd_pull_large_launch(const PullLargePlan& pl, const int32_t* row_ptr, const int32_t* col_idx, int64_t nnz,
                                const gt_batch* batch, int32_t max_dist, uint8_t* spd, void* workspace, cudaStream_t s)
{
    uint8_t* ws = (uint8_t*)workspace;
    LargeParams p{};
    p.row_ptr = row_ptr;
    p.col_idx = col_idx;
    p.order = (uint16_t*)(ws + pl.order_off);
    p.info = (uint32_t*)(ws + pl.info_off);
    p.hub_at = (uint32_t*)(ws + pl.hub_off);
    p.list = (uint32_t*)(ws + pl.list_off);
    p.planes = (uint32_t*)(ws + pl.plane_off);
    p.counts = (uint32_t*)ws + 4;
    p.component = (uint16_t*)(ws + pl.component_off);
    p.spd = spd;
    p.n = batch->n_total;
    p.n_pad = pl.n_pad;
    p.max_dist = max_dist;
    p.n_planes = pull_planes(max_dist);
    static std::atomic<uint64_t> order_granted{0}, pull_granted{0};
    gt_status st;
    if ((st = grant_smem(spd_large_order_kernel, order_granted, kLargeSmemLimit)) != GT_OK) return st;
    if ((st = grant_smem(spd_large_pull_kernel, pull_granted, kLargeSmemLimit)) != GT_OK) return st;
    if ((st = launch_overlapped(spd_large_order_kernel, dim3(1), 1024, 8 * (size_t)p.n, s, p)) != GT_OK) return st;
    const size_t tasks = (size_t)p.n / 32 + 2 + (size_t)nnz / (kLargeHubDegree + 1);
    if ((st = launch_overlapped(spd_large_lists_kernel, dim3((unsigned)tasks), 256, 0, s, p)) != GT_OK) return st;
    return launch_overlapped(spd_large_pull_kernel, dim3(pl.blocks), (unsigned)pl.threads, pl.smem_bytes, s, p);
}

}  // namespace gt
