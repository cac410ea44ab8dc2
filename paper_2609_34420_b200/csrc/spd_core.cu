// Targets that follow from others.  A path to t ends with an edge from one of t's in-neighbours, so
//     dist(s, t) = 1 + min over in-neighbours p of t of dist(s, p)        (s != t)
// and a target needs no search of its own if all its in-neighbours have one.  The build for large graphs searches for the
// others only, the core: bit rows are that much shorter, and so is all the traffic that bounds it; the expansion then
// forms the rest while it writes the matrix.  In a power-law graph of 65 536 nodes and degree 12 the core is 43 % of the nodes.
//
// The targets left out are an independent set among the vertices of up to kCoreMaxDegree in-neighbours, few first: of two
// joined vertices the one with more in-neighbours (then by a hash) loses, who has not lost to anyone is in, and a second round
// among the losers that are not joined to those.  No edge joins two of the set in either direction, so directed
// graphs need nothing else.
#include <type_traits>

#include "spd_core.cuh"
#include "spd_pull.cuh"

namespace gt {
namespace {

constexpr int kSegmentGroups = kCoreSegment / 32;
constexpr int kSegmentWarps = kSegmentGroups / 8;                    // that work on a segment, eight groups each
constexpr int kStageWords = 4 * kCoreSegment;                        // two segments of either half of a block
constexpr int kSegmentList = kCoreSegment * kCoreMaxDegree / 2;      // words
constexpr int kCoreSmem = 222 * 1024;                                // and 5 KB of static arrays
constexpr int kMaxWords = kCoreMaxNodes / 32;
constexpr uint16_t kPadding = 0xffff;                                // loc of a column past the last node

// Vertices of few edges, by their out-edges, which are there without counting: a graph without many of them is not looked at further.
__global__ void __launch_bounds__(1024) spd_core_candidates_kernel(CoreParams p)
{
    grid_wait();
    grid_release();
    const int v = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    const int few = __syncthreads_count(v < p.n && p.row_ptr[v + 1] - p.row_ptr[v] <= kCoreMaxDegree);
    if (threadIdx.x == 0) atomicAdd(p.candidates, (uint32_t)few);
}
__device__ __forceinline__ bool hopeless(const CoreParams& p) { return *p.candidates < (uint32_t)(0.3f * (float)p.n); }

// In-degrees and in-neighbours; a warp per work item of the search, up to 32 edges of a vertex (a warp per 32 vertices takes 500 us at
// 65 536 nodes where the hubs are neighbours).
__global__ void __launch_bounds__(256) spd_core_degree_kernel(CoreParams p)
{
    grid_wait();
    grid_release();
    if (hopeless(p)) return;
    const int item = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (item >= p.item_start[p.n]) return;
    const int4 rec = p.items[item];                      // vertex, first edge, one past the last
    const int e = rec.y + (int)(threadIdx.x & 31);
    if (e >= rec.z) return;
    const int t = p.col_idx[e];
    if (t == rec.x) return;
    const uint32_t at = atomicAdd(&p.in_degree[t], 1u);
    if (at < kCoreMaxDegree) p.slots[(size_t)t * kCoreMaxDegree + at] = (uint16_t)rec.x;
}

__device__ __forceinline__ bool candidate(uint32_t degree) { return degree <= kCoreMaxDegree; }
__device__ __forceinline__ uint32_t rank_of(uint32_t degree, int v) { return degree << 16 | (((uint32_t)v * 40503u) & 0xffffu); }

// f(p, in-degree of p) for t's in-neighbours that are candidates; d: t's in-degree
template <class F>
__device__ __forceinline__ void for_candidates(const CoreParams& p, int t, uint32_t d, F f)
{
    const uint4 s4 = *(const uint4*)(p.slots + (size_t)t * kCoreMaxDegree);
    const uint32_t s[4] = {s4.x, s4.y, s4.z, s4.w};
    uint32_t from[kCoreMaxDegree];
#pragma unroll
    for (int j = 0; j < kCoreMaxDegree; ++j) from[j] = j < (int)d ? p.in_degree[(s[j / 2] >> (16 * (j & 1))) & 0xffffu] : 0xffffffffu;
#pragma unroll
    for (int j = 0; j < kCoreMaxDegree; ++j)
        if (candidate(from[j])) f((int)((s[j / 2] >> (16 * (j & 1))) & 0xffffu), from[j]);
}

// kStep 0: the first round's losers, 1: who is joined to a winner, 2: the second round's losers
template <int kStep>
__global__ void __launch_bounds__(256) spd_core_round_kernel(CoreParams p)
{
    grid_wait();
    grid_release();
    const int t = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (t >= p.n || hopeless(p)) return;
    const uint32_t d = p.in_degree[t];
    if (!candidate(d)) return;
    const bool won = kStep > 0 && p.lost[t] == 0;
    const bool again = kStep == 2 && !won && p.out[t] == 0;
    if (kStep == 2 && !again) return;
    for_candidates(p, t, d, [&](int u, uint32_t du) {
        if (kStep == 1) {
            const bool won_u = p.lost[u] == 0;
            if (won && !won_u) p.out[u] = 1;
            if (won_u && !won) p.out[t] = 1;
        } else {
            if (kStep == 2 && (p.lost[u] == 0 || p.out[u] != 0)) return;
            uint8_t* mark = kStep == 0 ? p.lost : p.lost_again;
            mark[rank_of(du, u) > rank_of(d, t) ? u : t] = 1;
        }
    });
}

__global__ void __launch_bounds__(256) spd_core_bits_kernel(CoreParams p)
{
    grid_wait();
    grid_release();
    const int t = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    const bool in = t < p.n && candidate(p.in_degree[t]) && (p.lost[t] == 0 || (p.out[t] == 0 && p.lost_again[t] == 0));
    const uint32_t bits = __ballot_sync(0xffffffffu, in);
    if ((threadIdx.x & 31) == 0 && t < p.n) p.left_out[t / 32] = bits;
}

// Word of column c in the expansion's shared memory: 16-byte pieces of 32 columns are swapped, so that threads that write 32
// columns each do not meet in the same banks.
__device__ __forceinline__ uint32_t word_of_column(uint32_t c) { return (c & ~31u) | ((((c >> 2) ^ (c >> 5)) & 7u) << 2) | (c & 3u); }

// Segments are for the halves of a block in turn, and each has room for two.
__device__ __forceinline__ uint32_t stage_of(int seg) { return (uint32_t)(seg & 3) * kCoreSegment; }

// A block per segment of targets: columns, the targets left out by their number of in-neighbours in groups of 32, and their lists.
__global__ void __launch_bounds__(1024) spd_core_lists_kernel(CoreParams p)
{
    __shared__ uint32_t s_bits[kMaxWords], s_before[kMaxWords];      // vertices left out: bits, and how many before a word
    __shared__ uint32_t s_warp[32], s_class[kCoreMaxDegree + 2], s_off[kSegmentGroups];
    grid_wait();
    grid_release();
    const int n = p.n, n_words = (n + 31) / 32, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int w0 = 2 * (int)threadIdx.x;
    uint32_t bits[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        bits[k] = w0 + k < n_words ? p.left_out[w0 + k] : 0u;
        s_bits[w0 + k] = bits[k];
    }
    const int mine = __popc(bits[0]) + __popc(bits[1]);
    const int incl = warp_scan(mine, lane);
    if (lane == 31) s_warp[warp] = (uint32_t)incl;
    if (threadIdx.x < kCoreMaxDegree + 2) s_class[threadIdx.x] = 0u;
    __syncthreads();
    if (warp == 0) s_warp[lane] = (uint32_t)warp_scan((int)s_warp[lane], lane);
    __syncthreads();
    const uint32_t before = (warp ? s_warp[warp - 1] : 0u) + (uint32_t)(incl - mine);
    s_before[w0] = before;
    s_before[w0 + 1] = before + (uint32_t)__popc(bits[0]);
    const int n_cols = n - (int)s_warp[31];
    const int groups = max(1, (n_cols + 8191) / 8192);
    const int block_bits = max(1, ((n_cols + groups - 1) / groups + 127) / 128) * 128;
    const int n_planes = min(kCoreMaxLevels, p.plane_words / (groups * (block_bits / 32)));
    // Not worth while (the expansion reads what the search would have written) or no room
    const bool reduced = !hopeless(p) && n_cols <= (int)(0.7f * (float)n) && groups * block_bits <= n && groups <= p.n_groups && (groups * block_bits + 4 + kStageWords) * 4 <= kCoreSmem &&
                         n_planes + kCoreLateLevels >= kCoreMaxLevels;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        CoreInfo& o = *p.info;
        o.deep = 0;
        for (int g = 0; g < kCoreMaxGroups; ++g) o.levels[g] = 0;
        o.reduced = reduced ? 1 : 0;
        o.n_cols = n_cols;
        o.block_bits = block_bits;
        o.row_words = block_bits / 32;
        o.n_groups = groups;
        o.n_planes = n_planes;
    }
    if (!reduced) return;
    __syncthreads();
    auto column = [&](int v) -> uint32_t { return (uint32_t)v - s_before[v >> 5] - (uint32_t)__popc(s_bits[v >> 5] & ((1u << (v & 31)) - 1u)); };
    const int seg = (int)blockIdx.x, t_first = seg * kCoreSegment;
    const uint32_t stage = (uint32_t)(groups * block_bits) + 4u + stage_of(seg);
    const uint32_t none = (uint32_t)(groups * block_bits);           // a word that is "none" for all sources
    constexpr int kPer = kCoreSegment / 1024;
    uint32_t place[kPer];                                            // class << 16 | rank
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int t = t_first + k * 1024 + (int)threadIdx.x;
        const bool left = t < n && ((s_bits[t >> 5] >> (t & 31)) & 1u);
        const uint32_t cls = left ? p.in_degree[t] : kCoreMaxDegree + 1;
        const uint32_t peers = __match_any_sync(0xffffffffu, cls);
        const int leader = __ffs((int)peers) - 1;
        uint32_t at = 0;
        if (lane == leader) at = atomicAdd(&s_class[cls], (uint32_t)__popc(peers));
        at = __shfl_sync(0xffffffffu, at, leader) + (uint32_t)__popc(peers & ((1u << lane) - 1u));
        place[k] = cls << 16 | at;
        if (t < n) p.column[t] = left ? -1 : (int32_t)column(t);
    }
    __syncthreads();
    uint32_t first[kCoreMaxDegree + 2];
    first[0] = 0u;
#pragma unroll
    for (int c = 0; c <= kCoreMaxDegree; ++c) first[c + 1] = first[c] + s_class[c];
    const int n_left = (int)first[kCoreMaxDegree + 1], n_groups = (n_left + 31) / 32;
    auto class_at = [&](int pos) -> uint32_t {
        uint32_t c = 0;
#pragma unroll
        for (int k = 1; k <= kCoreMaxDegree; ++k) c = pos >= (int)first[k] ? (uint32_t)k : c;
        return c;
    };
    if (warp == 0) {                                     // lists in the order in which the expansion's warps go through them
        uint32_t at = 0;
        for (int o = lane; o < kSegmentGroups; o += 32) {
            const int q = (o >> 3) + kSegmentWarps * (o & 7);
            const uint32_t pairs = q < n_groups ? (class_at(min(32 * q + 31, n_left - 1)) + 1) / 2 : 0u;
            const int words = 32 * (int)pairs, x = warp_scan(words, lane);
            const uint32_t first_word = at + (uint32_t)(x - words);
            s_off[q] = first_word;
            uint32_t head = pairs << (3 * (o & 7)) | (q < n_groups ? 1u << 24 : 0u);       // of the eight groups of a warp: pairs of edges, and how many
#pragma unroll
            for (int off = 1; off < 8; off <<= 1) head += __shfl_xor_sync(0xffffffffu, head, off);
            if ((o & 7) == 0) p.groups[seg * kSegmentWarps + (o >> 3)] = make_uint2((uint32_t)seg * kSegmentList + first_word, head);
            at += (uint32_t)__shfl_sync(0xffffffffu, x, 31);
        }
    }
    __syncthreads();
    uint32_t* list = p.list + (size_t)seg * kSegmentList;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int t = t_first + k * 1024 + (int)threadIdx.x;
        const uint32_t cls = place[k] >> 16;
        if (t >= n) {
            if (t < ((n + 15) & ~15)) p.loc[t] = kPadding;
            continue;
        }
        if (cls > kCoreMaxDegree) {
            p.loc[t] = (uint16_t)word_of_column(column(t));
            continue;
        }
        uint32_t pos = place[k] & 0xffffu;
#pragma unroll
        for (int c = 0; c <= kCoreMaxDegree; ++c) pos += (uint32_t)c == cls ? first[c] : 0u;
        p.loc[t] = (uint16_t)(stage + pos);
        const uint32_t most = class_at(min((int)(pos | 31u), n_left - 1));
        const uint4 s4 = *(const uint4*)(p.slots + (size_t)t * kCoreMaxDegree);
        const uint32_t s[4] = {s4.x, s4.y, s4.z, s4.w};
        uint32_t* at = list + s_off[pos / 32] + (pos & 31u);
#pragma unroll
        for (int j = 0; j < kCoreMaxDegree / 2; ++j) {
            if (2 * j >= (int)most) continue;
            const uint32_t a = 2 * j < (int)cls ? word_of_column(column((int)(s[j] & 0xffffu))) : none;
            const uint32_t b = 2 * j + 1 < (int)cls ? word_of_column(column((int)(s[j] >> 16))) : none;
            at[32 * j] = a | b << 16;
        }
    }
    for (int pos = n_left + (int)threadIdx.x; pos < 32 * n_groups; pos += (int)blockDim.x) {       // lanes without a target
        const uint32_t most = class_at(n_left - 1);
        for (int j = 0; 2 * j < (int)most; ++j) list[s_off[pos / 32] + 32u * (uint32_t)j + ((uint32_t)pos & 31u)] = none | none << 16;
    }
}

struct ExpandParams {
    CoreParams c;
    const uint32_t* planes;                // [groups][levels][n][row_words]; further levels are in the rows of spd
    const uint8_t* nonempty;               // [groups][flag_planes][n_pad]
    uint8_t* spd;
    int32_t n_pad;
    int32_t flag_planes;
    int32_t max_dist;
    uint32_t minus_one;                    // not known to the compiler, which would subtract
};

// byte k: byte (s_k & 7) of hi:lo, s_k the k-th nibble of `select`; its sign eight times if s_k has bit 3
__device__ __forceinline__ uint32_t look_up4(uint32_t lo, uint32_t hi, uint32_t select)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(lo), "r"(hi), "r"(select));
    return r;
}

// rows of 32 bits -> columns: bit i of out[p] = bit p of in[i]
__device__ __forceinline__ void transpose32(uint32_t (&m)[32])
{
    uint32_t mask = 0x0000ffffu;
#pragma unroll
    for (int j = 16; j != 0; j >>= 1) {
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            if (k & j) continue;
            const uint32_t t = ((m[k] >> j) ^ m[k + j]) & mask;
            m[k] ^= t << j;
            m[k + j] ^= t;
        }
        mask ^= mask << (j >> 1);
    }
}

// four words with a byte per row -> four rows with a byte per word
__device__ __forceinline__ void transpose_bytes(const uint32_t (&w)[4], uint32_t (&r)[4])
{
    const uint32_t a = __byte_perm(w[0], w[1], 0x5140), b = __byte_perm(w[2], w[3], 0x5140);
    const uint32_t c = __byte_perm(w[0], w[1], 0x7362), d = __byte_perm(w[2], w[3], 0x7362);
    r[0] = __byte_perm(a, b, 0x5410);
    r[1] = __byte_perm(a, b, 0x7632);
    r[2] = __byte_perm(c, d, 0x5410);
    r[3] = __byte_perm(c, d, 0x7632);
}

// Field by field the smaller one of a and b, for fields whose values leave the bit `guard` of each free; it is set in a and stays so.
// (Logic and shifts share a pipe of half the rate, which bounds the expansion: the subtractions go to the other one as multiplications.)
template <int kGuardBit>
__device__ __forceinline__ uint32_t smaller(uint32_t a, uint32_t b, uint32_t guard, uint32_t minus_one)
{
    const uint32_t m = (b * minus_one + a) & guard;                              // a >= b
    const uint32_t mask = (m >> kGuardBit) * ((1u << kGuardBit) - 1u);           // the bits below the guard
    return (a & ~mask) | (b & mask);
}

// A thread block turns 32 / kBits source rows at a time into output bytes.  A word of shared memory holds one target's
// distances from these sources, kBits each: four (15: none) while all column blocks' frontiers were kept, else eight (the output's codes).
//   decode   the search's targets, 32 per thread, from the levels' frontiers (or the bytes that a deep search left)
//   gather   the targets left out: minima over their in-neighbours' words, a warp per 32 targets with the same number of them
//   output   words of eight neighbouring targets -> eight bytes of every row
// Of four-bit words without a distance beyond 6 the minimum is one of three-bit fields, whose fourth bit is the guard; else
// of every other field at a time.
// What bounds it: the pipe of logic and shifts, 61 % busy when all warps went through a segment together (issue slots as much; 2.0 TB/s
// of DRAM traffic): they gathered, then wrote, and waited for each other in between.  So each half of a block takes every other
// segment and meets only itself: one gathers while the other writes.
// 65 536 nodes, degree 12 (28 500 targets searched for, 37 000 with 3.0 in-neighbours on average): the whole build 4.96 -> 4.71 ms by the
// halves, the expansion 2.4 -> 2.15 ms of it; with four accumulators of 16-bit minima, which have no instruction here, and without the
// table of the output it took 3.3 ms.
template <int kBits>
__global__ void __launch_bounds__(1024, 1) spd_core_expand_kernel(ExpandParams p)
{
    constexpr int kSources = 32 / kBits;
    extern __shared__ __align__(16) uint32_t s_word[];
    __shared__ const uint32_t* s_row[kCoreMaxGroups][kCoreMaxLevels][kSources];      // frontier rows of the sources, by column block and level; nullptr: none
    __shared__ int s_levels[kCoreMaxGroups], s_far[2];
    const CoreInfo& info = *p.c.info;
    grid_wait();
    grid_release();
    if (!info.reduced || (info.deep != 0) != (kBits == 8)) return;
    const int n = p.c.n, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t ld = (int64_t)((n + 15) & ~15);
    const int row_words = info.row_words, n_words = info.n_groups * row_words, n_planes = info.n_planes;
    const int n_segments = (n + kCoreSegment - 1) / kCoreSegment, n_eights = (int)(ld / 8);
    const uint32_t max_dist = (uint32_t)p.max_dist;
    uint32_t* const stage = s_word + 32 * n_words + 4;
    if (threadIdx.x < kCoreMaxGroups) s_levels[threadIdx.x] = (int)threadIdx.x < info.n_groups ? info.levels[threadIdx.x] : 0;
    if (threadIdx.x < 4) s_word[32 * n_words + threadIdx.x] = 0xffffffffu;       // "none" (with eight bits: larger than any code, set right below)
    if (threadIdx.x < 2) s_far[threadIdx.x] = 0;
    __syncthreads();
    // The rows of the next sources, ahead of their use (and those of a plane to L2); s_far[turn]: some distance is beyond 6.
    auto fetch_rows = [&](int s0, int turn) {
        const int block = (int)threadIdx.x / kCoreMaxLevels, l = (int)threadIdx.x % kCoreMaxLevels;
        if (block >= kCoreMaxGroups || l >= s_levels[block]) return;
        const size_t at = ((size_t)block * p.flag_planes + l) * p.n_pad + s0;
        const uint32_t* plane = p.planes + (size_t)block * n_planes * n * row_words;
        const int here = min(kSources, n - s0);
        uint8_t set[kSources];                           // a byte per source, aligned to as many
        *(uint32_t*)set = *(const uint32_t*)(p.nonempty + at);
        if constexpr (kSources == 8) *(uint32_t*)(set + 4) = *(const uint32_t*)(p.nonempty + at + 4);
        bool any = false;
#pragma unroll
        for (int r = 0; r < kSources; ++r) {
            const bool there = r < here && set[r] != 0;
            const uint32_t* row = l < n_planes ? plane + ((size_t)l * n + s0 + r) * row_words : (const uint32_t*)(p.spd + (s0 + r) * ld + block * row_words * 32);
            s_row[block][l][r] = there ? row : nullptr;
            any = any || there;
        }
        if (any && l >= 6) s_far[turn] = 1;
        if (any && l < n_planes)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(plane + ((size_t)l * n + s0) * row_words), "r"((uint32_t)(here * row_words) * 4u) : "memory");
    };
    // A warp's groups of a segment, warp + 16 i: where their lists begin, pairs of edges of each (three bits), and how many; the words of
    // a list; a thread's targets.
    static_assert(kSegmentWarps == 16 && kCoreSegment == 8 * 512, "eight groups per warp and eight targets per thread of half a block");
    const int half = warp / kSegmentWarps, half_warp = warp % kSegmentWarps, half_thread = (int)threadIdx.x & 511;
    auto groups_of = [&](int seg) -> uint2 { return seg < n_segments ? __ldg(&p.c.groups[seg * kSegmentWarps + half_warp]) : make_uint2(0u, 0u); };
    auto words_at = [&](uint32_t off, int pairs, uint32_t (&u)[kCoreMaxDegree / 2]) {
#pragma unroll
        for (int j = 0; j < kCoreMaxDegree / 2; ++j)
            if (j < pairs) u[j] = __ldg(p.c.list + off + 32 * j);
    };
    auto locs_of = [&](int seg) -> uint4 {
        const int q = seg * 512 + half_thread;
        return seg < n_segments && q < n_eights ? __ldg((const uint4*)p.c.loc + q) : make_uint4(0u, 0u, 0u, 0u);
    };
    const uint32_t code_lo = (max_dist + 1u) | 1u << 8 | min(2u, max_dist) << 16 | min(3u, max_dist) << 24;
    const uint32_t code_hi = min(4u, max_dist) | min(5u, max_dist) << 8 | min(6u, max_dist) << 16 | min(7u, max_dist) << 24;
    fetch_rows(min((int)blockIdx.x * kSources, (n - 1) / kSources * kSources), 0);
    __syncthreads();

    for (int s0 = (int)blockIdx.x * kSources, turn = 0; s0 < n; s0 += (int)gridDim.x * kSources, turn ^= 1) {
        // ---- decode ----
        for (int w = threadIdx.x; w < n_words; w += (int)blockDim.x) {
            const int block = w / row_words, word = w - block * row_words, levels = s_levels[block];
            uint32_t bits[32];                                                   // [source][bit of the code]: the columns' bits
#pragma unroll
            for (int i = 0; i < 32; ++i) bits[i] = 0u;
            if (kBits == 4 || levels > 0) {
#pragma unroll
                for (int l = 0; l < kCoreMaxLevels; ++l) {
                    if (l >= levels) break;
                    const uint32_t at = l < n_planes ? (uint32_t)word : core_late_word(l - n_planes, word, row_words);
                    uint32_t x[kSources];
#pragma unroll
                    for (int r = 0; r < kSources; ++r) {
                        const uint32_t* row = s_row[block][l][r];
                        x[r] = row != nullptr ? __ldcs(row + at) : 0u;
                    }
#pragma unroll
                    for (int b = 0; b < 4; ++b)
                        if (((l + 1) >> b) & 1) {
#pragma unroll
                            for (int r = 0; r < kSources; ++r) bits[kBits * r + b] |= x[r];
                        }
                }
                if (kBits == 8) {                                                // levels -> codes
#pragma unroll
                    for (int r = 0; r < kSources; ++r) {
                        const uint32_t none = ~(bits[8 * r] | bits[8 * r + 1] | bits[8 * r + 2] | bits[8 * r + 3]);
                        uint32_t far = 0u, eq = 0xffffffffu;                     // level > max_dist
#pragma unroll
                        for (int b = 3; b >= 0; --b) {
                            const uint32_t m = max_dist >= 16u ? 0xffffffffu : 0u - ((max_dist >> b) & 1u);
                            far |= eq & bits[8 * r + b] & ~m;
                            eq &= ~(bits[8 * r + b] ^ m);
                        }
#pragma unroll
                        for (int b = 0; b < 8; ++b) {
                            const uint32_t m = 0u - ((max_dist >> b) & 1u), u = 0u - (((max_dist + 1u) >> b) & 1u);
                            bits[8 * r + b] = (bits[8 * r + b] & ~far) | (far & m) | (none & u);
                        }
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < kSources; ++r) {
                        const uint32_t none = ~(bits[4 * r] | bits[4 * r + 1] | bits[4 * r + 2] | bits[4 * r + 3]);
#pragma unroll
                        for (int b = 0; b < 4; ++b) bits[4 * r + b] |= none;
                    }
                }
#pragma unroll
                for (int r = 0; r < kSources; ++r) {                             // the source itself
                    const int own = s0 + r < n ? p.c.column[s0 + r] - 32 * w : -1;
                    if ((unsigned)own < 32u) {
                        const uint32_t self = 1u << Rows<32>::bit(own);
#pragma unroll
                        for (int b = 0; b < kBits; ++b) bits[kBits * r + b] &= ~self;
                    }
                }
                transpose32(bits);                                               // target 4 k + j at bits[8 j + k]
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    *(uint4*)&s_word[32 * w + 4 * (k ^ (w & 7))] = make_uint4(bits[k], bits[8 + k], bits[16 + k], bits[24 + k]);
            } else if (kBits == 8) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    uint32_t x[4], y[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) x[r] = s0 + r < n ? __ldcg((const uint32_t*)(p.spd + (int64_t)(s0 + r) * ld + 32 * w + 4 * k)) : 0u;
                    transpose_bytes(x, y);
                    *(uint4*)&s_word[32 * w + 4 * (k ^ (w & 7))] = make_uint4(y[0], y[1], y[2], y[3]);
                }
            }
        }
        const bool far = s_far[turn] != 0 || max_dist >= 127u;                   // (the table's first byte has no sign)
        if (threadIdx.x == 0) s_far[turn ^ 1] = 0;
        uint2 mine = groups_of(half);
        uint4 loc = locs_of(half);
        __syncthreads();
        if (s0 + (int)gridDim.x * kSources < n) fetch_rows(s0 + (int)gridDim.x * kSources, turn ^ 1);       // (read behind further barriers)
        uint32_t u[kCoreMaxDegree / 2];
        words_at(mine.x + lane, (int)(mine.y & 7u), u);
        // f(minimum over nothing, the words of a group's in-neighbours in pairs) -> word
        auto gather = [&](int seg, auto least) {
            uint32_t* to = stage + stage_of(seg) + 32 * half_warp + lane;
            uint32_t off = mine.x + (uint32_t)lane, head = mine.y;
            for (int left = (int)(head >> 24); left > 0; --left, to += 32 * kSegmentWarps, head >>= 3) {
                uint32_t v[kCoreMaxDegree / 2];
                const int k = (int)(head & 7u);
                off += 32u * (uint32_t)k;
                words_at(off, left > 1 ? (int)((head >> 3) & 7u) : 0, v);
                auto of = [&](auto pairs) {
                    constexpr int kPairs = decltype(pairs)::value;
                    uint32_t x[2 * kPairs + 1];
                    x[2 * kPairs] = 0xffffffffu;
#pragma unroll
                    for (int j = 0; j < kPairs; ++j) { x[2 * j] = s_word[u[j] & 0xffffu]; x[2 * j + 1] = s_word[u[j] >> 16]; }
                    *to = least(x);
                };
                if (k == 2) of(std::integral_constant<int, 2>{});
                else if (k == 1) of(std::integral_constant<int, 1>{});
                else if (k == 3) of(std::integral_constant<int, 3>{});
                else if (k == 4) of(std::integral_constant<int, 4>{});
                else of(std::integral_constant<int, 0>{});
#pragma unroll
                for (int j = 0; j < kCoreMaxDegree / 2; ++j) u[j] = v[j];
            }
        };
        // (the last element of x is "none")
        auto least_near = [&](auto& x) -> uint32_t {                             // four bits, distances up to 6
            constexpr uint32_t kGuard = 0x88888888u;
            constexpr int kCount = sizeof(x) / 4;
            uint32_t a = x[0] | kGuard;
#pragma unroll
            for (int j = 1; j + 1 < kCount; ++j) a = smaller<3>(a, x[j] & ~kGuard, kGuard, p.minus_one);
            const uint32_t r = (a & ~kGuard) + 0x11111111u, none = r & kGuard;   // one hop more; 8: none
            return r | (none - (none >> 3));
        };
        auto least_far = [&](auto& x) -> uint32_t {                              // four bits
            constexpr uint32_t kGuard = 0x80808080u, kLow = 0x0f0f0f0fu;
            constexpr int kCount = sizeof(x) / 4;
            uint32_t even = (x[0] & kLow) | kGuard, odd = ((x[0] >> 4) & kLow) | kGuard;
#pragma unroll
            for (int j = 1; j + 1 < kCount; ++j) {
                even = smaller<7>(even, x[j] & kLow, kGuard, p.minus_one);
                odd = smaller<7>(odd, (x[j] >> 4) & kLow, kGuard, p.minus_one);
            }
            even = (even & kLow) + 0x01010101u;
            odd = (odd & kLow) + 0x01010101u;
            even -= (even >> 4) & 0x01010101u;                                   // 16: 15 stays
            odd -= (odd >> 4) & 0x01010101u;
            return even | odd << 4;
        };
        auto least_code = [&](auto& x) -> uint32_t {                             // eight bits: codes
            constexpr int kCount = sizeof(x) / 4;
            uint32_t a = __vminu4(x[0], (max_dist + 1u) * 0x01010101u);          // (255 is "none", too)
#pragma unroll
            for (int j = 1; j + 1 < kCount; ++j) a = __vminu4(a, x[j]);
            return a + (__vcmpltu4(a, max_dist * 0x01010101u) & 0x01010101u);
        };
        auto output = [&](int seg, uint4 at) {
            const int q = seg * 512 + half_thread;
            if (q >= n_eights) return;
            const uint32_t at4[4] = {at.x, at.y, at.z, at.w};
            uint32_t x[8], past[2] = {0u, 0u};
            if (8 * q + 8 <= n) {
#pragma unroll
                for (int i = 0; i < 8; ++i) x[i] = s_word[i & 1 ? at4[i / 2] >> 16 : at4[i / 2] & 0xffffu];
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const bool in = 8 * q + i < n;
                    x[i] = in ? s_word[i & 1 ? at4[i / 2] >> 16 : at4[i / 2] & 0xffffu] : 0u;
                    if (!in) past[i / 4] |= 0xffu << (8 * (i % 4));              // columns behind the last node: 255
                }
            }
            const bool own = (unsigned)(8 * q - s0 + 7) < (unsigned)(kSources + 7);          // a source's own column
            if (own) {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int r = 8 * q + i - s0;
                    if ((unsigned)r < (unsigned)kSources) x[i] &= ~(((1u << kBits) - 1u) << (kBits * r));
                }
            }
            uint8_t* out = p.spd + (int64_t)s0 * ld + 8 * (int64_t)q;
            const int here = n - s0;
            auto store = [&](const uint32_t (&a)[4], const uint32_t (&b)[4], int first, int step) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (first + step * i < here) __stcs((uint2*)(out + (first + step * i) * ld), make_uint2(a[i] | past[0], b[i] | past[1]));
            };
            uint32_t a[4], b[4];
            if (kBits == 4 && !far) {
                // Distances up to 7: a byte permutation looks four of them up, and 8 is 0 (the sign of the first byte).  none -> 0, own column -> 8
#pragma unroll
                for (int i = 0; i < 8; ++i) x[i] -= ((x[i] >> 3) & 0x11111111u) * 15u;
                if (own) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int r = 8 * q + i - s0;
                        if ((unsigned)r < (unsigned)kSources) x[i] |= 8u << (4 * r);
                    }
                }
#pragma unroll
                for (int hlf = 0; hlf < 2; ++hlf) {                              // the first and the last four sources
                    uint32_t y[2][4];
#pragma unroll
                    for (int i = 0; i < 8; ++i) y[i / 4][i % 4] = look_up4(code_lo, code_hi, hlf ? x[i] >> 16 : x[i]);
                    transpose_bytes(y[0], a);
                    transpose_bytes(y[1], b);
                    store(a, b, 4 * hlf, 1);
                }
            } else if (kBits == 4) {
#pragma unroll
                for (int hlf = 0; hlf < 2; ++hlf) {                              // even and odd sources
                    uint32_t y[2][4];
#pragma unroll
                    for (int i = 0; i < 8; ++i) y[i / 4][i % 4] = (hlf ? x[i] >> 4 : x[i]) & 0x0f0f0f0fu;
                    transpose_bytes(y[0], a);
                    transpose_bytes(y[1], b);
                    auto code = [&](uint32_t v) -> uint32_t {
                        const uint32_t none = ((v + 0x01010101u) >> 4) & 0x01010101u;              // 15
                        if (max_dist >= 15u) return v + none * (max_dist - 14u);
                        const uint32_t over = ((v + (0x7fu - max_dist) * 0x01010101u) >> 7) & 0x01010101u;      // beyond max_dist
                        return ((v & ~(over * 0xffu)) | (over * max_dist)) + none;
                    };
#pragma unroll
                    for (int i = 0; i < 4; ++i) { a[i] = code(a[i]); b[i] = code(b[i]); }
                    store(a, b, hlf, 2);
                }
            } else {
                const uint32_t y[2][4] = {{x[0], x[1], x[2], x[3]}, {x[4], x[5], x[6], x[7]}};
                transpose_bytes(y[0], a);
                transpose_bytes(y[1], b);
                store(a, b, 0, 1);
            }
        };
        // The halves of the block take every other segment, each with its own barrier: one gathers while the other writes.
        for (int seg = half; seg < n_segments; seg += 2) {
            const uint2 next = groups_of(seg + 2);                               // ahead of their use
            const uint4 at = loc;
            if constexpr (kBits == 8) gather(seg, least_code);
            else if (far) gather(seg, least_far);
            else gather(seg, least_near);
            mine = next;
            words_at(mine.x + lane, (int)(mine.y & 7u), u);
            loc = locs_of(seg + 2);
            asm volatile("bar.sync %0, 512;" ::"r"(1 + half) : "memory");
            output(seg, at);
        }
        __syncthreads();                                                         // all words read
    }
}

}  // namespace

CorePlan spd_core_plan(int32_t n, int groups, size_t off, bool wanted)
{
    CorePlan c{};
    c.enabled = wanted && n >= kCoreMinNodes && n <= kCoreMaxNodes;
    c.groups = c.enabled && n > 8192 * groups * 10 / 7 ? groups + 1 : groups;
    if (c.groups > kCoreMaxGroups) c.groups = kCoreMaxGroups;
    c.clear_off = off;
    c.info_off = off;
    c.total_bytes = off;
    if (!c.enabled) return c;
    const size_t n_pad = align_up((size_t)n, 256);
    c.clear_bytes = 7 * n_pad + 256; off += c.clear_bytes;
    c.slot_off = off; off += n_pad * kCoreMaxDegree * sizeof(uint16_t);
    c.bits_off = off; off += align_up(n_pad / 8, 256);
    c.col_off = off; off += n_pad * sizeof(int32_t);
    c.loc_off = off; off += n_pad * sizeof(uint16_t);
    const size_t segments = ((size_t)n + kCoreSegment - 1) / kCoreSegment;
    c.group_off = off; off += align_up(segments * kSegmentWarps * sizeof(uint2), 256);
    c.list_off = off; off += segments * kSegmentList * sizeof(uint32_t);
    c.info_off = off; off += align_up(sizeof(CoreInfo), 256);
    c.total_bytes = off;
    return c;
}

gt_status spd_core_launch(const CorePlan& c, CoreParams& p, uint8_t* ws, const int32_t* row_ptr, const int32_t* col_idx,
                          int32_t n, int64_t nnz, const int4* items, const int32_t* item_start, int plane_words, cudaStream_t s)
{
    const size_t n_pad = align_up((size_t)n, 256);
    const int segments = (n + kCoreSegment - 1) / kCoreSegment;
    p.row_ptr = row_ptr;
    p.col_idx = col_idx;
    p.in_degree = (uint32_t*)(ws + c.clear_off);
    p.lost = ws + c.clear_off + 4 * n_pad;
    p.out = p.lost + n_pad;
    p.lost_again = p.out + n_pad;
    p.candidates = (uint32_t*)(p.lost_again + n_pad);
    p.slots = (uint16_t*)(ws + c.slot_off);
    p.left_out = (uint32_t*)(ws + c.bits_off);
    p.column = (int32_t*)(ws + c.col_off);
    p.loc = (uint16_t*)(ws + c.loc_off);
    p.groups = (uint2*)(ws + c.group_off);
    p.list = (uint32_t*)(ws + c.list_off);
    p.info = (CoreInfo*)(ws + c.info_off);
    p.items = items;
    p.item_start = item_start;
    p.n = n;
    p.n_groups = c.groups;
    p.plane_words = plane_words;
    GT_CUDA_TRY(cudaMemsetAsync(ws + c.clear_off, 0, c.clear_bytes, s));
    const dim3 per_vertex((unsigned)((n + 255) / 256));
    gt_status st;
    if ((st = launch_overlapped(spd_core_candidates_kernel, dim3((unsigned)((n + 1023) / 1024)), 1024, 0, s, p)) != GT_OK) return st;
    if ((st = launch_overlapped(spd_core_degree_kernel, dim3((unsigned)(((size_t)n + (size_t)nnz / 32 + 8) / 8)), 256, 0, s, p)) != GT_OK) return st;
    if ((st = launch_overlapped(spd_core_round_kernel<0>, per_vertex, 256, 0, s, p)) != GT_OK) return st;
    if ((st = launch_overlapped(spd_core_round_kernel<1>, per_vertex, 256, 0, s, p)) != GT_OK) return st;
    if ((st = launch_overlapped(spd_core_round_kernel<2>, per_vertex, 256, 0, s, p)) != GT_OK) return st;
    if ((st = launch_overlapped(spd_core_bits_kernel, per_vertex, 256, 0, s, p)) != GT_OK) return st;
    return launch_overlapped(spd_core_lists_kernel, dim3((unsigned)segments), 1024, 0, s, p);
}

gt_status spd_core_expand(const CoreParams& c, const uint32_t* planes, const uint8_t* nonempty, int32_t n_pad, int flag_planes,
                          int32_t max_dist, uint8_t* spd, cudaStream_t s)
{
    ExpandParams p{c, planes, nonempty, spd, n_pad, flag_planes, max_dist, 0xffffffffu};
    static std::atomic<uint64_t> granted4{0}, granted8{0};
    gt_status st;
    if ((st = grant_smem(spd_core_expand_kernel<4>, granted4, kCoreSmem)) != GT_OK) return st;
    if ((st = grant_smem(spd_core_expand_kernel<8>, granted8, kCoreSmem)) != GT_OK) return st;
    // the targets of the search are at most 0.7 n
    const size_t most = 4 * ((size_t)(0.7 * c.n) + 128 * kCoreMaxGroups + 32 + 4 + kStageWords);
    const size_t smem = most < (size_t)kCoreSmem ? most : (size_t)kCoreSmem;
    const dim3 grid((unsigned)sm_count());
    if ((st = launch_overlapped(spd_core_expand_kernel<4>, grid, 1024, smem, s, p)) != GT_OK) return st;
    return launch_overlapped(spd_core_expand_kernel<8>, grid, 1024, smem, s, p);
}

}  // namespace gt
