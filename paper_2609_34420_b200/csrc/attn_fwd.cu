// gt_biased_attn_fwd / gt_biased_attn_fwd_chunked: Eq. 1 forward,
//     O = Softmax(Q K^T / sqrt(d) + B_h[spd]) V,
// flash-style: score tiles are produced by tcgen05 MMAs into tensor memory, the bias is
// gathered from a per-head table by the SPD bucket and added BEFORE the running max / sum
// are updated (the rule the paper states for its context-parallel online softmax), P goes
// back to tensor memory as the A operand of the P V MMA.
//
// One CTA = one head x 256 query rows (two 128-row tiles, so the tensor pipe works on one tile
// while the other is in its softmax) x all key tiles of the graph (or of one key chunk, or several behind one
// another, for the chunked entry point).
//
//   warp 0      TMA producer: Q once; K and V through separate 2-stage rings; on a single graph
//               also the 256x128-byte SPD tile (3-stage ring, 128-byte swizzle)
//   warp 1      issues S_t = Q_t K^T (SS MMAs) for both query tiles
//   warp 3      issues O_t += P_t V (A from TMEM, B = V as MN-major)
//               (two issuing warps: a helper warp shares its scheduler with busy softmax warps
//               and gets few issue slots, so the MMA issue is split to keep it off the critical path)
//   warp 2      SPD loader for packed batches (per-graph pitch: cp.async with the same XOR swizzle)
//   warps 4-19  softmax: 8 warps per query tile, 4 per half of the 128 key columns (thread = query
//               row = TMEM lane, 64 score elements per thread).
//
// Softmax is single pass and speculative: a key tile is exponentiated against the row's current
// reference without looking at the tile's own maximum first; the row sum of the tile tells
// afterwards whether the reference was out of reach (sum above a threshold, or not finite), and only then the
// tile is redone the classical way (maximum, rescale of l and O, exponentials).  References are integers in log2
// units, so rescale factors are exact powers of two (a P entry depends on the reference in the rounding of its exponent's
// argument only).  They start at 0, as scores are mostly within some powers of two of 1; a few scores of the first tile tell where they
// are not.  With the first tile's maximum always taken first, and the first loads behind the set-up -> now: 4 096 nodes, 8 heads of 64:
// 59.4 -> 58.6 us, 64 graphs of 512-2 048 nodes, 16 heads: 1 052 -> 1 019; all scores shifted by -40: 60.7 -> 60.8, 1 088 -> 1 085.
//
// TMEM columns: three score buffers [0,128) [128,256) [256,384) used in rotation by the steps
// (key tile j, query tile t) -> buffer (2j+t) mod 3, so that the S MMA of a step never waits for a
// softmax; P overwrites the part of the score buffer its own thread has read (bf16, half the
// columns); O_0 [384,448), O_1 [448,512).
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>

#include "attn_common.cuh"
#include "sm100_primitives.cuh"

namespace gt {

namespace {

using namespace sm100;

constexpr int kRowsPerTile = 128;
constexpr int kQTiles = 2;
constexpr int kRowsPerCta = kRowsPerTile * kQTiles;
constexpr int kKvTile = 128;
constexpr int kKStages = 2;
constexpr int kVStages = 2;
constexpr int kSpdStages = 3;
constexpr int kHalves = 2;                    // softmax threads per query row (column halves)
constexpr int kCols = kKvTile / kHalves;      // score columns per softmax thread
constexpr int kCW = 16;                       // columns per TMEM load
constexpr int kChunks = kCols / kCW;
static_assert(kChunks == 4, "the softmax pass is written for four chunks");
constexpr float kSumThreshold = 0x1p24f;       // tile row sum above which the reference is raised
constexpr float kPeekReach = 24.0f;            // log2 units within which a row's first scores leave the starting reference as it is
constexpr int kNormRows = 256;                // precise variant: rows per entry of key_norms
constexpr float kReach = 60.0f;               // precise variant: log2 of the largest P entry that needs no new reference (and of the smallest at first)

struct FwdParams {
    const uint8_t* spd;
    const int64_t* spd_offsets;
    const int32_t* cu_seqlens;
    const float* bias;
    __nv_bfloat16* out;        // [T,H,D]          (unchunked)
    float* out_f32;            // [T,H,D] fp32     (unchunked, optional: the output before its rounding to bf16)
    float* lse;                // [H,T]            (unchunked)
    float* part_o;             // [C,T,H,D] fp32   (chunked)
    float* part_lse;           // [C,H,T]          (chunked)
    uint32_t* status;
    int32_t n_total;
    int32_t n_heads;
    int32_t n_buckets;
    int32_t kv_chunk_rows;     // chunked: keys of a share (multiple of 128): a chunk, or several behind one another
    float* chunk_sums;         //   sums over a share's chunks, [thread blocks][D / 8][softmax threads] of four channels of a row (nullptr: one chunk)
    int32_t chunk_tiles;       //   key tiles per chunk
    int32_t use_ranges;        // step entry point: key ranges given explicitly, one per grid z
    int32_t range_begin[2];
    int32_t range_end[2];
    int32_t q_block0;          // first 256-row query block of the launch
    float* state_o;            // step entry point, one key range: carried state merged in the epilogue
    float* state_lse;          //   ([T,H,D] fp32, [H,T]); rows [state_q_begin, state_q_end) only
    int32_t state_q_begin;
    int32_t state_q_end;
    const uint8_t* maps;       // packed batch: tensor maps of the graphs' SPD blocks
    const int4* list;          // packed batch: work list; block index = entry * heads + head (nullptr: grid of heads x blocks x graphs)
    int32_t split;             // one query tile: thread blocks (a cluster) that share its keys
    const __nv_bfloat16* q;    // precise variant: for the rows' norms
    const float* key_norms;    // precise variant: largest |k|^2 of every kNormRows rows, [H][blocks] (nullptr: always the classical way)
    int32_t early_release;     // let the next kernel start its set-up while this one runs
    int32_t spd_tma;           // 1: SPD tiles come by TMA; 0: packed batch without room for the maps, cp.async loader warp
    float c1;                  // log2(e) / sqrt(d)
};

enum FwdBarrier {
    kBarQFull = 0,
    kBarKFull = 1,                           // [kKStages]
    kBarKEmpty = kBarKFull + kKStages,       // [kKStages]  commit after S_1 of the key tile
    kBarVFull = kBarKEmpty + kKStages,       // [kVStages]
    kBarVEmpty = kBarVFull + kVStages,       // [kVStages]  commit after PV_1 of the key tile
    kBarSpdFull = kBarVEmpty + kVStages,     // [kSpdStages]
    kBarSpdEmpty = kBarSpdFull + kSpdStages, // [kSpdStages]
    kBarSFull = kBarSpdEmpty + kSpdStages,   // [3]  per score buffer
    kBarBufFree = kBarSFull + 3,             // [3]  P of the buffer consumed by its PV MMA
    kBarPFull = kBarBufFree + 3,             // [2 tiles][2 key-tile parities]
    kBarODone = kBarPFull + 4,               // [2 tiles][2 key-tile parities]
    kNumFwdBarriers = kBarODone + 4
};

// kPair: half of an SM's shared memory.
template <int D, bool kPair = false>
struct FwdSmem {
    static constexpr int kKStages = kPair ? 1 : gt::kKStages, kVStages = gt::kVStages, kSpdStages = kPair ? 2 : gt::kSpdStages;
    static constexpr int kRowBytes = D * 2;
    static constexpr int kTileBytes = 128 * kRowBytes;
    static constexpr int kSpdTileBytes = (kPair ? kRowsPerTile : kRowsPerCta) * kKvTile;
    static constexpr int kQ = 0;
    static constexpr int kK = kQ + (kPair ? 1 : kQTiles) * kTileBytes;
    static constexpr int kV = kK + kKStages * kTileBytes;
    static constexpr int kSpd = kV + kVStages * kTileBytes;
    static constexpr int kBias = kSpd + kSpdStages * kSpdTileBytes;
    static constexpr int kXchg = kBias + 256 * 4;             // [2 tiles][max | sum][2 halves][128 rows] float
    static constexpr int kBars = kXchg + 2 * 512 * 4;
    static constexpr int kMisc = kBars + kNumFwdBarriers * 8;
    static constexpr int kSums = kMisc + 16;                  // kFold: [softmax threads] {reference, l} of the chunks before
    static constexpr int kTotal = kSums + (kPair ? 0 : 512 * 8);
    static constexpr int kDynamic = kTotal + 1024;   // slack for the 1024-byte alignment
};

enum FwdNamedBarrier { kNbPair = 2 /* + 4 t + lane quarter: the two warps that share 32 query rows */ };

template <bool B> struct BoolTag { static constexpr bool value = B; };

template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[N])
{
    if constexpr (N == 32) tmem_ld32(taddr, r); else tmem_ld16(taddr, r);
}
template <int N>
__device__ __forceinline__ void tmem_st(uint32_t taddr, const uint32_t (&r)[N])
{
    if constexpr (N == 32) tmem_st32(taddr, r); else tmem_st16(taddr, r);
}

// Sum of the squares of eight bf16 values.
__device__ __forceinline__ float square_sum(const uint4& v)
{
    float a = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t w = i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
        const float lo = __uint_as_float(w << 16), hi = __uint_as_float(w & 0xffff0000u);
        a += lo * lo + hi * hi;
    }
    return a;
}
// Larger of two values that are not negative; NaN wins.
__device__ __forceinline__ float norm_max(float a, float b) { return __uint_as_float(max(__float_as_uint(a) & 0x7fffffffu, __float_as_uint(b) & 0x7fffffffu)); }

// kPrecise (the fp32-output entry point): P goes to the P V MMA as TWO bf16 terms, P = hi + lo with
// lo = bf16(P - hi) (16 mantissa bits instead of 8), so that the output is accurate to fp32 accumulation
// instead of to the 2^-9 relative rounding of a bf16 P.  The two terms of a 16-key chunk overwrite that
// chunk's own score columns ([0,8) hi, [8,16) lo) as soon as the chunk has been read, so a tile cannot be
// redone.  It may go the speculative way all the same where no score can overflow: |q_i| max|k_j| / sqrt(d) + max bias
// bounds a row's scores, and while that is within 2^60 of the row's reference, P, l and O stay far inside the range
// of fp32 and bf16, whose relative precision does not depend on the reference.  Rows (warps of 32) beyond it take the
// maximum first, which costs a second pass over the scores.  8 192 nodes, 8 heads of 64: 386 -> 251 us, norms included.
// kTiles = 1: thread blocks of one 128-row query tile and eight softmax warps, for grids that would leave half
// of the SMs idle or more (rows_per_block); a cluster of them may share the keys (FwdParams::split).  Two score buffers then: with three, a warp could be two key tiles ahead of another.
// kPair (with one tile): two thread blocks per SM, of which one computes while the other fills, drains or waits for its MMAs; one score
// buffer, and half of the shared and of the tensor memory (pairs_of_blocks).
// kFold: the chunked forward with all chunks behind one another.  Every chunk of keys is a chain of MMAs of its own, as if its share went
// through memory, and is added to the chunks before with rounding: one chain over all of them would be less exact, because the tensor
// core cuts off what its accumulator cannot hold, an error that grows with the chain.
template <int D, bool kPartial, bool kShflBias, bool kPrecise = false, int kTiles = kQTiles, bool kPair = false, bool kFold = false>
__global__ void __launch_bounds__(128 + 256 * kTiles, kPair ? 2 : 1)
attn_fwd_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ CUtensorMap tmap_spd,
                const FwdParams p)
{
    using L = FwdSmem<D, kPair>;
    constexpr int kRows = kRowsPerTile * kTiles, kThreads = 128 + 256 * kTiles, kBuffers = kPair ? 1 : kTiles + 1;
    constexpr int kKStages = L::kKStages, kVStages = L::kVStages, kSpdStages = L::kSpdStages;
    constexpr uint32_t kTmemCols = kPair ? 256 : 512, kOCol = kPair ? 128 : 384;
    extern __shared__ uint8_t smem_raw[];
    // 1024-byte alignment by pointer arithmetic on the __shared__ array itself, so that every derived
    // pointer keeps its shared address space (integer round trips would turn the accesses generic)
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    int h = blockIdx.x, g = kPartial ? 0 : (int)blockIdx.z;
    int32_t q_block = (int32_t)blockIdx.y + p.q_block0;
    const int chunk = kPartial ? (int)blockIdx.z : 0;
    constexpr bool kShared = kTiles == 1 && !kPartial && !kPair && !kFold;       // blocks of a cluster may share the keys
    const int rank = kShared ? (int)blockIdx.x % p.split : 0;
    if constexpr (kShared) h = (int)blockIdx.x / p.split;

    if (p.cu_seqlens) grid_wait();          // a single graph's blocks set up their barriers and tensor memory before they wait
    int32_t node0 = 0, n_g = p.n_total;
    if (!kPartial && p.list) {
        const int4 entry = p.list[blockIdx.x / (unsigned)p.n_heads];
        if (entry.x < 0) return;
        h = (int)(blockIdx.x % (unsigned)p.n_heads);
        g = entry.x;
        q_block = entry.y;
        node0 = entry.z;
        n_g = entry.w;
    } else if (p.cu_seqlens) {
        node0 = p.cu_seqlens[g];
        n_g = p.cu_seqlens[g + 1] - node0;
    }
    const int32_t q0 = q_block * kRows;
    if (q0 >= n_g) return;
    const int64_t ld = (int64_t)((n_g + 15) & ~15);
    const uint8_t* spd_g = p.spd + (p.spd_offsets ? p.spd_offsets[g] : 0);
    int32_t kv_begin = kPartial ? (p.use_ranges ? p.range_begin[chunk] : chunk * p.kv_chunk_rows) : 0;
    int32_t kv_end = kPartial ? (p.use_ranges ? p.range_end[chunk] : min(n_g, kv_begin + p.kv_chunk_rows)) : n_g;
    int sharers = 1;                        // blocks of the cluster that have keys
    if constexpr (kShared) {
        const int32_t tiles = (n_g + kKvTile - 1) / kKvTile, per = (tiles + p.split - 1) / p.split;
        sharers = (tiles + per - 1) / per;
        if (rank >= sharers) return;        // (the cluster's barriers wait for blocks that are still there)
        kv_begin = rank * per * kKvTile;
        kv_end = min(n_g, kv_begin + per * kKvTile);
    }
    const int32_t n_kv = kv_end > kv_begin ? (kv_end - kv_begin + kKvTile - 1) / kKvTile : 0;

    if (kPartial && n_kv == 0) {            // empty chunk: weight zero in the merge
        grid_wait();
        for (int i = tid; i < kRows; i += kThreads) {
            int q = q0 + i;
            if (q < n_g) {
                p.part_lse[((size_t)chunk * p.n_heads + h) * p.n_total + q] = -INFINITY;
                float* o = p.part_o + (((size_t)chunk * p.n_total + q) * p.n_heads + h) * D;
                for (int c = 0; c < D; ++c) o[c] = 0.f;
            }
        }
        return;
    }

    uint64_t* bars = (uint64_t*)(smem + L::kBars);
    uint32_t* misc = (uint32_t*)(smem + L::kMisc);       // [0] TMEM base, [1] abort flag
    float* s_bias = (float*)(smem + L::kBias);
    auto bar = [&](int i) { return smem_u32(&bars[i]); };
    volatile uint32_t* abort_flag = &misc[1];

    if (tid == 0) {
        misc[1] = 0u;
        mbar_init(bar(kBarQFull), 1);
        for (int s = 0; s < kKStages; ++s) { mbar_init(bar(kBarKFull + s), 1); mbar_init(bar(kBarKEmpty + s), 1); }
        for (int s = 0; s < kVStages; ++s) { mbar_init(bar(kBarVFull + s), 1); mbar_init(bar(kBarVEmpty + s), 1); }
        for (int s = 0; s < kSpdStages; ++s) { mbar_init(bar(kBarSpdFull + s), p.spd_tma ? 1 : 32); mbar_init(bar(kBarSpdEmpty + s), 8 * kTiles); }
        for (int b = 0; b < 3; ++b) { mbar_init(bar(kBarSFull + b), 1); mbar_init(bar(kBarBufFree + b), 1); }
        for (int t = 0; t < 4; ++t) mbar_init(bar(kBarPFull + t), 4 * kHalves);     // one arrival per warp
        for (int t = 0; t < 4; ++t) mbar_init(bar(kBarODone + t), 1);
        fence_mbar_init();
        prefetch_tensormap(&tmap_q);
        prefetch_tensormap(&tmap_k);
        prefetch_tensormap(&tmap_v);
        if (p.spd_tma && !p.maps) prefetch_tensormap(&tmap_spd);
    }
    if (warp == 1) { tmem_alloc(smem_u32(&misc[0]), kTmemCols); tmem_relinquish(); }
    grid_wait();
    // The first tiles are on their way while the block is still setting up: the thread that set up the barriers is the one that loads.
    const void* spd_map = !kPartial && p.maps ? (const void*)(p.maps + (size_t)g * kMapBytes) : &tmap_spd;
    auto load_k = [&](int j) {
        const int s = j % kKStages;
        mbar_arrive_expect_tx(bar(kBarKFull + s), L::kTileBytes);
        tma_load_3d(smem_u32(smem + L::kK + s * L::kTileBytes), &tmap_k, bar(kBarKFull + s), 0, h, node0 + kv_begin + j * kKvTile);
    };
    auto load_spd = [&](int j) {
        const int s = j % kSpdStages;
        mbar_arrive_expect_tx(bar(kBarSpdFull + s), kRows * kKvTile);
        tma_load_2d(smem_u32(smem + L::kSpd + s * L::kSpdTileBytes), spd_map, bar(kBarSpdFull + s), kv_begin + j * kKvTile, q0);
    };
    auto load_v = [&](int j) {
        const int s = j % kVStages;
        mbar_arrive_expect_tx(bar(kBarVFull + s), L::kTileBytes);
        tma_load_3d(smem_u32(smem + L::kV + s * L::kTileBytes), &tmap_v, bar(kBarVFull + s), 0, h, node0 + kv_begin + j * kKvTile);
    };
    if (tid == 0) {
        mbar_arrive_expect_tx(bar(kBarQFull), kTiles * L::kTileBytes);
        for (int t = 0; t < kTiles; ++t)
            tma_load_3d(smem_u32(smem + L::kQ + t * L::kTileBytes), &tmap_q, bar(kBarQFull), 0, h, node0 + q0 + t * kRowsPerTile);
        load_k(0);
        if (!kPartial && p.maps) acquire_tensor_map(spd_map);
        if (p.spd_tma) load_spd(0);
        load_v(0);
    }
    if (p.early_release) grid_release();
    for (int i = tid; i < 256; i += kThreads)
        s_bias[i] = p.bias[(size_t)h * p.n_buckets + min(i, p.n_buckets - 1)] * kLog2e;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = misc[0];

    if (warp < 4) {
        // =========================== producer / MMA / SPD warps ===========================
        if constexpr (kTiles == 2 || kPair) setmaxnreg_dec_32();
        if (warp == 0) {
            for (int j = 1; j < n_kv; ++j) {
                mbar_wait(bar(kBarKEmpty + j % kKStages), ((j / kKStages) & 1) ^ 1, abort_flag, p.status, 10);
                if (lane == 0) load_k(j);
                if (p.spd_tma) {
                    mbar_wait(bar(kBarSpdEmpty + j % kSpdStages), ((j / kSpdStages) & 1) ^ 1, abort_flag, p.status, 11);
                    if (lane == 0) load_spd(j);
                }
                mbar_wait(bar(kBarVEmpty + j % kVStages), ((j / kVStages) & 1) ^ 1, abort_flag, p.status, 12);
                if (lane == 0) load_v(j);
                __syncwarp();
            }
        } else if (warp == 1) {
            // ---- S issuer: step (j, t) goes to score buffer (2j+t) mod 3 once the PV MMA of the
            // step that used the buffer before has drained it ----
            constexpr uint32_t idesc_s = make_idesc_bf16(128, 128, false, false);
            const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
            const uint64_t desc_q0 = make_smem_desc(smem_u32(smem + L::kQ), L::kRowBytes, 0);
            const uint64_t desc_k0 = make_smem_desc(smem_u32(smem + L::kK), L::kRowBytes, 0);
            mbar_wait(bar(kBarQFull), 0, abort_flag, p.status, 20);
            for (int j = 0; j < n_kv; ++j) {
                const int ks = j % kKStages;
                mbar_wait(bar(kBarKFull + ks), (j / kKStages) & 1, abort_flag, p.status, 22);
#pragma unroll
                for (int t = 0; t < kTiles; ++t) {
                    const int step = kTiles * j + t, b = step % kBuffers;
                    if (step >= kBuffers) mbar_wait(bar(kBarBufFree + b), (step / kBuffers - 1) & 1, abort_flag, p.status, 23);
                    tc_fence_after();
                    if (elect_one()) {
                        const uint64_t da = advance_desc(desc_q0, t * L::kTileBytes);
                        const uint64_t db = advance_desc(desc_k0, ks * L::kTileBytes);
#pragma unroll
                        for (int k = 0; k < D / 16; ++k)
                            mma_ss(tm + b * 128, advance_desc(da, k * 32), advance_desc(db, k * 32), idesc_s, k > 0);
                        mma_commit(bar(kBarSFull + b));
                        if (t == kTiles - 1) mma_commit(bar(kBarKEmpty + ks));
                    }
                    __syncwarp();
                }
            }
        } else if (warp == 3) {
            // ---- PV issuer ----
            constexpr uint32_t idesc_o = make_idesc_bf16(128, D, false, true);
            const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
            const uint64_t desc_v0 = make_smem_desc(smem_u32(smem + L::kV), L::kRowBytes, 0);
            [[maybe_unused]] int begin = 0;             // key tile that begins the next chunk
            for (int j = 0; j < n_kv; ++j) {
                const int vs = j % kVStages;
                mbar_wait(bar(kBarVFull + vs), (j / kVStages) & 1, abort_flag, p.status, 25);
                const uint64_t dv = advance_desc(desc_v0, vs * L::kTileBytes);
                uint32_t acc0 = j > 0 ? 1u : 0u;
                if constexpr (kFold) {
                    acc0 = j != begin ? 1u : 0u;
                    if (j == begin) begin += p.chunk_tiles;
                }
#pragma unroll
                for (int t = 0; t < kTiles; ++t) {
                    const int b = (kTiles * j + t) % kBuffers;
                    mbar_wait(bar(kBarPFull + 2 * t + (j & 1)), (j >> 1) & 1, abort_flag, p.status, 24);
                    tc_fence_after();
                    if (elect_one()) {
                        if constexpr (kPrecise) {
#pragma unroll
                            for (int k = 0; k < kKvTile / 16; ++k) {    // hi and lo term of key chunk k at the start of its own 16 score columns
                                const uint32_t a = tm + b * 128 + (k / (kCols / 16)) * kCols + (k % (kCols / 16)) * 16;
                                mma_ts(tm + kOCol + t * 64, a, advance_desc(dv, k * 16 * L::kRowBytes), idesc_o, k > 0 ? 1u : acc0);
                                mma_ts(tm + kOCol + t * 64, a + 8, advance_desc(dv, k * 16 * L::kRowBytes), idesc_o, 1u);
                            }
                        } else {
#pragma unroll
                        for (int k = 0; k < kKvTile / 16; ++k)      // P of key half hf sits at the start of that half's score columns
                            mma_ts(tm + kOCol + t * 64, tm + b * 128 + (k / (kCols / 16)) * kCols + (k % (kCols / 16)) * 8,
                                   advance_desc(dv, k * 16 * L::kRowBytes), idesc_o, k > 0 ? 1u : acc0);
                        }
                        mma_commit(bar(kBarODone + 2 * t + (j & 1)));
                        mma_commit(bar(kBarBufFree + b));
                        if (t == kTiles - 1) mma_commit(bar(kBarVEmpty + vs));
                    }
                    __syncwarp();
                }
            }
        } else if (!p.spd_tma) {
            // ---- warp 2: SPD tile loader for packed batches ----
            // A lane copies 16-byte chunk cc of rows lr, lr + 4, ...; the 128-byte swizzle (chunk c of row r at c ^ (r & 7))
            // depends on the parity of the round only, so both shared-memory offsets and the source pointer are
            // formed once and a copy costs the instruction itself plus one multiply-add for its address.
            const int cc = lane & 7, lr = lane >> 3;
            const uint32_t dst_even = (uint32_t)(lr * 128 + ((cc ^ lr) << 4)), dst_odd = (uint32_t)(lr * 128 + ((cc ^ (4 + lr)) << 4));
            const uint8_t* lane_src = spd_g + (int64_t)(q0 + lr) * ld + cc * 16;
            const uint32_t step = 4u * (uint32_t)ld;      // every copy's address is base + (constant round) * step: no dependent chain
            const int32_t rows_valid = min(kRows, n_g - q0);
            for (int j = 0; j < n_kv; ++j) {
                const int s2 = j % kSpdStages;
                mbar_wait(bar(kBarSpdEmpty + s2), ((j / kSpdStages) & 1) ^ 1, abort_flag, p.status, 30);
                const int32_t kv0 = kv_begin + j * kKvTile;
                const uint32_t dst0 = smem_u32(smem + L::kSpd + s2 * L::kSpdTileBytes);
                const uint8_t* src = lane_src + kv0;
                if (rows_valid == kRows && (int64_t)kv0 + kKvTile <= ld) {
#pragma unroll 16
                    for (int i = 0; i < kRows / 4; ++i)
                        cp_async_16(dst0 + i * 512 + ((i & 1) ? dst_odd : dst_even), src + (uint64_t)step * (uint32_t)i, 16u);
                } else {
                    const int32_t lim = ((int64_t)kv0 + cc * 16 < ld) ? rows_valid - lr : 0;     // rounds 4 i < lim are in range
#pragma unroll 8
                    for (int i = 0; i < kRows / 4; ++i) {
                        const bool valid = 4 * i < lim;
                        cp_async_16(dst0 + i * 512 + ((i & 1) ? dst_odd : dst_even), valid ? src + (uint64_t)step * (uint32_t)i : spd_g, valid ? 16u : 0u);
                    }
                }
                cp_async_mbar_arrive_noinc(bar(kBarSpdFull + s2));
            }
        }
    } else {
        // =================================== softmax warps ===================================
        if constexpr (kTiles == 2) setmaxnreg_inc_112();
        if constexpr (kPair) setmaxnreg_inc_104();       // 128 x 32 + 256 x 104 = 384 x 80 registers, which the block was launched with
        const int sw = warp - 4;
        const int t = sw / (4 * kHalves);
        const int hf = (sw >> 2) & (kHalves - 1);
        const int r = ((warp & 3) << 5) | lane;
        const uint32_t lane_off = (uint32_t)((warp & 3) * 32) << 16;
        constexpr int kOC = D / kHalves;                 // output columns per thread
        constexpr int kOP = kOC < 32 ? kOC : 32;         // ... per TMEM access
        const uint32_t tO = tmem + kOCol + t * 64 + hf * kOC + lane_off;
        const uint32_t pair_bar = kNbPair + t * 4 + (warp & 3);
        float* xchg = (float*)(smem + L::kXchg) + t * 512;
        float m = 0.f, l = 0.f;
        // A form of the pass without the subtraction, for warps whose references are all 0.  8 192 nodes, 8 heads of 64, fp32 output: 255 -> 242 us; heads
        // of 32: 16 384 nodes, 4 heads 424 -> 409, 64 graphs of 512-2 048 nodes, 16 heads 955 -> 938.  Heads of 64 gain 1 % at 0 (217.2 -> 215.3) and
        // lose 2 % where references differ (223 -> 228), two blocks per SM lose either way (195 -> 198, 209 -> 217).
        constexpr bool kOwnFormAtZero = kPrecise || (D == 32 && !kPair);
        [[maybe_unused]] bool m_moved = false;             // some reference of this warp may not be 0
        // kFold: O and l are of the chunk at work; what the chunks before add up to is in memory and, {reference, l}, in `sums`
        [[maybe_unused]] int next_chunk = p.chunk_tiles;
        [[maybe_unused]] float2* sums = (float2*)(smem + L::kSums) + (kFold ? tid - 128 : 0);
        constexpr int kSumStep = 256 * kTiles;
        [[maybe_unused]] auto o_sum = [&]() -> float4* {            // of this thread's row, four channels every kSumStep
            uint32_t x, y, z, at;               // (by asm: nothing of the address is to be kept in registers through the loop, which costs 2 %)
            asm volatile("mov.u32 %0, %%ctaid.x; mov.u32 %1, %%ctaid.y; mov.u32 %2, %%ctaid.z; mov.u32 %3, %%tid.x;" : "=r"(x), "=r"(y), "=r"(z), "=r"(at));
            return (float4*)p.chunk_sums + ((size_t)((z * gridDim.y + y) * gridDim.x + x) * (kOC / 4)) * kSumStep + (at - 128);
        };

        // lane b of every softmax warp keeps table entry b (scaled by log2 e); entries past the
        // table repeat the last one.  With at most 32 buckets a score's bias is fetched by a
        // warp shuffle whose source lane is the raw SPD byte (only its low 5 bits select).
        const float tbl = s_bias[lane];
        const uint64_t c1c1 = pack_f32x2(p.c1, p.c1);

        // Precise variant: no score of this row exceeds |q| max|k| / sqrt(d) + max bias (log2 units; with room for rounding).
        float limit = INFINITY, low = -INFINITY;             // ... and none is below `low`
        if constexpr (kPrecise) {
            if (p.key_norms != nullptr) {
                const int32_t n_blocks = (p.n_total + kNormRows - 1) / kNormRows;
                float kk = 0.f, qq = 0.f, bmax = -INFINITY, bmin = INFINITY;
                for (int32_t b = node0 / kNormRows + lane; b <= (node0 + n_g - 1) / kNormRows; b += 32)
                    kk = norm_max(kk, p.key_norms[(size_t)h * n_blocks + b]);
                for (int i = lane; i < 256; i += 32) { bmax = fmaxf(bmax, s_bias[i]); bmin = fminf(bmin, s_bias[i]); }
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) {
                    kk = norm_max(kk, __shfl_xor_sync(0xffffffffu, kk, off));
                    bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, off));
                    bmin = fminf(bmin, __shfl_xor_sync(0xffffffffu, bmin, off));
                }
                const int32_t row = node0 + min(q0 + t * kRowsPerTile + r, n_g - 1);
                const uint4* src = (const uint4*)(p.q + ((size_t)row * p.n_heads + h) * D);
#pragma unroll 2
                for (int i = 0; i < D / 8; ++i) qq += square_sum(src[i]);
                limit = sqrtf(qq * kk) * p.c1 * 1.001f + 1.0f;
                low = bmin - limit;
                limit += bmax;
            }
        }

        uint32_t sa[kCW], sb[kCW];              // score chunks, alternating
        uint4 wa[kCW / 16], wb[kCW / 16];       // their SPD bytes
        uint32_t tS = 0;                        // this thread's score columns of the current step
        const uint8_t* srow = nullptr;          // this thread's row of the current SPD tile
        auto load_chunk = [&](int c, uint32_t (&sr)[kCW], uint4 (&ws)[kCW / 16]) {
            tmem_ld<kCW>(tS + c * kCW, sr);
#pragma unroll
            for (int i = 0; i < kCW / 16; ++i)
                ws[i] = *(const uint4*)(srow + (((hf * (kCols / 16) + c * (kCW / 16) + i) ^ (r & 7)) << 4));
        };
        // bias of 8 consecutive columns (two SPD words)
        auto lookup8 = [&](uint32_t w0, uint32_t w1, float (&bb)[8]) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const uint32_t word = k == 0 ? w0 : w1;
                if (kShflBias) {
                    bb[4 * k + 0] = __shfl_sync(0xffffffffu, tbl, word);
                    bb[4 * k + 1] = __shfl_sync(0xffffffffu, tbl, word >> 8);
                    bb[4 * k + 2] = __shfl_sync(0xffffffffu, tbl, word >> 16);
                    bb[4 * k + 3] = __shfl_sync(0xffffffffu, tbl, word >> 24);
                } else {
                    bb[4 * k + 0] = s_bias[word & 0xffu];
                    bb[4 * k + 1] = s_bias[(word >> 8) & 0xffu];
                    bb[4 * k + 2] = s_bias[(word >> 16) & 0xffu];
                    bb[4 * k + 3] = s_bias[word >> 24];
                }
            }
        };
        // first chunk of key tile j: fetched at the end of tile j-1, behind the P store
        auto begin_tile = [&](int j) {
            const int step = kTiles * j + t, b = step % kBuffers;
            tS = tmem + b * 128 + hf * kCols + lane_off;
            mbar_wait(bar(kBarSFull + b), (step / kBuffers) & 1, abort_flag, p.status, 40);
            tc_fence_after();
            mbar_wait(bar(kBarSpdFull + (j % kSpdStages)), (j / kSpdStages) & 1, abort_flag, p.status, 41);
            srow = smem + L::kSpd + (j % kSpdStages) * L::kSpdTileBytes + (t * 128 + r) * 128;
            load_chunk(0, sa, wa);
        };
        begin_tile(0);

        for (int j = 0; j < n_kv; ++j) {
            const int32_t kv0 = kv_begin + j * kKvTile;
            const bool ragged = kv0 + kKvTile > kv_end;          // last key tile of the range
            const int valid = kv_end - kv0 - hf * kCols;         // valid columns of this thread (may be <= 0)
            uint32_t pk[kCols / 64][32];           // P of this thread's columns, bf16 pairs
            float tile_sum = 0.f;
            bool loaded = true;                    // chunk 0 is already on its way
            bool exact = false;                    // take the tile maximum first
            // Is the starting reference in reach of the first tile?  Four of the thread's first 16 scores tell: none of them far above 0 and one not far
            // below, so that the row's sum is not, either.  Otherwise the tile takes the classical way at once.
            if (!kPrecise && j == 0) {
                tmem_wait_ld();
                const uint32_t word[4] = {wa[0].x, wa[0].y, wa[0].z, wa[0].w};
                float top = -INFINITY;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float b = kShflBias ? __shfl_sync(0xffffffffu, tbl, word[i]) : s_bias[word[i] & 0xffu];
                    if (4 * i < valid) top = fmaxf(top, fmaf(__uint_as_float(sa[4 * i]), p.c1, b));
                }
                exact = named_barrier_or(pair_bar, 64, valid > 0 && !(fabsf(top) <= kPeekReach));       // (a half without valid columns has no say)
            }
            // The precise variant's P overwrites the scores chunk by chunk, so a tile cannot be redone: it goes the speculative way
            // only where the row's reference leaves no score out of reach (both column halves decide alike).
            if constexpr (kPrecise) exact = __any_sync(0xffffffffu, !(limit <= m + kReach) || (j == 0 && !(low >= -kReach)));

            for (;;) {
                if (exact) {
                    // ---- classical way: tile maximum, new reference, rescale of l and O ----
                    float mx0 = -INFINITY, mx1 = -INFINITY;
                    auto max_chunk = [&](int c, const uint32_t (&sr)[kCW], const uint4 (&ws)[kCW / 16]) {
#pragma unroll
                        for (int q = 0; q < kCW / 8; ++q) {
                            const uint4& ww = ws[q >> 1];
                            float bb[8];
                            lookup8((q & 1) ? ww.z : ww.x, (q & 1) ? ww.w : ww.y, bb);
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                float lo, hi;
                                unpack_f32x2(fma_f32x2(pack_u32x2(sr[q * 8 + 2 * i], sr[q * 8 + 2 * i + 1]), c1c1,
                                                       pack_f32x2(bb[2 * i], bb[2 * i + 1])), lo, hi);
                                const int col = c * kCW + q * 8 + 2 * i;
                                if (ragged && col >= valid) lo = -INFINITY;
                                if (ragged && col + 1 >= valid) hi = -INFINITY;
                                mx0 = fmaxf(mx0, lo);
                                mx1 = fmaxf(mx1, hi);
                            }
                        }
                    };
                    if (!loaded) load_chunk(0, sa, wa);
                    tmem_wait_ld(); load_chunk(1, sb, wb); max_chunk(0, sa, wa);
                    tmem_wait_ld(); load_chunk(2, sa, wa); max_chunk(1, sb, wb);
                    tmem_wait_ld(); load_chunk(3, sb, wb); max_chunk(2, sa, wa);
                    tmem_wait_ld(); max_chunk(3, sb, wb);
                    loaded = false;
                    float mt = fmaxf(mx0, mx1);
                    xchg[hf * 128 + r] = mt;
                    named_barrier_sync(pair_bar, 64);
                    mt = fmaxf(mt, xchg[(hf ^ 1) * 128 + r]);
                    const float m_new = j == 0 ? ceilf(mt) : fmaxf(m, ceilf(mt));
                    const float alpha = j == 0 ? 0.f : ex2_approx(m - m_new);      // (there is nothing yet; a first reference far below 0 would give infinity)
                    l *= alpha;
                    if (j > 0) {
                        mbar_wait(bar(kBarODone + 2 * t + ((j - 1) & 1)), ((j - 1) >> 1) & 1, abort_flag, p.status, 42);
                        tc_fence_after();
#pragma unroll
                        for (int c = 0; c < kOC / kOP; ++c) {
                            uint32_t o[kOP];
                            tmem_ld<kOP>(tO + c * kOP, o);
                            tmem_wait_ld();
#pragma unroll
                            for (int i = 0; i < kOP; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                            tmem_st<kOP>(tO + c * kOP, o);
                        }
                    }
                    m = m_new;
                    m_moved = true;
                }

                // ---- P = 2^(s c1 + bias - m), row sum ----
                const uint64_t neg_m = pack_f32x2(-m, -m);
                uint64_t sum2 = pack_f32x2(0.f, 0.f);
                auto exp_chunk = [&](int c, const uint32_t (&sr)[kCW], const uint4 (&ws)[kCW / 16], auto rag, auto ref) {
                    [[maybe_unused]] uint32_t hl[kCW];   // precise variant: hi terms of the chunk, then its lo terms
#pragma unroll
                    for (int q = 0; q < kCW / 8; ++q) {
                        const uint4& ww = ws[q >> 1];
                        float bb[8];
                        lookup8((q & 1) ? ww.z : ww.x, (q & 1) ? ww.w : ww.y, bb);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            float lo, hi;
                            uint64_t x = fma_f32x2(pack_u32x2(sr[q * 8 + 2 * i], sr[q * 8 + 2 * i + 1]), c1c1, pack_f32x2(bb[2 * i], bb[2 * i + 1]));
                            if constexpr (decltype(ref)::value) x = add_f32x2(x, neg_m);
                            unpack_f32x2(x, lo, hi);
                            if constexpr (decltype(rag)::value) {
                                const int col = c * kCW + q * 8 + 2 * i;
                                if (col >= valid) lo = -INFINITY;
                                if (col + 1 >= valid) hi = -INFINITY;
                            }
                            lo = ex2_approx(lo);
                            hi = ex2_approx(hi);
                            sum2 = add_f32x2(sum2, pack_f32x2(lo, hi));
                            const uint32_t top = pack_bf16x2(lo, hi);
                            if constexpr (kPrecise) {
                                hl[q * 4 + i] = top;
                                hl[kCW / 2 + q * 4 + i] = pack_bf16x2(lo - __uint_as_float(top << 16), hi - __uint_as_float(top & 0xffff0000u));
                            } else {
                                pk[(c * (kCW / 2) + q * 4 + i) >> 5][(c * (kCW / 2) + q * 4 + i) & 31] = top;
                            }
                        }
                    }
                    if constexpr (kPrecise) tmem_st<kCW>(tS + c * kCW, hl);      // over the chunk's own score columns (already in registers)
                };
                auto exp_pass = [&](auto rag, auto ref) {
                    if (!loaded) load_chunk(0, sa, wa);
                    tmem_wait_ld(); load_chunk(1, sb, wb); exp_chunk(0, sa, wa, rag, ref);
                    tmem_wait_ld(); load_chunk(2, sa, wa); exp_chunk(1, sb, wb, rag, ref);
                    tmem_wait_ld(); load_chunk(3, sb, wb); exp_chunk(2, sa, wa, rag, ref);
                    tmem_wait_ld(); exp_chunk(3, sb, wb, rag, ref);
                };
                if (ragged) exp_pass(BoolTag<true>{}, BoolTag<true>{});
                else if (!kOwnFormAtZero || m_moved) exp_pass(BoolTag<false>{}, BoolTag<true>{});
                else exp_pass(BoolTag<false>{}, BoolTag<false>{});
                loaded = false;
                {
                    float lo, hi;
                    unpack_f32x2(sum2, lo, hi);
                    tile_sum = lo + hi;
                }
                if (kPrecise || exact) break;
                // reference too low for some row of this warp (pair of warps)?  Also catches inf / NaN.
                const bool need = !(tile_sum <= kSumThreshold);
                if (!named_barrier_or(pair_bar, 64, need)) break;
                exact = true;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kBarSpdEmpty + (j % kSpdStages)));
            if constexpr (!kFold) l += tile_sum;

            // P over the first half of this thread's own score columns
            if constexpr (!kPrecise) {
#pragma unroll
                for (int c = 0; c < kCols / 64; ++c) tmem_st32(tS + c * 32, pk[c]);
            }
            tmem_wait_st();
            if constexpr (kFold) {
                if (j == next_chunk) {          // the chunk before joins the sum; PV(j) then overwrites it
                    mbar_wait(bar(kBarODone + 2 * t + ((j - 1) & 1)), ((j - 1) >> 1) & 1, abort_flag, p.status, 44);
                    tc_fence_after();
                    float4* const sum = o_sum();
                    uint32_t o[kOC];
                    tmem_ld<kOC>(tO, o);
                    tmem_wait_ld();
                    if (j == p.chunk_tiles) {
#pragma unroll
                        for (int i = 0; i < kOC / 4; ++i) *(uint4*)&sum[i * kSumStep] = make_uint4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
                    } else {
                        const float m_sum = sums->x;
                        if (__any_sync(0xffffffffu, m != m_sum)) {
                            const float w = ex2_approx(m_sum - m);
#pragma unroll 1
                            for (int i = 0; i < kOC / 4; ++i) {
                                float4 a = __ldcg(&sum[i * kSumStep]);
                                a.x *= w; a.y *= w; a.z *= w; a.w *= w;
                                sum[i * kSumStep] = a;
                            }
                        }
#pragma unroll
                        for (int i = 0; i < kOC / 4; ++i) red_add_f32x4(&sum[i * kSumStep], o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
                    }
                    if (j > p.chunk_tiles) l += sums->y * ex2_approx(sums->x - m);
                    *sums = make_float2(m, l);
                    l = 0.f;
                    next_chunk += p.chunk_tiles;
                }
                l += tile_sum;
            }
            tc_fence_before();
            // Warps of a tile can be one step apart (nothing in the speculative pass waits for the
            // previous PV MMA), so odd and even key tiles use different barriers, here and for the
            // completion of the PV MMAs: a parity wait can only tell two states apart.  Two steps
            // apart is impossible because S(j+2) needs a score buffer that is only freed after PV(j).
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(kBarPFull + 2 * t + (j & 1)));
            if (j + 1 < n_kv) begin_tile(j + 1);
        }

        // ---- epilogue: O / l, LSE ----
        mbar_wait(bar(kBarODone + 2 * t + ((n_kv - 1) & 1)), ((n_kv - 1) >> 1) & 1, abort_flag, p.status, 43);
        tc_fence_after();
        [[maybe_unused]] float w_sum = 0.f;
        [[maybe_unused]] const bool summed = kFold && n_kv > p.chunk_tiles;
        if (summed) {
            w_sum = ex2_approx(sums->x - m);
            l += sums->y * w_sum;
        }
        xchg[256 + hf * 128 + r] = l;
        named_barrier_sync(pair_bar, 64);
        l += xchg[256 + (hf ^ 1) * 128 + r];
        const int32_t q = q0 + t * kRowsPerTile + r;
        const float inv_l = 1.0f / l;
        const float lse_nat = kFold ? m * kLn2 + logf(l) : (m + log2f(l)) * kLn2;       // (the merge of shares took a natural logarithm, too)
        if (kShared && sharers > 1) {
            // This block's share of O, not normalised, and its m and l, to its own shared memory (over K and V: every MMA is done).
#pragma unroll
            for (int c = 0; c < kOC / kOP; ++c) {
                uint32_t o[kOP];
                tmem_ld<kOP>(tO + c * kOP, o);
                tmem_wait_ld();
                uint4* part = (uint4*)(smem + L::kK) + ((hf * kOC + c * kOP) / 4) * 128 + r;
#pragma unroll
                for (int i = 0; i < kOP / 4; ++i) part[i * 128] = make_uint4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
            }
            if (hf == 0) *(float2*)(smem + L::kXchg + 512 * 4 + r * 8) = make_float2(m, l);
        } else if (kPartial && !kFold && p.state_o != nullptr) {
            // Merge into the carried state: lse' = log(e^lse0 + e^lse), o' = e^(lse0-lse') o0 + e^(lse-lse') o.
            const bool mine = q >= p.state_q_begin && q < p.state_q_end;
            float* lse_ptr = p.state_lse + (size_t)h * p.n_total + q;
            const float l0 = mine ? *lse_ptr : -INFINITY;
            named_barrier_sync(pair_bar, 64);   // both column halves have read lse0 before it is rewritten
            const float mx = fmaxf(l0, lse_nat);
            const float e0 = l0 == -INFINITY ? 0.f : exp2f((l0 - mx) * kLog2e);
            const float e1 = exp2f((lse_nat - mx) * kLog2e);
            const float inv = 1.0f / (e0 + e1);
            const float w0 = e0 * inv, w1 = e1 * inv * inv_l;
#pragma unroll
            for (int c = 0; c < kOC / kOP; ++c) {
                uint32_t o[kOP];
                tmem_ld<kOP>(tO + c * kOP, o);
                tmem_wait_ld();
                if (mine) {
                    float4* st = (float4*)(p.state_o + ((size_t)q * p.n_heads + h) * D + hf * kOC + c * kOP);
                    uint2* ob = p.out ? (uint2*)(p.out + ((size_t)q * p.n_heads + h) * D + hf * kOC + c * kOP) : nullptr;
#pragma unroll
                    for (int i = 0; i < kOP / 4; ++i) {
                        float4 a = make_float4(__uint_as_float(o[4 * i]) * w1, __uint_as_float(o[4 * i + 1]) * w1,
                                               __uint_as_float(o[4 * i + 2]) * w1, __uint_as_float(o[4 * i + 3]) * w1);
                        if (e0 != 0.f) {
                            const float4 b = st[i];
                            a.x += w0 * b.x; a.y += w0 * b.y; a.z += w0 * b.z; a.w += w0 * b.w;
                        }
                        st[i] = a;
                        if (ob) ob[i] = make_uint2(pack_bf16x2(a.x, a.y), pack_bf16x2(a.z, a.w));
                    }
                }
            }
            if (mine && hf == 0) *lse_ptr = mx + log2f(e0 + e1) * kLn2;
        } else {
#pragma unroll
        for (int c = 0; c < kOC / kOP; ++c) {
            uint32_t o[kOP];
            tmem_ld<kOP>(tO + c * kOP, o);
            tmem_wait_ld();
            if (summed) {
#pragma unroll
                for (int i = 0; i < kOP / 4; ++i) {
                    const float4 a = __ldcg(&o_sum()[(c * (kOP / 4) + i) * kSumStep]);
                    o[4 * i] = __float_as_uint(__uint_as_float(o[4 * i]) + w_sum * a.x);
                    o[4 * i + 1] = __float_as_uint(__uint_as_float(o[4 * i + 1]) + w_sum * a.y);
                    o[4 * i + 2] = __float_as_uint(__uint_as_float(o[4 * i + 2]) + w_sum * a.z);
                    o[4 * i + 3] = __float_as_uint(__uint_as_float(o[4 * i + 3]) + w_sum * a.w);
                }
            }
            if (q < n_g) {
                if (kPartial) {
                    float4* dst = (float4*)(p.part_o + (((size_t)chunk * p.n_total + q) * p.n_heads + h) * D + hf * kOC + c * kOP);
#pragma unroll
                    for (int i = 0; i < kOP / 4; ++i)
                        *(kFold ? &o_sum()[(c * (kOP / 4) + i) * kSumStep] : &dst[i]) = make_float4(__uint_as_float(o[4 * i]) * inv_l, __uint_as_float(o[4 * i + 1]) * inv_l,
                                             __uint_as_float(o[4 * i + 2]) * inv_l, __uint_as_float(o[4 * i + 3]) * inv_l);
                } else {
                    uint4* dst = (uint4*)(p.out + ((size_t)(node0 + q) * p.n_heads + h) * D + hf * kOC + c * kOP);
#pragma unroll
                    for (int i = 0; i < kOP / 8; ++i) {
                        uint4 v;
                        v.x = pack_bf16x2(__uint_as_float(o[8 * i]) * inv_l, __uint_as_float(o[8 * i + 1]) * inv_l);
                        v.y = pack_bf16x2(__uint_as_float(o[8 * i + 2]) * inv_l, __uint_as_float(o[8 * i + 3]) * inv_l);
                        v.z = pack_bf16x2(__uint_as_float(o[8 * i + 4]) * inv_l, __uint_as_float(o[8 * i + 5]) * inv_l);
                        v.w = pack_bf16x2(__uint_as_float(o[8 * i + 6]) * inv_l, __uint_as_float(o[8 * i + 7]) * inv_l);
                        dst[i] = v;
                    }
                    if (p.out_f32 != nullptr) {
                        float4* dst32 = (float4*)(p.out_f32 + ((size_t)(node0 + q) * p.n_heads + h) * D + hf * kOC + c * kOP);
#pragma unroll
                        for (int i = 0; i < kOP / 4; ++i)
                            dst32[i] = make_float4(__uint_as_float(o[4 * i]) * inv_l, __uint_as_float(o[4 * i + 1]) * inv_l,
                                                   __uint_as_float(o[4 * i + 2]) * inv_l, __uint_as_float(o[4 * i + 3]) * inv_l);
                    }
                }
            }
        }
        if (q < n_g && hf == 0) {
            if (kPartial) p.part_lse[((size_t)chunk * p.n_heads + h) * p.n_total + q] = lse_nat;
            else p.lse[(size_t)h * p.n_total + node0 + q] = lse_nat;
        }
        }
    }

    // ---- teardown ----
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) __nanosleep(200000);    // let copies that may still be in flight land
    if (warp == 1) tmem_dealloc(tmem, kTmemCols);
    if (kShared && sharers > 1) {
        // Every block merges its part of the rows' channels from all blocks' shares.
        cluster_sync();
        constexpr int kPieces = (D / 4) * 128;           // of four channels of a row
        const int per = (kPieces + sharers - 1) / sharers;
        for (int i = rank * per + tid; i < min(kPieces, (rank + 1) * per); i += kThreads) {
            const int row = i & 127, c4 = i >> 7;
            const uint32_t at = smem_u32(smem + L::kK) + (uint32_t)i * 16u, at_ml = smem_u32(smem + L::kXchg) + 512u * 4u + (uint32_t)row * 8u;
            float2 ml[kMaxSplit];
            float mx = -INFINITY;
#pragma unroll
            for (int k = 0; k < kMaxSplit; ++k) {
                ml[k] = k < sharers ? ld_cluster_float2(at_ml, (uint32_t)k) : make_float2(-INFINITY, 0.f);
                mx = fmaxf(mx, ml[k].x);
            }
            float den = 0.f;
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int k = 0; k < kMaxSplit; ++k) {
                if (ml[k].x == -INFINITY && mx != -INFINITY) continue;       // no such block, or nothing to attend to among its keys
                if (k >= sharers) continue;
                const float w = ex2_approx(ml[k].x - mx);                    // references are whole numbers: a power of two
                const float4 b = ld_cluster_float4(at, (uint32_t)k);
                den += w * ml[k].y;
                a.x += w * b.x; a.y += w * b.y; a.z += w * b.z; a.w += w * b.w;
            }
            const int32_t q = q0 + row;
            if (q >= n_g) continue;
            const float inv = 1.0f / den;
            a.x *= inv; a.y *= inv; a.z *= inv; a.w *= inv;
            const size_t to = ((size_t)(node0 + q) * p.n_heads + h) * D + c4 * 4;
            *(uint2*)(p.out + to) = make_uint2(pack_bf16x2(a.x, a.y), pack_bf16x2(a.z, a.w));
            if (kPrecise && p.out_f32 != nullptr) *(float4*)(p.out_f32 + to) = a;
            if (c4 == 0) p.lse[(size_t)h * p.n_total + node0 + q] = (mx + log2f(den)) * kLn2;
        }
        cluster_sync();                                  // no block leaves while another reads its share
    }
}

// Merge of per-chunk partials: lse = log sum_c exp(lse_c), out = sum_c exp(lse_c - lse) out_c.
// One thread per (row, head, 4 channels).
template <int D>
__global__ void chunk_merge_kernel(const float* __restrict__ part_o, const float* __restrict__ part_lse,
                                   __nv_bfloat16* __restrict__ out, float* __restrict__ lse, float* __restrict__ lse_chunks,
                                   int32_t n_total, int32_t n_heads, int32_t n_chunks)
{
    grid_wait();
    grid_release();
    constexpr int kVec = D / 4;
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t n_rows = (size_t)n_total * n_heads;
    if (idx >= n_rows * kVec) return;
    const size_t rh = idx / kVec;
    const int v = (int)(idx % kVec);
    const int32_t row = (int32_t)(rh / n_heads), h = (int32_t)(rh % n_heads);
    float mx = -INFINITY;
    for (int c = 0; c < n_chunks; ++c) mx = fmaxf(mx, part_lse[((size_t)c * n_heads + h) * n_total + row]);
    float den = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c = 0; c < n_chunks; ++c) {
        const float lc = part_lse[((size_t)c * n_heads + h) * n_total + row];
        if (v == 0 && lse_chunks) lse_chunks[((size_t)c * n_heads + h) * n_total + row] = lc;
        if (lc == -INFINITY) continue;                      // empty chunk: weight 0 (no inf - inf)
        const float w = exp2f((lc - mx) * kLog2e);
        den += w;
        const float4 o = *(const float4*)(part_o + (((size_t)c * n_total + row) * n_heads + h) * D + v * 4);
        acc.x += w * o.x; acc.y += w * o.y; acc.z += w * o.z; acc.w += w * o.w;
    }
    const float inv = 1.0f / den;
    uint2 pk;
    pk.x = pack_bf16x2(acc.x * inv, acc.y * inv);
    pk.y = pack_bf16x2(acc.z * inv, acc.w * inv);
    *(uint2*)(out + ((size_t)row * n_heads + h) * D + v * 4) = pk;
    if (v == 0) lse[(size_t)h * n_total + row] = mx + logf(den);
}

// The same for shares in the layout of FwdParams::chunk_sums, in thread blocks of 256 rows: block (rows and head, 16 channels).
template <int D>
__global__ void __launch_bounds__(kRowsPerCta) share_merge_kernel(const float4* __restrict__ sums, const float* __restrict__ part_lse, __nv_bfloat16* __restrict__ out,
                                                                  float* __restrict__ lse, int32_t n_total, int32_t n_heads, int32_t n_shares)
{
    grid_wait();
    grid_release();
    constexpr int kOC = D / kHalves;
    const int h = (int)(blockIdx.x % (unsigned)n_heads), row = (int)threadIdx.x, c = (int)blockIdx.y * 16;
    const int32_t q = (int32_t)(blockIdx.x / (unsigned)n_heads) * kRowsPerCta + row;
    if (q >= n_total) return;
    auto lse_of = [&](int k) -> float { return part_lse[((size_t)k * n_heads + h) * n_total + q]; };
    float mx = -INFINITY;
    for (int k = 0; k < n_shares; ++k) mx = fmaxf(mx, lse_of(k));
    float den = 0.f;
    float4 acc[4] = {};
    for (int k = 0; k < n_shares; ++k) {
        const float lc = lse_of(k);
        if (lc == -INFINITY) continue;
        const float w = exp2f((lc - mx) * kLog2e);
        den += w;
        const float4* src = sums + (((size_t)k * gridDim.x + blockIdx.x) * (kOC / 4) + (c % kOC) / 4) * 512 + (row / 128) * 256 + (c / kOC) * 128 + row % 128;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 o = src[i * 512];
            acc[i].x += w * o.x; acc[i].y += w * o.y; acc[i].z += w * o.z; acc[i].w += w * o.w;
        }
    }
    const float inv = 1.0f / den;
    uint4 pk[2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
        pk[i] = make_uint4(pack_bf16x2(acc[2 * i].x * inv, acc[2 * i].y * inv), pack_bf16x2(acc[2 * i].z * inv, acc[2 * i].w * inv),
                           pack_bf16x2(acc[2 * i + 1].x * inv, acc[2 * i + 1].y * inv), pack_bf16x2(acc[2 * i + 1].z * inv, acc[2 * i + 1].w * inv));
    uint4* to = (uint4*)(out + ((size_t)q * n_heads + h) * D + c);
    to[0] = pk[0];
    to[1] = pk[1];
    if (c == 0) lse[(size_t)h * n_total + q] = mx + logf(den);
}

// One ring step's merge: the carried state (normalised accumulator o_acc, lse_acc) of the query rows
// [q_begin, q_end) absorbs up to two partial results (the step's regular key range and its super-node
// range):  lse' = log sum exp(lse_i),  o' = sum exp(lse_i - lse') o_i.  Rows with nothing to attend to yet
// keep lse = -inf, o = 0.  One thread per (row, head, 4 channels).
template <int D>
__global__ void step_merge_kernel(const float* __restrict__ part_o, const float* __restrict__ part_lse, int32_t n_parts,
                                  float* __restrict__ o_acc, float* __restrict__ lse_acc, __nv_bfloat16* __restrict__ out,
                                  int32_t q_begin, int32_t q_end, int32_t n_total, int32_t n_heads)
{
    grid_wait();
    grid_release();
    constexpr int kVec = D / 4;
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t n_rows = (size_t)(q_end - q_begin) * n_heads;
    if (idx >= n_rows * kVec) return;
    const size_t rh = idx / kVec;
    const int v = (int)(idx % kVec);
    const int32_t row = q_begin + (int32_t)(rh / n_heads), h = (int32_t)(rh % n_heads);
    const float l0 = lse_acc[(size_t)h * n_total + row];
    float mx = l0;
    for (int c = 0; c < n_parts; ++c) mx = fmaxf(mx, part_lse[((size_t)c * n_heads + h) * n_total + row]);
    float4* acc_ptr = (float4*)(o_acc + ((size_t)row * n_heads + h) * D + v * 4);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    float den = 0.f;
    if (mx != -INFINITY) {
        if (l0 != -INFINITY) {
            const float w = exp2f((l0 - mx) * kLog2e);
            const float4 o = *acc_ptr;
            den += w;
            acc.x += w * o.x; acc.y += w * o.y; acc.z += w * o.z; acc.w += w * o.w;
        }
        for (int c = 0; c < n_parts; ++c) {
            const float lc = part_lse[((size_t)c * n_heads + h) * n_total + row];
            if (lc == -INFINITY) continue;
            const float w = exp2f((lc - mx) * kLog2e);
            const float4 o = *(const float4*)(part_o + (((size_t)c * n_total + row) * n_heads + h) * D + v * 4);
            den += w;
            acc.x += w * o.x; acc.y += w * o.y; acc.z += w * o.z; acc.w += w * o.w;
        }
        const float inv = 1.0f / den;
        acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
    }
    *acc_ptr = acc;
    if (out) {
        uint2 pk;
        pk.x = pack_bf16x2(acc.x, acc.y);
        pk.y = pack_bf16x2(acc.z, acc.w);
        *(uint2*)(out + ((size_t)row * n_heads + h) * D + v * 4) = pk;
    }
    __syncwarp();
    if (v == 0) lse_acc[(size_t)h * n_total + row] = mx == -INFINITY ? -INFINITY : mx + logf(den);
}

int32_t chunk_rows(int32_t n, int32_t n_chunks)
{
    int32_t w = (n + n_chunks - 1) / n_chunks;
    return (w + kKvTile - 1) / kKvTile * kKvTile;
}

constexpr size_t kListMinSaved = 128;     // thread blocks

// Largest |k|^2 of every kNormRows rows of a head: block (row block, head), D / 8 lanes per row.  Bound by its launch (8 192 rows,
// 8 heads: 3 us for 8 MB).
template <int D>
__global__ void __launch_bounds__(256) key_norms_kernel(const uint4* __restrict__ k, float* __restrict__ norms, int32_t n_total, int32_t n_heads)
{
    constexpr int kLanes = D / 8, kRowsAtOnce = 256 / kLanes;
    __shared__ float part[8];
    grid_wait();
    grid_release();
    const int part_of_row = threadIdx.x % kLanes, first = blockIdx.x * kNormRows + threadIdx.x / kLanes;
    uint4 v[kNormRows / kRowsAtOnce];
#pragma unroll
    for (int i = 0; i < kNormRows / kRowsAtOnce; ++i) {
        const int row = first + i * kRowsAtOnce;
        v[i] = row < n_total ? k[((size_t)row * n_heads + blockIdx.y) * kLanes + part_of_row] : make_uint4(0, 0, 0, 0);
    }
    float best = 0.f;
#pragma unroll
    for (int i = 0; i < kNormRows / kRowsAtOnce; ++i) {
        float a = square_sum(v[i]);
#pragma unroll
        for (int off = kLanes / 2; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
        best = norm_max(best, a);
    }
#pragma unroll
    for (int off = 16; off >= kLanes; off >>= 1) best = norm_max(best, __shfl_xor_sync(0xffffffffu, best, off));
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) best = norm_max(best, part[w]);
        norms[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = best;
    }
}

inline size_t norms_bytes(const gt_batch* b, int32_t n_heads) { return (size_t)((b->n_total + kNormRows - 1) / kNormRows) * (size_t)n_heads * sizeof(float); }
// Precise forward: a tile saves half its softmax time (1 us) from the second one of a graph on; the norms cost about 3 us.
constexpr int32_t kNormsMinNodes = 513;

// Tensor maps of a packed batch, a thread per graph, behind its work list (unless `list` is null), a warp per graph.
constexpr int kBatchThreads = 128;
template <int kRows>
__global__ void __launch_bounds__(kBatchThreads) fwd_batch_kernel(const __grid_constant__ CUtensorMap model, uint8_t* maps, int4* list, int32_t entries,
                                                                  const uint8_t* spd, const int64_t* spd_offsets, const int32_t* cu_seqlens, int32_t n_graphs)
{
    grid_wait();
    grid_release();
    int32_t w = (int32_t)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (list != nullptr) {
        if (w < n_graphs) {
            write_work_list<kRows>(list, entries, cu_seqlens, n_graphs, w);
            return;
        }
        w -= n_graphs;
    }
    const int32_t g = w * 32 + (int32_t)(threadIdx.x & 31);
    if (g >= n_graphs) return;
    const int32_t n = cu_seqlens[g + 1] - cu_seqlens[g];
    if (n > 0) make_spd_map(maps + (size_t)g * kMapBytes, model, spd + spd_offsets[g], n);
}

// Rows per thread block.  One tile where the grid of two would leave at least half of the SMs idle: the softmax of a tile is bound
// by its SM's issue slots and exponentials, so two SMs with a tile each are faster than one with both: 1 000 nodes, 8 heads of 64:
// 19.5 -> 13.8 us; 2 048 nodes 31.8 -> 23.0; 4 096 nodes, 4 heads: 56.4 -> 40.3; up to 256 nodes no difference.
inline int32_t rows_per_block(const gt_batch* b, int32_t n_heads)
{
    return (int64_t)((b->max_seqlen + kRowsPerTile - 1) / kRowsPerTile) * b->n_graphs * n_heads <= sm_count() ? kRowsPerTile : kRowsPerCta;
}

// Chunks of a chunked forward that the same thread blocks take one behind the other.  Blocks of several fill and drain less often and leave
// fewer shares to merge; more blocks fill the grid's last wave better.  `room`: floats in the workspace for the shares.  A 256 x 128 tile
// takes 1.50 to 1.61 us (heads of 32 and of 64), a 128 x 128 tile 1.0 where all blocks are of one, a block's fill and drain 7, an addition
// to the sums 0.9 to 2.5, the merge 3 and its bytes (5 TB/s).  us with every chunk in blocks of its own -> by this rule, 8 chunks: 8 heads of
// 64: 4 096 nodes 110 -> 66 (one share), 10 000 nodes 466 -> 380 (two), 65 536 nodes 14 060 -> 13 660 (one); 4 heads: 6 000 nodes 111 -> 78
// (three), 4 096 nodes 62 -> 42 (one-tile blocks); 5 000 nodes, 5 chunks stay with 69 (98 in one share).
int32_t chunks_in_turn(const gt_batch* b, int32_t n_heads, int32_t head_dim, int32_t n_chunks, int32_t chunk_tiles, size_t room)
{
    const int64_t n = b->n_total, sms = sm_count(), blocks = (n + kRowsPerCta - 1) / kRowsPerCta * n_heads, tiles = (n + kKvTile - 1) / kKvTile;
    const bool one_tile = rows_per_block(b, n_heads) == kRowsPerTile;
    int32_t best = n_chunks;
    double least = one_tile ? 1.0 * tiles + 0.8 * (n_chunks - 1) + 7.0 : 1e30;
    for (int32_t shares = 1; shares <= n_chunks && shares <= 64; ++shares) {
        const int32_t per = (n_chunks + shares - 1) / shares;
        if ((n_chunks + per - 1) / per != shares) continue;                // (the same as fewer shares)
        if (shares == 1 && one_tile) continue;
        if (shares > 1 && per > 1 && (size_t)shares * blocks * kRowsPerCta * head_dim > room) continue;
        const int64_t longest = std::min<int64_t>(tiles, (int64_t)per * chunk_tiles);
        double us = (double)((blocks * shares + sms - 1) / sms) * (1.55 * longest + 1.5 * (per - 1) + 7.0);
        if (shares > 1) us += 3.0 + 8e-6 / 5.0 * shares * (double)n * n_heads * head_dim;
        if (us < 0.97 * least) {
            best = per;
            least = us;
        }
    }
    return best;
}

// Two blocks of one tile per SM, for packed batches of small graphs.  A block of ten key tiles spends a quarter of its time filling and draining,
// and padding of 256 rows is more than half of a graph of a hundred; a tile itself takes a fifth longer, with one score buffer.
// Graphs and nodes each, heads of d: 64 of 16-300, 4 of 32: 25.7 -> 21.2 us; 200 of 64-1 000, 4 of 32: 217 -> 209; 20 of 1 000-1 100, 8 of 64:
// 129 -> 120; but 64 of 512-2 048, 16 of 64: 1 035 -> 1 076, and where every block has an SM of its own: 8 of 500-600, 2 of 64: 14.9 -> 16.1.
constexpr int32_t kPairMaxNodes = 1152;
constexpr int kPairRegisters = 80;           // per thread at launch: what setmaxnreg shares out, which would wait forever for more than there are
template <int D>
auto pair_kernel(bool shfl, bool precise)
{
    if (precise) return shfl ? attn_fwd_kernel<D, false, true, true, 1, true> : attn_fwd_kernel<D, false, false, true, 1, true>;
    return shfl ? attn_fwd_kernel<D, false, true, false, 1, true> : attn_fwd_kernel<D, false, false, false, 1, true>;
}
template <int D>
bool pair_registers(bool shfl, bool precise)
{
    static std::atomic<int> registers[4] = {};               // as compiled (allocated in eights); 0: not asked yet
    std::atomic<int>& known = registers[(shfl ? 1 : 0) + (precise ? 2 : 0)];
    int n = known.load(std::memory_order_relaxed);
    if (n == 0) {
        cudaFuncAttributes a;
        if (cudaFuncGetAttributes(&a, pair_kernel<D>(shfl, precise)) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        n = (a.numRegs + 7) / 8 * 8;
        known.store(n, std::memory_order_relaxed);
    }
    return n >= kPairRegisters;
}
inline bool small_graphs(const gt_batch* b) { return b->n_graphs > 1 && b->max_seqlen <= kPairMaxNodes; }
inline size_t fwd_workspace(const gt_batch* b, int32_t n_heads, int32_t list_rows)
{
    return kHeaderBytes + maps_bytes(b->n_graphs) + list_bytes(b, list_rows) + norms_bytes(b, n_heads);
}
// A workspace without room for a list by 128 rows is used as for large graphs, and so is everything if the kernel came out with too few registers.
inline bool pairs_of_blocks(const gt_batch* b, int32_t n_heads, int32_t head_dim, int32_t n_buckets, bool precise, size_t workspace_bytes)
{
    return small_graphs(b) && rows_per_block(b, n_heads) == kRowsPerCta && workspace_bytes >= fwd_workspace(b, n_heads, kRowsPerTile) &&
           (head_dim == 64 ? pair_registers<64>(n_buckets <= 32, precise) : pair_registers<32>(n_buckets <= 32, precise));
}

// Blocks that share a query tile's keys (cluster_split): a key tile takes 1.2 us, the cluster and the merge 2 to 3 us.  1 000 nodes, heads
// of 64: 8 heads 13.9 -> 12.6 us, 4 heads 13.7 -> 10.8; 2 048 nodes, 4 heads 22.3 -> 17.1; 512 nodes, 8 heads 10.5 -> 10.7; 8 graphs of
// 500 nodes, 2 heads 11.6 -> 12.2: from six key tiles on.
constexpr int32_t kMinSplitTiles = 6;

template <int D, bool kPartial>
gt_status launch_fwd(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tspd,
                     FwdParams p, const gt_batch* batch, int grid_z, cudaStream_t s, int grid_y = 0, bool pair = false)
{
    const bool shfl = p.n_buckets <= 32, in_turn = p.chunk_sums != nullptr;
    const int32_t rows = kPartial ? kRowsPerCta : pair ? kRowsPerTile : rows_per_block(batch, p.n_heads);
    auto kern = shfl ? attn_fwd_kernel<D, kPartial, true> : attn_fwd_kernel<D, kPartial, false>;
    if (in_turn) kern = shfl ? attn_fwd_kernel<D, kPartial, true, false, kQTiles, false, true> : attn_fwd_kernel<D, kPartial, false, false, kQTiles, false, true>;
    if constexpr (!kPartial) {
        if (p.out_f32 != nullptr) kern = shfl ? attn_fwd_kernel<D, false, true, true> : attn_fwd_kernel<D, false, false, true>;
        if (rows == kRowsPerTile) {
            kern = shfl ? attn_fwd_kernel<D, false, true, false, 1> : attn_fwd_kernel<D, false, false, false, 1>;
            if (p.out_f32 != nullptr) kern = shfl ? attn_fwd_kernel<D, false, true, true, 1> : attn_fwd_kernel<D, false, false, true, 1>;
        }
        if (in_turn && rows == kRowsPerTile) kern = shfl ? attn_fwd_kernel<D, false, true, false, 1, false, true> : attn_fwd_kernel<D, false, false, false, 1, false, true>;
        if (pair) kern = pair_kernel<D>(shfl, p.out_f32 != nullptr);
    }
    const size_t smem = pair ? FwdSmem<D, true>::kDynamic : FwdSmem<D>::kDynamic;
    static std::atomic<uint64_t> granted[16] = {};
    static ClusterFit max_clusters[4];
    const int form = (shfl ? 1 : 0) + (!kPartial && p.out_f32 ? 2 : 0);
    const gt_status st = grant_smem(kern, granted[form + (in_turn ? (rows == kRowsPerTile ? 14 : 12) : pair ? 8 : rows == kRowsPerTile ? 4 : 0)], smem);
    if (st != GT_OK) return st;
    const int32_t row_blocks = grid_y > 0 ? grid_y : (batch->max_seqlen + rows - 1) / rows;
    dim3 grid = p.list ? dim3((unsigned)(list_entries(batch, rows) * p.n_heads))
                       : dim3((unsigned)p.n_heads, (unsigned)row_blocks, (unsigned)grid_z);
    p.split = 1;
    const int32_t tiles = (batch->max_seqlen + kKvTile - 1) / kKvTile;
    if (!pair && !in_turn && rows == kRowsPerTile && tiles >= kMinSplitTiles)
        p.split = cluster_split(kern, 128 + 2 * rows, smem, max_clusters[form], (int64_t)grid.x * grid.y * grid.z, tiles, 3.0f, 2.0f);
    grid.x *= (unsigned)p.split;
    // As in the backward: with several waves of blocks the next kernel's blocks take SMs that the last wave frees one by one, and a
    // backward behind this forward starts ragged (forward and backward, 8 heads of 64: 14 000 nodes 2 452 -> 2 329 us, 16 384 nodes
    // 3 400 -> 3 228, 24 000 nodes 7 349 -> 7 176; the forward alone the same).
    p.early_release = (int64_t)grid.x * grid.y * grid.z <= (pair ? 2 : 1) * sm_count();
    return launch_overlapped_cluster(kern, grid, 128 + 2 * rows, smem, p.split, s, tq, tk, tv, tspd, p);
}

gt_status check_fwd_args(const void* q, const void* k, const void* v, const uint8_t* spd, const int64_t* spd_offsets,
                         const float* bias, const gt_batch* batch, int32_t n_heads, int32_t head_dim, int32_t max_dist,
                         void* out, float* lse)
{
    gt_status st = validate_attn_common(batch, n_heads, head_dim, max_dist, spd_offsets);
    if (st != GT_OK) return st;
    if (!q || !k || !v || !spd || !bias || !out || !lse) return GT_ERR_INVALID_ARG;
    if (misaligned16(q) || misaligned16(k) || misaligned16(v) || misaligned16(spd) || misaligned16(out)) return GT_ERR_INVALID_ARG;
    if (n_heads > 65535 || batch->n_graphs > 65535) return GT_ERR_UNSUPPORTED;
    return GT_OK;
}

}  // namespace
}  // namespace gt

extern "C" size_t gt_biased_attn_fwd_workspace(const gt_batch* batch, int32_t n_heads, int32_t head_dim)
{
    (void)head_dim;
    if (gt::validate_batch(batch) != GT_OK || n_heads < 1) return gt::kHeaderBytes;
    return gt::fwd_workspace(batch, n_heads, gt::small_graphs(batch) ? gt::kRowsPerTile : gt::kRowsPerCta);
}

extern "C" gt_status gt_biased_attn_fwd(const void* q, const void* k, const void* v,
                                        const uint8_t* spd, const int64_t* spd_offsets, const float* bias,
                                        const gt_batch* batch, int32_t n_heads, int32_t head_dim, int32_t max_dist,
                                        void* out, float* lse,
                                        void* workspace, size_t workspace_bytes, void* stream)
{
    return gt_biased_attn_fwd_ex(q, k, v, spd, spd_offsets, bias, batch, n_heads, head_dim, max_dist, out, lse, nullptr,
                                 workspace, workspace_bytes, stream);
}

extern "C" gt_status gt_biased_attn_fwd_ex(const void* q, const void* k, const void* v,
                                           const uint8_t* spd, const int64_t* spd_offsets, const float* bias,
                                           const gt_batch* batch, int32_t n_heads, int32_t head_dim, int32_t max_dist,
                                           void* out, float* lse, float* out_f32,
                                           void* workspace, size_t workspace_bytes, void* stream)
{
    using namespace gt;
    gt_status st = check_fwd_args(q, k, v, spd, spd_offsets, bias, batch, n_heads, head_dim, max_dist, out, lse);
    if (st != GT_OK) return st;
    if (out_f32 != nullptr && misaligned16(out_f32)) return GT_ERR_INVALID_ARG;
    if (workspace == nullptr || workspace_bytes < kHeaderBytes || misaligned16(workspace)) return GT_ERR_WORKSPACE;
    if (sm_count() <= 0) return GT_ERR_NO_DEVICE;
    CUtensorMap tq, tk, tv;
    if ((st = encode_thd_map(&tq, q, batch->n_total, n_heads, head_dim)) != GT_OK) return st;
    if ((st = encode_thd_map(&tk, k, batch->n_total, n_heads, head_dim)) != GT_OK) return st;
    if ((st = encode_thd_map(&tv, v, batch->n_total, n_heads, head_dim)) != GT_OK) return st;
    CUtensorMap tspd = tq;                       // placeholder when the cp.async loader is used
    FwdParams p{};
    const bool pair = pairs_of_blocks(batch, n_heads, head_dim, max_dist + 2, out_f32 != nullptr, workspace_bytes);
    const int32_t list_rows = pair ? kRowsPerTile : kRowsPerCta;
    const int32_t rows = pair ? kRowsPerTile : rows_per_block(batch, n_heads);
    p.spd_tma = batch->n_graphs == 1 ? 1 : 0;
    const bool room = workspace_bytes >= fwd_workspace(batch, n_heads, list_rows);
    if (batch->n_graphs > 1 && room) {
        p.maps = maps_at((uint8_t*)workspace + kHeaderBytes);
        // The list costs 1 us before the first block; that has to come back from the empty blocks that it saves.
        if ((pair || rows == kRowsPerCta) && list_saves(batch, rows, n_heads, kListMinSaved))
            p.list = (const int4*)((uint8_t*)workspace + kHeaderBytes + maps_bytes(batch->n_graphs));
        p.spd_tma = 1;
    }
    if (p.spd_tma && (st = encode_spd_map(&tspd, spd, batch->max_seqlen, rows)) != GT_OK) return st;
    p.spd = spd;
    p.spd_offsets = batch->n_graphs > 1 ? spd_offsets : nullptr;
    p.cu_seqlens = batch->n_graphs > 1 ? batch->cu_seqlens : nullptr;
    p.bias = bias;
    p.out = (__nv_bfloat16*)out;
    p.out_f32 = out_f32;
    p.lse = lse;
    p.status = (uint32_t*)workspace;
    p.n_total = batch->n_total;
    p.n_heads = n_heads;
    p.n_buckets = max_dist + 2;
    p.c1 = kLog2e / sqrtf((float)head_dim);
    cudaStream_t s = (cudaStream_t)stream;
    if (out_f32 != nullptr && room && batch->max_seqlen >= kNormsMinNodes) {
        float* norms = (float*)((uint8_t*)workspace + kHeaderBytes + maps_bytes(batch->n_graphs) + list_bytes(batch, list_rows));
        const dim3 grid((unsigned)((batch->n_total + kNormRows - 1) / kNormRows), (unsigned)n_heads);
        st = head_dim == 64 ? launch_overlapped(key_norms_kernel<64>, grid, 256, 0, s, (const uint4*)k, norms, batch->n_total, n_heads)
                            : launch_overlapped(key_norms_kernel<32>, grid, 256, 0, s, (const uint4*)k, norms, batch->n_total, n_heads);
        if (st != GT_OK) return st;
        p.q = (const __nv_bfloat16*)q;
        p.key_norms = norms;
    }
    if (p.maps) {
        const int32_t warps = (batch->n_graphs + 31) / 32 + (p.list ? batch->n_graphs : 0);
        st = launch_overlapped(pair ? fwd_batch_kernel<kRowsPerTile> : fwd_batch_kernel<kRowsPerCta>, dim3((unsigned)((warps * 32 + kBatchThreads - 1) / kBatchThreads)), kBatchThreads, 0, s, tspd,
                               (uint8_t*)p.maps, (int4*)p.list, (int32_t)list_entries(batch, list_rows), spd, p.spd_offsets, p.cu_seqlens, batch->n_graphs);
        if (st != GT_OK) return st;
    }
    return head_dim == 64 ? launch_fwd<64, false>(tq, tk, tv, tspd, p, batch, batch->n_graphs, s, 0, pair)
                          : launch_fwd<32, false>(tq, tk, tv, tspd, p, batch, batch->n_graphs, s, 0, pair);
}

extern "C" size_t gt_biased_attn_fwd_chunked_workspace(const gt_batch* batch, int32_t n_heads, int32_t head_dim,
                                                       int32_t n_kv_chunks)
{
    if (gt::validate_batch(batch) != GT_OK || n_heads < 1 || n_kv_chunks < 1) return 0;
    size_t rows = (size_t)batch->n_total * n_heads;
    return gt::kHeaderBytes + (size_t)n_kv_chunks * rows * head_dim * sizeof(float)
         + gt::align_up((size_t)n_kv_chunks * rows * sizeof(float), 256);
}

extern "C" gt_status gt_biased_attn_fwd_chunked(const void* q, const void* k, const void* v,
                                                const uint8_t* spd, const int64_t* spd_offsets, const float* bias,
                                                const gt_batch* batch, int32_t n_heads, int32_t head_dim, int32_t max_dist,
                                                void* out, float* lse, int32_t n_kv_chunks, float* lse_chunks,
                                                void* workspace, size_t workspace_bytes, void* stream)
{
    using namespace gt;
    gt_status st = check_fwd_args(q, k, v, spd, spd_offsets, bias, batch, n_heads, head_dim, max_dist, out, lse);
    if (st != GT_OK) return st;
    if (n_kv_chunks < 1 || n_kv_chunks > 65535) return GT_ERR_INVALID_ARG;
    if (batch->n_graphs != 1) return GT_ERR_UNSUPPORTED;
    const size_t need = gt_biased_attn_fwd_chunked_workspace(batch, n_heads, head_dim, n_kv_chunks);
    if (workspace == nullptr || workspace_bytes < need || misaligned16(workspace)) return GT_ERR_WORKSPACE;
    if (sm_count() <= 0) return GT_ERR_NO_DEVICE;
    const int32_t width = chunk_rows(batch->n_total, n_kv_chunks), n_filled = (batch->n_total + width - 1) / width;      // (chunks behind those are empty)
    const size_t rows = (size_t)batch->n_total * n_heads, room = (size_t)n_kv_chunks * rows * head_dim;
    const int32_t per = lse_chunks != nullptr ? 1 : chunks_in_turn(batch, n_heads, head_dim, n_filled, width / kKvTile, room);      // (each chunk's own lse is wanted)
    const int32_t shares = lse_chunks != nullptr ? n_kv_chunks : (n_filled + per - 1) / per;
    const bool whole = shares == 1 && lse_chunks == nullptr;                           // nothing to merge
    if (n_filled == 1 && lse_chunks == nullptr)
        return gt_biased_attn_fwd_ex(q, k, v, spd, nullptr, bias, batch, n_heads, head_dim, max_dist, out, lse, nullptr, workspace, workspace_bytes, stream);
    CUtensorMap tq, tk, tv;
    if ((st = encode_thd_map(&tq, q, batch->n_total, n_heads, head_dim)) != GT_OK) return st;
    if ((st = encode_thd_map(&tk, k, batch->n_total, n_heads, head_dim)) != GT_OK) return st;
    if ((st = encode_thd_map(&tv, v, batch->n_total, n_heads, head_dim)) != GT_OK) return st;
    uint8_t* ws = (uint8_t*)workspace;
    CUtensorMap tspd;
    if ((st = encode_spd_map(&tspd, spd, batch->n_total, whole ? rows_per_block(batch, n_heads) : kRowsPerCta)) != GT_OK) return st;
    FwdParams p{};
    p.spd_tma = 1;
    p.spd = spd;
    p.bias = bias;
    p.part_lse = (float*)(ws + kHeaderBytes);
    p.part_o = (float*)(ws + kHeaderBytes + align_up((size_t)n_kv_chunks * rows * sizeof(float), 256));
    if (per > 1) {                               // (one share: there is room for two, which is more than whole blocks of rows take)
        p.chunk_sums = p.part_o;
        p.chunk_tiles = width / kKvTile;
    }
    if (whole) {
        p.out = (__nv_bfloat16*)out;
        p.lse = lse;
    }
    p.status = (uint32_t*)workspace;
    p.n_total = batch->n_total;
    p.n_heads = n_heads;
    p.n_buckets = max_dist + 2;
    p.kv_chunk_rows = width * per;
    p.c1 = kLog2e / sqrtf((float)head_dim);
    cudaStream_t s = (cudaStream_t)stream;
    if (whole)
        return head_dim == 64 ? launch_fwd<64, false>(tq, tk, tv, tspd, p, batch, 1, s) : launch_fwd<32, false>(tq, tk, tv, tspd, p, batch, 1, s);
    st = head_dim == 64 ? launch_fwd<64, true>(tq, tk, tv, tspd, p, batch, shares, s)
                        : launch_fwd<32, true>(tq, tk, tv, tspd, p, batch, shares, s);
    if (st != GT_OK) return st;
    if (per > 1) {
        const dim3 merge((unsigned)((batch->n_total + kRowsPerCta - 1) / kRowsPerCta * n_heads), (unsigned)head_dim / 16);
        return head_dim == 64 ? launch_overlapped(share_merge_kernel<64>, merge, kRowsPerCta, 0, s, (const float4*)p.chunk_sums, p.part_lse, (__nv_bfloat16*)out, lse, batch->n_total, n_heads, shares)
                              : launch_overlapped(share_merge_kernel<32>, merge, kRowsPerCta, 0, s, (const float4*)p.chunk_sums, p.part_lse, (__nv_bfloat16*)out, lse, batch->n_total, n_heads, shares);
    }
    const size_t n_thr = rows * (head_dim / 4);
    const unsigned blocks = (unsigned)((n_thr + 255) / 256);
    if (head_dim == 64)
        st = launch_overlapped(chunk_merge_kernel<64>, dim3(blocks), 256, 0, s, p.part_o, p.part_lse, (__nv_bfloat16*)out, lse, lse_chunks,
                                                      batch->n_total, n_heads, shares);
    else
        st = launch_overlapped(chunk_merge_kernel<32>, dim3(blocks), 256, 0, s, p.part_o, p.part_lse, (__nv_bfloat16*)out, lse, lse_chunks,
                                                      batch->n_total, n_heads, shares);
    return st;
}

extern "C" size_t gt_biased_attn_fwd_step_workspace(const gt_batch* batch, int32_t n_heads, int32_t head_dim)
{
    return gt_biased_attn_fwd_chunked_workspace(batch, n_heads, head_dim, 2);
}

extern "C" gt_status gt_biased_attn_fwd_step(const void* q, const void* k, const void* v,
                                             const uint8_t* spd, const float* bias,
                                             const gt_batch* batch, int32_t n_heads, int32_t head_dim, int32_t max_dist,
                                             int32_t q_begin, int32_t q_end,
                                             int32_t kv_begin0, int32_t kv_end0, int32_t kv_begin1, int32_t kv_end1,
                                             float* o_acc, float* lse_acc, void* out,
                                             void* workspace, size_t workspace_bytes, void* stream)
{
    using namespace gt;
    gt_status st = validate_attn_common(batch, n_heads, head_dim, max_dist, nullptr);
    if (st != GT_OK) return st;
    if (!q || !k || !v || !spd || !bias || !o_acc || !lse_acc) return GT_ERR_INVALID_ARG;
    if (misaligned16(q) || misaligned16(k) || misaligned16(v) || misaligned16(spd) || misaligned16(o_acc) || (out && misaligned16(out)))
        return GT_ERR_INVALID_ARG;
    if (batch->n_graphs != 1 || n_heads > 65535) return GT_ERR_UNSUPPORTED;
    const int32_t n = batch->n_total;
    if (q_begin < 0 || q_end > n || q_begin >= q_end) return GT_ERR_INVALID_ARG;
    if (kv_begin0 < 0 || kv_end0 > n || kv_begin0 > kv_end0 || kv_begin1 < 0 || kv_end1 > n || kv_begin1 > kv_end1) return GT_ERR_INVALID_ARG;
    // a key range starts at a multiple of 16: the SPD tile of a range is fetched by TMA from that column
    if ((kv_end0 > kv_begin0 && (kv_begin0 & 15)) || (kv_end1 > kv_begin1 && (kv_begin1 & 15))) return GT_ERR_UNSUPPORTED;
    const size_t need = gt_biased_attn_fwd_step_workspace(batch, n_heads, head_dim);
    if (workspace == nullptr || workspace_bytes < need || misaligned16(workspace)) return GT_ERR_WORKSPACE;
    if (sm_count() <= 0) return GT_ERR_NO_DEVICE;
    CUtensorMap tq, tk, tv, tspd;
    if ((st = encode_thd_map(&tq, q, n, n_heads, head_dim)) != GT_OK) return st;
    if ((st = encode_thd_map(&tk, k, n, n_heads, head_dim)) != GT_OK) return st;
    if ((st = encode_thd_map(&tv, v, n, n_heads, head_dim)) != GT_OK) return st;
    if ((st = encode_spd_map(&tspd, spd, n, 256)) != GT_OK) return st;
    const size_t rows = (size_t)n * n_heads;
    uint8_t* ws = (uint8_t*)workspace;
    FwdParams p{};
    p.spd_tma = 1;
    p.spd = spd;
    p.bias = bias;
    p.part_lse = (float*)(ws + kHeaderBytes);
    p.part_o = (float*)(ws + kHeaderBytes + align_up((size_t)2 * rows * sizeof(float), 256));
    p.status = (uint32_t*)workspace;
    p.n_total = n;
    p.n_heads = n_heads;
    p.n_buckets = max_dist + 2;
    p.use_ranges = 1;
    p.range_begin[0] = kv_begin0; p.range_end[0] = kv_end0;
    p.range_begin[1] = kv_begin1; p.range_end[1] = kv_end1;
    const int n_parts = kv_end1 > kv_begin1 ? 2 : 1;
    p.q_block0 = q_begin / kRowsPerCta;
    const int grid_y = (q_end - 1) / kRowsPerCta - p.q_block0 + 1;
    p.c1 = kLog2e / sqrtf((float)head_dim);
    cudaStream_t s = (cudaStream_t)stream;
    // One non-empty key range: the kernel's epilogue merges into the carried state itself.
    const bool fused = n_parts == 1 && kv_end0 > kv_begin0;
    if (fused) {
        p.state_o = o_acc; p.state_lse = lse_acc;
        p.state_q_begin = q_begin; p.state_q_end = q_end;
        p.out = (__nv_bfloat16*)out;
    }
    st = head_dim == 64 ? launch_fwd<64, true>(tq, tk, tv, tspd, p, batch, n_parts, s, grid_y)
                        : launch_fwd<32, true>(tq, tk, tv, tspd, p, batch, n_parts, s, grid_y);
    if (st != GT_OK || fused) return st;
    const size_t n_thr = (size_t)(q_end - q_begin) * n_heads * (head_dim / 4);
    const unsigned blocks = (unsigned)((n_thr + 255) / 256);
    if (head_dim == 64)
        st = launch_overlapped(step_merge_kernel<64>, dim3(blocks), 256, 0, s, p.part_o, p.part_lse, n_parts, o_acc, lse_acc, (__nv_bfloat16*)out,
                                                     q_begin, q_end, n, n_heads);
    else
        st = launch_overlapped(step_merge_kernel<32>, dim3(blocks), 256, 0, s, p.part_o, p.part_lse, n_parts, o_acc, lse_acc, (__nv_bfloat16*)out,
                                                     q_begin, q_end, n, n_heads);
    return st;
}
