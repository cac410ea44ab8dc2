// gt_feature_encode and friends: categorical bias features as a code matrix plus a dictionary.
//
// The feature bias of the model the paper trains (four features per node pair, weighted per head: Sec.
// "Experiments", end-to-end configuration) is   b[h,i,j] = sum_x W[h,x] f[i,j,x].   When the pairs of a graph
// carry only a few distinct feature vectors -- structural encodings are categorical -- numbering the distinct
// vectors c = 0..n_codes-1 turns this into the bucket form of Eq. 1 exactly:
//     b[h,i,j] = table[h, code[i,j]],   table[h,c] = sum_x W[h,x] vec[c,x],   dW[h,x] = sum_c dTable[h,c] vec[c,x],
// so the tensor-core kernels of the bucket form (gt_biased_attn_fwd / _bwd with the code matrix in place of the SPD
// matrix) serve it, and the weights enter and leave through two tiny kernels.  The encoding is done once per batch,
// like the SPD build.  Codes follow the ascending order of the 32-bit feature word, so the result does not depend on
// the order in which threads meet the vectors.
#include "gt_common.cuh"

namespace gt {
namespace {

constexpr int kMaxCodes = 256;
constexpr int kSlots = 4096;                     // open-addressing table, at most 1/16 full
constexpr uint64_t kOccupied = 1ull << 32;      // a slot holds 0 (empty) or kOccupied | word

// workspace: header | slots uint64[kSlots]
constexpr size_t kSlotsOff = kHeaderBytes;
constexpr size_t kEncodeWorkspace = kSlotsOff + sizeof(uint64_t) * kSlots;
// header words used here: [0] status, [4] number of distinct vectors met (may overshoot kMaxCodes), [5] final count,
// [6] thread blocks that are done collecting

__device__ __forceinline__ uint32_t slot_hash(uint32_t w)
{
    w ^= w >> 16; w *= 0x7feb352du; w ^= w >> 15; w *= 0x846ca68bu; w ^= w >> 16;
    return w & (kSlots - 1);
}

// Adds a word to the global set.  False: there are too many already, and the caller of the library is told.  A slot is
// written once (empty -> key), so a stale read can only show "empty", and the compare-and-swap that follows returns what the
// slot really holds.
__device__ bool add_word(uint32_t w, unsigned long long* __restrict__ slots, uint32_t* __restrict__ header)
{
    const unsigned long long key = kOccupied | w;
    uint32_t h = slot_hash(w);
    for (int probe = 0; probe < kSlots; ++probe, h = (h + 1) & (kSlots - 1)) {
        unsigned long long cur = *(volatile unsigned long long*)&slots[h];
        if (cur == key) return true;
        if (cur == 0ull) {
            if (*(volatile uint32_t*)&header[4] > (uint32_t)kMaxCodes) return false;
            cur = atomicCAS(&slots[h], 0ull, key);
            if (cur == 0ull) {
                if (atomicAdd(&header[4], 1u) >= (uint32_t)kMaxCodes) atomicCAS(&header[0], 0u, (uint32_t)GT_ERR_UNSUPPORTED);
                return true;
            }
            if (cur == key) return true;
        }
    }
    return false;
}

// Small tables in shared memory, looked up once per pair.
constexpr int kCacheSlots = 2048;
__device__ __forceinline__ uint32_t cache_hash(uint32_t w) { return (w * 0x9E3779B1u) >> 21; }

// Pass 1: the set of distinct feature words, and (the thread block that is last to finish) their numbers in ascending order.
// Nearly every word has been met before: a thread block keeps the words it has met in shared memory, where one hash and one
// load dismiss a pair, and goes to the global set only for a word that is new to the block.  Four pairs per load, four loads
// in flight.  What bounds it: HBM (4 bytes per pair).
__global__ void __launch_bounds__(512) feature_collect_kernel(const uint32_t* __restrict__ f, int64_t n_pairs, unsigned long long* __restrict__ slots,
                                                              uint32_t* __restrict__ vectors, uint32_t* __restrict__ header)
{
    // Buckets of two words; an empty place holds a word that belongs to another bucket, so a pair needs no test for it.
    __shared__ __align__(8) uint32_t s_met[kCacheSlots];
    __shared__ uint32_t s_full, s_cnt, s_last;
    auto bucket_of = [](uint32_t w) -> uint32_t { return (w * 0x9E3779B1u) >> 22; };
    static_assert(kCacheSlots == 2048, "1 024 buckets");
    auto nobody = [](uint32_t bucket) -> uint32_t { return bucket == 0u ? 1u : 0u; };      // 0 is in bucket 0, 1 is not
    for (int i = threadIdx.x; i < kCacheSlots; i += blockDim.x) s_met[i] = nobody((uint32_t)i >> 1);
    if (threadIdx.x == 0) { s_full = 0u; s_cnt = 0u; }
    __syncthreads();
    auto met = [&](uint32_t w) -> bool {
        const uint2 e = *(const uint2*)&s_met[2 * bucket_of(w)];
        return e.x == w || e.y == w;
    };
    auto meet = [&](uint32_t w) {                          // a bucket that is full sends its other words to the global set every time
        if (met(w)) return;
        if (!add_word(w, slots, header)) { s_full = 1u; return; }
        const uint32_t b = bucket_of(w), none = nobody(b);
        const uint32_t first = atomicCAS(&s_met[2 * b], none, w);
        if (first != none && first != w) atomicCAS(&s_met[2 * b + 1], none, w);
    };
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int head = (int)min((int64_t)((16 - (reinterpret_cast<uintptr_t>(f) & 15)) & 15) / 4, n_pairs);       // pairs before the first aligned vector
    const int64_t n_vec = (n_pairs - head) / 4;
    const uint4* __restrict__ f4 = (const uint4*)(f + head);
    if (blockIdx.x == 0) {
        if ((int)threadIdx.x < head) meet(f[threadIdx.x]);
        const int64_t tail = head + 4 * n_vec;
        if (tail + threadIdx.x < n_pairs) meet(f[tail + threadIdx.x]);
    }
    for (int64_t i = first; i < n_vec; i += 4 * stride) {
        uint4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i + k * stride < n_vec) v[k] = __ldcs(&f4[i + k * stride]);
        if (*(volatile uint32_t*)&s_full) break;           // more vectors than codes: nothing to collect any more
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i + k * stride < n_vec && !(met(v[k].x) & met(v[k].y) & met(v[k].z) & met(v[k].w))) { meet(v[k].x); meet(v[k].y); meet(v[k].z); meet(v[k].w); }
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&header[6], 1u) == gridDim.x - 1 ? 1u : 0u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    uint32_t* words = s_met;
    for (int s = threadIdx.x; s < kSlots; s += blockDim.x) {
        const unsigned long long v = __ldcg(&slots[s]);
        if (v != 0ull) {
            const uint32_t at = atomicAdd(&s_cnt, 1u);
            if (at < (uint32_t)kMaxCodes) words[at] = (uint32_t)v;
        }
    }
    __syncthreads();
    const int n = min((int)s_cnt, kMaxCodes);
    for (int c = threadIdx.x; c < kMaxCodes; c += blockDim.x)
        if (c >= n) vectors[c] = 0u;
    if ((int)threadIdx.x < n) {
        const uint32_t mine = words[threadIdx.x];
        int rank = 0;
        for (int k = 0; k < n; ++k) rank += words[k] < mine;
        vectors[rank] = mine;
    }
    if (threadIdx.x == 0) header[5] = s_cnt;
}

// Pass 2: code[i][j] for the n x n pairs, row pitch ld = n rounded up to 16 as for the SPD matrix, padding bytes 255.
// A warp takes 512 columns of a row, a lane four consecutive ones at a time (one 16-byte load where rows are aligned, one
// 4-byte store), four loads in flight.  What bounds it: HBM (4 bytes read and one written per pair).
__global__ void __launch_bounds__(512) feature_encode_kernel(const uint32_t* __restrict__ f, int32_t n, int32_t ld, const uint32_t* __restrict__ vectors,
                                                             uint8_t* __restrict__ codes, const uint32_t* __restrict__ header)
{
    __shared__ uint2 s_code[kCacheSlots];                 // {word, code}; code ~0: empty
    grid_wait();
    grid_release();
    if (header[0] != 0u) return;                          // too many distinct vectors: nothing sensible to write
    for (int i = threadIdx.x; i < kCacheSlots; i += blockDim.x) s_code[i] = make_uint2(0u, ~0u);
    __syncthreads();
    const int n_codes = min((int)header[5], kMaxCodes);
    if ((int)threadIdx.x < n_codes) {
        const uint32_t w = vectors[threadIdx.x];
        uint32_t h = cache_hash(w);
        while (atomicCAS(&s_code[h].y, ~0u, threadIdx.x) != ~0u) h = (h + 1) & (kCacheSlots - 1);     // at most 1/8 full
        s_code[h].x = w;
    }
    __syncthreads();
    auto code_of = [&](uint32_t w) -> uint32_t {
        uint32_t h = cache_hash(w);
        uint2 e = s_code[h];
        for (int probe = 0; probe < kCacheSlots && (e.x != w || e.y == ~0u); ++probe) { h = (h + 1) & (kCacheSlots - 1); e = s_code[h]; }
        return e.y & 0xffu;
    };
    const int lane = threadIdx.x & 31;
    const uint32_t segs = (uint32_t)(ld + 511) / 512;
    const uint64_t items = (uint64_t)n * segs;
    const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
    const bool words = (reinterpret_cast<uintptr_t>(codes) & 3) == 0;
    const bool aligned = (n & 3) == 0 && (reinterpret_cast<uintptr_t>(f) & 15) == 0;
    for (uint64_t it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < items; it += warps) {
        const int32_t i = (int32_t)(it / segs), j0 = (int32_t)(it % segs) * 512 + 4 * lane;
        const uint32_t* __restrict__ row = f + (size_t)i * n;
        uint4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int32_t j = j0 + 128 * k;
            v[k] = make_uint4(0u, 0u, 0u, 0u);
            if (aligned) {
                if (j < n) v[k] = __ldcs((const uint4*)(row + j));
            } else {
                if (j < n) v[k].x = row[j];
                if (j + 1 < n) v[k].y = row[j + 1];
                if (j + 2 < n) v[k].z = row[j + 2];
                if (j + 3 < n) v[k].w = row[j + 3];
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int32_t j = j0 + 128 * k;
            if (j >= ld) continue;
            uint32_t out;
            if (j + 4 <= n) {
                out = code_of(v[k].x) | code_of(v[k].y) << 8 | code_of(v[k].z) << 16 | code_of(v[k].w) << 24;
            } else {
                out = 0xffffffffu;
                if (j < n) out = (out & ~0xffu) | code_of(v[k].x);
                if (j + 1 < n) out = (out & ~0xff00u) | code_of(v[k].y) << 8;
                if (j + 2 < n) out = (out & ~0xff0000u) | code_of(v[k].z) << 16;
            }
            uint8_t* to = codes + (size_t)i * ld + j;
            if (words) *(uint32_t*)to = out;
            else
                for (int b = 0; b < 4; ++b) to[b] = (uint8_t)(out >> (8 * b));
        }
    }
}

__device__ __forceinline__ float vec_feature(uint32_t word, int x) { return (float)((word >> (8 * x)) & 0xffu); }

// table[h][c] = sum_x W[h][x] vec[c][x]
__global__ void feature_code_table_kernel(const float* __restrict__ w, const uint32_t* __restrict__ vectors, int32_t n_heads,
                                          int32_t n_codes, float* __restrict__ table)
{
    grid_wait();
    grid_release();
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n_heads * n_codes) return;
    const int h = idx / n_codes, c = idx % n_codes;
    const uint32_t word = c < kMaxCodes ? vectors[c] : 0u;
    float b = 0.f;
#pragma unroll
    for (int x = 0; x < 4; ++x) b = fmaf(w[h * 4 + x], vec_feature(word, x), b);
    table[idx] = b;
}

// dW[h][x] = sum_c dTable[h][c] vec[c][x]: one warp per head, fp64 sums (the table gradients of a head cancel to
// rounding, and the vectors may share a large common part)
__global__ void __launch_bounds__(32) feature_code_dweights_kernel(const float* __restrict__ dtable, const uint32_t* __restrict__ vectors,
                                                                   int32_t n_codes, float* __restrict__ dw)
{
    grid_wait();
    grid_release();
    const int h = blockIdx.x, lane = threadIdx.x;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int c = lane; c < n_codes && c < kMaxCodes; c += 32) {
        const double g = (double)dtable[(size_t)h * n_codes + c];
        const uint32_t word = vectors[c];
#pragma unroll
        for (int x = 0; x < 4; ++x) acc[x] += g * (double)((word >> (8 * x)) & 0xffu);
    }
#pragma unroll
    for (int x = 0; x < 4; ++x) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) acc[x] += __shfl_xor_sync(0xffffffffu, acc[x], off);
        if (lane == 0) dw[h * 4 + x] = (float)acc[x];
    }
}

}  // namespace
}  // namespace gt

extern "C" size_t gt_feature_encode_workspace(void) { return gt::kEncodeWorkspace; }

extern "C" gt_status gt_feature_encode(const uint8_t* features, const gt_batch* batch, uint8_t* codes, uint32_t* vectors,
                                       void* workspace, size_t workspace_bytes, void* stream)
{
    using namespace gt;
    gt_status st = validate_batch(batch);
    if (st != GT_OK) return st;
    if (batch->n_graphs != 1) return GT_ERR_UNSUPPORTED;
    if (features == nullptr || codes == nullptr || vectors == nullptr || (reinterpret_cast<uintptr_t>(features) & 3u) != 0 ||
        (reinterpret_cast<uintptr_t>(vectors) & 3u) != 0)
        return GT_ERR_INVALID_ARG;
    if (workspace == nullptr || workspace_bytes < kEncodeWorkspace || misaligned16(workspace)) return GT_ERR_WORKSPACE;
    const int sms = sm_count();
    if (sms <= 0) return GT_ERR_NO_DEVICE;
    cudaStream_t s = (cudaStream_t)stream;
    uint8_t* ws = (uint8_t*)workspace;
    const int32_t n = batch->n_total, ld = (n + 15) & ~15;
    const int64_t n_pairs = (int64_t)n * n;
    GT_CUDA_TRY(cudaMemsetAsync(ws + 16, 0, kEncodeWorkspace - 16, s));  // counters and slots (the status word is the caller's)
    const int64_t want = (n_pairs / 4 + 4095) / 4096 + 1;
    const unsigned grid1 = (unsigned)(want < (int64_t)sms * 4 ? want : (int64_t)sms * 4);
    feature_collect_kernel<<<grid1, 512, 0, s>>>((const uint32_t*)features, n_pairs, (unsigned long long*)(ws + kSlotsOff), vectors, (uint32_t*)ws);
    GT_CUDA_TRY(cudaGetLastError());
    const int64_t items = (int64_t)n * ((ld + 511) / 512);
    const int64_t want2 = (items + 15) / 16;
    const unsigned grid2 = (unsigned)(want2 < (int64_t)sms * 4 ? want2 : (int64_t)sms * 4);
    return launch_overlapped(feature_encode_kernel, dim3(grid2), 512, 0, s, (const uint32_t*)features, n, ld, vectors, codes, (const uint32_t*)ws);
}

extern "C" gt_status gt_feature_encode_count(void* workspace, void* stream, int32_t* n_codes_host)
{
    using namespace gt;
    if (workspace == nullptr || n_codes_host == nullptr) return GT_ERR_INVALID_ARG;
    GT_CUDA_TRY(cudaStreamSynchronize((cudaStream_t)stream));
    uint32_t c = 0;
    GT_CUDA_TRY(cudaMemcpy(&c, (const uint8_t*)workspace + 20, sizeof(c), cudaMemcpyDeviceToHost));
    *n_codes_host = (int32_t)c;
    return GT_OK;
}

extern "C" gt_status gt_feature_code_table(const float* weights, const uint32_t* vectors, int32_t n_heads, int32_t n_codes,
                                           float* table, void* stream)
{
    using namespace gt;
    if (weights == nullptr || vectors == nullptr || table == nullptr || n_heads < 1 || n_codes < 1 || n_codes > kMaxCodes)
        return GT_ERR_INVALID_ARG;
    const int total = n_heads * n_codes;
    return launch_overlapped(feature_code_table_kernel, dim3((unsigned)(total + 255) / 256), 256, 0, (cudaStream_t)stream, weights, vectors, n_heads, n_codes, table);
}

extern "C" gt_status gt_feature_code_dweights(const float* dtable, const uint32_t* vectors, int32_t n_heads, int32_t n_codes,
                                              float* dweights, void* stream)
{
    using namespace gt;
    if (dtable == nullptr || vectors == nullptr || dweights == nullptr || n_heads < 1 || n_codes < 1 || n_codes > kMaxCodes)
        return GT_ERR_INVALID_ARG;
    return launch_overlapped(feature_code_dweights_kernel, dim3((unsigned)n_heads), 32, 0, (cudaStream_t)stream, dtable, vectors, n_codes, dweights);
}
