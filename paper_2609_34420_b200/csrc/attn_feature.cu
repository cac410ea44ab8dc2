// gt_feature_attn_fwd / gt_feature_attn_bwd: Eq. 1 with a FEATURE bias,
//     S_ij = (q_i . k_j)/sqrt(d) + sum_c W[h][c] * f[i][j][c],      f uint8 [N][N][4],  W fp32 [H][4]
// (the end-to-end model of the paper has an "attention bias dimension of 4"; the paper gives the dimension
// only, the linear form is the reading taken here).  The bias gradient is a plain contraction,
// dW[h][c] = sum_ij dS_ij f[i][j][c], instead of the scatter of the bucket form.
//
// The contractions run on the tensor cores without giving up fp32: the bf16 inputs are exact operands, and a probability or
// a score gradient, an fp32 number, goes in as three bf16 terms (8 + 8 + 8 bits of mantissa: the sum is the number); sums
// over more than one MMA block are fp32 adds (add_product).  Against fp64, lse and dW are no further off than the same sums
// formed element by element on the fp32 pipes, and fewer of the bf16 results miss the nearest value.  Three kernels of one shape:
//   forward      a warp owns 16 query rows and walks over keys:   S = Q K^T, online softmax, O += P V
//   query side   the same rows and keys, twice:  S and dP = dO V^T for Delta_i = sum_j P_ij dP_ij, then again for dS = P (dP - Delta),
//                dQ += dS K and dW += dS f
//   key side     a warp owns 16 key rows and walks over queries:  S^T, dP^T, dV += P^T dO, dK += dS^T Q
// The score fragments of one product are the operand fragments of the next (mma.sync keeps both in registers), a pair's four
// features are read straight into the lane that holds its score, and Delta is formed from the same P as the gradients: the
// features have a large common part, which a Delta from a rounded output would turn into an error of dW.  A thread block is
// two row groups times two halves of each 64-row tile of the other side (small graphs have few rows: the halves keep twice as
// many warps busy), whose partial results are added at the end.
//
// mma.sync and not tcgen05: at the 500 - 8 192 nodes this form is meant for, a 128-row tile per thread block would leave
// most SMs empty, and the three-term operands would have to travel through tensor memory.
// What bounds it: the latency of an element's chain of instructions at ten warps per SM (1 500 nodes have no more rows; issue slots
// 45 %, tensor pipe 33-42 % busy).  12 of the 19 contractions are the terms of P and dS; fp32 arithmetic goes by pairs of neighbouring
// columns (one instruction, the same results), and a chain's first MMA adds to zero.  1 500 nodes, H = 8, d = 64: forward 60 us,
// backward 195 us (64 and 199 element by element; 54 and 172 with one chain of MMAs over all keys, ex2 in the forward and one walk on
// the query side, whose results are further off); the same sums on the fp32 pipes took 3 000 us.
#include <cuda_bf16.h>
#include <math.h>

#include <initializer_list>

#include "attn_common.cuh"
#include "sm100_primitives.cuh"

namespace gt {
namespace {

using namespace sm100;

constexpr int kFeat = 4;              // bias features per node pair
constexpr int kRows = 32;             // rows of a thread block: two groups of 16
constexpr int kTile = 64;             // rows of the other side per stage: two halves of 32
constexpr int kThreads = 128;

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// the same on an empty accumulator
__device__ __forceinline__ void mma16816_first(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                 : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ void ldm4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldm4_trans(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16u : 0u) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kLeft>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(kLeft) : "memory"); }

// Two fp32 numbers as three pairs of bf16 whose sum they are.
__device__ __forceinline__ void split3(uint64_t x, uint32_t& hi, uint32_t& mid, uint32_t& lo)
{
    auto pack = [](uint64_t v) {
        float a, b;
        unpack_f32x2(v, a, b);
        uint32_t r;
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(b), "f"(a));
        return r;
    };
    auto rest = [](uint64_t v, uint32_t term) {
        return fma_f32x2(pack_u32x2(term << 16, term & 0xffff0000u), pack_f32x2(-1.f, -1.f), v);
    };
    hi = pack(x);
    x = rest(x, hi);
    mid = pack(x);
    lo = pack(rest(x, mid));
}

// A tile of rows of D bf16 in shared memory: 16-byte chunks, XOR-swizzled so that eight rows of one chunk column lie in
// different banks (ldmatrix reads them together).
template <int D>
struct Tile {
    static constexpr int kRowBytes = 2 * D;
    static __device__ __forceinline__ uint32_t at(uint32_t base, int row, int chunk)
    {
        const int x = D == 64 ? (row & 7) : ((row >> 1) & 3);
        return base + (uint32_t)(row * kRowBytes + ((chunk ^ x) * 16));
    }
    // rows [r0, r0 + kCount) of head h of a [n, H, D] tensor; rows past n are zero.  kAligned: the tensor begins at a multiple of 16 bytes
    template <int kCount, bool kAligned>
    static __device__ __forceinline__ void fetch(uint32_t base, const __nv_bfloat16* __restrict__ x, int32_t n, int32_t n_heads, int32_t h, int32_t r0)
    {
        constexpr int kChunks = D / 8;
#pragma unroll
        for (int e = 0; e < kCount * kChunks / kThreads; ++e) {
            const int i = e * kThreads + (int)threadIdx.x, r = i / kChunks, c = i % kChunks;
            const bool ok = r0 + r < n;
            const __nv_bfloat16* src = x + ((size_t)(ok ? r0 + r : 0) * n_heads + h) * D + c * 8;
            if constexpr (kAligned) {
                cp16(at(base, r, c), src, ok);
            } else {
                uint32_t w[4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    w[k] = ok ? (uint32_t)((const uint16_t*)src)[2 * k] | (uint32_t)((const uint16_t*)src)[2 * k + 1] << 16 : 0u;
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at(base, r, c)), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
            }
        }
    }
    // A fragments (16 rows from `row`, all of D)
    static __device__ __forceinline__ void load_a(uint32_t (&a)[D / 16][4], uint32_t base, int row, int lane)
    {
#pragma unroll
        for (int k = 0; k < D / 16; ++k) ldm4(a[k], at(base, row + (lane & 15), 2 * k + (lane >> 4)));
    }
    // B fragments of 16 rows (two column tiles of the product) for channels 16 k .. : b[0..1] first tile, b[2..3] second
    static __device__ __forceinline__ void load_b(uint32_t (&b)[4], uint32_t base, int row, int k, int lane)
    {
        ldm4(b, at(base, row + (lane & 7) + ((lane >> 4) << 3), 2 * k + ((lane >> 3) & 1)));
    }
    // B fragments of 16 rows as the contracted index, channels 16 c .. (two column tiles)
    static __device__ __forceinline__ void load_bt(uint32_t (&b)[4], uint32_t base, int row, int c, int lane)
    {
        ldm4_trans(b, at(base, row + (lane & 15), 2 * c + (lane >> 4)));
    }
};

// S (16 x 32, two blocks of 16 columns) = A (16 x D) B^T, B = 32 rows of a tile
template <int D>
__device__ __forceinline__ void scores(float (&s)[2][2][4], const uint32_t (&a)[D / 16][4], uint32_t base, int row, int lane)
{
#pragma unroll
    for (int k = 0; k < D / 16; ++k) {
        uint32_t b[4], c[4];
        Tile<D>::load_b(b, base, row, k, lane);
        Tile<D>::load_b(c, base, row + 16, k, lane);
        auto step = [&](auto mma) {
            mma(s[0][0], a[k], b[0], b[1]);
            mma(s[0][1], a[k], b[2], b[3]);
            mma(s[1][0], a[k], c[0], c[1]);
            mma(s[1][1], a[k], c[2], c[3]);
        };
        if (k == 0) step(mma16816_first);
        else step(mma16816);
    }
}

// Two such products with A read from 16 rows of a tile as it goes.  Their steps alternate: an MMA that adds to the result of
// the one before it would wait for it.
template <int D>
__device__ __forceinline__ void two_scores(float (&s)[2][4], uint32_t own_s, float (&u)[2][4], uint32_t own_u, int own_row,
                                           uint32_t base_s, uint32_t base_u, int row, int lane)
{
#pragma unroll
    for (int k = 0; k < D / 16; ++k) {
        uint32_t a[4], b[4], c[4], d[4];
        ldm4(a, Tile<D>::at(own_s, own_row + (lane & 15), 2 * k + (lane >> 4)));
        Tile<D>::load_b(b, base_s, row, k, lane);
        ldm4(c, Tile<D>::at(own_u, own_row + (lane & 15), 2 * k + (lane >> 4)));
        Tile<D>::load_b(d, base_u, row, k, lane);
        auto step = [&](auto mma) {
            mma(s[0], a, b[0], b[1]);
            mma(u[0], c, d[0], d[1]);
            mma(s[1], a, b[2], b[3]);
            mma(u[1], c, d[2], d[3]);
        };
        if (k == 0) step(mma16816_first);
        else step(mma16816);
    }
}

// a 16 x 16 block of fp32 in score fragments (pairs of neighbouring columns) -> its three bf16 operand fragments
__device__ __forceinline__ void split_block(const uint64_t (&p)[2][2], uint32_t (&t)[3][4])
{
#pragma unroll
    for (int k = 0; k < 4; ++k) split3(p[k >> 1][k & 1], t[0][k], t[1][k], t[2][k]);
}

// acc (16 x D) += P (16 x 16, three terms; smallest first) times 16 rows of a tile.  The tensor core cuts off what its
// accumulator cannot hold instead of rounding it, an error that grows with every MMA of a chain and does not cancel: a chain is
// one block of 16 long and its result is added to the sum by an fp32 add.  (With chains over all keys two to five times as many
// outputs miss the nearest bf16 value, growing with n.)  Four chains alternate: an MMA that adds to the result of the one before
// it would wait for it.
template <int D>
__device__ __forceinline__ void add_product(uint64_t (&acc)[D / 8][2], const uint32_t (&t)[3][4], uint32_t base, int row, int lane)
{
#pragma unroll
    for (int c = 0; c < D / 16; c += 2) {
        uint32_t b0[4], b1[4];
        Tile<D>::load_bt(b0, base, row, c, lane);
        Tile<D>::load_bt(b1, base, row, c + 1, lane);
        float u[4][4];
#pragma unroll
        for (int x = 2; x >= 0; --x) {
            auto step = [&](auto mma) {
                mma(u[0], t[x], b0[0], b0[1]);
                mma(u[2], t[x], b1[0], b1[1]);
                mma(u[1], t[x], b0[2], b0[3]);
                mma(u[3], t[x], b1[2], b1[3]);
            };
            if (x == 2) step(mma16816_first);
            else step(mma16816);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            acc[2 * c + k][0] = add_f32x2(acc[2 * c + k][0], pack_f32x2(u[k][0], u[k][1]));
            acc[2 * c + k][1] = add_f32x2(acc[2 * c + k][1], pack_f32x2(u[k][2], u[k][3]));
        }
    }
}

__device__ __forceinline__ uint64_t both(float x) { return pack_f32x2(x, x); }

// The features of two pairs.  Byte -> fp32 without the conversion pipe: 2^15 + b has b in its mantissa's second byte, and 2^15
// comes off exactly.
__device__ __forceinline__ void unpack_features(uint32_t f4, uint32_t g4, uint64_t (&f)[kFeat])
{
#pragma unroll
    for (int c = 0; c < kFeat; ++c) {
        const uint32_t pick = 0x7404u | ((uint32_t)c << 4);
        f[c] = add_f32x2(pack_u32x2(__byte_perm(f4, 0x47000000u, pick), __byte_perm(g4, 0x47000000u, pick)), both(-32768.f));
    }
}

template <bool B> struct BoolConst { static constexpr bool value = B; };

// Two neighbouring results.
template <bool kAligned>
__device__ __forceinline__ void store_pair(__nv_bfloat16* to, float a, float b)
{
    if constexpr (kAligned) {
        *(__nv_bfloat162*)to = __floats2bfloat162_rn(a, b);
    } else {
        to[0] = __float2bfloat16_rn(a);
        to[1] = __float2bfloat16_rn(b);
    }
}

struct FeatureArgs {
    const __nv_bfloat16 *q, *k, *v, *dout;
    const uint32_t* feat;         // the four features of a pair as one word, [n][n]
    const float* weights;
    const float* lse_in;
    float* lse;
    float* delta;                 // [H][n]
    double* dw_part;              // [H][row blocks][4]
    __nv_bfloat16 *out, *dq, *dk, *dv;
    float* dweights;
    int32_t n, n_heads;
    float scale;                  // 1 / sqrt(d)
};

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint64_t ex2_pair(uint64_t x)
{
    float a, b;
    unpack_f32x2(x, a, b);
    return pack_f32x2(ex2(a), ex2(b));
}
// e^x for the backward's P, off by up to |x| 2^-24 beside the 2 ulp of ex2, and less than P matters where x is large.
__device__ __forceinline__ uint64_t exp_of(uint64_t x) { return ex2_pair(mul_f32x2(x, both(kLog2e))); }
// The forward keeps expf, because its lse is returned in fp32.
__device__ __forceinline__ uint64_t expf_pair(uint64_t x)
{
    float a, b;
    unpack_f32x2(x, a, b);
    return pack_f32x2(expf(a), expf(b));
}

// words of pairs (i, j) and (i, j + 1), j even; out of range: 0
__device__ __forceinline__ uint2 feature_pair(const uint32_t* __restrict__ feat, int32_t n, bool pairs, int32_t i, int32_t j)
{
    uint2 r = make_uint2(0u, 0u);
    if (i < n && j < n) {
        const uint32_t* at = feat + (size_t)i * n + j;
        if (pairs) r = __ldg((const uint2*)at);            // n even: j + 1 < n too
        else {
            r.x = __ldg(at);
            if (j + 1 < n) r.y = __ldg(at + 1);
        }
    }
    return r;
}
__device__ __forceinline__ uint64_t bias_of(const uint64_t (&f)[kFeat], const uint64_t (&w)[kFeat])
{
    return fma_f32x2(w[3], f[3], fma_f32x2(w[2], f[2], fma_f32x2(w[1], f[1], mul_f32x2(w[0], f[0]))));
}
// sum over the four lanes that share a fragment row
__device__ __forceinline__ float quad_sum(float x)
{
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    return x + __shfl_xor_sync(0xffffffffu, x, 2);
}
__device__ __forceinline__ float quad_max(float x)
{
    x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 1));
    return fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 2));
}

// ---------------------------------------------------------------------------------------------------
// Forward: a warp owns 16 query rows and one half of the keys.
// ---------------------------------------------------------------------------------------------------
template <int D, bool kAligned>
__global__ void __launch_bounds__(kThreads, 3) feature_fwd_kernel(FeatureArgs p)
{
    grid_wait();
    grid_release();
    constexpr int kTileBytes = kTile * 2 * D;
    __shared__ __align__(128) uint8_t s_tiles[4 * kTileBytes];                    // two stages of K and V
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, group = warp >> 1, half = warp & 1;
    const int h = blockIdx.y;
    const int32_t n = p.n, i0 = (int32_t)blockIdx.x * kRows + 16 * group;
    const int g = lane >> 2, t4 = lane & 3;
    const uint32_t base = smem_addr(s_tiles);
    const bool pairs = (n & 1) == 0 && (reinterpret_cast<uintptr_t>(p.feat) & 7u) == 0;
    uint64_t w[kFeat];
#pragma unroll
    for (int c = 0; c < kFeat; ++c) w[c] = both(p.weights[h * kFeat + c]);
    const uint64_t scale = both(p.scale);

    uint32_t qa[D / 16][4];
    Tile<D>::template fetch<kRows, kAligned>(base, p.q, n, p.n_heads, h, (int32_t)blockIdx.x * kRows);
    cp_commit();
    cp_wait<0>();
    __syncthreads();
    Tile<D>::load_a(qa, base, 16 * group, lane);
    __syncthreads();

    uint64_t o[D / 8][2];
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
#pragma unroll
    for (int c = 0; c < D / 8; ++c) o[c][0] = o[c][1] = 0ull;
    const int32_t n_tiles = (n + kTile - 1) / kTile;
    auto stage = [&](int32_t tile) {
        const uint32_t at = base + (uint32_t)(tile & 1) * 2 * kTileBytes;
        Tile<D>::template fetch<kTile, kAligned>(at, p.k, n, p.n_heads, h, tile * kTile);
        Tile<D>::template fetch<kTile, kAligned>(at + kTileBytes, p.v, n, p.n_heads, h, tile * kTile);
        cp_commit();
    };
    stage(0);
    for (int32_t tile = 0; tile < n_tiles; ++tile) {
        const int32_t j0 = tile * kTile + 32 * half;
        uint2 f[2][2][2];                                                        // [16 keys][column tile][row g, g + 8]
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int r = 0; r < 2; ++r) f[b][t][r] = feature_pair(p.feat, n, pairs, i0 + g + 8 * r, j0 + 16 * b + 8 * t + 2 * t4);
        if (tile + 1 < n_tiles) { stage(tile + 1); cp_wait<1>(); } else cp_wait<0>();
        __syncthreads();
        const uint32_t kt = base + (uint32_t)(tile & 1) * 2 * kTileBytes, vt = kt + kTileBytes;
        const bool ragged = j0 + 32 > n;
        float s[2][2][4], top[2] = {m[0], m[1]};
        scores<D>(s, qa, kt, 32 * half, lane);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const int32_t j = j0 + 16 * b + 8 * t + 2 * t4;
                    uint64_t fv[kFeat];
                    unpack_features(f[b][t][r].x, f[b][t][r].y, fv);
                    float(&s2)[2] = *(float(*)[2])&s[b][t][2 * r];
                    unpack_f32x2(fma_f32x2(pack_f32x2(s2[0], s2[1]), scale, bias_of(fv, w)), s2[0], s2[1]);     // bias added before the softmax statistics
                    if (ragged && j >= n) s2[0] = -INFINITY;
                    if (ragged && j + 1 >= n) s2[1] = -INFINITY;
                    top[r] = fmaxf(top[r], fmaxf(s2[0], s2[1]));
                }
        }
        top[0] = quad_max(top[0]);
        top[1] = quad_max(top[1]);
        if (__any_sync(0xffffffffu, top[0] > m[0] || top[1] > m[1])) {
            const float a0 = m[0] == top[0] ? 1.f : expf(m[0] - top[0]), a1 = m[1] == top[1] ? 1.f : expf(m[1] - top[1]);
            l[0] *= a0; l[1] *= a1;
#pragma unroll
            for (int c = 0; c < D / 8; ++c) { o[c][0] = mul_f32x2(o[c][0], both(a0)); o[c][1] = mul_f32x2(o[c][1], both(a1)); }
            m[0] = top[0]; m[1] = top[1];
        }
        uint64_t less[2];                                                        // minus the reference (0: a half without keys so far)
#pragma unroll
        for (int r = 0; r < 2; ++r) less[r] = both(m[r] == -INFINITY ? 0.f : -m[r]);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            uint64_t pr[2][2];                                                   // 0 for keys past the end
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int r = 0; r < 2; ++r) pr[t][r] = expf_pair(add_f32x2(pack_f32x2(s[b][t][2 * r], s[b][t][2 * r + 1]), less[r]));
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                float x, y;
                unpack_f32x2(add_f32x2(pr[0][r], pr[1][r]), x, y);
                l[r] += x + y;
            }
            uint32_t pt[3][4];
            split_block(pr, pt);
            add_product<D>(o, pt, vt, 32 * half + 16 * b, lane);
        }
        __syncthreads();
    }
    l[0] = quad_sum(l[0]);
    l[1] = quad_sum(l[1]);
    // the second half's share, merged by the first
    float* part = (float*)s_tiles + group * (16 * (D + 2));
    if (half == 1) {
#pragma unroll
        for (int c = 0; c < D / 8; ++c)
#pragma unroll
            for (int r = 0; r < 2; ++r) *(uint64_t*)&part[(g + 8 * r) * D + 8 * c + 2 * t4] = o[c][r];
        if (t4 == 0) {
#pragma unroll
            for (int r = 0; r < 2; ++r) { part[16 * D + g + 8 * r] = m[r]; part[16 * D + 16 + g + 8 * r] = l[r]; }
        }
    }
    __syncthreads();
    if (half == 0) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int32_t i = i0 + g + 8 * r;
            const float m2 = part[16 * D + g + 8 * r], l2 = part[16 * D + 16 + g + 8 * r];
            const float mm = fmaxf(m[r], m2), a = expf(m[r] - mm), b = m2 == -INFINITY ? 0.f : expf(m2 - mm);
            const float ll = l[r] * a + l2 * b, inv = 1.0f / ll;
            if (i < n) {
#pragma unroll
                for (int c = 0; c < D / 8; ++c) {
                    const float* o2 = part + (g + 8 * r) * D + 8 * c + 2 * t4;
                    float x, y;
                    unpack_f32x2(o[c][r], x, y);
                    x = (x * a + o2[0] * b) * inv;
                    y = (y * a + o2[1] * b) * inv;
                    store_pair<kAligned>(p.out + ((size_t)i * p.n_heads + h) * D + 8 * c + 2 * t4, x, y);
                }
                if (t4 == 0) p.lse[(size_t)h * n + i] = mm + logf(ll);
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------------
// Backward, query side: dQ, Delta and the row block's share of dW.  Two walks over the keys: first Delta_i = sum_j P_ij dP_ij,
// divided by sum_j P_ij (1 up to the rounding of lse, whose share of a dP with a large common part would come back as an error of
// dW), then dS.  (One walk that takes Delta_i sum_j P_ij K_j from sum_j P_ij dP_ij K_j at its end needs one MMA more per 16 keys
// and channels and loses what the two sums have in common.)
// ---------------------------------------------------------------------------------------------------
template <int D, bool kAligned>
__global__ void __launch_bounds__(kThreads, 3) feature_bwd_q_kernel(FeatureArgs p)
{
    grid_wait();
    grid_release();
    constexpr int kTileBytes = kTile * 2 * D;
    __shared__ __align__(128) uint8_t s_tiles[4 * kTileBytes];
    __shared__ __align__(128) uint8_t s_own[2 * kRows * 2 * D];                   // the rows' Q and dO (in registers they would cost a block per SM)
    __shared__ float2 s_sums[2][2][16];                                           // [half][group][row]: sums of P dP and of P
    __shared__ double s_dw[4][kFeat];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, group = warp >> 1, half = warp & 1;
    const int h = blockIdx.y;
    const int32_t n = p.n, i0 = (int32_t)blockIdx.x * kRows + 16 * group;
    const int g = lane >> 2, t4 = lane & 3;
    const uint32_t base = smem_addr(s_tiles);
    const bool pairs = (n & 1) == 0 && (reinterpret_cast<uintptr_t>(p.feat) & 7u) == 0;
    uint64_t w[kFeat];
#pragma unroll
    for (int c = 0; c < kFeat; ++c) w[c] = both(p.weights[h * kFeat + c]);
    const uint64_t scale = both(p.scale);

    const uint32_t own_q = smem_addr(s_own), own_d = own_q + kRows * 2 * D;
    Tile<D>::template fetch<kRows, kAligned>(own_q, p.q, n, p.n_heads, h, (int32_t)blockIdx.x * kRows);
    Tile<D>::template fetch<kRows, kAligned>(own_d, p.dout, n, p.n_heads, h, (int32_t)blockIdx.x * kRows);
    cp_commit();

    float lse[2], delta[2] = {0.f, 0.f}, sum_px[2] = {0.f, 0.f}, sum_p[2] = {0.f, 0.f};
    uint64_t dq[D / 8][2], xf[kFeat];                                             // sums of dS K and of dS f (even and odd columns)
#pragma unroll
    for (int r = 0; r < 2; ++r) lse[r] = i0 + g + 8 * r < n ? p.lse_in[(size_t)h * n + i0 + g + 8 * r] : INFINITY;     // P = 0
#pragma unroll
    for (int c = 0; c < D / 8; ++c) dq[c][0] = dq[c][1] = 0ull;
#pragma unroll
    for (int c = 0; c < kFeat; ++c) xf[c] = 0ull;
    const int32_t n_tiles = (n + kTile - 1) / kTile;
    auto stage = [&](int32_t tile) {
        const uint32_t at = base + (uint32_t)(tile & 1) * 2 * kTileBytes;
        Tile<D>::template fetch<kTile, kAligned>(at, p.k, n, p.n_heads, h, tile * kTile);
        Tile<D>::template fetch<kTile, kAligned>(at + kTileBytes, p.v, n, p.n_heads, h, tile * kTile);
        cp_commit();
    };
    auto walk = [&](auto for_delta) {
        constexpr bool kForDelta = decltype(for_delta)::value;
        stage(0);
        for (int32_t tile = 0; tile < n_tiles; ++tile) {
            const int32_t j0 = tile * kTile + 32 * half;
            uint2 f[2][2];                                                        // of the next 16 keys
            auto fetch_features = [&](int b) {
#pragma unroll
                for (int t = 0; t < 2; ++t)
#pragma unroll
                    for (int r = 0; r < 2; ++r) f[t][r] = feature_pair(p.feat, n, pairs, i0 + g + 8 * r, j0 + 16 * b + 8 * t + 2 * t4);
            };
            fetch_features(0);
            if (tile + 1 < n_tiles) { stage(tile + 1); cp_wait<1>(); } else cp_wait<0>();
            __syncthreads();
            const uint32_t kt = base + (uint32_t)(tile & 1) * 2 * kTileBytes, vt = kt + kTileBytes;
#pragma unroll 1
            for (int b = 0; b < 2; ++b) {
                float s[2][4], dp[2][4];
                uint64_t y[kFeat] = {}, px[2][2], pr[2][2];
                two_scores<D>(s, own_q, dp, own_d, 16 * group, kt, vt, 32 * half + 16 * b, lane);
                const bool ragged = j0 + 16 * b + 16 > n;
#pragma unroll
                for (int t = 0; t < 2; ++t)
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const int32_t j = j0 + 16 * b + 8 * t + 2 * t4;
                        uint64_t fv[kFeat];
                        unpack_features(f[t][r].x, f[t][r].y, fv);
                        const uint64_t x = fma_f32x2(pack_f32x2(s[t][2 * r], s[t][2 * r + 1]), scale, bias_of(fv, w));
                        pr[t][r] = exp_of(add_f32x2(x, both(-lse[r])));
                        if (ragged && j + 1 >= n) pr[t][r] &= j >= n ? 0ull : 0xffffffffull;
                        const uint64_t d = pack_f32x2(dp[t][2 * r], dp[t][2 * r + 1]);
                        if constexpr (kForDelta) {
                            px[t][r] = mul_f32x2(d, pr[t][r]);
                        } else {
                            px[t][r] = mul_f32x2(pr[t][r], add_f32x2(d, both(-delta[r])));
#pragma unroll
                            for (int c = 0; c < kFeat; ++c) y[c] = fma_f32x2(px[t][r], fv[c], y[c]);
                        }
                    }
                if (b == 0) fetch_features(1);
                if constexpr (kForDelta) {
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        float a, c;
                        unpack_f32x2(add_f32x2(px[0][r], px[1][r]), a, c);
                        sum_px[r] += a + c;
                        unpack_f32x2(add_f32x2(pr[0][r], pr[1][r]), a, c);
                        sum_p[r] += a + c;
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < kFeat; ++c) xf[c] = add_f32x2(xf[c], y[c]);
                    uint32_t xt[3][4];
                    split_block(px, xt);
                    add_product<D>(dq, xt, kt, 32 * half + 16 * b, lane);
                }
            }
            __syncthreads();
        }
    };
    walk(BoolConst<true>{});
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        sum_px[r] = quad_sum(sum_px[r]);
        sum_p[r] = quad_sum(sum_p[r]);
        if (t4 == 0) s_sums[half][group][g + 8 * r] = make_float2(sum_px[r], sum_p[r]);
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int32_t i = i0 + g + 8 * r;
        const float2 a = s_sums[0][group][g + 8 * r], b = s_sums[1][group][g + 8 * r];
        delta[r] = a.y + b.y > 0.f ? (a.x + b.x) / (a.y + b.y) : a.x + b.x;      // (rows past the end: 0)
        if (half == 0 && t4 == 0 && i < n) p.delta[(size_t)h * n + i] = delta[r];
    }
    walk(BoolConst<false>{});
    float* part = (float*)s_tiles + group * (16 * D);
    if (half == 1) {
#pragma unroll
        for (int c = 0; c < D / 8; ++c)
#pragma unroll
            for (int r = 0; r < 2; ++r) *(uint64_t*)&part[(g + 8 * r) * D + 8 * c + 2 * t4] = dq[c][r];
    }
#pragma unroll
    for (int c = 0; c < kFeat; ++c) {
        float even, odd;
        unpack_f32x2(xf[c], even, odd);
        double dw = (double)even + (double)odd;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) dw += __shfl_xor_sync(0xffffffffu, dw, off);
        if (lane == 0) s_dw[warp][c] = dw;
    }
    __syncthreads();
    if (half == 0) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int32_t i = i0 + g + 8 * r;
            if (i >= n) continue;
#pragma unroll
            for (int c = 0; c < D / 8; ++c) {
                const float* x2 = part + (g + 8 * r) * D + 8 * c + 2 * t4;
                float x, y;
                unpack_f32x2(dq[c][r], x, y);
                store_pair<kAligned>(p.dq + ((size_t)i * p.n_heads + h) * D + 8 * c + 2 * t4, (x + x2[0]) * p.scale, (y + x2[1]) * p.scale);
            }
        }
    }
    if (threadIdx.x < kFeat)
        p.dw_part[((size_t)h * gridDim.x + blockIdx.x) * kFeat + threadIdx.x] =
            s_dw[0][threadIdx.x] + s_dw[1][threadIdx.x] + s_dw[2][threadIdx.x] + s_dw[3][threadIdx.x];
}

// ---------------------------------------------------------------------------------------------------
// Backward, key side: dK and dV (and, by the first block of a head, the sum of the row blocks' shares of dW).
// ---------------------------------------------------------------------------------------------------
template <int D, bool kAligned>
__global__ void __launch_bounds__(kThreads, 3) feature_bwd_kv_kernel(FeatureArgs p)
{
    grid_wait();
    grid_release();
    constexpr int kTileBytes = kTile * 2 * D;
    __shared__ __align__(128) uint8_t s_tiles[4 * kTileBytes];                    // two stages of Q and dO
    __shared__ __align__(128) uint8_t s_own[2 * kRows * 2 * D];                   // the rows' K and V
    __shared__ __align__(16) float s_lse[2][kTile], s_delta[2][kTile];            // minus lse and minus Delta of the queries
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, group = warp >> 1, half = warp & 1;
    const int h = blockIdx.y;
    const int32_t n = p.n, j0 = (int32_t)blockIdx.x * kRows + 16 * group;
    const int g = lane >> 2, t4 = lane & 3;
    const uint32_t base = smem_addr(s_tiles);
    if (blockIdx.x == 0 && warp == 0) {
        double dw = 0.0;                                                          // lane: feature lane & 3, every eighth block
        for (unsigned b = lane >> 2; b < gridDim.x; b += 8) dw += p.dw_part[((size_t)h * gridDim.x + b) * kFeat + (lane & 3)];
#pragma unroll
        for (int off = 16; off >= 4; off >>= 1) dw += __shfl_xor_sync(0xffffffffu, dw, off);
        if (lane < kFeat) p.dweights[h * kFeat + lane] = (float)dw;
    }
    uint64_t w[kFeat];
#pragma unroll
    for (int c = 0; c < kFeat; ++c) w[c] = both(p.weights[h * kFeat + c]);
    const uint64_t scale = both(p.scale);

    const uint32_t own_k = smem_addr(s_own), own_v = own_k + kRows * 2 * D;
    Tile<D>::template fetch<kRows, kAligned>(own_k, p.k, n, p.n_heads, h, (int32_t)blockIdx.x * kRows);
    Tile<D>::template fetch<kRows, kAligned>(own_v, p.v, n, p.n_heads, h, (int32_t)blockIdx.x * kRows);
    cp_commit();

    uint64_t dk[D / 8][2], dv[D / 8][2];
#pragma unroll
    for (int c = 0; c < D / 8; ++c) dk[c][0] = dk[c][1] = dv[c][0] = dv[c][1] = 0ull;
    const int32_t n_tiles = (n + kTile - 1) / kTile;
    auto stage = [&](int32_t tile) {
        const uint32_t at = base + (uint32_t)(tile & 1) * 2 * kTileBytes;
        Tile<D>::template fetch<kTile, kAligned>(at, p.q, n, p.n_heads, h, tile * kTile);
        Tile<D>::template fetch<kTile, kAligned>(at + kTileBytes, p.dout, n, p.n_heads, h, tile * kTile);
        cp_commit();
        if (threadIdx.x < kTile) {
            const int32_t i = tile * kTile + (int32_t)threadIdx.x;
            s_lse[tile & 1][threadIdx.x] = i < n ? -p.lse_in[(size_t)h * n + i] : -INFINITY;
            s_delta[tile & 1][threadIdx.x] = i < n ? -p.delta[(size_t)h * n + i] : 0.f;
        }
    };
    stage(0);
    for (int32_t tile = 0; tile < n_tiles; ++tile) {
        const int32_t i0 = tile * kTile + 32 * half;
        uint32_t f[2][4];                                                         // fragment order: (key g, query 2t4), (g, 2t4+1), (g+8, ..)
        auto fetch_features = [&](int b) {
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const int32_t i = i0 + 16 * b + 8 * t + 2 * t4 + (x & 1), j = j0 + g + 8 * (x >> 1);
                    f[t][x] = i < n && j < n ? __ldg(p.feat + (size_t)i * n + j) : 0u;         // the pair is (query i -> key j)
                }
        };
        fetch_features(0);
        if (tile + 1 < n_tiles) { stage(tile + 1); cp_wait<1>(); } else cp_wait<0>();
        __syncthreads();
        const uint32_t qt = base + (uint32_t)(tile & 1) * 2 * kTileBytes, dt = qt + kTileBytes;
#pragma unroll 1
        for (int b = 0; b < 2; ++b) {
            float s[2][4], dp[2][4];
            uint64_t pr[2][2], ds[2][2];
            two_scores<D>(s, own_k, dp, own_v, 16 * group, qt, dt, 32 * half + 16 * b, lane);
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const int i = 32 * half + 16 * b + 8 * t + 2 * t4;
                const uint64_t lse = *(const uint64_t*)&s_lse[tile & 1][i], delta = *(const uint64_t*)&s_delta[tile & 1][i];
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    uint64_t fv[kFeat];
                    unpack_features(f[t][2 * r], f[t][2 * r + 1], fv);
                    const uint64_t x = fma_f32x2(pack_f32x2(s[t][2 * r], s[t][2 * r + 1]), scale, bias_of(fv, w));
                    pr[t][r] = exp_of(add_f32x2(x, lse));                         // 0 for queries past the end
                    ds[t][r] = mul_f32x2(pr[t][r], add_f32x2(pack_f32x2(dp[t][2 * r], dp[t][2 * r + 1]), delta));
                }
            }
            if (b == 0) fetch_features(1);
            uint32_t terms[3][4];
            split_block(pr, terms);
            add_product<D>(dv, terms, dt, 32 * half + 16 * b, lane);
            split_block(ds, terms);
            add_product<D>(dk, terms, qt, 32 * half + 16 * b, lane);
        }
        __syncthreads();
    }
    float* part = (float*)s_tiles + group * (2 * 16 * D);
    if (half == 1) {
#pragma unroll
        for (int c = 0; c < D / 8; ++c)
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int at = (g + 8 * r) * D + 8 * c + 2 * t4;
                *(uint64_t*)&part[at] = dk[c][r];
                *(uint64_t*)&part[16 * D + at] = dv[c][r];
            }
    }
    __syncthreads();
    if (half == 0) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int32_t j = j0 + g + 8 * r;
            if (j >= n) continue;
#pragma unroll
            for (int c = 0; c < D / 8; ++c) {
                const float* x2 = part + (g + 8 * r) * D + 8 * c + 2 * t4;
                const size_t at = ((size_t)j * p.n_heads + h) * D + 8 * c + 2 * t4;
                float x, y;
                unpack_f32x2(dk[c][r], x, y);
                store_pair<kAligned>(p.dk + at, (x + x2[0]) * p.scale, (y + x2[1]) * p.scale);
                unpack_f32x2(dv[c][r], x, y);
                store_pair<kAligned>(p.dv + at, x + x2[16 * D], y + x2[16 * D + 1]);
            }
        }
    }
}

gt_status check_feature_common(const gt_batch* batch, int32_t n_heads, int32_t head_dim)
{
    gt_status st = validate_batch(batch);
    if (st != GT_OK) return st;
    if (n_heads < 1) return GT_ERR_INVALID_ARG;
    if (head_dim != 32 && head_dim != 64) return GT_ERR_UNSUPPORTED;
    if (batch->n_graphs != 1 || n_heads > 65535) return GT_ERR_UNSUPPORTED;
    return GT_OK;
}

// What the pointers have in common: 16: vectors and bf16 pairs; 2: element by element; 1: not a bf16 tensor.
unsigned alignment(std::initializer_list<const void*> tensors)
{
    uintptr_t bits = 16;
    for (const void* t : tensors) bits |= reinterpret_cast<uintptr_t>(t);
    return (bits & 15u) == 0 ? 16u : ((bits & 1u) == 0 ? 2u : 1u);
}

// launches kernel<head_dim, aligned>
#define FEATURE_LAUNCH(kernel, grid, s, p)                                                                                            \
    (head_dim == 64 ? launch_overlapped(aligned ? kernel<64, true> : kernel<64, false>, grid, kThreads, 0, s, p)                     \
                    : launch_overlapped(aligned ? kernel<32, true> : kernel<32, false>, grid, kThreads, 0, s, p))

size_t dw_part_bytes(int32_t n, int32_t n_heads)
{
    return align_up((size_t)n_heads * (size_t)((n + kRows - 1) / kRows) * kFeat * sizeof(double), 256);
}

}  // namespace
}  // namespace gt

extern "C" gt_status gt_feature_attn_fwd(const void* q, const void* k, const void* v, const uint8_t* features, const float* weights,
                                         const gt_batch* batch, int32_t n_heads, int32_t head_dim,
                                         void* out, float* lse, void* stream)
{
    using namespace gt;
    gt_status st = check_feature_common(batch, n_heads, head_dim);
    if (st != GT_OK) return st;
    if (!q || !k || !v || !features || !weights || !out || !lse) return GT_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(features) & 3u) != 0) return GT_ERR_INVALID_ARG;
    const unsigned bytes = alignment({q, k, v, out});
    if (bytes < 2) return GT_ERR_INVALID_ARG;
    const bool aligned = bytes == 16;
    if (sm_count() <= 0) return GT_ERR_NO_DEVICE;
    FeatureArgs p{};
    p.q = (const __nv_bfloat16*)q; p.k = (const __nv_bfloat16*)k; p.v = (const __nv_bfloat16*)v;
    p.feat = (const uint32_t*)features;
    p.weights = weights;
    p.lse = lse;
    p.out = (__nv_bfloat16*)out;
    p.n = batch->n_total;
    p.n_heads = n_heads;
    p.scale = 1.0f / sqrtf((float)head_dim);
    const dim3 grid((unsigned)((p.n + kRows - 1) / kRows), (unsigned)n_heads);
    return FEATURE_LAUNCH(feature_fwd_kernel, grid, (cudaStream_t)stream, p);
}

extern "C" size_t gt_feature_attn_bwd_workspace(const gt_batch* batch, int32_t n_heads)
{
    if (gt::validate_batch(batch) != GT_OK || n_heads < 1) return 0;
    return gt::kHeaderBytes + gt::dw_part_bytes(batch->n_total, n_heads) + (size_t)batch->n_total * n_heads * sizeof(float);
}

extern "C" gt_status gt_feature_attn_bwd(const void* q, const void* k, const void* v, const void* dout, const float* lse,
                                         const uint8_t* features, const float* weights,
                                         const gt_batch* batch, int32_t n_heads, int32_t head_dim,
                                         void* dq, void* dk, void* dv, float* dweights,
                                         void* workspace, size_t workspace_bytes, void* stream)
{
    using namespace gt;
    gt_status st = check_feature_common(batch, n_heads, head_dim);
    if (st != GT_OK) return st;
    if (!q || !k || !v || !dout || !lse || !features || !weights || !dq || !dk || !dv || !dweights) return GT_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(features) & 3u) != 0) return GT_ERR_INVALID_ARG;
    const unsigned bytes = alignment({q, k, v, dout, dq, dk, dv});
    if (bytes < 2) return GT_ERR_INVALID_ARG;
    const bool aligned = bytes == 16;
    if (workspace == nullptr || workspace_bytes < gt_feature_attn_bwd_workspace(batch, n_heads) || misaligned16(workspace)) return GT_ERR_WORKSPACE;
    if (sm_count() <= 0) return GT_ERR_NO_DEVICE;
    uint8_t* ws = (uint8_t*)workspace;
    FeatureArgs p{};
    p.q = (const __nv_bfloat16*)q; p.k = (const __nv_bfloat16*)k; p.v = (const __nv_bfloat16*)v; p.dout = (const __nv_bfloat16*)dout;
    p.feat = (const uint32_t*)features;
    p.weights = weights;
    p.lse_in = lse;
    p.dw_part = (double*)(ws + kHeaderBytes);
    p.delta = (float*)(ws + kHeaderBytes + dw_part_bytes(batch->n_total, n_heads));
    p.dq = (__nv_bfloat16*)dq; p.dk = (__nv_bfloat16*)dk; p.dv = (__nv_bfloat16*)dv;
    p.dweights = dweights;
    p.n = batch->n_total;
    p.n_heads = n_heads;
    p.scale = 1.0f / sqrtf((float)head_dim);
    const dim3 grid((unsigned)((p.n + kRows - 1) / kRows), (unsigned)n_heads);
    cudaStream_t s = (cudaStream_t)stream;
    st = FEATURE_LAUNCH(feature_bwd_q_kernel, grid, s, p);
    if (st != GT_OK) return st;
    return FEATURE_LAUNCH(feature_bwd_kv_kernel, grid, s, p);
}
