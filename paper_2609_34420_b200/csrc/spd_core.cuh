// Targets that the bit-matrix build (spd_build.cu) does not search for: their distances follow from their in-neighbours'.
#pragma once

#include "gt_common.cuh"

namespace gt {

constexpr int kCoreMaxDegree = 8;          // in-neighbours of a target that is left out, at most
constexpr int kCoreSegment = 4096;         // targets of one step of half a block of the expansion
// All targets searched for -> the core.  Power-law graphs: 32 768 nodes of degree 8 1.73 -> 1.47 ms, 33 000 of degree 6 2.52 -> 1.60, 40 000 of
// degree 12 3.30 -> 2.31, 65 536 6.95 -> 4.76 (of degree 22 7.00 -> 5.70).  60 000 nodes: preferential attachment of degree 10 5.09 -> 4.76,
// Erdos-Renyi of degree 6 13.0 -> 6.6, a random tree 53 -> 22; geometric of 33 000 nodes, degree 4 10.7 -> 8.2.  Below, the shorter rows leave
// the chip idle and the expansion costs more than they save: 24 000 of degree 12 1.03 -> 1.23, 19 000 of degree 8 0.93 -> 1.18.  A graph
// that is turned down pays for the choice: 15 us without many vertices of few edges, else up to 115 (power law of 65 536 nodes, degree 26:
// 6.51 -> 6.62 ms; geometric of 33 000 nodes, degree 6: 118 ms either way).
constexpr int kCoreMinNodes = 32768;
constexpr int kCoreMaxNodes = 65536;       // vertices are numbered in 16 bits
constexpr int kCoreMaxGroups = 5;
constexpr int kCoreMaxLevels = 13;         // a distance and "none" in four bits, after one hop more
// Levels without a plane of their own wait in the rows of the matrix, where a target has a byte and these levels have a bit of it each.
// Five column blocks leave five or six planes: what came later went through a pool of rows in the workspace, and where that ran over through
// bytes that were written, blended and read again (of the graphs above, those of degree 10, 6 and 22: 7.38, 13.7 and 8.39 ms).
constexpr int kCoreLateLevels = 8;
// Word `w` of a bit row of `row_words` at the k-th of them, in words from where the column block begins in a row of the matrix.  All
// levels of 128 words lie together, where the output pass puts these words' bytes (a warp reads and then writes as much at a time).
__host__ __device__ constexpr uint32_t core_late_word(int k, int w, int row_words)
{
    return (uint32_t)((w >> 7) * 1024 + k * (row_words - (w & ~127) < 128 ? row_words - (w & ~127) : 128) + (w & 127));
}

// What the search is told, and what it tells the expansion.  In the workspace.
struct CoreInfo {
    int32_t reduced;                       // 0: every vertex is a target of the search, and it writes the matrix itself
    int32_t n_cols;                        // targets of the search
    int32_t block_bits;                    // targets of a column block, a multiple of 128
    int32_t row_words;                     // pitch of a bit row
    int32_t n_groups;                      // column blocks in work at a time
    int32_t n_planes;                      // levels with a plane of their own
    int32_t deep;                          // some block has more than kCoreMaxLevels: its distances are bytes at the rows' beginnings
    int32_t levels[kCoreMaxGroups];        // levels of a column block; 0: bytes
};

struct CorePlan {
    bool enabled;
    int groups;                            // column blocks that bit rows are allocated for
    size_t clear_off, clear_bytes;         // in-degrees and marks, to be zeroed
    size_t slot_off, bits_off, col_off, loc_off, group_off, list_off, info_off, total_bytes;
};

CorePlan spd_core_plan(int32_t n, int groups, size_t off, bool wanted);

struct CoreParams {
    const int32_t* row_ptr;
    const int32_t* col_idx;
    const int4* items;                     // the search's work items {vertex, first edge, one past the last, ..}, up to 32 edges each
    const int32_t* item_start;             // [n]: how many
    uint32_t* in_degree;                   // [n]
    uint8_t *lost, *out, *lost_again;      // [n] marks of the choice
    uint32_t* candidates;                  // vertices of few out-edges
    uint16_t* slots;                       // [n][kCoreMaxDegree] in-neighbours
    uint32_t* left_out;                    // [n / 32] a bit per vertex
    int32_t* column;                       // [n] column of a target of the search, -1: left out
    uint16_t* loc;                         // [pitch] word of a target in the expansion's shared memory
    uint2* groups;                         // [segments][16] a warp's groups of 32 targets: their lists, and how long they are
    uint32_t* list;                        // [segments][kCoreSegment * kCoreMaxDegree / 2] pairs of words
    CoreInfo* info;
    int32_t n;
    int32_t n_groups;                      // as allocated
    int32_t plane_words;                   // words per vertex that the frontiers may take
};

// Chooses the targets; fills *info and the expansion's lists.
gt_status spd_core_launch(const CorePlan& plan, CoreParams& p, uint8_t* ws, const int32_t* row_ptr, const int32_t* col_idx,
                          int32_t n, int64_t nnz, const int4* items, const int32_t* item_start, int plane_words, cudaStream_t s);

// The matrix from the frontiers (or the bytes) of the search's targets.
gt_status spd_core_expand(const CoreParams& p, const uint32_t* planes, const uint8_t* nonempty, int32_t n_pad, int flag_planes,
                          int32_t max_dist, uint8_t* spd, cudaStream_t s);

}  // namespace gt
