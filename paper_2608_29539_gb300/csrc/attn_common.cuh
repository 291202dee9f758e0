// attn_common.cuh -- pieces shared by the attention forward and backward
// kernels: tile geometry, work-item decoding for the local (Eq. 6) and the
// query-sparse global (Eq. 8) branches, and the row/key visibility rule.
#pragma once
#include <cuda.h>

#include <cstdint>

#include "../../include/logo.h"

namespace logo {

constexpr int kBM = 128;              // query rows per tile (TMEM lanes)
constexpr int kBN = 128;              // keys per KV block
constexpr int kNoWindow = 1 << 30;    // "window" of the global branch (C^inf_t)
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

// One schedule entry of the global branch: a tile of up to 128 packed rows of
// one sequence, the range of real positions it covers (App. B: the KV blocks
// before min_pos need no causal predicate, those after max_pos none at all),
// and the KV blocks this entry visits: all of [0, max_pos / 128], or, when the
// tiles are too few to fill the GPU, one share of that range whose partial
// softmax result goes to a slot that a merge kernel combines with the others.
struct GlobalTile {
    int row0;     // first packed row
    int nrows;    // rows in the tile (1..128)
    int b;        // sequence
    int min_pos;  // position of the first row
    int max_pos;  // position of the last row
    int blk_lo;   // KV blocks visited (inclusive)
    int blk_hi;
    int slot;     // -1: the whole range, output written directly; else the partial-result slot
    int cost;     // KV blocks visited (the ordering key)
    int pad0, pad1, pad2;
};

// A tile whose KV range is split: the merge kernel combines slots
// slot0 .. slot0 + nsplit - 1 into its output rows.
struct SplitTile {
    int row0, nrows, slot0, nsplit;
};

// Everything the roles of a forward CTA need to know about one work item.
struct FwdItem {
    int b, h, kvh;
    int row0;       // local: first query position; global: first packed row
    int nrows;      // valid rows
    int pos_min, pos_max;
    int blk_lo, blk_hi;  // inclusive KV block range
    int slot;            // global split entry: partial-result slot; otherwise -1
};

// Rows see keys s with pos - W < s <= pos.
__device__ __forceinline__ bool key_visible(int key, int pos, int window)
{
    return key <= pos && key > pos - window;
}

// 32 columns as a bit mask: bit c set for lo <= c <= hi (either may lie
// outside 0..31; PTX shifts by 32 and more give 0).
__device__ __forceinline__ uint32_t column_mask(int lo, int hi)
{
    uint32_t up, down;
    asm("shr.u32 %0, 0xffffffff, %1;" : "=r"(up) : "r"(max(31 - hi, 0)));
    asm("shl.b32 %0, 0xffffffff, %1;" : "=r"(down) : "r"(max(lo, 0)));
    return up & down;
}

// Four lanes (a quad) hold, each, the bf16 pair of columns 8k + 2j, 8k + 2j + 1
// of a row for k = 0..3 (j the lane's place in the quad): afterwards lane j has
// the 8 adjacent columns 8j .. 8j + 7.
__device__ __forceinline__ uint4 quad_gather8(const uint32_t (&x)[4], int lane)
{
    const bool b0 = lane & 1, b1 = lane & 2;
    const uint32_t r0 = __shfl_xor_sync(0xffffffffu, b0 ? x[0] : x[1], 1);
    const uint32_t r1 = __shfl_xor_sync(0xffffffffu, b0 ? x[2] : x[3], 1);
    const uint32_t y0 = b0 ? r0 : x[0], y1 = b0 ? x[1] : r0, y2 = b0 ? r1 : x[2], y3 = b0 ? x[3] : r1;
    const uint32_t q0 = __shfl_xor_sync(0xffffffffu, b1 ? y0 : y2, 2);
    const uint32_t q1 = __shfl_xor_sync(0xffffffffu, b1 ? y1 : y3, 2);
    return b1 ? make_uint4(q0, q1, y2, y3) : make_uint4(y0, y1, q0, q1);
}

// Sequence of packed row `row`: the b with cu_q[b] <= row < cu_q[b+1].
__device__ __forceinline__ int seq_of_row(const int32_t* cu_q, int B, int row)
{
    int lo = 0, hi = B - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (cu_q[mid] <= row) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

}  // namespace logo
