// Structures shared by the host entry points and the kernels.
#pragma once
#include <cstdint>
#include <cuda.h>

namespace vpp {

constexpr int kTileM = 128;  // query rows per MMA tile
constexpr int kTileN = 128;  // keys per KV tile

// One schedulable unit: a run of consecutive query rows of one request restricted to a range of KV tiles.
// The attention kernel turns (unit, head slot) pairs into work items.
struct __align__(16) WorkUnit {
    int32_t req;        // request index
    int32_t q_row0;     // first packed query row of the tile
    int32_t rows;       // query rows (tokens) of the unit (at most 256) and its number of splits (merge launches): rows | splits << 16
    int32_t pos0;       // absolute position of the tile's first row (prefix_len + row offset)
    int32_t kv_begin;   // first KV tile (units of kTileN keys)
    int32_t kv_end;     // one past the last KV tile
    int32_t split;      // split index of this unit, or -1 when the tile is not split (final output)
    int32_t kv_len;     // prefix_len + chunk_len of the request: keys at or beyond it do not exist
};
// A unit as the attention kernels use it: `rows` alone, the split count aside.
__device__ __forceinline__ int take_splits(WorkUnit& u) {
    const int n = u.rows >> 16;
    u.rows &= 0xffff;
    return n;
}

constexpr int kMaxCheckers = 8;   // blocks of the work-decomposition kernel that check the block table

// Head of the workspace; written by the work-decomposition kernel, read in one go (read_header).
struct __align__(16) WorkHeader {
    int32_t num_units;    // units in the sorted list
    int32_t num_short;    // the last num_short units of the list are the short ones: their rows fill at most one tile
    int32_t unit_block;   // units per locality block of the item order (see decode_item)
    int32_t error;        // VPP_DEV_* (0 = ok) of the lengths
    int32_t counter;      // persistent-kernel work counter
    int32_t num_checkers; // blocks that checked a part of the block table
    int32_t num_lead;     // units at the start of the list that are handed out before the short ones (d = 128 kernel)
    int32_t pad;
    int32_t bad_table[kMaxCheckers];   // one word each: VPP_DEV_BAD_BLOCK if it found an entry out of range, else 0
};
static_assert(kMaxCheckers == 8, "read_header");

// The head of the work list as the kernels after the decomposition see it: nothing to do when a check failed.
struct WorkList {
    int32_t num_units, num_short, unit_block, error, num_lead;
};
__device__ __forceinline__ WorkList read_header(const WorkHeader* h) {
    const int4* q = reinterpret_cast<const int4*>(h);
    const int4 a = q[0], b = q[1], c = q[2], d = q[3];   // (independent loads: one round trip)
    const int bad[8] = {c.x, c.y, c.z, c.w, d.x, d.y, d.z, d.w};
    WorkList w{a.x, a.y, a.z, a.w, b.z};
#pragma unroll
    for (int i = 0; i < 8; ++i)
        if (w.error == 0 && i < b.y) w.error = bad[i];
    if (w.error != 0) w.num_units = w.num_short = w.num_lead = 0;
    return w;
}

struct WorkspaceLayout {
    size_t header;      // WorkHeader
    size_t units;       // WorkUnit[max_units]
    size_t row_splits;  // int32[total_q]: number of partials to merge for each query row (0/1: none)
    size_t o_parts;     // float[S][total_q][Hq][Dv]
    size_t lse_parts;   // float[S][total_q][Hq]
    size_t total;
    int32_t max_units;
    int32_t splits;     // S, the most parts a unit may get
    int32_t balanced;   // 1: the work decomposition chooses each unit's own number (prep.cuh)
};

struct AttnParams {
    const int32_t* block_table;   // may be null (contiguous)
    int32_t max_blocks_per_req;
    int32_t block_shift;          // log2(block_size) (paged only)
    int32_t num_blocks;
    int32_t num_q_heads;
    int32_t num_kv_heads;
    int32_t total_q;
    // d = 128 kernel, how tile rows are packed: row r of a tile is q-head h0 + r % group of token r / group
    int32_t group, tile_tokens;               // items of two tiles
    int32_t short_group, short_tokens;        // items of one tile (short units)
    // d = 128 kernel, K/V copies: (block b, kv-head g) is coordinate b * block_units + g * head_units of a cache's map
    int32_t k_block_units, k_head_units, k_end;   // (k_end: one past the last: reads as zero)
    int32_t v_block_units, v_head_units, v_end;
    int32_t exact_from;                       // tiles that reach past this position take the copies of 8 keys
    float scale_log2e;            // softmax_scale * log2(e)
    void* out;                    // bf16 [T, Hq, Dv]
    float* lse;                   // [T, Hq] or null
    float* o_parts;               // [S, T, Hq, Dv]
    float* lse_parts;             // [S, T, Hq]
    const WorkHeader* header_ro;
    WorkHeader* header;
    const WorkUnit* units;
    int32_t* row_splits;          // [T] number of partial results of every query row, for the merge kernel (null: no merge)
    int32_t* status;              // may be null
};

constexpr int kSlabBytes = kTileM * 128;  // 128 rows x 64 bf16, 128B-swizzled

// Which (unit, head slot) a flat work index means.  Units arrive sorted by decreasing cost; inside
// a block of `unit_block` consecutive units the items are ordered kv-head-major so that CTAs
// running at the same time read the same K/V pages (L2 reuse), while blocks keep the longest-first order.
__device__ __forceinline__ void decode_item(int w, int num_units, int unit_block, int items_per_unit, int per_kv_head, int& unit,
                                            int& slot) {
    const int blk_items = unit_block * items_per_unit;
    const int ub = w / blk_items;
    const int rem = w - ub * blk_items;
    const int left = num_units - ub * unit_block;
    const int nblk = left < unit_block ? left : unit_block;
    const int per_g = nblk * per_kv_head;
    const int g = rem / per_g;
    const int rem2 = rem - g * per_g;
    unit = ub * unit_block + rem2 / per_kv_head;
    slot = g * per_kv_head + rem2 % per_kv_head;
}

}  // namespace vpp
