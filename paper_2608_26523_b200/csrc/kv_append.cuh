// Paged KV-cache append: the chunk's new key / value rows go to cache positions [prefix_len, prefix_len + chunk_len)
// of their request (the step that precedes the attention of the same chunk; the paper's chunked-prefill section).
// Pure data movement, HBM-bound: every byte is read once and written once.
//
// A warp takes one piece of a token row at a time: up to kAppendPiece 16-byte vectors of the row's (kv-head, vector)
// units, a 4 KB row of eight kv-heads whole.  Its loads are all issued first -- kAppendUnroll in flight per lane -- and the
// row's destination is looked up while they are in flight: lane 0 finds the request (binary search in the exclusive scan
// of chunk_len that every block builds in shared memory) and the page.  The block after the copying ones checks the
// lengths and pages of the whole launch and writes *status, so that the call needs no memset before it.
// 134 MB (16384 rows of eight kv-heads): 28.0 -> 24.4 us a call, 5.5 TB/s; the rest to the copy rate (20.6 us) is one launch.
#pragma once
#include <cstdint>

#include "ptx.cuh"

namespace vpp {

constexpr int kAppendThreads = 256;
constexpr int kAppendUnroll = 8;
constexpr int kAppendPiece = 32 * kAppendUnroll;   // 16-byte vectors a warp moves at a time
constexpr int kAppendMaxReqs = 8192;   // the scan of chunk_len lives in shared memory (32 KB + 4)

struct AppendParams {
    const uint4* k_new;      // [total_q, Hkv, Dqk] bf16 as 16-byte vectors
    const uint4* v_new;      // [total_q, Hkv, Dv] or null
    uint8_t* k_cache;
    uint8_t* v_cache;
    long long k_block_stride, k_token_stride, k_head_stride;   // bytes
    long long v_block_stride, v_token_stride, v_head_stride;   // bytes
    const int32_t* block_table;
    const int32_t* prefix_len;
    const int32_t* chunk_len;
    int num_reqs, max_blocks_per_req, block_shift, num_blocks;
    long long capacity;      // positions a request can hold: max_blocks_per_req * block_size (or the contiguous extent)
    int total_q, num_kv_heads;
    int k_vecs, v_vecs;      // 16-byte vectors per (token, kv-head) row of K and of V (0 when v_new is null)
    int32_t* status;
};

__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

// Exclusive scan of chunk_len into cu[0 .. num_reqs] (shared memory); true if the lengths describe the launch.
__device__ __forceinline__ bool append_scan(const AppendParams& p, int32_t* cu) {
    __shared__ int s_bad;
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) s_bad = 0;
    __syncthreads();
    bool bad = false;
    for (int r = tid; r < p.num_reqs; r += kAppendThreads) {   // (all loads at once, then the scan from shared memory)
        int c = p.chunk_len[r];
        const int pre = p.prefix_len[r];
        if (c < 0 || pre < 0 || static_cast<long long>(pre) + c > p.capacity) {
            bad = true;
            c = 0;
        }
        cu[r] = c;
    }
    if (bad) s_bad = 1;
    __syncthreads();
    if (tid < 32) {
        int carry = 0;
        for (int base = 0; base < p.num_reqs; base += 32) {
            const int r = base + lane;
            const int c = r < p.num_reqs ? cu[r] : 0;
            int x = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (r < p.num_reqs) cu[r] = carry + x - c;
            carry += __shfl_sync(0xffffffffu, x, 31);
        }
        if (lane == 0) cu[p.num_reqs] = carry;
    }
    __syncthreads();
    return !s_bad && cu[p.num_reqs] == p.total_q;
}

// Request of row g (0 <= g < total_q): the last r with cu[r] <= g.
__device__ __forceinline__ int append_request(const int32_t* cu, int num_reqs, int g) {
    int lo = 0, hi = num_reqs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (cu[mid] <= g) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// The verdict on the launch (one block): lengths, and the pages of every row.  Looked up are the pages of each request's first and
// last row and of every block_size-th row of the launch: rows of a request that follow one another among these are at most a page
// apart, so every page is among theirs.  The threads share the rows, not the requests (one long chunk among many short ones: 8192
// rows in pages of 16 and 255 single rows took 37 us with a thread walking the long one's pages, 11.6 now), with kAppendProbes look-ups in flight each.
constexpr int kAppendProbes = 4;
__device__ __forceinline__ void append_status(const AppendParams& p, const int32_t* cu, bool lengths_ok) {
    bool bad = false;
    if (lengths_ok && p.block_table != nullptr) {
        auto outside = [&](int r, int pos) {
            const int e = __ldg(p.block_table + static_cast<long long>(r) * p.max_blocks_per_req + (pos >> p.block_shift));
            return e < 0 || e >= p.num_blocks;
        };
        for (int r0 = threadIdx.x; r0 < p.num_reqs; r0 += kAppendProbes * kAppendThreads) {
            int pre[kAppendProbes], n[kAppendProbes];
#pragma unroll
            for (int i = 0; i < kAppendProbes; ++i) {
                const int r = r0 + i * kAppendThreads;
                n[i] = r < p.num_reqs ? cu[r + 1] - cu[r] : 0;
                pre[i] = n[i] > 0 ? __ldg(p.prefix_len + r) : 0;
            }
#pragma unroll
            for (int i = 0; i < kAppendProbes; ++i)
                if (n[i] > 0) bad |= outside(r0 + i * kAppendThreads, pre[i]) | outside(r0 + i * kAppendThreads, pre[i] + n[i] - 1);
        }
        const long long step = 1ll << p.block_shift;
        for (long long g0 = threadIdx.x * step; g0 < p.total_q; g0 += kAppendProbes * kAppendThreads * step) {
            int r[kAppendProbes], pos[kAppendProbes];
#pragma unroll
            for (int i = 0; i < kAppendProbes; ++i) {
                const long long g = g0 + i * kAppendThreads * step;
                r[i] = g < p.total_q ? append_request(cu, p.num_reqs, static_cast<int>(g)) : -1;
                pos[i] = r[i] >= 0 ? __ldg(p.prefix_len + r[i]) + static_cast<int>(g - cu[r[i]]) : 0;
            }
#pragma unroll
            for (int i = 0; i < kAppendProbes; ++i)
                if (r[i] >= 0) bad |= outside(r[i], pos[i]);
        }
    }
    const int any = __syncthreads_or(bad);
    if (threadIdx.x == 0) *p.status = !lengths_ok ? 1 /* VPP_DEV_BAD_LENGTHS */ : any ? 2 /* VPP_DEV_BAD_BLOCK */ : 0;
}

// The first copy_blocks blocks copy; the block after them, if there is one, writes the status.
__global__ void __launch_bounds__(kAppendThreads) kv_append_kernel(const AppendParams p, const int copy_blocks) {
    extern __shared__ int32_t cu[];   // cu[r] = rows before request r; cu[num_reqs] = total
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_launch_dependents();
    pdl_wait();                       // the rows and the lengths may come from the kernel launched just before
    const bool ok = append_scan(p, cu);
    if (static_cast<int>(blockIdx.x) >= copy_blocks) {
        append_status(p, cu, ok);
        return;
    }
    if (!ok) return;                  // lengths that do not describe this launch: write nothing
    const int units_k = p.num_kv_heads * p.k_vecs, units = units_k + p.num_kv_heads * p.v_vecs;
    const int pieces = (units + kAppendPiece - 1) / kAppendPiece;
    const long long tasks = static_cast<long long>(p.total_q) * pieces, stride = copy_blocks * (kAppendThreads / 32);
    for (long long task = blockIdx.x * (kAppendThreads / 32) + warp; task < tasks; task += stride) {
        const int row = static_cast<int>(task / pieces);
        const int u0 = static_cast<int>(task - static_cast<long long>(row) * pieces) * kAppendPiece + lane;
        const uint4* k_src = p.k_new + static_cast<long long>(row) * units_k;
        const uint4* v_src = p.v_new + static_cast<long long>(row) * (units - units_k);
        uint4 v[kAppendUnroll];
#pragma unroll
        for (int i = 0; i < kAppendUnroll; ++i) {
            const int u = u0 + 32 * i;
            if (u < units) v[i] = ld_stream(u < units_k ? k_src + u : v_src + (u - units_k));
        }
        long long blk = 0;
        int slot = 0;
        if (lane == 0) {
            const int lo = append_request(cu, p.num_reqs, row);
            const int pos = p.prefix_len[lo] + (row - cu[lo]);
            if (p.block_table == nullptr) {
                blk = lo;
                slot = pos;
            } else {
                blk = p.block_table[static_cast<long long>(lo) * p.max_blocks_per_req + (pos >> p.block_shift)];
                slot = pos & ((1 << p.block_shift) - 1);
                if (blk < 0 || blk >= p.num_blocks) blk = -1;
            }
        }
        blk = __shfl_sync(0xffffffffu, blk, 0);
        slot = __shfl_sync(0xffffffffu, slot, 0);
        if (blk < 0) continue;   // the row's page is not valid: skip the row
        uint8_t* k_dst = p.k_cache + blk * p.k_block_stride + slot * p.k_token_stride;
        uint8_t* v_dst = p.v_cache + blk * p.v_block_stride + slot * p.v_token_stride;
#pragma unroll
        for (int i = 0; i < kAppendUnroll; ++i) {
            const int u = u0 + 32 * i;
            if (u >= units) continue;
            if (u < units_k) {
                const int g = u / p.k_vecs, j = u - g * p.k_vecs;
                *reinterpret_cast<uint4*>(k_dst + g * p.k_head_stride + j * 16) = v[i];
            } else {
                const int w = u - units_k, g = w / p.v_vecs, j = w - g * p.v_vecs;
                *reinterpret_cast<uint4*>(v_dst + g * p.v_head_stride + j * 16) = v[i];
            }
        }
    }
}

}  // namespace vpp
