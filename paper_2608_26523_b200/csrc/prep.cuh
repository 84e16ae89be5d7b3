// Work decomposition: from the per-request (prefix_len, chunk_len) on the device, build the list of
// work units (a run of query rows x key-range split) ordered by decreasing cost, so that the
// persistent attention kernel can hand out tiles of very unequal cost longest-first.
//
// A unit whose first row sits at absolute position pos0 needs the KV tiles
// [0, ceil((pos0 + rows) / 128)); its cost is that count -- it grows linearly with the prefix,
// which is the per-chunk imbalance the paper's Eq. 2 models.
//
// Latency-bound (a launch of a few work items waits for it), so: one block of as many threads as the launch has units,
// the requests' lengths and scans in shared memory, one scan for both prefix sums, two cost bins per thread.
#pragma once
#include "common.cuh"
#include "ptx.cuh"

namespace vpp {

constexpr int kPrepMinThreads = 128, kPrepMaxThreads = 1024;
constexpr int kPrepSmemReqs = 1024;   // up to so many requests the lengths and scans live in shared memory

struct PrepParams {
    const int32_t* prefix_len;
    const int32_t* chunk_len;
    const int32_t* block_table;  // may be null
    int32_t num_reqs;
    int32_t total_q;
    int32_t max_seq_len;
    int32_t max_blocks_per_req;
    int32_t block_shift;
    int32_t num_blocks;
    int32_t splits;      // S >= 1
    int32_t max_units;
    int32_t unit_rows;   // query rows per unit
    int32_t short_rows;  // units of at most so many rows go to the end of the list (packed items)
    int32_t unit_block, ragged_unit_block;   // units per locality block of the item order (common.cuh): about equally long units, others (parts of a balanced cut: 1)
    // Balanced cut (the library's own choice of splits for launches of few work items):
    int32_t balanced;    // 1: cut the launch's KV tiles into equal shares of the SMs, `splits` being the most a unit may get
    int32_t slots;       // CTAs (or CTA pairs) that take work items
    int32_t unit_items, short_items;      // work items of a unit and of a short unit
    int32_t ranges, short_ranges;         // into how many equal ranges a launch of one kind of units is cut
    float unit_us, short_us;              // time of a KV tile of an item
    float short_per_unit;                 // short_us / unit_us
    int32_t lead_items;                   // launches of fewer items put the long units of two tiles before the short ones (0: none)
    int32_t min_len, min_short_len;       // fewest KV tiles worth a work item
    int32_t lead, short_lead;             // what starting and ending a work item costs, in KV tiles
    int32_t partial;     // 1: key-range restricted launch whose results are partial (o fp32, lse) of "split 0"
    int32_t range_begin; // first KV tile of the key range (partial launches)
    int32_t range_end;   // one past its last KV tile
    WorkHeader* header;
    WorkUnit* units;
    int32_t* q_start;     // [num_reqs + 1] scratch
    int32_t* tile_start;  // [num_reqs + 1] scratch
};

// Exclusive scan of two counts per thread over the block: (before a, before b, total a, total b).  Out of line and rolled up:
// the kernel runs once through its code, which comes from far away, so its size is its latency.
__device__ __noinline__ int4 block_scan2(int a, int b, int2* warp_sums) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int ia = a, ib = b;
#pragma unroll 1
    for (int o = 1; o < 32; o <<= 1) {
        const int ta = __shfl_up_sync(0xffffffffu, ia, o), tb = __shfl_up_sync(0xffffffffu, ib, o);
        if (lane >= o) {
            ia += ta;
            ib += tb;
        }
    }
    if (lane == 31) warp_sums[warp] = make_int2(ia, ib);
    __syncthreads();
    // every warp scans the warp totals for itself
    const int2 w = lane < nw ? warp_sums[lane] : make_int2(0, 0);
    int wa = w.x, wb = w.y;
#pragma unroll 1
    for (int o = 1; o < 32; o <<= 1) {
        const int ta = __shfl_up_sync(0xffffffffu, wa, o), tb = __shfl_up_sync(0xffffffffu, wb, o);
        if (lane >= o) {
            wa += ta;
            wb += tb;
        }
    }
    int4 r;
    r.z = __shfl_sync(0xffffffffu, wa, 31);
    r.w = __shfl_sync(0xffffffffu, wb, 31);
    r.x = __shfl_sync(0xffffffffu, wa - w.x, warp) + ia - a;
    r.y = __shfl_sync(0xffffffffu, wb - w.y, warp) + ib - b;
    __syncthreads();
    return r;
}

// Number of key-range splits of the unit whose first row is at absolute position pos0:
// every split must start at or before pos0 so that each row sees at least one key in each split.
__device__ __forceinline__ int tile_num_splits(int pos0, int S) {
    const int splittable = pos0 / kTileN + 1;  // KV tiles that start at or before pos0
    return S < splittable ? S : splittable;
}

__device__ __forceinline__ void split_range(int pos0, int n_tiles, int nsplit, int s, int& kb, int& ke) {
    const int splittable = pos0 / kTileN + 1;
    // (at most 64 splits of at most 2^24 tiles: 32 bits are enough, and a division of 64 is the longest step of a small launch)
    kb = static_cast<uint32_t>(s) * splittable / static_cast<uint32_t>(nsplit);
    ke = (s + 1 == nsplit) ? n_tiles : static_cast<uint32_t>(s + 1) * splittable / static_cast<uint32_t>(nsplit);
}

// Every block-table entry a request needs must name a real block.  A batch of decode rows over small pages needs a
// hundred thousand entries, so blocks 1 .. gridDim.x - 1 of the work-decomposition kernel check them while block 0 does
// the decomposition: the warps of all these blocks share the requests (several warps to a request when there are few),
// four loads in flight per lane, one verdict word per block.  (Measured on 256 rows with 16-token pages: 187 us when one
// block walked the requests one after the other, a quarter of the launch; the launch is 1.22 times as fast now.)
__device__ __forceinline__ void check_block_table(const PrepParams& p, int checker, int num_checkers) {
    const int warps = blockDim.x >> 5, lane = threadIdx.x & 31;
    const int n_warps = num_checkers * warps, w = checker * warps + (threadIdx.x >> 5);
    const int per_req = p.num_reqs >= n_warps ? 1 : n_warps / p.num_reqs;    // warps that share a request
    const int groups = n_warps / per_req, grp = w / per_req, part = w % per_req;
    bool bad = false;
    for (int r = grp; r < p.num_reqs && grp < groups; r += groups) {
        const int P = p.prefix_len[r], C = p.chunk_len[r];
        const long long kv_len = static_cast<long long>(P) + C;
        if (P < 0 || C <= 0 || kv_len > p.max_seq_len) continue;             // (block 0 reports bad lengths)
        const int nb = static_cast<int>((kv_len + (1 << p.block_shift) - 1) >> p.block_shift);
        if (nb > p.max_blocks_per_req) {
            bad = true;
            continue;
        }
        const int32_t* row = p.block_table + static_cast<long long>(r) * p.max_blocks_per_req;
        for (int b = part * 128 + lane; b < nb; b += per_req * 128) {
            int e[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) e[i] = b + 32 * i < nb ? __ldg(row + b + 32 * i) : 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) bad |= e[i] < 0 || e[i] >= p.num_blocks;
        }
    }
    const int any = __syncthreads_or(bad);
    if (threadIdx.x == 0) p.header->bad_table[checker] = any ? 2 /* VPP_DEV_BAD_BLOCK */ : 0;
}

// In a batch of few items, the units of two tiles that take longer than the longest short one go before the short ones: those in front
// of the bin of this length.  (64 tokens at 8000 keys and 30 decode rows at 4000 to 4400 of 64/8 heads: 212 us with all of them at
// the end, 155 so.  Where there are several items to a slot the end is filled anyway: a mixed batch of 14 lost 0.5 %.)
// (out of line: see block_scan2)
__device__ __noinline__ void put_long_units_first(WorkHeader* header, const int* bins, int short_bin, float bin_scale, float short_per_unit,
                                                  int lead, int short_lead) {
    const int nthr = blockDim.x;
    const float as_long = (2 * nthr - 1 - short_bin) * short_per_unit + (short_lead * short_per_unit - lead) * bin_scale;
    if (threadIdx.x == 0) header->num_lead = bins[min(max(nthr - 1 - static_cast<int>(as_long), 0), nthr - 1)];
    __syncthreads();
}

__global__ void __launch_bounds__(kPrepMaxThreads, 1) prep_kernel(const PrepParams p) {
    __shared__ int2 warp_sums[32];
    __shared__ int bins[2 * kPrepMaxThreads];   // blockDim.x bins of decreasing cost, then as many for the short units
    __shared__ int s_P[kPrepSmemReqs], s_C[kPrepSmemReqs], s_q[kPrepSmemReqs], s_t[kPrepSmemReqs + 1];
    __shared__ int s_error, s_max, s_min, s_normal, s_items, s_short_bin;
    const int tid = threadIdx.x, nthr = blockDim.x;
    pdl_launch_dependents();   // the attention kernel may set itself up (barriers, tensor memory) while this runs
    pdl_wait();                // the lengths may come from the kernel launched just before; the workspace may be in use by it
    if (blockIdx.x > 0) {
        check_block_table(p, blockIdx.x - 1, gridDim.x - 1);
        return;
    }
    const bool in_smem = p.num_reqs <= kPrepSmemReqs;
    int* const qs = in_smem ? s_q : p.q_start;     // first packed row / first unit of every request
    int* const ts = in_smem ? s_t : p.tile_start;
    const int* const Ps = in_smem ? s_P : p.prefix_len;
    const int* const Cs = in_smem ? s_C : p.chunk_len;
    if (tid == 0) {
        s_error = 0;
        s_max = 1;
        s_min = 1 << 30;
        s_short_bin = 2 * nthr;
        p.header->num_checkers = gridDim.x - 1;
    }
    bins[tid] = 0;
    bins[nthr + tid] = 0;
    __syncthreads();

    // ---- phase 1: validate lengths, scan chunk lengths and unit counts over requests ----
    int carry_q = 0, carry_t = 0;
#pragma unroll 1
    for (int base = 0; base < p.num_reqs; base += nthr) {
        const int r = base + tid;
        int P = 0, c = 0;
        if (r < p.num_reqs) {
            P = p.prefix_len[r];
            c = p.chunk_len[r];
            // (a key range must start inside every request's prefix, so that each query row sees at least one of its keys)
            if (P < 0 || c < 0 || static_cast<long long>(P) + c > p.max_seq_len ||
                (p.partial && c > 0 && P < p.range_begin * kTileN)) {
                s_error = 1;
                c = 0;
            }
            if (c > 0) {
                atomicMax(&s_max, (P + c + kTileN - 1) / kTileN);                                      // longest unit,
                atomicMin(&s_min, (P + (c < p.unit_rows ? c : p.unit_rows) + kTileN - 1) / kTileN);   // shortest
            }
        }
        const int4 sc = block_scan2(c, (c + p.unit_rows - 1) / p.unit_rows, warp_sums);
        if (r < p.num_reqs) {
            if (in_smem) {
                s_P[r] = P;
                s_C[r] = c;
            }
            qs[r] = carry_q + sc.x;
            ts[r] = carry_t + sc.y;
        }
        carry_q += sc.z;
        carry_t += sc.w;
    }
    const int total_units = carry_t;
    if (tid == 0) ts[p.num_reqs] = total_units;
    __syncthreads();
    if (s_error != 0 || carry_q != p.total_q) {
        if (tid == 0) {
            p.header->num_units = 0;
            p.header->num_short = 0;
            p.header->counter = 0;
            p.header->error = 1 /* VPP_DEV_BAD_LENGTHS */;
        }
        return;
    }

    // ---- phase 2: counting sort of the units by decreasing cost, two passes; before them, for a balanced cut, one that
    //      adds the KV tiles up: how many of them does a work item get? ----
    // The KV tiles of the units of a kind (the short ones, the others) laid end to end are cut at the multiples of the kind's `len`, so
    // that every range is one slot's share and a unit is cut only where a share ends in it (few partial results); every unit
    // begins with `lead` tiles that stand for the start and end of one more item in the share it begins in.
    int sum = 0, sum_short = 0, len = 0, len_short = 0;
    float bin_scale = static_cast<float>(nthr - 1) / static_cast<float>(s_max);
    // this thread's unit, its parts: the first of `first` KV tiles, then `part` each, the last what is left (part = 0: equal parts)
    const bool once = total_units <= nthr;   // (then both are worked out once)
    int r = 0, row_off = 0, rows = 0, pos0 = 0, n_tiles = 0, nsplit = 0;
    int before = 0, first = 0, part = 0;
    const int first_pass = p.balanced ? 0 : 1;
#pragma unroll 1
    for (int pass = first_pass; pass < 3; ++pass) {
        int carry = 0, carry_short = 0;
#pragma unroll 1
        for (int base = 0; base < total_units; base += nthr) {
            const int gt = base + tid;
            if (pass == first_pass || !once) {
                r = 0;
                n_tiles = 0;
                rows = 0;
                nsplit = 0;
                if (gt < total_units) {
                    int hi = p.num_reqs - 1;          // request of unit gt: last r with ts[r] <= gt
                    while (r < hi) {
                        const int mid = (r + hi + 1) >> 1;
                        if (ts[mid] <= gt) r = mid; else hi = mid - 1;
                    }
                    row_off = (gt - ts[r]) * p.unit_rows;
                    rows = Cs[r] - row_off < p.unit_rows ? Cs[r] - row_off : p.unit_rows;
                    pos0 = Ps[r] + row_off;
                    n_tiles = (pos0 + rows + kTileN - 1) / kTileN;
                }
            }
            const bool is_short = rows <= p.short_rows;
            if (p.balanced && (pass == 0 || !once)) {
                const int lead = is_short ? p.short_lead : p.lead, n = n_tiles > 0 ? n_tiles + lead : 0;
                const int4 sc = block_scan2(is_short ? 0 : n, is_short ? n : 0, warp_sums);
                before = (is_short ? carry_short + sc.y : carry + sc.x) + lead;
                carry += sc.z;
                carry_short += sc.w;
                if (pass == 0) {
                    sum += sc.z;
                    sum_short += sc.w;
                }
            }
            if (pass == 0) continue;
            if ((pass == 1 || !once) && n_tiles > 0) {
                nsplit = p.partial ? 1 : tile_num_splits(pos0, p.splits);
                part = 0;
                if (p.balanced) {
                    const int most = nsplit, share = is_short ? len_short : len;
                    // A sliver that costs more to start than it holds is left out, or rather given to its neighbour (and one under an
                    // eighth of a short share).  Left out below an eighth of any share, parts of 53 tiles grew to 58: 2048 tokens of
                    // eight heads at 14321 keys 142.8 -> 140.1 us.
                    const int least = min(max(share / 8, 1), (is_short ? p.short_lead : p.lead) + 1);
                    first = share - before % share;
                    if (first < least) first += share;
                    const int last = min(n_tiles - least, pos0 / kTileN);   // (a part starts at or before the first row)
                    nsplit = last >= first ? (last - first) / share + 2 : 1;
                    if (nsplit > 1) part = share;
                    if (nsplit > most) {
                        nsplit = most;
                        part = 0;
                    }
                }
            }
            int* const my_bins = bins + (is_short ? nthr : 0);
            auto bin = [&](int n) {
                const int b = nthr - 1 - static_cast<int>(static_cast<float>(n) * bin_scale);
                return my_bins + (b < 0 ? 0 : b);
            };
            const int ends = part > 0 ? 2 : 0;     // parts that are not of the common length
            // Uniform splits take their places in rounds, one split of every unit after the other: CTAs that run at the same time
            // then stream the same key range, where a unit's splits side by side kept several ranges going at once (16384
            // tokens at 344064 keys, four splits: 187 ms, so 164).
            const int rounds = pass == 2 && !p.balanced ? p.splits : 1;
#pragma unroll 1
            for (int round = 0; round < rounds; ++round) {
                int s0 = 0, s1 = nsplit;
                if (rounds > 1) {
                    __syncthreads();
                    s0 = min(round, nsplit);
                    s1 = min(round + 1, nsplit);
                }
                int slot = 0, slot_first = 0, slot_last = 0;
                if (s1 - s0 > ends) slot = atomicAdd(bin(part > 0 ? part : (n_tiles + nsplit - 1) / nsplit), s1 - s0 - ends) - s0;
                if (ends > 0) {
                    slot_first = atomicAdd(bin(first), 1);
                    slot_last = atomicAdd(bin(n_tiles - first - (nsplit - 2) * part), 1);
                }
                if (pass == 1) break;
#pragma unroll 1
                for (int s = s0; s < s1; ++s) {
                    int kb, ke, at = slot + s;
                    if (part > 0) {
                        kb = s == 0 ? 0 : first + (s - 1) * part;
                        ke = s + 1 == nsplit ? n_tiles : first + s * part;
                        at = s == 0 ? slot_first : s + 1 == nsplit ? slot_last : at - 1;
                    } else if (p.partial) {
                        kb = p.range_begin;
                        ke = n_tiles < p.range_end ? n_tiles : p.range_end;
                    } else {
                        split_range(pos0, n_tiles, nsplit, s, kb, ke);
                    }
                    if (at < p.max_units) {
                        WorkUnit u;
                        u.req = r;
                        u.q_row0 = qs[r] + row_off;
                        u.rows = rows | nsplit << 16;
                        u.pos0 = pos0;
                        u.kv_begin = kb;
                        u.kv_end = ke;
                        u.split = (nsplit > 1 || p.partial) ? s : -1;
                        u.kv_len = Ps[r] + Cs[r];
                        p.units[at] = u;
                    }
                }
            }
        }
        __syncthreads();
        if (pass == 0) {
            int ranges = p.ranges, ranges_short = p.short_ranges;
            if (sum > 0 && sum_short > 0) {     // both kinds share the slots by the work they have
                const float work = sum * p.unit_items * p.unit_us, work_short = sum_short * p.short_items * p.short_us;
                ranges = max(1, static_cast<int>(p.slots * (work / (work + work_short))) / p.unit_items);
                ranges_short = max(1, (p.slots - ranges * p.unit_items) / p.short_items);
            }
            len = max((sum + ranges - 1) / ranges, p.min_len);
            len_short = max((sum_short + ranges_short - 1) / ranges_short, p.min_short_len);
            const int longest = max(len, len_short);
            bin_scale = static_cast<float>(nthr - 1) / static_cast<float>(min(s_max, longest + longest / 8));
        }
        if (pass == 1) {
            // exclusive scan of the bins, two per thread (bin 0 = most expensive first, the short units' bins last)
            const int b0 = bins[2 * tid], b1 = bins[2 * tid + 1];
            const int4 sc = block_scan2(b0 + b1, 0, warp_sums);
            bins[2 * tid] = sc.x;
            bins[2 * tid + 1] = sc.x + b0;
            if (p.lead_items > 0 && 2 * tid >= nthr && b0 + b1 > 0) atomicMin(&s_short_bin, b0 > 0 ? 2 * tid : 2 * tid + 1);   // the longest short unit's
            if (2 * tid == nthr) {   // the first of the short units' bins
                const int n = sc.z < p.max_units ? sc.z : p.max_units;
                p.header->num_units = n;
                p.header->num_short = n - (sc.x < n ? sc.x : n);
                // Parts of a balanced cut are of very different lengths even where the units are not, so they go longest first over all
                // heads: 256 tokens of 64/8 heads at 32768 keys 329 us with the whole launch in one block (the last heads' long parts
                // started when the others were done), 300 with blocks of 256 rows, 253 so.
                p.header->unit_block = p.balanced ? 1 : 4 * s_min >= 3 * s_max ? p.unit_block : p.ragged_unit_block;
                p.header->counter = 0;
                p.header->error = 0;
                p.header->num_lead = 0;
                s_normal = sc.x;
                s_items = sc.x * p.unit_items + (sc.z - sc.x) * p.short_items;
            }
            __syncthreads();
            if (p.lead_items > 0 && s_normal > 0 && s_short_bin < 2 * nthr && s_items < p.lead_items)
                put_long_units_first(p.header, bins, s_short_bin, bin_scale, p.short_per_unit, p.lead, p.short_lead);
        }
    }
}

}  // namespace vpp
