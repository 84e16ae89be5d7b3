// Warp-specialised persistent chunked-prefill attention kernel for head_dim 128 (MHA / GQA / MQA).
//
// One CTA per SM, 12 warps:
//   warp 0      scheduler + TMA producer: takes work item blockIdx.x, then pops from the global counter, publishes them in a
//               2-deep shared ring, loads the two Q tiles of the item and streams K/V pages through a
//               ring of 128B-swizzled 32 KB stages (K0 V0 K1 V1 ...), gathered through the block table.
//   warp 1      MMA issuer: tcgen05.mma  S_t = Q_t K^T  and  O_t += P_t V  for the two query tiles
//               t = 0, 1 of the item, which use the same K/V stages.
//   warp 2      tensor-memory allocation.
//   warps 4-7   softmax group for tile 0: one query row per thread, fp32 online softmax on S_0 read
//               from tensor memory, P_0 written back to tensor memory as bf16 over S_0.
//   warps 8-11  the same for tile 1.
// (Shared-out items, below, differ in that: there a row stands in a lane of each warp of a group.)
// While one group works on its S tile the tensor core runs the other tile's MMAs.
//
// The rows of a tile are (token, q-head) pairs: `group` q-heads of one kv-head over `tile_tokens` consecutive tokens,
// group * tile_tokens = 125 .. 128 (group = the whole group of a kv-head where that fills a tile; 1 for MHA, which gives
// tiles of 128 tokens of one head).  A tile of few tokens wastes little on a ragged chunk: a request of 200 tokens with
// groups of eight takes seven units of 32 tokens where tiles of 128 tokens of one head took 256 (32 ragged chunks of 8192
// tokens together with 16 decode rows: 4.11 -> 3.50 ms).
// A work unit whose (token, q-head) rows fill at most one tile -- a decode step, a few tokens, the tail of a chunk -- is
// run "packed": both tiles of its item use that one Q tile and split the KV tiles between
// them (even ones to tile 0, odd ones to tile 1) as two independent online softmaxes whose results softmax group 0
// merges at the end -- one softmax chain per KV tile would leave the memory system idle most of the time.
// In large batches of decode rows (kQuarters) a packed item of one token is "shared out" as well: each warp of a group has the item's rows
// in its lanes and takes 32 of a tile's 128 keys, and group 0 joins eight results instead of two (ws_run_quarters).
// Tensor memory: S_0 | S_1 | O_0 | O_1, 128 fp32 columns each (all 512 columns).
//
// The math per row is the paper's Eq. 1 with the causal rule, evaluated KV tile by KV tile with a
// running maximum; O is rescaled lazily (only when the maximum has grown by more than 2^8).
#pragma once
#include <type_traits>

#include "common.cuh"
#include "ptx.cuh"

namespace vpp {

constexpr int kWsThreads = 384;
// Register budget per thread after the roles split (setmaxnreg).  The launch gives every warp 168 registers (three warps
// per sub-partition); warps 0-3 (one per sub-partition: producer, MMA issuer, allocator, idle) hand back down to
// kWsRegsLow and each of the two softmax warps of a sub-partition takes kWsRegsHigh: 72 + 2 * 216 = 3 * 168.  With 216
// registers the softmax loop (128 scores of a row live at once) has no spills.
constexpr int kWsRegsLow = 72, kWsRegsHigh = 216;
static_assert(kWsRegsLow + 2 * kWsRegsHigh <= 3 * 168 && kWsRegsLow % 8 == 0 && kWsRegsHigh % 8 == 0, "register budget");
constexpr int kWsStages = 4;                  // 32 KB each
constexpr int kTileBytes = 2 * kSlabBytes;    // one 128 x 128 bf16 tile
// (the two alternating slots of the V-tail barrier cover a producer that runs at most two V tiles ahead of the MMA thread:
//  a ring of more than four stages would need more slots -- five stages failed parity on short items)
static_assert(kWsStages <= 4, "V-tail barrier slots");
constexpr int kWsStageBytes = 8 * 32 * 128;   // 4 KB per softmax warp for the epilogue's stores (the join of shared-out items: 8 KB per warp of group 0)
constexpr int kWsSmemBytes = 2 * kTileBytes + kWsStages * kTileBytes + 1024 /*align*/ + 2048 /*barriers, ring, merge exchange*/ + kWsStageBytes;
static_assert(kWsSmemBytes <= 232448, "shared memory of one CTA");
// (bytes from the first barrier)
constexpr int kWsBarS = 48, kWsBarP = 64, kWsBarO = 80, kWsBarJoin = 104, kWsBarX1 = 128 + 16 * kWsStages, kWsBarX0 = kWsBarX1 + 8, kWsBarPart = 208;
constexpr int kWsAbort = 512, kWsXm = 1024, kWsStage = 2048;
constexpr float kRescaleThreshold = 8.f;      // log2 units
// Early hand-overs of P: bit c set = the key columns up to 32 (c + 1) are handed to the MMA thread as soon as they are in
// tensor memory, so that O += P V starts on them while the rest of the exponentials are computed (0: P is handed over whole).
constexpr int kPartMask = 3;   // after 32 and after 64 columns (measured best: a hand-over after 96 columns costs more than it gains)
static_assert(kPartMask >= 0 && kPartMask < 8, "hand-overs after 32, 64 and 96 columns only");
constexpr int kPartWaitDefer = 8;             // pairs of columns of the next chunk computed before that hand-over's store is awaited (0: none)
static_assert(kPartWaitDefer >= 1 && kPartWaitDefer <= 16, "the wait sits inside the next chunk");

struct WsItem {
    WorkUnit u;
    int32_t h0;      // first q-head of the item's rows
    int32_t valid;   // 0: no more work
    int32_t packed;  // 1: the rows fill at most tile 0; both tiles use it and split the KV tiles
    int32_t pad;
};


// Merge of the two tiles' partial results of a packed item (rare path, kept out of line to spare the main loop's
// registers):  out = (a0 O_0 + a1 O_1) / (a0 l_0 + a1 l_1),  a_t = 2^(m_t - m).  O_1 sits 128 columns after O_0.
// (every argument by value: a reference to the kernel's parameter block or to the work unit would force them into
// local memory for the whole kernel)
__device__ __noinline__ void ws_packed_merge(void* out, float* lse_out, float* o_parts, float* lse_parts, bool final,
                                             long long out_row, bool second, const float* xm,
                                             uint32_t tO, int row, int tile_rows, float m_ref, float l_run) {
    const float m1 = xm[row], l1 = xm[128 + row];
    const float m = fmaxf(m_ref, m1);
    const float a0 = m_ref == -INFINITY ? 0.f : ex2(m_ref - m), a1 = m1 == -INFINITY ? 0.f : ex2(m1 - m);
    const float l_tot = a0 * l_run + a1 * l1;
    const float s0 = a0 / l_tot, s1 = a1 / l_tot;
    const bool live = row < tile_rows;
    uint32_t r[16], r1[16];
#pragma unroll 1
    for (int c = 0; c < 8; ++c) {     // 16 output columns at a time (registers)
        tmem_ld16(tO + c * 16, r);
        if (second) tmem_ld16(tO + 128 + c * 16, r1);
        tc_wait_ld();
        if (!live) continue;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            float v = __uint_as_float(r[i]) * s0;
            if (second) v = fmaf(__uint_as_float(r1[i]), s1, v);
            r[i] = __float_as_uint(v);
        }
        if (final) {
            uint4* dst = reinterpret_cast<uint4*>(static_cast<uint8_t*>(out) + (out_row * 128 + c * 16) * 2);
#pragma unroll
            for (int q4 = 0; q4 < 2; ++q4) {
                uint32_t w[4];
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    w[e] = pack_bf16x2(__uint_as_float(r[q4 * 8 + 2 * e]), __uint_as_float(r[q4 * 8 + 2 * e + 1]));
                dst[q4] = make_uint4(w[0], w[1], w[2], w[3]);
            }
        } else {
            float4* dst = reinterpret_cast<float4*>(o_parts + out_row * 128 + c * 16);
#pragma unroll
            for (int q4 = 0; q4 < 4; ++q4)
                dst[q4] = make_float4(__uint_as_float(r[q4 * 4]), __uint_as_float(r[q4 * 4 + 1]),
                                      __uint_as_float(r[q4 * 4 + 2]), __uint_as_float(r[q4 * 4 + 3]));
        }
    }
    if (live) {
        const float lse = (m + log2f(l_tot)) * 0.6931471805599453f;
        if (final) {
            if (lse_out) lse_out[out_row] = lse;
        } else {
            lse_parts[out_row] = lse;
        }
    }
}

// Whole items of one token and up to kQuarterHeads q-heads (decode rows that are not cut): the item's rows stand in Q four times, once in the 32 lanes of
// each softmax warp, and the warps share out the 128 keys of a tile -- 32 each, an online softmax of its own -- where one warp would take
// them all and the others idle.  The MMAs of a warp's keys write that warp's lanes of O only (zero weights for the others' would do as well
// but for infinite values, 0 * inf).  Tile t's O is then the sum of four over the lanes, and an item's
// result the sum of eight, joined by group 0: every warp weighs its two and leaves them in the stage, all sum.
// A warp has 32 exponentials a tile instead of 128, so that what ends an item hides behind the copies of the next: 256 decode rows of 64/8
// heads, contexts to 8192 tokens, 802 us packed and 771 so (6.3 TB/s); all of 8192 tokens 1361 and 1322 us, which is 6.5 TB/s, the copy rate.  Where
// contexts differ, the rest is the start of the launch and the SMs' unequal ends; what share each has is not measured.
// (Against 64 bits, 40 to 200 rows: results 2.16 - 2.21e-3 off before, 2.06 - 2.13e-3 now, log-sum-exps 3.5e-7 and 3.6e-7.)
constexpr int kQuarterHeads = 16;             // rows of 512 bytes in a warp's 8 KB of the stage
static_assert(4 * kQuarterHeads * 512 <= kWsStageBytes, "the stage of both groups");
// dst: row of the item's first head; lse: its log-sum-exp, or null; area: the CTA's barriers, xm and stage
__device__ __forceinline__ bool ws_quarter_join(uint8_t* dst, float* lse, bool second, uint8_t* area, uint32_t bar, uint32_t tO,
                                                int heads, float m_ref, float l_run) {
    volatile int* const s_abort = reinterpret_cast<volatile int*>(area + kWsAbort);
    float* const xm = reinterpret_cast<float*>(area + kWsXm);
    uint8_t* const stage = area + kWsStage;
    const int row = threadIdx.x & 127, w = row >> 5, lane = row & 31;
    const float m1 = xm[row], l1 = xm[128 + row];
    const float m = fmaxf(m_ref, m1);
    const float a0 = m_ref == -INFINITY ? 0.f : ex2(m_ref - m), a1 = m1 == -INFINITY ? 0.f : ex2(m1 - m);
    xm[row] = m;              // (read by this thread alone so far)
    xm[128 + row] = a0 * l_run + a1 * l1;
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
    if (!mbar_wait(bar, 0, s_abort, 406)) return false;      // (two phases an item: the same parities every time)
    float M = -INFINITY, L = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) M = fmaxf(M, xm[k * 32 + lane]);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float mk = xm[k * 32 + lane];     // (-inf: no key of its own, or scores of NaN, whose sum is NaN and must stay so)
        L = fmaf(mk == -INFINITY ? 0.f : ex2(mk - M), xm[128 + k * 32 + lane], L);
    }
    const float f = (m == -INFINITY ? 0.f : ex2(m - M)) / L;     // (all scores -inf: 0 / 0, as the definition has it)
    const float s0 = a0 * f, s1 = a1 * f;
    uint8_t* const mine = stage + w * (kQuarterHeads * 512) + lane * 512;
#pragma unroll 1
    for (int c = 0; c < 8; ++c) {     // 16 output columns at a time (registers)
        uint32_t r[16], r1[16];
        tmem_ld16(tO + c * 16, r);
        if (second) tmem_ld16(tO + 128 + c * 16, r1);
        tc_wait_ld();
        if (lane < heads) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                float v = __uint_as_float(r[i]) * s0;
                if (second) v = fmaf(__uint_as_float(r1[i]), s1, v);
                r[i] = __float_as_uint(v);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
                *reinterpret_cast<uint4*>(mine + (((c * 4 + q) ^ (lane & 7)) << 4)) = make_uint4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
        }
    }
    if (lane < heads && w == 0 && lse) lse[lane] = (M + log2f(L)) * 0.6931471805599453f;
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
    if (!mbar_wait(bar, 1, s_abort, 407)) return false;
    for (int i = row; i < heads * 16; i += 128) {     // eight columns of a row
        const int h = i >> 4, c8 = i & 15;
        float acc[8] = {};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint8_t* const from = stage + k * (kQuarterHeads * 512) + h * 512;
            const float4 x = *reinterpret_cast<const float4*>(from + (((2 * c8) ^ (h & 7)) << 4));
            const float4 y = *reinterpret_cast<const float4*>(from + (((2 * c8 + 1) ^ (h & 7)) << 4));
            acc[0] += x.x; acc[1] += x.y; acc[2] += x.z; acc[3] += x.w;
            acc[4] += y.x; acc[5] += y.y; acc[6] += y.z; acc[7] += y.w;
        }
        *reinterpret_cast<uint4*>(dst + (h * 128 + c8 * 8) * 2) =
            make_uint4(pack_bf16x2(acc[0], acc[1]), pack_bf16x2(acc[2], acc[3]), pack_bf16x2(acc[4], acc[5]), pack_bf16x2(acc[6], acc[7]));
    }
    return true;
}

// Softmax of one item of quarters, by a warp of group t: 32 of the keys of every second tile, then the join.
// (in line: out of line, the twelve arguments and what lives across the call cost a stack frame and 52 bytes of spills; the other
// instantiations of the kernel do not have it)
__device__ __forceinline__ bool ws_run_quarters(uint8_t* dst, float* lse, int kv_end, int pos, int heads, float sc, uint32_t sBar,
                                                uint8_t* area, uint32_t tmem_base, uint32_t s_it, uint32_t o_it, uint32_t x_it) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t = (warp - 4) >> 2, wq = warp & 3, row = threadIdx.x & 127;
    const uint32_t lane_off = static_cast<uint32_t>(wq * 32) << 16, tS = tmem_base + t * 128 + lane_off, tO = tmem_base + 256 + t * 128 + lane_off;
    volatile int* const s_abort = reinterpret_cast<volatile int*>(area + kWsAbort);
    float* const xm = reinterpret_cast<float*>(area + kWsXm);
    float m_ref = -INFINITY, l_run = 0.f;
    const int first = t;                      // (a whole row begins at its first tile)
#pragma unroll 1
    for (int j = first; j < kv_end; j += 2) {
        if (!mbar_wait(sBar + kWsBarS + 8 * t, s_it & 1, s_abort, 402)) return false;
        ++s_it;
        tc_fence_after();
        uint32_t s[32];
        tmem_ld32(tS + 32 * wq, s);
        tc_wait_ld();
        const int lim = pos - j * kTileN - 32 * wq;      // columns <= lim are visible
        if (lim < 31) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
                if (i > lim) s[i] = 0xff800000u;  // -inf
        }
        float mx[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) mx[k] = fmaxf(__uint_as_float(s[k]), __uint_as_float(s[4 + k]));
#pragma unroll
        for (int i = 8; i < 32; i += 8)
#pragma unroll
            for (int k = 0; k < 4; ++k) mx[k] = fmax3(mx[k], __uint_as_float(s[i + k]), __uint_as_float(s[i + 4 + k]));
        const float m_new = fmaxf(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * sc, m_ref);
        // (lanes beyond the heads hold leftovers: they never ask for a rescale)
        const bool grow = lane < heads && ((m_new - m_ref > kRescaleThreshold) || (m_ref == -INFINITY && m_new != -INFINITY));
        if (__any_sync(0xffffffffu, grow)) {
            const float alpha = grow ? ex2(m_ref - m_new) : 1.f;  // m_ref = -inf gives 0
            if (grow) m_ref = m_new;
            l_run *= alpha;
            if (j > first) {   // O of this tile already holds something
                uint32_t o[16];
#pragma unroll 1
                for (int c = 0; c < 8; ++c) {
                    tmem_ld16(tO + c * 16, o);
                    tc_wait_ld();
#pragma unroll
                    for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                    tmem_st16(tO + c * 16, o);
                }
            }
        }
        const float m_use = (m_ref == -INFINITY) ? 0.f : m_ref;
        float sum0 = 0.f, sum1 = 0.f;
        uint32_t pk[16];     // (the columns of the other warps' keys stay as they are: the MMAs of those keys leave these lanes of O alone)
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
            const float p0 = ex2(fmaf(__uint_as_float(s[i]), sc, -m_use)), p1 = ex2(fmaf(__uint_as_float(s[i + 1]), sc, -m_use));
            sum0 += p0;
            sum1 += p1;
            pk[i >> 1] = pack_bf16x2(p0, p1);
        }
        tmem_st16(tS + wq * 16, pk);
        l_run += sum0 + sum1;
        tc_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
#pragma unroll
            for (int c = 0; c < 3; ++c)
                if ((kPartMask >> c) & 1) mbar_arrive(sBar + kWsBarPart + 16 * c + 8 * t);
            mbar_arrive(sBar + kWsBarP + 8 * t);
        }
    }
    if (first < kv_end && !mbar_wait(sBar + kWsBarO + 8 * t, o_it & 1, s_abort, 403)) return false;   // (tile 1 of a one-tile item has none)
    tc_fence_after();
    if (t == 1) {
        xm[row] = m_ref;
        xm[128 + row] = l_run;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(sBar + kWsBarX1);
        return mbar_wait(sBar + kWsBarX0, x_it & 1, s_abort, 404);
    }
    if (!mbar_wait(sBar + kWsBarX1, x_it & 1, s_abort, 405)) return false;
    tc_fence_after();
    if (!ws_quarter_join(dst, lse, 1 < kv_end, area, sBar + kWsBarJoin, tO, heads, m_ref, l_run)) return false;
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(sBar + kWsBarX0);
    return true;
}

// K / V tile in shared memory: 8-key groups of 2 KB, features 0-63 then 64-127 of the eight keys, 128-byte swizzle.  Keys of a
// page are consecutive in it, so a page of any size is ONE copy (issuing a copy costs a producer lane over 100 clk; with the
// two 64-feature slabs 16 KB apart a page under 128 tokens took two).  256 decode rows over pages of 16
// tokens: 576 -> 543 us; 2048-token chunks over pages of 16 .. 64: 1020 -> 989 us, as over pages of 128.
constexpr int kGroupBytes = 2048, kHalfBytes = 1024;
constexpr int kExactRows = 8;                 // keys per copy of the exact map

// kQuarters: for launches that are not cut, of up to kQuarterHeads q-heads a kv-head (an instantiation of its own: cut launches of decode rows
// lose 1 % to the registers and the size of the code)
template <bool kVWarp, bool kQuarters>
__global__ void __launch_bounds__(kWsThreads, 1)
attn128_ws_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_qs, const __grid_constant__ CUtensorMap tm_q1,
                  const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                  const __grid_constant__ CUtensorMap tm_kx, const __grid_constant__ CUtensorMap tm_vx, const AttnParams p,
                  const int kv_box_rows) {
    // tm_q:  q with a box of (64 features, group heads, tile_tokens tokens): one 64-column slab of a tile
    // tm_qs / tm_q1: the same with (64, short_group, short_tokens) and (64, short_group, 1), for packed items of several tokens and of one
    // tm_k / tm_v: (64 features, 8 keys, 2 halves, 8-key groups, (block, kv-head)), box (64, 8, 2, kv_box_rows / 8, 1): the keys of
    //        a page, or of a whole tile where pages are that large
    // tm_kx / tm_vx: (64 features, keys, 2 halves, kv-head, block), box (64, 8, 2, 1, 1): eight keys, the extent of the keys exact --
    //        for the last tile of a contiguous cache whose length is no multiple of 8, and strides the other maps cannot express
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* gen_base = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t sQ = smem_base;                       // 2 tiles
    const uint32_t sKV = sQ + 2 * kTileBytes;            // kWsStages tiles
    const uint32_t sBar = sKV + kWsStages * kTileBytes;  // barriers
    // barrier map (8 bytes each)
    const uint32_t bar_item_full = sBar + 0;     // [2]
    const uint32_t bar_item_empty = sBar + 16;   // [2]
    const uint32_t bar_q_full = sBar + 32;
    const uint32_t bar_q_empty = sBar + 40;
    const uint32_t bar_s_full = sBar + kWsBarS;       // [2]
    const uint32_t bar_p_full = sBar + kWsBarP;       // [2]
    const uint32_t bar_o_full = sBar + kWsBarO;       // [2]
    // Two slots used alternately: the producer can fix up the V tile of the next short item before the MMA thread has
    // looked at the barrier for this one (slot k & 1 for the k-th such tile, 24 bytes apart).
    const uint32_t bar_vfix = sBar + 96;         // (and + 120; kWsBarJoin is between)
    // [3][2] early hand-overs of P: part c (the key columns up to 32 (c + 1)) of tile t is in place.  One barrier per part:
    // the MMA thread may look at part 0 only after part 1 has arrived too, which a shared barrier could not tell apart.
    const uint32_t bar_p_part = sBar + kWsBarPart;
    const uint32_t bar_kv_full = sBar + 128;     // [kWsStages]
    const uint32_t bar_kv_empty = sBar + 128 + 8 * kWsStages;
    const uint32_t bar_x1 = sBar + kWsBarX1;       // packed item: group 1 has published its (m, l) per row (shared out: per lane)
    const uint32_t bar_x0 = sBar + kWsBarX0;       // packed item: group 0 has merged, tile 1, xm and group 1's stage may be reused
    // (kWsBarJoin, shared-out items: the warps of group 0 have published their own (m, l), then their weighed results: two phases an item)
    uint8_t* gen_bar = gen_base + (2 + kWsStages) * kTileBytes;
    volatile int* s_abort = reinterpret_cast<volatile int*>(gen_bar + kWsAbort);
    volatile uint32_t* s_tmem = reinterpret_cast<volatile uint32_t*>(gen_bar + 516);
    WsItem* ring = reinterpret_cast<WsItem*>(gen_bar + 576);  // 2 x 48 bytes
    // [2][128]: running maximum and row sum of tile 1 (packed items); shared out, of each lane of tile 1, then of both tiles together
    float* xm = reinterpret_cast<float*>(gen_bar + kWsXm);

    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar_item_full + 8 * i, 1);
            mbar_init(bar_item_empty + 8 * i, kVWarp ? 10 : 9);   // 8 softmax warps, the MMA thread, (the second producer)
            mbar_init(bar_s_full + 8 * i, 1);
            mbar_init(bar_p_full + 8 * i, 4);   // one arrival per softmax warp
            for (int c = 0; c < 3; ++c) mbar_init(bar_p_part + 16 * c + 8 * i, 4);
            mbar_init(bar_o_full + 8 * i, 1);
        }
        mbar_init(bar_q_full, 1);
        mbar_init(bar_q_empty, 1);
        mbar_init(bar_vfix, 1);
        mbar_init(bar_vfix + 24, 1);
        mbar_init(bar_x1, 4);
        mbar_init(sBar + kWsBarJoin, 4);
        mbar_init(bar_x0, 4);
        for (int i = 0; i < kWsStages; ++i) {
            mbar_init(bar_kv_full + 8 * i, 1);
            mbar_init(bar_kv_empty + 8 * i, 1);
        }
        fence_mbar_init();
        *s_abort = 0;
        prefetch_tmap(&tm_q);
        prefetch_tmap(&tm_k);
        prefetch_tmap(&tm_v);
        prefetch_tmap(&tm_qs);
        prefetch_tmap(&tm_q1);
    }
    __syncthreads();
    if (warp == 2) {
        tmem_alloc(smem_u32(const_cast<uint32_t*>(s_tmem)), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *s_tmem;

    pdl_wait();                  // the work list comes from the work-decomposition kernel launched just before
    pdl_launch_dependents();     // (the merge kernel, if any, waits for this grid to finish in the same way)
    const WorkList list = read_header(p.header_ro);
    if (blockIdx.x == 0 && tid == 0 && p.status) *p.status = list.error;
    const int G = p.num_q_heads / p.num_kv_heads;
    // Items: the short units' (unit, group of q-heads), which run packed (their groups are larger where a kv-head's group
    // does not fill a tile well), and those of the units of two tiles.  Whatever is long comes early, since such an item started
    // last would run alone: the short ones, which sit at the end of long contexts, in a batch of few items behind the units that take longer than any of
    // them (prep.cuh), then the rest.
    const int num_packed = list.num_short;
    const int num_normal = list.num_units - num_packed;
    const int normal_slots = p.num_q_heads / p.group, packed_slots = p.num_q_heads / p.short_group;
    const int packed_items = num_packed * packed_slots, unit_block = list.unit_block, lead_items = list.num_lead * normal_slots;
    const int total_items = packed_items + num_normal * normal_slots;

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kWsRegsLow));
        // One K (which = 0) or V (which = 1) tile of the item into the next ring stage, by the calling warp.
        auto load_kv_tile = [&](const WorkUnit& u, int g, int tile0, int which, uint32_t kv_it, uint32_t& vfix_cnt) -> bool {
            bool ok = true;
                const uint32_t st = kv_it % kWsStages;
                const uint32_t ph = (kv_it / kWsStages) & 1;
                const uint32_t dst = sKV + st * kTileBytes;
                const uint32_t full = bar_kv_full + 8 * st;
                // a lane per page (or per eight keys); its page is looked up before the wait for the stage
                const bool exact = tile0 + kTileN > p.exact_from;
                const int rows = exact ? kExactRows : kv_box_rows, off = lane * rows, pos = tile0 + off;
                int blk = p.num_blocks, slot_in = 0;     // (past the end: reads as zero)
                if (off < kTileN) {
                    if (p.block_table == nullptr) {
                        blk = u.req;
                        slot_in = pos;
                    } else if (pos < u.kv_len) {
                        blk = __ldg(p.block_table + static_cast<long long>(u.req) * p.max_blocks_per_req + (pos >> p.block_shift));
                        slot_in = pos & ((1 << p.block_shift) - 1);
                    }
                }
                if (lane == 0) {
                    ok = mbar_wait(bar_kv_empty + 8 * st, ph ^ 1, s_abort, 203);
                    if (ok) mbar_arrive_expect_tx(full, kTileBytes);
                }
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) return false;
                if (off < kTileN) {
                    const uint32_t d = dst + static_cast<uint32_t>(off) * (kGroupBytes / 8);
                    if (exact) {
                        tma_load_5d(d, which == 0 ? &tm_kx : &tm_vx, full, 0, slot_in, 0, g, blk);
                    } else {
                        const int at = blk == p.num_blocks ? (which == 0 ? p.k_end : p.v_end)
                                       : which == 0 ? blk * p.k_block_units + g * p.k_head_units : blk * p.v_block_units + g * p.v_head_units;
                        tma_load_5d(d, which == 0 ? &tm_k : &tm_v, full, 0, 0, 0, slot_in >> 3, at);
                    }
                }
                __syncwarp();
                if (which == 1 && tile0 + kTileN > u.kv_len) {
                    // Keys at or beyond kv_len do not exist; zero their V rows so that 0 * garbage
                    // cannot poison O.  The MMA warp waits for bar_vfix on such a tile.
                    if (lane == 0) ok = mbar_wait(full, ph, s_abort, 204);
                    ok = __shfl_sync(0xffffffffu, ok, 0);
                    if (!ok) return false;
                    uint8_t* vb = gen_base + 2 * kTileBytes + st * kTileBytes;
                    const int first = u.kv_len > tile0 ? u.kv_len - tile0 : 0;
                    const uint4 z = make_uint4(0, 0, 0, 0);
                    for (int r = first + lane; r < kTileN; r += 32) {
                        uint4* a = reinterpret_cast<uint4*>(vb + (r >> 3) * kGroupBytes + (r & 7) * 128);
                        uint4* b = a + kHalfBytes / 16;
#pragma unroll
                        for (int c = 0; c < 8; ++c) {
                            a[c] = z;
                            b[c] = z;
                        }
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_vfix + 24 * (vfix_cnt & 1));
                    ++vfix_cnt;
                }
            return true;
        };
        // kVWarp: a second producer warp (warp 2) loads the V tiles, warp 0 the K tiles.  The host chooses it for the launches
        // that are bound by how fast K/V arrives: batches of decode rows, which stream K/V at memory speed (+10 to 18 % with K
        // and V requested by two warps).  Prefill keeps the single producer (a second one costs it 1 to 2 %).
        constexpr bool split_v = kVWarp;
        if (warp == 0) {
            // ============================ scheduler + TMA producer ============================
            uint32_t item_it = 0, q_it = 0, kv_it = 0, vfix_cnt = 0;
            while (true) {
                int item = blockIdx.x;     // (the first without a round trip to the counter)
                if (item_it > 0) {
                    if (lane == 0) item = gridDim.x + atomicAdd(&p.header->counter, 1);
                    item = __shfl_sync(0xffffffffu, item, 0);
                }
                const bool have = item < total_items;
                WorkUnit u{};
                int h0 = 0;
                bool packed = false;
                packed = have && static_cast<uint32_t>(item - lead_items) < static_cast<uint32_t>(packed_items);
                if (packed) {
                    const int k = item - lead_items;
                    u = p.units[num_normal + k / packed_slots];
                    h0 = (k % packed_slots) * p.short_group;
                } else if (have) {
                    int ui, hs;
                    decode_item(item < lead_items ? item : item - packed_items, num_normal, unit_block, normal_slots, G / p.group, ui, hs);
                    u = p.units[ui];
                    h0 = hs * p.group;
                }
                const uint32_t slot = item_it & 1;
                bool ok = true;
                if (lane == 0) ok = mbar_wait(bar_item_empty + 8 * slot, ((item_it >> 1) & 1) ^ 1, s_abort, 201);
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) break;
                if (lane == 0) {
                    ring[slot].u = u;     // (its split count with it)
                    ring[slot].h0 = h0;
                    ring[slot].valid = have ? 1 : 0;
                    ring[slot].packed = packed ? 1 : 0;
                    mbar_arrive(bar_item_full + 8 * slot);
                }
                ++item_it;
                if (!have) break;
                const int g = h0 / G;

                if (lane == 0) {
                    ok = mbar_wait(bar_q_empty, (q_it & 1) ^ 1, s_abort, 202);
                    // (tokens past the end of q read as zero; rows of a following request are never stored; tile rows the
                    // boxes do not cover keep whatever they held)
                    if (ok && packed) {
                        const bool one = (u.rows & 0xffff) == 1;
                        const CUtensorMap* tm = one ? &tm_q1 : &tm_qs;
                        const int copies = kQuarters && one ? 4 : 1;     // (one for the lanes of each softmax warp)
                        mbar_arrive_expect_tx(bar_q_full, copies * 2 * p.short_group * (one ? 1 : p.short_tokens) * 128);
#pragma unroll 1
                        for (int i = 0; i < copies; ++i) {
                            tma_load_3d(sQ + i * 4096, tm, bar_q_full, 0, h0, u.q_row0);
                            tma_load_3d(sQ + i * 4096 + kSlabBytes, tm, bar_q_full, 64, h0, u.q_row0);
                        }
                    } else if (ok) {
                        mbar_arrive_expect_tx(bar_q_full, 4 * p.group * p.tile_tokens * 128);
#pragma unroll
                        for (int t = 0; t < 2; ++t) {
                            tma_load_3d(sQ + t * kTileBytes, &tm_q, bar_q_full, 0, h0, u.q_row0 + t * p.tile_tokens);
                            tma_load_3d(sQ + t * kTileBytes + kSlabBytes, &tm_q, bar_q_full, 64, h0, u.q_row0 + t * p.tile_tokens);
                        }
                    }
                }
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) break;
                ++q_it;

                for (int j = u.kv_begin; j < u.kv_end && ok; ++j) {
#pragma unroll
                    for (int which = 0; which < 2; ++which) {  // 0: K, 1: V
                        if (!(split_v && which == 1)) ok = load_kv_tile(u, g, j * kTileN, which, kv_it, vfix_cnt);
                        if (!ok) break;
                        ++kv_it;
                    }
                }
                if (!ok) break;
            }
        } else if (warp == 2 && split_v) {
            // ============================ second producer: the V tiles ============================
            // (follows the item ring like every other role)
            uint32_t item_it = 0, kv_it = 0, vfix_cnt = 0;
            while (true) {
                const uint32_t slot = item_it & 1;
                bool ok = true;
                if (lane == 0) ok = mbar_wait(bar_item_full + 8 * slot, (item_it >> 1) & 1, s_abort, 211);
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) break;
                WorkUnit u = ring[slot].u;
                take_splits(u);
                const int g = ring[slot].h0 / G;
                const int valid = ring[slot].valid;
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_item_empty + 8 * slot);
                ++item_it;
                if (!valid) break;
                for (int j = u.kv_begin; j < u.kv_end && ok; ++j) {
                    ++kv_it;                                             // (the K tile: warp 0's)
                    ok = load_kv_tile(u, g, j * kTileN, 1, kv_it, vfix_cnt);
                    ++kv_it;
                }
                if (!ok) break;
            }
        } else if (warp == 1 && lane == 0) {
            // ============================ MMA issuer (a single thread) ============================
            constexpr uint32_t kIdescQK = idesc_bf16(128, 128, false, false);
            constexpr uint32_t kIdescPV = idesc_bf16(128, 128, false, true);
            const uint32_t tS0 = tmem_base, tS1 = tmem_base + 128, tO0 = tmem_base + 256, tO1 = tmem_base + 384;
            uint32_t item_it = 0, q_it = 0, kv_it = 0, vfix_it = 0, p_it = 0, p_it1 = 0;   // P hand-offs seen per tile
            auto wait1 = [&](uint32_t bar, uint32_t parity, int where) -> bool {
                return mbar_wait(bar, parity, s_abort, where);
            };
            // Descriptors are advanced by adding constants to their low word: the single issuing thread
            // must not spend longer building operands than the tensor core spends on the MMA.
            constexpr uint32_t kHiQ = desc_hi_sw128(1024), kHiKV = desc_hi_sw128(kGroupBytes);
            const uint32_t q_lo0 = desc_lo_sw128(sQ, 16), q_lo1 = desc_lo_sw128(sQ + kTileBytes, 16);
            auto issue_qk = [&](uint32_t tS, uint32_t q_lo, uint32_t k_stage) {
                const uint32_t k_lo = desc_lo_sw128(k_stage, 16);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const uint32_t qoff = ((k >> 2) * kSlabBytes + (k & 3) * 32) >> 4, koff = ((k >> 2) * kHalfBytes + (k & 3) * 32) >> 4;
                    mma_ss_lhh(tS, q_lo + qoff, kHiQ, k_lo + koff, kHiKV, kIdescQK, k > 0);
                }
            };
            // (quarter: the 16 keys of a step go to the lanes of the warp whose keys they are, and to no others)
            auto issue_pv = [&](uint32_t tO, uint32_t tP, uint32_t v_stage, bool first, int k0, int k1, bool quarter) {
                const uint32_t v_lo = desc_lo_sw128(v_stage, kHalfBytes);
#pragma unroll
                for (int k = k0; k < k1; ++k) {
                    const uint32_t a = tP + k * 8, b_lo = v_lo + k * (2 * kGroupBytes >> 4);
                    if constexpr (kQuarters) {
                        const uint32_t off = quarter ? 0xffffffffu : 0u;
                        const int w = k >> 1;
                        mma_ts_lh_lanes(tO, a, b_lo, kHiKV, kIdescPV, (!first || (quarter ? (k & 1) : k) > 0) ? 1u : 0u,
                                        w == 0 ? 0u : off, w == 1 ? 0u : off, w == 2 ? 0u : off, w == 3 ? 0u : off);
                    } else {
                        mma_ts_lh(tO, a, b_lo, kHiKV, kIdescPV, (!first || k > 0) ? 1u : 0u);
                    }
                }
            };
            // O_t += P_t V for one KV tile, following the hand-overs: every early part as soon as it is there, the rest after
            // the whole of P.  pit = hand-overs of P_t seen so far (tile visits).
            auto pv_tile = [&](int t, uint32_t tO, uint32_t tS, uint32_t v_stage, bool first, uint32_t pit, int where, bool quarter) -> bool {
                int k0 = 0;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    if ((kPartMask >> c) & 1) {
                        if (!wait1(bar_p_part + 16 * c + 8 * t, pit & 1, where)) return false;
                        tc_fence_after();
                        issue_pv(tO, tS, v_stage, first, k0, 2 * (c + 1), quarter);
                        k0 = 2 * (c + 1);
                    }
                }
                if (!wait1(bar_p_full + 8 * t, pit & 1, where + 1)) return false;
                tc_fence_after();
                issue_pv(tO, tS, v_stage, first, k0, 8, quarter);
                return true;
            };
            while (true) {
                const uint32_t slot = item_it & 1;
                if (!wait1(bar_item_full + 8 * slot, (item_it >> 1) & 1, 301)) break;
                WorkUnit u = ring[slot].u;
                take_splits(u);
                const int valid = ring[slot].valid;
                const bool packed = ring[slot].packed != 0;
                mbar_arrive(bar_item_empty + 8 * slot);
                ++item_it;
                if (!valid) break;
                const int n = u.kv_end - u.kv_begin;
                if (!wait1(bar_q_full, q_it & 1, 302)) break;
                ++q_it;
                if (packed) {
                    // Packed item (a short unit): both tiles use the same Q (the unit's tokens x the heads of one kv-head) and share the KV
                    // range -- tile t takes the KV tiles kv_begin + t, + t + 2, ... as an independent online softmax
                    // (its own S_t, O_t); the two partial results are merged by softmax group 0 at the end.
                    // Ring index of K(jj) is base + 2 jj, of V(jj) base + 2 jj + 1.
                    const uint32_t base = kv_it;
                    bool ok = true;
                    auto do_qk = [&](int jj) {
                        const uint32_t idx = base + 2 * jj, st = idx % kWsStages;
                        if (!wait1(bar_kv_full + 8 * st, (idx / kWsStages) & 1, 321)) return false;
                        tc_fence_after();
                        issue_qk((jj & 1) ? tS1 : tS0, q_lo0, sKV + st * kTileBytes);
                        tc_commit(bar_s_full + 8 * (jj & 1));
                        tc_commit(bar_kv_empty + 8 * st);
                        if (jj + 1 == n) tc_commit(bar_q_empty);
                        return true;
                    };
                    ok = do_qk(0);
                    if (ok && n > 1) ok = do_qk(1);
                    for (int jj = 0; jj < n && ok; ++jj) {
                        const int t = jj & 1;
                        const int tile0 = (u.kv_begin + jj) * kTileN;
                        const uint32_t idx = base + 2 * jj + 1, st = idx % kWsStages;
                        const uint32_t pit = t ? p_it1 : p_it;   // (no reference: the counters must stay in registers)
                        ok = wait1(bar_kv_full + 8 * st, (idx / kWsStages) & 1, 322);
                        if (!ok) break;
                        if (tile0 + kTileN > u.kv_len) {
                            ok = wait1(bar_vfix + 24 * (vfix_it & 1), (vfix_it >> 1) & 1, 323);
                            if (!ok) break;
                            ++vfix_it;
                        }
                        const uint32_t tO = t ? tO1 : tO0, tS = t ? tS1 : tS0;
                        ok = pv_tile(t, tO, tS, sKV + st * kTileBytes, jj < 2, pit, 324, kQuarters && u.rows == 1);
                        if (!ok) break;
                        tc_commit(bar_kv_empty + 8 * st);
                        if (t) ++p_it1; else ++p_it;
                        if (jj + 2 < n) ok = do_qk(jj + 2);
                        else tc_commit(bar_o_full + 8 * t);     // this tile's last KV tile
                    }
                    if (!ok) break;
                    kv_it = base + 2 * n;
                    continue;
                }
                // S_t(0) = Q_t K(0)^T
                uint32_t stK = kv_it % kWsStages;
                if (!wait1(bar_kv_full + 8 * stK, (kv_it / kWsStages) & 1, 303)) break;
                ++kv_it;
                tc_fence_after();
                if (lane == 0) {
                    issue_qk(tS0, q_lo0, sKV + stK * kTileBytes);
                    tc_commit(bar_s_full);
                    issue_qk(tS1, q_lo1, sKV + stK * kTileBytes);
                    tc_commit(bar_s_full + 8);
                    tc_commit(bar_kv_empty + 8 * stK);
                    if (n == 1) tc_commit(bar_q_empty);
                }
                bool ok = true;
                for (int jj = 0; jj < n && ok; ++jj) {
                    const int tile0 = (u.kv_begin + jj) * kTileN;
                    const uint32_t stV = kv_it % kWsStages;
                    ok = wait1(bar_kv_full + 8 * stV, (kv_it / kWsStages) & 1, 304);
                    if (!ok) break;
                    ++kv_it;
                    if (tile0 + kTileN > u.kv_len) {
                        ok = wait1(bar_vfix + 24 * (vfix_it & 1), (vfix_it >> 1) & 1, 305);
                        if (!ok) break;
                        ++vfix_it;
                    }
                    const bool has_next = jj + 1 < n;
                    stK = kv_it % kWsStages;
                    // ---- tile 0 ----
                    ok = pv_tile(0, tO0, tS0, sKV + stV * kTileBytes, jj == 0, p_it, 308, false);
                    if (!ok) break;
                    if (has_next) {
                        ok = wait1(bar_kv_full + 8 * stK, (kv_it / kWsStages) & 1, 307);
                        if (!ok) break;
                        tc_fence_after();
                        if (lane == 0) {
                            issue_qk(tS0, q_lo0, sKV + stK * kTileBytes);
                            tc_commit(bar_s_full);
                        }
                    } else if (lane == 0) {
                        tc_commit(bar_o_full);
                    }
                    // ---- tile 1 ----
                    ok = pv_tile(1, tO1, tS1, sKV + stV * kTileBytes, jj == 0, p_it1, 312, false);
                    if (!ok) break;
                    if (lane == 0) {
                        tc_commit(bar_kv_empty + 8 * stV);
                        if (has_next) {
                            issue_qk(tS1, q_lo1, sKV + stK * kTileBytes);
                            tc_commit(bar_s_full + 8);
                            tc_commit(bar_kv_empty + 8 * stK);
                            if (jj + 2 == n) tc_commit(bar_q_empty);
                        } else {
                            tc_commit(bar_o_full + 8);
                        }
                    }
                    if (has_next) ++kv_it;
                    ++p_it;
                    ++p_it1;
                }
                if (!ok) break;
            }
        }
        // warps 2 and 3 have nothing to do until teardown
    } else {
        // ===================================== softmax groups =====================================
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kWsRegsHigh));
        const int t = (warp - 4) >> 2;                 // query tile / softmax group
        const int row = ((warp & 3) << 5) | lane;      // row of the tile = TMEM lane
        const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
        const uint32_t tS = tmem_base + t * 128 + lane_off;
        const uint32_t tO = tmem_base + 256 + t * 128 + lane_off;
        const uint32_t bar_s = bar_s_full + 8 * t, bar_p = bar_p_full + 8 * t, bar_o = bar_o_full + 8 * t;
        uint32_t item_it = 0, s_it = 0, o_it = 0, x_it = 0;
        const float sc = p.scale_log2e;
        while (true) {
            const uint32_t slot = item_it & 1;
            if (!mbar_wait(bar_item_full + 8 * slot, (item_it >> 1) & 1, s_abort, 401)) break;
            WorkUnit u = ring[slot].u;
            const int n_splits = take_splits(u);
            const bool packed = ring[slot].packed != 0;
            // this thread's row: token `tok` of the unit, q-head h0 + row % grp
            const int grp = packed ? p.short_group : p.group;
            const int tile_tok0 = packed ? 0 : t * p.tile_tokens;     // first token of the tile within the unit
            const int tok = tile_tok0 + row / grp;
            const int ring_h0 = ring[slot].h0;
            const int out_row0 = (u.q_row0 + tok) * p.num_q_heads + ring_h0 + row % grp;   // its row of out / lse
            const int tile_toks = packed || u.rows - tile_tok0 < p.tile_tokens ? u.rows - tile_tok0 : p.tile_tokens;
            const int tile_rows = tile_toks * grp;                    // rows of this tile that exist (<= 0: none)
            const int valid = ring[slot].valid;
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_item_empty + 8 * slot);
            ++item_it;
            if (!valid) break;
            // the first part and head of a unit says how many partial results its rows have
            if (p.row_splits && u.split <= 0 && ring_h0 == 0 && row < tile_rows && row % grp == 0 && !(packed && t == 1)) p.row_splits[u.q_row0 + tok] = n_splits;
            // One item's softmax work.  The packed variant (short units) is compiled separately so that the
            // prefill path keeps the registers and the instruction count it had without it.
            auto run_item = [&](auto packed_tag) -> bool {
            constexpr bool kPacked = decltype(packed_tag)::value;
            // a warp of a packed tile without a row that exists only keeps the barriers moving
            const bool warp_idle = kPacked && (warp & 3) * 32 >= tile_rows;

            const int tile_pos0 = u.pos0 + tile_tok0;              // position of the tile's first row
            const int my_pos = u.pos0 + tok;
            float m_ref = -INFINITY, l_run = 0.f;
            bool ok = true;
            // a packed item: this group's tile takes every second KV tile
            for (int j = u.kv_begin + (kPacked ? t : 0); j < u.kv_end; j += kPacked ? 2 : 1) {
                const int tile0 = j * kTileN;
                ok = mbar_wait(bar_s, s_it & 1, s_abort, 402);
                if (!ok) break;
                ++s_it;
                tc_fence_after();
                if (warp_idle) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
#pragma unroll
                        for (int c = 0; c < 3; ++c)
                            if ((kPartMask >> c) & 1) mbar_arrive(bar_p_part + 16 * c + 8 * t);
                        mbar_arrive(bar_p);
                    }
                    continue;
                }
                uint32_t s[128];
                const bool diag = tile0 + kTileN - 1 > tile_pos0;  // keys beyond the row's position are masked
                const int lim = my_pos - tile0;                 // columns <= lim are visible
                float mx[8];
                // the second half of the row is still in flight while the first half is reduced
                tmem_ld32(tS, reinterpret_cast<uint32_t(&)[32]>(s[0]));
                tmem_ld32(tS + 32, reinterpret_cast<uint32_t(&)[32]>(s[32]));
                tc_wait_ld();
                tmem_ld32(tS + 64, reinterpret_cast<uint32_t(&)[32]>(s[64]));
                tmem_ld32(tS + 96, reinterpret_cast<uint32_t(&)[32]>(s[96]));
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    if (hh == 1) tc_wait_ld();
                    if (diag) {
#pragma unroll
                        for (int i = 0; i < 64; ++i)
                            if (hh * 64 + i > lim) s[hh * 64 + i] = 0xff800000u;  // -inf
                    }
#pragma unroll
                    for (int i = 0; i < 64; i += 16)
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const float v0 = __uint_as_float(s[hh * 64 + i + k]), v1 = __uint_as_float(s[hh * 64 + i + 8 + k]);
                            mx[k] = (hh == 0 && i == 0) ? fmaxf(v0, v1) : fmax3(mx[k], v0, v1);
                        }
                }
                const float mxa = fmaxf(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])),
                                        fmaxf(fmaxf(mx[4], mx[5]), fmaxf(mx[6], mx[7])));
                const float m_new = fmaxf(mxa * sc, m_ref);
                // lazy rescale: keep the old reference unless the maximum moved by more than 2^8
                // (rows beyond the tile's last one hold leftovers: they never ask for a rescale)
                const bool grow = row < tile_rows &&
                                  ((m_new - m_ref > kRescaleThreshold) || (m_ref == -INFINITY && m_new != -INFINITY));
                if (__any_sync(0xffffffffu, grow)) {
                    const float alpha = grow ? ex2(m_ref - m_new) : 1.f;  // m_ref = -inf gives 0
                    if (grow) m_ref = m_new;
                    l_run *= alpha;
                    if (j > u.kv_begin + (kPacked ? t : 0)) {   // O of this tile already holds something
                        uint32_t o[32];
#pragma unroll 1
                        for (int c = 0; c < 4; ++c) {
                            tmem_ld32(tO + c * 32, o);
                            tc_wait_ld();
#pragma unroll
                            for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                            tmem_st32(tO + c * 32, o);
                        }
                    }
                }
                const float m_use = (m_ref == -INFINITY) ? 0.f : m_ref;
                // Scale and reference of two columns in one packed fma: the loop is bound by the issue slots around the exponentials and,
                // in long launches, by power.  8192 tokens of 64/4 heads at 65536 keys 16.26 -> 15.79 ms, 4096 tokens of 32/32 184 -> 179 us.
                // (The sums stay scalar: packed ones took it back, 144.0 against 139.6 us on 2048 tokens of 8/1 heads at 14321 keys.)
                const uint64_t sc2 = pack_f32x2(sc, sc), neg_m2 = pack_f32x2(-m_use, -m_use);
                float sum0 = 0.f, sum1 = 0.f;
                // The wait for the early hand-over's store comes kPartWaitDefer pairs into the next chunk, so that the warp keeps
                // issuing exponentials while the store completes.
                constexpr int kDefer = kPartWaitDefer;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    uint32_t pk[16];
#pragma unroll
                    for (int i = 0; i < 32; i += 2) {
                        float x0, x1;
                        unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s[c * 32 + i]), __uint_as_float(s[c * 32 + i + 1])), sc2, neg_m2), x0, x1);
                        const float p0 = ex2(x0), p1 = ex2(x1);
                        sum0 += p0;
                        sum1 += p1;
                        pk[i >> 1] = pack_bf16x2(p0, p1);
                        if (c > 0 && ((kPartMask >> (c - 1)) & 1) && (i >> 1) == kDefer - 1) {
                            tc_wait_st();
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(bar_p_part + 16 * (c - 1) + 8 * t);
                        }
                    }
                    tmem_st16(tS + c * 16, pk);
                }
                l_run += sum0 + sum1;
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_p);
            }
            if (!ok) return false;

            // ---- epilogue ----
            const bool have_tiles = !kPacked || u.kv_begin + t < u.kv_end;   // (tile 1 of a one-tile packed item has none)
            if (have_tiles) {
                ok = mbar_wait(bar_o, o_it & 1, s_abort, 403);
                if (!ok) return false;
                ++o_it;
            }
            tc_fence_after();
            // the row of out / lse, or of the partials (split, token, q-head)
            const long long part_row = u.split < 0 ? out_row0 : static_cast<long long>(u.split) * p.total_q * p.num_q_heads + out_row0;
            if (kPacked && t == 1) {
                // hand (m, l) of every row to group 0, which also reads O_1; wait until it is done with them
                xm[row] = m_ref;
                xm[128 + row] = l_run;
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_x1);
                ok = mbar_wait(bar_x0, x_it & 1, s_abort, 404);
                if (!ok) return false;
                ++x_it;
                return true;
            }
            if (kPacked) {
                // merge the two tiles' partial results:  out = (a0 O_0 + a1 O_1) / (a0 l_0 + a1 l_1),  a_t = 2^(m_t - m)
                ok = mbar_wait(bar_x1, x_it & 1, s_abort, 405);
                if (!ok) return false;
                ++x_it;
                tc_fence_after();
                ws_packed_merge(p.out, p.lse, p.o_parts, p.lse_parts, u.split < 0, part_row,
                                u.kv_begin + 1 < u.kv_end /* O_1 was written at all */, xm, tO, row, tile_rows, m_ref, l_run);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_x0);
                return true;
            }
            {
                const float inv_l = 1.f / l_run;
                const bool live = row < tile_rows;
                // whole runs of 128 bytes: 64 bf16 or 32 fp32 columns of the warp's 32 rows at a time
                uint8_t* const stage = gen_bar + kWsStage + (warp - 4) * 4096;
                const int warp_row0 = (warp & 3) * 32;
                if (u.split < 0) {
#pragma unroll 1
                    for (int c = 0; c < 2; ++c) {
#pragma unroll
                        for (int hf = 0; hf < 2; ++hf) {
                            uint32_t r[32];
                            tmem_ld32(tO + c * 64 + hf * 32, r);
                            tc_wait_ld();
#pragma unroll
                            for (int q4 = 0; q4 < 4; ++q4) {
                                uint32_t w[4];
#pragma unroll
                                for (int e = 0; e < 4; ++e)
                                    w[e] = pack_bf16x2(__uint_as_float(r[q4 * 8 + 2 * e]) * inv_l,
                                                       __uint_as_float(r[q4 * 8 + 2 * e + 1]) * inv_l);
                                stage_put(stage, lane, hf * 4 + q4, make_uint4(w[0], w[1], w[2], w[3]));
                            }
                        }
                        stage_flush(stage, lane, 32, [&](int i) -> uint8_t* {
                            const int orow = __shfl_sync(0xffffffffu, out_row0, i);
                            return warp_row0 + i < tile_rows ? static_cast<uint8_t*>(p.out) + (static_cast<long long>(orow) * 128 + c * 64) * 2 : nullptr;
                        });
                    }
                } else {
                    const long long part0 = part_row - out_row0;
#pragma unroll 1
                    for (int c = 0; c < 4; ++c) {
                        uint32_t r[32];
                        tmem_ld32(tO + c * 32, r);
                        tc_wait_ld();
#pragma unroll
                        for (int q4 = 0; q4 < 8; ++q4)
                            stage_put(stage, lane, q4,
                                      make_uint4(__float_as_uint(__uint_as_float(r[q4 * 4]) * inv_l), __float_as_uint(__uint_as_float(r[q4 * 4 + 1]) * inv_l),
                                                 __float_as_uint(__uint_as_float(r[q4 * 4 + 2]) * inv_l), __float_as_uint(__uint_as_float(r[q4 * 4 + 3]) * inv_l)));
                        stage_flush(stage, lane, 32, [&](int i) -> uint8_t* {
                            const int orow = __shfl_sync(0xffffffffu, out_row0, i);
                            return warp_row0 + i < tile_rows ? reinterpret_cast<uint8_t*>(p.o_parts + (part0 + orow) * 128 + c * 32) : nullptr;
                        });
                    }
                }
                if (live) {
                    const float lse = (m_ref + log2f(l_run)) * 0.6931471805599453f;
                    if (u.split < 0) {
                        if (p.lse) p.lse[part_row] = lse;
                    } else {
                        p.lse_parts[part_row] = lse;
                    }
                }
            }
            tc_fence_before();
            return true;
            };
            if (kQuarters && packed && u.rows == 1) {
                const long long row0 = static_cast<long long>(u.q_row0) * p.num_q_heads + ring_h0;
                if (!ws_run_quarters(static_cast<uint8_t*>(p.out) + row0 * 256, p.lse ? p.lse + row0 : nullptr, u.kv_end, u.pos0, grp, sc, sBar, gen_bar, tmem_base,
                                     s_it, o_it, x_it))
                    break;
                const int n = (u.kv_end + 1 - t) >> 1;      // tiles of this group
                s_it += n;
                o_it += n > 0 ? 1 : 0;
                ++x_it;
                continue;
            }
            if (!(packed ? run_item(std::true_type{}) : run_item(std::false_type{}))) break;
        }
    }

    // ---- teardown ----
    __syncthreads();
    if (*s_abort != 0) {
        if (tid == 0 && p.status) atomicCAS(p.status, 0, 3 /* VPP_DEV_TIMEOUT */);
        for (int i = 0; i < 64; ++i) __nanosleep(1000);  // let copies and MMAs in flight drain
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 2) tmem_dealloc(tmem_base, 512);
}

}  // namespace vpp
