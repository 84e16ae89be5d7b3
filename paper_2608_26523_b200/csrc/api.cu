// Host side of the C ABI declared in include/vpp.h: argument validation, workspace layout,
// tensor-map construction and kernel launches.  Nothing here synchronises or allocates device memory.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdarg>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <numeric>

#include "../../include/vpp.h"
#include "attn_mla2.cuh"
#include "attn_dsa.cuh"
#include "attn_ws.cuh"
#include "bounded.h"
#include "common.cuh"
#include "kv_append.cuh"
#include "merge.cuh"
#include "prep.cuh"
#include "wait_test.cuh"

namespace {

thread_local char g_err[512] = "";
thread_local int32_t g_launches = 0;

vpp_status fail(vpp_status s, const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof g_err, fmt, ap);
    va_end(ap);
    return s;
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// The status word of a call that launches nothing.
vpp_status zero_status(int32_t* status, cudaStream_t stream) {
    if (status && cudaMemsetAsync(status, 0, sizeof(int32_t), stream) != cudaSuccess)
        return fail(VPP_ERR_CUDA, "memset status: %s", cudaGetErrorString(cudaGetLastError()));
    return VPP_OK;
}

// Launch with programmatic stream serialization: the kernel may start (and set itself up) while its predecessor in the
// stream still runs, and waits for it (griddepcontrol.wait) before it touches memory.
template <typename... Params, typename... Args>
cudaError_t launch(void (*kernel)(Params...), unsigned blocks, unsigned threads, size_t smem, cudaStream_t stream, Args... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

// ---- device facts, cached per device -------------------------------------------------------------
struct DeviceInfo {
    bool ready = false;
    int sm_count = 0;
    bool attrs_set = false;
};
std::mutex g_mu;
DeviceInfo g_dev[64];

int sm_count_or_default() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return 148;
    }
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_dev[dev].ready) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
            cudaGetLastError();
            n = 148;
        }
        g_dev[dev].sm_count = n;
        g_dev[dev].ready = true;
    }
    return g_dev[dev].sm_count;
}

// ---- tensor maps ------------------------------------------------------------------------------------
using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn get_encode() {
    static EncodeFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeFn>(p);
        else
            cudaGetLastError();
    });
    return fn;
}

// Encoded tensor maps are cached: a serving loop calls with the same buffers and shapes again and again, and seven
// (d = 128) or four (MLA) driver encodes per call are a visible part of a short launch.  A map depends only on (base address, rank,
// extents, strides, box), so an entry never goes stale; the cache is a small 4-way set-associative table (least recently
// used way replaced) guarded by a mutex.
struct TmapKey {
    const void* base;
    uint64_t dims[5];
    uint64_t strides[4];
    uint32_t box[5];
    uint32_t rank;
};
using RawEncodeFn = bool (*)(CUtensorMap*, const TmapKey&);

class TmapCache {
public:
    static constexpr int kSets = 64, kWays = 4;   // a call uses up to seven maps; 256 entries serve a few dozen distinct launches
    bool get(const TmapKey& key, RawEncodeFn encode, CUtensorMap* out) {
        const uint64_t h = hash(key);
        Slot* set = slots_ + (h % kSets) * kWays;
        std::lock_guard<std::mutex> lk(mu_);
        ++lookups_;
        ++clock_;
        Slot* victim = set;
        for (int w = 0; w < kWays; ++w) {
            Slot& sl = set[w];
            if (sl.valid && sl.hash == h && std::memcmp(&sl.key, &key, sizeof key) == 0) {
                sl.stamp = clock_;
                *out = sl.map;
                return true;
            }
            // the way to replace on a miss: an empty one if there is any, else the least recently used
            if (victim->valid && (!sl.valid || sl.stamp < victim->stamp)) victim = &sl;
        }
        CUtensorMap m;
        if (!encode(&m, key)) return false;
        ++encodes_;
        victim->key = key;
        victim->hash = h;
        victim->map = m;
        victim->valid = true;
        victim->stamp = clock_;
        *out = m;
        return true;
    }
    void stats(int64_t* lookups, int64_t* encodes) {
        std::lock_guard<std::mutex> lk(mu_);
        *lookups = lookups_;
        *encodes = encodes_;
    }
private:
    struct Slot {
        TmapKey key;
        uint64_t hash = 0, stamp = 0;
        CUtensorMap map;
        bool valid = false;
    };
    static uint64_t hash(const TmapKey& k) {   // over the key's words (the key is zero-initialised, padding included)
        static_assert(sizeof(TmapKey) % 8 == 0, "whole words");
        uint64_t w[sizeof k / 8], h = 1469598103934665603ull;
        std::memcpy(w, &k, sizeof k);
        for (uint64_t x : w) h = (h ^ x ^ (h >> 29)) * 0x9E3779B97F4A7C15ull;
        return h ^ (h >> 32);
    }
    std::mutex mu_;
    Slot slots_[kSets * kWays];
    int64_t lookups_ = 0, encodes_ = 0;
    uint64_t clock_ = 0;
};
TmapCache g_tmaps;

// bf16 tensor, innermost dimension contiguous, 128-byte swizzle, zero fill out of bounds.
bool encode_with_driver(CUtensorMap* m, const TmapKey& k) {
    EncodeFn enc = get_encode();
    if (!enc) return false;
    cuuint64_t gd[5], gs[4];
    cuuint32_t bx[5], es[5];
    for (uint32_t i = 0; i < k.rank; ++i) {
        gd[i] = k.dims[i];
        bx[i] = k.box[i];
        es[i] = 1;
        if (i > 0) gs[i - 1] = k.strides[i - 1];
    }
    CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, k.rank, const_cast<void*>(k.base), gd, gs, bx, es,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

TmapKey make_key(const void* base, int rank, const uint64_t* dims, const uint64_t* strides_bytes, const uint32_t* box) {
    TmapKey k;
    std::memset(&k, 0, sizeof k);
    k.base = base;
    k.rank = static_cast<uint32_t>(rank);
    for (int i = 0; i < rank; ++i) {
        k.dims[i] = dims[i];
        k.box[i] = box[i];
        if (i > 0) k.strides[i - 1] = strides_bytes[i - 1];
    }
    return k;
}

bool make_tmap(CUtensorMap* m, const void* base, int rank, const uint64_t* dims, const uint64_t* strides_bytes,
               const uint32_t* box) {
    return g_tmaps.get(make_key(base, rank, dims, strides_bytes, box), encode_with_driver, m);
}

// The two maps of a K or V cache of the d = 128 kernel (attn_ws.cuh) and how (block, kv-head) becomes one coordinate of the
// first: both strides are whole numbers of `unit`.  Where that coordinate would not fit an int32 (strides with hardly a common
// divisor in a huge cache) every tile takes the exact map.
bool make_kv_maps(const void* base, int64_t block_stride, int64_t token_stride, int64_t head_stride, int B, int n_blocks, int heads, int box_rows,
                  CUtensorMap* tm, CUtensorMap* tm_exact, int32_t* block_units, int32_t* head_units, int32_t* end, int32_t* exact_from) {
    const uint64_t dx[5] = {64, static_cast<uint64_t>(B), 2, static_cast<uint64_t>(heads), static_cast<uint64_t>(n_blocks)};
    const uint64_t sx[4] = {static_cast<uint64_t>(token_stride) * 2, 128, static_cast<uint64_t>(head_stride) * 2,
                            static_cast<uint64_t>(block_stride) * 2};
    const uint32_t bx[5] = {64, vpp::kExactRows, 2, 1, 1};
    if (!make_tmap(tm_exact, base, 5, dx, sx, bx)) return false;
    const int64_t unit = std::gcd(block_stride, head_stride);
    const int64_t last = ((n_blocks - 1) * block_stride + (heads - 1) * head_stride) / unit;
    if (last >= INT32_MAX) {
        *tm = *tm_exact;
        *exact_from = 0;
        return true;
    }
    *block_units = static_cast<int32_t>(block_stride / unit);
    *head_units = static_cast<int32_t>(head_stride / unit);
    *end = static_cast<int32_t>(last + 1);
    const int groups = B / vpp::kExactRows;
    const uint64_t d[5] = {64, vpp::kExactRows, 2, static_cast<uint64_t>(groups > 0 ? groups : 1), static_cast<uint64_t>(last + 1)};
    const uint64_t s[4] = {static_cast<uint64_t>(token_stride) * 2, 128, static_cast<uint64_t>(token_stride) * 2 * vpp::kExactRows,
                           static_cast<uint64_t>(unit) * 2};
    const uint32_t b[5] = {64, vpp::kExactRows, 2, static_cast<uint32_t>(box_rows / vpp::kExactRows), 1};
    return make_tmap(tm, base, 5, d, s, b);
}

// ---- validation -------------------------------------------------------------------------------------
bool is_pow2(int x) { return x > 0 && (x & (x - 1)) == 0; }
int ilog2(int x) {
    int s = 0;
    while ((1 << s) < x) ++s;
    return s;
}

enum class Family { kGqa128, kMla576, kNone };

vpp_status validate(const vpp_chunk_attn_args* a, Family* fam) {
    if (!a) return fail(VPP_ERR_INVALID_ARG, "args is null");
    if (a->num_reqs < 0 || a->total_q < 0 || a->max_seq_len < 0)
        return fail(VPP_ERR_INVALID_ARG, "num_reqs, total_q and max_seq_len must be >= 0");
    if (a->num_q_heads <= 0 || a->num_kv_heads <= 0 || a->num_q_heads % a->num_kv_heads != 0)
        return fail(VPP_ERR_INVALID_ARG, "num_q_heads (%d) must be a positive multiple of num_kv_heads (%d)",
                    a->num_q_heads, a->num_kv_heads);
    if (!(a->softmax_scale > 0.f) || !std::isfinite(a->softmax_scale))
        return fail(VPP_ERR_INVALID_ARG, "softmax_scale must be positive and finite");
    if (a->num_kv_splits < 0 || a->num_kv_splits > 64)
        return fail(VPP_ERR_INVALID_ARG, "num_kv_splits must be in [0, 64]");
    if (a->head_dim_qk == 128 && a->head_dim_v == 128)
        *fam = Family::kGqa128;
    else if (a->head_dim_qk == 576 && a->head_dim_v == 512 && a->num_kv_heads == 1)
        *fam = Family::kMla576;
    else
        return fail(VPP_ERR_UNSUPPORTED, "no kernel for head dims (%d, %d) with %d kv heads", a->head_dim_qk,
                    a->head_dim_v, a->num_kv_heads);
    if (a->block_table != nullptr) {
        if (!is_pow2(a->block_size) || a->block_size < 16)
            return fail(VPP_ERR_UNSUPPORTED, "block_size %d: need a power of two >= 16", a->block_size);
        if (a->max_blocks_per_req <= 0 || a->num_blocks <= 0)
            return fail(VPP_ERR_INVALID_ARG, "paged cache needs max_blocks_per_req > 0 and num_blocks > 0");
    }
    return VPP_OK;
}

vpp_status validate_pointers(const vpp_chunk_attn_args* a) {
    if (a->num_reqs > 0 && (!a->prefix_len || !a->chunk_len))
        return fail(VPP_ERR_INVALID_ARG, "prefix_len / chunk_len is null");
    if (a->total_q > 0 && (!a->q || !a->out || !a->k_cache || !a->v_cache))
        return fail(VPP_ERR_INVALID_ARG, "q, k_cache, v_cache and out must be non-null");
    auto mis16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) != 0; };
    if (mis16(a->q) || mis16(a->out) || mis16(a->k_cache) || mis16(a->v_cache))
        return fail(VPP_ERR_INVALID_ARG, "q, out, k_cache and v_cache must be 16-byte aligned");
    const int64_t st[6] = {a->k_block_stride, a->k_token_stride, a->k_head_stride,
                           a->v_block_stride, a->v_token_stride, a->v_head_stride};
    for (int i = 0; i < 6; ++i)
        if (st[i] <= 0 || st[i] % 8 != 0)
            return fail(VPP_ERR_INVALID_ARG, "cache strides must be positive multiples of 8 elements");
    if (a->block_table == nullptr && a->num_reqs > 1 &&
        (a->k_block_stride < a->k_token_stride * a->max_seq_len || a->v_block_stride < a->v_token_stride * a->max_seq_len))
        return fail(VPP_ERR_INVALID_ARG,
                    "contiguous cache: every request's region must hold max_seq_len (%d) slots, but the block strides are "
                    "shorter than max_seq_len token strides", a->max_seq_len);
    return VPP_OK;
}

// Key-range splits of a launch: the most a work unit may get, and whether the work decomposition chooses each unit's own
// number so that the KV tiles are shared out evenly over the SMs (prep.cuh) instead of cutting every unit into that many.
struct SplitPlan {
    int splits;
    bool balanced;
};
// How the work decomposition counts work items of this launch.
struct ItemCounts {
    int unit_rows, unit_items, short_items, slots;
};

// How the d = 128 kernel packs (token, q-head) pairs into the rows of a tile (attn_ws.cuh).
struct RowPacking {
    int group, tile_tokens;         // items of two tiles: q-heads x tokens of a tile
    int short_group, short_tokens;  // items of one tile
    int unit_rows;                  // query rows (tokens) per work unit
};
RowPacking row_packing(const vpp_chunk_attn_args* a) {
    const int G = a->num_q_heads / a->num_kv_heads;
    RowPacking r{};
    // the largest part of a kv-head's group that fills at least 125 of the 128 rows (1 always does)
    auto fills = [&](int d) { return G % d == 0 && d * (vpp::kTileM / d) >= 125; };
    r.group = 1;
    for (int d = 1; d <= vpp::kTileM && d <= G; ++d)
        if (fills(d)) r.group = d;
    // a packed item streams its K/V for these rows alone: the whole group if it fits a tile, however well it fills it
    r.short_group = G <= vpp::kTileM ? G : r.group;
    r.short_tokens = vpp::kTileM / r.short_group;
    if (a->num_reqs == 1 && (G & (G - 1)) != 0) {
        // One chunk, of a known length, in groups that are no power of two (whose units divide one another): a smaller part of the group where the largest leaves a tail that goes over all the keys for a
        // few tokens.  512 tokens of groups of three are six units of 84 and eight tokens over, or, head by head, two units of
        // 256: 512 tokens of 24/8 heads at 16384 keys 143 us and 101, 768 tokens of 48/8 at 65536 1650 and 1050.
        auto visits = [&](int d) {    // tile visits per KV tile and kv-head
            const int unit = 2 * (vpp::kTileM / d), rest = a->total_q % unit;
            return (a->total_q / unit + (rest > r.short_tokens ? 1 : 0)) * 2.0 * (G / d) + (rest > 0 && rest <= r.short_tokens ? 2.0 : 0.0);
        };
        const int largest = r.group;
        for (int d = largest - 1; d >= 1; --d)
            if (fills(d) && visits(d) < 0.95 * visits(largest) && visits(d) < visits(r.group)) r.group = d;
    }
    r.tile_tokens = vpp::kTileM / r.group;
    r.unit_rows = 2 * r.tile_tokens;
    return r;
}
// Query rows of a work unit.
int unit_rows_of(const vpp_chunk_attn_args* a, Family fam) { return fam == Family::kGqa128 ? row_packing(a).unit_rows : vpp::kTileM; }

// The absorbed-MLA kernel runs on pairs of SMs (2-CTA clusters).
bool mla_kernel_available() { return sm_count_or_default() >= 2; }

ItemCounts item_counts(const vpp_chunk_attn_args* a, Family fam) {
    const int sms = sm_count_or_default();
    if (fam == Family::kMla576) {
        const bool packs = a->num_q_heads <= 2 * vpp::kMla2Rows;
        return {vpp::kTileM, a->num_q_heads, packs ? 1 : a->num_q_heads, sms / 2 > 0 ? sms / 2 : 1};
    }
    const RowPacking r = row_packing(a);
    return {r.unit_rows, a->num_q_heads / r.group, a->num_q_heads / r.short_group, sms};
}

// The start and end of a work item (query load, first K/V, epilogue) in KV tiles: ~4 us of ~2 us a tile; packed items
// ~4.5 us of ~1.5 us; MLA items (144 KB of queries, 256 KB of partial results) ~9 us of ~1.9.
constexpr int kLead = 2, kShortLead = 3, kMlaLead = 5;
constexpr double kL2Keeps = 96e6;   // bytes of keys and values that stay in the 126 MB of L2 while a launch goes over them
constexpr int kMinLen = 2, kMinShortLen = 4;   // fewest KV tiles worth a work item (start-up ~4 us, ~2 / ~1 us per tile)

// Does the d = 128 kernel run with a second producer warp, for the V tiles?  Where most of the work is packed items, which are bound by the
// arrival of K/V: batches of requests of 64 tokens or fewer on average.  64/8 heads, without it and with it: 30 decode rows at 4000 to
// 4400 keys and 64 tokens at 8000 155 and 130 us, 200 rows and 1000 tokens 1046 and 916, 32 requests of 4 tokens 165 and 144; the
// other way round 60 rows and 4000 tokens 1351 and 1384, a chunk by itself 1 to 2 %.
bool v_producer(const vpp_chunk_attn_args* a) { return a->total_q <= (a->num_reqs > 1 ? 64ll * a->num_reqs : 1); }

// Does the d = 128 kernel share out the keys of a decode row's tiles over the softmax warps (attn_ws.cuh)?  Its items end later (the join of
// eight results) and hand the SM to the next one earlier, so it pays where an SM runs several, one after the other, and not where
// each has one; groups of more heads have a longer join.  Uncut rows of the same batch packed and shared out, us, contexts to 8192 / to 512 / of 128
// tokens: 8 rows of 64/8 heads (64 items) 75.3 and 76.8 / 17.5 and 17.9 / 12.7 both; 24 of 32/8 (192) 83.7 and 84.5 / 19.9 and 20.1 / 17.9
// and 17.1; 40 of 32/8 (320) 134.6 and 134.2 / 27.6 and 27.4 / 23.9 and 22.7; 300 of 64/8 to 512 126.7 and 117.8; 256 to 8192 765 and 748.  Groups of
// 16: 64 rows of 64/4 (256) 106.2 and 106.6 / 23.8 and 24.5 / 24.4 and 24.3; 96 (384) 150.6 both / 30.8 and 31.2 / 26.5 and 25.4;
// 149 (596) 216.9 and 214.9 / 41.8 and 40.8 / 31.6 and 31.0.
// (Which of more requests than tokens are decode rows only the device knows: a chunk of 1500 tokens among 2000 empty requests takes 70.8 us so, 69.2
// otherwise; 256 rows among 768 empty ones 219 and 231.)
bool shares_out_keys(const vpp_chunk_attn_args* a, int short_group) {
    const long long items = static_cast<long long>(a->total_q) * (a->num_q_heads / short_group);
    return a->total_q <= a->num_reqs && short_group <= vpp::kQuarterHeads && items >= (short_group <= 8 ? 2ll : 3ll) * sm_count_or_default();
}

// Time of a KV tile of a work item, measured at full clock.
struct TileTimes {
    double unit_us, short_us;
};
TileTimes tile_times(const vpp_chunk_attn_args* a, Family fam) {
    if (fam == Family::kMla576) return {1.6, 1.6};
    return {1.75, v_producer(a) ? 0.85 : 1.3};
}

// Ranges of a balanced cut when every unit has `items` work items: as many as fill the slots in one round, or in up to four where
// one would leave a fifth of them idle.
int ranges_of(int slots, int items) {
    int best = 1;
    double fill = 0;
    for (int k = 1; k <= 4 && fill < 0.8; ++k) {
        const int r = k * slots / items;
        const double f = static_cast<double>(r) * items / (k * slots);
        if (r >= 1 && f > fill) {
            fill = f;
            best = r;
        }
    }
    return best;
}

// Equal splits of a batch of decode rows that fills the SMs (80 % of them or more): as many as leave the least idle last wave,
// charged with what splitting costs (measured: partials + merge ~5 %, ~1 % per extra split, ~4 us of start-up per unit against
// ~1.5 us per KV tile when all SMs stream).
int decode_splits(long long items, int slots, double tiles) {
    int best = 1;
    double best_cost = 0.0;
    for (int s = 1; s <= 4; ++s) {
        if (s > 1 && tiles / s < 4.0) break;   // keep at least 4 KV tiles per split
        const double waves = static_cast<double>(items) * s / slots;
        double cost = std::ceil(waves) / waves;
        if (s > 1) cost *= 1.05 + 0.01 * s;
        cost *= 1.0 + (s - 1) * 4.0 / (tiles * 1.5 + 1.0);
        if (s == 1 || cost < best_cost) {
            best = s;
            best_cost = cost;
        }
    }
    return best;
}

// Equal splits of one request's chunk, and the time they take: waves of items, the last of them as idle as the items are equally long
// (a chunk that is half the context or more has items of all lengths, which go longest first), and the partial results (whose
// stores mostly hide behind the items).  Measured on 8192-token chunks at 64K-128K prefixes: 512 items (3.46 waves) gain 7-9 % from two splits, 256 items 1.5 % from
// four, 128 and 1024 items are best unsplit; 4096 tokens of 32/32 heads without a prefix (512 items) 131 us unsplit, 215 in two.
int chunk_splits(long long items, int slots, double tiles, double chunk_tiles, double unit_us, double parts_us, int most, double* us) {
    const double mean = tiles - 0.5 * chunk_tiles, equal = chunk_tiles < 0.5 * tiles ? 1.0 - chunk_tiles / tiles : 0.0;
    int best = 1;
    for (int s = 1; s <= 8 && s <= most; ++s) {
        if (s > 1 && tiles / s < 4.0) break;   // keep at least 4 KV tiles per split
        const double w = static_cast<double>(items) * s / slots;
        const double waves = std::fmax(w + (std::ceil(w) - w) * equal, 1.0);
        const double t = std::fmax(waves * (mean / s + kLead), tiles / s + kLead) * unit_us * (1.0 + 0.01 * (s - 1)) + (s > 1 ? 8.0 + 0.4 * parts_us * s : 0.0);
        if (s == 1 || t < 0.975 * *us) {
            best = s;
            *us = t;
        }
    }
    return best;
}

// most: parts a unit of a launch of few items may get.
SplitPlan plan_splits(const vpp_chunk_attn_args* a, Family fam, int most = vpp::kMergeMaxSplits) {
    if (a->num_kv_splits >= 1) return {a->num_kv_splits, false};
    if (a->total_q <= 0 || a->num_reqs <= 0) return {1, false};
    // An upper bound on the work items of an uncut launch.  Where they fill the slots several times the dynamic longest-first
    // order balances them well enough; where they do not, the shares are cut to measure.
    const ItemCounts c = item_counts(a, fam);
    const bool decode = a->total_q <= a->num_reqs, one_request = a->num_reqs == 1, mla = fam == Family::kMla576;
    const long long units = decode ? a->total_q : (a->total_q + c.unit_rows - 1) / c.unit_rows + (one_request ? 0 : a->num_reqs);
    const int per_unit = decode ? c.short_items : c.unit_items;
    const long long items = units * per_unit, tiles = (a->max_seq_len + vpp::kTileN - 1) / vpp::kTileN;
    // (one request, or a batch of decode rows, of the d = 128 family: from 80 % of the SMs on the split count that leaves the
    //  least idle last wave, below; MLA's pairs of SMs take their items in a fixed order, so more items than pairs are left alone:
    //  110 decode rows 75 us uncut, 88 cut; mixed batches of d = 128: up to two items per slot)
    const bool few = mla ? items <= c.slots : decode || one_request ? items * 5 < c.slots * 4ll : items < 2ll * c.slots;
    const double chunk_tiles = a->total_q / static_cast<double>(vpp::kTileN);
    const double parts_us = 8.0 * a->total_q * a->num_q_heads * a->head_dim_v / 3e6;      // of one partial result per row, written and read
    if (few) {
        // Is it worth it?  Uncut, the longest unit takes tiles * us, or a ragged batch of more items than slots about half of that
        // after the mean ends.  Cut, everybody takes its share, plus the decomposition's and the merge's part and the partial
        // results, written and read once at ~3 TB/s.  (Lengths are only known to be at most max_seq_len: one request's units
        // are taken to end there, a batch's to be half as long.)  200 tokens of 64 heads at 2048 keys: 40 us uncut, 47 cut; 256 tokens of 4
        // heads at 1024 keys 24 uncut, 21 cut.
        const TileTimes t = tile_times(a, fam);
        const double us = decode ? t.short_us : t.unit_us, mean = one_request ? (decode ? tiles : tiles - 0.5 * chunk_tiles) : 0.5 * tiles;
        const int least = decode ? kMinShortLen : kMinLen;
        double share = mean * units / ranges_of(c.slots, per_unit);
        if (share < least) share = least;
        if (share < mean / most) share = mean / most;
        const double uncut_us = us * (items <= c.slots ? tiles : std::fmax(tiles, mean * items / c.slots + 0.5 * tiles));
        double cut_us = us * share + (decode && !mla ? 6.0 : 8.0) + parts_us * (mean / share > 1 ? mean / share : 1);
        const double kv_bytes = 512.0 * a->max_seq_len * a->num_kv_heads;
        if (one_request && !mla && units > 1 && kv_bytes > kL2Keeps) {
            // The parts of a balanced cut read different keys at the same time, so that every unit fetches keys that L2 does not keep
            // from memory for itself (4.1 TB/s); equal splits of all units go over them together.  400 tokens of 64/8 heads at 65536 keys
            // 949 us balanced, 804 equal; 256 tokens of 64/4 heads at 131072 keys 1003, 944; 300 of 32/8 there 684, 600.
            cut_us = std::fmax(cut_us, units * kv_bytes / 4.1e6 + 8.0);
            double equal_us = 0;
            const int equal = chunk_splits(items, c.slots, tiles, chunk_tiles, us, parts_us, most, &equal_us);
            if (equal_us < cut_us) return {equal, false};
        }
        if (cut_us >= uncut_us) return {1, false};
        // what a unit may need: its share of the slots when all are equally long; several times that when they are ragged (one
        // long context among short ones gets most of the slots)
        long long s = one_request ? (c.slots + items - 1) / items + 1 : (2ll * c.slots + items - 1) / items + 2;
        if (s > tiles / least) s = tiles / least;
        if (s > most) s = most;
        return s < 2 ? SplitPlan{1, false} : SplitPlan{static_cast<int>(s), true};
    }
    if (mla || !(decode || one_request)) return {1, false};   // (others have two items a slot or more here, of different lengths)
    if (decode) return {decode_splits(items, c.slots, a->max_seq_len / static_cast<double>(vpp::kTileN)), false};
    // (a last unit whose rows fit one tile runs packed)
    const int rest = a->total_q % c.unit_rows;
    const long long tail = rest > 0 && rest <= row_packing(a).short_tokens ? c.short_items - c.unit_items : 0;
    double equal_us = 0;
    return {chunk_splits(items + tail, c.slots, tiles, chunk_tiles, tile_times(a, fam).unit_us, parts_us, most, &equal_us), false};
}

using MergeKernel = void (*)(const float*, const float*, int, long long, int, int, const int32_t*, const vpp::WorkHeader*, __nv_bfloat16*,
                             float*);
// The kernel and the grid for a merge of `splits` partials of total_q x num_q_heads rows of head_dim_v features.
MergeKernel pick_merge_kernel(int splits, long long total_q, int num_q_heads, int head_dim_v, int sms, unsigned* blocks) {
    const long long pairs = total_q * num_q_heads;
    const long long pieces = pairs * (head_dim_v / 4);
    if (splits <= vpp::kMergeSmallMax && head_dim_v % 4 == 0 && pieces < (1ll << 31)) {
        long long b = (pieces + vpp::kMergeThreads - 1) / vpp::kMergeThreads;
        if (b > 12ll * sms) b = 12ll * sms;
        *blocks = static_cast<unsigned>(b);
        if (splits <= 2) return vpp::lse_merge_small_kernel<2, 4>;
        if (splits <= 4) return vpp::lse_merge_small_kernel<4, 2>;
        return vpp::lse_merge_small_kernel<8, 1>;
    }
    long long b = (pairs * 32 + vpp::kMergeThreads - 1) / vpp::kMergeThreads;
    if (b > 8ll * sms) b = 8ll * sms;
    *blocks = static_cast<unsigned>(b);
    return vpp::lse_merge_kernel<2, 4>;
}

vpp::WorkspaceLayout layout_of(const vpp_chunk_attn_args* a, Family fam, SplitPlan plan) {
    vpp::WorkspaceLayout L{};
    const int S = plan.splits;
    L.balanced = plan.balanced && S > 1 ? 1 : 0;
    const int unit_rows = unit_rows_of(a, fam);
    const long long tiles = (a->total_q + unit_rows - 1) / unit_rows + a->num_reqs;
    L.splits = S;
    L.max_units = static_cast<int32_t>(tiles * S);
    size_t off = 0;
    L.header = off;
    off = align_up(off + sizeof(vpp::WorkHeader), 256);
    L.units = off;
    off = align_up(off + sizeof(vpp::WorkUnit) * static_cast<size_t>(L.max_units > 0 ? L.max_units : 1), 256);
    L.row_splits = off;  // followed by q_start and tile_start scratch
    off = align_up(off + sizeof(int32_t) * (static_cast<size_t>(a->total_q) + 2 * (static_cast<size_t>(a->num_reqs) + 1)),
                   256);
    L.o_parts = off;
    if (S > 1)
        off = align_up(off + sizeof(float) * static_cast<size_t>(S) * a->total_q * a->num_q_heads * a->head_dim_v, 256);
    L.lse_parts = off;
    if (S > 1) off = align_up(off + sizeof(float) * static_cast<size_t>(S) * a->total_q * a->num_q_heads, 256);
    L.total = off;
    return L;
}

// The layout of a launch whose workspace may hold `limit` bytes: where the library's own cut needs more, its units get fewer parts
// (2048 tokens of 8/1 heads at 16369 keys: 32.3 MiB with four, 24.2 with three; 119 us, 137, and 229 uncut), and none if that does
// not do.  The equal splits of a launch that fills the SMs are not made fewer: their number is that of the best last wave.
vpp::WorkspaceLayout layout_for(const vpp_chunk_attn_args* a, Family fam, size_t limit) {
    SplitPlan plan = plan_splits(a, fam);
    vpp::WorkspaceLayout L = layout_of(a, fam, plan);
    if (L.total <= limit || a->num_kv_splits != 0 || plan.splits == 1) return L;
    const vpp::WorkspaceLayout uncut = layout_of(a, fam, {1, false});
    if (uncut.total > limit) return uncut;
    const size_t part = (L.total - uncut.total) / (plan.splits - 1);     // bytes that one more part takes
    for (int most = 1 + static_cast<int>((limit - uncut.total) / part); most > 1; --most) {   // (the first or, by alignment, the second fits)
        plan = plan_splits(a, fam, most);
        L = layout_of(a, fam, plan);
        if (L.total <= limit) return L;
    }
    return uncut;
}

}  // namespace

size_t vpp::workspace_size_within(const vpp_chunk_attn_args* a, size_t limit) {
    Family fam = Family::kNone;
    if (validate(a, &fam) != VPP_OK) return 0;
    return layout_for(a, fam, limit).total;
}

extern "C" {

const char* vpp_status_string(vpp_status s) {
    switch (s) {
        case VPP_OK: return "ok";
        case VPP_ERR_INVALID_ARG: return "invalid argument";
        case VPP_ERR_UNSUPPORTED: return "unsupported shape";
        case VPP_ERR_WORKSPACE: return "workspace missing or too small";
        case VPP_ERR_CUDA: return "CUDA call failed";
        case VPP_ERR_TIMEOUT: return "device wait timed out";
    }
    return "unknown status";
}

const char* vpp_last_error(void) { return g_err; }
int32_t vpp_last_launch_count(void) { return g_launches; }

size_t vpp_chunk_attn_workspace_size(const vpp_chunk_attn_args* a) { return vpp::workspace_size_within(a, SIZE_MAX); }

namespace {
// Key range of a partial launch, in KV tiles of kTileN keys (null: the whole causal range, final results).
struct KeyRange {
    int32_t begin_tile, end_tile;
};
vpp_status run_chunk_attn(const vpp_chunk_attn_args* a, vpp_stream_t stream_, const KeyRange* range, size_t limit);
}  // namespace

vpp_status vpp_chunk_attn_fwd(const vpp_chunk_attn_args* a, vpp_stream_t stream_) {
    return run_chunk_attn(a, stream_, nullptr, SIZE_MAX);
}

vpp_status vpp_chunk_attn_partial_fwd(const vpp_chunk_attn_args* args, int32_t kv_begin, int32_t kv_end, float* o_part,
                                      float* lse_part, vpp_stream_t stream_) {
    g_err[0] = 0;
    if (!args) return fail(VPP_ERR_INVALID_ARG, "args is null");
    if (kv_begin < 0 || kv_end <= kv_begin) return fail(VPP_ERR_INVALID_ARG, "need 0 <= kv_begin < kv_end");
    if (kv_begin % vpp::kTileN != 0 || (kv_end % vpp::kTileN != 0 && kv_end < args->max_seq_len))
        return fail(VPP_ERR_INVALID_ARG, "kv_begin must be a multiple of %d, and so must kv_end unless it is >= max_seq_len",
                    vpp::kTileN);
    if (args->total_q > 0 && (!o_part || !lse_part)) return fail(VPP_ERR_INVALID_ARG, "o_part and lse_part must be non-null");
    vpp_chunk_attn_args b = *args;
    b.num_kv_splits = 1;       // the caller's ranges are the split
    b.out = o_part;            // (fp32 here; only checked for null and alignment)
    b.lse = lse_part;
    KeyRange r;
    r.begin_tile = kv_begin / vpp::kTileN;
    r.end_tile = static_cast<int32_t>((static_cast<int64_t>(kv_end) + vpp::kTileN - 1) / vpp::kTileN);
    return run_chunk_attn(&b, stream_, &r, SIZE_MAX);
}

namespace {
vpp_status run_chunk_attn(const vpp_chunk_attn_args* a, vpp_stream_t stream_, const KeyRange* range, size_t limit) {
    g_err[0] = 0;
    Family fam = Family::kNone;
    vpp_status st = validate(a, &fam);
    if (st != VPP_OK) return st;
    st = validate_pointers(a);
    if (st != VPP_OK) return st;
    const vpp::WorkspaceLayout L = layout_for(a, fam, limit);
    if (!a->workspace || a->workspace_bytes < L.total)
        return fail(VPP_ERR_WORKSPACE, "workspace: need %zu bytes, got %zu", L.total, a->workspace_bytes);
    if (reinterpret_cast<uintptr_t>(a->workspace) & 255u)
        return fail(VPP_ERR_INVALID_ARG, "workspace must be 256-byte aligned");
    if (fam == Family::kMla576 &&
        (a->v_cache != a->k_cache || a->v_block_stride != a->k_block_stride || a->v_token_stride != a->k_token_stride ||
         a->v_head_stride != a->k_head_stride))
        return fail(VPP_ERR_UNSUPPORTED,
                    "the (576, 512) kernel needs v_cache to alias k_cache with the same strides (V = first 512 features)");

    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    g_launches = 0;
    if (a->total_q == 0 || a->num_reqs == 0) return zero_status(a->status, stream);
    // (otherwise the attention kernel writes the status word: a memset node and its gap cost a short launch 4 us)
    if (fam == Family::kMla576 && !mla_kernel_available())
        return fail(VPP_ERR_UNSUPPORTED, "the absorbed-MLA kernel needs clusters of two SMs");

    uint8_t* ws = static_cast<uint8_t*>(a->workspace);
    const bool paged = a->block_table != nullptr;
    const int B = paged ? a->block_size : a->max_seq_len;
    const int n_blocks = paged ? a->num_blocks : a->num_reqs;
    const int tile_n = fam == Family::kMla576 ? vpp::kMla2BoxRows : vpp::kTileN;  // keys one copy can bring (MLA: a CTA's 64 of the pair's tile)
    const int box_rows = paged ? (B < tile_n ? B : tile_n) : tile_n;

    // ---- tensor maps ----
    CUtensorMap tm_q, tm_qs, tm_q1, tm_k, tm_v, tm_kx, tm_vx;
    vpp::AttnParams ap{};
    const RowPacking rp = row_packing(a);
    if (fam == Family::kGqa128) {
        const uint64_t dq[3] = {static_cast<uint64_t>(a->head_dim_qk), static_cast<uint64_t>(a->num_q_heads),
                                static_cast<uint64_t>(a->total_q)};
        const uint64_t sq[2] = {static_cast<uint64_t>(a->head_dim_qk) * 2,
                                static_cast<uint64_t>(a->head_dim_qk) * a->num_q_heads * 2};
        const uint32_t bq[3] = {64, static_cast<uint32_t>(rp.group), static_cast<uint32_t>(rp.tile_tokens)};
        // a packed item of one token has a box of its own: with the box of all the tokens that such an item may have, 256 decode rows
        // of 64/8 heads took 546 us instead of 538
        const uint32_t b1[3] = {64, static_cast<uint32_t>(rp.short_group), 1};
        const uint32_t bs[3] = {64, static_cast<uint32_t>(rp.short_group), static_cast<uint32_t>(rp.short_tokens)};
        if (!make_tmap(&tm_q, a->q, 3, dq, sq, bq) || !make_tmap(&tm_qs, a->q, 3, dq, sq, bs) || !make_tmap(&tm_q1, a->q, 3, dq, sq, b1))
            return fail(VPP_ERR_CUDA, "cuTensorMapEncodeTiled(q) failed");
        ap.exact_from = paged || B % vpp::kExactRows == 0 ? INT32_MAX : B / vpp::kExactRows * vpp::kExactRows;
        if (!make_kv_maps(a->k_cache, a->k_block_stride, a->k_token_stride, a->k_head_stride, B, n_blocks, a->num_kv_heads, box_rows, &tm_k,
                          &tm_kx, &ap.k_block_units, &ap.k_head_units, &ap.k_end, &ap.exact_from) ||
            !make_kv_maps(a->v_cache, a->v_block_stride, a->v_token_stride, a->v_head_stride, B, n_blocks, a->num_kv_heads, box_rows, &tm_v,
                          &tm_vx, &ap.v_block_units, &ap.v_head_units, &ap.v_end, &ap.exact_from))
            return fail(VPP_ERR_CUDA, "cuTensorMapEncodeTiled(k/v) failed");
    }
    CUtensorMap tm_q9, tm_qh9, tm_k93, tm_k92;  // attn_mla2.cuh
    const bool mla_pair = fam == Family::kMla576, mla_small_pages = mla_pair && box_rows < vpp::kMla2BoxRows;
    if (mla_pair) {
        const uint64_t dq[4] = {64, static_cast<uint64_t>(a->total_q), static_cast<uint64_t>(vpp::kMlaSlabs),
                                static_cast<uint64_t>(a->num_q_heads)};
        const uint64_t sq[3] = {static_cast<uint64_t>(a->head_dim_qk) * a->num_q_heads * 2, 128,
                                static_cast<uint64_t>(a->head_dim_qk) * 2};
        const uint32_t bq[4] = {vpp::kMla2BoxCols, vpp::kMla2BoxRows, static_cast<uint32_t>(vpp::kMlaSlabs), 1};   // all nine slabs in one copy
        const uint64_t tok = static_cast<uint64_t>(a->k_token_stride) * 2, blk = static_cast<uint64_t>(a->k_block_stride) * 2;
        const uint64_t slabs = static_cast<uint64_t>(vpp::kMlaSlabs), blocks = static_cast<uint64_t>(n_blocks);
        const uint32_t rows = static_cast<uint32_t>(box_rows);
        // pages under 64 tokens: the keys seen as 8-key groups; larger ones: 64 keys of three / two slabs
        const uint64_t d8[5] = {64, 8, slabs, static_cast<uint64_t>(B) / 8, blocks}, s8[4] = {tok, 128, 8 * tok, blk};
        const uint64_t d64[5] = {64, static_cast<uint64_t>(B), slabs, static_cast<uint64_t>(a->num_kv_heads), blocks};
        const uint64_t s64[4] = {tok, 128, static_cast<uint64_t>(a->k_head_stride) * 2, blk};
        auto kv_map = [&](CUtensorMap* m, uint32_t n_slabs) {
            const uint32_t b8[5] = {vpp::kMla2BoxCols, 8, n_slabs, rows / 8, 1}, b64[5] = {vpp::kMla2BoxCols, rows, n_slabs, 1, 1};
            return mla_small_pages ? make_tmap(m, a->k_cache, 5, d8, s8, b8) : make_tmap(m, a->k_cache, 5, d64, s64, b64);
        };
        if (!make_tmap(&tm_q9, a->q, 4, dq, sq, bq) || !kv_map(&tm_k93, vpp::kKG) || !kv_map(&tm_k92, vpp::kMla2VBoxSlabs))
            return fail(VPP_ERR_CUDA, "cuTensorMapEncodeTiled(mla pair) failed");
        // packed single-token items: 64 q-heads of one token as the rows of a CTA's Q tile
        const uint64_t dh[4] = {64, static_cast<uint64_t>(a->num_q_heads), static_cast<uint64_t>(vpp::kMlaSlabs),
                                static_cast<uint64_t>(a->total_q)};
        const uint64_t sh[3] = {static_cast<uint64_t>(a->head_dim_qk) * 2, 128,
                                static_cast<uint64_t>(a->head_dim_qk) * a->num_q_heads * 2};
        const uint32_t bh[4] = {64, 64, static_cast<uint32_t>(vpp::kMlaSlabs), 1};   // heads past num_q_heads read as zero
        if (!make_tmap(&tm_qh9, a->q, 4, dh, sh, bh)) return fail(VPP_ERR_CUDA, "cuTensorMapEncodeTiled(mla q heads) failed");
    }
    // ---- work decomposition ----
    int32_t* row_splits = reinterpret_cast<int32_t*>(ws + L.row_splits);
    vpp::PrepParams pp{};
    pp.prefix_len = a->prefix_len;
    pp.chunk_len = a->chunk_len;
    pp.block_table = a->block_table;
    pp.num_reqs = a->num_reqs;
    pp.total_q = a->total_q;
    pp.max_seq_len = a->max_seq_len;
    pp.max_blocks_per_req = a->max_blocks_per_req;
    pp.block_shift = paged ? ilog2(B) : 0;
    pp.num_blocks = n_blocks;
    pp.splits = L.splits;
    {
        const ItemCounts c = item_counts(a, fam);
        pp.balanced = L.balanced;
        pp.slots = c.slots;
        pp.unit_items = c.unit_items;
        pp.short_items = c.short_items;
        pp.ranges = ranges_of(c.slots, c.unit_items);
        pp.short_ranges = ranges_of(c.slots, c.short_items);
        const TileTimes t = tile_times(a, fam);
        pp.unit_us = static_cast<float>(t.unit_us);
        pp.short_us = static_cast<float>(t.short_us);
        pp.short_per_unit = static_cast<float>(t.short_us / t.unit_us);
        // (several requests, not all of them decode rows: the others have units of one kind, or of one length)
        pp.lead_items = fam == Family::kGqa128 && a->num_reqs > 1 && a->total_q > a->num_reqs ? 4 * c.slots : 0;
        pp.min_len = kMinLen;
        pp.min_short_len = kMinShortLen;
        pp.lead = fam == Family::kMla576 ? kMlaLead : kLead;
        pp.short_lead = fam == Family::kMla576 ? kMlaLead : kShortLead;
    }
    pp.max_units = L.max_units;
    pp.unit_rows = unit_rows_of(a, fam);
    pp.short_rows = fam == Family::kGqa128 ? rp.short_tokens : 1;   // (the box of a packed item's Q copy)
    // Item order: kv-head-major inside blocks of so many query rows.  Large blocks keep more CTAs on the same K/V pages, small
    // ones keep the order longest-first where units differ (no long one is started near the end): a first chunk of 4096 tokens
    // and 32 heads took 205 us with blocks of 4096 rows, 186 of 512 (and later 182, 180 of 256, 184 of 1024); 8192 tokens at prefix
    // 65536 16.46 ms with the large blocks against 16.58.
    pp.unit_block = 4096 / pp.unit_rows > 1 ? 4096 / pp.unit_rows : 1;
    pp.ragged_unit_block = 256 / pp.unit_rows > 1 ? 256 / pp.unit_rows : 1;
    pp.partial = range ? 1 : 0;
    pp.range_begin = range ? range->begin_tile : 0;
    pp.range_end = range ? range->end_tile : 0;
    pp.header = reinterpret_cast<vpp::WorkHeader*>(ws + L.header);
    pp.units = reinterpret_cast<vpp::WorkUnit*>(ws + L.units);
    pp.q_start = row_splits + a->total_q;
    pp.tile_start = pp.q_start + a->num_reqs + 1;
    {
        // a thread per request and per unit of an unsplit launch, as far as a block goes
        const long long units_ub = (a->total_q + pp.unit_rows - 1) / pp.unit_rows + a->num_reqs;
        unsigned threads = vpp::kPrepMinThreads;
        while (threads < vpp::kPrepMaxThreads && threads < units_ub) threads *= 2;
        // blocks that check the block table: one per 4 entries a thread can have in flight, at most kMaxCheckers
        long long checkers = 0;
        if (paged) {
            const long long entries = static_cast<long long>(a->num_reqs) * a->max_blocks_per_req;
            checkers = (entries + 4 * threads - 1) / (4 * threads);
            if (checkers > vpp::kMaxCheckers) checkers = vpp::kMaxCheckers;
        }
        const cudaError_t pe = launch(vpp::prep_kernel, static_cast<unsigned>(1 + checkers), threads,
                                      0, stream, pp);
        if (pe != cudaSuccess) return fail(VPP_ERR_CUDA, "work decomposition launch: %s", cudaGetErrorString(pe));
    }
    ++g_launches;

    // ---- attention ----
    ap.block_table = a->block_table;
    ap.max_blocks_per_req = a->max_blocks_per_req;
    ap.block_shift = pp.block_shift;
    ap.num_blocks = n_blocks;
    ap.num_q_heads = a->num_q_heads;
    ap.num_kv_heads = a->num_kv_heads;
    ap.total_q = a->total_q;
    ap.group = rp.group;
    ap.tile_tokens = rp.tile_tokens;
    ap.short_group = rp.short_group;
    ap.short_tokens = rp.short_tokens;
    ap.scale_log2e = a->softmax_scale * 1.4426950408889634f;
    ap.out = a->out;
    ap.lse = a->lse;
    // a partial launch writes "split 0" of the caller's buffers, which have the merge kernel's input layout
    ap.o_parts = range ? static_cast<float*>(a->out) : reinterpret_cast<float*>(ws + L.o_parts);
    ap.lse_parts = range ? a->lse : reinterpret_cast<float*>(ws + L.lse_parts);
    ap.header_ro = pp.header;
    ap.header = pp.header;
    ap.units = pp.units;
    ap.row_splits = L.splits > 1 ? row_splits : nullptr;
    ap.status = a->status;

    const int sms = sm_count_or_default();
    cudaError_t ce;
    if (mla_pair) {
        auto kern = mla_small_pages ? vpp::attn_mla2_kernel<true> : vpp::attn_mla2_kernel<false>;
        ce = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, vpp::kMla2SmemBytes);
        if (ce == cudaSuccess)
            ce = launch(kern, static_cast<unsigned>((sms / 2) * 2), vpp::kMla2Threads, vpp::kMla2SmemBytes, stream, tm_q9, tm_qh9, tm_k93,
                        tm_k92, ap, box_rows);
    } else {
        const bool quarters = L.splits == 1 && !range && shares_out_keys(a, rp.short_group);
        auto kern = !v_producer(a) ? vpp::attn128_ws_kernel<false, false> : quarters ? vpp::attn128_ws_kernel<true, true> : vpp::attn128_ws_kernel<true, false>;
        ce = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, vpp::kWsSmemBytes);
        if (ce == cudaSuccess)
            ce = launch(kern, static_cast<unsigned>(sms), vpp::kWsThreads, vpp::kWsSmemBytes, stream, tm_q, tm_qs, tm_q1, tm_k, tm_v, tm_kx,
                        tm_vx, ap, box_rows);
    }
    if (ce != cudaSuccess) return fail(VPP_ERR_CUDA, "attention kernel attributes: %s", cudaGetErrorString(ce));
    ++g_launches;

    // ---- merge of split partials ----
    if (L.splits > 1) {
        unsigned blocks = 1;
        const MergeKernel mk = pick_merge_kernel(L.splits, a->total_q, a->num_q_heads, a->head_dim_v, sms, &blocks);
        ce = launch(mk, blocks, vpp::kMergeThreads, 0, stream, ap.o_parts, ap.lse_parts, L.splits, a->total_q, a->num_q_heads,
                    a->head_dim_v, row_splits, pp.header, static_cast<__nv_bfloat16*>(a->out), a->lse);
        if (ce != cudaSuccess) return fail(VPP_ERR_CUDA, "merge launch: %s", cudaGetErrorString(ce));
        ++g_launches;
    }
    ce = cudaGetLastError();
    if (ce != cudaSuccess) return fail(VPP_ERR_CUDA, "kernel launch: %s", cudaGetErrorString(ce));
    return VPP_OK;
}
}  // namespace

vpp_status vpp_lse_merge(const float* o_parts, const float* lse_parts, int32_t num_splits, int32_t total_q,
                         int32_t num_q_heads, int32_t head_dim_v, void* out, float* lse, vpp_stream_t stream_) {
    g_err[0] = 0;
    if (num_splits <= 0 || total_q < 0 || num_q_heads <= 0 || head_dim_v <= 0)
        return fail(VPP_ERR_INVALID_ARG, "num_splits, num_q_heads, head_dim_v must be > 0 and total_q >= 0");
    if (head_dim_v % 8 != 0) return fail(VPP_ERR_UNSUPPORTED, "head_dim_v must be a multiple of 8");
    if (num_splits > vpp::kMergeMaxSplits) return fail(VPP_ERR_UNSUPPORTED, "at most %d splits", vpp::kMergeMaxSplits);
    if (total_q == 0) return VPP_OK;
    if (!o_parts || !lse_parts || !out) return fail(VPP_ERR_INVALID_ARG, "o_parts, lse_parts and out must be non-null");
    if ((reinterpret_cast<uintptr_t>(o_parts) | reinterpret_cast<uintptr_t>(out)) & 15u)
        return fail(VPP_ERR_INVALID_ARG, "o_parts and out must be 16-byte aligned");
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    unsigned blocks = 1;
    const MergeKernel mk = pick_merge_kernel(num_splits, total_q, num_q_heads, head_dim_v, sm_count_or_default(), &blocks);
    const cudaError_t ce = launch(mk, blocks, vpp::kMergeThreads, 0, stream, o_parts, lse_parts, num_splits, total_q, num_q_heads,
                                  head_dim_v, nullptr, nullptr, static_cast<__nv_bfloat16*>(out), lse);
    if (ce != cudaSuccess) return fail(VPP_ERR_CUDA, "merge launch: %s", cudaGetErrorString(ce));
    return VPP_OK;
}

vpp_status vpp_kv_append(const vpp_kv_append_args* a, vpp_stream_t stream_) {
    g_err[0] = 0;
    if (!a) return fail(VPP_ERR_INVALID_ARG, "args is null");
    if (a->num_reqs < 0 || a->total_q < 0 || a->num_kv_heads <= 0 || a->head_dim_qk <= 0 || a->head_dim_v <= 0)
        return fail(VPP_ERR_INVALID_ARG, "num_reqs, total_q >= 0 and num_kv_heads, head dims > 0 required");
    if (a->head_dim_qk % 8 || a->head_dim_v % 8) return fail(VPP_ERR_UNSUPPORTED, "head dims must be multiples of 8");
    if (a->num_reqs > vpp::kAppendMaxReqs) return fail(VPP_ERR_UNSUPPORTED, "at most %d requests", vpp::kAppendMaxReqs);
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (a->total_q == 0 || a->num_reqs == 0) return zero_status(a->status, stream);
    if (!a->k_new || !a->k_cache || !a->prefix_len || !a->chunk_len)
        return fail(VPP_ERR_INVALID_ARG, "k_new, k_cache, prefix_len and chunk_len must be non-null");
    if (a->v_new && !a->v_cache) return fail(VPP_ERR_INVALID_ARG, "v_new given without v_cache");
    int shift = 0;
    long long capacity = a->max_seq_len;
    if (a->block_table) {
        if (a->block_size < 1 || (a->block_size & (a->block_size - 1)))
            return fail(VPP_ERR_UNSUPPORTED, "block_size must be a power of two");
        if (a->max_blocks_per_req <= 0 || a->num_blocks <= 0)
            return fail(VPP_ERR_INVALID_ARG, "max_blocks_per_req and num_blocks must be > 0 with a block table");
        while ((1 << shift) < a->block_size) ++shift;
        capacity = static_cast<long long>(a->max_blocks_per_req) * a->block_size;
    } else if (a->max_seq_len <= 0) {
        return fail(VPP_ERR_INVALID_ARG, "max_seq_len must be > 0 for a contiguous cache");
    }
    const int64_t strides[6] = {a->k_block_stride, a->k_token_stride, a->k_head_stride,
                                a->v_block_stride, a->v_token_stride, a->v_head_stride};
    for (int i = 0; i < (a->v_new ? 6 : 3); ++i)
        if (strides[i] < 0 || strides[i] % 8) return fail(VPP_ERR_INVALID_ARG, "strides must be non-negative multiples of 8 elements");
    uintptr_t al = reinterpret_cast<uintptr_t>(a->k_new) | reinterpret_cast<uintptr_t>(a->k_cache);
    if (a->v_new) al |= reinterpret_cast<uintptr_t>(a->v_new) | reinterpret_cast<uintptr_t>(a->v_cache);
    if (al & 15u) return fail(VPP_ERR_INVALID_ARG, "k_new, v_new and the caches must be 16-byte aligned");

    vpp::AppendParams p{};
    p.k_new = static_cast<const uint4*>(a->k_new);
    p.v_new = static_cast<const uint4*>(a->v_new);
    p.k_cache = static_cast<uint8_t*>(a->k_cache);
    p.v_cache = static_cast<uint8_t*>(a->v_cache);
    p.k_block_stride = a->k_block_stride * 2; p.k_token_stride = a->k_token_stride * 2; p.k_head_stride = a->k_head_stride * 2;
    p.v_block_stride = a->v_block_stride * 2; p.v_token_stride = a->v_token_stride * 2; p.v_head_stride = a->v_head_stride * 2;
    p.block_table = a->block_table;
    p.prefix_len = a->prefix_len;
    p.chunk_len = a->chunk_len;
    p.num_reqs = a->num_reqs;
    p.max_blocks_per_req = a->max_blocks_per_req;
    p.block_shift = shift;
    p.num_blocks = a->num_blocks;
    p.capacity = capacity;
    p.total_q = a->total_q;
    p.num_kv_heads = a->num_kv_heads;
    p.k_vecs = a->head_dim_qk / 8;
    p.v_vecs = a->v_new ? a->head_dim_v / 8 : 0;
    p.status = a->status;
    const int vecs = p.num_kv_heads * (p.k_vecs + p.v_vecs), warps_per_block = vpp::kAppendThreads / 32;
    const long long tasks = static_cast<long long>(a->total_q) * ((vecs + vpp::kAppendPiece - 1) / vpp::kAppendPiece);
    long long blocks = (tasks + warps_per_block - 1) / warps_per_block;
    const long long cap = 16ll * sm_count_or_default();
    if (blocks > cap) blocks = cap;
    const size_t smem = sizeof(int32_t) * (static_cast<size_t>(a->num_reqs) + 1);
    const int copy_blocks = static_cast<int>(blocks);
    const cudaError_t ce = launch(vpp::kv_append_kernel, static_cast<unsigned>(copy_blocks + (a->status ? 1 : 0)), vpp::kAppendThreads, smem,
                                  stream, p, copy_blocks);
    if (ce != cudaSuccess) return fail(VPP_ERR_CUDA, "append launch: %s", cudaGetErrorString(ce));
    return VPP_OK;
}

namespace {
// Workspace of a sparse launch: the token table, then -- for launches of so few tokens that their lists are cut into
// parts -- the number of parts of every token and the partial results.
struct SparseLayout {
    size_t row_splits, o_parts, lse_parts, total, base;   // base: without the partials
    int max_splits;
};
constexpr int kSparseMaxSplits = 8;
SparseLayout sparse_layout(int32_t total_q) {
    const size_t T = static_cast<size_t>(total_q > 0 ? total_q : 0);
    SparseLayout L{};
    L.base = 256 + sizeof(int2) * T;
    L.total = L.base;
    // A list is cut only where a whole number of parts, two or more, keeps every item in the one wave of SM pairs: 16 tokens
    // with 2048-entry lists ran 54 us on 16 of 74 pairs, cut in four they run on 64 pairs.  More tokens fill the pairs
    // by themselves well enough that a second wave of shorter items costs what it saves.
    const int pairs = sm_count_or_default() / 2;
    L.max_splits = T > 0 && pairs >= 2 * static_cast<int>(T) ? pairs / static_cast<int>(T) : 1;
    if (L.max_splits > kSparseMaxSplits) L.max_splits = kSparseMaxSplits;
    if (L.max_splits > 1) {
        const size_t rows = T * L.max_splits * 2 * vpp::kMla2Rows;
        L.row_splits = align_up(L.base, 256);
        L.o_parts = align_up(L.row_splits + sizeof(int32_t) * T, 256);
        L.lse_parts = align_up(L.o_parts + sizeof(float) * rows * vpp::kMlaDv, 256);
        L.total = L.lse_parts + sizeof(float) * rows;
    }
    return L;
}
}  // namespace

size_t vpp_sparse_attn_workspace_size(int32_t total_q) { return sparse_layout(total_q).total; }

vpp_status vpp_sparse_mla_fwd(const vpp_sparse_attn_args* a, vpp_stream_t stream_) {
    g_err[0] = 0;
    if (!a) return fail(VPP_ERR_INVALID_ARG, "args is null");
    if (a->num_reqs < 0 || a->total_q < 0) return fail(VPP_ERR_INVALID_ARG, "num_reqs and total_q must be >= 0");
    if (a->num_q_heads <= 0 || a->num_q_heads > 2 * vpp::kMla2Rows)
        return fail(VPP_ERR_UNSUPPORTED, "num_q_heads must be in 1..%d", 2 * vpp::kMla2Rows);
    if (a->topk < 1) return fail(VPP_ERR_INVALID_ARG, "topk must be >= 1");
    if (!(a->softmax_scale > 0.f) || !std::isfinite(a->softmax_scale))
        return fail(VPP_ERR_INVALID_ARG, "softmax_scale must be positive and finite");
    if (a->num_reqs > vpp::kDsaMaxReqs) return fail(VPP_ERR_UNSUPPORTED, "at most %d requests", vpp::kDsaMaxReqs);
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (a->total_q == 0 || a->num_reqs == 0) return zero_status(a->status, stream);
    if (!a->q || !a->kv_cache || !a->indices || !a->prefix_len || !a->chunk_len || !a->out)
        return fail(VPP_ERR_INVALID_ARG, "q, kv_cache, indices, prefix_len, chunk_len and out must be non-null");
    if ((reinterpret_cast<uintptr_t>(a->q) | reinterpret_cast<uintptr_t>(a->kv_cache) | reinterpret_cast<uintptr_t>(a->out) |
         reinterpret_cast<uintptr_t>(a->workspace)) & 15u)
        return fail(VPP_ERR_INVALID_ARG, "q, kv_cache, out and workspace must be 16-byte aligned");
    if (a->kv_row_stride < vpp::kMlaDqk || a->kv_row_stride % 8)
        return fail(VPP_ERR_INVALID_ARG, "kv_row_stride must be a multiple of 8 elements and at least %d", vpp::kMlaDqk);
    const SparseLayout L = sparse_layout(a->total_q);
    if (!a->workspace || a->workspace_bytes < L.base)
        return fail(VPP_ERR_WORKSPACE, "workspace too small: %zu bytes needed", L.total);
    // parts of at least two tiles; a workspace that holds the token table only runs unsplit
    const int list_tiles = (a->topk + vpp::kTileN - 1) / vpp::kTileN;
    int splits = a->workspace_bytes < L.total ? 1 : L.max_splits;
    if (splits > list_tiles / 2) splits = list_tiles / 2;
    if (splits < 1) splits = 1;
    int shift = 0;
    long long capacity, num_rows;
    if (a->block_table) {
        if (a->block_size < 1 || (a->block_size & (a->block_size - 1)))
            return fail(VPP_ERR_UNSUPPORTED, "block_size must be a power of two");
        if (a->max_blocks_per_req <= 0 || a->num_blocks <= 0)
            return fail(VPP_ERR_INVALID_ARG, "max_blocks_per_req and num_blocks must be > 0 with a block table");
        while ((1 << shift) < a->block_size) ++shift;
        capacity = static_cast<long long>(a->max_blocks_per_req) * a->block_size;
        num_rows = static_cast<long long>(a->num_blocks) * a->block_size;
    } else {
        if (a->max_seq_len <= 0) return fail(VPP_ERR_INVALID_ARG, "max_seq_len must be > 0 for a contiguous cache");
        capacity = a->max_seq_len;
        num_rows = static_cast<long long>(a->num_reqs) * a->max_seq_len;
    }
    if (num_rows >= (1ll << 31)) return fail(VPP_ERR_UNSUPPORTED, "the cache must have fewer than 2^31 rows");

    CUtensorMap tm_qh, tm_rows;
    {
        const uint64_t dh[4] = {64, static_cast<uint64_t>(a->num_q_heads), static_cast<uint64_t>(vpp::kMlaSlabs),
                                static_cast<uint64_t>(a->total_q)};
        const uint64_t sh[3] = {static_cast<uint64_t>(vpp::kMlaDqk) * 2, 128,
                                static_cast<uint64_t>(vpp::kMlaDqk) * a->num_q_heads * 2};
        const uint32_t bh[4] = {64, 64, static_cast<uint32_t>(vpp::kMlaSlabs), 1};   // heads past num_q_heads read as zero
        // gather form: a box of one row; each copy names four rows
        const uint64_t dr[2] = {static_cast<uint64_t>(vpp::kMlaDqk), static_cast<uint64_t>(num_rows)};
        const uint64_t sr[1] = {static_cast<uint64_t>(a->kv_row_stride) * 2};
        const uint32_t br[2] = {64, 1};
        if (!make_tmap(&tm_qh, a->q, 4, dh, sh, bh) || !make_tmap(&tm_rows, a->kv_cache, 2, dr, sr, br))
            return fail(VPP_ERR_CUDA, "cuTensorMapEncodeTiled(sparse mla) failed");
    }
    uint8_t* ws = static_cast<uint8_t*>(a->workspace);
    int2* tok = reinterpret_cast<int2*>(ws);
    int32_t* row_splits = reinterpret_cast<int32_t*>(ws + L.row_splits);
    const int sms = sm_count_or_default();
    {
        long long blocks = (static_cast<long long>(a->total_q) + vpp::kDsaPrepThreads - 1) / vpp::kDsaPrepThreads;
        if (blocks > 4ll * sms) blocks = 4ll * sms;
        const size_t smem = sizeof(int32_t) * (static_cast<size_t>(a->num_reqs) + 1);
        const cudaError_t te = launch(vpp::dsa_tokens_kernel, static_cast<unsigned>(blocks), vpp::kDsaPrepThreads, smem, stream, a->prefix_len,
                                      a->chunk_len, a->num_reqs, a->total_q, capacity, splits, tok, row_splits, a->status);
        if (te != cudaSuccess) return fail(VPP_ERR_CUDA, "token table launch: %s", cudaGetErrorString(te));
    }
    vpp::DsaParams p{};
    p.indices = a->indices;
    p.topk = a->topk;
    p.tok = tok;
    p.block_table = a->block_table;
    p.max_blocks_per_req = a->max_blocks_per_req;
    p.block_shift = shift;
    p.num_blocks = a->num_blocks;
    p.max_seq_len = a->max_seq_len;
    p.num_q_heads = a->num_q_heads;
    p.total_q = a->total_q;
    p.scale_log2e = a->softmax_scale * 1.4426950408889634f;
    p.splits = splits;
    p.out = a->out;
    p.lse = a->lse;
    p.o_parts = reinterpret_cast<float*>(ws + L.o_parts);
    p.lse_parts = reinterpret_cast<float*>(ws + L.lse_parts);
    p.status = a->status;
    auto kern = splits > 1 ? vpp::dsa_attn_kernel<true> : vpp::dsa_attn_kernel<false>;
    cudaError_t ce = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, vpp::kMla2SmemBytes);
    if (ce == cudaSuccess) {
        long long pairs = sms / 2, items = static_cast<long long>(a->total_q) * splits;
        if (pairs > items) pairs = items;
        ce = launch(kern, static_cast<unsigned>(pairs * 2), vpp::kDsaThreads, vpp::kMla2SmemBytes, stream, tm_qh, tm_rows, p);
    }
    if (ce != cudaSuccess) return fail(VPP_ERR_CUDA, "sparse attention launch: %s", cudaGetErrorString(ce));
    g_launches = 2;
    if (splits > 1) {
        unsigned blocks = 1;
        const MergeKernel mk = pick_merge_kernel(splits, a->total_q, a->num_q_heads, vpp::kMlaDv, sms, &blocks);
        ce = launch(mk, blocks, vpp::kMergeThreads, 0, stream, p.o_parts, p.lse_parts, splits, a->total_q, a->num_q_heads, vpp::kMlaDv,
                    row_splits, nullptr, static_cast<__nv_bfloat16*>(a->out), a->lse);
        if (ce != cudaSuccess) return fail(VPP_ERR_CUDA, "merge launch: %s", cudaGetErrorString(ce));
        ++g_launches;
    }
    return VPP_OK;
}


void vpp_tensor_map_cache_stats(int64_t* lookups, int64_t* encodes) {
    int64_t l = 0, e = 0;
    g_tmaps.stats(&l, &e);
    if (lookups) *lookups = l;
    if (encodes) *encodes = e;
}

int32_t vpp_test_tensor_map_cache(int32_t repeats) {
    // the cache logic with a stand-in for the driver's encoder (pure host code)
    static TmapCache cache;
    auto fake = +[](CUtensorMap* m, const TmapKey& k) {
        std::memset(m, 0, sizeof *m);
        std::memcpy(m, &k, sizeof k < sizeof *m ? sizeof k : sizeof *m);
        return true;
    };
    const uint64_t d1[3] = {128, 8, 1000}, s1[2] = {256, 2048}, d2[3] = {128, 8, 1001};
    const uint32_t b1[3] = {64, 1, 128};
    static const char anchor[64] = {0};
    int64_t l0, e0, l1, e1;
    cache.stats(&l0, &e0);
    for (int i = 0; i < repeats; ++i) {
        CUtensorMap m, ref;
        const TmapKey k = make_key(anchor, 3, d1, s1, b1);
        if (!cache.get(k, fake, &m)) return -1;
        fake(&ref, k);
        if (std::memcmp(&m, &ref, sizeof m) != 0) return -2;     // a hit must return what the encoder produced
    }
    CUtensorMap m;
    if (!cache.get(make_key(anchor, 3, d2, s1, b1), fake, &m)) return -1;    // another extent: another map
    if (!cache.get(make_key(anchor + 16, 3, d1, s1, b1), fake, &m)) return -1;   // another base: another map
    cache.stats(&l1, &e1);
    if (l1 - l0 != repeats + 2) return -3;
    return static_cast<int32_t>(e1 - e0);
}

vpp_status vpp_test_bounded_wait(int32_t* status, int64_t limit_cycles, vpp_stream_t stream_) {
    g_err[0] = 0;
    if (!status || limit_cycles <= 0 || limit_cycles > (1ll << 31))
        return fail(VPP_ERR_INVALID_ARG, "status must be non-null and limit_cycles in (0, 2^31]");
    vpp::bounded_wait_test_kernel<<<1, 64, 0, static_cast<cudaStream_t>(stream_)>>>(status, limit_cycles);
    const cudaError_t ce = cudaGetLastError();
    if (ce != cudaSuccess) return fail(VPP_ERR_CUDA, "test kernel launch: %s", cudaGetErrorString(ce));
    return VPP_OK;
}

}  // extern "C"

vpp_status vpp::chunk_attn_fwd_within(const vpp_chunk_attn_args* a, vpp_stream_t stream_, size_t limit) {
    return run_chunk_attn(a, stream_, nullptr, limit);
}
