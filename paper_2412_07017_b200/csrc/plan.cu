// Host planner: validates one step's batch, tiles it into (unit, KV chunk) work items, balances the
// items over persistent CTAs and uploads the packed plan with one asynchronous copy.
//
// The step being planned is the "next decoding step" after the interrupt manager has appended its
// queued interrupt tokens (paper Section 5.3): q_len 1 = decode, > 1 = interrupt span, 0 = a
// sequence paused by a trap (Section 3.2).  All work here is integer work on the host.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <climits>
#include <cstring>
#include <vector>

#include "asynclm.h"
#include "kernels.h"
#include "plan_internal.h"

namespace asynclm {

static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

int resolve_num_sms(const asynclm_plan_options* opts, bool need_device, int* out) {
    if (opts && opts->num_sms > 0) { *out = opts->num_sms; return ASYNCLM_OK; }
    if (!need_device) { *out = 148; return ASYNCLM_OK; }
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return ASYNCLM_ERR_CUDA;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return ASYNCLM_ERR_CUDA;
    *out = n;
    return ASYNCLM_OK;
}

static int check_shape(const asynclm_shape* s) {
    if (!s) return ASYNCLM_ERR_INVALID_ARG;
    if (s->num_q_heads <= 0 || s->num_kv_heads <= 0 || s->num_pages < 0 || s->reserved != 0)
        return ASYNCLM_ERR_INVALID_ARG;
    if (s->num_q_heads % s->num_kv_heads != 0) return ASYNCLM_ERR_UNSUPPORTED_SHAPE;
    const int g = s->num_q_heads / s->num_kv_heads;
    if (!(g == 1 || g == 2 || g == 4 || g == 8)) return ASYNCLM_ERR_UNSUPPORTED_SHAPE;
    if (!(s->head_dim == 64 || s->head_dim == 128)) return ASYNCLM_ERR_UNSUPPORTED_SHAPE;
    if (s->page_size != kPage) return ASYNCLM_ERR_UNSUPPORTED_SHAPE;
    return ASYNCLM_OK;
}

// Tokens of a span that one tensor-core work item covers: two row tiles of 128 (token, head) rows.
int tensor_tile_tokens(int group) { return 256 / group; }

// Rows (G * q_len) from which a (sequence, kv head) goes to the span body (tcgen05).  Below it the
// warp body reads the keys once per 8 (token, head) columns, which costs less than a span item's
// start-up; decode rows (G rows) always stay on the warp body, which runs at the memory rate for
// every supported G.  At head_dim 64 a re-read of the keys costs half as much.
static int default_tensor_min_rows(int head_dim) { return head_dim == 64 ? 64 : 32; }

// Sizes of the sections of the packed blob (identical offsets on host and device).
struct BlobLayout {
    size_t off_q_indptr, off_kv_len, off_page_indptr, off_page_indices, off_row_seq, off_row_slot, off_units,
        off_items, off_works, off_heads, off_cta_cuda, off_cta_tensor, off_split, off_merge, off_status,
        off_arrivals, blob_bytes;
};

static BlobLayout layout_blob(int batch, int total_q, int64_t total_pages, int64_t n_units,
                              int64_t n_items, int ctas_cuda, int ctas_tensor, int64_t n_split,
                              int64_t n_merge_blocks) {
    BlobLayout L{};
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t at = o; o = align_up(o + bytes, 256); return at; };
    L.off_status = take(256);
    L.off_q_indptr = take(sizeof(int32_t) * (size_t)(batch + 1));
    L.off_kv_len = take(sizeof(int32_t) * (size_t)std::max(batch, 1));
    L.off_page_indptr = take(sizeof(int32_t) * (size_t)(batch + 1));
    L.off_page_indices = take(sizeof(int32_t) * (size_t)std::max<int64_t>(total_pages, 1));
    L.off_row_seq = take(sizeof(int32_t) * (size_t)std::max(total_q, 1));
    L.off_row_slot = take(sizeof(int64_t) * (size_t)std::max(total_q, 1));
    L.off_units = take(sizeof(Unit) * (size_t)std::max<int64_t>(n_units, 1));
    L.off_items = take(sizeof(Item) * (size_t)std::max<int64_t>(n_items, 1));
    L.off_works = take(sizeof(Work) * (size_t)std::max<int64_t>(n_items, 1));
    L.off_heads = take(sizeof(int32_t) * kHeadWords * (size_t)std::max(ctas_cuda, ctas_tensor));
    L.off_cta_cuda = take(sizeof(int32_t) * (size_t)(ctas_cuda + 1));
    L.off_cta_tensor = take(sizeof(int32_t) * (size_t)(ctas_tensor + 1));
    L.off_split = take(sizeof(int32_t) * (size_t)std::max<int64_t>(n_split, 1));
    L.off_merge = take(sizeof(int32_t) * (size_t)std::max<int64_t>(n_merge_blocks, 1));
    L.off_arrivals = take(sizeof(int32_t) * (size_t)std::max<int64_t>(n_units, 1));
    L.blob_bytes = o;
    return L;
}

static size_t partial_bytes(int64_t rows, int group, int head_dim) {
    return align_up((size_t)rows * (size_t)group * (size_t)head_dim * sizeof(float), 256) +
           align_up((size_t)rows * (size_t)group * sizeof(float), 256);
}

// Warp-body units: a sixth of the work is cut into short chunks for the end of the queue, about
// kTailChunksPerCta per CTA and never shorter than kMinChunkTiles tiles (see deal_dynamic), unless the shortest
// units, which stand at the end of the queue anyway, are short enough to even out the CTAs' finishing times: those
// that make up a sixth of the work are no longer than kShortUnitShare of a CTA's share.  Cutting costs item boundaries,
// partial rows and merges, and a CTA that is late streams faster once others have left the memory to it (which takes
// kSaturatingCtas to begin with).  (us of attention a layer, cut | not: 64 decoding sequences of 1-3 K keys 85.3 | 83.4, 256 of
// 0.3-2 K with 5 spans 192 | 186, 32 of 0.5-4 K with 8 spans 62.1 | 60.0, 40 of 64/8 heads with 8 123 | 114; the longest of the
// shortest sixth has 0.05 to 0.6 of a share there.  Near a share, cutting wins: 19 of 3 K keys 45.4 | 50.)
constexpr int kTailChunksPerCta = 2;
constexpr int kMinChunkTiles = 4;
constexpr int kShortUnitShareNum = 2, kShortUnitShareDen = 3;
constexpr int kSaturatingCtas = 74;      // stream 6.2 TB/s of pages, 148 6.6, 37 4.4
// That alone leaves the last wave nearly empty where the units are of about one length and not a multiple of the CTAs, so
// an uncut queue is followed to its end (queue_ns) and cut after all if it ends later than the cut one by more than cutting
// costs.  (us of attention a layer, cut | not | chosen: sequences of one length, 38 of 4 K keys 104 | 117 | cut, 48 135 | 124 | not,
// 57 of 6 K 208 | 224 | cut, at head_dim 64 38 of 6 K 85.6 | 108 | cut, 74 156 | 145 | not.  Of 290 batches, half of them of one
// length or nearly, the chosen form takes 0.2 % longer than the faster one on average and 6 % at most, the rule above
// alone 2.1 % and 26 %.)
struct StreamCost {
    int64_t tile_ns, least_tile_ns;      // 128 keys on a CTA while kStreamCtas stream, and while few do
    int64_t cut_ns;                      // what a cut sixth costs at the end: more boundaries, partial rows, merges
};
// (Those of head_dim 64 were taken with a warp body that had one page of a stage for each warp; 640 and 570 are what it takes with two.
// 11 batches of one length and 11 others come out the same with either.)
constexpr int kStreamCtas = 148;
constexpr StreamCost stream_cost(int head_dim) {
    return head_dim == 64 ? StreamCost{700, 630, 2500} : StreamCost{1390, 834, 5000};
}
// The other units are cut into pieces of at most kBulkTiles tiles (50-90 us) or an eighth of a CTA's share: with
// contexts of 10^5 tokens, pieces of two fifths of the step, which used to be the only limit, left some CTAs on
// a last piece of half a millisecond.  (8 sequences of 32-131 K tokens, two 256-token spans: 1083 us of attention
// a layer without this limit, 910-970 with it, run to run; 32 and 128 tiles the same; 128 sequences of 64 / 8
// heads 489 at 32 tiles, 480 at 64 and 128.)
constexpr int kBulkTiles = 64;
// Span units of two row tiles are cut by keys instead of divided by rows where the pieces are at least this
// long, because the divided halves each stream the keys: 128 keys take a CTA 2.4 us for two row tiles and
// 1.55 us for one, when all CTAs stream.  (8 sequences of 32-131 K tokens, two 256-token spans: 1065-1096 us of
// attention a layer with divided units, 910-970 with as many cut ones as the fixed array has room for.)  Below,
// the partial rows and their merge cost more than they save (32 sequences of up to 4 K tokens, 8 spans: 62.5 us
// divided, 68.7 cut).
constexpr int kLongPieceTiles = 64;
// Tokens of one warp-body unit: its MMAs have 8 (token, head) columns.
static int warp_unit_tokens(int group) { return 8 / group; }

// Upper bounds on what the automatic policy produces, for C CTAs and W tiles of warp-body work in all.
//   Warp body, only units longer than 1.5 pieces are cut, into ceil(t / piece) <= 1.5 t / piece pieces (the
// worst is just over two).  A long piece is at least min(2/5 of a CTA's share, max(kBulkTiles, an eighth of
// it)) >= W / (8 C) tiles: at most 12 C pieces.  A short one is at least W / (12 C) less the rounding, and
// never below kMinChunkTiles, so below 1.25 times as many: 15 C pieces if one unit holds all the work; a unit
// goes to the short ones only until they hold a sixth of W, so all but the last add at most 1.5 * 15 C / 6.
// The worst mixture, a sixth of W in small units and the rest in the last one, stays below 17 C.
//   Span body: a unit is cut only if it is longer than what a fresh CTA takes, into pieces longer than half of
// that (or of one tile, which each need a CTA of their own), so a CTA holds fewer than three.
//   A unit that is not cut is one item, and a divided unit is two; only cut units hold partial rows.
static int64_t auto_item_bound(int64_t units, int ctas) { return 2 * units + (int64_t)20 * ctas; }
static int64_t auto_partial_row_bound(int ctas, int group) {
    return (int64_t)20 * ctas * warp_unit_tokens(group) + (int64_t)3 * ctas * tensor_tile_tokens(group);
}

}  // namespace asynclm

using namespace asynclm;

extern "C" int asynclm_plan_workspace_size(const asynclm_shape* shape,
                                           const asynclm_plan_options* opts, int32_t max_batch,
                                           int32_t max_total_q, int64_t max_total_pages,
                                           size_t* host_bytes, size_t* device_bytes) {
    int rc = check_shape(shape);
    if (rc != ASYNCLM_OK) return rc;
    if (max_batch < 0 || max_total_q < 0 || max_total_pages < 0 || !host_bytes || !device_bytes)
        return ASYNCLM_ERR_INVALID_ARG;
    int n_sms = 0;
    if (resolve_num_sms(opts, true, &n_sms) != ASYNCLM_OK) n_sms = 160;
    const int G = shape->num_q_heads / shape->num_kv_heads;
    const int ctas_cuda = n_sms * kCudaSlotsPerSm;
    const int ctas_tensor = n_sms;
    const int64_t max_units = (int64_t)max_total_q * shape->num_kv_heads;
    int64_t max_items, max_partial_rows;
    if (opts && opts->kv_chunk_tokens > 0) {
        // fixed chunk length: every unit may be cut into ceil(n/chunk) pieces
        const int64_t per_unit = (max_total_pages * kPage) / opts->kv_chunk_tokens + 1;
        max_items = max_units * per_unit;
        max_partial_rows = max_items;   // ntok tokens per unit are already counted in max_units
    } else {
        max_items = auto_item_bound(max_units, ctas_cuda);
        max_partial_rows = auto_partial_row_bound(ctas_cuda, G);      // only cut units hold partial rows
    }
    BlobLayout L = layout_blob(max_batch, max_total_q, max_total_pages, max_units, max_items,
                               ctas_cuda, ctas_tensor, max_units,
                               (int64_t)max_total_q * shape->num_q_heads / 4 + max_units);
    *host_bytes = align_up(sizeof(asynclm_plan_s), 256) + L.blob_bytes +
                  align_up(sizeof(int32_t) * (size_t)std::max<int64_t>(max_items, 1), 256);
    *device_bytes = L.blob_bytes + partial_bytes(max_partial_rows, G, shape->head_dim);
    return ASYNCLM_OK;
}

namespace {

struct UnitBuild {
    Unit u;
    int path;
    int64_t n_keys;   // keys visible to the unit's last token
};

// Cuts the units of one path into items and deals them to `n_ctas` persistent CTAs.
// fixed_chunk > 0: equal chunks of that many tokens, then a contiguous equal-cost partition of the
// item sequence.  Otherwise: the concatenated tile sequence of all units is cut into n_ctas nearly
// equal contiguous ranges (a unit is split only where a range boundary falls inside it).
void cut_and_deal(const std::vector<int>& unit_ids, std::vector<UnitBuild>& units, int fixed_chunk,
                  int n_ctas, int item_overhead_tiles, std::vector<Item>& items,
                  std::vector<int32_t>& cta_indptr, std::vector<int32_t>& item_cta) {
    const size_t first_item = items.size();
    cta_indptr.assign((size_t)n_ctas + 1, (int32_t)first_item);
    if (unit_ids.empty() || n_ctas <= 0) return;
    auto tiles_of = [](int64_t tokens) { return (tokens + kKvTile - 1) / kKvTile; };
    if (fixed_chunk > 0) {
        for (int id : unit_ids) {
            UnitBuild& ub = units[id];
            int c = 0;
            for (int64_t k0 = 0; k0 < ub.n_keys; k0 += fixed_chunk, ++c) {
                Item it{id, (int32_t)k0, (int32_t)std::min<int64_t>(ub.n_keys, k0 + fixed_chunk), c};
                items.push_back(it);
            }
            ub.u.n_chunks = c;
        }
        int64_t total = 0;
        for (size_t i = first_item; i < items.size(); ++i)
            total += item_overhead_tiles + tiles_of(items[i].kv1 - items[i].kv0);
        // contiguous partition: an item goes to the CTA in whose share of the total its midpoint falls
        int64_t cum = 0;
        for (size_t i = first_item; i < items.size(); ++i) {
            const int64_t c = item_overhead_tiles + tiles_of(items[i].kv1 - items[i].kv0);
            const int64_t cta = std::min<int64_t>(n_ctas - 1, ((2 * cum + c) * n_ctas) / (2 * total));
            item_cta.push_back((int32_t)cta);
            cum += c;
        }
    } else {
        int64_t total_tiles = 0;
        for (int id : unit_ids) total_tiles += tiles_of(units[id].n_keys);
        const int64_t total_cost =
            total_tiles + (int64_t)item_overhead_tiles * ((int64_t)unit_ids.size() + n_ctas);
        const int64_t quota = std::max<int64_t>(1 + item_overhead_tiles,
                                                (total_cost + n_ctas - 1) / n_ctas);
        int cta = 0;
        int64_t budget = quota;
        for (int id : unit_ids) {
            UnitBuild& ub = units[id];
            int64_t tiles_left = tiles_of(ub.n_keys);
            int64_t k0 = 0;
            int c = 0;
            while (tiles_left > 0) {
                if (budget <= item_overhead_tiles && cta + 1 < n_ctas) {
                    ++cta;
                    budget = quota;
                }
                int64_t take = cta + 1 < n_ctas
                                   ? std::min<int64_t>(tiles_left, std::max<int64_t>(1, budget - item_overhead_tiles))
                                   : tiles_left;
                const int64_t k1 = std::min<int64_t>(ub.n_keys, k0 + take * kKvTile);
                items.push_back(Item{id, (int32_t)k0, (int32_t)k1, c});
                item_cta.push_back(cta);
                budget -= item_overhead_tiles + take;
                tiles_left -= take;
                k0 = k1;
                ++c;
            }
            ub.u.n_chunks = c;
        }
    }
    // items were emitted in CTA order; build the CSR
    std::vector<int32_t> count((size_t)n_ctas, 0);
    for (size_t i = first_item; i < items.size(); ++i) count[(size_t)item_cta[i]]++;
    int32_t at = (int32_t)first_item;
    for (int k = 0; k < n_ctas; ++k) {
        cta_indptr[(size_t)k] = at;
        at += count[(size_t)k];
    }
    cta_indptr[(size_t)n_ctas] = at;
}

// Costs of the attention kernels on B200 as the packing sees them, in nanoseconds, used only to size the span
// CTAs.  At head_dim 128 they are those of an earlier form of the span body with 128-key tiles, which the margins
// below were chosen with; the present body takes, per 128 keys with one | two row tiles, 0.9 | 1.55 us on a CTA
// alone and 1.4 | 2.4 on all 148, where memory and power bound it (with 900 | 1800 here, 48 sequences with 6 spans took
// 120 us instead of 112).  At head_dim 64 it takes 0.93 | 1.55 alone and 1.0 | 1.9 on all.
struct PathCost {
    int gran;            // tokens per tile of the path (cuts fall on multiples of it)
    int64_t tile_ns;     // one tile in steady state
    int64_t item_ns;     // starting and finishing an item (pipeline fill and drain, merge, write)
    int64_t phase_ns;    // first item of the path on a CTA (descriptor chain, first loads)
};
// Span body: a KV tile of 128 keys against one row tile, an item, the body's start on a CTA.
constexpr PathCost kTensorCost{128, 1170, 8000, 11800};
constexpr int64_t kTensorDualTileNs = 2435;   // a KV tile of an item with two row tiles (more than 128 rows)
// When every unit runs on the span body all SMs stream K/V tiles at once and the tile time is set by
// the memory system (64 KB per tile and SM); the producers run ahead across item boundaries.
constexpr PathCost kTensorOnlyCost{128, 1543, 8000, 2400};
constexpr int64_t kTensorOnlyDualTileNs = 3126;
// Warp body: 64 KB per 128-key tile (32 KB at head_dim 64).  It is bound by memory, so its tile time depends on
// how many SMs stream at once: 1.39 us when all 148 do, 1.05 us (62 KB/us) when half of them run span tiles,
// which draw some bandwidth too, 0.79 us for 74 and 0.73 for one by themselves; at head_dim 64 0.64, 0.58 for 37 to
// 100 and 0.53 for one.  The model takes the second figure for both.  (At head_dim 64 900 here gives layers of 0.88 to 1.08 of the time
// with 1050, 750 of 0.90 to 1.11, without a rule to tell which batch gains.)
constexpr PathCost kWarpCost{128, 1050, 400, 2000};
// No step ends before its bytes have crossed the memory bus: K/V pages stream at about 6 bytes per
// nanosecond on this access pattern (4 KB runs through a shuffled page table), after about 3 us in
// which the CTAs start.  Without this floor the model would spread the span units over so many CTAs
// that too few were left streaming to keep the memory busy (one SM streams 60-75 KB/us at most).
// Each (sequence, kv head) counts once: the row tiles of a long span re-read it, mostly from L2.
constexpr int64_t kDramBytesPerUs = 6000000;
// A span CTA that finishes early joins the queue; one that finishes late delays the whole step, so the span CTAs
// are filled to the load limit divided by this margin (in 1/64).  The costs above are head_dim 128's of a
// slower body, which leaves a margin by itself.  Attention of a layer in us at 66 | 68 | 72 | 88, head_dim 128: 32
// sequences with 8 spans 60.0 | 61.5 | 61.4 | 61.6, 64 with 12 73.3 | 73.1 | 72.8 | 79.2, 40 of 16/8 heads with 10 65.1 | 64.7 |
// 64.5 | 69.2, 40 of 64/8 heads with 8 114 | 121 | 120 | 122, 128 of 64/8 heads with 13 492 | 489 | 488 | 479 (469 | 465 | 463 |
// 463 at best: power); at head_dim 64, 64 | 72 | 76 | 88: 32 with 8 50.0 | 49.8 | 49.4 | 55.4, 64 with 16 83.3 | 81.1 | 80.7 |
// 80.2, 64 of 8/8 heads with 8 103 | 103 | 104 | 106, 100 of 8/2 heads with 20 48.1 | 50.4 | 50.7 | 55.1.
constexpr int64_t span_margin64(int head_dim) { return head_dim == 64 ? 72 : 66; }
// The same, for the decision to divide a unit by rows.  At head_dim 128 it lies above the span CTAs' margin, so that a unit
// between the two limits is divided although it would fit a CTA whole.  Both ways measured: with 66 here 28 of 1632 random
// batches come out otherwise, attention of a layer 0.80 to 1.18 of the time with 72, 1.002 on average.
constexpr int64_t kDivideMargin64 = 72;
// Share (in 1/64) of the queue that the CTAs without span work must be able to stream by themselves.
constexpr int64_t kStreamShare64 = 58;
constexpr int64_t kStartNs = 3000;

// Sorts `v` by falling key, equal keys in the order they stand in.  What stands here comes in runs of equal keys (the
// kv heads of a sequence, a unit's pieces), so the runs are sorted and written out again.
template <typename T, typename Key>
void sort_falling(std::vector<T>& v, Key key) {
    struct Run { int64_t key; uint32_t at, count; };
    std::vector<Run> runs;
    runs.reserve(v.size() / 4 + 8);
    for (size_t i = 0; i < v.size(); ++i) {
        const int64_t k = key(v[i]);
        if (!runs.empty() && runs.back().key == k) ++runs.back().count;
        else runs.push_back(Run{k, (uint32_t)i, 1});
    }
    auto before = [](const Run& x, const Run& y) { return x.key != y.key ? x.key > y.key : x.at < y.at; };
    if (std::is_sorted(runs.begin(), runs.end(), before)) return;
    std::sort(runs.begin(), runs.end(), before);
    std::vector<T> sorted;
    sorted.reserve(v.size());
    for (const Run& r : runs) sorted.insert(sorted.end(), v.begin() + r.at, v.begin() + r.at + r.count);
    v.swap(sorted);
}

// How span units and long decode units are cut.  The default is the fastest; asynclm_plan asks for fewer cuts
// where the partial results would outgrow the fixed array of asynclm_attn_mixed_static.
struct CutPolicy {
    int units_by_keys = INT_MAX;      // long span units (kLongPieceTiles) that may be cut by keys, the longest first
    bool bound_pieces = true;         // kBulkTiles
};

// Modelled time until the last CTA is through with the warp body's queue: `joins` holds when the CTAs with span work join
// (the others are there from the start), each takes the next item as soon as it is through with one, and those that are
// still busy when nothing is left stream faster.  Time runs in steps of 1/1024 of the mean (longer ones where
// an item or a join is very long); *mean_ns, the mean finish, is what no other order of the same items ends before.
int64_t queue_ns(const std::vector<Item>& queue, const std::vector<int64_t>& joins, int n_ctas, int head_dim, int64_t* mean_ns) {
    const StreamCost cost = stream_cost(head_dim);
    auto tile_ns = [&](int64_t ctas) { return std::max(cost.least_tile_ns, cost.tile_ns * ctas / kStreamCtas); };
    const int64_t tile = tile_ns(n_ctas);
    struct Run { int64_t ns, count; };      // items of equal cost
    std::vector<Run> runs;
    int64_t sum = 0, tiles_before = -1, longest = 0;
    for (const Item& it : queue) {
        const int64_t tiles = ((int64_t)it.kv1 - it.kv0 + kWarpCost.gran - 1) / kWarpCost.gran;
        if (tiles != tiles_before) runs.push_back(Run{kWarpCost.item_ns + tiles * tile, 0});
        tiles_before = tiles;
        ++runs.back().count;
        sum += runs.back().ns;
        longest = std::max(longest, runs.back().ns);
    }
    for (int64_t at : joins) sum += at, longest = std::max(longest, at);
    const int64_t step = std::max<int64_t>(16, std::max(sum / n_ctas / 1024, longest / 4096));
    std::vector<int32_t> free(2048);      // CTAs that are free from step i on
    auto add = [&](int64_t at, int64_t ctas) {
        if (at >= (int64_t)free.size()) free.resize((size_t)at + 1024);
        free[(size_t)at] += (int32_t)ctas;
    };
    add(0, n_ctas - (int64_t)joins.size());
    for (int64_t at : joins) add(at / step, 1);
    size_t now = 0;
    for (const Run& r : runs) {
        const int64_t need = std::max<int64_t>(1, (r.ns + step / 2) / step);
        for (int64_t left = r.count; left > 0;) {
            while (free[now] == 0) ++now;
            const int64_t n = std::min<int64_t>(left, free[now]);
            free[now] -= (int32_t)n;
            add((int64_t)now + need, n);
            left -= n;
        }
    }
    // (CTAs that join when nothing is left have no part in it)
    int64_t late = 0;
    for (int64_t at : joins)
        if (at / step > (int64_t)now) --free[(size_t)(at / step)], ++late, sum -= at;
    *mean_ns = sum / (n_ctas - late);
    int64_t end = (int64_t)now * step, busy = n_ctas - late - free[now];
    for (size_t at = now + 1; busy > 0; ++at) {
        if (free[at] == 0) continue;
        end += (int64_t)(at - now) * step * tile_ns(busy) / tile;
        now = at;
        busy -= free[at];
    }
    return end;
}

// Default policy for the fused kernel.
//   Span units (tensor-core body) are compute-heavy and predictable: they are packed whole onto as few
// persistent CTAs as the load limit allows (largest first, each into the fullest CTA that still has
// room; a unit larger than a CTA's share is cut into equal pieces), so that most of them write final
// bf16 rows instead of fp32 partial rows.
//   Warp-body units (decode rows, short spans) are bandwidth-bound, and how fast a CTA streams depends
// on what the other SMs are doing, which no static cost predicts.  They are cut into chunks of a few
// tiles, sorted by length (longest first), and handed out at run time: the CTAs without span work
// start on one chunk each, every other chunk waits in a queue from which a CTA that runs out of work
// (a span CTA included) takes the next one with one atomic add.  Partial results are indexed by chunk
// and merged in chunk order, so the output does not depend on which CTA ran what.
//   The load limit is the smallest one under which the span units fit and the room left on all CTAs
// covers the modelled time of the queue; it is found by bisection.
//   Returns false, with only the units (their division and n_chunks) filled in, if the cuts leave more than
// max_partial_rows partial rows.
bool deal_dynamic(std::vector<int>& ids_tensor, const std::vector<int>& ids_warp,
                  std::vector<UnitBuild>& units, int group, int head_dim, int64_t kv_bytes, int n_ctas, const CutPolicy& policy,
                  int64_t max_partial_rows, std::vector<Item>& items,
                  std::vector<int32_t>& cta_indptr_warp, std::vector<int32_t>& cta_indptr_tensor,
                  std::vector<int32_t>& item_cta, int32_t* queue_first, int32_t* queue_count) {
    struct Piece { Item it; int32_t cta; };
    const bool tensor_only = ids_warp.empty();
    const PathCost tc = tensor_only ? kTensorOnlyCost : kTensorCost;
    const int64_t dual_tile_ns = tensor_only ? kTensorOnlyDualTileNs : kTensorDualTileNs;
    auto tiles_of = [](int64_t keys, int gran) { return (keys + gran - 1) / gran; };

    // ---- warp-body work as the model sees it (the chunks are cut below, once the number of CTAs
    // that start on the queue is known)
    int64_t warp_tiles = 0;
    for (int id : ids_warp) warp_tiles += tiles_of(units[id].n_keys, kWarpCost.gran);
    const int64_t warp_ns = warp_tiles * kWarpCost.tile_ns + (int64_t)ids_warp.size() * 2 * kWarpCost.item_ns;

    // ---- span units with two row tiles that would not fit a CTA whole are divided by rows into two
    // units of one row tile each (the second reader of the keys finds most of them in L2) rather than by
    // keys, which would cost fp32 partial rows and a merge, unless the pieces would be long (kLongPieceTiles).
    // The limit used for the decision is the lower bound of the one found below.
    {
        int64_t work = warp_ns;
        for (int id : ids_tensor)
            work += tc.item_ns + tiles_of(units[id].n_keys, tc.gran) * (units[id].u.ntok * group > 128 ? dual_tile_ns : tc.tile_ns);
        const int64_t limit0 = std::max(work / n_ctas, kStartNs + kv_bytes * 1000 / kDramBytesPerUs) * 64 / kDivideMargin64;
        const int half = 128 / group;      // tokens of one row tile
        // which of them are left to be cut by keys (below): the longest, because a divided half stays whole and would
        // be a CTA's longest item
        std::vector<char> by_keys;
        if (policy.units_by_keys > 0 && limit0 - tc.phase_ns - tc.item_ns >= kLongPieceTiles * dual_tile_ns) {
            std::vector<int> longest(ids_tensor);
            std::stable_sort(longest.begin(), longest.end(), [&](int x, int y) { return units[x].n_keys > units[y].n_keys; });
            by_keys.assign(units.size(), 0);
            int n = 0;
            for (int id : longest)
                if (units[(size_t)id].u.ntok * group > 128 && n < policy.units_by_keys) by_keys[(size_t)id] = 1, ++n;
        }
        const size_t n0 = ids_tensor.size();
        for (size_t i = 0; i < n0; ++i) {
            const int id = ids_tensor[i];
            UnitBuild& ub = units[(size_t)id];
            if (ub.u.ntok * group <= 128) continue;
            if (tc.phase_ns + tc.item_ns + tiles_of(ub.n_keys, tc.gran) * dual_tile_ns <= limit0) continue;
            if (!by_keys.empty() && by_keys[(size_t)id]) continue;
            UnitBuild second = ub;
            second.u.q_row0 += half;
            second.u.ntok -= half;
            second.u.kv_limit0 += half;
            ub.u.ntok = half;
            ub.n_keys = (int64_t)ub.u.kv_limit0 + ub.u.ntok - 1;
            ids_tensor.push_back((int)units.size());
            units.push_back(second);
        }
    }

    // ---- span units under a load limit
    std::vector<int> order(ids_tensor);
    std::vector<int64_t> tiles(units.size()), tns(units.size());
    for (int id : order) {
        tiles[(size_t)id] = tiles_of(units[id].n_keys, tc.gran);
        tns[(size_t)id] = units[id].u.ntok * group > 128 ? dual_tile_ns : tc.tile_ns;
    }
    sort_falling(order, [&](int id) { return tiles[(size_t)id] * tns[(size_t)id]; });
    // units of the same cost one after the other: (first in `order`, how many)
    struct Batch { int64_t tiles, ns; uint32_t at, count; };
    std::vector<Batch> batches;
    for (size_t i = 0; i < order.size(); ++i) {
        const int64_t t = tiles[(size_t)order[i]], ns = tns[(size_t)order[i]];
        if (!batches.empty() && batches.back().tiles == t && batches.back().ns == ns) ++batches.back().count;
        else batches.push_back(Batch{t, ns, (uint32_t)i, 1});
    }
    struct Cta { int64_t load; int32_t id; };
    std::vector<Cta> ctas((size_t)n_ctas);      // those in use, the fullest first, equal loads by id
    std::vector<Piece> pieces_out;
    int used = 0;
    // Packs the span units under `cap`; returns false if they do not fit or leave too little room for
    // the queue.  With emit == false only the verdict is computed (the bisection's probes).
    int64_t span_work = 0;      // all span items without the per-CTA start
    for (int id : order) span_work += tc.item_ns + tiles[(size_t)id] * tns[(size_t)id];
    const int64_t floor_ns = kStartNs + kv_bytes * 1000 / kDramBytesPerUs;
    const int64_t bound = std::max<int64_t>(std::max<int64_t>(1, (warp_ns + span_work) / n_ctas), floor_ns);      // of the load limit
    auto fill = [&](int64_t limit, bool emit) {
        // CTAs that may hold span work: the others have to be able to stream most of the queue by
        // themselves (span CTAs draw little bandwidth, and one SM streams only so much)
        const int64_t stream_ctas = limit > kStartNs
            ? (warp_tiles * kWarpCost.tile_ns * kStreamShare64 / 64 + (limit - kStartNs) - 1) / (limit - kStartNs) : n_ctas;
        // (a lone CTA does both)
        const int64_t span_ctas = ids_warp.empty() || n_ctas == 1 ? n_ctas : n_ctas - stream_ctas;
        if (!order.empty() && span_ctas < 1) return false;
        // what a span CTA may be given: the span work spread over those CTAs with some slack for the
        // packing, at most the load limit less the safety margin.  Spreading the spans thin costs little (a
        // span CTA that is done early joins the queue), filling span CTAs to the brim risks a late finish.
        const int64_t thin = order.empty() ? 0 : span_work / span_ctas * 5 / 4 + tc.phase_ns + tc.item_ns + dual_tile_ns;
        // (Past twice the lower bound the spread is given up: items of more than half of `thin` take a CTA each,
        // and there may be more of them than CTAs.)
        const int64_t full = limit * 64 / span_margin64(head_dim);
        const int64_t cap = limit > 2 * bound ? full : std::min(full, std::max(thin, 2 * (tc.phase_ns + tc.item_ns)));
        pieces_out.clear();
        used = 0;
        // moves the CTA at position `at` of `ctas` to where its new load belongs
        auto add_load = [&](int at, int64_t more) {
            Cta c = ctas[(size_t)at];
            c.load += more;
            auto fuller = [](const Cta& x, const Cta& y) { return x.load != y.load ? x.load > y.load : x.id < y.id; };
            if (at == 0 || fuller(ctas[(size_t)at - 1], c)) {
                ctas[(size_t)at] = c;
                return;
            }
            const int to = (int)(std::upper_bound(ctas.begin(), ctas.begin() + at, c, fuller) - ctas.begin());
            std::move_backward(ctas.begin() + to, ctas.begin() + at, ctas.begin() + at + 1);
            ctas[(size_t)to] = c;
        };
        for (const Batch& batch : batches) {
            const int64_t t = batch.tiles, ns = batch.ns;
            const int64_t fresh_room = std::max<int64_t>(1, (cap - tc.phase_ns - tc.item_ns) / ns);
            const int64_t pieces = t <= fresh_room ? 1 : (t + fresh_room - 1) / fresh_room;
            // pieces of a unit one after the other, units one after the other; whole units go to one CTA several at once
            // as long as it stays the fullest that has room (nobody fuller has, and it only gets fuller)
            const int64_t todo = pieces * batch.count;
            for (int64_t k = 0; k < todo;) {
                const int64_t c = k % pieces;
                const int64_t take = pieces == 1 ? t : t / pieces + (c < t % pieces ? 1 : 0);
                const int64_t need = tc.item_ns + take * ns;
                int at = used;
                if (used > 0 && ctas[(size_t)used - 1].load + need <= cap)
                    at = (int)(std::partition_point(ctas.begin(), ctas.begin() + used, [&](const Cta& x) { return x.load + need > cap; }) - ctas.begin());
                if (at == used) {
                    if (used < n_ctas) {
                        ctas[(size_t)used] = Cta{tc.phase_ns, (int32_t)used};
                        ++used;
                        if (!emit && used > span_ctas) return false;
                    } else {
                        if (!emit) return false;
                        --at;      // the least loaded
                        while (at > 0 && ctas[(size_t)at - 1].load == ctas[(size_t)at].load) --at;
                    }
                }
                const int64_t n = pieces > 1 ? 1 : std::min(todo - k, 1 + std::max<int64_t>(0, cap - need - ctas[(size_t)at].load) / need);
                if (emit)
                    for (int64_t j = k; j < k + n; ++j) {
                        const int id = order[batch.at + (size_t)(j / pieces)];
                        const int64_t k0 = c * (t / pieces) + std::min(c, t % pieces);      // tiles before piece c
                        pieces_out.push_back(Piece{Item{id, (int32_t)(k0 * tc.gran), (int32_t)std::min<int64_t>(units[id].n_keys, (k0 + take) * tc.gran),
                                                        (int32_t)c}, ctas[(size_t)at].id});
                    }
                add_load(at, n * need);
                k += n;
            }
        }
        // room for the queue: what the span CTAs have left after restarting on the warp body, and the
        // whole limit on the others
        int64_t room = (n_ctas - used) * std::max<int64_t>(0, limit - kWarpCost.phase_ns);
        for (int k = 0; k < used; ++k)
            room += std::max<int64_t>(0, limit - ctas[(size_t)k].load - kWarpCost.phase_ns);
        return used <= span_ctas && room >= warp_ns;
    };
    int64_t lo = bound;
    int64_t hi = lo + lo / 4 + tc.item_ns + tc.phase_ns + kWarpCost.phase_ns;
    while (!fill(hi, false)) { lo = hi; hi += hi / 2; }
    for (int iter = 0; iter < 24 && hi - lo > std::max<int64_t>(50, hi / 128); ++iter) {      // to 0.8 %
        const int64_t mid = (lo + hi) / 2;
        if (fill(mid, false)) hi = mid; else lo = mid;
    }
    fill(hi, true);
    for (const Piece& pz : pieces_out) units[pz.it.unit].u.n_chunks = std::max(units[pz.it.unit].u.n_chunks, pz.it.chunk + 1);

    // ---- warp-body chunks.  An item boundary costs time and a split unit costs partial rows and a
    // merge, so most of the work stays in long pieces: where the shortest units are long themselves (kShortUnitShare), a
    // few units, a sixth of all tiles, are cut into short chunks that go to the END of the queue, where they even out
    // the CTAs' finishing times; every other unit stays whole unless it is longer than two fifths of the step (or than kBulkTiles tiles
    // and an eighth of a CTA's share), in which case it is cut into equal pieces.  The queue holds the long pieces longest first, then the short chunks.
    std::vector<int> warp_order(ids_warp);
    sort_falling(warp_order, [&](int id) { return units[id].n_keys; });
    std::vector<Item> chunks, tail;
    chunks.reserve(ids_warp.size() + (size_t)n_ctas * 4);
    auto longest_piece = [&](int64_t limit) {
        int64_t t = limit * 2 / 5 / kWarpCost.tile_ns;
        if (policy.bound_pieces) t = std::min(t, std::max<int64_t>(kBulkTiles, warp_tiles / (8 * (int64_t)n_ctas)));
        return std::max<int64_t>(t, kMinChunkTiles);
    };
    int64_t bulk_max = longest_piece(hi);
    const int64_t tail_target = warp_tiles / 6;
    const int64_t tail_chunk = std::max<int64_t>(kMinChunkTiles, tail_target / ((int64_t)n_ctas * kTailChunksPerCta));
    // cuts the units; which are cut short: first those of up to four chunks (their merge is one round trip to
    // L2), longest first; longer ones only if that does not give a sixth of the tiles
    std::vector<char> to_tail(units.size());
    auto cut = [&](bool cut_tail) {
        chunks.clear();
        tail.clear();
        std::fill(to_tail.begin(), to_tail.end(), 0);
        int64_t tail_tiles = 0;
        for (int pass = 0; pass < 2 && cut_tail && tail_tiles < tail_target; ++pass)
            for (int id : warp_order) {
                const int64_t t = tiles_of(units[id].n_keys, kWarpCost.gran);
                if (tail_tiles >= tail_target) break;
                if (to_tail[(size_t)id] || t <= tail_chunk + tail_chunk / 2 || (pass == 0 && t > 4 * tail_chunk)) continue;
                to_tail[(size_t)id] = 1;
                tail_tiles += t;
            }
        for (int id : warp_order) {
            const int64_t t = tiles_of(units[id].n_keys, kWarpCost.gran);
            const bool short_chunks = to_tail[(size_t)id] != 0;
            const int64_t piece_max = short_chunks ? tail_chunk : bulk_max;
            const int64_t pieces = t <= piece_max + piece_max / 2 ? 1 : (t + piece_max - 1) / piece_max;
            int64_t k0 = 0;
            for (int64_t c = 0; c < pieces; ++c) {
                const int64_t take = t / pieces + (c < t % pieces ? 1 : 0);
                const int64_t k1 = std::min<int64_t>(units[id].n_keys, k0 + take * kWarpCost.gran);
                (short_chunks ? tail : chunks).push_back(Item{id, (int32_t)k0, (int32_t)k1, (int32_t)c});
                k0 = k1;
            }
            units[id].u.n_chunks = (int32_t)pieces;
        }
    };
    // the queue in its order: long pieces, then short chunks, the longest first
    bool queued = false;
    auto queue_up = [&]() {
        auto length = [](const Item& x) { return (int64_t)x.kv1 - x.kv0; };
        sort_falling(chunks, length);
        sort_falling(tail, length);
        chunks.insert(chunks.end(), tail.begin(), tail.end());
        queued = true;
    };
    bool cut_tail = n_ctas < kSaturatingCtas;
    int64_t shortest = 0;
    for (size_t i = warp_order.size(); i-- > 0 && shortest < tail_target && !cut_tail;) {
        const int64_t t = tiles_of(units[(size_t)warp_order[i]].n_keys, kWarpCost.gran);
        shortest += t;
        cut_tail = t * n_ctas * kShortUnitShareDen > warp_tiles * kShortUnitShareNum;
    }
    int64_t decode_tiles = 0;
    for (int id : ids_warp)
        if (units[(size_t)id].u.ntok == 1) decode_tiles += tiles_of(units[(size_t)id].n_keys, kWarpCost.gran);
    cut_tail = cut_tail || 2 * decode_tiles < warp_tiles;      // (spans on the warp body: not measured without)
    cut(cut_tail);
    // Two fifths of the limit were chosen when the span CTAs had a margin of 88 and the limit came out that much higher. Where
    // pieces of that length leave no queue, they are taken: a CTA that comes from span tiles passes through the warp
    // body's start and end (3 us) to find a queue empty.  (us of attention a layer, with a queue | without: 4 sequences of 4/2
    // heads over 5-7 K keys, one with 75 tokens, 41 pieces on 40 CTAs 29.3 | 26.1; 23 of 4/2 heads with 2-44 tokens 30.3 | 23.2.)
    if (used > 0 && chunks.size() + tail.size() > (size_t)(n_ctas - used) && warp_order.size() <= (size_t)(n_ctas - used)) {
        const int64_t shorter = bulk_max;
        bulk_max = longest_piece(hi * 88 / span_margin64(head_dim));
        cut(cut_tail);
        if (chunks.size() + tail.size() > (size_t)(n_ctas - used)) {
            bulk_max = shorter;
            cut(cut_tail);
        }
    }
    if (!cut_tail && chunks.size() > (size_t)(n_ctas - used)) {      // (else every CTA has one to begin with and nothing is left)
        std::vector<int64_t> joins;
        for (int k = 0; k < used; ++k) joins.push_back(ctas[(size_t)k].load);
        int64_t mean = 0;
        queue_up();
        const int64_t whole = queue_ns(chunks, joins, n_ctas, head_dim, &mean);
        // (Span CTAs join at times of their own, which evens the waves out better than modelled: where a gain of 6 to 11 % of the
        // mean was predicted, cutting was 1 to 7 % slower; where 20 %, 6 % faster.)
        const int64_t cut_ns = std::max(stream_cost(head_dim).cut_ns, used > 0 ? mean / 8 : 0);
        if (whole - mean > cut_ns) {
            const std::vector<Item> uncut(chunks);
            cut(true);
            queue_up();
            if (whole - queue_ns(chunks, joins, n_ctas, head_dim, &mean) <= cut_ns) {
                chunks = uncut;
                for (int id : warp_order) units[(size_t)id].u.n_chunks = 1;
                for (const Item& it : chunks) units[(size_t)it.unit].u.n_chunks = std::max(units[(size_t)it.unit].u.n_chunks, it.chunk + 1);
            }
        }
    }
    int64_t partial_rows = 0;
    for (const UnitBuild& ub : units)
        if (ub.u.n_chunks > 1) partial_rows += (int64_t)ub.u.n_chunks * ub.u.ntok;
    if (partial_rows > max_partial_rows) return false;
    if (!queued) queue_up();

    // ---- emit: warp-body items first (one start chunk for every CTA without span work, then the
    // queue), then the span items grouped by CTA
    cta_indptr_warp.assign((size_t)n_ctas + 1, 0);
    cta_indptr_tensor.assign((size_t)n_ctas + 1, 0);
    const int n_start = (int)std::min<size_t>(chunks.size(), (size_t)(n_ctas - used));
    items.reserve(chunks.size() + pieces_out.size());
    item_cta.reserve(chunks.size() + pieces_out.size());
    for (size_t i = 0; i < chunks.size(); ++i) {
        items.push_back(chunks[i]);
        item_cta.push_back(i < (size_t)n_start ? used + (int32_t)i : -1);
    }
    for (int k = 0; k <= n_ctas; ++k)
        cta_indptr_warp[(size_t)k] = std::min(std::max(k - used, 0), n_start);
    *queue_first = n_start;
    *queue_count = (int32_t)chunks.size() - n_start;
    const int32_t first = (int32_t)items.size();
    std::stable_sort(pieces_out.begin(), pieces_out.end(), [](const Piece& x, const Piece& y) { return x.cta < y.cta; });
    std::vector<int32_t> count((size_t)n_ctas, 0);
    for (const Piece& pz : pieces_out) {
        items.push_back(pz.it);
        item_cta.push_back(pz.cta);
        count[(size_t)pz.cta]++;
    }
    int32_t at = first;
    for (int k = 0; k < n_ctas; ++k) {
        cta_indptr_tensor[(size_t)k] = at;
        at += count[(size_t)k];
    }
    cta_indptr_tensor[(size_t)n_ctas] = at;
    return true;
}

}  // namespace

extern "C" int asynclm_plan(const asynclm_shape* shape, const asynclm_plan_options* opts,
                            const asynclm_batch* batch, void* host_ws, size_t host_bytes,
                            void* dev_ws, size_t dev_bytes, void* stream,
                            asynclm_plan_t** out_plan) {
    int rc = check_shape(shape);
    if (rc != ASYNCLM_OK) return rc;
    if (!batch || !host_ws || !out_plan || batch->batch < 0) return ASYNCLM_ERR_INVALID_ARG;
    if (((uintptr_t)host_ws & 15) != 0 || ((uintptr_t)dev_ws & 255) != 0)
        return ASYNCLM_ERR_INVALID_ARG;
    const int B = batch->batch;
    if (B > 0 && (!batch->q_indptr || !batch->kv_len_before || !batch->page_indptr))
        return ASYNCLM_ERR_INVALID_ARG;
    if (opts && (opts->kv_chunk_tokens < 0 || opts->num_sms < 0 || opts->tensor_min_rows < 0))
        return ASYNCLM_ERR_INVALID_ARG;
    if (opts && opts->kv_chunk_tokens > 0 && opts->kv_chunk_tokens % 64 != 0)
        return ASYNCLM_ERR_INVALID_ARG;
    const bool host_only = dev_ws == nullptr;
    if (host_only && !(opts && opts->num_sms > 0)) return ASYNCLM_ERR_INVALID_ARG;

    int device = -1;
    if (!host_only) {
        if (cudaGetDevice(&device) != cudaSuccess) return ASYNCLM_ERR_CUDA;
        int major = 0;
        if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device) != cudaSuccess)
            return ASYNCLM_ERR_CUDA;
        if (major != 10) return ASYNCLM_ERR_ARCH;
    }
    int n_sms = 0;
    rc = resolve_num_sms(opts, !host_only, &n_sms);
    if (rc != ASYNCLM_OK) return rc;

    const int Hkv = shape->num_kv_heads;
    const int G = shape->num_q_heads / Hkv;
    const int P = shape->page_size;

    // ---- validation -------------------------------------------------------------------------
    static const int32_t zero_indptr[1] = {0};
    const int32_t* q_indptr = B > 0 ? batch->q_indptr : zero_indptr;
    const int32_t* page_indptr = B > 0 ? batch->page_indptr : zero_indptr;
    if (q_indptr[0] != 0 || page_indptr[0] != 0) return ASYNCLM_ERR_INVALID_ARG;
    int64_t total_kv = 0;
    for (int b = 0; b < B; ++b) {
        const int64_t ql = (int64_t)q_indptr[b + 1] - q_indptr[b];
        const int64_t np = (int64_t)page_indptr[b + 1] - page_indptr[b];
        if (ql < 0 || np < 0 || batch->kv_len_before[b] < 0) return ASYNCLM_ERR_INVALID_ARG;
        const int64_t n = (int64_t)batch->kv_len_before[b] + ql;
        if (n > INT32_MAX - kKvTile) return ASYNCLM_ERR_INVALID_ARG;
        if (ql > 0) {
            if (np * P < n) return ASYNCLM_ERR_PAGE_TABLE;
            total_kv += n;
        }
    }
    const int T = q_indptr[B];
    const int64_t total_pages = page_indptr[B];
    if (total_pages > 0 && !batch->page_indices) return ASYNCLM_ERR_INVALID_ARG;
    for (int b = 0; b < B; ++b) {
        const int64_t ql = (int64_t)q_indptr[b + 1] - q_indptr[b];
        if (ql == 0) continue;   // paused sequences are not read or written: their ids are not checked
        const int64_t need = ((int64_t)batch->kv_len_before[b] + ql + P - 1) / P;
        // (as unsigned numbers, the negative ids are the largest; no exit inside the loop, so that it runs in vectors)
        const int32_t* ids = batch->page_indices + page_indptr[b];
        const uint32_t end = (uint32_t)std::min<int64_t>(shape->num_pages, (int64_t)INT32_MAX + 1);
        uint32_t bad = 0;
        for (int64_t j = 0; j < need; ++j) bad |= (uint32_t)((uint32_t)ids[j] >= end);
        if (bad) return ASYNCLM_ERR_PAGE_TABLE;
    }
    if (opts && (opts->flags & ASYNCLM_PLAN_REJECT_ALIASED_WRITES)) {
        std::vector<int32_t> written;
        for (int b = 0; b < B; ++b) {
            const int ql = q_indptr[b + 1] - q_indptr[b];
            if (ql == 0) continue;
            const int lo = batch->kv_len_before[b] / P;
            const int hi = (batch->kv_len_before[b] + ql - 1) / P;
            for (int j = lo; j <= hi; ++j) written.push_back(batch->page_indices[page_indptr[b] + j]);
        }
        std::sort(written.begin(), written.end());
        if (std::adjacent_find(written.begin(), written.end()) != written.end())
            return ASYNCLM_ERR_PAGE_TABLE;
    }

    // ---- units ------------------------------------------------------------------------------
    const bool tensor_wanted = !(opts && (opts->flags & ASYNCLM_PLAN_NO_TENSOR_PATH));
    const int tensor_min_rows =
        (opts && opts->tensor_min_rows > 0) ? opts->tensor_min_rows : default_tensor_min_rows(shape->head_dim);
    const int TQ = tensor_tile_tokens(G);
    const int fixed_chunk = opts ? opts->kv_chunk_tokens : 0;
    const int ctas_cuda = n_sms * kCudaSlotsPerSm;
    const int ctas_tensor = n_sms;
    std::vector<UnitBuild> units;
    std::vector<int> ids_cuda, ids_tensor;
    std::vector<Item> items;
    std::vector<int32_t> item_cta, cta_indptr_cuda, cta_indptr_tensor;
    int n_items_cuda = 0;
    int32_t queue_first = 0, queue_count = 0;
    std::vector<int32_t> split_units, merge_blocks;   // merge block: 4 (token, head) rows of a split unit
    int64_t partial_rows = 0;
    // (too_many: the cuts leave more than max_partial_rows partial rows, and nothing is dealt)
    bool too_many = false;
    auto deal = [&](const CutPolicy& policy, bool tensor_on, int64_t max_partial_rows) -> int {
        units.clear(); ids_cuda.clear(); ids_tensor.clear(); items.clear(); item_cta.clear();
        units.reserve(std::min<size_t>((size_t)std::min(B, T) * Hkv, 65536));
        ids_cuda.reserve(units.capacity());
        split_units.clear(); merge_blocks.clear();
        n_items_cuda = queue_first = queue_count = 0;
        partial_rows = 0;
        for (int b = 0; b < B; ++b) {
            const int ql = q_indptr[b + 1] - q_indptr[b];
            if (ql == 0) continue;
            const int ctx = batch->kv_len_before[b];
            const bool tensor = tensor_on && (int64_t)G * ql >= tensor_min_rows;
            const int step = tensor ? TQ : warp_unit_tokens(G);
            for (int h = 0; h < Hkv; ++h) {
                for (int t0 = 0; t0 < ql; t0 += step) {
                    UnitBuild ub{};
                    ub.u.seq = b;
                    ub.u.kv_head = h;
                    ub.u.q_row0 = q_indptr[b] + t0;
                    ub.u.ntok = std::min(step, ql - t0);
                    ub.u.kv_limit0 = ctx + t0 + 1;
                    ub.u.n_chunks = 0;
                    ub.u.partial_base = -1;
                    ub.u.page_base = page_indptr[b];
                    ub.path = tensor ? kPathTensor : kPathCuda;
                    ub.n_keys = (int64_t)ub.u.kv_limit0 + ub.u.ntok - 1;
                    (tensor ? ids_tensor : ids_cuda).push_back((int)units.size());
                    units.push_back(ub);
                }
            }
        }

        // ---- items and CTA assignment --------------------------------------------------------------
        if (fixed_chunk > 0 || ctas_cuda != ctas_tensor) {
            cut_and_deal(ids_cuda, units, fixed_chunk, ctas_cuda, kCudaItemOverheadTiles, items,
                         cta_indptr_cuda, item_cta);
            n_items_cuda = (int)items.size();
            cut_and_deal(ids_tensor, units, fixed_chunk, ctas_tensor, kTensorItemOverheadTiles, items,
                         cta_indptr_tensor, item_cta);
        } else {
            // bytes of K and V the step has to read, each (sequence, kv head) counted once
            const int64_t kv_bytes = total_kv * Hkv * 4 * shape->head_dim;
            too_many = !deal_dynamic(ids_tensor, ids_cuda, units, G, shape->head_dim, kv_bytes, ctas_cuda, policy, max_partial_rows, items,
                                     cta_indptr_cuda, cta_indptr_tensor, item_cta, &queue_first, &queue_count);
            if (too_many) return ASYNCLM_OK;
            n_items_cuda = queue_first + queue_count;
        }

        // ---- partial rows ------------------------------------------------------------------------
        for (size_t i = 0; i < units.size(); ++i) {
            if (units[i].u.n_chunks > 1) {
                units[i].u.partial_base = (int32_t)partial_rows;
                partial_rows += (int64_t)units[i].u.n_chunks * units[i].u.ntok;
                split_units.push_back((int32_t)i);
                if (i >= (size_t)(INT32_MAX >> 6)) return ASYNCLM_ERR_WORKSPACE_TOO_SMALL;
                // split units of the warp body are merged inside the attention kernel; those of the span
                // body by the merge kernel
                if (units[i].path == kPathTensor)
                    for (int rb = 0; rb * 4 < units[i].u.ntok * G; ++rb) merge_blocks.push_back((int32_t)((i << 6) | (size_t)rb));
                if (partial_rows > INT32_MAX / 2) return ASYNCLM_ERR_WORKSPACE_TOO_SMALL;
            }
        }
        return ASYNCLM_OK;
    };
    // The fastest cuts, as long as their partial results fit the fixed array of asynclm_attn_mixed_static; else as
    // many of the long span units cut by keys as it has room for, none of them, long pieces in the queue as
    // well, and at head_dim 64 no span units at all (warp units have far fewer partial rows).  If nothing fits,
    // the fastest again: that call then refuses the plan.  A try that does not fit ends when its cuts are
    // known, before the items are sorted and dealt.
    int64_t static_rows = (int64_t)(ASYNCLM_STATIC_SCRATCH_BYTES / ((size_t)G * (shape->head_dim + 1) * sizeof(float)));
    while (partial_bytes(static_rows, G, shape->head_dim) > ASYNCLM_STATIC_SCRATCH_BYTES) --static_rows;
    auto fits_static = [&]() { return !too_many && partial_rows <= static_rows; };
    const CutPolicy fastest;
    rc = deal(fastest, tensor_wanted, static_rows);
    if (rc == ASYNCLM_OK && !fits_static()) {
        if (fixed_chunk == 0) {
            int64_t span_rows = 0, span_units = 0, warp_rows = 0;
            for (const UnitBuild& ub : units) {
                const int64_t rows = ub.u.n_chunks > 1 ? (int64_t)ub.u.n_chunks * ub.u.ntok : 0;
                if (ub.path != kPathTensor) warp_rows += rows;
                else if (rows > 0) span_rows += rows, ++span_units;
            }
            const int64_t room = (int64_t)(ASYNCLM_STATIC_SCRATCH_BYTES / ((size_t)G * (shape->head_dim + 1) * sizeof(float))) - warp_rows;
            CutPolicy fewer;
            fewer.units_by_keys = room <= 0 ? 0 : (int)(span_units * room / std::max<int64_t>(1, span_rows) * 15 / 16);
            if (fewer.units_by_keys > 0) rc = deal(fewer, tensor_wanted, static_rows);
            if (rc == ASYNCLM_OK && !fits_static()) rc = deal(CutPolicy{0, true}, tensor_wanted, static_rows);
            if (rc == ASYNCLM_OK && !fits_static()) rc = deal(CutPolicy{0, false}, tensor_wanted, static_rows);
        }
        if (rc == ASYNCLM_OK && !fits_static() && tensor_wanted && shape->head_dim == 64)
            rc = deal(CutPolicy{0, false}, false, static_rows);
        if (rc == ASYNCLM_OK && !fits_static()) rc = deal(fastest, tensor_wanted, INT64_MAX);
    }
    if (rc != ASYNCLM_OK) return rc;
    const int n_items = (int)items.size();

    const int n_split = (int)split_units.size();

    // CTAs without an item, which stand at the end, have something to do only where there is a queue: else they are not
    // launched, and their headers (384 bytes each, of which a small plan mostly consists) are neither cleared nor uploaded.
    int grid_cuda = ctas_cuda, grid_tensor = ctas_tensor;
    if (queue_count == 0 && ctas_cuda == ctas_tensor) {
        auto idle = [&](int c) { return cta_indptr_cuda[(size_t)c] == cta_indptr_cuda[(size_t)c + 1] && cta_indptr_tensor[(size_t)c] == cta_indptr_tensor[(size_t)c + 1]; };
        while (grid_cuda > 1 && idle(grid_cuda - 1)) --grid_cuda;
        grid_tensor = grid_cuda;
    }

    // ---- pack ---------------------------------------------------------------------------------
    BlobLayout L = layout_blob(B, T, total_pages, (int64_t)units.size(), n_items, grid_cuda,
                               grid_tensor, (int64_t)n_split, (int64_t)merge_blocks.size());
    const size_t plan_bytes = align_up(sizeof(asynclm_plan_s), 256);
    const size_t item_cta_bytes = align_up(sizeof(int32_t) * (size_t)std::max(n_items, 1), 256);
    const size_t host_need = plan_bytes + L.blob_bytes + item_cta_bytes;
    const size_t dev_need = L.blob_bytes + partial_bytes(partial_rows, G, shape->head_dim);
    if (host_bytes < host_need) return ASYNCLM_ERR_WORKSPACE_TOO_SMALL;
    if (!host_only && dev_bytes < dev_need) return ASYNCLM_ERR_WORKSPACE_TOO_SMALL;

    char* hb = (char*)host_ws + plan_bytes;
    std::memset(hb + L.off_status, 0, 256);
    std::memset(hb + L.off_arrivals, 0, sizeof(int32_t) * std::max<size_t>(units.size(), 1));
    if (B > 0) {
        std::memcpy(hb + L.off_q_indptr, q_indptr, sizeof(int32_t) * (size_t)(B + 1));
        std::memcpy(hb + L.off_kv_len, batch->kv_len_before, sizeof(int32_t) * (size_t)B);
        std::memcpy(hb + L.off_page_indptr, page_indptr, sizeof(int32_t) * (size_t)(B + 1));
    } else {
        std::memset(hb + L.off_q_indptr, 0, sizeof(int32_t));
        std::memset(hb + L.off_page_indptr, 0, sizeof(int32_t));
    }
    if (total_pages > 0)
        std::memcpy(hb + L.off_page_indices, batch->page_indices, sizeof(int32_t) * (size_t)total_pages);
    int32_t* row_seq = (int32_t*)(hb + L.off_row_seq);
    int64_t* row_slot = (int64_t*)(hb + L.off_row_slot);
    for (int b = 0; b < B; ++b)
        for (int r = q_indptr[b]; r < q_indptr[b + 1]; ++r) {
            row_seq[r] = b;
            const int pos = batch->kv_len_before[b] + (r - q_indptr[b]);
            row_slot[r] = (int64_t)batch->page_indices[page_indptr[b] + pos / P] * P + pos % P;
        }
    Unit* h_units = (Unit*)(hb + L.off_units);
    for (size_t i = 0; i < units.size(); ++i) h_units[i] = units[i].u;
    if (n_items > 0) std::memcpy(hb + L.off_items, items.data(), sizeof(Item) * (size_t)n_items);
    int32_t* h_heads = (int32_t*)(hb + L.off_heads);
    std::memset(h_heads, 0, sizeof(int32_t) * kHeadWords * (size_t)std::max(grid_cuda, grid_tensor));
    Work* h_works = (Work*)(hb + L.off_works);
    for (int i = 0; i < n_items; ++i) {
        const Item& it = items[(size_t)i];
        const Unit& u = units[(size_t)it.unit].u;
        Work w;
        w.kv0 = it.kv0;
        w.kv_end = std::min(it.kv1, u.kv_limit0 + u.ntok - 1);
        w.q_row0 = u.q_row0;
        w.ntok = u.ntok;
        w.kv_limit0 = u.kv_limit0;
        w.kv_head = u.kv_head;
        w.partial_row0 = u.partial_base < 0 ? -1 : u.partial_base + it.chunk * u.ntok;
        w.page0 = u.page_base + it.kv0 / kPage;
        w.unit = it.unit;
        w.n_chunks = u.n_chunks;
        w.partial_base = u.partial_base;
        w.q_seq0 = q_indptr[u.seq];
        h_works[i] = w;
    }
    for (int c = 0; c < std::max(grid_cuda, grid_tensor); ++c) {
        int32_t* h = h_heads + (size_t)c * kHeadWords;
        const int32_t range[4] = {c < grid_tensor ? cta_indptr_tensor[(size_t)c] : 0,
                                  c < grid_tensor ? cta_indptr_tensor[(size_t)c + 1] : 0,
                                  c < grid_cuda ? cta_indptr_cuda[(size_t)c] : 0,
                                  c < grid_cuda ? cta_indptr_cuda[(size_t)c + 1] : 0};
        std::memcpy(h, range, sizeof(range));
        for (int path = 0; path < 2; ++path) {
            const int first = range[2 * path], last = range[2 * path + 1];
            if (first >= last) continue;
            const Work& w = h_works[first];
            std::memcpy(h + (path == 0 ? kHeadWorkTensor : kHeadWorkCuda), &w, sizeof(Work));
            const int npg = (w.kv_end - w.kv0 + kPage - 1) / kPage;
            for (int k = 0; k < 32 && k < npg; ++k)
                h[(path == 0 ? kHeadPagesTensor : kHeadPagesCuda) + k] = batch->page_indices[w.page0 + k];
        }
    }
    std::memcpy(hb + L.off_cta_cuda, cta_indptr_cuda.data(), sizeof(int32_t) * (size_t)(grid_cuda + 1));
    std::memcpy(hb + L.off_cta_tensor, cta_indptr_tensor.data(),
                sizeof(int32_t) * (size_t)(grid_tensor + 1));
    if (n_split > 0) std::memcpy(hb + L.off_split, split_units.data(), sizeof(int32_t) * split_units.size());
    if (!merge_blocks.empty())
        std::memcpy(hb + L.off_merge, merge_blocks.data(), sizeof(int32_t) * merge_blocks.size());
    int32_t* h_item_cta = (int32_t*)(hb + L.blob_bytes);
    if (n_items > 0) std::memcpy(h_item_cta, item_cta.data(), sizeof(int32_t) * (size_t)n_items);

    asynclm_plan_s* plan = (asynclm_plan_s*)host_ws;
    std::memset(plan, 0, sizeof(*plan));
    plan->magic = kPlanMagic;
    plan->shape = *shape;
    plan->device = device;
    plan->host_only = host_only ? 1 : 0;
    plan->h_units = h_units;
    plan->h_items = (const Item*)(hb + L.off_items);
    plan->h_item_cta = h_item_cta;
    plan->h_kv_len_before = (const int32_t*)(hb + L.off_kv_len);
    plan->h_units_path_split = n_items_cuda;
    for (int b = 0; b < B; ++b) plan->max_q_len = std::max(plan->max_q_len, q_indptr[b + 1] - q_indptr[b]);

    char* db = (char*)dev_ws;
    DevPlan& d = plan->dev;
    auto dp = [&](size_t off) { return host_only ? nullptr : (void*)(db + off); };
    d.status = (int32_t*)dp(L.off_status);
    d.counters = (int32_t*)dp(L.off_status + 64);
    d.queue_first = queue_first;
    d.queue_count = queue_count;
    d.q_indptr = (const int32_t*)dp(L.off_q_indptr);
    d.kv_len_before = (const int32_t*)dp(L.off_kv_len);
    d.page_indptr = (const int32_t*)dp(L.off_page_indptr);
    d.page_indices = (const int32_t*)dp(L.off_page_indices);
    d.row_seq = (const int32_t*)dp(L.off_row_seq);
    d.row_slot = (const int64_t*)dp(L.off_row_slot);
    d.units = (const Unit*)dp(L.off_units);
    d.items = (const Item*)dp(L.off_items);
    d.works = (const Work*)dp(L.off_works);
    d.cta_heads = (const int32_t*)dp(L.off_heads);
    d.cta_indptr_cuda = (const int32_t*)dp(L.off_cta_cuda);
    d.cta_indptr_tensor = (const int32_t*)dp(L.off_cta_tensor);
    d.split_units = (const int32_t*)dp(L.off_split);
    d.merge_blocks = (const int32_t*)dp(L.off_merge);
    d.unit_arrivals = (int32_t*)dp(L.off_arrivals);
    d.partial_o = (float*)dp(L.blob_bytes);
    d.partial_lse = (float*)dp(L.blob_bytes + align_up((size_t)partial_rows * (size_t)G *
                                                           (size_t)shape->head_dim * sizeof(float), 256));
    d.batch = B;
    d.total_q = T;
    d.num_units = (int32_t)units.size();
    d.num_items = n_items;
    d.num_items_cuda = n_items_cuda;
    d.num_items_tensor = n_items - n_items_cuda;
    d.num_split_units = n_split;
    d.num_merge_blocks = (int32_t)merge_blocks.size();
    d.num_ctas_cuda = grid_cuda;
    d.num_ctas_tensor = grid_tensor;
    d.num_q_heads = shape->num_q_heads;
    d.num_kv_heads = Hkv;
    d.head_dim = shape->head_dim;
    d.group = G;
    d.num_pages = shape->num_pages;
    // at least the smallest normal number: the kernels flush smaller ones to zero, and the span body scales masked
    // scores (-inf) as well
    d.sm_scale = shape->sm_scale > 0.f ? std::max(shape->sm_scale, FLT_MIN) : 1.0f / sqrtf((float)shape->head_dim);

    asynclm_plan_info& info = plan->info;
    info.total_q = T;
    info.num_units = d.num_units;
    info.num_items = n_items;
    info.num_split_units = d.num_split_units;
    info.partial_rows = (int32_t)partial_rows;
    int max_chunk = 0;
    for (const Item& it : items) max_chunk = std::max(max_chunk, it.kv1 - it.kv0);
    info.kv_chunk_tokens = fixed_chunk > 0 ? fixed_chunk : (d.num_split_units ? max_chunk : INT32_MAX);
    info.num_ctas_cuda = grid_cuda;
    info.num_ctas_tensor = grid_tensor;
    info.num_items_tensor = d.num_items_tensor;
    info.launches_append = T > 0 ? 1 : 0;
    // span tiles and decode rows share one fused launch when a step has both
    info.launches_attn = ((n_items_cuda > 0 || d.num_items_tensor > 0) ? 1 : 0) + (merge_blocks.empty() ? 0 : 1);
    info.num_sms = n_sms;
    info.total_kv_tokens = total_kv;
    info.device_bytes_used = dev_need;
    info.host_bytes_used = host_need;

    if (!host_only) {
        // By kernel where the workspace is page-locked, so that kernels can read it, and the plan neither so small that the
        // copy engine is as fast nor so large that the bus is what takes the time.
        const void* by_kernel = L.blob_bytes >= kUploadMinBytes && L.blob_bytes <= kUploadMaxBytes ? page_locked_on_device(hb, L.blob_bytes) : nullptr;
        cudaError_t e = by_kernel ? upload_plan(db, by_kernel, L.blob_bytes, (cudaStream_t)stream)
                                  : cudaMemcpyAsync(db, hb, L.blob_bytes, cudaMemcpyHostToDevice, (cudaStream_t)stream);
        if (int rc = cuda_status(e)) return rc;
        plan->fresh = by_kernel ? 1 : 0;
    }
    *out_plan = plan;
    return ASYNCLM_OK;
}

extern "C" int asynclm_plan_get_info(const asynclm_plan_t* plan, asynclm_plan_info* info) {
    if (!plan || !info || plan->magic != kPlanMagic) return ASYNCLM_ERR_INVALID_ARG;
    *info = plan->info;
    return ASYNCLM_OK;
}

extern "C" int asynclm_plan_get_items(const asynclm_plan_t* plan, asynclm_item_view* out,
                                      int32_t capacity) {
    if (!plan || plan->magic != kPlanMagic || capacity < 0 || (capacity > 0 && !out))
        return ASYNCLM_ERR_INVALID_ARG;
    const int n = plan->dev.num_items;
    for (int i = 0; i < n && i < capacity; ++i) {
        const Item& it = plan->h_items[i];
        const Unit& u = plan->h_units[it.unit];
        asynclm_item_view v;
        v.seq = u.seq;
        v.kv_head = u.kv_head;
        v.tok0 = u.kv_limit0 - 1 - plan->h_kv_len_before[u.seq];
        v.ntok = u.ntok;
        v.kv0 = it.kv0;
        v.kv1 = it.kv1;
        v.path = i < plan->h_units_path_split ? kPathCuda : kPathTensor;
        v.cta = plan->h_item_cta[i];
        out[i] = v;
    }
    return n;
}
