// Tables and launchers of the direct bucketed form (tiles.cu).
#pragma once
#include <algorithm>
#include <cstdint>

#include "kernels.h"

namespace turtle {

constexpr int TL_MAX_BITS = 10;           // bucket-index bits one level sorts by, at most
constexpr uint32_t TL_MAX_GROUP = 1024;   // runs gathered into one second-level tile, at most

constexpr int TILE_THREADS = 512;         // threads of an extraction or gather CTA; 1024 threads per SM
constexpr uint32_t tile_keys(int key_words) { return 16u * TILE_THREADS / (uint32_t)key_words; }  // keys per tile
constexpr uint32_t TL_STEP_KEYS = 256;    // a tile is written when fewer keys than one warp step fit

// Tiles of one level: run starts, first key of each tile, continuation rows (second level), the tile
// counter and the key cursor (both zero before the first launch). The run starts (bins + 1 16-bit entries
// a tile) of eight tiles are interleaved, entry by entry, so that one 32-byte sector holds a run's
// bounds in eight tiles: a gather reads the same run of consecutive tiles.
struct TileTable {
    uint16_t *starts;
    uint64_t *base;
    uint32_t *next;
    uint32_t pitch, max_tiles;
    uint32_t *n_tiles;
    unsigned long long *cursor;
};
inline uint64_t tile_start_bytes(uint64_t tiles, uint32_t pitch) { return 16 * ((tiles + 7) / 8) * pitch; }
__host__ __device__ inline uint64_t tile_start_index(const TileTable &t, uint32_t row, uint32_t bin) {
    return ((uint64_t)(row >> 3) * t.pitch + bin) * 8 + (row & 7);
}

// Windows to extract: starts in packed words [w_begin, w_end), 32 to a word.
struct ExtractArgs {
    const uint64_t *P;
    const uint32_t *V32;
    uint64_t w_begin, w_end;
    int k;
    uint32_t top_lo, top_span;  // top_span != 0: only windows whose left-aligned key's top 32 bits less top_lo are below it
    const uint64_t *lib_starts;  // batched form (n_libs > 0), as launch_pass1
    const int *lib_k;
    int n_libs, tag_shift;
};
// 1024 threads per SM; a thread takes one word at a time. Small libraries leave three quarters of a CTA's warps idle
// rather than SMs: 20 kbase 12.7 us against 19.4 with full CTAs; one busy warp per CTA gained nothing more.
inline int extract_grid(int sms, uint64_t words) {
    return (int)std::max<uint64_t>(1, std::min<uint64_t>((words + TILE_THREADS / 4 - 1) / (TILE_THREADS / 4),
                                                         (uint64_t)sms * (1024 / TILE_THREADS)));
}

// Bucket index of a left-aligned key: floor((f - f_lo) * scale / 2^32), f the high word of v (2^32 - v) for
// the key's top 31 bits v, in [0, n_buckets) for the keys of the range. lib.lib != null (batches): bucket_of(key,
// lib). slices != null (plain keys): f = the top 32 bits of key << align (all ones when the key has more bits than that
// leaves room for), clamped to [f_lo, f_lo + span], less f_lo; slice f >> slice_shift has its first bucket and its
// number of buckets in slices[].
struct TileGeom {
    BucketGeom lib;
    uint32_t f_lo, scale, n_buckets;
    uint32_t span;
    int align, slice_shift;
    const uint2 *slices;
};

// A sample of an array's keys: the n sampled keys' largest left shift, the least and greatest of their top 32 bits
// after it, the slices between (of 2^shift values, at most KS_SLICES) and, per slice, its first bucket and number
// of buckets in proportion to its sampled keys; crowd = most sampled keys in one of KS_CHECK equal groups of buckets.
constexpr uint32_t KS_SLICES = 256, KS_CHECK = 1024;
struct KeySample {
    uint32_t n, align, lo, hi, shift, crowd, pad[2];
    uint2 slice[KS_SLICES];
};
// Place of the j-th of 2^log2m sampled keys among n (a whole stride of n >> log2m would leave up to half of the array
// unseen at its end).
__host__ __device__ inline uint64_t sample_place(uint64_t n, int log2m, uint32_t j) { return n * j >> log2m; }
// Buckets for keys like the sample's (sample: its device copy); false when some group of buckets holds more than
// four times its share: one key, or a cluster below the slices' resolution, that a single CTA would have to count.
// (40M keys in even buckets: 0.98 ms against 2.7 by radix sort; in two clusters 2.78 by radix sort, of which the
// look at the sample, and the wait for it, are 0.035.) False, too, when a sampled key has bits above key_bits, which the
// tiles would only find out on the way (40M such keys: 2.67 ms by tiles and then by radix sort, which takes 1.88).
inline bool sample_geom(const KeySample &k, const KeySample *sample, uint32_t n_buckets, int key_words, int key_bits,
                        TileGeom *g) {
    if (k.crowd > 4 * (k.n / KS_CHECK) + 32 || 64 * key_words - (int)k.align > key_bits) return false;
    g->f_lo = k.lo;
    g->span = k.hi - k.lo;
    g->align = (int)k.align;
    g->slice_shift = (int)k.shift;
    g->n_buckets = n_buckets;
    g->slices = sample->slice;
    return true;
}

// A range of a large bucket's keys, moved into tiles of its own: run `digit` of rows row0 .. row0 + rows - 1. Its kept
// keys are segment seg of bucket `bucket`'s chain.
struct SubBucket {
    uint32_t row0, rows, digit, bucket, seg;
};

struct CountArgs {
    uint32_t n_buckets, min_count;
    const SubBucket *sub;                 // the buckets, when they are ranges of large ones (null: those of the levels)
    uint32_t first_extra;                 // first segment that belongs to no bucket (their number without sub)
    uint32_t *retry;                      // null, or where the second kernel lists what it would have to split into more
    unsigned long long *n_retry;          // than a few ranges, and their number (zero)
    int low_bits;                         // bucket-index bits of the second level; -1: one level
    uint32_t row_stride, group;           // second level: rows per first-level bin, first-level tiles per row
    const uint32_t *n_tiles;              // first-level tiles written
    uint32_t max_tiles;
    uint32_t *ticket;                     // two, zero
    uint32_t *large;                      // buckets left to the second kernel, and their number (zero)
    unsigned long long *n_large;
    unsigned long long *n_distinct, *largest;  // += distinct keys; max= keys of one segment
    bool check;                           // a count could reach 2^32 - 1
};

// Windows per bucket aimed at: three quarters of what one CTA's shared memory holds; for plain keys, whose
// buckets' sizes are estimated from a sample, nine sixteenths.
// (Fly-shaped library: 6400 13.2 ms, 5632 and 4864 more, a bucket's fixed cost being spread over fewer keys.)
constexpr uint32_t tile_bucket_windows(int key_words) { return 6400u / (uint32_t)key_words; }
constexpr uint32_t tile_bucket_keys(int key_words) { return 4608u / (uint32_t)key_words; }

// Kept keys of each bucket, unordered: segment b of bucket b, chained to further ones in key order.
struct SegmentTable {
    unsigned long long *at;
    uint32_t *n, *next, *bucket_n;
    uint32_t max_segments;
    uint32_t *n_extra;           // zero
    unsigned long long *cursor;  // zero; keys kept in all
    uint64_t cap;                // room in the temporary arrays
};

template <class K>
void launch_extract_tiles(const LaunchCfg &c, const ExtractArgs &a, const TileGeom &tg, int digit_shift,
                          uint32_t bins, K *out, uint64_t cap, const TileTable &tt, uint32_t *err);
// n plain keys (8-byte aligned) -> tiles; ERR_KEY_FORM when one has bits above key_bits. Keys of all ones, which
// are the tiles' padding, are counted in *n_ones instead.
template <class K>
void launch_array_tiles(const LaunchCfg &c, const uint64_t *keys, uint64_t n, int key_bits, const TileGeom &tg,
                        int digit_shift, uint32_t bins, K *out, uint64_t cap, const TileTable &tt,
                        unsigned long long *n_ones, uint32_t *err);
template <class K>
void launch_sample_keys(const LaunchCfg &c, const uint64_t *keys, uint64_t n, uint32_t n_buckets, KeySample *out);
template <class K>
void launch_regroup_tiles(const LaunchCfg &c, const K *in, const TileTable &t1, uint32_t bins1, uint32_t group,
                          uint32_t groups_max, const TileGeom &tg, uint32_t bins2, K *out, uint64_t cap,
                          const TileTable &t2, uint32_t *err);
// Counts the buckets that fit shared memory and lists the others in a.large, *a.n_large of them. wide_buckets: 128-bit
// keys, more than CS_WIDE_WINDOWS windows a bucket on average, of which the ordinary kernel has room for 4,096 (k = 64,
// four ranges of 240M windows, all of the counting: mean 4,100 11.4 ms wide, 10.1 ordinary and large; 4,550 10.8, 11.2;
// 5,200 10.1, 11.3; 7,000 9.3, 11.1; at 3,200, ordinary, 8.8).
constexpr uint64_t CS_WIDE_WINDOWS = 4300, CS_WIDE_BUCKET = 7000, CS_MAX_WINDOWS = 8192;
template <class K>
void launch_count_small(const LaunchCfg &c, const K *keys, const TileTable &t, const CountArgs &a, bool wide_buckets,
                        K *tmp_keys, uint32_t *tmp_counts, const SegmentTable &seg, uint32_t *err);
// Counts the listed buckets; n_large: at most as many as that. With a.retry not those of many distinct keys.
template <class K>
void launch_count_buckets(const LaunchCfg &c, const K *keys, const TileTable &t, const CountArgs &a, uint64_t n_large,
                          K *tmp_keys, uint32_t *tmp_counts, const SegmentTable &seg, uint32_t *err);
// ---- large buckets in ranges (k_plan_large, k_refine_tiles)
// A large bucket's ranges: `subs` of them; their inner bounds are splitters[spl .. spl + subs - 1); `rows` tiles.
struct LargePlan {
    uint32_t bucket, subs, rows, spl;
};
constexpr uint32_t RF_SLICES = 16;  // the list's sixteenths, whose sizes are added up apart (room for one at a time is enough)
// First list item of a sixteenth.
inline uint32_t refine_first(uint32_t n_list, uint32_t slice) {
    return (uint32_t)(((uint64_t)n_list * slice + RF_SLICES - 1) / RF_SLICES);
}
constexpr uint32_t RF_MAX_SUBS = 1u << TL_MAX_BITS;
constexpr uint32_t refine_keys(int key_words) { return tile_bucket_keys(key_words); }  // keys per range aimed at
struct RefineCounts {  // zero before the plan
    unsigned long long keys[RF_SLICES], rows[RF_SLICES], subs[RF_SLICES];  // keys: with the room for their padding
    unsigned long long n_spl;
    // zero before each k_refine_tiles
    unsigned long long cursor, n_large;
    uint32_t n_tiles, n_subs, ticket[2];
};
template <class K>
void launch_plan_large(const LaunchCfg &c, const K *keys, const TileTable &t, const CountArgs &a, uint32_t n_list,
                       LargePlan *plan, K *splitters, uint32_t splitter_cap, RefineCounts *counts, uint32_t *err);
// List items [first, end): their keys to `out` and the tiles t3 (pitch RF_MAX_SUBS + 1), their ranges to sub[0 ..
// *n_subs) and their buckets' chains.
template <class K>
void launch_refine_tiles(const LaunchCfg &c, const K *in, const TileTable &t, const CountArgs &a, const LargePlan *plan,
                         const K *splitters, uint32_t first, uint32_t end, K *out, uint64_t cap, const TileTable &t3,
                         SubBucket *sub, uint32_t *n_subs, const SegmentTable &seg, uint32_t *err);
// Segments in key order to okeys/ocounts; out_off[b] = first entry of bucket b; largest: of any
// segment; drop: zero bits below the keys, shifted out.
template <class K>
void launch_sort_segments(const LaunchCfg &c, const K *tmp_keys, const uint32_t *tmp_counts, const SegmentTable &seg,
                          uint64_t largest, const unsigned long long *out_off, uint32_t n_buckets, int drop, K *okeys,
                          uint32_t *ocounts, const uint32_t *err);
// out[i] = sum of in[0 .. i), i = 0 .. n; words: scan_many_words(n) zeroed words.
uint64_t scan_many_words(uint32_t n);
void launch_scan_many(const LaunchCfg &c, const uint32_t *in, uint32_t n, unsigned long long *out, uint64_t *words,
                      uint32_t *err);

}  // namespace turtle
