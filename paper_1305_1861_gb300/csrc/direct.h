// Host side of the direct bucketed form (tiles.cu): its geometry, its buffers and its launches.
#pragma once
#include <algorithm>
#include <cstdint>

#include "kernels.h"
#include "tiles.cuh"

namespace turtle {

// Buckets the first level's tiles are grouped by directly: a tile of 8,192 keys in 1,024 runs of eight is still gathered
// well; more runs would be shorter than a sector, and a second level (9.3 ms of the fly-shaped library's 37) is cheaper.
constexpr uint32_t ONE_LEVEL_BUCKETS = 1u << TL_MAX_BITS;
constexpr int DIRECT_MAX_BITS = 2 * TL_MAX_BITS;  // bucket-index bits, at most

// Buckets for n keys. A small input gets up to 304 buckets (one for every CTA of the counting kernel) of 512
// keys or more. Past 2^20 buckets they grow: beyond 8,192 64-bit keys (ranges of 8.6G windows) they are counted by the
// second kernel, which the fly-shaped library pays with 37.4 to 39.1 ms in buckets of 8,500 to 16,384 windows
// against 36.4.
inline uint32_t direct_buckets(uint64_t n, uint64_t per_bucket) {
    uint64_t b = (n + per_bucket - 1) / per_bucket;
    b = std::max<uint64_t>(b, std::min<uint64_t>(304, n / 512));
    return (uint32_t)std::min<uint64_t>(std::max<uint64_t>(b, 1), (uint64_t)1 << DIRECT_MAX_BITS);
}

// Windows per bucket: min_count 1 keeps every distinct key, and buckets that keep up to 4,096 are ordered faster (60M
// windows, 37M distinct: 0.46 ms in buckets of 5,600 windows, 0.63 of 6,400; counting takes 0.61 either way).
// 128-bit keys whose ordinary buckets would need all the bits of the second level's index: its runs are four keys
// short then, and fewer, wider buckets gather better, by more the larger the range (k = 64; extraction to order, one
// key range): 4.77G windows 154 against 181 ms, 2.4G 70.4 against 72.3, 1.7G 50.1 against 51.1; at 1.1G and at 0.6G no
// difference, 0.24G 7.71 against 7.66.
// The caller's number (`asked`) holds up to the counting kernel's room. Wider buckets are gathered there in vain, and the
// distinct keys of most libraries overflow the second kernel's tables, so that they are split and walked again: ragged
// reads, k = 55, 4.1 ms by default, 5.5 in buckets of 8,192 windows, 22.2 of 16,384 (the forms with a filter's default)
// and 120 of 65,536; contigs, k = 21, 1.7, 2.0, 8.9 and 31.2.
inline uint64_t direct_bucket_windows(uint32_t asked, int key_words, uint32_t min_count, uint64_t W) {
    if (asked && asked <= CS_MAX_WINDOWS) return asked;
    const uint64_t w = tile_bucket_windows(key_words);
    if (key_words == 2 && W / w >= (uint64_t)1 << (DIRECT_MAX_BITS - 1)) return CS_WIDE_BUCKET;
    return min_count == 1 && key_words == 1 ? w * 7 / 8 : w;
}

// Layout of one key range of at most W keys, in B = tg.n_buckets buckets. Buffers come from `alloc(bytes)`
// (256-byte aligned, or throws); the caller zeroes words[0 .. n_words) before the first launch.
template <class K>
struct Direct {
    static constexpr int KW = sizeof(K) / 8;
    TileGeom tg;
    uint64_t W;
    int low_bits = -1;  // bucket-index bits of the second level; -1: one level
    bool wide_buckets = false;  // of 128-bit keys, more of them than the ordinary counting kernel has room for
    uint32_t bins1, bins2 = 0, group = 1, groups_max = 0, min_count = 1;
    uint64_t tiles, rows = 0, cap1, cap2 = 0, cand_cap, kept_max = 0, n_words;
    TileTable t1{}, t2{};
    SegmentTable seg{};
    K *keys1 = nullptr, *keys2 = nullptr, *tmp_keys = nullptr;
    uint32_t *tmp_counts = nullptr, *large = nullptr;
    unsigned long long *out_off = nullptr;
    unsigned long long *words = nullptr;  // counters, then the output scan's words

    // The first level is written by `launches` launches that end with at most `partial` tiles not full each.
    Direct(const TileGeom &tg_, uint64_t W_, uint64_t launches, uint64_t partial, uint64_t cand_cap_,
           double fill_target = 0.9)
        : tg(tg_), W(W_) {
        const uint32_t cap = tile_keys(KW), B = tg.n_buckets;
        if (B > ONE_LEVEL_BUCKETS) {  // about as many bins on both levels: runs of similar length
            low_bits = 0;
            while (((uint64_t)2 << (2 * low_bits)) <= B) low_bits++;
            low_bits = std::min(low_bits, TL_MAX_BITS);
        }
        bins1 = low_bits < 0 ? B : ((B - 1) >> low_bits) + 1;
        tiles = W / (cap - TL_STEP_KEYS) + launches * partial + 1;
        const uint64_t pad = KW == 1 ? 1 : 0;  // keys a run may be padded by
        cap1 = W + pad * tiles * bins1 + cap;
        cand_cap = cand_cap_ < W ? cand_cap_ : cap1;  // (failure injection: less room)
        t1.pitch = bins1 + 1;
        t1.max_tiles = (uint32_t)tiles;
        n_words = 8 + scan_many_words(B);
        if (low_bits >= 0) {
            bins2 = 1u << low_bits;
            // tiles whose runs of one bin are gathered into one second-level tile: fill_target of a tile's keys
            // on average, so that the usual spread of the bins' sizes rarely needs a second tile
            const double fill = (double)W / ((double)W / cap + (double)(launches * partial));
            const double run = std::max(fill / bins1 + 0.5 * pad, 1e-3);
            group = (uint32_t)std::min<double>(TL_MAX_GROUP, std::max(1.0, fill_target * cap / run));
            if (group > 8) group &= ~7u;  // (the bounds of eight tiles share a sector)
            groups_max = (uint32_t)((tiles + group - 1) / group + 7) & ~7u;
            rows = (uint64_t)bins1 * groups_max + cap1 / cap + 2;
            t2.max_tiles = (uint32_t)rows;
            t2.pitch = bins2 + 1;
            cap2 = W + pad * std::min<uint64_t>(W, rows * bins2) + cap;
        }
    }

    // Buffers of the first level and the tables.
    template <class A>
    void allocate(A &&alloc) {
        keys1 = (K *)alloc(sizeof(K) * cap1);
        words = (unsigned long long *)alloc(8 * n_words);
        t1.cursor = words;
        t1.n_tiles = (uint32_t *)(words + 2);
        t2.cursor = words + 1;
        t2.n_tiles = (uint32_t *)(words + 2) + 1;
        seg.n_extra = (uint32_t *)(words + 3);
        const uint64_t pairs = (tiles + 1) / 2 * 2;  // a gather reads two tiles' first keys at a time
        const uint64_t s1 = tile_start_bytes(tiles, t1.pitch), s2 = rows ? tile_start_bytes(rows, t2.pitch) : 0;
        char *p = (char *)alloc(s1 + s2 + 8 * pairs + 12 * rows);
        t1.starts = (uint16_t *)p;
        t2.starts = (uint16_t *)(p + s1);
        t1.base = (uint64_t *)(p + s1 + s2);
        t2.base = t1.base + pairs;
        t2.next = (uint32_t *)(t2.base + rows);
    }

    // Buffers of the other steps, once the threshold is known; the first level's keys give their place to the
    // kept keys when a second level moves them on.
    template <class A>
    void allocate_rest(uint32_t min_count_, A &&alloc) {
        min_count = min_count_;
        kept_max = W / min_count;
        if (low_bits >= 0) keys2 = (K *)alloc(sizeof(K) * cap2);
        tmp_keys = low_bits >= 0 ? keys1 : (K *)alloc(sizeof(K) * (kept_max + 1));
        tmp_counts = (uint32_t *)alloc(4 * (kept_max + 1));
        const uint64_t B = tg.n_buckets;
        seg.max_segments = (uint32_t)std::min<uint64_t>(B + W / 64 + 1024, 0x7fffffffu);
        out_off = (unsigned long long *)alloc(8 * (B + 1) + 16 * (uint64_t)seg.max_segments + 8 * B);
        seg.at = out_off + B + 1;
        seg.n = (uint32_t *)(seg.at + seg.max_segments);
        seg.next = seg.n + seg.max_segments;
        seg.bucket_n = seg.next + seg.max_segments;
        large = seg.bucket_n + B;
        seg.cap = kept_max + 1;
    }

    // `windows`, by estimate, in buckets of per_bucket or, when they are too many for that, more.
    void choose_width(uint64_t windows, uint64_t per_bucket) {
        wide_buckets = KW == 2 && std::max(per_bucket, windows >> DIRECT_MAX_BITS) > CS_WIDE_WINDOWS;
    }
    int digit_shift() const { return low_bits < 0 ? 0 : low_bits; }
    void extract(const LaunchCfg &lc, const ExtractArgs &a, uint32_t *err) const {
        launch_extract_tiles<K>(lc, a, tg, digit_shift(), bins1, keys1, cand_cap, t1, err);
    }
    void regroup(const LaunchCfg &lc, uint32_t *err) const {
        if (low_bits >= 0)
            launch_regroup_tiles<K>(lc, keys1, t1, bins1, group, groups_max, tg, bins2, keys2, cap2, t2, err);
    }
    // Counts and the threshold: *kept (zero) += kept keys, *distinct += distinct keys, *largest max= keys of one
    // segment, *n_large (zero) = buckets left to count_large.
    CountArgs count_args(unsigned long long *kept, unsigned long long *distinct, unsigned long long *largest,
                         unsigned long long *n_large) {
        seg.cursor = kept;
        CountArgs a{};
        a.n_buckets = a.first_extra = tg.n_buckets;
        a.min_count = min_count;
        a.low_bits = low_bits;
        a.row_stride = groups_max;
        a.group = group;
        a.n_tiles = t1.n_tiles;
        a.max_tiles = t1.max_tiles;
        a.ticket = (uint32_t *)(words + 4);
        a.large = large;
        a.n_large = n_large;
        a.n_distinct = distinct;
        a.largest = largest;
        a.check = W >= 0xfffffffeull;
        return a;
    }
    void count(const LaunchCfg &lc, const CountArgs &a, uint32_t *err) const {
        launch_count_small<K>(lc, low_bits < 0 ? keys1 : keys2, low_bits < 0 ? t1 : t2, a, wide_buckets, tmp_keys,
                              tmp_counts, seg, err);
    }
    const K *counted_keys() const { return low_bits < 0 ? keys1 : keys2; }
    const TileTable &counted_tiles() const { return low_bits < 0 ? t1 : t2; }
    // n_large: buckets listed, or n_buckets when the host does not know.
    void count_large(const LaunchCfg &lc, const CountArgs &a, uint64_t n_large, uint32_t *err) const {
        launch_count_buckets<K>(lc, low_bits < 0 ? keys1 : keys2, low_bits < 0 ? t1 : t2, a, n_large, tmp_keys, tmp_counts,
                                seg, err);
    }
    // The buckets' places in the output.
    void place(const LaunchCfg &lc, uint32_t *err) const {
        launch_scan_many(lc, seg.bucket_n, tg.n_buckets, out_off, (uint64_t *)(words + 8), err);
    }
    // After order() of a caller's keys: the key of all ones, which comes last, and its count (the low word of
    // *n_ones).
    cudaError_t append_ones(cudaStream_t s, uint64_t at, const unsigned long long *n_ones, K *okeys, uint32_t *ocounts) const {
        const cudaError_t e = cudaMemsetAsync(okeys + at, 0xff, sizeof(K), s);
        return e != cudaSuccess ? e : cudaMemcpyAsync(ocounts + at, n_ones, 4, cudaMemcpyDeviceToDevice, s);
    }
    // The kept keys in order. largest: of any segment (0: not known to the host).
    void order(const LaunchCfg &lc, uint64_t largest, int drop, K *okeys, uint32_t *ocounts, const uint32_t *err) const {
        launch_sort_segments<K>(lc, tmp_keys, tmp_counts, seg, largest, out_off, tg.n_buckets, drop, okeys, ocounts, err);
    }
};

}  // namespace turtle
