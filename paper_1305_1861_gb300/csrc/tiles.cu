// Direct bucketed sort-and-compact: every valid window's canonical key is grouped by key range
// ("bucket") and counted in shared memory, with no filter, no radix sort and no first-sighting stream.
//
// The paper's filter keeps once-seen k-mers out of the working array so that the array stays small
// (Sec. 2.1.3). This form keeps every key in device memory anyway, so a filter could only save slots in
// a bucket's table, and it would pay for them with one random 32-byte probe per window (a whole DRAM
// line on a miss). What it keeps of the paper is the cache-sized working set of Sec. 2.1.4: keys are
// moved until a bucket fits one CTA's shared memory, and there duplicates are merged.
//
//   k_extract_tiles  windows -> canonical keys, appended to a tile in shared memory; a full tile is
//                    grouped by the leading bits of its keys' bucket index and written out whole
//   k_regroup_tiles  (second level, for more than 2^TL_MAX_BITS buckets) the runs of one leading
//                    value are gathered from a group of tiles, grouped by the remaining bits, written out
//   k_count_small    a bucket's runs are gathered from all its tiles into shared memory and counted there; keys
//                    that reach min_count leave unordered
//   k_count_buckets  the same for buckets that do not fit, in a hash table of their distinct keys
//   k_refine_tiles   moves the keys of buckets whose distinct keys are too many for that into ranges that fit
//   k_sort_segments  each bucket's kept keys are ordered in shared memory and written to their place
//
// Times below are of a fly-shaped library: 30M reads of 100 bases, 2.07G windows, k = 31, 64-bit keys. The form
// before (filter, two radix passes, buckets of 32,768 windows) took 88 ms: pass 1 with its filter 45, radix
// passes 23, buckets 15. This one takes 37: 10.9, 9.2, 13.2 and 1.2 ms for the four kernels, and 1.3 for packing and
// validity. At k = 64 (957M windows, four key ranges) it was 84 ms and is 33.
//
// A tile is written where one atomic reserves room for it, and a row of 16-bit run starts describes
// it, so no kernel needs the sizes of the buckets beforehand (a histogram pass over every key), waits
// for an earlier tile (look-back) or scatters single keys to device memory: every store is a whole tile
// (one bulk copy), every load a run of consecutive keys. Runs start on 16-byte boundaries: a run of
// 64-bit keys with an odd length is padded with the all-ones word, which is no canonical key.
#include <algorithm>

#include "bucket.cuh"
#include "tiles.cuh"

namespace turtle {

namespace {

constexpr int TL_THREADS = TILE_THREADS, TL_WARPS = TL_THREADS / WARP, TL_CTAS = 1024 / TL_THREADS;
constexpr int CT_THREADS = 512, CT_WARPS = CT_THREADS / WARP;
constexpr int TL_MAX_BINS = 1 << TL_MAX_BITS;
constexpr int TL_BPT = TL_MAX_BINS / TL_THREADS;  // bins per thread in a tile's scan
constexpr int TL_RPT = TL_MAX_GROUP / TL_THREADS;  // runs per thread in a gather's scan
constexpr uint32_t TL_NONE = ~0u;

// Keys per tile: 128 bytes of keys per thread.
template <class K> struct TileCfg {
    static constexpr int CAP = 128 * TL_THREADS / (int)sizeof(K);
    static constexpr int ITEMS = CAP / TL_THREADS;
    static constexpr int PER16 = 16 / (int)sizeof(K);  // keys per 16-byte chunk
    static constexpr int BUF = CAP + (PER16 > 1 ? TL_MAX_BINS : 0);  // + one pad key per run
};
static_assert(TileCfg<uint64_t>::CAP == tile_keys(1) && TileCfg<Key128>::CAP == tile_keys(2), "host geometry");

// Exclusive scan of one value per thread over the CTA: one barrier inside (each warp adds up the warps before
// it for itself); the caller's next barrier must come before warp_sums is used again.
template <int WARPS>
__device__ __forceinline__ uint32_t tile_scan(uint32_t v, uint32_t *warp_sums /* WARPS */, uint32_t *total) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(FULL, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    const uint32_t w = lane < WARPS ? warp_sums[lane] : 0u;
    const uint32_t before = __reduce_add_sync(FULL, lane < warp ? w : 0u);
    *total = __reduce_add_sync(FULL, w);
    return before + x - v;
}

template <class K> __device__ __forceinline__ K pad_key();
template <> __device__ __forceinline__ uint64_t pad_key<uint64_t>() { return ~0ull; }
template <> __device__ __forceinline__ Key128 pad_key<Key128>() { return Key128{~0ull, ~0ull}; }
__device__ __forceinline__ bool is_pad(uint64_t k) { return k == ~0ull; }
__device__ __forceinline__ bool is_pad(const Key128 &k) { return (k.hi & k.lo) == ~0ull; }

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp_async_16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_4(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// Bulk copy shared -> global of `bytes` (a multiple of 16, both addresses 16-byte aligned), and its waits.
__device__ __forceinline__ void bulk_store(void *dst, const void *src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)),
                 "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Shared state of one tile, after its keys.
struct TileShared {
    uint32_t cnt[TL_MAX_BINS + 2], start[TL_MAX_BINS];  // cnt[TL_MAX_BINS]: pads (never read)
    uint32_t scan[2 * TL_WARPS];
    uint32_t row, pad;
};

// Group the n keys in s_keys by digit (bins of them, at most TL_MAX_BINS) and write the tile: its run
// starts to the table's row, its keys to out at the row's base, which one atomic on the cursor reserves.
// sh.cnt is zero on entry and a barrier has passed since the keys were written. The order of a run's keys
// carries no meaning, so one shared atomic per key ranks it. The keys sit in registers between the two phases:
// the tile is permuted in place.
// pads: the tile's keys may hold pads, which are left out. Thread 0 calls begin() before the first barrier
// here (it gives the tile's row) and end() after it. The bulk copy may still be reading s_keys on return: thread 0
// waits for it (bulk_wait_read) before a barrier after which they are written again.
template <class K, class D, class F, class G>
__device__ __forceinline__ void write_tile(bool pads, K *s_keys, uint32_t n, uint32_t bins, const D &digit, TileShared &sh,
                                           K *__restrict__ out, uint64_t cap, const TileTable &tt, F &&begin, G &&end,
                                           uint32_t *err) {
    constexpr int ITEMS = TileCfg<K>::ITEMS, PER16 = TileCfg<K>::PER16;
    constexpr uint32_t NO_BIN = (uint32_t)TL_MAX_BINS << 16;
    const uint32_t tid = threadIdx.x;
    uint32_t row0 = 0;
    if (tid == 0) row0 = begin();  // the answers of this atomic and the next are awaited where they are used
    K key[ITEMS];
    uint32_t place[ITEMS];  // bin << 16 | rank inside it; pads count in a bin of their own
#pragma unroll
    for (int i = 0; i < ITEMS; i++) key[i] = s_keys[tid + i * TL_THREADS];
    if (!pads && n > (ITEMS - 1) * TL_THREADS) {  // every thread's first ITEMS - 1 keys exist
#pragma unroll
        for (int i = 0; i < ITEMS; i++) {
            const uint32_t d = i < ITEMS - 1 || tid + i * TL_THREADS < n ? digit(key[i]) : (uint32_t)TL_MAX_BINS;
            place[i] = atomicAdd(&sh.cnt[d], 1u) | (d << 16);
        }
    } else {
#pragma unroll
        for (int i = 0; i < ITEMS; i++) {
            place[i] = NO_BIN;
            if (tid + i * TL_THREADS < n && !(pads && is_pad(key[i]))) {
                const uint32_t d = digit(key[i]);
                place[i] = atomicAdd(&sh.cnt[d], 1u) | (d << 16);
            }
        }
    }
    if (tid == 0) sh.row = row0;
    __syncthreads();
    const uint32_t row = sh.row;
    if (tid == 0) end();
    uint32_t c[TL_BPT], sum = 0, total;  // the thread's bins; bins past `bins` are empty
#pragma unroll
    for (int j = 0; j < TL_BPT; j++) {
        c[j] = sh.cnt[TL_BPT * tid + j];
        sum += (c[j] + PER16 - 1) / PER16 * PER16;
    }
    uint32_t run = tile_scan<TL_WARPS>(sum, sh.scan, &total);
    uint16_t *starts = tt.starts + tile_start_index(tt, row, 0);
#pragma unroll
    for (int j = 0; j < TL_BPT; j++) {
        const uint32_t d = TL_BPT * tid + j;
        sh.start[d] = run;
        if (d <= bins) starts[8 * d] = (uint16_t)run;  // entry `bins` holds the tile's length
        const uint32_t end = run + (c[j] + PER16 - 1) / PER16 * PER16;
        if (run + c[j] < end) s_keys[run + c[j]] = pad_key<K>();
        run = end;
        sh.cnt[d] = 0;  // for the next tile
    }
    unsigned long long base = 0;
    if (tid == 0) {
        if (bins == TL_MAX_BINS) starts[8 * bins] = (uint16_t)total;
        base = atomicAdd(tt.cursor, (unsigned long long)total);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; i++)
        if (place[i] < NO_BIN) s_keys[sh.start[place[i] >> 16] + (place[i] & 0xffffu)] = key[i];
    fence_async_smem();  // this thread's writes of the tile come before the bulk copy that reads them
    __syncthreads();
    if (tid == 0) {
        tt.base[row] = base;
        if (base + total > cap) atomicOr(err, ERR_CAND_OVERFLOW);
        else if (total) bulk_store(out + base, s_keys, total * (uint32_t)sizeof(K));
    }
}

// Keys of one library (no tags) are kept left-aligned in the tiles and the table: the 2k bits at the top of
// the 64- or 128-bit word, zeros below. Shifting all keys alike keeps their order, the window streams
// need no masks before the two strands are compared, and the key's top 31 bits v are a constant shift
// away. Buckets are equal slices of f(v) = v (2^32 - v), which the canonical keys of random sequence fill about
// equally (the map of the key-range parts); the product's high word is fine enough: a part holds 2^24 of its
// values and at most 2^20 buckets.
__device__ __forceinline__ uint32_t top_word(uint64_t key) { return (uint32_t)(key >> 32); }
__device__ __forceinline__ uint32_t top_word(const Key128 &key) { return (uint32_t)(key.hi >> 32); }
template <class K> __device__ __forceinline__ uint32_t f_high(const K &key) {
    const uint32_t v = top_word(key) >> 1;
    return __umulhi(v, 0u - v);
}

// One level's digit of the bucket index: (index >> shift) & mask. Keys are of three kinds: a library's,
// left-aligned; tagged ones of a batch (KEYS_LIB), right-aligned with the tag above them and indexed through the
// library table; plain ones of a caller's array (KEYS_PLAIN), in slices of the span they cover, each with as many
// buckets as a sample says.
enum KeyKind { KEYS_ONE, KEYS_LIB, KEYS_PLAIN };
// Top 32 bits of key << align. A key of more bits than the shift leaves room for (align is a sample's, which need not
// hold the widest key) is above every key that fits: all ones, so that it takes a place past all of theirs.
__device__ __forceinline__ uint32_t top_after(uint64_t key, int align) {  // align < 64
    return key > ~0ull >> align ? ~0u : (uint32_t)(key << align >> 32);
}
__device__ __forceinline__ uint32_t top_after(const Key128 &key, int align) {  // align < 128
    const bool over = align < 64 ? key.hi > ~0ull >> align : key.hi || key.lo > ~0ull >> (align - 64);
    const uint64_t hi = align < 64 ? (key.hi << align) | ((key.lo >> 1) >> (63 - align)) : key.lo << (align - 64);
    return over ? ~0u : (uint32_t)(hi >> 32);
}
__device__ __forceinline__ uint32_t plain_index(uint32_t top, uint32_t lo, uint32_t span, int shift, const uint2 *slices,
                                                uint32_t n_buckets) {
    const uint32_t f = min(max(top, lo) - lo, span);
    const uint2 s = slices[f >> shift];
    return min(s.x + __umulhi(f << (32 - shift), s.y), n_buckets - 1);  // shift >= 1
}
template <class K, KeyKind KIND>
struct TileDigit {
    TileGeom g;
    int shift;
    uint32_t mask;
    // s_slices (plain keys): shared copy of g.slices, complete after the next barrier
    __device__ __forceinline__ TileDigit(const TileGeom &g_, int shift_, uint32_t mask_, uint2 *s_slices = nullptr)
        : g(g_), shift(shift_), mask(mask_) {
        if (KIND == KEYS_PLAIN) {
            for (uint32_t i = threadIdx.x; i < KS_SLICES; i += TL_THREADS) s_slices[i] = g_.slices[i];
            g.slices = s_slices;
        }
    }
    __device__ __forceinline__ uint32_t operator()(const K &key) const {
        uint32_t index;
        if (KIND == KEYS_LIB) {
            index = bucket_of(key, g.lib);
        } else if (KIND == KEYS_PLAIN) {
            index = plain_index(top_after(key, g.align), g.f_lo, g.span, g.slice_shift, g.slices, g.n_buckets);
        } else {
            index = __umulhi(f_high(key) - g.f_lo, g.scale);
        }
        return (index >> shift) & mask;
    }
};

// ---------------------------------------------------------------- extraction
// The canonical keys of the 32 windows that start in one packed word, as shifts of two streams: f is
// the word's bases and the following ones; r is the reverse complement of the same bases, shifted so that
// its low 64 or 128 bits begin with the first window's reverse complement. Window j is then f shifted
// left and r shifted right by 2j bits, constants once the loop over j is unrolled. Both begin at the
// top bit; below their 2k bits come other bases, which cannot decide the comparison unless the window is its
// own reverse complement, when either will do. LIB (batches): keys right-aligned and masked first, so that
// a tag fits above them.
__device__ __forceinline__ uint32_t word_lo(uint64_t x) { return (uint32_t)x; }
__device__ __forceinline__ uint32_t word_hi(uint64_t x) { return (uint32_t)(x >> 32); }
__device__ __forceinline__ uint64_t words(uint32_t hi, uint32_t lo) { return ((uint64_t)hi << 32) | lo; }

template <class K, bool LIB> struct Windows;
template <bool LIB> struct Windows<uint64_t, LIB> {
    static constexpr int SUB = 8;  // windows per lane and step
    uint32_t f[4], r[4];           // 32-bit words, least significant first
    uint32_t mask_hi, mask_lo;
    __device__ __forceinline__ void load(uint64_t a, uint64_t b, int k) {
        const int s = 64 - 2 * k;
        uint64_t f1 = a, f0 = b, r0 = ~rev2(a), r1 = ~rev2(b), mask = ~0ull << s;
        if (LIB) {
            f1 = a >> s;
            f0 = (b >> s) | ((a << 1) << (63 - s));
            mask = ~0ull >> s;
        } else {
            r1 = (r1 << s) | ((r0 >> 1) >> (63 - s));
            r0 <<= s;
        }
        f[3] = word_hi(f1); f[2] = word_lo(f1); f[1] = word_hi(f0); f[0] = word_lo(f0);
        r[0] = word_lo(r0); r[1] = word_hi(r0); r[2] = word_lo(r1); r[3] = word_hi(r1);
        mask_hi = word_hi(mask);
        mask_lo = word_lo(mask);
    }
    __device__ __forceinline__ void step() {  // SUB windows on
#pragma unroll
        for (int i = 3; i > 0; i--) f[i] = __funnelshift_l(f[i - 1], f[i], 2 * SUB);
        f[0] <<= 2 * SUB;
#pragma unroll
        for (int i = 0; i < 3; i++) r[i] = __funnelshift_r(r[i], r[i + 1], 2 * SUB);
        r[3] >>= 2 * SUB;
    }
    __device__ __forceinline__ uint64_t key(int j) const {  // j a constant in [0, SUB)
        uint64_t x = words(__funnelshift_l(f[2], f[3], 2 * j), __funnelshift_l(f[1], f[2], 2 * j));
        uint64_t y = words(__funnelshift_r(r[1], r[2], 2 * j), __funnelshift_r(r[0], r[1], 2 * j));
        const uint64_t m = words(mask_hi, mask_lo);
        if (LIB) {
            x &= m;
            y &= m;
            return x < y ? x : y;
        }
        return (x < y ? x : y) & m;
    }
    // top 32 bits of window j's key (j a constant in [0, 32), no step taken)
    __device__ __forceinline__ uint32_t top(int j) const {
        const uint32_t x = j < 16 ? __funnelshift_l(f[2], f[3], 2 * j) : __funnelshift_l(f[1], f[2], 2 * j - 32);
        const uint32_t y = j < 16 ? __funnelshift_r(r[1], r[2], 2 * j) : __funnelshift_r(r[2], r[3], 2 * j - 32);
        return min(x, y) & mask_hi;
    }
    __device__ __forceinline__ uint64_t key_at(int j) const {  // any j in [0, 32), no step taken
        const bool far = j >= 16;
        const uint32_t a = far ? f[2] : f[3], b = far ? f[1] : f[2], c = far ? f[0] : f[1];
        const uint32_t d = far ? r[1] : r[0], e = far ? r[2] : r[1], g = far ? r[3] : r[2];
        const uint64_t x = words(__funnelshift_l(b, a, 2 * j), __funnelshift_l(c, b, 2 * j));
        const uint64_t y = words(__funnelshift_r(e, g, 2 * j), __funnelshift_r(d, e, 2 * j));
        return (x < y ? x : y) & words(mask_hi, mask_lo);
    }
};
template <bool LIB> struct Windows<Key128, LIB> {
    static constexpr int SUB = 4;
    uint32_t f[6], r[6];
    uint64_t mask_hi, mask_lo;
    __device__ __forceinline__ void load(uint64_t a, uint64_t b, uint64_t c, int k) {
        int s = 128 - 2 * k;  // 0..62; LIB: 0..126 (a mixed batch also keeps short keys in 128 bits)
        uint64_t f2 = a, f1 = b, f0 = c, r0 = ~rev2(a), r1 = ~rev2(b), r2 = ~rev2(c);
        if (LIB) {
            if (s >= 64) {
                f0 = f1;
                f1 = f2;
                f2 = 0;
                s -= 64;
                mask_hi = 0;
                mask_lo = ~0ull >> s;
            } else {
                mask_hi = ~0ull >> s;
                mask_lo = ~0ull;
            }
            f0 = (f0 >> s) | ((f1 << 1) << (63 - s));
            f1 = (f1 >> s) | ((f2 << 1) << (63 - s));
            f2 >>= s;
        } else {
            mask_hi = ~0ull;
            mask_lo = ~0ull << s;
            r2 = (r2 << s) | ((r1 >> 1) >> (63 - s));
            r1 = (r1 << s) | ((r0 >> 1) >> (63 - s));
            r0 <<= s;
        }
        f[5] = word_hi(f2); f[4] = word_lo(f2); f[3] = word_hi(f1);
        f[2] = word_lo(f1); f[1] = word_hi(f0); f[0] = word_lo(f0);
        r[0] = word_lo(r0); r[1] = word_hi(r0); r[2] = word_lo(r1);
        r[3] = word_hi(r1); r[4] = word_lo(r2); r[5] = word_hi(r2);
    }
    __device__ __forceinline__ void step() {
#pragma unroll
        for (int i = 5; i > 0; i--) f[i] = __funnelshift_l(f[i - 1], f[i], 2 * SUB);
        f[0] <<= 2 * SUB;
#pragma unroll
        for (int i = 0; i < 5; i++) r[i] = __funnelshift_r(r[i], r[i + 1], 2 * SUB);
        r[5] >>= 2 * SUB;
    }
    __device__ __forceinline__ Key128 key(int j) const {
        uint64_t fh = words(__funnelshift_l(f[4], f[5], 2 * j), __funnelshift_l(f[3], f[4], 2 * j));
        uint64_t fl = words(__funnelshift_l(f[2], f[3], 2 * j), __funnelshift_l(f[1], f[2], 2 * j));
        uint64_t rh = words(__funnelshift_r(r[3], r[4], 2 * j), __funnelshift_r(r[2], r[3], 2 * j));
        uint64_t rl = words(__funnelshift_r(r[1], r[2], 2 * j), __funnelshift_r(r[0], r[1], 2 * j));
        if (LIB) {
            fh &= mask_hi;
            rh &= mask_hi;
            fl &= mask_lo;
            rl &= mask_lo;
        }
        const bool fwd = fh < rh || (fh == rh && fl < rl);
        return Key128{fwd ? fh : rh, (fwd ? fl : rl) & mask_lo};
    }
    __device__ __forceinline__ uint32_t top(int j) const {
        const uint32_t x = j < 16 ? __funnelshift_l(f[4], f[5], 2 * j) : __funnelshift_l(f[3], f[4], 2 * j - 32);
        const uint32_t y = j < 16 ? __funnelshift_r(r[3], r[4], 2 * j) : __funnelshift_r(r[4], r[5], 2 * j - 32);
        return min(x, y);
    }
    __device__ __forceinline__ Key128 key_at(int j) const {
        const bool far = j >= 16;
        uint32_t a[5], b[5];
#pragma unroll
        for (int i = 0; i < 5; i++) {
            a[i] = far ? f[i] : f[i + 1];
            b[i] = far ? r[i + 1] : r[i];
        }
        const uint64_t fh = words(__funnelshift_l(a[3], a[4], 2 * j), __funnelshift_l(a[2], a[3], 2 * j));
        const uint64_t fl = words(__funnelshift_l(a[1], a[2], 2 * j), __funnelshift_l(a[0], a[1], 2 * j));
        const uint64_t rh = words(__funnelshift_r(b[3], b[4], 2 * j), __funnelshift_r(b[2], b[3], 2 * j));
        const uint64_t rl = words(__funnelshift_r(b[1], b[2], 2 * j), __funnelshift_r(b[0], b[1], 2 * j));
        const bool fwd = fh < rh || (fh == rh && fl < rl);
        return Key128{fwd ? fh : rh, (fwd ? fl : rl) & mask_lo};
    }
};

// Packed words [w_begin, w_end) (32 window starts each) -> tiles. A warp takes 32 words at a time, one per
// lane, and Windows::SUB starts of each per step; it reserves room in the tile for the step's keys and
// appends them. The first warp that finds no room ends the tile (later, larger positions fail as well,
// so the keys below the smallest failed position are exactly the appended ones); the whole CTA then
// writes it, and the warp's step starts the next tile. Tiles are thus full to within one step whatever
// share of the windows is valid or, with PARTED, in the key range.
//
// The step's keys are appended window by window (window j of every lane, then window j + 1): each lane's
// validity bits are spread to one byte per window and summed over the lanes below, so that eight appends
// take one packed scan instead of eight ballots and bit counts, and a window's stores are consecutive.
// A warp's next 32 words are copied to shared memory while it works on the current ones.
//
// Bound by shared memory and the ALUs together: of the peaks, shared-memory wavefronts 61 %, ALU 44 %, issue 51 %;
// DRAM 30 %. 11.0 ms = 1.6 TB/s for the fly-shaped library (13.0 with keys right-aligned and eight ballots
// a step). Two CTAs of 512 threads with 64 KB tiles: tiles of half the size make runs of half the length, which
// cost the next kernel more than twice its time (23.6 against 11.9 ms).
//
// PARTED: a key range takes a fraction of the windows, and building every key to find out which costs more
// than the keys themselves. The range is an interval of the key's top 32 bits, which are the smaller of the
// two strands' (the smaller strand's top bits, or both the same), so eight instructions per window mark the
// windows that count; then each lane takes its marked windows one after the other, at shifts of its own: four
// ranges of 957M windows, k = 64, 14.0 ms in all, against 20 when every key was built.
template <class K, bool LIB, bool PARTED>
__global__ void __launch_bounds__(TL_THREADS, TL_CTAS) k_extract_tiles(ExtractArgs a, TileGeom tg, int digit_shift,
                                                                 uint32_t bins, K *__restrict__ out, uint64_t cap,
                                                                 TileTable tt, uint32_t *err) {
    extern __shared__ __align__(16) unsigned char smem[];
    K *s_keys = reinterpret_cast<K *>(smem);
    TileShared &sh = *reinterpret_cast<TileShared *>(smem + sizeof(K) * TileCfg<K>::BUF);
    __shared__ uint32_t s_fill, s_end;
    __shared__ uint64_t s_lib[LIB ? 65 : 1];
    __shared__ int s_libk[LIB ? 64 : 1];
    __shared__ __align__(16) uint64_t s_p[TL_WARPS][2][36];  // a warp's words and the ones after them; the next
    __shared__ __align__(16) uint32_t s_v[TL_WARPS][2][32];  // their validity bits
    constexpr int SUB = Windows<K, LIB>::SUB, STEPS = 32 / SUB, REGS = SUB / 4;
    constexpr uint32_t CAP = TileCfg<K>::CAP;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const TileDigit<K, LIB ? KEYS_LIB : KEYS_ONE> digit(tg, digit_shift, TL_MAX_BINS - 1);
    for (int i = tid; i < TL_MAX_BINS; i += TL_THREADS) sh.cnt[i] = 0;
    if (LIB) {
        for (int i = tid; i <= a.n_libs; i += TL_THREADS) s_lib[i] = a.lib_starts[i];
        if (a.lib_k)
            for (int i = tid; i < a.n_libs; i += TL_THREADS) s_libk[i] = a.lib_k[i];
    }
    const uint64_t stride = (uint64_t)gridDim.x * TL_WARPS * 32;
    uint64_t w0 = a.w_begin + ((uint64_t)warp * gridDim.x + blockIdx.x) * 32;  // the warp's words: w0 + lane
    // w_begin is a multiple of four words (whole 128-position tiles). P holds at least w_end + 4 words and V32
    // as many; 16-byte pieces that start past the words the windows need are left out.
    auto fetch = [&](uint64_t w, int buf) {
        if (w >= a.w_end) return;
        if (lane < 18) {
            if (w + 2 * lane < a.w_end + 3) cp_async_16(&s_p[warp][buf][2 * lane], a.P + w + 2 * lane);
        } else if (lane < 26) {
            const uint32_t i = 4 * (lane - 18);
            if (w + i < a.w_end) cp_async_16(&s_v[warp][buf][i], a.V32 + w + i);
        }
    };
    Windows<K, LIB> win;
    uint32_t v = 0;
    int k = a.k, lib = 0, sub = STEPS, cur = 1;
    auto load = [&]() {  // the warp's words from buffer cur
        v = w0 + lane < a.w_end ? s_v[warp][cur][lane] : 0u;
        if (LIB) {  // library of the word's first position
            lib = 0;
            int hi = a.n_libs;
            while (hi - lib > 1) {
                const int mid = (lib + hi) >> 1;
                if (s_lib[mid] <= 32 * (w0 + lane)) lib = mid;
                else hi = mid;
            }
            k = a.lib_k ? s_libk[lib] : a.k;  // mixed batches: a word lies in one library
        }
        const uint64_t *p = &s_p[warp][cur][lane];
        if constexpr (sizeof(K) == 8) win.load(p[0], p[1], k);
        else win.load(p[0], p[1], p[2], k);
    };
    fetch(w0, 0);
    if (tid == 0) {
        s_fill = 0;
        s_end = CAP;
    }
    __syncthreads();
    for (;;) {
        bool room = true;
        if (sub < STEPS) {  // resumed in the middle of the words (nothing of them is kept over a tile's writing)
            const uint32_t left = v;
            load();
            if (PARTED) v = left;
            else
                for (int i = 0; i < sub; i++) win.step();
        }
        while (w0 < a.w_end) {
            if (sub >= STEPS) {  // new words
                cur ^= 1;
                cp_async_wait();
                __syncwarp();  // every lane's pieces have landed, and every lane is done with the other buffer
                load();
                fetch(w0 + stride, cur ^ 1);
                sub = 0;
                if (PARTED) {
                    uint32_t in = 0;
#pragma unroll
                    for (int j = 0; j < 32; j++) in |= win.top(j) - a.top_lo < a.top_span ? 1u << j : 0u;
                    v &= in;
                }
            }
            if constexpr (PARTED) {  // the marked windows, up to eight a lane at a time
                for (;;) {
                    const uint32_t mine = min(__popc(v), 8);
                    const uint32_t n = __reduce_add_sync(FULL, mine);
                    if (n == 0) break;
                    uint32_t at = 0;
                    if (lane == 0) {
                        at = atomicAdd(&s_fill, n);
                        if (at + n > CAP) atomicMin(&s_end, at);
                    }
                    at = __shfl_sync(FULL, at, 0);
                    if (at + n > CAP) {
                        room = false;
                        break;
                    }
                    const uint32_t rounds = __reduce_max_sync(FULL, mine);
                    for (uint32_t i = 0; i < rounds; i++) {
                        const bool ok = i < mine;
                        const uint32_t b = __ballot_sync(FULL, ok);
                        if (ok) s_keys[at + __popc(b & lanemask_lt())] = win.key_at(__ffs((int)v) - 1);
                        v &= ok ? v - 1 : ~0u;
                        at += __popc(b);
                    }
                }
                if (room) sub = STEPS;
            } else
            for (; sub < STEPS; sub++) {
                const uint32_t in = (v >> (SUB * sub)) & ((1u << SUB) - 1u);
                uint32_t own[REGS], pos[REGS], n = 0;  // one byte per window
#pragma unroll
                for (int q = 0; q < REGS; q++) {
                    own[q] = (((in >> (4 * q)) & 15u) * 0x00204081u) & 0x01010101u;
                    pos[q] = own[q];
                }
#pragma unroll
                for (int d = 1; d < 32; d <<= 1)
#pragma unroll
                    for (int q = 0; q < REGS; q++) {
                        const uint32_t y = __shfl_up_sync(FULL, pos[q], d);
                        if (lane >= d) pos[q] += y;  // at most 32 per byte
                    }
#pragma unroll
                for (int q = 0; q < REGS; q++) {
                    const uint32_t all = __shfl_sync(FULL, pos[q], 31);
                    pos[q] += all * 0x01010100u + n * 0x01010101u - own[q];  // places below 256: no carries
                    n += (all * 0x01010101u) >> 24;
                }
                if (n) {
                    uint32_t at = 0;
                    if (lane == 0) {
                        at = atomicAdd(&s_fill, n);
                        if (at + n > CAP) atomicMin(&s_end, at);
                    }
                    at = __shfl_sync(FULL, at, 0);
                    if (at + n > CAP) {
                        room = false;
                        break;
                    }
                    K *dst = s_keys + at;
#pragma unroll
                    for (int j = 0; j < SUB; j++) {
                        K key = win.key(j);
                        if ((in >> j) & 1u) {
                            if (LIB) {
                                const uint64_t s = 32 * (w0 + lane) + SUB * sub + j;
                                while (lib + 1 < a.n_libs && s_lib[lib + 1] <= s) lib++;
                                key = add_tag(key, (uint32_t)lib, a.tag_shift);
                            }
                            dst[(pos[j / 4] >> (8 * (j & 3))) & 255u] = key;
                        }
                    }
                }
                win.step();
            }
            if (!room) break;
            w0 += stride;  // sub == STEPS
        }
        const bool more = __syncthreads_or(!room);
        const uint32_t n = min(s_fill, s_end);
        if (n)
            write_tile<K>(false, s_keys, n, bins, digit, sh, out, cap, tt,
                [&] {
                    uint32_t row = atomicAdd(tt.n_tiles, 1u);
                    if (row >= tt.max_tiles) {  // cannot happen: sized for every tile
                        atomicOr(err, ERR_CAND_OVERFLOW);
                        row = 0;
                    }
                    return row;
                },
                [&] {  // every thread has seen n: the next tile may begin
                    s_fill = 0;
                    s_end = CAP;
                },
                err);
        if (!more) break;
        if (tid == 0) bulk_wait_read();
        __syncthreads();
    }
    cp_async_wait();
    if (tid == 0) bulk_wait_all();
}

// Valid windows of each of the 2^part_bits key-range parts (sizes the super-partitions and the shards): a lane
// takes a word's 32 windows, whose parts follow from the top words alone; each warp counts in its own bins. ALU-bound.
constexpr int PC_THREADS = 256, PC_WARPS = PC_THREADS / WARP, PC_PARTS = 64;
template <class K>
__global__ void __launch_bounds__(PC_THREADS) k_part_count(const uint64_t *__restrict__ P,
                                                           const uint32_t *__restrict__ V32, uint64_t n_words, int k,
                                                           int part_bits, unsigned long long *counts) {
    __shared__ uint32_t s_cnt[PC_WARPS][PC_PARTS];
    for (int i = threadIdx.x; i < PC_WARPS * PC_PARTS; i += PC_THREADS) (&s_cnt[0][0])[i] = 0;
    __syncthreads();
    uint32_t *mine = s_cnt[threadIdx.x >> 5];
    for (uint64_t w = blockIdx.x * (uint64_t)PC_THREADS + threadIdx.x; w < n_words; w += (uint64_t)gridDim.x * PC_THREADS) {
        const uint32_t v = __ldg(V32 + w);
        if (!v) continue;
        Windows<K, false> win;
        if constexpr (sizeof(K) == 8) win.load(__ldg(P + w), __ldg(P + w + 1), k);
        else win.load(__ldg(P + w), __ldg(P + w + 1), __ldg(P + w + 2), k);
#pragma unroll
        for (int j = 0; j < 32; j++) {
            const uint32_t t = win.top(j) >> 1;
            if ((v >> j) & 1u) atomicAdd(&mine[__umulhi(t, 0u - t) >> (30 - part_bits)], 1u);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 1 << part_bits; i += PC_THREADS) {
        uint32_t c = 0;
        for (int w = 0; w < PC_WARPS; w++) c += s_cnt[w][i];
        if (c) atomicAdd(&counts[i], (unsigned long long)c);
    }
}

// ---------------------------------------------------------------- a caller's keys
__device__ __forceinline__ uint64_t load_key(const uint64_t *p, uint64_t i, uint64_t) { return __ldcs(p + i); }
__device__ __forceinline__ Key128 load_key(const uint64_t *p, uint64_t i, Key128) {  // 8-byte aligned
    return Key128{__ldcs(p + 2 * i), __ldcs(p + 2 * i + 1)};
}
__device__ __forceinline__ bool above_bits(uint64_t key, int bits) { return bits < 64 && key >> bits; }
__device__ __forceinline__ bool above_bits(const Key128 &key, int bits) {
    return bits < 64 ? key.hi || key.lo >> bits : bits < 128 && key.hi >> (bits - 64);
}

// The array's keys, a tile's worth at a time: loads of the next tile do not wait for the bulk store of the last. The
// same bound as k_extract_tiles' tiles. With the later kernels, 40M 64-bit keys, each four times: 0.98 ms, where
// eight radix passes and a run-length pass took 2.7. Pieces of 512 bytes are dealt to the tiles in turn, so that each
// tile has keys from all over the array: tiles of consecutive keys of a sorted array hold one or two buckets, whose
// runs fill chains of second-level tiles that the counting kernel follows one by one (each four times, sorted: 40M 1.16
// against 2.72 ms, 200M 5.1 against 18.3; in no order: 64-bit keys 0.998 against 0.991, 128-bit ones 1.51 against
// 1.57; pieces of 256 bytes 1.01 and 1.53).
template <class K>
__global__ void __launch_bounds__(TL_THREADS, TL_CTAS) k_array_tiles(const uint64_t *__restrict__ keys, uint64_t n,
                                                                     int key_bits, TileGeom tg, int digit_shift,
                                                                     uint32_t bins, K *__restrict__ out, uint64_t cap,
                                                                     TileTable tt, unsigned long long *n_ones,
                                                                     uint32_t *err) {
    extern __shared__ __align__(16) unsigned char smem[];
    K *s_keys = reinterpret_cast<K *>(smem);
    TileShared &sh = *reinterpret_cast<TileShared *>(smem + sizeof(K) * TileCfg<K>::BUF);
    constexpr int ITEMS = TileCfg<K>::ITEMS;
    const uint32_t tid = threadIdx.x;
    __shared__ uint2 s_slices[KS_SLICES];
    __shared__ uint32_t s_ones;  // keys of all ones in this tile
    const TileDigit<K, KEYS_PLAIN> digit(tg, digit_shift, TL_MAX_BINS - 1, s_slices);
    for (int i = tid; i < TL_MAX_BINS; i += TL_THREADS) sh.cnt[i] = 0;
    if (tid == 0) s_ones = 0;
    bool odd = false;  // a key that this form does not take
    constexpr int PIECE = 512 / (int)sizeof(K), ROWS = PIECE / WARP;
    const uint64_t tiles = (n + TileCfg<K>::CAP - 1) / TileCfg<K>::CAP, pieces = (n + PIECE - 1) / PIECE;
    const uint64_t step = PIECE * TL_WARPS * tiles;
    // a warp takes whole pieces; thread's place in the tile for its i-th key
    const uint32_t at0 = PIECE * (tid / WARP) + tid % WARP;
    auto at = [&](int i) { return at0 + PIECE * TL_WARPS * (i / ROWS) + WARP * (i % ROWS); };
    for (uint64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const uint64_t last = (pieces - 1 - t) / tiles;  // the tile's pieces: t + j tiles, j = 0 .. last
        const uint32_t m = (uint32_t)(PIECE * last + min((uint64_t)PIECE, n - PIECE * (t + last * tiles)));
        const uint64_t from = PIECE * (t + tid / WARP * tiles) + tid % WARP;
        K key[ITEMS];
#pragma unroll
        for (int i = 0; i < ITEMS; i++)
            if (at(i) < m) key[i] = load_key(keys, from + i / ROWS * step + WARP * (i % ROWS), K{});
        if (tid == 0) bulk_wait_read();
        __syncthreads();  // the tile before has left s_keys
#pragma unroll
        for (int i = 0; i < ITEMS; i++)
            if (at(i) < m) {
                odd |= above_bits(key[i], key_bits);
                if (is_pad(key[i])) atomicAdd(&s_ones, 1u);
                s_keys[at(i)] = key[i];
            }
        __syncthreads();
        const uint32_t ones = s_ones;
        // Keys of all ones are counted apart: 64-bit runs are padded with them, so the later steps pass over them;
        // tiles of 128-bit keys, which need no padding, leave them out.
        write_tile<K>(
            sizeof(K) == 16 && ones, s_keys, m, bins, digit, sh, out, cap, tt,
            [&] {
                atomicAdd(tt.n_tiles, 1u);
                return (uint32_t)t;
            },
            [&] {  // (after a barrier that every thread passes with its copy of s_ones)
                if (ones) atomicAdd(n_ones, (unsigned long long)ones);
                s_ones = 0;
            },
            err);
    }
    if (odd) atomicOr(err, ERR_KEY_FORM);
    if (tid == 0) bulk_wait_all();
}

// One CTA looks at up to KS_MAX keys, evenly spaced (KeySample).
constexpr uint32_t KS_MAX = 16384, KS_THREADS = 1024;
template <class K>
__global__ void __launch_bounds__(KS_THREADS) k_sample_keys(const uint64_t *__restrict__ keys, uint64_t n,
                                                           uint32_t n_buckets, uint32_t check_scale, KeySample *out) {
    __shared__ uint32_t s_cnt[KS_CHECK];
    __shared__ uint2 s_slice[KS_SLICES];
    __shared__ uint32_t s_align, s_lo, s_hi, s_crowd;
    constexpr int PER = KS_MAX / KS_THREADS;
    static_assert(KS_CHECK == KS_THREADS, "one counter per thread");
    const uint32_t tid = threadIdx.x;
    // a sixteenth of the keys, 1,024 to KS_MAX, and a power of two
    const int log2m = min(min(63 - __clzll((long long)n), max(59 - __clzll((long long)n), 10)), 31 - __clz((int)KS_MAX));
    const uint32_t m = 1u << log2m;  // sampled keys
    s_cnt[tid] = 0;
    if (tid == 0) {
        s_align = 8 * sizeof(K) - 1;
        s_lo = ~0u;
        s_hi = 0;
        s_crowd = 0;
    }
    __syncthreads();
    K key[PER];
    uint32_t align = 8 * sizeof(K) - 1;  // zero bits above the largest key
#pragma unroll
    for (int i = 0; i < PER; i++) {
        const uint32_t j = tid + i * KS_THREADS;
        if (j < m) {
            key[i] = load_key(keys, sample_place(n, log2m, j), K{});
            uint32_t z;
            if constexpr (sizeof(K) == 8) z = (uint32_t)__clzll((long long)key[i]);
            else z = key[i].hi ? (uint32_t)__clzll((long long)key[i].hi) : 64u + (uint32_t)__clzll((long long)key[i].lo);
            align = min(align, z);
        }
    }
    align = __reduce_min_sync(FULL, align);
    if ((tid & 31) == 0) atomicMin(&s_align, align);
    __syncthreads();
    align = s_align;
    uint32_t lo = ~0u, hi = 0, top[PER];
#pragma unroll
    for (int i = 0; i < PER; i++)
        if (tid + i * KS_THREADS < m) {
            top[i] = top_after(key[i], (int)align);
            lo = min(lo, top[i]);
            hi = max(hi, top[i]);
        }
    lo = __reduce_min_sync(FULL, lo);
    hi = __reduce_max_sync(FULL, hi);
    if ((tid & 31) == 0) {
        atomicMin(&s_lo, lo);
        atomicMax(&s_hi, hi);
    }
    __syncthreads();
    // The array reaches past its sample, by one mean gap between sampled keys at each end: with four gaps of room the
    // keys there don't all join the first and the last bucket. (40M keys, a gap of 2,441: without, one of those two did
    // not fit the counting kernel in 13 of 32 arrays, 1.09 ms instead of 0.99; with it, some bucket in 1 of 32.)
    const uint32_t beyond = log2m > 2 ? (s_hi - s_lo) >> (log2m - 2) : 0u;
    lo = s_lo > beyond ? s_lo - beyond : 0u;
    hi = s_hi < ~beyond ? s_hi + beyond : ~0u;
    const int shift = max(1, 32 - 8 - __clz((int)(hi - lo)));  // (hi - lo) >> shift < KS_SLICES
    static_assert(KS_SLICES == 256, "slices by the top eight bits");
#pragma unroll
    for (int i = 0; i < PER; i++)
        if (tid + i * KS_THREADS < m) atomicAdd(&s_cnt[(top[i] - lo) >> shift], 1u);
    __syncthreads();
    if (tid < WARP) {  // slices' first buckets: n_buckets times the share below of the sample and one key more a slice
        const uint64_t share = ((uint64_t)n_buckets << 32) / (m + KS_SLICES);
        uint32_t below = 0;
        for (uint32_t j = tid * (KS_SLICES / WARP); j < (tid + 1) * (KS_SLICES / WARP); j++) below += s_cnt[j] + 1;
        uint32_t x = below;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(FULL, x, d);
            if ((int)tid >= d) x += y;
        }
        below = x - below;
        for (uint32_t j = tid * (KS_SLICES / WARP); j < (tid + 1) * (KS_SLICES / WARP); j++) {
            const uint32_t a = (uint32_t)(share * below >> 32);
            below += s_cnt[j] + 1;
            const uint32_t e = (uint32_t)(share * below >> 32);
            s_slice[j] = make_uint2(a, e - a);
        }
    }
    __syncthreads();
    if (tid < KS_SLICES) out->slice[tid] = s_slice[tid];
    s_cnt[tid] = 0;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < PER; i++)
        if (tid + i * KS_THREADS < m) {
            const uint32_t b = plain_index(top[i], lo, hi - lo, shift, s_slice, n_buckets);
            atomicAdd(&s_cnt[min(n_buckets < KS_CHECK ? b : __umulhi(b, check_scale), KS_CHECK - 1)], 1u);
        }
    __syncthreads();
    // buckets fewer than the groups: a group is one bucket, which may hold its share of the sample
    const uint32_t share = n_buckets < KS_CHECK ? m / n_buckets : 0u;
    const uint32_t mine = s_cnt[tid] > share ? s_cnt[tid] - share : 0u;
    const uint32_t most = __reduce_max_sync(FULL, mine);
    if ((tid & 31) == 0) atomicMax(&s_crowd, most);
    __syncthreads();
    if (tid == 0) {
        out->n = m;
        out->align = align;
        out->lo = lo;
        out->hi = hi;
        out->shift = (uint32_t)shift;
        out->crowd = s_crowd;
    }
}

// ---------------------------------------------------------------- runs of several tiles as one sequence
// The non-empty runs of a list, in order, as one sequence of 16-byte chunks: run i holds chunks [off[i],
// off[i + 1]) and starts at chunk ptr[i] + off[i] of the keys; off[n .. n + 32] = the total. A warp walks
// its share of the sequence 32 chunks at a time: one load per lane brings the next 32 run ends, each
// marks its place among the 32 chunks, and the marks below a lane's chunk number its run. (Searching on
// from the lane's previous run, one end after the other, cost more than the copies themselves.)
struct RunWalk {
    const uint32_t *off;
    uint32_t x, r0;  // the warp's next chunk and the run it lies in
    // Start at chunk x0 < total; n <= 1024 runs.
    __device__ __forceinline__ RunWalk(const uint32_t *off_, uint32_t n, uint32_t x0) : off(off_), x(x0) {
        const uint32_t lane = threadIdx.x & 31, step = (n + 31) / 32;
        uint32_t i = min(lane * step, n);
        const uint32_t block = __popc(__ballot_sync(FULL, off[i] <= x0)) - 1;  // off[0] = 0; off[n] > x0
        i = min(block * step + lane, n);
        r0 = block * step + __popc(__ballot_sync(FULL, lane < step && off[i] <= x0)) - 1;
    }
    // Run of chunk x + lane (which must lie before the total for the answer to mean anything); moves on.
    __device__ __forceinline__ uint32_t next() {
        const uint32_t lane = threadIdx.x & 31;
        const uint32_t rel = off[r0 + 1 + lane] - x;  // >= 1: run r0 holds chunk x; distinct below the total
        const uint32_t marks = __reduce_or_sync(FULL, rel < 32 ? 1u << rel : 0u);
        const uint32_t run = r0 + __popc(marks & (FULL >> (31 - lane)));
        r0 += __popc(__ballot_sync(FULL, rel <= 32));
        x += 32;
        return run;
    }
};

// Compact list of a CTA's runs, RPT per thread in thread order: len[j] chunks from chunk src[j] of the keys.
// Returns the number of non-empty runs; *total = their chunks. One barrier inside, one needed after.
template <int WARPS, int RPT>
__device__ __forceinline__ uint32_t list_runs(const uint64_t (&src)[RPT], const uint32_t (&len)[RPT], uint64_t *ptr,
                                              uint32_t *off, uint32_t *warp_sums /* 2 WARPS */,
                                              uint32_t *total) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t runs = 0, chunks = 0;
#pragma unroll
    for (int j = 0; j < RPT; j++) {
        runs += len[j] ? 1u : 0u;
        chunks += len[j];
    }
    uint32_t r = runs, c = chunks;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t x = __shfl_up_sync(FULL, r, d), y = __shfl_up_sync(FULL, c, d);
        if (lane >= d) {
            r += x;
            c += y;
        }
    }
    if (lane == 31) {
        warp_sums[warp] = r;
        warp_sums[WARPS + warp] = c;
    }
    __syncthreads();
    const uint32_t wr = lane < WARPS ? warp_sums[lane] : 0u, wc = lane < WARPS ? warp_sums[WARPS + lane] : 0u;
    const uint32_t n = __reduce_add_sync(FULL, wr);
    *total = __reduce_add_sync(FULL, wc);
    uint32_t i = __reduce_add_sync(FULL, lane < warp ? wr : 0u) + r - runs;
    uint32_t o = __reduce_add_sync(FULL, lane < warp ? wc : 0u) + c - chunks;
#pragma unroll
    for (int j = 0; j < RPT; j++)
        if (len[j]) {
            off[i] = o;
            ptr[i] = src[j] - o;
            i++;
            o += len[j];
        }
    if (threadIdx.x <= 32) off[n + threadIdx.x] = *total;
    return n;
}

// ---------------------------------------------------------------- second level
// Unit (bin c, group g): the runs of bin c in tiles [g G, (g + 1) G), at most TL_MAX_GROUP of them, are
// copied into shared memory as one sequence, grouped by the low bits of the bucket index and written
// as tile c * groups_max + g of the second level. A sequence longer than a tile (skewed input)
// continues in further tiles, chained by next[]. Units go through eight groups of a bin, then the next bin:
// the lines that neighbouring bins share and the table lines that eight groups share are still in L2.
// Runs are eight keys long (64 bytes): 9.3 ms = 3.6 TB/s, bound by shared memory (wavefronts 54 %) and the barriers
// of its phases at 32 warps per SM; DRAM moves 16.8 bytes a key, 16 of them keys. 28.7 ms with lanes that
// each searched their own runs, 11.9 before keys were left-aligned and run bounds prefetched.
template <class K, KeyKind KIND>
__global__ void __launch_bounds__(TL_THREADS, TL_CTAS) k_regroup_tiles(const K *__restrict__ in, TileTable t1, uint32_t bins1,
                                                                 uint32_t group, uint32_t groups_max, TileGeom tg,
                                                                 uint32_t bins2, K *__restrict__ out, uint64_t cap,
                                                                 TileTable t2, uint32_t *err) {
    extern __shared__ __align__(16) unsigned char smem[];
    K *s_keys = reinterpret_cast<K *>(smem);
    TileShared &sh = *reinterpret_cast<TileShared *>(smem + sizeof(K) * TileCfg<K>::BUF);
    uint64_t *s_ptr = reinterpret_cast<uint64_t *>(&sh + 1);
    uint32_t *s_off = reinterpret_cast<uint32_t *>(s_ptr + TL_MAX_GROUP);  // TL_MAX_GROUP + 33
    __shared__ uint32_t s_raw[2][TL_THREADS];                     // two 16-bit bounds each
    __shared__ __align__(16) uint64_t s_base[TL_RPT * TL_THREADS];
    static_assert(TL_RPT == 2, "run bounds are staged two tiles a thread");
    const ulonglong2 *in16 = reinterpret_cast<const ulonglong2 *>(in);
    constexpr int PER16 = TileCfg<K>::PER16;
    constexpr uint32_t CAP16 = TileCfg<K>::CAP / PER16;
    const uint32_t tid = threadIdx.x;
    __shared__ uint2 s_slices[KIND == KEYS_PLAIN ? KS_SLICES : 1];
    const TileDigit<K, KIND> digit(tg, 0, bins2 - 1, s_slices);
    for (int i = tid; i < TL_MAX_BINS; i += TL_THREADS) sh.cnt[i] = 0;
    if (tid == 0) sh.row = *(volatile uint32_t *)err & ERR_CAND_OVERFLOW;
    __syncthreads();
    if (sh.row) return;  // the first level had no room for its keys: its tiles are not there
    __syncthreads();
    const uint32_t n_tiles = min(*t1.n_tiles, t1.max_tiles);
    const uint32_t groups = (n_tiles + group - 1) / group;
    const uint64_t units = (uint64_t)((groups + 7) / 8 * 8) * bins1;
    // Unit -> its bin and group; false past the last group (the last eight are only partly there).
    auto locate = [&](uint64_t u, uint32_t &c, uint32_t &g) {
        c = (uint32_t)(u / 8 % bins1);
        g = (uint32_t)(u / 8 / bins1) * 8 + (uint32_t)(u & 7);
        return g < groups;
    };
    // Each thread's run bounds (TL_RPT consecutive tiles) of a unit, copied while the unit before is written.
    // Groups of fewer than eight tiles, whose bounds are not aligned for that, are loaded when needed.
    const bool staged = group % 8 == 0;
    auto fetch = [&](uint64_t u) {
        uint32_t c, g;
        if (!staged || u >= units || !locate(u, c, g)) return;
        const uint32_t t = g * group + TL_RPT * tid;
        if (TL_RPT * tid < group && t < n_tiles) {
            const uint16_t *st = t1.starts + tile_start_index(t1, t, c);
            cp_async_4(&s_raw[0][tid], st);
            cp_async_4(&s_raw[1][tid], st + 8);
            cp_async_16(&s_base[TL_RPT * tid], t1.base + t);
        }
    };
    fetch(blockIdx.x);
    for (uint64_t u = blockIdx.x; u < units; u += gridDim.x) {
        uint32_t g, c;
        if (!locate(u, c, g)) {
            fetch(u + gridDim.x);
            continue;
        }
        const uint32_t n_tile_runs = min(group, n_tiles - g * group);
        uint64_t src[TL_RPT];
        uint32_t len[TL_RPT], total;
        cp_async_wait();  // this thread's bounds
#pragma unroll
        for (int h = 0; h < TL_RPT; h++) {
            const uint32_t i = TL_RPT * tid + h;
            len[h] = 0;
            if (i < n_tile_runs) {
                uint32_t a, b;
                uint64_t base;
                if (staged) {
                    a = s_raw[0][tid] >> (16 * h) & 0xffffu;
                    b = s_raw[1][tid] >> (16 * h) & 0xffffu;
                    base = s_base[i];
                } else {
                    const uint32_t t = g * group + i;
                    const uint16_t *st = t1.starts + tile_start_index(t1, t, c);
                    a = st[0];
                    b = st[8];
                    base = t1.base[t];
                }
                len[h] = (b - a) / PER16;
                src[h] = (base + a) / PER16;
            }
        }
        if (tid == 0) bulk_wait_read();  // the unit before has left s_keys when the next barrier is passed
        const uint32_t n_runs = list_runs<TL_WARPS, TL_RPT>(src, len, s_ptr, s_off, sh.scan, &total);
        uint32_t row = c * groups_max + g;
        __syncthreads();
        fetch(u + gridDim.x);
        for (uint32_t x0 = 0;;) {
            const uint32_t n16 = min(CAP16, total - x0);
            // each warp copies a contiguous share of the chunks
            const uint32_t warp = tid >> 5, x_end = x0 + n16 * (warp + 1) / TL_WARPS, xw = x0 + n16 * warp / TL_WARPS;
            if (xw < x_end) {
                RunWalk walk(s_off, n_runs, xw);
                for (uint32_t x = xw + (tid & 31); walk.x < x_end; x += 32) {
                    const uint32_t run = walk.next();
                    if (x < x_end) cp_async_16(s_keys + (x - x0) * PER16, in16 + s_ptr[run] + x);
                }
            }
            cp_async_wait();
            __syncthreads();
            write_tile<K>(true, s_keys, n16 * PER16, bins2, digit, sh, out, cap, t2, [&] { return row; },
                [&] { t2.next[row] = TL_NONE; }, err);
            x0 += n16;
            if (x0 >= total) break;
            // the sequence goes on in a further tile
            if (tid == 0) {
                uint32_t nx = bins1 * groups_max + atomicAdd(t2.n_tiles, 1u);
                if (nx >= t2.max_tiles) {  // cannot happen: sized for every tile
                    atomicOr(err, ERR_CAND_OVERFLOW);
                    nx = t2.max_tiles - 1;
                }
                t2.next[row] = nx;
                sh.row = nx;
                bulk_wait_read();
            }
            __syncthreads();
            row = sh.row;
        }
    }
    cp_async_wait();
    if (tid == 0) bulk_wait_all();
}

// ---------------------------------------------------------------- counting
typedef unsigned __int128 u128;
__device__ __forceinline__ u128 wide(uint64_t k) { return (u128)k; }
__device__ __forceinline__ u128 wide(const Key128 &k) { return ((u128)k.hi << 64) | (u128)k.lo; }

// Table slots: 12 (64-bit keys) or 20 bytes (128-bit keys) a slot, two CTAs per SM.
template <class K> struct CountCfg;
template <> struct CountCfg<uint64_t> { static constexpr uint32_t SLOTS = 8192; };
template <> struct CountCfg<Key128> { static constexpr uint32_t SLOTS = 5120; };
constexpr uint32_t CT_PROBES = 96;  // probes of one key after which the table counts as full
constexpr uint32_t CT_SPLIT16 = 8192;  // 16-byte chunks of a bucket up to which it is split here: two or three ranges
constexpr int CT_STACK = 136;       // pending key ranges (2 per split level, 128-bit ranges)

__device__ __forceinline__ uint32_t count_hash(uint64_t k) {
    return ((uint32_t)(k >> 32) * 0x85ebca6bu ^ (uint32_t)k) * 0x9e3779b1u;
}
__device__ __forceinline__ uint32_t count_hash(const Key128 &k) {
    const uint32_t a = ((uint32_t)(k.lo >> 32) * 0x85ebca6bu ^ (uint32_t)k.lo) * 0x9e3779b1u;
    const uint32_t b = ((uint32_t)(k.hi >> 32) * 0xc2b2ae35u ^ (uint32_t)k.hi) * 0x27d4eb2fu;
    return (a ^ (b >> 15) ^ b) * 0x9e3779b1u;
}
template <uint32_t SLOTS, class K> __device__ __forceinline__ uint32_t count_slot(const K &k) {
    return __umulhi(count_hash(k), SLOTS);
}
__device__ __forceinline__ uint64_t swap_key(uint64_t *slot, uint64_t desired) {
    return atomicCAS(reinterpret_cast<unsigned long long *>(slot), ~0ull, desired);
}
// 16-byte compare-and-swap against the all-ones key; the low 64 bits of the operand are the word at the
// lower address, Key128::hi.
__device__ __forceinline__ Key128 swap_key(Key128 *slot, const Key128 &desired) {
    uint64_t o0, o1;
    asm volatile(
        "{\n\t.reg .b128 d, c, v;\n\t"
        "mov.b128 c, {%2, %2};\n\t"
        "mov.b128 v, {%3, %4};\n\t"
        "atom.shared.cas.b128 d, [%5], c, v;\n\t"
        "mov.b128 {%0, %1}, d;\n\t}"
        : "=l"(o0), "=l"(o1)
        : "l"(~0ull), "l"(desired.hi), "l"(desired.lo), "r"(smem_u32(slot))
        : "memory");
    return Key128{o0, o1};
}

template <class K> struct CountShared {
    static constexpr uint32_t SLOTS = CountCfg<K>::SLOTS;
    K key[SLOTS];
    uint32_t count[SLOTS];
    uint64_t ptr[CT_THREADS];
    uint32_t off[CT_THREADS + 33];
    u128 lo[CT_STACK], hi[CT_STACK];
    K wmin[CT_WARPS], wmax[CT_WARPS];
    uint32_t scan[2 * CT_WARPS];
    uint32_t full, top, next_item;
    unsigned long long at;
};

template <class K>
__device__ __forceinline__ void count_key(CountShared<K> &sm, const K &key, bool check, uint32_t *err) {
    constexpr uint32_t SLOTS = CountCfg<K>::SLOTS;
    uint32_t h = count_slot<SLOTS>(key);
    for (uint32_t left = CT_PROBES;;) {
        const K old = swap_key(&sm.key[h], key);
        if (is_pad(old) || KeyT<K>::eq(old, key)) break;
        h = h + 1 < SLOTS ? h + 1 : 0;
        if (--left == 0) {
            sm.full = 1;
            return;
        }
    }
    if (check) {
        if (atomicAdd(&sm.count[h], 1u) >= 0xfffffffeu) atomicOr(err, ERR_COUNT_OVERFLOW);
    } else {
        atomicAdd(&sm.count[h], 1u);
    }
}

// One 16-byte chunk of a run: two 64-bit keys or one 128-bit key.
__device__ __forceinline__ void unpack16(const ulonglong2 &v, uint64_t (&k)[2]) {
    k[0] = v.x;
    k[1] = v.y;
}
__device__ __forceinline__ void unpack16(const ulonglong2 &v, Key128 (&k)[1]) { k[0] = Key128{v.x, v.y}; }

// The rows (tiles) that hold bucket b's runs: rows r0 .. r0 + n - 1 and what they chain to, run d of each.
struct BucketRows {
    uint32_t r0, n, d;
};
template <bool SUB = true>  // whether there can be ranges of large buckets
__device__ __forceinline__ BucketRows rows_of(uint32_t b, const CountArgs &a, uint32_t n_rows) {
    if (SUB && a.sub) return BucketRows{a.sub[b].row0, a.sub[b].rows, a.sub[b].digit};
    if (a.low_bits < 0) return BucketRows{0u, n_rows, b};
    return BucketRows{(b >> a.low_bits) * a.row_stride, n_rows, b & ((1u << a.low_bits) - 1u)};
}

// ---- buckets that fit shared memory whole
// The bucket's keys are gathered into shared memory first. The table then needs no keys of its own: a slot is
// one 32-bit word, the place of the key that claimed it and the count so far, so a window costs a 32-bit
// swap, a comparison with the claimer's key and a 32-bit add instead of a swap of the whole key (64-bit
// shared swaps set the pace of a table that holds keys: 21 of its 34 shared wavefronts per 32 keys). Each
// thread walks its 64-bit keys by itself: a key that needs more probes holds up only its own thread, not the
// warp's other keys. Probes go on in steps of the hash's odd low bits: with as many distinct keys as slots (a
// library of nearly unique k-mers) a key still meets few others, where neighbouring slots would run full. A
// bucket with more keys than fit is left to k_count_buckets.
// 13.2 ms = 1.4 TB/s, bound by issue and ALU (50 to 59 %) and the probes' shared wavefronts (36 to 54 %); a table of
// 64-bit keys took 14.8. 512 threads and 8,192 slots, two CTAs per SM: 768 threads 13.3, 1,024 threads 14.5, four CTAs
// of 256 threads and 4,096 slots 15.1 ms; buckets of 4,864 or 5,632 windows instead of 6,400 were slower too.
// WIDE: one CTA of 1,024 threads per SM and twice the room, for 128-bit keys in buckets that are wider because a
// key range has too many windows for ordinary ones: 9.3 ms against 8.8 per 957M keys, but see CS_WIDE_WINDOWS.
constexpr uint32_t CS_IDX_BITS = 13, CS_ONE = 1u << CS_IDX_BITS, CS_EMPTY = ~0u;
template <class K, bool WIDE> struct SmallShared {
    static constexpr int THREADS = WIDE ? 1024 : 512, WARPS = THREADS / WARP;
    static constexpr int RPT = 1024 / THREADS;  // rows per thread and block of rows
    static constexpr int LOG2 = WIDE ? 14 : 13;
    static constexpr uint32_t SLOTS = 1u << LOG2, CAP = (WIDE ? 131072 : 65536) / sizeof(K);
    static_assert(CAP <= CS_ONE, "a key's place fits its bits");
    K key[CAP];
    uint32_t slot[SLOTS];
    uint64_t ptr[RPT * THREADS];
    uint32_t off[RPT * THREADS + 33];
    uint32_t scan[2 * WARPS], kept_scan[WARPS];
    uint32_t next_bucket, stop;
    unsigned long long at;
};

template <class K, bool WIDE, bool SUB>
__global__ void __launch_bounds__(WIDE ? 1024 : 512, WIDE ? 1 : 2) k_count_small(
    const K *__restrict__ keys, TileTable t, CountArgs a, K *__restrict__ tmp_keys, uint32_t *__restrict__ tmp_counts,
    SegmentTable seg, uint32_t *err) {
    extern __shared__ __align__(16) unsigned char smem[];
    using Shared = SmallShared<K, WIDE>;
    Shared &sm = *reinterpret_cast<Shared *>(smem);
    constexpr int CS_THREADS = Shared::THREADS, CS_WARPS = Shared::WARPS, CS_RPT = Shared::RPT, CS_LOG2 = Shared::LOG2;
    constexpr uint32_t CS_SLOTS = Shared::SLOTS;
    constexpr int PER16 = TileCfg<K>::PER16;
    constexpr uint32_t CAP16 = Shared::CAP / PER16, BLOCK = CS_RPT * CS_THREADS;
    constexpr int QUADS = CS_SLOTS / 4 / CS_THREADS;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) sm.stop = *(volatile uint32_t *)err & ERR_CAND_OVERFLOW;
    for (uint32_t i = tid; i < CS_SLOTS; i += CS_THREADS) sm.slot[i] = CS_EMPTY;
    __syncthreads();
    if (sm.stop) return;  // the keys are not all there
    const ulonglong2 *keys16 = reinterpret_cast<const ulonglong2 *>(keys);
    const uint32_t n_tiles = min(*a.n_tiles, a.max_tiles);
    const uint32_t n_rows = a.low_bits < 0 ? n_tiles : (n_tiles + a.group - 1) / a.group;
    uint64_t distinct = 0;
    uint32_t largest = 0;
    // run bounds of the thread's rows, and the rows that continue them
    uint64_t src[CS_RPT];
    uint32_t len[CS_RPT], next[CS_RPT];
    auto fetch_row = [&](int h, uint32_t row, uint32_t d) {
        const uint16_t *st = t.starts + tile_start_index(t, row, d);
        const uint32_t x = st[0], y = st[8];
        src[h] = (t.base[row] + x) / PER16;
        len[h] = (y - x) / PER16;
        next[h] = t.next ? t.next[row] : TL_NONE;
    };
    auto fetch = [&](const BucketRows &br, uint32_t r) {
#pragma unroll
        for (int h = 0; h < CS_RPT; h++) {
            const uint32_t i = r + CS_RPT * tid + h;
            len[h] = 0;
            next[h] = TL_NONE;
            if (i < br.n) fetch_row(h, br.r0 + i, br.d);
        }
    };
    auto continued = [&] {
        bool any = false;
#pragma unroll
        for (int h = 0; h < CS_RPT; h++) any |= next[h] != TL_NONE;
        return any;
    };
    uint32_t b = blockIdx.x, n_runs, listed;  // runs and chunks in the list
    bool fits;
    auto list = [&] {
        n_runs = list_runs<CS_WARPS, CS_RPT>(src, len, sm.ptr, sm.off, sm.scan, &listed);
    };
    bool more;  // some of the listed rows are continued
    fetch(rows_of<SUB>(b, a, n_rows), 0);  // the grid has at most one CTA per bucket
    list();
    more = __syncthreads_or(continued());
    while (b < a.n_buckets) {
        const BucketRows br = rows_of<SUB>(b, a, n_rows);
        uint32_t ticket = 0;
        if (tid == 0) ticket = gridDim.x + atomicAdd(a.ticket, 1u);
        // gather: every row's run d, one after the other; the first rows' runs are listed already
        uint32_t n16 = 0;
        fits = listed <= CAP16;
        for (uint32_t r = 0; fits;) {
            const uint32_t x_end = listed * (warp + 1) / CS_WARPS, xw = listed * warp / CS_WARPS;
            if (xw < x_end) {
                RunWalk walk(sm.off, n_runs, xw);
                for (uint32_t x = xw + lane; walk.x < x_end; x += 32) {
                    const uint32_t run = walk.next();
                    if (x < x_end) cp_async_16(sm.key + (n16 + x) * PER16, keys16 + sm.ptr[run] + x);
                }
            }
            n16 += listed;
            if (more) {
#pragma unroll
                for (int h = 0; h < CS_RPT; h++) {
                    len[h] = 0;
                    if (next[h] != TL_NONE) fetch_row(h, next[h], br.d);
                }
            } else {
                r += BLOCK;
                if (r >= br.n) break;
                fetch(br, r);
            }
            __syncthreads();  // every warp is done with the list
            list();
            more = __syncthreads_or(continued());
            fits = n16 + listed <= CAP16;
        }
        cp_async_wait();
        if (tid == 0) sm.next_bucket = ticket;
        __syncthreads();
        const uint32_t nb = sm.next_bucket;
        fetch(nb < a.n_buckets ? rows_of<SUB>(nb, a, n_rows) : BucketRows{0u, 0u, 0u}, 0);  // the next bucket's, listed below
        if (!fits) {
            if (tid == 0) {
                a.large[atomicAdd(a.n_large, 1ull)] = b;
                if (!SUB) seg.bucket_n[b] = 0;
            }
            list();
            more = __syncthreads_or(continued());
            b = nb;
            continue;
        }
        const uint32_t n = n16 * PER16;
        if constexpr (sizeof(K) == 8) {
            if (tid < n) {
                K key = sm.key[tid];
                uint32_t i = tid, hash = count_hash(key), h = hash >> (32 - CS_LOG2);
#pragma unroll 1
                do {  // one probe of the thread's current key; the warp's threads need not be at the same one
                    bool done = is_pad(key);
                    if (!done) {
                        const uint32_t old = atomicCAS(&sm.slot[h], CS_EMPTY, CS_ONE | i);
                        done = old == CS_EMPTY;
                        if (!done && KeyT<K>::eq(sm.key[old & (CS_ONE - 1)], key)) {
                            atomicAdd(&sm.slot[h], CS_ONE);
                            done = true;
                        }
                    }
                    if (done) {
                        i += CS_THREADS;
                        if (i < n) key = sm.key[i];
                        hash = count_hash(key);
                        h = hash >> (32 - CS_LOG2);
                    } else {
                        h = (h + (hash | 1u)) & (CS_SLOTS - 1);
                    }
                } while (i < n);
            }
        } else {  // half as many keys in as many slots: most need one probe
            for (uint32_t i = tid; i < n; i += CS_THREADS) {
                const K key = sm.key[i];
                const uint32_t hash = count_hash(key);
                uint32_t h = hash >> (32 - CS_LOG2);
                for (;;) {
                    const uint32_t old = atomicCAS(&sm.slot[h], CS_EMPTY, CS_ONE | i);
                    if (old == CS_EMPTY) break;
                    if (KeyT<K>::eq(sm.key[old & (CS_ONE - 1)], key)) {
                        atomicAdd(&sm.slot[h], CS_ONE);
                        break;
                    }
                    h = (h + (hash | 1u)) & (CS_SLOTS - 1);
                }
            }
        }
        __syncthreads();
        // keep count >= min_count: each thread its groups of four slots
        uint4 s4[QUADS];
        uint32_t kept = 0;
#pragma unroll
        for (int q = 0; q < QUADS; q++) {
            s4[q] = reinterpret_cast<const uint4 *>(sm.slot)[q * CS_THREADS + tid];
            const uint32_t s[4] = {s4[q].x, s4[q].y, s4[q].z, s4[q].w};
#pragma unroll
            for (int h = 0; h < 4; h++)
                if (s[h] != CS_EMPTY) kept += 0x10000u + (s[h] >> CS_IDX_BITS >= a.min_count ? 1u : 0u);
            reinterpret_cast<uint4 *>(sm.slot)[q * CS_THREADS + tid] = make_uint4(CS_EMPTY, CS_EMPTY, CS_EMPTY, CS_EMPTY);
        }
        uint32_t total;
        const uint32_t pos = tile_scan<CS_WARPS>(kept, sm.kept_scan, &total) & 0xffffu;
        unsigned long long reserved = 0;
        if (tid == 0) {
            const uint32_t n_kept = total & 0xffffu;
            distinct += total >> 16;
            largest = max(largest, n_kept);
            reserved = atomicAdd(seg.cursor, (unsigned long long)n_kept);  // its answer comes while the list is made
            if (SUB) {  // a link of its bucket's chain
                seg.n[a.sub[b].seg] = n_kept;
                atomicAdd(&seg.bucket_n[a.sub[b].bucket], n_kept);
            } else {
                seg.n[b] = n_kept;
                seg.next[b] = TL_NONE;
                seg.bucket_n[b] = n_kept;
            }
        }
        list();
        if (tid == 0) {
            seg.at[SUB ? a.sub[b].seg : b] = reserved;
            sm.at = reserved;
        }
        more = __syncthreads_or(continued());
        uint64_t at = sm.at + pos;
#pragma unroll
        for (int q = 0; q < QUADS; q++) {
            const uint32_t s[4] = {s4[q].x, s4[q].y, s4[q].z, s4[q].w};
#pragma unroll
            for (int h = 0; h < 4; h++)
                if (s[h] != CS_EMPTY && s[h] >> CS_IDX_BITS >= a.min_count) {
                    if (at < seg.cap) {
                        store_key(tmp_keys + at, sm.key[s[h] & (CS_ONE - 1)]);
                        tmp_counts[at] = s[h] >> CS_IDX_BITS;
                    }
                    at++;
                }
        }
        __syncthreads();
        b = nb;
    }
    if (tid == 0) {
        if (distinct) atomicAdd(a.n_distinct, (unsigned long long)distinct);
        if (largest) atomicMax(a.largest, (unsigned long long)largest);
    }
}

// ---- the other buckets
// One CTA at a time per listed bucket, taken in ticket order. The bucket's runs are gathered from its tiles and
// counted; keys with count >= min_count go, unordered, to tmp at an offset that one atomic reserves. A
// bucket whose distinct keys do not fit the table (a key meets CT_PROBES other keys) is listed in a.retry, or, when it
// is small or there is no such list, split into two
// key ranges, each counted from the runs again; its ranges leave as a chain of segments in key order.
// The table is emptied while it is read out, and the next bucket's run bounds are fetched meanwhile. Reached by
// skewed libraries and wide buckets only: 14.8 ms when it counted all of the fly-shaped library's buckets, bound by
// the 64-bit swaps in shared memory.
template <class K>
__global__ void __launch_bounds__(CT_THREADS, 2) k_count_buckets(const K *__restrict__ keys, TileTable t, CountArgs a,
                                                                 K *__restrict__ tmp_keys,
                                                                 uint32_t *__restrict__ tmp_counts,
                                                                 SegmentTable seg, uint32_t *err) {
    extern __shared__ __align__(16) unsigned char smem[];
    CountShared<K> &sm = *reinterpret_cast<CountShared<K> *>(smem);
    constexpr uint32_t SLOTS = CountCfg<K>::SLOTS;
    constexpr int PER16 = TileCfg<K>::PER16;
    constexpr int QUADS = (SLOTS / 4 + CT_THREADS - 1) / CT_THREADS;  // groups of four slots per thread
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) sm.full = *(volatile uint32_t *)err & ERR_CAND_OVERFLOW;
    __syncthreads();
    if (sm.full) return;  // the keys are not all there
    __syncthreads();
    const uint32_t n_list = (uint32_t)*a.n_large;
    if (blockIdx.x >= n_list) return;
    for (uint32_t i = tid; i < SLOTS; i += CT_THREADS) {
        sm.key[i] = pad_key<K>();
        sm.count[i] = 0;
    }
    const ulonglong2 *keys16 = reinterpret_cast<const ulonglong2 *>(keys);
    const uint32_t n_tiles = min(*a.n_tiles, a.max_tiles);
    const uint32_t n_rows = a.low_bits < 0 ? n_tiles : (n_tiles + a.group - 1) / a.group;
    uint64_t distinct = 0;
    uint32_t largest = 0;
    // bounds of run d in row r
    auto fetch = [&](uint32_t r, uint32_t d, uint64_t &src, uint32_t &len, uint32_t &nx) {
        const uint16_t *st = t.starts + tile_start_index(t, r, d);
        const uint32_t x = st[0], y = st[8];
        src = (t.base[r] + x) / PER16;
        len = (y - x) / PER16;
        nx = t.next ? t.next[r] : TL_NONE;
    };
    uint32_t item = blockIdx.x, b = a.large[item];
    uint64_t p_src = 0;
    uint32_t p_len = 0, p_next = TL_NONE;
    {
        const BucketRows br = rows_of(b, a, n_rows);
        if (tid < br.n) fetch(br.r0 + tid, br.d, p_src, p_len, p_next);
    }
    if (tid == 0) sm.full = 0;
    __syncthreads();
    while (item < n_list) {
        const BucketRows br = rows_of(b, a, n_rows);
        if (tid == 0) {
            sm.next_item = gridDim.x + atomicAdd(a.ticket + 1, 1u);
            sm.top = 1;
            sm.lo[0] = 0;
            sm.hi[0] = ~(u128)0;
        }
        auto fetch_next = [&] {  // the next bucket's run bounds, used after this one is written
            const uint32_t ni = sm.next_item;
            if (ni >= n_list) return;
            const BucketRows nr = rows_of(a.large[ni], a, n_rows);
            p_len = 0;
            p_next = TL_NONE;
            if (tid < nr.n) fetch(nr.r0 + tid, nr.d, p_src, p_len, p_next);
        };
        bool narrowed = false, first_try = true, last = false, counting = true;
        uint64_t seen = 0;  // the bucket's chunks
        uint32_t seg_at = a.sub ? a.sub[b].seg : b;                   // the segment to write next
        const uint32_t after = a.sub ? seg.next[seg_at] : TL_NONE;  // what the chain goes on with after this bucket
        uint32_t bucket_kept = 0;
        __syncthreads();
        while (!last) {
            const uint32_t depth = sm.top;
            const u128 lo = sm.lo[depth - 1], hi = sm.hi[depth - 1];
            const bool whole = lo == 0 && hi == ~(u128)0;
            // every key of the range into the table; `only_span` instead finds the keys' least and greatest
            K mn = pad_key<K>(), mx{};
            auto walk = [&](auto &&take) {
                for (uint32_t r = 0; r < br.n; r += CT_THREADS) {
                    uint64_t src = p_src;
                    uint32_t len = p_len, nx = p_next;
                    if (!(first_try && r == 0)) {
                        len = 0;
                        nx = TL_NONE;
                        if (r + tid < br.n) fetch(br.r0 + r + tid, br.d, src, len, nx);
                    }
                    for (;;) {
                        uint32_t total;
                        const uint64_t src1[1] = {src};
                        const uint32_t len1[1] = {len};
                        const uint32_t n_runs = list_runs<CT_WARPS, 1>(src1, len1, sm.ptr, sm.off, sm.scan, &total);
                        if (first_try) seen += total;
                        __syncthreads();
                        // each warp a contiguous share of the chunks, four loads in flight
                        const uint32_t x_end = (uint32_t)((uint64_t)total * (warp + 1) / CT_WARPS);
                        const uint32_t xw = (uint32_t)((uint64_t)total * warp / CT_WARPS);
                        if (xw < x_end) {
                            RunWalk rw(sm.off, n_runs, xw);
                            uint32_t x = xw + lane;
                            // a full table ends the walk; the warp's lanes, out of step after their probes, agree on it
                            while (rw.x < x_end && !__any_sync(FULL, counting && *(volatile uint32_t *)&sm.full)) {
                                ulonglong2 v[4];
#pragma unroll
                                for (int q = 0; q < 4; q++, x += 32) {
                                    v[q] = make_ulonglong2(~0ull, ~0ull);
                                    if (rw.x < x_end) {
                                        const uint32_t run = rw.next();
                                        if (x < x_end) v[q] = __ldcs(keys16 + sm.ptr[run] + x);
                                    }
                                }
#pragma unroll
                                for (int q = 0; q < 4; q++) {
                                    K kk[PER16];
                                    unpack16(v[q], kk);
#pragma unroll
                                    for (int h = 0; h < PER16; h++)
                                        if (!is_pad(kk[h])) take(kk[h]);
                                }
                            }
                        }
                        const bool chained = nx != TL_NONE;
                        if (!__syncthreads_or(chained)) break;
                        len = 0;
                        if (chained) fetch(nx, br.d, src, len, nx);
                    }
                }
            };
            if (whole)
                walk([&](const K &key) { count_key<K>(sm, key, a.check, err); });
            else
                walk([&](const K &key) {
                    const u128 v = wide(key);
                    if (v >= lo && v <= hi) count_key<K>(sm, key, a.check, err);
                });
            first_try = false;
            __syncthreads();
            if (sm.full) {
                for (uint32_t i = tid; i < SLOTS; i += CT_THREADS) {
                    sm.key[i] = pad_key<K>();
                    sm.count[i] = 0;
                }
                if (a.retry && seen > CT_SPLIT16) {  // left to another kernel
                    __syncthreads();
                    last = true;
                    if (tid == 0) {
                        a.retry[atomicAdd(a.n_retry, 1ull)] = b;
                        sm.full = 0;
                    }
                    fetch_next();
                    continue;
                }
                u128 nlo = lo, nhi = hi;
                if (!narrowed) {  // first split: shrink to the bucket's own key span
                    bool any = false;
                    counting = false;
                    walk([&](const K &key) {
                        if (!any || KeyT<K>::lt(key, mn)) mn = key;
                        if (!any || KeyT<K>::lt(mx, key)) mx = key;
                        any = true;
                    });
                    counting = true;
                    for (int d = 16; d > 0; d >>= 1) {
                        const K x = shfl_down_key(mn, d), y = shfl_down_key(mx, d);
                        if (KeyT<K>::lt(x, mn)) mn = x;
                        if (KeyT<K>::lt(mx, y)) mx = y;
                    }
                    if (lane == 0) {
                        sm.wmin[warp] = mn;
                        sm.wmax[warp] = mx;
                    }
                    __syncthreads();
                    mn = sm.wmin[0];
                    mx = sm.wmax[0];
                    for (int q = 1; q < CT_WARPS; q++) {
                        if (KeyT<K>::lt(sm.wmin[q], mn)) mn = sm.wmin[q];
                        if (KeyT<K>::lt(mx, sm.wmax[q])) mx = sm.wmax[q];
                    }
                    nlo = wide(mn);
                    nhi = wide(mx);
                    narrowed = true;
                }
                __syncthreads();
                if (tid == 0) {
                    sm.full = 0;
                    if (nhi > nlo && depth + 1 <= (uint32_t)CT_STACK) {  // lower half on top
                        const u128 mid = nlo + (nhi - nlo) / 2;
                        sm.lo[depth - 1] = mid + 1;
                        sm.hi[depth - 1] = nhi;
                        sm.lo[depth] = nlo;
                        sm.hi[depth] = mid;
                        sm.top = depth + 1;
                    } else {
                        atomicOr(err, ERR_TABLE_FULL);  // cannot happen: one key is one slot
                        sm.top = depth - 1;
                    }
                }
                __syncthreads();
                last = sm.top == 0;
                continue;
            }
            last = depth == 1;
            if (last) fetch_next();
            // keep count >= min_count: each thread its groups of four slots
            uint4 c4[QUADS];
            uint32_t kept = 0;
#pragma unroll
            for (int q = 0; q < QUADS; q++) {
                const uint32_t i = q * CT_THREADS + tid;
                c4[q] = i < SLOTS / 4 ? reinterpret_cast<const uint4 *>(sm.count)[i] : make_uint4(0, 0, 0, 0);
                const uint32_t c[4] = {c4[q].x, c4[q].y, c4[q].z, c4[q].w};
#pragma unroll
                for (int h = 0; h < 4; h++) kept += (c[h] ? 0x10000u : 0u) + (c[h] >= a.min_count ? 1u : 0u);
            }
            uint32_t total;
            uint32_t pos = tile_scan<CT_WARPS>(kept, sm.scan, &total) & 0xffffu;
            const uint32_t n_kept = total & 0xffffu;
            if (tid == 0) {
                distinct += total >> 16;
                largest = max(largest, n_kept);
                bucket_kept += n_kept;
                if (n_kept || last) {  // a range that keeps nothing needs no segment, unless it ends the chain
                    const unsigned long long at = atomicAdd(seg.cursor, (unsigned long long)n_kept);
                    sm.at = at;
                    seg.at[seg_at] = at;
                    seg.n[seg_at] = n_kept;
                    uint32_t nx = after;
                    if (!last) {
                        nx = a.first_extra + atomicAdd(seg.n_extra, 1u);
                        if (nx >= seg.max_segments) {
                            atomicOr(err, ERR_TABLE_FULL);
                            nx = TL_NONE;
                        }
                    }
                    seg.next[seg_at] = nx;
                    if (!last && nx != TL_NONE) seg_at = nx;
                    if (last && a.sub) atomicAdd(&seg.bucket_n[a.sub[b].bucket], bucket_kept);
                    else if (last) seg.bucket_n[b] = bucket_kept;
                }
                sm.top = depth - 1;
            }
            __syncthreads();
            const uint64_t at = sm.at + pos;
            uint32_t w = 0;
#pragma unroll
            for (int q = 0; q < QUADS; q++) {
                const uint32_t i = q * CT_THREADS + tid;
                const uint32_t c[4] = {c4[q].x, c4[q].y, c4[q].z, c4[q].w};
                if ((c[0] | c[1] | c[2] | c[3]) == 0) continue;
#pragma unroll
                for (int h = 0; h < 4; h++) {
                    if (c[h] == 0) continue;
                    if (c[h] >= a.min_count) {
                        if (at + w < seg.cap) {
                            store_key(tmp_keys + at + w, sm.key[4 * i + h]);
                            tmp_counts[at + w] = c[h];
                        }
                        w++;
                    }
                    sm.key[4 * i + h] = pad_key<K>();
                }
                reinterpret_cast<uint4 *>(sm.count)[i] = make_uint4(0, 0, 0, 0);
            }
            if (!last) __syncthreads();
        }
        item = sm.next_item;
        __syncthreads();
        if (item < n_list) b = a.large[item];
    }
    if (tid == 0) {
        if (distinct) atomicAdd(a.n_distinct, (unsigned long long)distinct);
        if (largest) atomicMax(a.largest, (unsigned long long)largest);
    }
}

// ---- large buckets in ranges
// Sequences of uneven composition (a genome of 20 % G and C) put most of their k-mers into a few of the buckets: 300
// Mbase, k = 31, in buckets of 80,000 windows on average, seen from a window. Halving those by value and walking each
// again per half, as k_count_buckets does, is quadratic: 78 ms a call. Here a sample of a large bucket's own keys
// gives it as many ranges as it needs, its keys move once more, into tiles grouped by range, and k_count_small
// counts the ranges: 9.9 ms (3.7 with equal bases; k = 55 131 and 13; 3 Gbase 1,088 and 90). Tiles and gathers are
// k_regroup_tiles' and bound like it, plus the binary search of each key's range. The splitters are the sample's
// quantiles, so the ranges are about equal whatever the distribution is; a range that one key fills by itself is
// left to k_count_buckets. (k_count_buckets has tried the bucket first: few distinct keys fit its table, however many
// windows they have, and it gives up as soon as they don't.) 200 Mbase at 20 %, k = 31, of 6.0 ms: the try 1.41, the plan
// 0.06, the ranges 1.55, their counts 0.63; the last buckets' CTAs leave the others idle (37 to 40 % of the warps active).
constexpr int PL_THREADS = 256, PL_WARPS = PL_THREADS / WARP;
constexpr uint32_t PL_SAMPLE = 4096, PL_PER_SUB = 16;  // sampled keys: at most, and per range aimed at
template <class K>
__global__ void __launch_bounds__(PL_THREADS) k_plan_large(const K *__restrict__ keys, TileTable t, CountArgs a,
                                                           uint32_t n_list, LargePlan *plan, K *splitters,
                                                           uint32_t splitter_cap, RefineCounts *counts, uint32_t *err) {
    extern __shared__ __align__(16) unsigned char smem[];
    K *s_key = reinterpret_cast<K *>(smem);
    __shared__ unsigned long long s_sum[PL_WARPS];
    __shared__ uint32_t s_spl;
    constexpr int PER16 = TileCfg<K>::PER16;
    constexpr uint32_t CAP16 = TileCfg<K>::CAP / PER16;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t n_tiles = min(*a.n_tiles, a.max_tiles);
    const uint32_t n_rows = a.low_bits < 0 ? n_tiles : (n_tiles + a.group - 1) / a.group;
    for (uint32_t item = blockIdx.x; item < n_list; item += gridDim.x) {
        const uint32_t b = a.large[item];
        const BucketRows br = rows_of(b, a, n_rows);
        // take(first chunk, chunks) for each run of the thread's rows and of what continues them
        auto runs = [&](auto &&take) {
            for (uint32_t r = tid; r < br.n; r += PL_THREADS) {
                for (uint32_t row = br.r0 + r; row != TL_NONE; row = t.next ? t.next[row] : TL_NONE) {
                    const uint16_t *st = t.starts + tile_start_index(t, row, br.d);
                    const uint32_t x = st[0], y = st[8];
                    take((t.base[row] + x) / PER16, (y - x) / PER16);
                }
            }
        };
        unsigned long long mine = 0;
        runs([&](uint64_t, uint32_t len) { mine += len; });
        unsigned long long x = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long y = __shfl_up_sync(FULL, x, d);
            if ((int)lane >= d) x += y;
        }
        if (lane == 31) s_sum[warp] = x;
        __syncthreads();
        unsigned long long n16 = 0;
        x -= mine;  // chunks before the thread's
        for (uint32_t w = 0; w < PL_WARPS; w++) {
            if (w < warp) x += s_sum[w];
            n16 += s_sum[w];
        }
        const uint64_t want = (n16 * PER16 + refine_keys(sizeof(K) / 8) - 1) / refine_keys(sizeof(K) / 8);
        const uint32_t subs = (uint32_t)min(max(want, (uint64_t)2), (uint64_t)RF_MAX_SUBS);
        uint32_t m = PL_PER_SUB;  // sampled keys, a power of two
        while (m < PL_PER_SUB * subs && m < PL_SAMPLE) m *= 2;
        // sample j is the first key of chunk floor(j n16 / m)
        runs([&](uint64_t src, uint32_t len) {
            const uint64_t q1 = ((x + len) * m + n16 - 1) / n16;
            for (uint64_t q = (x * m + n16 - 1) / n16; q < q1; q++) s_key[q] = keys[(src + (q * n16 / m - x)) * PER16];
            x += len;
        });
        __syncthreads();
        for (uint32_t size = 2; size <= m; size <<= 1)
            for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
                for (uint32_t q = tid; q < m / 2; q += PL_THREADS) {
                    const uint32_t i = 2 * q - (q & (stride - 1)), j = i + stride;
                    const bool up = (i & size) == 0;
                    const K k0 = s_key[i], k1 = s_key[j];
                    if (KeyT<K>::lt(k1, k0) == up) {
                        s_key[i] = k1;
                        s_key[j] = k0;
                    }
                }
                __syncthreads();
            }
        if (tid == 0) {
            const uint64_t rows = (n16 + CAP16 - 1) / CAP16, pads = PER16 > 1 ? min((uint64_t)(n16 * PER16), rows * subs) : 0;
            const uint32_t slice = (uint32_t)((uint64_t)item * RF_SLICES / n_list);
            s_spl = (uint32_t)atomicAdd(&counts->n_spl, (unsigned long long)subs);
            if (s_spl + subs > splitter_cap) {  // cannot happen: sized for every key of the level
                atomicOr(err, ERR_CAND_OVERFLOW);
                s_spl = 0;
            }
            plan[item] = LargePlan{b, subs, (uint32_t)rows, s_spl};
            atomicAdd(&counts->keys[slice], n16 * PER16 + pads);
            atomicAdd(&counts->rows[slice], rows);
            atomicAdd(&counts->subs[slice], (unsigned long long)subs);
        }
        __syncthreads();
        for (uint32_t j = tid; j + 1 < subs; j += PL_THREADS) splitters[s_spl + j] = s_key[(uint64_t)(j + 1) * m / subs];
        __syncthreads();
    }
}

// Number of splitters not above the key.
template <class K> struct SplitterDigit {
    const K *spl;
    uint32_t n, top;  // top: the greatest power of two <= n
    __device__ __forceinline__ uint32_t operator()(const K &key) const {
        uint32_t at = 0;
        for (uint32_t step = top; step; step >>= 1)
            if (at + step <= n && !KeyT<K>::lt(key, spl[at + step - 1])) at += step;
        return at;
    }
};

template <class K>
__global__ void __launch_bounds__(TL_THREADS, TL_CTAS) k_refine_tiles(const K *__restrict__ in, TileTable t, CountArgs a,
                                                                const LargePlan *__restrict__ plan,
                                                                const K *__restrict__ splitters, uint32_t first,
                                                                uint32_t end, K *__restrict__ out, uint64_t cap,
                                                                TileTable t3, SubBucket *sub, uint32_t *n_subs,
                                                                SegmentTable seg, uint32_t *err) {
    extern __shared__ __align__(16) unsigned char smem[];
    K *s_keys = reinterpret_cast<K *>(smem);
    K *s_spl = s_keys + TileCfg<K>::BUF;
    TileShared &sh = *reinterpret_cast<TileShared *>(s_spl + RF_MAX_SUBS);
    uint64_t *s_ptr = reinterpret_cast<uint64_t *>(&sh + 1);
    uint32_t *s_off = reinterpret_cast<uint32_t *>(s_ptr + TL_MAX_GROUP);  // TL_MAX_GROUP + 33
    __shared__ uint32_t s_row0, s_sub0, s_seg0, s_stop;
    const ulonglong2 *in16 = reinterpret_cast<const ulonglong2 *>(in);
    constexpr int PER16 = TileCfg<K>::PER16;
    constexpr uint32_t CAP16 = TileCfg<K>::CAP / PER16, BLOCK = TL_RPT * TL_THREADS;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < TL_MAX_BINS; i += TL_THREADS) sh.cnt[i] = 0;
    if (tid == 0) s_stop = *(volatile uint32_t *)err & ERR_CAND_OVERFLOW;
    __syncthreads();
    if (s_stop) return;  // the keys are not all there
    const uint32_t n_tiles = min(*a.n_tiles, a.max_tiles);
    const uint32_t n_rows = a.low_bits < 0 ? n_tiles : (n_tiles + a.group - 1) / a.group;
    for (uint32_t item = first + blockIdx.x; item < end; item += gridDim.x) {
        const LargePlan p = plan[item];
        const BucketRows br = rows_of(p.bucket, a, n_rows);
        for (uint32_t j = tid; j + 1 < p.subs; j += TL_THREADS) s_spl[j] = splitters[p.spl + j];
        if (tid == 0) {
            s_row0 = atomicAdd(t3.n_tiles, p.rows);
            s_sub0 = atomicAdd(n_subs, p.subs);
            s_seg0 = a.first_extra + atomicAdd(seg.n_extra, p.subs);
            if (s_row0 + p.rows > t3.max_tiles || s_seg0 + p.subs > seg.max_segments) {  // cannot happen: sized for all
                atomicOr(err, ERR_CAND_OVERFLOW);
                s_stop = 1;
            }
            bulk_wait_read();
        }
        __syncthreads();
        if (s_stop) break;
        const SplitterDigit<K> digit{s_spl, p.subs - 1, 1u << (31 - __clz((int)(p.subs - 1)))};
        uint64_t src[TL_RPT];
        uint32_t len[TL_RPT], next[TL_RPT];
        auto fetch_row = [&](int h, uint32_t row) {
            const uint16_t *st = t.starts + tile_start_index(t, row, br.d);
            const uint32_t x = st[0], y = st[8];
            src[h] = (t.base[row] + x) / PER16;
            len[h] = (y - x) / PER16;
            next[h] = t.next ? t.next[row] : TL_NONE;
        };
        auto fetch = [&](uint32_t r) {
#pragma unroll
            for (int h = 0; h < TL_RPT; h++) {
                const uint32_t i = r + TL_RPT * tid + h;
                len[h] = 0;
                next[h] = TL_NONE;
                if (i < br.n) fetch_row(h, br.r0 + i);
            }
        };
        uint32_t used = 0, filled = 0;  // tiles written, chunks in the next one
        auto write = [&] {
            cp_async_wait();
            __syncthreads();
            const uint32_t row = s_row0 + min(used, p.rows - 1);
            write_tile<K>(true, s_keys, filled * PER16, p.subs, digit, sh, out, cap, t3, [&] { return row; }, [] {}, err);
            if (used >= p.rows) atomicOr(err, ERR_CAND_OVERFLOW);  // cannot happen
            used++;
            filled = 0;
            if (tid == 0) bulk_wait_read();
            __syncthreads();
        };
        fetch(0);
        for (uint32_t r = 0;;) {
            uint32_t total;
            const uint32_t n_runs = list_runs<TL_WARPS, TL_RPT>(src, len, s_ptr, s_off, sh.scan, &total);
            bool goes_on = false;
#pragma unroll
            for (int h = 0; h < TL_RPT; h++) goes_on |= next[h] != TL_NONE;
            const bool more = __syncthreads_or(goes_on);
            for (uint32_t x0 = 0; x0 < total;) {
                const uint32_t n16 = min(CAP16 - filled, total - x0);
                const uint32_t x_end = x0 + n16 * (warp + 1) / TL_WARPS, xw = x0 + n16 * warp / TL_WARPS;
                if (xw < x_end) {
                    RunWalk walk(s_off, n_runs, xw);
                    for (uint32_t x = xw + lane; walk.x < x_end; x += 32) {
                        const uint32_t run = walk.next();
                        if (x < x_end) cp_async_16(s_keys + (filled + x - x0) * PER16, in16 + s_ptr[run] + x);
                    }
                }
                filled += n16;
                x0 += n16;
                if (filled == CAP16) write();
            }
            if (more) {
#pragma unroll
                for (int h = 0; h < TL_RPT; h++) {
                    len[h] = 0;
                    if (next[h] != TL_NONE) fetch_row(h, next[h]);
                }
            } else {
                r += BLOCK;
                if (r >= br.n) break;
                fetch(r);
            }
            __syncthreads();  // every warp is done with the list
        }
        if (filled) write();
        // the ranges, and the bucket's chain: an empty segment of its own, then one per range
        for (uint32_t j = tid; j < p.subs; j += TL_THREADS) {
            const uint32_t sg = s_seg0 + j;
            sub[s_sub0 + j] = SubBucket{s_row0, min(used, p.rows), j, p.bucket, sg};
            seg.at[sg] = 0;
            seg.n[sg] = 0;
            seg.next[sg] = j + 1 < p.subs ? sg + 1 : TL_NONE;
        }
        if (tid == 0) {
            seg.at[p.bucket] = 0;
            seg.n[p.bucket] = 0;
            seg.next[p.bucket] = s_seg0;
            seg.bucket_n[p.bucket] = 0;
        }
        __syncthreads();
    }
    if (tid == 0) bulk_wait_all();
}

// ---------------------------------------------------------------- output order
__device__ __forceinline__ uint64_t key_diff(uint64_t a, uint64_t b) { return a - b; }
__device__ __forceinline__ u128 key_diff(const Key128 &a, const Key128 &b) { return wide(a) - wide(b); }
__device__ __forceinline__ int key_bits_of(uint64_t x) { return 64 - __clzll((long long)x); }
__device__ __forceinline__ int key_bits_of(u128 x) {
    return (uint64_t)(x >> 64) ? 64 + key_bits_of((uint64_t)(x >> 64)) : key_bits_of((uint64_t)x);
}
__device__ __forceinline__ uint64_t shfl_xor_key(uint64_t k, int d) { return __shfl_xor_sync(FULL, k, d); }
__device__ __forceinline__ Key128 shfl_xor_key(const Key128 &k, int d) {
    return Key128{__shfl_xor_sync(FULL, k.hi, d), __shfl_xor_sync(FULL, k.lo, d)};
}
// The least of the warp's mn and the greatest of its mx, in every lane.
template <class K> __device__ __forceinline__ void warp_span(K &mn, K &mx) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const K x = shfl_xor_key(mn, d), y = shfl_xor_key(mx, d);
        if (KeyT<K>::lt(x, mn)) mn = x;
        if (KeyT<K>::lt(mx, y)) mx = y;
    }
}

// Segment by segment: the n kept keys are spread over n / 2 or more sub-ranges of the segment's own key span (one or two
// keys each for keys that are spread evenly), grouped by sub-range in shared memory, and each key's
// place is its sub-range's start plus the number of smaller keys in it. Keys that crowd into one
// sub-range (more than SS_CROWD) are ordered by a bitonic sort instead. ALU-bound (65 %, issue 70 %): 1.2 ms for 115M
// kept keys and counts (2.3 TB/s).
constexpr uint32_t SS_CROWD = 48;
__device__ __forceinline__ uint64_t right_aligned(uint64_t k, int drop) { return k >> drop; }
__device__ __forceinline__ Key128 right_aligned(const Key128 &k, int drop) {  // drop < 64
    return Key128{k.hi >> drop, (k.lo >> drop) | ((k.hi << 1) << (63 - drop))};
}
template <class K, uint32_t N, uint32_t THREADS>
__global__ void __launch_bounds__(THREADS) k_sort_segments(const K *__restrict__ tmp_keys,
                                                           const uint32_t *__restrict__ tmp_counts, SegmentTable seg,
                                                           const unsigned long long *__restrict__ out_off,
                                                           uint32_t n_buckets, int drop, K *__restrict__ okeys,
                                                           uint32_t *__restrict__ ocounts, const uint32_t *err) {
    extern __shared__ __align__(16) unsigned char smem[];
    // the segments are not all there, or the radix sort takes the keys instead (okeys may be their own buffer)
    if (*err & ~ERR_COUNT_OVERFLOW) return;
    constexpr uint32_t ITEMS = N / THREADS, NW = THREADS / WARP;
    K *s_key = reinterpret_cast<K *>(smem);
    uint32_t *s_cnt = reinterpret_cast<uint32_t *>(s_key + N);  // keys per sub-range; bitonic: N key indices
    uint32_t *s_start = s_cnt + N / 2;
    __shared__ K s_min[NW], s_max[NW];
    __shared__ uint32_t s_scan[NW], s_crowd;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t sg = blockIdx.x, b = sg;
    uint64_t dst = out_off[b], src = seg.at[sg];
    uint32_t n = seg.n[sg], next = seg.next[sg];
    while (b < n_buckets) {
        {
            // the segment after this one, known by the time this one is written
            const bool goes_on = next != TL_NONE;
            const uint32_t b1 = goes_on ? b : b + gridDim.x, sg1 = goes_on ? next : b1;
            uint64_t src1 = 0, dst1 = 0;
            uint32_t n1 = 0, next1 = TL_NONE;
            if (b1 < n_buckets) {
                src1 = seg.at[sg1];
                n1 = seg.n[sg1];
                next1 = seg.next[sg1];
                dst1 = goes_on ? dst + n : out_off[b1];
            }
            auto advance = [&] {
                b = b1;
                src = src1;
                dst = dst1;
                n = n1;
                next = next1;
            };
            if (n == 0) {
                advance();
                continue;
            }
            // sub-ranges: half the power of two >= n, and one per thread at least
            const int log2s = max(31 - __clz((int)n - 1), 31 - __clz((int)THREADS));
            const uint32_t per = 1u << log2s >> (31 - __clz((int)THREADS));  // per thread
            for (uint32_t i = tid; i < 1u << log2s; i += THREADS) s_cnt[i] = 0;
            K key[ITEMS];
            uint32_t cnt[ITEMS];
            K mn = pad_key<K>(), mx{};
#pragma unroll
            for (uint32_t i = 0; i < ITEMS; i++)  // all loads first: one memory latency a segment
                if (tid + i * THREADS < n) {
                    key[i] = tmp_keys[src + tid + i * THREADS];
                    cnt[i] = tmp_counts[src + tid + i * THREADS];
                }
#pragma unroll
            for (uint32_t i = 0; i < ITEMS; i++)
                if (tid + i * THREADS < n) {
                    if (KeyT<K>::lt(key[i], mn)) mn = key[i];
                    if (KeyT<K>::lt(mx, key[i])) mx = key[i];
                }
            warp_span(mn, mx);
            if (lane == 0) {
                s_min[warp] = mn;
                s_max[warp] = mx;
            }
            if (tid == 0) s_crowd = 0;
            __syncthreads();
            mn = s_min[lane % NW];  // every warp adds up the warps' spans for itself
            mx = s_max[lane % NW];
            warp_span(mn, mx);
            const int bits = key_bits_of(key_diff(mx, mn));
            const int shift = bits > log2s ? bits - log2s : 0;
            uint32_t place[ITEMS];  // sub-range | rank inside it << 16
#pragma unroll
            for (uint32_t i = 0; i < ITEMS; i++)
                if (tid + i * THREADS < n) {
                    const uint32_t d = (uint32_t)(key_diff(key[i], mn) >> shift);
                    const uint32_t r = atomicAdd(&s_cnt[d], 1u);
                    if (r >= SS_CROWD) s_crowd = 1;
                    place[i] = d | (r << 16);
                }
            __syncthreads();
            if (!s_crowd) {
                uint32_t sum = 0;
                for (uint32_t i = 0; i < per; i++) sum += s_cnt[tid * per + i];
                uint32_t run = block_exclusive_scan<THREADS>(sum, s_scan, nullptr);
                for (uint32_t i = 0; i < per; i++) {
                    s_start[tid * per + i] = run;
                    run += s_cnt[tid * per + i];
                }
                __syncthreads();
#pragma unroll
                for (uint32_t i = 0; i < ITEMS; i++)
                    if (tid + i * THREADS < n) s_key[s_start[place[i] & 0xffffu] + (place[i] >> 16)] = key[i];
                __syncthreads();
#pragma unroll
                for (uint32_t i = 0; i < ITEMS; i++)
                    if (tid + i * THREADS < n) {
                        const uint32_t d = place[i] & 0xffffu, a = s_start[d], m = s_cnt[d];
                        uint32_t r = 0;
                        for (uint32_t x = 0; x < m; x++) r += KeyT<K>::lt(s_key[a + x], key[i]) ? 1u : 0u;
                        store_key(okeys + dst + a + r, right_aligned(key[i], drop));
                        ocounts[dst + a + r] = cnt[i];
                    }
            } else {
                __syncthreads();  // every thread has seen s_crowd and is done with s_cnt
                uint32_t m = 1;
                while (m < n) m <<= 1;  // <= N
                for (uint32_t i = tid; i < m; i += THREADS) {
                    s_key[i] = i < n ? tmp_keys[src + i] : pad_key<K>();
                    s_cnt[i] = i;
                }
                __syncthreads();
                for (uint32_t size = 2; size <= m; size <<= 1)
                    for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
                        for (uint32_t q = tid; q < m / 2; q += THREADS) {
                            const uint32_t i = 2 * q - (q & (stride - 1)), j = i + stride;
                            const bool up = (i & size) == 0;
                            const K x = s_key[i], y = s_key[j];
                            if (KeyT<K>::lt(y, x) == up) {
                                s_key[i] = y;
                                s_key[j] = x;
                                const uint32_t e = s_cnt[i];
                                s_cnt[i] = s_cnt[j];
                                s_cnt[j] = e;
                            }
                        }
                        __syncthreads();
                    }
                for (uint32_t i = tid; i < n; i += THREADS) {
                    store_key(okeys + dst + i, right_aligned(s_key[i], drop));
                    ocounts[dst + i] = tmp_counts[src + s_cnt[i]];
                }
            }
            __syncthreads();
            advance();
        }
    }
}

// Exclusive scan of n counters by many CTAs (decoupled look-back); out[n] = total. status: one zeroed word
// per 4096 counters, then the ticket word (zeroed).
constexpr int SN_THREADS = 512, SN_ITEMS = 8;
__global__ void __launch_bounds__(SN_THREADS) k_scan_many(const uint32_t *__restrict__ in, uint32_t n,
                                                          unsigned long long *__restrict__ out, uint64_t *status,
                                                          uint32_t *ticket, uint32_t *err) {
    __shared__ uint32_t s_scan[SN_THREADS / WARP], s_tile;
    __shared__ uint64_t s_excl;
    const uint32_t tid = threadIdx.x;
    if (tid == 0) s_tile = atomicAdd(ticket, 1u);  // tiles start in ticket order: look-back always progresses
    __syncthreads();
    const uint32_t tile = s_tile, first = tile * SN_THREADS * SN_ITEMS + tid * SN_ITEMS;
    uint32_t v[SN_ITEMS], sum = 0;
#pragma unroll
    for (int i = 0; i < SN_ITEMS; i++) {
        v[i] = first + i < n ? in[first + i] : 0u;
        sum += v[i];
    }
    uint32_t total;
    const uint32_t mine = block_exclusive_scan<SN_THREADS>(sum, s_scan, &total);
    if (tid < WARP) {
        const uint64_t e = lookback_prefix_warp(status, tile, total, 1, err);
        if (tid == 0) s_excl = e;
    }
    __syncthreads();
    unsigned long long run = s_excl + mine;
#pragma unroll
    for (int i = 0; i < SN_ITEMS; i++) {
        if (first + i < n) out[first + i] = run;
        run += v[i];
        if (first + i + 1 == n) out[n] = run;
    }
}

template <class K> constexpr size_t extract_smem() { return sizeof(K) * TileCfg<K>::BUF + sizeof(TileShared); }
template <class K> constexpr size_t regroup_smem() {
    return extract_smem<K>() + 8 * TL_MAX_GROUP + 4 * (TL_MAX_GROUP + 34);
}
static_assert(sizeof(TileShared) % 8 == 0, "run sources are 8-byte aligned after it");

}  // namespace

template <class K>
void launch_extract_tiles(const LaunchCfg &c, const ExtractArgs &a, const TileGeom &tg, int digit_shift,
                          uint32_t bins, K *out, uint64_t cap, const TileTable &tt, uint32_t *err) {
    if (a.w_begin >= a.w_end) return;
    auto kern = a.n_libs ? k_extract_tiles<K, true, false>  // batches are never split into key ranges
                         : (a.top_span ? k_extract_tiles<K, false, true> : k_extract_tiles<K, false, false>);
    constexpr size_t smem = extract_smem<K>();
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    kern<<<extract_grid(c.sms, a.w_end - a.w_begin), TL_THREADS, smem, c.stream>>>(a, tg, digit_shift, bins, out, cap,
                                                                                  tt, err);
}

template <class K>
void launch_part_count(const LaunchCfg &c, const PackLayout &L, int k, const uint64_t *P, const uint64_t *V,
                       int part_bits, unsigned long long *counts) {
    const uint64_t words = (L.n_bases + 31) / 32;
    const uint64_t need = (words + PC_THREADS - 1) / PC_THREADS, cap = (uint64_t)c.sms * 8;
    k_part_count<K><<<(int)(need < cap ? (need ? need : 1) : cap), PC_THREADS, 0, c.stream>>>(
        P, reinterpret_cast<const uint32_t *>(V), words, k, part_bits, counts);
}

template <class K>
void launch_array_tiles(const LaunchCfg &c, const uint64_t *keys, uint64_t n, int key_bits, const TileGeom &tg,
                        int digit_shift, uint32_t bins, K *out, uint64_t cap, const TileTable &tt,
                        unsigned long long *n_ones, uint32_t *err) {
    constexpr size_t smem = extract_smem<K>();
    cudaFuncSetAttribute(k_array_tiles<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const uint64_t tiles = (n + TileCfg<K>::CAP - 1) / TileCfg<K>::CAP;
    const int grid = (int)std::min<uint64_t>(tiles, (uint64_t)c.sms * TL_CTAS);
    k_array_tiles<K><<<grid, TL_THREADS, smem, c.stream>>>(keys, n, key_bits, tg, digit_shift, bins, out, cap, tt, n_ones,
                                                           err);
}

template <class K>
void launch_sample_keys(const LaunchCfg &c, const uint64_t *keys, uint64_t n, uint32_t n_buckets, KeySample *out) {
    // bucket -> one of KS_CHECK groups: umulhi(bucket, 2^32 KS_CHECK / n_buckets) (n_buckets >= KS_CHECK)
    const uint32_t scale = (uint32_t)std::min<uint64_t>(0xffffffffu, ((uint64_t)KS_CHECK << 32) / n_buckets);
    k_sample_keys<K><<<1, KS_THREADS, 0, c.stream>>>(keys, n, n_buckets, scale, out);
}

template <class K>
void launch_regroup_tiles(const LaunchCfg &c, const K *in, const TileTable &t1, uint32_t bins1, uint32_t group,
                          uint32_t groups_max, const TileGeom &tg, uint32_t bins2, K *out, uint64_t cap,
                          const TileTable &t2, uint32_t *err) {
    constexpr size_t smem = regroup_smem<K>();
    auto kern = tg.lib.lib ? k_regroup_tiles<K, KEYS_LIB>
                : tg.slices ? k_regroup_tiles<K, KEYS_PLAIN>
                            : k_regroup_tiles<K, KEYS_ONE>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const uint64_t units = (uint64_t)groups_max * bins1;
    const int grid = (int)std::min<uint64_t>(units, (uint64_t)c.sms * TL_CTAS);
    kern<<<grid, TL_THREADS, smem, c.stream>>>(in, t1, bins1, group, groups_max, tg, bins2, out, cap, t2, err);
}

template <class K, bool WIDE, bool SUB>
static void count_small_cfg(const LaunchCfg &c, const K *keys, const TileTable &t, const CountArgs &a, K *tmp_keys,
                            uint32_t *tmp_counts, const SegmentTable &seg, uint32_t *err) {
    using Shared = SmallShared<K, WIDE>;
    auto kern = k_count_small<K, WIDE, SUB>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Shared));
    const int grid = (int)std::min<uint64_t>(a.n_buckets, (uint64_t)c.sms * (WIDE ? 1 : 2));
    kern<<<grid, Shared::THREADS, sizeof(Shared), c.stream>>>(keys, t, a, tmp_keys, tmp_counts, seg, err);
}
template <class K>
void launch_count_small(const LaunchCfg &c, const K *keys, const TileTable &t, const CountArgs &a, bool wide_buckets,
                        K *tmp_keys, uint32_t *tmp_counts, const SegmentTable &seg, uint32_t *err) {
    if (a.sub) return count_small_cfg<K, false, true>(c, keys, t, a, tmp_keys, tmp_counts, seg, err);
    if constexpr (sizeof(K) == 16)
        if (wide_buckets) return count_small_cfg<K, true, false>(c, keys, t, a, tmp_keys, tmp_counts, seg, err);
    count_small_cfg<K, false, false>(c, keys, t, a, tmp_keys, tmp_counts, seg, err);
}

template <class K>
void launch_count_buckets(const LaunchCfg &c, const K *keys, const TileTable &t, const CountArgs &a, uint64_t n_large,
                          K *tmp_keys, uint32_t *tmp_counts, const SegmentTable &seg, uint32_t *err) {
    cudaFuncSetAttribute(k_count_buckets<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(CountShared<K>));
    const int grid = (int)std::min<uint64_t>(n_large, (uint64_t)c.sms * 2);
    k_count_buckets<K><<<grid, CT_THREADS, sizeof(CountShared<K>), c.stream>>>(keys, t, a, tmp_keys, tmp_counts, seg,
                                                                             err);
}

template <class K>
void launch_plan_large(const LaunchCfg &c, const K *keys, const TileTable &t, const CountArgs &a, uint32_t n_list,
                       LargePlan *plan, K *splitters, uint32_t splitter_cap, RefineCounts *counts, uint32_t *err) {
    constexpr size_t smem = PL_SAMPLE * sizeof(K);
    cudaFuncSetAttribute(k_plan_large<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const int grid = (int)std::min<uint64_t>(n_list, (uint64_t)c.sms * (sizeof(K) == 8 ? 6 : 3));
    k_plan_large<K><<<grid, PL_THREADS, smem, c.stream>>>(keys, t, a, n_list, plan, splitters, splitter_cap, counts, err);
}

template <class K>
void launch_refine_tiles(const LaunchCfg &c, const K *in, const TileTable &t, const CountArgs &a, const LargePlan *plan,
                         const K *splitters, uint32_t first, uint32_t end, K *out, uint64_t cap, const TileTable &t3,
                         SubBucket *sub, uint32_t *n_subs, const SegmentTable &seg, uint32_t *err) {
    constexpr size_t smem = regroup_smem<K>() + sizeof(K) * RF_MAX_SUBS;
    cudaFuncSetAttribute(k_refine_tiles<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const int grid = (int)std::min<uint64_t>(end - first, (uint64_t)c.sms * TL_CTAS);
    k_refine_tiles<K><<<grid, TL_THREADS, smem, c.stream>>>(in, t, a, plan, splitters, first, end, out, cap, t3, sub, n_subs,
                                                           seg, err);
}

template <class K, uint32_t N, uint32_t THREADS>
static void sort_segments_cfg(const LaunchCfg &c, const K *tmp_keys, const uint32_t *tmp_counts,
                              const SegmentTable &seg, const unsigned long long *out_off, uint32_t n_buckets, int drop,
                              K *okeys, uint32_t *ocounts, const uint32_t *err) {
    constexpr size_t smem = (sizeof(K) + 4) * N;
    auto kern = k_sort_segments<K, N, THREADS>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const int grid = (int)std::min<uint64_t>(n_buckets, (uint64_t)c.sms * 64);
    kern<<<grid, THREADS, smem, c.stream>>>(tmp_keys, tmp_counts, seg, out_off, n_buckets, drop, okeys, ocounts, err);
}

template <class K>
void launch_sort_segments(const LaunchCfg &c, const K *tmp_keys, const uint32_t *tmp_counts, const SegmentTable &seg,
                          uint64_t largest, const unsigned long long *out_off, uint32_t n_buckets, int drop, K *okeys,
                          uint32_t *ocounts, const uint32_t *err) {
    // eight keys a thread whatever the segments' size: fewer threads were slower at each size, and a CTA for segments
    // larger than there are leaves most of its threads idle (up to 512 keys in the form for 1,024: 1.49 against 1.21 ms
    // for 115M 64-bit keys, 2.02 against 1.08 for 52M of 128 bits in segments of 170)
    if (largest && largest <= 256)
        sort_segments_cfg<K, 256, 32>(c, tmp_keys, tmp_counts, seg, out_off, n_buckets, drop, okeys, ocounts, err);
    else if (largest && largest <= 512)
        sort_segments_cfg<K, 512, 64>(c, tmp_keys, tmp_counts, seg, out_off, n_buckets, drop, okeys, ocounts, err);
    else if (largest && largest <= 1024)
        sort_segments_cfg<K, 1024, 128>(c, tmp_keys, tmp_counts, seg, out_off, n_buckets, drop, okeys, ocounts, err);
    else if (largest && largest <= 2048)
        sort_segments_cfg<K, 2048, 256>(c, tmp_keys, tmp_counts, seg, out_off, n_buckets, drop, okeys, ocounts, err);
    else if (largest && largest <= 4096)
        sort_segments_cfg<K, 4096, 512>(c, tmp_keys, tmp_counts, seg, out_off, n_buckets, drop, okeys, ocounts, err);
    else
        sort_segments_cfg<K, 8192, 1024>(c, tmp_keys, tmp_counts, seg, out_off, n_buckets, drop, okeys, ocounts, err);
}
static_assert(CountCfg<uint64_t>::SLOTS <= 8192 && CountCfg<Key128>::SLOTS <= 8192, "a segment fits the largest sort");

uint64_t scan_many_words(uint32_t n) { return (n + SN_THREADS * SN_ITEMS - 1) / (SN_THREADS * SN_ITEMS) + 1; }
void launch_scan_many(const LaunchCfg &c, const uint32_t *in, uint32_t n, unsigned long long *out, uint64_t *words,
                      uint32_t *err) {
    const uint64_t tiles = scan_many_words(n) - 1;
    k_scan_many<<<(int)tiles, SN_THREADS, 0, c.stream>>>(in, n, out, words, reinterpret_cast<uint32_t *>(words + tiles),
                                                         err);
}

#define INST(K)                                                                                                     \
    template void launch_extract_tiles<K>(const LaunchCfg &, const ExtractArgs &, const TileGeom &, int, uint32_t, \
                                          K *, uint64_t, const TileTable &, uint32_t *);                            \
    template void launch_part_count<K>(const LaunchCfg &, const PackLayout &, int, const uint64_t *, const uint64_t *, \
                                       int, unsigned long long *);                                                  \
    template void launch_array_tiles<K>(const LaunchCfg &, const uint64_t *, uint64_t, int, const TileGeom &, int,   \
                                        uint32_t, K *, uint64_t, const TileTable &, unsigned long long *,           \
                                        uint32_t *);                                                                \
    template void launch_sample_keys<K>(const LaunchCfg &, const uint64_t *, uint64_t, uint32_t, KeySample *);      \
    template void launch_regroup_tiles<K>(const LaunchCfg &, const K *, const TileTable &, uint32_t, uint32_t,       \
                                          uint32_t, const TileGeom &, uint32_t, K *, uint64_t, const TileTable &, \
                                          uint32_t *);                                                              \
    template void launch_count_small<K>(const LaunchCfg &, const K *, const TileTable &, const CountArgs &, bool,    \
                                        K *, uint32_t *, const SegmentTable &, uint32_t *);                         \
    template void launch_count_buckets<K>(const LaunchCfg &, const K *, const TileTable &, const CountArgs &,        \
                                          uint64_t, K *, uint32_t *, const SegmentTable &, uint32_t *);             \
    template void launch_plan_large<K>(const LaunchCfg &, const K *, const TileTable &, const CountArgs &, uint32_t, \
                                       LargePlan *, K *, uint32_t, RefineCounts *, uint32_t *);                     \
    template void launch_refine_tiles<K>(const LaunchCfg &, const K *, const TileTable &, const CountArgs &,         \
                                         const LargePlan *, const K *, uint32_t, uint32_t, K *, uint64_t,            \
                                         const TileTable &, SubBucket *, uint32_t *, const SegmentTable &,           \
                                         uint32_t *);                                                                \
    template void launch_sort_segments<K>(const LaunchCfg &, const K *, const uint32_t *, const SegmentTable &,      \
                                          uint64_t, const unsigned long long *, uint32_t, int, K *, uint32_t *,    \
                                          const uint32_t *);
INST(uint64_t)
INST(Key128)
#undef INST

}  // namespace turtle
