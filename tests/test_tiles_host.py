"""Host side of counting and sorting by tiles (csrc/direct.h, csrc/tiles.cuh), on the CPU: a C++ program compiled
against the headers lays out tables and looks at what the launches would be given."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = """
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <vector>
#include <cuda_runtime.h>
namespace turtle { struct alignas(16) Key128 { uint64_t hi, lo; }; }
#include "direct.h"
using namespace turtle;
namespace turtle {
uint64_t scan_many_words(uint32_t n) { return (n + 4095) / 4096 + 1; }
}
"""


def _run(tmp_path, body):
    if not shutil.which("g++"):
        pytest.skip("no C++ compiler")
    cuda = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))
    src, exe = tmp_path / "host.cpp", tmp_path / "host"
    src.write_text(HEAD + body)
    subprocess.run(["g++", "-std=c++20", "-O1", "-I", os.path.join(ROOT, "paper_1305_1861_gb300", "csrc"), "-I",
                    os.path.join(cuda, "include"), str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()


# Every table inside its allocation, none over another, over numbers of windows and tiles (odd and even), buckets on
# both sides of one level, and thresholds.
TABLES = """
static std::map<uint64_t, uint64_t> blocks;  // allocation -> bytes
static uint64_t top = 1 << 20;
static void *take(uint64_t bytes) {
    void *p = (void *)top;
    blocks[top] = bytes;
    top += (bytes + 511) / 256 * 256;
    return p;
}
static int bad = 0, odd_two_levels = 0;
struct Span { uint64_t a, n, align; };
template <class K> void look(uint64_t W, uint32_t B, uint64_t launches, uint64_t partial, uint32_t min_count) {
    blocks.clear();
    TileGeom tg{};
    tg.n_buckets = B;
    Direct<K> d(tg, W, launches, partial, W);
    d.allocate(take);
    d.allocate_rest(min_count, take);
    std::vector<Span> s = {
        {(uint64_t)d.keys1, sizeof(K) * d.cap1, 16},
        {(uint64_t)d.words, 8 * (8 + scan_many_words(B)), 8},
        {(uint64_t)d.t1.starts, 16 * ((d.tiles + 7) / 8) * d.t1.pitch, 16},
        {(uint64_t)d.t1.base, 8 * ((d.tiles + 1) / 2 * 2), 16},  // read in pairs
        {(uint64_t)d.tmp_counts, 4 * d.seg.cap, 4},
        {(uint64_t)d.out_off, 8 * ((uint64_t)B + 1), 8},
        {(uint64_t)d.seg.at, 8ull * d.seg.max_segments, 8},
        {(uint64_t)d.seg.n, 4ull * d.seg.max_segments, 4},
        {(uint64_t)d.seg.next, 4ull * d.seg.max_segments, 4},
        {(uint64_t)d.seg.bucket_n, 4ull * B, 4},
        {(uint64_t)d.large, 4ull * B, 4}};
    if (d.low_bits >= 0) {
        odd_two_levels += d.tiles & 1;
        s.push_back({(uint64_t)d.keys2, sizeof(K) * d.cap2, 16});
        s.push_back({(uint64_t)d.t2.starts, 16 * ((d.rows + 7) / 8) * d.t2.pitch, 16});
        s.push_back({(uint64_t)d.t2.base, 8 * d.rows, 8});
        s.push_back({(uint64_t)d.t2.next, 4 * d.rows, 4});
    } else {
        s.push_back({(uint64_t)d.tmp_keys, sizeof(K) * d.seg.cap, 16});
    }
    for (size_t i = 0; i < s.size(); i++) {
        auto it = blocks.upper_bound(s[i].a);
        bool ok = it != blocks.begin() && s[i].a % s[i].align == 0;
        if (ok) --it, ok = s[i].a + s[i].n <= it->first + it->second;
        for (size_t j = 0; j < i; j++) ok &= s[i].a >= s[j].a + s[j].n || s[j].a >= s[i].a + s[i].n;
        if (!ok && bad++ < 5)
            fprintf(stderr, "span %zu W %llu B %u tiles %llu\\n", i, (unsigned long long)W, B, (unsigned long long)d.tiles);
    }
}
int main() {
    srand(1);
    const uint64_t Ws[] = {1, 255, 8193, 100003, 6553600, 6553601, 6561537, 13107200, 33554432, 240000000, 2070000000, 9000000000};
    for (uint64_t W0 : Ws)
        for (int i = 0; i < 64; i++) {
            const uint64_t W = W0 + (i ? rand() % (W0 / 4 + 1) : 0);
            for (uint32_t B : {direct_buckets(W, 6400), direct_buckets(W, 3200), 1024u, 1025u, 1u << 20})
                for (uint64_t l : {1, 9})
                    look<uint64_t>(W, B, l, 1 + i % 304, 1 + i % 3), look<Key128>(W, B, l, 1 + i % 304, 1 + i % 3);
        }
    printf("%d %d\\n", bad, odd_two_levels > 0);
}
"""


def test_tables_lie_inside_their_allocations(tmp_path):
    assert _run(tmp_path, TABLES) == ["0", "1"]


# The sampled places are distinct and evenly spread: no gap, the one to the array's end among them, is more than a key
# longer than another.
PLACES = """
int main() {
    int bad = 0;
    for (uint64_t n : {1024ull, 1025ull, 2047ull, 5119ull, 32767ull, 278527ull, 40000003ull, 9000000000ull, 1ull << 40})
        for (int log2m = 10; log2m <= 14 && n >> log2m; log2m++) {
            const uint64_t m = 1ull << log2m;
            bool ok = sample_place(n, log2m, 0) == 0;
            for (uint64_t j = 0; j < m; j++) {
                const uint64_t gap = (j + 1 < m ? sample_place(n, log2m, j + 1) : n) - sample_place(n, log2m, j);
                ok &= gap == n / m || gap == n / m + 1;
            }
            bad += !ok;
        }
    printf("%d\\n", bad);
}
"""


def test_the_sample_spans_the_array(tmp_path):
    assert _run(tmp_path, PLACES) == ["0"]


# Keys go by tiles when the widest sampled one (leading zeros `align`) has no bits above key_bits, and to the radix sort
# otherwise; a crowded sample goes there either way.
WIDTHS = """
int main() {
    int bad = 0;
    for (int words : {1, 2})
        for (int bits : {1, 16, 40, 62, 63, 64, 65, 110, 128}) {
            if (bits > 64 * words) continue;
            for (int widest = 1; widest <= 64 * words; widest++) {
                KeySample k{};
                TileGeom g{};
                k.n = 16384;
                k.align = 64 * words - widest;
                k.shift = 1;
                bad += sample_geom(k, &k, 100, words, bits, &g) != (widest <= bits);
                k.crowd = 97;
                bad += sample_geom(k, &k, 100, words, bits, &g);
            }
        }
    printf("%d\\n", bad);
}
"""


def test_keys_wider_than_key_bits_go_to_the_radix_sort(tmp_path):
    assert _run(tmp_path, WIDTHS) == ["0"]


# The caller's windows per bucket hold up to the counting kernel's room; more are taken as the default.
WINDOWS = """
int main() {
    int bad = 0;
    for (int words : {1, 2})
        for (uint64_t W : {1000ull, 46000000ull, 9000000000ull})
            for (uint32_t min_count : {1u, 2u}) {
                const uint64_t d = direct_bucket_windows(0, words, min_count, W);
                bad += d < 3200 || d > 7000;
                for (uint32_t asked : {1024u, 6400u, 8192u})
                    bad += direct_bucket_windows(asked, words, min_count, W) != asked;
                for (uint32_t asked : {8193u, 16384u, 65536u, 1u << 20})
                    bad += direct_bucket_windows(asked, words, min_count, W) != d;
            }
    printf("%d\\n", bad);
}
"""


def test_windows_that_no_bucket_holds_are_the_default(tmp_path):
    assert _run(tmp_path, WINDOWS) == ["0"]


# The sixteenths of a list of large buckets: the items that the plan adds up in one (item 16 / n) are those launched for it.
SLICES = """
int main() {
    int bad = 0;
    for (uint32_t n : {1u, 2u, 15u, 16u, 17u, 100u, 4097u, 1000003u}) {
        bad += refine_first(n, 0) != 0 || refine_first(n, RF_SLICES) != n;
        for (uint32_t s = 0; s < RF_SLICES; s++)
            for (uint32_t item = refine_first(n, s); item < refine_first(n, s + 1); item++)
                bad += (uint32_t)((uint64_t)item * RF_SLICES / n) != s;
    }
    printf("%d\\n", bad);
}
"""


def test_sixteenths_of_the_large_buckets(tmp_path):
    assert _run(tmp_path, SLICES) == ["0"]
