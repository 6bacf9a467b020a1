"""Counting and sort-and-compact by tiles vs the CPU oracle and vs the other forms, where they can go wrong:
tile edges, one and two levels of tiles, key ranges, buckets larger than shared memory, key arrays of every
kind of distribution, packing of every byte value. Integer work: the bar is bit-exact."""
import numpy as np
import pytest

import oracle
from tests import brute

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg(have_gpu):
    import paper_1305_1861_gb300 as pkg

    pkg.build()
    return pkg


@pytest.fixture(scope="module")
def ctx(pkg):
    c = pkg.Context(0)
    yield c
    c.close()


def _dev(bases, offsets):
    import torch

    return torch.from_numpy(np.ascontiguousarray(bases)).cuda(), \
        torch.from_numpy(np.ascontiguousarray(offsets).astype(np.int64)).cuda()


def _letters(seed, n):
    return np.frombuffer(b"ACGT", np.uint8)[np.random.default_rng(seed).integers(0, 4, n)]


def _check(ctx, bases, offs, k, min_count, params=None):
    ok, oc, onw = oracle.count(bases, offs, k, min_count)
    keys, counts, nw = ctx.turtle_count_device(*_dev(bases, offs), k, min_count, params)
    assert nw == onw
    assert np.array_equal(keys.cpu().numpy().view(np.uint64).reshape(ok.shape), ok)
    assert np.array_equal(counts.cpu().numpy().view(np.uint32).astype(np.uint64), oc)
    return ctx.stats()


# A tile holds 8,192 64-bit or 4,096 128-bit keys and is written when a step of 256 might not fit.
@pytest.mark.parametrize("k,cap", [(31, 8192), (55, 4096)])
def test_tile_edges(ctx, k, cap):
    for n in (1, 31, 32, 33, 511, 512, 513, cap - 257, cap - 256, cap - 255, cap - 1, cap, cap + 1, 2 * cap + 1):
        bases = _letters(n, n + k - 1)
        _check(ctx, bases, np.array([0, bases.size], np.uint64), k, 1)


# 1,024 buckets are one level, 1,025 two; one, five or fifteen key ranges; the wait for the number of windows is
# left out only when every base's window would fit the budget.
@pytest.mark.parametrize("budget", [0, 8, 2])
@pytest.mark.parametrize("k,min_count", [(11, 2), (31, 1), (32, 2), (55, 1), (64, 3)])
def test_levels_and_key_ranges(ctx, pkg, k, min_count, budget):
    for n in (1024 * 1024, 1024 * 1024 + 1024):
        g = _letters(k, n // 3)
        reads = np.concatenate([g, g[::-1], g])[:n + k - 1]  # keys once, twice and in palindromic halves
        reads = np.concatenate([reads, _letters(7, n + k - 1 - reads.size)])
        st = _check(ctx, reads, np.array([0, reads.size], np.uint64), k, min_count,
                    pkg.Params.default(bucket_windows=1024, budget_mib=budget))
        assert (st["super_partitions"] > 1) == (budget > 0)


# Buckets left to the second counting kernel: one key in half of the windows, many windows in a narrow key range
# (more distinct keys than its table holds: split into key ranges), and wide buckets.
@pytest.mark.parametrize("k", [21, 47])
@pytest.mark.parametrize("kind", ["heavy", "skew", "wide"])
def test_large_buckets(ctx, pkg, k, kind):
    rng = np.random.default_rng(k)
    if kind == "heavy":
        seq = [np.full(150_000, ord("A"), np.uint8), _letters(1, 150_000)]
    elif kind == "skew":  # a long run of A before 6 to 9 random letters
        seq = [np.concatenate([np.full(k - 8, ord("A"), np.uint8), _letters(100 + i, 8)]) for i in range(30_000)]
    else:
        seq = [_letters(1, 300_000)]
    offs = np.concatenate([[0], np.cumsum([s.size for s in seq])]).astype(np.uint64)
    bases = np.concatenate(seq)
    for min_count in (1, 2):
        for bw in (0, 1 << 20) if kind == "wide" else (0, 1024):
            _check(ctx, bases, offs, k, min_count, pkg.Params.default(bucket_windows=bw))


# Buckets of 128-bit keys wider than the ordinary counting kernel's: on both sides of the line, and with some that do
# not fit the wide one either.
@pytest.mark.parametrize("bucket_windows", [4300, 4301, 7000, 8192])
def test_wide_buckets(ctx, pkg, bucket_windows):
    for n in (1, 4097, 8192, 8193, 300_000):
        bases = np.concatenate([_letters(n, n)] * 3)
        for min_count in (1, 3):
            _check(ctx, bases, np.array([0, bases.size], np.uint64), 40, min_count,
                   pkg.Params.default(bucket_windows=bucket_windows))


# Segments of kept keys on both sides of each of the ordering kernel's sizes: one bucket, and 304 whose sizes vary
# around 512, 1,024, 2,048 and 4,096.
@pytest.mark.parametrize("k", [31, 40])
def test_order_at_its_sizes(ctx, pkg, k):
    for n in (1, 255, 256, 257, 511, 155_000, 311_000, 622_000, 1_245_000):
        bases = _letters(n, n + k - 1)
        _check(ctx, bases, np.array([0, bases.size], np.uint64), k, 1, pkg.Params.default(bucket_windows=1 << 20))


# Every k through the tiles, against the global form of the same call, whole and in key ranges.
@pytest.mark.parametrize("min_count", [1, 2, 3])
def test_every_k_matches_the_global_form(ctx, pkg, min_count):
    g = _letters(3, 9000)
    reads = [g[s:s + int(n)].tobytes().decode() for s, n in
             zip(np.random.default_rng(4).integers(0, 8800, 600), np.random.default_rng(5).integers(0, 200, 600))]
    b, o = _dev(*brute.pack(reads))
    for k in range(1, 65):
        ref = [x.clone() for x in ctx.turtle_count_device(b, o, k, min_count, pkg.Params.default(compact=1))[:2]]
        for budget in (0, 1):
            keys, counts, _ = ctx.turtle_count_device(b, o, k, min_count, pkg.Params.default(budget_mib=budget))
            assert keys.equal(ref[0]) and counts.equal(ref[1]), (k, budget)


@pytest.mark.parametrize("mixed", [1, 2])
def test_batch_libraries_at_tile_edges(pkg, mixed):
    jobs = []
    for i, n in enumerate((1, 8191, 8192, 8193, 4095, 4097, 300, 20_000)):
        k = (21, 33)[i % 2]
        bases = np.concatenate([_letters(i, n + k - 1)] * 2)
        jobs.append((bases, np.array([0, n + k - 1, bases.size], np.uint64), k, 2))
    got = pkg.turtle_count_batch(jobs, pkg.Params.default(batch_mixed=mixed))
    for (b, o, k, m), (keys, counts, nw) in zip(jobs, got):
        ok, oc, onw = oracle.count(b, o, k, m)
        assert nw == onw and np.array_equal(keys, ok) and np.array_equal(counts.astype(np.uint64), oc)


def test_batch_runs_a_large_library_alone(pkg):
    """On both sides of 64 MiB, beside small libraries of the same k, in the callers' order."""
    g = _letters(9, 1_000_000)
    def lib(n, k):
        starts = np.random.default_rng(n).integers(0, g.size - 150, n // 150 + 1)
        bases = g[(starts[:, None] + np.arange(150)).ravel()][:n]
        return bases, np.append(np.arange(0, n, 150), n).astype(np.uint64), k, 2
    jobs = [lib(40_000, 31), lib((64 << 20) + 1, 31), lib(50_000, 31), lib(64 << 20, 55), lib((64 << 20) - 1, 31)]
    for (b, o, k, m), (keys, counts, nw) in zip(jobs, pkg.turtle_count_batch(jobs)):
        pk, pc, pn = pkg.turtle_count(b, o, k, m)
        assert nw == pn and np.array_equal(keys, pk) and np.array_equal(counts, pc)


def _keys(kind, n, words, rng):
    top = 2**62 if words == 1 else 2**46
    def uniform(m):
        hi = rng.integers(0, top, m, dtype=np.uint64)
        return hi if words == 1 else np.stack([hi, rng.integers(0, 2**64, m, dtype=np.uint64)], 1)
    x = uniform(max(n // 4, 1))[rng.integers(0, max(n // 4, 1), n)]
    if kind == "distinct":
        x = uniform(n)
    elif kind == "small":
        x = np.zeros_like(x)
        x.reshape(n, words)[:, -1] = rng.integers(0, 5000, n)
    elif kind == "constant":
        x[:] = x[0]
    elif kind == "ones":
        x[rng.random(n) < 0.01] = ~np.uint64(0)
    elif kind == "all ones":
        x[:] = ~np.uint64(0)
    elif kind == "heavy":
        x[rng.random(n) < 0.4] = x[0]
    elif kind == "clusters":
        x = uniform(n) >> np.uint64(40)
        x.reshape(n, words)[n // 2:, 0] |= np.uint64(top // 2)
    elif kind == "sorted":
        x = np.sort(x) if words == 1 else x[np.lexsort((x[:, 1], x[:, 0]))]
    return x


# Sizes around the tiles and the sample (a sixteenth of the keys, 1,024 at least); the array may start at any
# multiple of eight bytes, also for 128-bit keys.
@pytest.mark.parametrize("words", [1, 2])
@pytest.mark.parametrize("kind", ["plain", "distinct", "small", "constant", "ones", "all ones", "heavy", "clusters", "sorted"])
def test_sort_by_tiles(ctx, pkg, kind, words):
    import torch

    rng = np.random.default_rng(len(kind) + words)
    for n in (1, 2, 1023, 4095, 4097, 8191, 8193, 70_001, 262_144):
        x = _keys(kind, n, words, rng)
        ok, oc = oracle.sort_compact(x)
        room = torch.zeros(n * words + 1, dtype=torch.int64, device="cuda")
        d = room[1:].view(x.shape)
        d.copy_(torch.from_numpy(x.view(np.int64)))
        bits = 64 * words if "ones" in kind else 62 if words == 1 else 110
        u, c = torch.empty(x.shape, dtype=torch.int64, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda")
        m = pkg.turtle_sort_compact_noalloc(d, bits, u, c)
        for keys, counts in ((u[:m], c[:m]), ctx.turtle_sort_compact(d, bits)):
            assert np.array_equal(keys.cpu().numpy().view(np.uint64), ok), n
            assert np.array_equal(counts.cpu().numpy().astype(np.uint64), oc), n


def test_keys_with_bits_above_key_bits_are_ordered_by_the_others(ctx, pkg):
    """As before: a stable order by the digits of key_bits, runs of equal whole keys compacted."""
    import torch

    rng = np.random.default_rng(2)
    x = rng.integers(0, 1 << 16, 50_000, dtype=np.uint64) | (rng.integers(0, 2, 50_000, dtype=np.uint64) << np.uint64(40))
    s = x[np.argsort(x & np.uint64(0xffff), kind="stable")]
    first = np.flatnonzero(np.concatenate([[True], s[1:] != s[:-1]]))
    d = torch.from_numpy(x.view(np.int64)).cuda()
    u, c = torch.empty_like(d), torch.empty(x.size, dtype=torch.int32, device="cuda")
    m = pkg.turtle_sort_compact_noalloc(d, 16, u, c)
    for keys, counts in ((u[:m], c[:m]), ctx.turtle_sort_compact(d, 16)):
        assert np.array_equal(keys.cpu().numpy().view(np.uint64), s[first])
        assert np.array_equal(counts.cpu().numpy(), np.diff(np.append(first, s.size)))


# Every byte value, reads that end at and around 32- and 64-base words, every window length's smear.
@pytest.mark.parametrize("k", [1, 2, 17, 31, 32, 33, 63, 64])
def test_packing_every_byte_value_and_read_ends(ctx, k):
    rng = np.random.default_rng(k)
    lens = np.array([256, 0, 1, 31, 32, 33, 63, 64, 65, 127, 128, 129, 5000, 20_000])
    offs = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    bases = _letters(k, int(offs[-1])).copy()
    bases[:256] = rng.permutation(256)
    odd = rng.random(bases.size) < np.where(np.arange(bases.size) < 6000, 0.1, 0.002)
    odd[:256] = False
    bases[odd] = rng.integers(0, 256, int(odd.sum()))
    pos, okeys = oracle.windows(bases, offs, k)
    keys, valid, nw = ctx.turtle_extract(*_dev(bases, offs), k)
    bits = np.unpackbits(valid.cpu().numpy().view(np.uint8), bitorder="little")[:bases.size].astype(bool)
    assert nw == len(pos) and np.array_equal(np.flatnonzero(bits), pos.astype(np.int64))
    assert np.array_equal(keys.cpu().numpy().view(np.uint64)[pos.astype(np.int64)], okeys)
