"""Sort-and-compact of keys that the sample does not show: wider or narrower than every sampled key, or in a part of
the array that no sampled key comes from. Bit-exact against the oracle, both entry points, both key widths."""
import ctypes

import numpy as np
import pytest

import oracle

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


def _check(pkg, ctx, x, bits):
    import torch

    n, words = x.shape[0], x.ndim
    ok, oc = oracle.sort_compact(x)
    d = torch.from_numpy(x.view(np.int64)).cuda()
    u, c = torch.empty_like(d), torch.empty(n, dtype=torch.int32, device="cuda")
    m = pkg.turtle_sort_compact_noalloc(d, bits, u, c) if n <= (1 << 20) // words else None
    for keys, counts in ([] if m is None else [(u[:m], c[:m])]) + [ctx.turtle_sort_compact(d, bits)]:
        assert np.array_equal(keys.cpu().numpy().view(np.uint64), ok)
        assert np.array_equal(counts.cpu().numpy().astype(np.uint64), oc)


def _wide(x, words, shift):
    """Keys of `words` words: x << shift over 128 bits (shift <= 63 past the low word's when words is 2)."""
    if words == 1:
        return x << np.uint64(shift)
    if shift >= 64:
        return np.stack([x << np.uint64(shift - 64), np.zeros_like(x)], 1)
    return np.stack([(x >> np.uint64(1)) >> np.uint64(63 - shift), x << np.uint64(shift)], 1)


# Consecutive keys: just above a power of two, only the last have its bit, and the sample ends before them; at 2,047
# the 1,024 sampled keys could be the first half.
@pytest.mark.parametrize("words,shift", [(1, 0), (1, 40), (2, 0), (2, 50), (2, 70), (2, 100)])
def test_consecutive_keys(pkg, ctx, words, shift):
    for n in (2047, 16_384, 16_389, 65_586, (1 << 18) + 100, (1 << 21) + 9):
        if shift + n.bit_length() > 64 * words:
            continue
        for x in (np.arange(n, dtype=np.uint64), np.arange(n, dtype=np.uint64)[::-1].copy()):
            _check(pkg, ctx, _wide(x, words, shift), 64 * words)


# One key or many of more bits, or of fewer, than every sampled one, at places the sample passes over: next to sampled
# ones, and the last. (2^log2m keys are sampled, the j-th at n j / 2^log2m.)
@pytest.mark.parametrize("words", [1, 2])
@pytest.mark.parametrize("n", [40_000, 100_003, 300_001])
@pytest.mark.parametrize("outlier", [0, 1, 3 << 38, 1 << 41, 1 << 45, 1 << 61, (1 << 63) - 1, 1 << 63])
def test_keys_outside_the_samples_span(pkg, ctx, words, n, outlier):
    rng = np.random.default_rng(n + words)
    narrow = rng.integers(1 << 39, 1 << 40, n, dtype=np.uint64)
    log2m = min(max(n.bit_length() - 5, 10), 14)
    beside = (n * np.arange(0, 1 << log2m, 2) >> log2m) + 1
    for at in ([1], [n - 1], [1, 7, n - 2, n - 1], beside):
        for shift in (0, 64) if words == 2 else (0,):
            x = narrow.copy()
            x[at] = outlier
            x = _wide(x, words, shift)
            if words == 2 and shift == 0 and outlier > 1 << 45:  # the high word alone holds it
                x[at] = (np.uint64(outlier), np.uint64(3))
            _check(pkg, ctx, x, 64 * words)


@pytest.mark.parametrize("words", [1, 2])
@pytest.mark.parametrize("at", [[], [1], [1, 7, 4095, 49_999]])
def test_results_over_the_keys_themselves(pkg, ctx, words, at):
    """unique may be the keys' own buffer, also when keys (here unsampled ones) have bits above key_bits, which the
    tiles only find out on the way."""
    import torch

    rng = np.random.default_rng(words)
    x = rng.integers(0, 1 << 16, 50_000, dtype=np.uint64)
    x[at] |= np.uint64(1 << 40)
    s = x[np.argsort(x & np.uint64(0xffff), kind="stable")]
    first = np.flatnonzero(np.concatenate([[True], s[1:] != s[:-1]]))
    counts = np.diff(np.append(first, s.size))
    for noalloc in (True, False):
        d = torch.from_numpy(_wide(x, words, 0).view(np.int64)).cuda()
        c = torch.empty(x.size, dtype=torch.int32, device="cuda")
        if noalloc:
            m = pkg.turtle_sort_compact_noalloc(d, 16, d, c)
        else:
            nu = ctypes.c_uint64()
            rc = pkg.load().turtle_sort_compact(ctx._h, d.data_ptr(), x.size, words, 16, d.data_ptr(), c.data_ptr(),
                                                ctypes.byref(nu), None)
            assert rc == 0
            m = nu.value
        assert np.array_equal(d[:m].cpu().numpy().view(np.uint64), _wide(s[first], words, 0))
        assert np.array_equal(c[:m].cpu().numpy(), counts)


# A sorted array takes about as long as the same keys in no order (less than twice as long: its keys meet in the same
# counters), where tiles of consecutive keys took 2.6 times as long for keys that come four times.
@pytest.mark.parametrize("copies", [1, 4])
def test_sorted_arrays_take_no_detour(ctx, copies):
    import torch

    n = 40_000_000
    x = torch.arange(n, device="cuda").div(copies, rounding_mode="floor")
    y = x[torch.randperm(n, device="cuda", generator=torch.Generator("cuda").manual_seed(1))]
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    ms = {}
    for turn in range(7):
        for name, keys in (("sorted", x), ("shuffled", y)):
            ev[0].record()
            u, c = ctx.turtle_sort_compact(keys, 62)
            ev[1].record()
            ev[1].synchronize()
            ms.setdefault(name, []).append(ev[0].elapsed_time(ev[1]))
            if turn == 0:
                assert torch.equal(u, torch.arange(n // copies, device="cuda")) and bool((c == copies).all())
    print(ms)
    assert sorted(ms["sorted"])[3] < 2 * sorted(ms["shuffled"])[3]
