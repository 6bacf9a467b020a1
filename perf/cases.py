"""Performance cases: what a user of the library has it do, through its public entry points.

The read libraries are synthetic, made on the GPU, in the shapes of this repository's own
workloads (`synth/`): iid genomes with or without inserted repeat copies, reads from either
strand at uniform or per-region log-normal coverage, 0.5-1% substitutions, a few N calls, 100 or
150 bases or ragged (quality-trimmed) lengths, and assembled contigs. The genome's bases come from
the seed; where the reads start, where they are wrong and which segments repeat belongs to the
case, so that libraries of different seeds hold about equally many reportable k-mers (the host
forms, whose results come as they are, equally many: no repeats, k >= 29). A case is a plain dict:

  form        device | host | batch | served | sort | noalloc
  k, min_count, genome, coverage, read, err, nrate, ragged, repeats, skew, budget_mib
                                       (read libraries)
  jobs                                 (batch, served: libraries, whose sizes are drawn per library)
  n, words, bits                       (sort, noalloc)
"""
import math
import random
import zlib

import numpy as np
import torch

import paper_1305_1861_gb300 as turtle

_ASCII = (65, 67, 71, 84)  # A C G T
_handles = {}


def _context():
    """One context per program, as a user keeps it: it owns the device scratch and the last result."""
    if "ctx" not in _handles:
        _handles["ctx"] = turtle.Context(0)
    return _handles["ctx"]


def _server():
    if "srv" not in _handles:
        _handles["srv"] = turtle.Server(0, max_batch=4, executors=2)
    return _handles["srv"]


# ---------------------------------------------------------------- the cases
def _library(form, k, min_count, genome, coverage, read, err=0.01, nrate=0.0, ragged=False, repeats=False,
             skew=False, budget_mib=0):
    return {"form": form, "k": k, "min_count": min_count, "genome": genome, "coverage": coverage, "read": read,
            "err": err, "nrate": nrate, "ragged": ragged, "repeats": repeats, "skew": skew,
            "budget_mib": budget_mib}


def listed():
    return [
        # the smallest calls: one amplicon or plasmid sample; launches and synchronisations are what it costs
        {"name": "device_20kb_k25", **_library("device", 25, 2, 1_003, 20, 100)},
        # the repository's `small` library: a bacterial-scale sample, 200,000 x 100 bp
        {"name": "device_small_k31", **_library("device", 31, 2, 1_000_000, 20, 100)},
        # one served-size job with long k-mers and a higher threshold (error-free k-mers only)
        {"name": "device_20Mb_k63_min3", **_library("device", 63, 3, 1_000_000, 20, 100)},
        # quality-trimmed reads of two lanes of a small eukaryote, 128-bit keys
        {"name": "device_ragged_k55", **_library("device", 55, 2, 7_000_001, 40, 150, ragged=True, nrate=0.0005)},
        # the k-mer table of a draft assembly: long overlapping contigs, every k-mer reported, most of them unique
        {"name": "device_contigs_k21_min1", **_library("device", 21, 1, 60_000_000, 1, 20_000, err=0.0, ragged=True,
                                                       repeats=True)},
        # the repository's headline library (fly-shaped): 30M x 100 bp, 5% repeats, 0.05% N
        {"name": "device_fly_k31", **_library("device", 31, 2, 105_000_000, 28.5714286, 100, nrate=0.0005,
                                              repeats=True)},
        # the long-k library at 1/20 scale under a memory budget that makes it run as four key ranges
        {"name": "device_longk_ranges_k64", **_library("device", 64, 2, 50_000_000, 33, 150, err=0.005, skew=True,
                                                       budget_mib=10_240)},
        # host arrays in, host arrays out, at a tenth of the fly-shaped library's size: its copies are in the call
        {"name": "host_300Mb_k31", **_library("host", 31, 2, 10_500_000, 28.5714286, 100, err=0.005, nrate=0.0005)},
        # many small libraries (a sequencing plate) in one call
        {"name": "batch_16_libraries", "form": "batch", "jobs": 16, "low": 2_000, "high": 400_000, "scale": 1.0},
        # the served form under a burst of jobs of mixed k
        {"name": "served_12_jobs", "form": "served", "jobs": 12, "low": 1_000_000, "high": 8_000_000, "scale": 1.0},
        # sort-and-compact alone: k-mers another program extracted (k = 31)
        {"name": "sort_40M_62bit", "form": "sort", "n": 40_000_003, "words": 1, "bits": 62},
        # the same for a caller that owns every allocation, in a loop over small batches
        {"name": "noalloc_100k_62bit", "form": "noalloc", "n": 100_003, "words": 1, "bits": 62},
    ]


def _log_uniform(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng: random.Random):
    form = rng.choice(["device"] * 6 + ["host", "host", "batch", "served", "sort", "noalloc"])
    if form == "batch":
        return {"form": form, "jobs": rng.randint(5, 16), "low": 2_000, "high": _log_uniform(rng, 50_000, 400_000),
                "scale": round(rng.uniform(0.5, 1.0), 3)}
    if form == "served":
        return {"form": form, "jobs": rng.randint(4, 12), "low": 1_000_000,
                "high": _log_uniform(rng, 2_000_000, 8_000_000), "scale": round(rng.uniform(0.5, 1.0), 3)}
    if form in ("sort", "noalloc"):
        words = rng.choice([1, 1, 2])
        k = rng.randint(17, 32) if words == 1 else rng.randint(33, 64)
        n = _log_uniform(rng, 1_000, 40_000_000 // words if form == "sort" else 400_000)
        return {"form": form, "n": n, "words": words, "bits": 2 * k}
    k = rng.choice([rng.randint(15 if form == "device" else 29, 32), rng.choice([21, 25, 27, 31]) if form == "device" else 31,
                    rng.randint(33, 64)])
    bases = _log_uniform(rng, 20_000, 1_500_000_000 if form == "device" else 200_000_000)
    if k > 32:
        bases = min(bases, 700_000_000)
    read = rng.choice([75, 100, 125, 150, 151, 250])
    coverage = round(rng.uniform(8, 60), 2)
    budget = 0
    if form == "device" and bases > 100_000_000 and rng.random() < 0.4:  # two to five key ranges
        budget = max(64, int(bases * (1 - (k - 1) / read) * (40 if k > 32 else 24) / rng.uniform(1.5, 4.5) / 2**20))
    return _library(form, k, rng.choice([1, 2, 2, 2, 3, 5]), max(1_000, int(bases / coverage)), coverage, read,
                    err=rng.choice([0.0, 0.005, 0.01] if form == "device" else [0.0, 0.005]),
                    nrate=rng.choice([0.0, 0.0005, 0.002]), ragged=rng.random() < 0.4,
                    repeats=form == "device" and rng.random() < 0.4, skew=rng.random() < 0.3,
                    budget_mib=budget)


# ---------------------------------------------------------------- inputs
def _rng(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _own_seed(c):
    """The seed of what belongs to the case rather than to its inputs' seed."""
    return zlib.crc32(repr(sorted((k, v) for k, v in c.items() if k != "name")).encode())


def _genome(size, repeats, seed, g, r):
    seq = torch.randint(0, 4, (size,), dtype=torch.uint8, device="cuda", generator=_rng(seed))
    if repeats and size > 20_000:  # 5% of the length: families of 1-5 kb, 2-20 copies, 2% divergence
        done = 0
        while done < 0.05 * size:
            n = r.randint(1_000, 5_000)
            src = r.randrange(size - n)
            for _ in range(r.randint(2, 20)):
                dst = r.randrange(size - n)
                copy = seq[src:src + n].clone()
                change = torch.rand(n, device="cuda", generator=g) < 0.02
                copy = torch.where(change, (copy + 1 + done % 3) & 3, copy)
                seq[dst:dst + n] = copy
                done += n
                if done >= 0.05 * size:
                    break
    return seq


def _reads(c, seed):
    """(bases uint8, offsets int64) on the GPU."""
    g = _rng(_own_seed(c))
    size, read = c["genome"], min(c["read"], c["genome"])
    seq = _genome(size, c["repeats"], seed, g, random.Random(_own_seed(c)))
    lut = torch.tensor(_ASCII, dtype=torch.uint8, device="cuda")
    mean = 0.75 * read if c["ragged"] else read
    n = max(1, int(round(c["coverage"] * size / mean)))
    cum = None
    if c["skew"]:  # log-normal coverage per 10 kb
        cum = torch.randn(max(1, size // 10_000), device="cuda", generator=g).exp().double().cumsum(0)
    parts, lens = [], []
    step = max(1, (1 << 26) // read)
    cols = torch.arange(read, dtype=torch.int32, device="cuda")
    for first in range(0, n, step):
        m = min(step, n - first)
        span = size - read + 1
        if cum is not None:
            u = torch.rand(m, device="cuda", generator=g, dtype=torch.float64) * cum[-1]
            region = torch.searchsorted(cum, u).clamp_(max=cum.numel() - 1)
            start = region * 10_000 + torch.randint(0, 10_000, (m,), device="cuda", generator=g)
            start = start.clamp_(max=span - 1).to(torch.int32)
        else:
            start = torch.randint(0, span, (m,), device="cuda", generator=g, dtype=torch.int32)
        minus = torch.rand(m, device="cuda", generator=g) < 0.5
        at = torch.where(minus[:, None], start[:, None] + (read - 1) - cols, start[:, None] + cols)
        base = seq[at.reshape(-1).long()].reshape(m, read)
        del at
        base = torch.where(minus[:, None], 3 - base, base)
        if c["err"] > 0 or c["nrate"] > 0:
            u = torch.rand((m, read), device="cuda", generator=g)
            other = (base + 1 + (u * (3 / max(c["err"], 1e-9))).clamp_(max=2).to(torch.uint8)) & 3
            base = torch.where(u < c["err"], other, base)
            text = lut[base.long()]
            if c["nrate"] > 0:
                text = torch.where(u > 1 - c["nrate"], torch.full_like(text, 78), text)
            del u, other
        else:
            text = lut[base.long()]
        if c["ragged"]:
            length = torch.randint(read // 2, read + 1, (m,), device="cuda", generator=g)
            text = text[cols[None, :] < length[:, None]]
        else:
            length = torch.full((m,), read, device="cuda")
        parts.append(text.reshape(-1))
        lens.append(length)
        del base, text
    offsets = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    offsets[1:] = torch.cat(lens).cumsum(0)
    return torch.cat(parts), offsets


def _host_reads(c, seed):
    b, o = _reads(c, seed)
    return b.cpu().numpy(), o.cpu().numpy().astype(np.uint64)


def _job_specs(c):
    """Libraries of a batch or of a burst of jobs: the sizes belong to the case, the reads to the seed."""
    r = random.Random(7)
    specs = []
    for _ in range(c["jobs"]):
        size = int(_log_uniform(r, c["low"], c["high"]) * c["scale"])
        if c["form"] == "batch":  # genome sizes; coverage 10-60
            specs.append(_library("host", r.choice([29, 31, 55]), 2, max(1_000, size), round(r.uniform(10, 60), 2),
                                  r.choice([100, 150])))
        else:  # read bases; 20x
            specs.append(_library("host", r.choice([29, 31, 63]), r.choice([2, 3]), max(1_000, size // 20), 20, 100))
    return specs


def _mix(x, bits, odd):
    """A bijection of the integers below 2^bits (bits <= 63)."""
    m = (1 << bits) - 1
    x = (x * odd) & m
    return ((x ^ (x >> (bits // 2))) * odd) & m


def _keys(c, seed):
    """Distinct keys, each about four times, in random order (a pool of n / 4)."""
    pool, n = max(1, c["n"] // 4), c["n"]
    at = torch.randint(0, pool, (n,), device="cuda", generator=_rng(_own_seed(c)))
    r = random.Random(seed)
    first = r.randrange(1 << 30)
    odd = r.randrange(1 << 29) * 2 + 1
    bits = min(c["bits"], 62) if c["words"] == 1 else min(c["bits"] - 64, 62)
    lo = torch.arange(first, first + pool, device="cuda")
    if c["words"] == 1:
        return _mix(lo, bits, odd)[at].contiguous()
    hi = _mix(lo, bits, odd)
    lo = _mix(lo, 62, odd) - (1 << 61)
    return torch.stack([hi, lo], dim=1)[at].contiguous()


def _room(c):
    """Entries the program sets aside for a device result."""
    bases = int(1.05 * c["coverage"] * c["genome"]) + 2 * c["read"]
    return (bases if c["min_count"] == 1 else min(bases // c["min_count"], 6 * c["genome"])) + 1024


def prepare(case, seed):
    form = case["form"]
    state = {"form": form, "case": case}
    if form == "device":
        state["ctx"] = _context()
        state["bases"], state["offsets"] = _reads(case, seed)
        state["params"] = turtle.Params.default(budget_mib=case["budget_mib"]) if case["budget_mib"] else None
        n = _room(case)
        state["keys"] = torch.zeros((n,) if case["k"] <= 32 else (n, 2), dtype=torch.int64, device="cuda")
        state["counts"] = torch.zeros(n, dtype=torch.int32, device="cuda")
    elif form == "host":
        state["bases"], state["offsets"] = _host_reads(case, seed)
    elif form in ("batch", "served"):
        jobs = []
        for i, spec in enumerate(_job_specs(case)):
            b, o = _host_reads(spec, seed * 1_000 + i)
            jobs.append((b, o, spec["k"], spec["min_count"]))
        state["jobs"] = jobs
        if form == "served":
            state["server"] = _server()
    else:
        state["keys"] = _keys(case, seed)
        if form == "sort":
            state["ctx"] = _context()
        else:
            state["unique"] = torch.empty_like(state["keys"])
            state["counts"] = torch.empty(case["n"], dtype=torch.int32, device="cuda")
    return state


# ---------------------------------------------------------------- one pass
def _signed(keys, counts, n_windows):
    return keys.view(np.int64), counts.view(np.int32), n_windows


def run(state):
    form = state["form"]
    if form == "device":
        c = state["case"]
        keys, counts, n_windows = state["ctx"].turtle_count_device(state["bases"], state["offsets"], c["k"],
                                                                   c["min_count"], state["params"])
        n = counts.numel()  # the result is the context's until its next call: the program keeps a copy
        state["keys"][:n] = keys
        state["counts"][:n] = counts
        return state["keys"], state["counts"], n, n_windows
    if form == "host":
        c = state["case"]
        return _signed(*turtle.turtle_count(state["bases"], state["offsets"], c["k"], c["min_count"]))
    if form == "batch":
        return [_signed(*r) for r in turtle.turtle_count_batch(state["jobs"])]
    if form == "served":
        srv = state["server"]
        tickets = [srv.submit(*job) for job in state["jobs"]]
        return [_signed(*srv.poll(t)[:3]) for t in tickets]
    if form == "sort":
        return state["ctx"].turtle_sort_compact(state["keys"], state["case"]["bits"])
    n = turtle.turtle_sort_compact_noalloc(state["keys"], state["case"]["bits"], state["unique"], state["counts"])
    return state["unique"][:n], state["counts"][:n]


# ---------------------------------------------------------------- what a pass cannot do without
def _library_bytes(c):
    """Reads and offsets in, reported keys and counts out (their number is estimated: the genome's
    k-mers, and for min_count 1 the k-mers of the erroneous windows)."""
    bases = c["coverage"] * c["genome"]
    reads = bases / (c["read"] * (0.75 if c["ragged"] else 1.0))
    windows = max(0.0, bases - reads * (c["k"] - 1))
    out = min(windows, c["genome"])
    if c["min_count"] == 1:
        out = min(windows, out + windows * (1 - (1 - c["err"]) ** c["k"]))
    return bases + 8 * (reads + 1) + out * ((8 if c["k"] <= 32 else 16) + 4)


def work(case):
    if case["form"] in ("device", "host"):
        return {"bytes": _library_bytes(case), "flops": 0}
    if case["form"] in ("batch", "served"):
        return {"bytes": sum(_library_bytes(s) for s in _job_specs(case)), "flops": 0}
    distinct = case["n"] / 4 * (1 - math.exp(-4))
    return {"bytes": 8 * case["words"] * case["n"] + distinct * (8 * case["words"] + 4), "flops": 0}
