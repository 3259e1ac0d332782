"""The counting work whose speed is measured: read sets of the sizes and shapes that the
repository's own workloads have, each counted through the package's public calls.

A case is a dict of plain values:
  call       how the program counts: "count" (kc_count on device-resident reads), "submit"
             (kc_submit, then kc_job_wait: a served request), "batch" (kc_count_batch of
             several samples), "host" (pinned host reads submitted one after another, each
             result copied out to pinned host memory: the pipelined end-to-end form)
  kind       the genome: "uniform" (i.i.d. bases), "repeats" (a fifth of it copies of 500
             repeat families, 2% divergence), "satellite" (a few percent of it (AATGG)_n
             arrays, the heavy hitters of large genomes), "long" (i.i.d. bases, read by long
             noisy reads with insertions and deletions)
  genome     bases of the genome; with several samples, of the largest one
  genome_min with several samples, bases of the smallest (sizes are spread over the logarithm)
  samples    read sets in one pass
  coverage   bases read per genome base (with several samples: of the largest; the others
             take 5x to 40x)
  read_min, read_max   read lengths, uniform in between (long reads: log-normal lengths, the
             median given by read_max)
  errors     rate of wrong bases; n_rate: rate of N
  k, canonical

Reads are ASCII on the device, offsets int64 on the device, and one plan (KmerCounter) is
kept for as long as any read set is, as a program that counts many read sets keeps it.  A
result is kept in the program's own table (keys and counts of all samples back to back, the
samples' sizes beside them) and released: its buffers are sized for the bases, not for the
distinct keys.  Entries past the last one stay zero.
"""
from __future__ import annotations

import math
import weakref

import numpy as np
import torch

from paper_2505_04431_gb300 import KmerCounter

_CHUNK = 1 << 27  # bases generated at a time
_plans = weakref.WeakValueDictionary()


def _case(name, call, kind, genome, coverage, k, canonical=True, read_min=150, read_max=150, errors=0.005, n_rate=0.0,
          samples=1, genome_min=0):
    c = {"call": call, "kind": kind, "genome": genome, "coverage": coverage, "k": k, "canonical": canonical,
         "read_min": read_min, "read_max": read_max, "errors": errors, "n_rate": n_rate, "samples": samples,
         "genome_min": genome_min}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one amplicon or plasmid panel: the smallest call, where launches and host work count
        _case("tiny_k31", "count", "uniform", 20_000, 10.0, 31, read_min=100, read_max=100, n_rate=1e-4),
        # the plain small workload: 1 Mbp genome, 100 bp reads at 10x with errors and N
        _case("uniform_10mb_k31", "count", "uniform", 1_000_000, 10.0, 31, read_min=100, read_max=100, n_rate=1e-4),
        # a served request of middling size, reads of ragged length after quality trimming
        _case("served_ragged_k21", "submit", "uniform", 1_234_567, 17.0, 21, read_min=31, read_max=150),
        # a served request with 128-bit keys
        _case("served_100mb_k63", "submit", "uniform", 5_000_000, 20.0, 63),
        # strand-specific counting: forward keys only
        _case("forward_45mb_k25", "count", "uniform", 1_500_000, 30.0, 25, canonical=False),
        # a genome with satellite arrays: a few k-mers hold several percent of all windows
        _case("satellite_90mb_k31", "count", "satellite", 3_000_000, 30.0, 31),
        # an ordinary eukaryotic sample: the headline workload at a tenth of its size
        _case("repeats_300mb_k31", "count", "repeats", 10_000_000, 30.0, 31),
        # the headline workload: 100 Mbp repeat genome, 150 bp reads, 30x
        _case("repeats_3gb_k31", "count", "repeats", 100_000_000, 30.0, 31),
        # long noisy reads, 128-bit keys, nearly all windows distinct
        _case("long_1gb_k63", "count", "long", 50_000_000, 20.0, 63, read_min=64, read_max=10_000, errors=0.05),
        # a plate of small samples counted in batched launches
        _case("batch_32_small_k31", "batch", "uniform", 40_000, 10.0, 31, samples=32, genome_min=10_000),
        # samples of uneven size, the range of the batched workload
        _case("batch_12_uneven_k31", "batch", "uniform", 20_000_000, 20.0, 31, samples=12, genome_min=100_000),
        # end to end from pinned host memory and back, four read sets in a row
        _case("host_4x24mb_k31", "host", "uniform", 1_200_000, 20.0, 31, samples=4, genome_min=800_000),
    ]


def draw(rng):
    def log_uniform(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    call = rng.choice(["count", "count", "count", "submit", "batch", "host"])
    k = rng.choice([17, 21, 25, 27, 31, 31, 31, 32, 41, 55, 63, 63])
    wide = k > 32
    cov = round(rng.uniform(5.0, 40.0), 2)
    read = rng.choice([76, 100, 125, 150, 150, 250])
    low = read if rng.random() < 0.6 else rng.randrange(30, read)
    canonical = rng.random() < 0.85
    n_rate = rng.choice([0.0, 0.0, 1e-4, 1e-3])
    if call == "batch":
        return _case(None, call, "uniform", log_uniform(30_000, 15_000_000), cov, k, canonical, low, read, 0.005, n_rate,
                     rng.randrange(2, 24), rng.randrange(5_000, 30_000))
    if call == "host":
        g = log_uniform(50_000, 2_000_000)
        return _case(None, call, "uniform", g, cov, k, canonical, low, read, 0.005, n_rate, rng.randrange(1, 5),
                     max(5_000, g // 2))
    kind = rng.choice(["uniform", "uniform", "repeats", "satellite", "long"])
    bases = log_uniform(200_000, 100_000_000 if kind == "satellite" else 600_000_000 if wide else 1_500_000_000)
    if kind == "long":
        med = rng.choice([2_000, 10_000, 10_000, 25_000])
        return _case(None, call, kind, max(20_000, int(bases / cov)), cov, k, canonical, 64, med, 0.05, n_rate)
    return _case(None, call, kind, max(10_000, int(bases / cov)), cov, k, canonical, low, read, 0.005, n_rate)


# ------------------------------------------------------------------ sizes
def _samples(case):
    """(genome bases, coverage) of every read set of the case."""
    n = case["samples"]
    if n == 1:
        return [(case["genome"], case["coverage"])]
    ratio = case["genome"] / case["genome_min"]
    out = []
    for i in range(n):
        g = int(round(case["genome_min"] * ratio ** (i / (n - 1))))
        out.append((g, case["coverage"] if i == n - 1 else 5.0 + 35.0 * ((i * 0.6180339887) % 1.0)))
    return out


def _mean_read(case):
    if case["kind"] == "long":
        return case["read_max"] * math.exp(0.125)  # log-normal, sigma 0.5
    return (case["read_min"] + case["read_max"]) / 2


def _expected(case, g, cov):
    """(reads, bases, distinct keys) expected of one read set: the distinct keys are the covered
    genome and the windows that hold a wrong base (fewer where the genome repeats itself)."""
    k, mean, strands = case["k"], _mean_read(case), 1 if case["canonical"] else 2
    if case["kind"] == "long":
        per_read = mean - (k - 1)
    else:
        lengths = range(case["read_min"], case["read_max"] + 1)
        per_read = sum(max(0, n - k + 1) for n in lengths) / len(lengths)
    n_reads = max(1, round(cov * g / mean))
    bases = n_reads * mean
    windows = n_reads * per_read
    good = (1.0 - case["errors"]) ** k
    distinct = strands * g * (1.0 - math.exp(-windows * good / g / strands)) + windows * (1.0 - good)
    return n_reads, bases, min(distinct, windows)


def _room(case, g, cov):
    """Entries that the program's table keeps for one read set."""
    return int(1.05 * _expected(case, g, cov)[2]) + 16384


def work(case):
    """Reads and offsets read once, the histogram written once."""
    total = 0.0
    for g, cov in _samples(case):
        n_reads, bases, distinct = _expected(case, g, cov)
        total += bases + 8 * (n_reads + 1) + distinct * ((8 if case["k"] <= 32 else 16) + 4)
    return {"bytes": total, "flops": 0.0}


# ------------------------------------------------------------------ read sets
def _genome(gen, kind, size):
    """Base codes 0..3 (uint8) of a genome of `size` bases."""
    dev = gen.device
    g = torch.randint(0, 4, (size,), generator=gen, device=dev, dtype=torch.uint8)
    if kind == "repeats":
        # 500 families of 300 to 6000 bases, copy numbers by Zipf's law (1.2), a fifth of the genome
        families = max(1, min(500, size // 20_000))
        length = torch.randint(300, 6001, (families,), generator=gen, device=dev)
        weight = torch.arange(1, families + 1, device=dev, dtype=torch.float64) ** -1.2
        copies = (weight * (0.2 * size / (weight * length).sum())).round().clamp(min=1).long()
        consensus = torch.randint(0, 4, (families, 6000), generator=gen, device=dev, dtype=torch.uint8)
        family = torch.arange(families, device=dev).repeat_interleave(copies)
        family = family[torch.randperm(family.numel(), generator=gen, device=dev)]
        slot = size // family.numel()  # one copy somewhere in each slot
        n = length[family].clamp(max=slot)
        start = (torch.rand(n.numel(), generator=gen, device=dev, dtype=torch.float64) * (slot - n + 1)).long()
        start += torch.arange(n.numel(), device=dev) * slot
        copy = torch.arange(n.numel(), device=dev).repeat_interleave(n)
        at = torch.arange(copy.numel(), device=dev) - (n.cumsum(0) - n)[copy]
        base = consensus[family[copy], at]
        g[start[copy] + at] = _substitute(gen, base, 0.02)
    elif kind == "satellite":
        # arrays of (AATGG)_n, 2500 bases each, on 3% of the genome
        unit = torch.tensor([0, 0, 3, 2, 2], dtype=torch.uint8, device=dev)
        n = max(1, int(0.03 * size / 2500))
        slot = size // n
        width = min(2500, slot)
        start = torch.arange(n, device=dev) * slot
        at = torch.arange(width, device=dev)
        g[(start[:, None] + at).reshape(-1)] = unit[at % 5].repeat(n)
    return g


def _substitute(gen, codes, rate):
    hit = torch.rand(codes.shape, generator=gen, device=codes.device) < rate
    other = torch.randint(1, 4, codes.shape, generator=gen, device=codes.device, dtype=torch.uint8)
    return torch.where(hit, (codes + other) & 3, codes)


def _reads(gen, case, genome, coverage):
    """(reads uint8, offsets int64) on the device: reads from uniform starts on both strands."""
    dev, size = gen.device, genome.numel()
    n = max(1, round(coverage * size / _mean_read(case)))
    if case["kind"] == "long":
        # the quantiles of the distribution in random order: the bases read hardly vary
        z = torch.special.ndtri((torch.randperm(n, generator=gen, device=dev).double() + 0.5) / n)
        span = (case["read_max"] * torch.exp(0.5 * z)).round().long()
    else:
        span = torch.randint(case["read_min"], case["read_max"] + 1, (n,), generator=gen, device=dev)
    span = span.clamp(min=min(case["read_min"], size), max=size)
    start = (torch.rand(n, generator=gen, device=dev, dtype=torch.float64) * (size - span + 1)).long()
    reverse = torch.rand(n, generator=gen, device=dev) < 0.5
    end = span.cumsum(0)
    letters = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device=dev)
    n_chunks = max(1, -(-int(end[-1]) // _CHUNK))
    cuts = torch.searchsorted(end, torch.arange(1, n_chunks, device=dev) * _CHUNK).tolist()
    pieces, lengths = [], []
    for a, b in zip([0] + cuts, cuts + [n]):
        if a == b:
            continue
        m = span[a:b]
        read = torch.arange(b - a, device=dev).repeat_interleave(m)
        at = torch.arange(read.numel(), device=dev) - (m.cumsum(0) - m)[read]
        back = reverse[a:b][read]
        at = torch.where(back, m[read] - 1 - at, at) + start[a:b][read]
        codes = genome[at]
        del at
        codes = torch.where(back, 3 - codes, codes)
        del back
        if case["kind"] == "long":
            # wrong bases: 60% substitutions, 20% insertions before the base, 20% deletions
            u = torch.rand(codes.shape, generator=gen, device=dev) / case["errors"]
            other = torch.randint(1, 4, codes.shape, generator=gen, device=dev, dtype=torch.uint8)
            codes = torch.where(u < 0.6, (codes + other) & 3, codes)
            times = 1 + ((u >= 0.6) & (u < 0.8)).long() - ((u >= 0.8) & (u < 1.0)).long()
            del u, other
            lengths.append(torch.zeros(b - a, dtype=torch.int64, device=dev).index_add_(0, read, times))
            first = (times.cumsum(0) - times)[times == 2]
            codes = codes.repeat_interleave(times)
            codes[first] = torch.randint(0, 4, first.shape, generator=gen, device=dev, dtype=torch.uint8)
            del times, first
        else:
            codes = _substitute(gen, codes, case["errors"])
            lengths.append(m)
        del read
        text = letters.index_select(0, codes.int())
        if case["n_rate"]:
            text[torch.rand(text.shape, generator=gen, device=dev) < case["n_rate"]] = ord("N")
        pieces.append(text)
    reads = torch.cat(pieces) if len(pieces) > 1 else pieces[0]
    offsets = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    torch.cumsum(torch.cat(lengths), 0, out=offsets[1:])
    return reads, offsets


def _read_sets(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return [_reads(gen, case, _genome(gen, case["kind"], g), cov) for g, cov in _samples(case)]


def _plan():
    plan = _plans.get("plan")
    if plan is None:
        plan = _plans["plan"] = KmerCounter()
    return plan


def prepare(case, seed):
    sets = _read_sets(case, seed)
    rooms = [_room(case, g, cov) for g, cov in _samples(case)]
    width = 1 if case["k"] <= 32 else 2
    state = {"call": case["call"], "k": case["k"], "canonical": case["canonical"], "plan": _plan()}
    if case["call"] == "host":
        state["sets"] = [(reads.cpu().pin_memory(), offsets.cpu().pin_memory(), reads.numel(),
                          torch.zeros(room * width, dtype=torch.int64).pin_memory(),
                          torch.zeros(room, dtype=torch.int32).pin_memory())
                         for (reads, offsets), room in zip(sets, rooms)]
    else:
        state["sets"] = [(reads, offsets, reads.numel()) for reads, offsets in sets]
        shape = (sum(rooms),) if width == 1 else (sum(rooms), 2)
        state["keys"] = torch.zeros(shape, dtype=torch.int64, device="cuda")
        state["counts"] = torch.zeros(sum(rooms), dtype=torch.int32, device="cuda")
    return state


def _keep(state, results):
    """The results in the program's own table; they are released."""
    sizes = [r.n for r in results]
    total = sum(sizes)
    torch.cat([r.keys_tensor() for r in results], out=state["keys"][:total])
    torch.cat([r.counts_tensor() for r in results], out=state["counts"][:total])
    windows = [r.n_valid_windows for r in results]
    for r in results:
        r.free()
    return {"keys": state["keys"], "counts": state["counts"], "sizes": np.array(sizes), "windows": np.array(windows)}


def run(state):
    plan, k, canonical, sets = state["plan"], state["k"], state["canonical"], state["sets"]
    if state["call"] == "count":
        return _keep(state, [plan.count(sets[0][0], sets[0][1], k, canonical)])
    if state["call"] == "submit":
        return _keep(state, [plan.wait(plan.submit(sets[0][0], sets[0][1], k, canonical, n_bases=sets[0][2]))])
    if state["call"] == "batch":
        return _keep(state, plan.count_batch(sets, k, canonical))
    jobs = []
    for reads, offsets, n, keys, counts in sets:
        job = plan.submit(reads, offsets, k, canonical, n_bases=n)
        plan.copy_to_host(job, keys, counts)
        jobs.append(job)
    sizes, windows = [], []
    for job in jobs:
        res = plan.wait(job)
        sizes.append(res.n)
        windows.append(res.n_valid_windows)
        res.free()
    return {"keys": [s[3] for s in sets], "counts": [s[4] for s in sets], "sizes": np.array(sizes),
            "windows": np.array(windows)}


# ------------------------------------------------------------------ the same, computed plainly
def _exact_one(reads, offsets, k, canonical):
    """Sorted histogram of the windows' keys in plain torch: (keys, counts, windows)."""
    dev, n = reads.device, reads.numel()
    code = torch.full((256,), 4, dtype=torch.int64, device=dev)
    for i, letter in enumerate("ACGT"):
        code[ord(letter)] = code[ord(letter.lower())] = i
    c = code[reads.long()]
    read = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    read.index_add_(0, offsets[:-1], torch.ones(offsets.numel() - 1, dtype=torch.int64, device=dev))
    read = read.cumsum(0)[:n]
    bad = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    torch.cumsum((c > 3).long(), 0, out=bad[1:])
    m = n - k + 1
    ok = (read[:m] == read[k - 1:]) & (bad[k:] == bad[:m])
    first = torch.nonzero(ok).flatten()
    f = [torch.zeros_like(first), torch.zeros_like(first)]  # words of the forward key: high, low
    r = [torch.zeros_like(first), torch.zeros_like(first)]
    for d in range(k):
        digit, word = c[first + d], 1 if k - 1 - d < 32 else 0
        f[word] = (f[word] << 2) | digit
        word, digit = 1 if d < 32 else 0, 3 - digit
        r[word] = r[word] | (digit << (2 * (d % 32)))
    sign = -(1 << 63)
    if canonical:
        less = ((r[0] ^ sign) < (f[0] ^ sign)) | ((r[0] == f[0]) & ((r[1] ^ sign) < (f[1] ^ sign)))
        f = [torch.where(less, y, x) for x, y in zip(f, r)]
    if k <= 32:
        keys, counts = torch.unique_consecutive((f[1] ^ sign).sort()[0], return_counts=True)
        return keys ^ sign, counts, first.numel()
    order = (f[1] ^ sign).argsort()
    order = order[(f[0][order] ^ sign).argsort(stable=True)]
    pairs = torch.stack([f[1][order], f[0][order]], 1)  # low word first
    new = torch.ones(len(pairs), dtype=torch.bool, device=dev)
    new[1:] = (pairs[1:] != pairs[:-1]).any(1)
    at = torch.nonzero(new).flatten()
    return pairs[at], torch.diff(torch.cat([at, at.new_tensor([len(pairs)])])), first.numel()


def _padded(pieces, room, device):
    x = torch.cat(pieces)
    out = torch.zeros((room,) + x.shape[1:], dtype=x.dtype, device=device)
    out[: x.shape[0]] = x
    return out


def exact(case, seed):
    if sum(g * cov for g, cov in _samples(case)) > 150e6:
        return None
    rooms = [_room(case, g, cov) for g, cov in _samples(case)]
    got = [_exact_one(reads, offsets, case["k"], case["canonical"]) for reads, offsets in _read_sets(case, seed)]
    sizes, windows = np.array([len(c) for _, c, _ in got]), np.array([w for _, _, w in got])
    if case["call"] == "host":
        keys = [_padded([k.flatten()], room * k[:1].numel(), "cpu") for (k, _, _), room in zip(got, rooms)]
        counts = [_padded([c.int()], room, "cpu") for (_, c, _), room in zip(got, rooms)]
    else:
        keys = _padded([k for k, _, _ in got], sum(rooms), "cuda")
        counts = _padded([c.int() for _, c, _ in got], sum(rooms), "cuda")
    return {"keys": keys, "counts": counts, "sizes": sizes, "windows": windows}
