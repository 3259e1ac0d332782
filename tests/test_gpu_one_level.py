"""Inputs of a single coarse partition are partitioned once (pass A plans the fine partitions,
pass B writes them).  The result is compared with the oracle and with the general two-level
path, which a plan that asks for a partition count takes."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def counters(torch_cuda):
    from paper_2505_04431_gb300 import KmerCounter
    made = {name: KmerCounter(**kw) for name, kw in (
        ("one", {}), ("two", {"n_partitions_hint": 1}), ("one deferred", {"defer_all": True}),
        ("one, small tables", {"table_slots_max": 1024}))}
    yield made
    for c in made.values():
        c.close()


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return torch


def check(torch, counters, reads, offsets, k, canonical):
    want_k, want_c, want_n = oracle.count(reads, offsets, k, canonical)
    r = torch.from_numpy(reads).cuda()
    o = torch.from_numpy(offsets.view(np.int64)).cuda()
    for name, c in counters.items():
        res = c.count(r, o, k, canonical)
        keys, counts = res.to_numpy()
        n = res.n_valid_windows
        res.free()
        assert n == want_n and np.array_equal(keys, want_k) and np.array_equal(counts, want_c), name
        assert (c.stats()["kernel_launches"] == 5) == (name != "two"), name


# one read start to a few tiles of 8192 bases, with the lengths around a tile's edge
@pytest.mark.parametrize("bases", [1, 64, 8191, 8192, 8193, 16383, 70_001, 400_000])
@pytest.mark.parametrize("k,canonical", [(5, True), (21, False), (31, True), (32, True), (33, False), (63, True)])
def test_one_level_sizes(torch_cuda, counters, bases, k, canonical):
    rng = np.random.default_rng(bases * 100 + k)
    reads, offsets = synth.random_reads(rng, max(1, bases // 100), 200)
    reads, offsets = reads[:bases], np.minimum(offsets, bases).astype(np.uint64)
    offsets[-1] = len(reads)
    check(torch_cuda, counters, reads, offsets, k, canonical)


@pytest.mark.parametrize("k", [31, 63])
def test_one_level_uneven_bins(torch_cuda, counters, k):
    # 14 000 distinct keys under one 15-base prefix (one bin, larger than any table), a last
    # bin that holds many keys, and ordinary reads around them
    rng = np.random.default_rng(k)
    acgt = np.frombuffer(b"ACGT", np.uint8)
    n = 14_000
    clump = acgt[rng.integers(0, 4, (n, k))]
    clump[:, :15] = ord("A")
    last = acgt[rng.integers(0, 4, (3000, k))]
    last[:, :16] = ord("T")
    rest = acgt[rng.integers(0, 4, (500, k))]
    reads = np.ascontiguousarray(np.concatenate([rest, clump, last, rest])).reshape(-1)
    offsets = np.arange(0, len(reads) + 1, k, dtype=np.uint64)
    check(torch_cuda, counters, reads, offsets, k, False)
    assert counters["one"].stats()["n_overflow_fine"] > 0


# Two-level counts: the plan and the scans take one block per coarse partition, and the scan of
# the distinct counts one per 4096 possible fine partitions (of which repeats leave few)
@pytest.mark.parametrize("hint,slots,genome", [(1, 64, 700), (2, 64, 5000), (64, 64, 60_000), (4096, 0, 3000)])
def test_two_level_plan_and_scans(torch_cuda, hint, slots, genome):
    from paper_2505_04431_gb300 import KmerCounter
    rng = np.random.default_rng(hint + genome)
    acgt = np.frombuffer(b"ACGT", np.uint8)
    g = acgt[rng.integers(0, 4, genome)]
    starts = rng.integers(0, genome - 100, 6000)
    reads = np.ascontiguousarray(g[starts[:, None] + np.arange(100)]).reshape(-1)
    offsets = np.arange(0, len(reads) + 1, 100, dtype=np.uint64)
    want_k, want_c, _ = oracle.count(reads, offsets, 31, True)
    for kw in ({}, {"defer_all": True}, {"test_fine_sampled": True}):
        c = KmerCounter(n_partitions_hint=hint, table_slots_max=slots, **kw)
        res = c.count(torch_cuda.from_numpy(reads).cuda(), torch_cuda.from_numpy(offsets.view(np.int64)).cuda(), 31, True)
        keys, counts = res.to_numpy()
        res.free()
        c.close()
        assert np.array_equal(keys, want_k) and np.array_equal(counts, want_c), kw


# From 12 Mi bases on the number of fine partitions decides: a 30x genome leaves few (one level),
# unrelated reads leave more than 2048 (two levels).  Compared with a plan that always takes two.
@pytest.mark.parametrize("genome,few", [(450_000, True), (0, False)])
@pytest.mark.parametrize("k,canonical", [(31, True), (12, True), (32, False)])
@pytest.mark.parametrize("defer", [False, True])
def test_either_level(torch_cuda, genome, few, k, canonical, defer):
    from paper_2505_04431_gb300 import KmerCounter
    torch = torch_cuda
    gen = torch.Generator(device="cuda")
    gen.manual_seed(genome + k)
    n, length = 90_001, 147
    letters = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device="cuda")
    if genome:
        g = torch.randint(0, 4, (genome,), generator=gen, device="cuda")
        at = torch.randint(0, genome - length, (n, 1), generator=gen, device="cuda")
        codes = g[at + torch.arange(length, device="cuda")]
    else:
        codes = torch.randint(0, 4, (n, length), generator=gen, device="cuda")
    reads = letters[codes].reshape(-1)
    offsets = torch.arange(n + 1, device="cuda") * length
    got = []
    for kw in ({}, {"n_partitions_hint": 2}):
        c = KmerCounter(defer_all=defer, **kw)
        res = c.count(reads, offsets, k, canonical)
        got.append((res.keys_tensor().clone(), res.counts_tensor().clone(), res.n_valid_windows, c.stats()["n_fine"]))
        res.free()
        c.close()
    assert got[0][2] == got[1][2] and torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    if k >= 31:
        assert (got[0][3] <= 2048) == few


@pytest.mark.parametrize("k", [12, 16, 21, 31, 32, 33, 48, 63, 64])
def test_sketch_of_sampled_windows(torch_cuda, k):
    """The sketch takes its keys from a thread's noted windows by their index.  Sixteen copies
    of a sequence and eight of each strand have the same canonical keys, so the same estimate
    and the same number of fine partitions; that number gives the distinct keys within 20%:
    5 x (1.04 / sqrt(1024) for the sketch and 1 / sqrt(5900) for the sample it sees), and less
    than 1% for the partitions rounded up in each of four coarse ones."""
    from paper_2505_04431_gb300 import KmerCounter
    rng = np.random.default_rng(k)
    seq = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, 380_000)]
    other = np.frombuffer(b"TGCA", np.uint8)[np.searchsorted(np.frombuffer(b"ACGT", np.uint8), seq)][::-1]
    offsets = torch_cuda.from_numpy(np.arange(17, dtype=np.int64) * len(seq)).cuda()
    for options in ({"n_partitions_hint": 4, "table_slots_max": 256, "table_load": 0.5}, {}):
        c = KmerCounter(**options)
        n_fine = []
        for copies in ([seq] * 16, [seq, other] * 8):
            res = c.count(torch_cuda.from_numpy(np.concatenate(copies)).cuda(), offsets, k)
            distinct = res.n
            res.free()
            n_fine.append(c.stats()["n_fine"])
        c.close()
        assert n_fine[0] == n_fine[1]
        if options:
            assert abs(n_fine[0] * 128 * 0.9 / distinct - 1) < 0.2


@pytest.mark.parametrize("genome", [100_000, 140_000, 700_000])  # two where registers stay empty, one where none does
@pytest.mark.parametrize("k,canonical", [(31, True), (63, True), (21, False)])
def test_fine_partitions_from_the_sketch(torch_cuda, genome, k, canonical):
    """The fine partitions are those that the sketch's estimate gives in double precision (a
    coarse partition of n windows is cut into ceil(n / T), T = 0.9 fine_target K / D rounded up);
    K / T is beyond 16 per SM, where the target is the estimate's alone."""
    from paper_2505_04431_gb300 import KmerCounter
    rng = np.random.default_rng(genome + k)
    length = 100 + k
    n = 2_500_000 // (length - k + 1)
    codes = rng.integers(0, 4, genome)
    at = rng.integers(0, genome - length, n)
    windows = codes[at[:, None] + np.arange(length)].astype(np.uint64)  # [read, base]
    reads = np.frombuffer(b"ACGT", np.uint8)[windows.astype(np.int64)].reshape(-1)
    offsets = np.arange(n + 1, dtype=np.uint64) * length
    last = length - k + 1

    def value(cols, a, b):  # 64-bit value of the bases a .. b - 1 of every window
        v = np.zeros((n, last), np.uint64)
        for i in range(a, b):
            v = (v << np.uint64(2)) | cols(i)
        return v

    fwd = lambda i: windows[:, i:i + last]
    rev = lambda i: np.uint64(3) - windows[:, k - 1 - i:k - 1 - i + last]
    hi_n = max(0, k - 32)
    f = (value(fwd, 0, hi_n), value(fwd, hi_n, k))
    r = (value(rev, 0, hi_n), value(rev, hi_n, k))
    take = ((r[0] < f[0]) | ((r[0] == f[0]) & (r[1] < f[1]))) & canonical
    hi, lo = np.where(take, r[0], f[0]), np.where(take, r[1], f[1])
    top_f, top_r = value(fwd, 0, 16), value(rev, 0, 16)
    x = np.where(take, top_r, top_f)
    y = np.uint64(0xffffffff) - x
    u = np.uint64(0xffffffff) - ((y * y) >> np.uint64(32)) if canonical else x
    n_c = np.bincount((u >> np.uint64(30)).astype(np.int64).reshape(-1), minlength=4)
    sampled = (((top_f + top_r) * np.uint64(0x9E3779B1)) & np.uint64(0xffffffff)) >> np.uint64(26) == 0
    h = ((lo ^ (hi * np.uint64(0xC2B2AE3D27D4EB4F))) * np.uint64(0x9E3779B97F4A7C15))[sampled]
    regs = np.zeros(1024, np.int64)
    low = [int(v) & ((1 << 54) - 1) for v in np.unique(h)]
    np.maximum.at(regs, (np.unique(h) >> np.uint64(54)).astype(np.int64), [min(55 - v.bit_length(), 55) for v in low])
    e = 0.7213 / (1 + 1.079 / 1024) * 1024.0 ** 2 / np.sum(2.0 ** -regs)
    zeros = int(np.sum(regs == 0))
    if e < 2560 and zeros:
        e = 1024 * np.log(1024 / zeros)
    assert (e < 2560) == (genome < 700_000)
    total = n * last
    dup = min(max(total / (64 * e), 1.0), 32.0)
    T = int(np.ceil(35 * max(0.9 * dup, 1.0)))
    assert total / T > 17 * 152
    c = KmerCounter(n_partitions_hint=4, table_slots_max=64)
    res = c.count(torch_cuda.from_numpy(reads.copy()).cuda(), torch_cuda.from_numpy(offsets.view(np.int64)).cuda(), k,
                  canonical)
    assert res.n_valid_windows == total
    res.free()
    got = c.stats()["n_fine"]
    c.close()
    assert got == sum(min(max(1, -(-int(v) // T)), 4096) for v in n_c)


def random_reads_dev(torch, n_bases, seed, genome=0):
    """n_bases bases in reads of 150 (the last one shorter), of a genome or of i.i.d. bases."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n = -(-n_bases // 150)
    if genome:
        g = torch.randint(0, 4, (genome,), generator=gen, device="cuda")
        at = torch.randint(0, genome - 150, (n, 1), generator=gen, device="cuda")
        codes = g[at + torch.arange(150, device="cuda")].reshape(-1)[:n_bases]
    else:
        codes = torch.randint(0, 4, (n_bases,), generator=gen, device="cuda")
    reads = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device="cuda")[codes]
    return reads, torch.clamp(torch.arange(n + 1, device="cuda") * 150, max=n_bases)


def same(torch, a, b):
    return (a.n_valid_windows == b.n_valid_windows and torch.equal(a.keys_tensor(), b.keys_tensor())
            and torch.equal(a.counts_tensor(), b.counts_tensor()))


# the lengths at which one level, the choice by pass A and two levels meet; just below 6 Mi bases
# of 128-bit keys a block of pass A takes several tiles
@pytest.mark.parametrize("k,line", [(31, 12 << 20), (31, 48 << 20), (63, 6 << 20)])
@pytest.mark.parametrize("more", [-1, 0, 1])
@pytest.mark.parametrize("genome", [0, 400_000])
def test_lengths_around_the_paths_lines(torch_cuda, k, line, more, genome):
    from paper_2505_04431_gb300 import KmerCounter
    r, o = random_reads_dev(torch_cuda, line + more, k + genome, genome)
    a, b = KmerCounter(), KmerCounter(n_partitions_hint=8)
    x, y = a.count(r, o, k), b.count(r, o, k)
    assert same(torch_cuda, x, y)
    for res in (x, y):
        res.free()
    a.close()
    b.close()


# one group of batched launches with counts of every path: one level, either level (both
# outcomes), two levels (128-bit keys: beyond 6 Mi bases) and an empty one
@pytest.mark.parametrize("k,canonical,defer", [(31, True, False), (31, True, True), (63, True, False), (21, False, False)])
def test_paths_side_by_side_in_a_batch(torch_cuda, k, canonical, defer):
    from paper_2505_04431_gb300 import KmerCounter
    torch = torch_cuda
    sets = [random_reads_dev(torch, n, i + k, g) for i, (n, g) in enumerate(
        [(300_000, 0), (13_631_489, 0), (13_700_001, 450_000), (1, 0), (5_900_003, 0), (20_000_000, 700_000)])]
    sets.insert(2, (torch.zeros(0, dtype=torch.uint8, device="cuda"), torch.zeros(1, dtype=torch.int64, device="cuda")))
    a, b = KmerCounter(defer_all=defer), KmerCounter(n_partitions_hint=2)
    for i, ((r, o), x) in enumerate(zip(sets, a.count_batch([(r, o, r.numel()) for r, o in sets], k, canonical))):
        y = b.count(r, o, k, canonical)
        assert same(torch, x, y), i
        x.free()
        y.free()
    a.close()
    b.close()
