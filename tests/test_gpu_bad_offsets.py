"""Read offsets that do not ascend are refused (KC_EINVAL) by every call that counts, whatever
path the count would take, and the plan counts correctly afterwards.  Passes A and B walk the
offsets in steps of their own, so no kernel after pass A may work on such a count."""
import ctypes

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.fixture(scope="module")
def counters(torch_cuda):
    from paper_2505_04431_gb300 import KmerCounter
    made = {"default": KmerCounter(), "two levels": KmerCounter(n_partitions_hint=2),
            "sampled": KmerCounter(test_fine_sampled=True), "direct": KmerCounter(no_smem_buckets=True)}
    yield made
    for c in made.values():
        c.close()


def bad_offsets(kind, n_bases):
    """Offsets from 0 to n_bases that decrease somewhere."""
    good = np.arange(0, n_bases + 1, 150, dtype=np.uint64)
    good[-1] = n_bases
    if kind == "few":
        return np.array([0, n_bases // 2, 100, n_bases], dtype=np.uint64)
    if kind == "swapped":  # one pair in the middle
        m = len(good) // 2
        good[m], good[m + 1] = good[m + 1], good[m]
    elif kind == "past the end":  # a start behind the reads, before the last offset
        good[-2] = n_bases + 12345
    elif kind == "huge":
        good[len(good) // 3] = 1 << 63
    elif kind == "reversed":
        good[1:-1] = good[1:-1][::-1].copy()
    elif kind == "after empty reads":  # more offsets than the tiles' blocks would look at
        good = np.concatenate([good, np.full(400_000, n_bases, np.uint64)])
        good[-2] -= np.uint64(1)
    return good


KINDS = ["few", "swapped", "past the end", "huge", "reversed", "after empty reads"]


def assert_counts(counter, torch, reads, offsets, k, canonical):
    res = counter.count(torch.from_numpy(reads).cuda(), torch.from_numpy(offsets.view(np.int64)).cuda(), k, canonical)
    keys, counts = res.to_numpy()
    n = res.n_valid_windows
    res.free()
    want_k, want_c, want_n = oracle.count(reads, offsets, k, canonical)
    assert n == want_n and np.array_equal(keys, want_k) and np.array_equal(counts, want_c)


@pytest.mark.parametrize("n_bases", [8000, 300_000])
@pytest.mark.parametrize("k,canonical", [(15, True), (31, False), (33, True), (63, True), (64, False)])
def test_decreasing_offsets_are_refused(torch_cuda, counters, n_bases, k, canonical):
    from paper_2505_04431_gb300 import KC_EINVAL, KcError, load_library
    torch, lib = torch_cuda, load_library()
    rng = np.random.default_rng(n_bases + k)
    reads = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, n_bases)]
    r = torch.from_numpy(reads).cuda()
    good = np.arange(0, n_bases + 1, 100, dtype=np.uint64)
    good_dev = torch.from_numpy(good.view(np.int64)).cuda()
    for kind in KINDS:
        bad = bad_offsets(kind, n_bases)
        o = torch.from_numpy(bad.view(np.int64)).cuda()
        for c in counters.values():
            for call in (lambda: c.count(r, o, k, canonical), lambda: c.count(reads, bad, k, canonical),
                         lambda: c.wait(c.submit(r, o, k, canonical, n_bases=n_bases)),
                         lambda: c.count_batch([(r, good_dev, n_bases), (r, o, n_bases)], k, canonical)):
                with pytest.raises(KcError) as e:
                    call()
                assert e.value.status == KC_EINVAL, (kind, str(e.value))
        jobs = counters["default"].submit_batch([(r, o, n_bases), (r, good_dev, n_bases)], k, canonical)
        with pytest.raises(KcError) as e:
            counters["default"].wait(jobs[0])
        assert e.value.status == KC_EINVAL
        counters["default"].wait(jobs[1]).free()  # its neighbour in the batch is counted
        out_k = torch.empty(2 * n_bases, dtype=torch.int64, device="cuda")
        out_c = torch.empty(n_bases, dtype=torch.int32, device="cuda")
        nd, nv = ctypes.c_uint64(), ctypes.c_uint64()
        st = lib.kc_count_noalloc(r.data_ptr(), o.data_ptr(), len(bad) - 1, k, int(canonical), out_k.data_ptr(),
                                  out_c.data_ptr(), n_bases, ctypes.byref(nd), ctypes.byref(nv),
                                  torch.cuda.current_stream().cuda_stream)
        assert st == KC_EINVAL, kind
    for c in counters.values():
        assert_counts(c, torch, reads, good, k, canonical)


# larger counts: the path chosen by pass A's last block, and two levels
@pytest.mark.parametrize("n_bases,k", [(13 << 20, 31), (13 << 20, 63), (50 << 20, 21)])
def test_decreasing_offsets_of_larger_counts(torch_cuda, counters, n_bases, k):
    from paper_2505_04431_gb300 import KC_EINVAL, KcError
    torch = torch_cuda
    gen = torch.Generator(device="cuda")
    gen.manual_seed(k)
    r = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device="cuda")[
        torch.randint(0, 4, (n_bases,), generator=gen, device="cuda")]
    c = counters["default"]
    for kind in KINDS:
        o = torch.from_numpy(bad_offsets(kind, n_bases).view(np.int64)).cuda()
        with pytest.raises(KcError) as e:
            c.count(r, o, k)
        assert e.value.status == KC_EINVAL, (kind, str(e.value))
    small, offsets = synth.random_reads(np.random.default_rng(k), 2000, 150)
    assert_counts(c, torch, small, offsets.astype(np.uint64), k, True)


# ascending offsets with many empty reads: more offsets than bases
@pytest.mark.parametrize("k", [31, 63])
def test_many_empty_reads(torch_cuda, counters, k):
    rng = np.random.default_rng(k)
    reads = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, 20_000)]
    offsets = np.sort(np.concatenate([np.zeros(200_000), np.arange(0, 20_001, 100), np.full(300_000, 20_000),
                                      np.full(50_000, 12_300)])).astype(np.uint64)
    for c in counters.values():
        assert_counts(c, torch_cuda, reads, offsets, k, True)
