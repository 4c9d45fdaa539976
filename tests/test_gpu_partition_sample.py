"""The class cut of large inputs, from the partition pre-pass's sample of the k-mers: the
classes hold about the same number of distinct k-mers, whatever the sample comes across."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

K = 25


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_05856_gb300 import build
    build.build()


def T():
    from paper_1602_05856_gb300 import twopaco
    return twopaco


def _random(seed, m):
    rng = np.random.Generator(np.random.PCG64(seed))
    return np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, m, dtype=np.uint8)]


def _offsets(*ends):
    return np.array((0,) + ends, np.uint64)


def _hashes(bases):
    """The library's hash of every k-mer's normalized form (splitmix64's finalizer)."""
    code = np.zeros(256, np.uint64)
    code[list(b"ACGT")] = range(4)
    x, n = code[bases], bases.size - K + 1
    f, r = np.zeros(n, np.uint64), np.zeros(n, np.uint64)
    for j in range(K):
        f = (f << np.uint64(2)) | x[j:j + n]
        r |= (np.uint64(3) - x[j:j + n]) << np.uint64(2 * j)
    z = np.minimum(f, r)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xbf58476d1ce4e5b9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94d049bb133111eb)
    return z ^ (z >> np.uint64(31))


@pytest.mark.parametrize("m,q", [((1 << 23) - 3, 1 << 16), (1 << 23, 1 << 16), ((1 << 23) + 5, 1 << 18),
                                 ((1 << 25) - 1, 1 << 16), ((1 << 25) + 3, 1 << 17), ((1 << 26) + 7, 1 << 16)])
@pytest.mark.parametrize("rounds", [4, 16])
def test_classes_of_a_sampled_cut_are_balanced(m, q, rounds):
    """All k-mers distinct: a class's share, of the counted and of all k-mers, is 1 / rounds. 2^17
    counted k-mers at least: 1.1% of a class of 16, and a bin's granularity on top; 6% is five of it."""
    bases = _random(m, m)
    run = T().DeviceBuild(bases, _offsets(m), K, 1 << 30, rounds,
                          T().Options(partition_bins=q, ordered_first_pass=1, partial=True))
    run.run()
    assert run.stats()["ordered_rounds"] == rounds  # no class beyond a quarter more than its share
    bins, cuts = run.state(T().STATE_BINS, q).astype(np.int64), run.state(T().STATE_CUTS, rounds + 1).astype(np.int64)
    assert 1 << 17 <= bins.sum() <= m
    counted = np.add.reduceat(bins, cuts[:-1]) / bins.sum()
    assert np.all(np.abs(counted * rounds - 1) < 0.06), counted
    H = _hashes(bases[:4_000_000])
    share = np.histogram((H & np.uint64(q - 1)).astype(np.int64), cuts)[0] / H.size
    assert np.all(np.abs(share * rounds - 1) < 0.06), share


@pytest.mark.parametrize("how", ["n", "short", "repeat"])
def test_chunks_that_the_sample_walks_hold_no_or_few_k_mers(how):
    """Every other chunk of 65536 positions holds none (N, or strings shorter than k) or one
    k-mer; the others hold 16 M. Each class gets its share, and the run fits a table of twice
    that (all of them in one class do not). (The repeat's k-mer borders several bases: 16 M junctions.)"""
    m, c, rounds = 1 << 25, 1 << 16, 4
    bases = _random(9, m).reshape(-1, c)
    off = _offsets(m)
    if how == "n":
        bases[::2] = ord("N")
    elif how == "repeat":
        bases[::2] = ord("A")
    else:
        at = np.arange(0, m, 2 * c)[:, None] + np.arange(0, c, 16)[None, :]
        off = np.unique(np.concatenate((at.ravel(), np.arange(0, m + 1, c)))).astype(np.uint64)
    bases = bases.reshape(-1)
    base = dict(split_at_n=how == "n")
    run = T().DeviceBuild(bases, off, K, 1 << 20, rounds, T().Options(table_slots=1 << 23, **base), capacity=m)
    run.run()
    st = run.stats()
    cuts = run.state(T().STATE_CUTS, rounds + 1).astype(np.int64)
    assert np.all(np.abs(np.diff(cuts) - (1 << 16) // rounds) < 1000), cuts
    one = T().DeviceBuild(bases, off, K, 1 << 26, 1, T().Options(**base), capacity=m)
    one.run()
    assert one.stats()["pass2_marks"] == st["pass2_marks"]
    for a, b in zip(run.result(), one.result()):
        assert np.array_equal(a, b)
