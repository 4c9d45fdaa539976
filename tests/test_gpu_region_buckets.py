"""First-pass inserts through region buckets in one round, where the region-ordered passes
do not go: asked for with ordered_first_pass=2, and by default for k > 63 on a dense filter
beyond L2. The same filter as direct inserts and as the oracle's, bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_1602_05856_gb300 import genomes as G

pytestmark = pytest.mark.gpu


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


@pytest.mark.parametrize("k,bits,h,extra", [
    (25, 1 << 20, 4, {}), (25, 1 << 18, 6, {}), (31, 1 << 22, 1, {}), (63, 1 << 20, 6, {}), (32, 1 << 20, 3, {}),
    (21, 1 << 20, 4, {"wide_layout": 1}), (63, 1 << 20, 4, {"wide_layout": 1}), (100, 1 << 20, 4, {}),
    (64, 1 << 18, 6, {"wide_layout": 1}), (25, 1 << 20, 4, {"partial": True}), (24, 1 << 20, 4, {"split_at_n": True}),
    (100, 1 << 20, 5, {"both_strands": False}),
])
def test_one_round_of_bucketed_inserts(k, bits, h, extra):
    """Bucket by bucket, with and without descriptors, every k-mer width; a homopolymer sends
    all its records to one bucket, which overflows into direct ORs."""
    seqs = list(G.named_set("plain_single", 0.05)) + [np.frombuffer(b"A" * 60_000, np.uint8)]
    split, both = extra.get("split_at_n", False), extra.get("both_strands", True)
    if split:
        seqs = G.plant_n_runs(5, seqs)
    bases, off = G.concat(seqs)
    m = int(off[-1])
    base = dict(hashes=h, ordered_first_pass=2, **extra)
    a = T().DeviceBuild(bases, off, k, bits, 1, T().Options(bucket_inserts=2, **base))
    b = T().DeviceBuild(bases, off, k, bits, 1, T().Options(bucket_inserts=1, **base))
    assert b.ws_bytes > a.ws_bytes  # the buckets
    a.run()
    b.run()
    sa, sb = a.stats(), b.stats()
    assert sb["ordered_rounds"] == 0
    for key in ("positions", "pass1_marks", "pass2_marks"):
        assert sa[key] == sb[key], key
    for x, y in zip(b.result(), a.result() if extra.get("partial") else
                    O.junctions((bases, off), k, both_strands=both, split_n=split)):
        assert np.array_equal(x, y)
    marks, _, _, kept = O.pass1_marks((bases, off), k, bits, h, both_strands=both, split_n=split)
    for run in (a, b):
        words = run.state(T().STATE_CANDIDATES, (m + 31) // 32)
        assert np.array_equal(np.unpackbits(words.view(np.uint8), bitorder="little")[:m], marks)
    assert sb["pass1_marks"] == kept


def test_buckets_are_the_default_for_long_k_on_a_dense_filter():
    """k = 100 with 2^30 bits and 22 positions per filter sector."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(100)
    m = 92_000_003
    bases = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device="cuda")[
        torch.randint(0, 4, (m,), generator=g, device="cuda")]
    bases[m // 2:m // 2 + m // 3] = bases[:m // 3].clone()
    off = np.array([0, m // 2, m], np.uint64)
    runs = [T().DeviceBuild(bases, off, 100, 1 << 30, 1, T().Options(bucket_inserts=b, table_slots=1 << 26), capacity=m)
            for b in (0, 2)]
    assert runs[0].ws_bytes > runs[1].ws_bytes
    for r in runs:
        r.run()
    assert runs[0].stats()["pass1_marks"] == runs[1].stats()["pass1_marks"] > 0
    assert np.array_equal(*(r.state(T().STATE_CANDIDATES, (m + 31) // 32) for r in runs))
    for x, y in zip(*(r.result() for r in runs)):
        assert np.array_equal(x, y)
