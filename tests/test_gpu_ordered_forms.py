"""The region-ordered passes in one round and over the forms they accept, and pass 2
bucket by bucket, against the direct kernels and the oracle.

One-round runs take the region-ordered passes where bucket_inserts asks for them; pass 2
then runs on the records (k <= 31, at least 64 regions), bucket by bucket (k >= 32 with a
table far beyond L2) or over the candidate list. The junctions must equal the oracle's
element by element, and C_temp the oracle's first pass bit for bit.
"""
import functools

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


def _eq(got, want):
    assert len(got) == len(want)
    for t, (g, w) in enumerate(zip(got, want)):
        assert np.array_equal(np.asarray(g, np.uint64), np.asarray(w, np.uint64)), f"string {t}"


@functools.lru_cache(maxsize=None)
def _input(split=False):
    """Several tiles of 16384 positions, strings that start and end at and around tile and
    16-position boundaries, tandem repeats (palindromes at even k) and a homopolymer."""
    seqs = list(G.named_set("plain_single", 0.04))
    seqs += [s for n in (1, 15, 16, 17, 31, 63, 64, 65, 127, 16383, 16384, 16385)
             for s in G.random_strings(900 + n, 1, n, n)]
    seqs += [np.frombuffer(b"ACGT" * 60, np.uint8), np.frombuffer(b"A" * 20_000, np.uint8)]
    seqs += G.random_strings(78, 30, 0, 300)
    if split:
        seqs = G.plant_n_runs(6, seqs)
    return G.concat(seqs)


FORMS = [  # k, filter bits, hashes, rounds, options: widths of k-mer words and their edges
    (1, 1 << 14, 1, 1, {}), (16, 1 << 16, 4, 1, {}), (17, 1 << 18, 6, 1, {"both_strands": False}),
    (27, 1 << 20, 2, 1, {"split_at_n": True}), (28, 1 << 20, 4, 1, {}), (30, 1 << 18, 3, 5, {"both_strands": False}),
    (31, 1 << 18, 4, 1, {"split_at_n": True}), (32, 1 << 20, 4, 1, {}), (33, 1 << 18, 5, 2, {"split_at_n": True}),
    (62, 1 << 20, 1, 1, {}), (63, 1 << 18, 4, 1, {"partial": True}), (25, 1 << 20, 4, 64, {}),
    (24, 1 << 18, 4, 16, {"split_at_n": True}), (31, 1 << 20, 4, 1, {"partial": True}),
    # a table with room for fewer than 64 parts: the candidate list, which overflows: pass 2 over C_temp
    (25, 1 << 21, 4, 1, {"table_slots": 1 << 15, "candidate_records": 600}),
]


@pytest.mark.parametrize("k,bits,h,rounds,extra", FORMS)
def test_ordered_forms_match_oracle_and_direct(k, bits, h, rounds, extra):
    split, both = extra.get("split_at_n", False), extra.get("both_strands", True)
    bases, off = _input(split)
    m = int(off[-1])
    base = dict(hashes=h, partition_bins=256, **{**dict(table_slots=1 << 20), **extra})
    a = T().DeviceBuild(bases, off, k, bits, rounds, T().Options(bucket_inserts=2, ordered_first_pass=2, **base))
    a.shard_begin(compute_cut=True)
    a.shard_rounds(0, 1)
    a.write_output()
    cut = a.state_tensor(T().STATE_CUTS)
    b = T().DeviceBuild(bases, off, k, bits, rounds,
                        T().Options(bucket_inserts=1, ordered_first_pass=1 if rounds > 1 else 0, **base))
    b.shard_begin(compute_cut=False)
    b.shard_rounds(0, 1, class_cut=cut)
    b.write_output()
    sa, sb = a.stats(), b.stats()
    assert sa["ordered_rounds"] == 0 and sb["ordered_rounds"] >= 1
    for key in ("positions", "pass1_marks", "pass2_marks"):
        assert sa[key] == sb[key], key
    _eq(b.result(), a.result())
    if not extra.get("partial"):
        _eq(b.result(), O.junctions((bases, off), k, both_strands=both, split_n=split))
    if rounds == 1:
        marks, _, _, kept = O.pass1_marks((bases, off), k, bits, h, both_strands=both, split_n=split)
        words = b.state(T().STATE_CANDIDATES, (m + 31) // 32)
        assert np.array_equal(np.unpackbits(words.view(np.uint8), bitorder="little")[:m], marks)


@pytest.mark.parametrize("table_slots,parted", [(1 << 25, True), (1 << 24, False)])
def test_pass2_bucket_by_bucket(table_slots, parted):
    """k = 63 and a saturated filter: 12 M candidates, nearly all distinct, whose table (26 M
    slots of 32 bytes) is far beyond L2. With room for one part per region pass 2 runs
    bucket by bucket; a reserve without it keeps one table and the list."""
    anc = G.random_strings(4242, 1, 6_000_000, 6_000_000)[0]
    rng = np.random.Generator(np.random.PCG64(7))
    seqs = [anc, G.substitute(rng, anc, 0.01)]
    bases, off = G.concat(seqs)
    base = dict(hashes=4, candidate_records=12_000_000)
    a = T().DeviceBuild(bases, off, 63, 1 << 20, 1, T().Options(bucket_inserts=2, table_slots=1 << 25, **base))
    b = T().DeviceBuild(bases, off, 63, 1 << 20, 1, T().Options(bucket_inserts=1, table_slots=table_slots, **base))
    a.run()
    b.run()
    sa, sb = a.stats(), b.stats()
    assert sb["ordered_rounds"] == 1 and sb["pass1_marks"] == sa["pass1_marks"] > 11_000_000
    assert (sb["table_slots"] * 32 > 512 << 20 and sb["table_slots"] > 1 << 24) == parted
    _eq(b.result(), a.result())
