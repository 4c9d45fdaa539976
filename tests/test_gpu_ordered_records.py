"""Pass 2 on the region-ordered records at the edges of what it accepts: the smallest
filters, and tables whose parts fill up. Against the oracle, the direct kernels and the
first pass bit for bit."""
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


# Two 31-mers each whose hashes differ only in the two bits below the block index of that
# filter, with one (predecessor, successor) pair each: no junction.
PAIRS = {12: ("AACCTTCGGGAGATACTAACACCTTGTACCT", "TACGGCTGTCTTAACGCTAGAATATGCAAGA"),
         13: ("CACAAGTGATTCCAACTAGAACATGCCAGTC", "TACTATTCAGTCAGAGGACTTGAATCGCCAA")}


@pytest.mark.parametrize("lg_bits", [11, 12, 13, 14])
@pytest.mark.parametrize("rounds", [1, 2])
@pytest.mark.parametrize("strings", [0, 6])
def test_filters_smaller_than_64_blocks(lg_bits, rounds, strings):
    """With as many regions as filter words a region is smaller than a filter block, and its
    number holds bits that are not the hash's: the k-mers' hashes must not come from it."""
    first, second = PAIRS.get(lg_bits, PAIRS[12])
    seqs = [np.frombuffer(s.encode(), np.uint8) for s in ("A" + first + "A", "C" + second + "G")]
    seqs += G.random_strings(31 + lg_bits, strings, 40, 60)  # a filter partly full
    bases, off = G.concat(seqs)
    m = int(off[-1])
    base = dict(hashes=2, partition_bins=256, table_slots=1 << 18)
    a = T().DeviceBuild(bases, off, 31, 1 << lg_bits, rounds, T().Options(bucket_inserts=2, ordered_first_pass=2, **base))
    a.shard_begin(compute_cut=True)
    a.shard_rounds(0, 1)
    a.write_output()
    b = T().DeviceBuild(bases, off, 31, 1 << lg_bits, rounds, T().Options(bucket_inserts=1, ordered_first_pass=int(rounds > 1), **base))
    b.shard_begin(compute_cut=False)
    b.shard_rounds(0, 1, class_cut=a.state_tensor(T().STATE_CUTS))
    b.write_output()
    sa, sb = a.stats(), b.stats()
    assert sa["ordered_rounds"] == 0 and sb["ordered_rounds"] >= 1
    _eq(b.result(), O.junctions((bases, off), 31))
    for key in ("positions", "pass1_marks", "pass2_marks"):
        assert sa[key] == sb[key], key
    if rounds == 1:
        marks, _, _, kept = O.pass1_marks((bases, off), 31, 1 << lg_bits, 2)
        words = b.state(T().STATE_CANDIDATES, (m + 31) // 32)
        assert np.array_equal(np.unpackbits(words.view(np.uint8), bitorder="little")[:m], marks)
        assert sb["pass1_marks"] == kept
