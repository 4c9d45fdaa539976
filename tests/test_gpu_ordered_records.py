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


def _full_parts(k, rounds, seed=5):
    """Distinct k-mers, all of them candidates of a saturated filter: 250 to 260 thousand a
    round, which 2^18 slots hold but 256 parts of 1024 do not (a part's share of them has a
    standard deviation of 31)."""
    n = 259_000 if rounds == 1 else 500_000
    return G.concat(G.random_strings(seed, 1, n, n) + [np.frombuffer(b"ACGT" * 40, np.uint8)])


@pytest.mark.parametrize("k,rounds,extra", [
    (25, 1, {}), (31, 1, {}), (25, 2, {}), (30, 2, {}), (27, 1, {"wide_layout": 1}),
    (31, 1, {"wide_layout": 2}), (24, 1, {"candidate_records": 5000}), (25, 1, {"both_strands": False}),
])
def test_a_full_part_of_the_table_takes_one_table(k, rounds, extra):
    bases, off = _full_parts(k, rounds)
    base = dict(hashes=4, partition_bins=256, table_slots=1 << 18, **extra)
    run = T().DeviceBuild(bases, off, k, 1 << 16, rounds,
                          T().Options(bucket_inserts=1, ordered_first_pass=int(rounds > 1), **base))
    want = O.junctions((bases, off), k, both_strands=extra.get("both_strands", True))
    for again in range(3):  # launched twice, then replayed
        if again == 2:
            run.capture()
        run.run()
        st = run.stats()
        assert st["ordered_rounds"] == rounds and st["table_slots"] == 1 << 18
        assert st["positions"] == st["pass1_marks"]  # saturated: the parts are as full as they get
        assert st["pass2_marks"] == sum(len(w) for w in want)
        _eq(run.result(), want)
    run.release_plan()


@pytest.mark.parametrize("n,slots", [(259_000, 1 << 17), (3_000_000, 1 << 21), (3_000_000, 1 << 20)])
def test_a_full_reserve_is_reported_and_recovered(n, slots):
    """Fewer slots than k-mers: the parts fill up and the one table too. The run says so, and
    the host build grows the reserve and runs again, on the records."""
    bases, off = G.concat(G.random_strings(5, 1, n, n) + [np.frombuffer(b"ACGT" * 40, np.uint8)])
    opts = T().Options(hashes=4, bucket_inserts=1, table_slots=slots)
    run = T().DeviceBuild(bases, off, 25, 1 << 16, 1, opts)
    run.run()
    st = run.stats(check=False)
    assert st["rc"] == T().EOVERFLOW and st["overflow"] and st["ordered_rounds"] == 1
    seqs = [bases[int(off[t]):int(off[t + 1])] for t in range(len(off) - 1)]
    got, st = T().twopaco_build_ex(seqs, 25, 1 << 16, 1, opts)
    _eq(got, O.junctions((bases, off), 25))
    assert st["table_slots"] == 4 * slots and st["ordered_rounds"] == 1


@pytest.mark.parametrize("k,rounds", [(25, 1), (31, 1), (28, 4)])
def test_a_sparse_filter_takes_a_slot_per_record(k, rounds):
    """With fewer than 16 positions per filter sector the parts of the table take 1.25 slots per
    position, but at least 1024 each, whatever the reserve (a round clears them all); a filled
    filter takes it all."""
    bases, off = G.concat(G.named_set("plain_single", 0.3))
    m = int(off[-1])
    want = O.junctions((bases, off), k)
    parts = max(256 * 1024, m // rounds * 5 // 4)  # 256 regions; the records' rounding on top
    for lg, all_of_it in ((26, False), (18, True)):
        run = T().DeviceBuild(bases, off, k, 1 << lg, rounds,
                              T().Options(partition_bins=256, table_slots=1 << 22, bucket_inserts=1,
                                          ordered_first_pass=int(rounds > 1)))
        run.run()
        st = run.stats()
        assert st["ordered_rounds"] == rounds
        if all_of_it:
            assert st["table_slots"] == 1 << 22
        else:
            assert parts <= st["table_slots"] <= parts + 64 * 256 + 4096
        _eq(run.result(), want)
