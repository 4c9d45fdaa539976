"""Where the region-ordered passes go without being asked for by name: the workspace that
they may take, and the filters about as large as L2 (host only)."""
import random

import pytest

GIB = 1 << 30


def _ws(m, bits, rounds, k=25, **kw):
    from paper_1602_05856_gb300 import build, twopaco as T
    build.build()
    return T.twopaco_workspace_size(m, 8, k, bits, rounds, T.Options(**kw))


@pytest.mark.parametrize("m,lg,rounds,kw", [
    (24_000_000_000, 36, 1, dict(table_slots=1 << 33, candidate_records=1 << 20)),
    (24_000_000_000, 36, 1, dict(table_slots=1 << 30, candidate_records=3_000_000_000)),
    (16_000_000_000, 36, 1, dict(table_slots=1 << 33)),
    (12_000_000_000, 35, 1, dict(table_slots=1 << 30)),
    (6_000_000_000, 34, 1, {}),
    (24_000_000_000, 36, 1, dict(table_slots=1 << 33, bucket_inserts=1)),
    (24_000_000_000, 32, 16, {}),
    (24_000_000_000, 32, 8, dict(k=63)),
])
def test_large_runs_keep_the_direct_workspace(m, lg, rounds, kw):
    assert _ws(m, 1 << lg, rounds, **kw) == _ws(m, 1 << lg, rounds, ordered_first_pass=2, **kw)


def test_automatic_growth_is_bounded():
    rng = random.Random(5)
    ordered = 0
    for _ in range(20_000):
        m = int(1000 * 3e7 ** rng.random())
        rounds = rng.choice((1, 1, 2, 3, 4, 8, 16, 64))
        lg = rng.randint(8, 38 if rounds == 1 else 32)
        kw = dict(k=rng.choice((15, 25, 28, 31, 32, 63, 64)), hashes=rng.choice((3, 4, 6, 7)),
                  bucket_inserts=rng.randint(0, 2 if rounds > 1 else 1), partial=rng.random() < 0.2)
        if rng.random() < 0.5:
            kw["table_slots"] = 1 << rng.randint(2, 33)
        if rng.random() < 0.5:
            kw["candidate_records"] = rng.randint(1, m)
        auto, direct = _ws(m, 1 << lg, rounds, **kw), _ws(m, 1 << lg, rounds, ordered_first_pass=2, **kw)
        assert auto <= direct + 8 * GIB, (m, lg, rounds, kw)
        ordered += auto != direct
    assert ordered > 1000


def test_sizes_within_the_bound_stay_ordered():
    for m, lg, rounds, k in ((338_000_000, 30, 1, 25), (338_000_000, 30, 1, 63), (1_700_000_000, 34, 1, 25),
                             (200_000_000, 31, 4, 25), (2_000_000_000, 32, 8, 25)):
        assert _ws(m, 1 << lg, rounds, k=k) != _ws(m, 1 << lg, rounds, k=k, ordered_first_pass=2)
    # several rounds with a filter of 1 GiB and more: the rule there was, whatever it asks for
    assert _ws(24_000_000_000, 1 << 36, 4) == _ws(24_000_000_000, 1 << 36, 4, ordered_first_pass=1)


@pytest.mark.parametrize("m,k,lg,rounds,kw", [
    (6_450_000, 15, 17, 16, {}), (8_780_000, 63, 18, 12, dict(partial=True)),
    (6_060_000, 31, 22, 24, dict(split_at_n=True)), (8_940_000, 25, 16, 64, dict(table_slots=1 << 18)),
    (5_880_000, 45, 23, 7, dict(table_slots=1 << 16)),
])
def test_asked_for_by_name_the_small_runs_fit_the_allocation_free_scratch(m, k, lg, rounds, kw):
    """Runs just within the 32 MiB with 64 regions, a class byte and a region byte per position."""
    assert _ws(m, 1 << lg, rounds, k=k, ordered_first_pass=1, **kw) <= 32 << 20


@pytest.mark.parametrize("k,partial,least", [(25, False, 9), (31, False, 9), (25, True, 6), (32, False, 16), (63, True, 16)])
def test_one_round_with_a_filter_about_as_large_as_l2(k, partial, least):
    """A 128 MiB filter, nearly in L2: one-round runs below so many positions per 32-byte sector
    are faster direct (17 M positions, k = 25: 0.60 ms direct, 0.75 ordered)."""
    def ordered(m, lg, rounds=1):
        kw = dict(k=k, partial=partial)
        return _ws(m, 1 << lg, rounds, **kw) != _ws(m, 1 << lg, rounds, ordered_first_pass=2, **kw)

    sectors = 1 << 22
    assert not ordered(4 * sectors, 30) and not ordered(least * sectors - 1, 30)
    assert ordered(least * sectors, 30) and ordered(338_000_000, 30)
    # larger filters, and several rounds: from 4 on
    assert ordered(8 * sectors, 31) and not ordered(8 * sectors - 1, 31)
    assert ordered(8 * sectors, 30, 2)
