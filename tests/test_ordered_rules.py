"""Which runs the region-ordered passes take, by the workspace they ask for (host only)."""


def _ws(m, bits, rounds=1, k=25, **kw):
    from paper_1602_05856_gb300 import build, twopaco as T
    build.build()
    return T.twopaco_workspace_size(m, 8, k, bits, rounds, T.Options(**kw))


def test_one_round_takes_the_ordered_passes_where_the_filter_is_beyond_l2_and_dense():
    ordered = lambda m, bits, k=25, **kw: _ws(m, bits, 1, k, **kw) != _ws(m, bits, 1, k, ordered_first_pass=2, **kw)
    assert ordered(310_000_000, 1 << 30) and ordered(310_000_000, 1 << 30, k=63)
    assert ordered(40_000_000, 1 << 30) and not ordered(16_000_000, 1 << 30)  # 4 positions per filter sector
    assert not ordered(310_000_000, 1 << 29)                                 # 64 MiB: within L2
    assert not ordered(310_000_000, 1 << 30, k=64) and not ordered(310_000_000, 1 << 30, hashes=7)
    assert not ordered(310_000_000, 1 << 30, bucket_inserts=2)
    assert ordered(1_000_000, 1 << 24, bucket_inserts=1)
    # two bytes a position and the records instead of eight-byte descriptors and buckets
    assert _ws(310_000_000, 1 << 30) < _ws(310_000_000, 1 << 30, ordered_first_pass=2)


def test_rounds_take_the_ordered_passes_where_the_filter_is_beyond_l2_and_dense():
    auto = lambda m, bits, r, **kw: _ws(m, bits, r, **kw) == _ws(m, bits, r, ordered_first_pass=1, **kw)
    assert auto(200_000_000, 1 << 31, 4)
    assert not auto(100_000_000, 1 << 31, 4) and not auto(200_000_000, 1 << 29, 4)
    assert auto(10_000_000, 1 << 33, 4)                                      # 1 GiB: always


def test_small_workspaces_did_not_grow():
    """What fits the allocation-free run's 32 MiB stays as it was: the direct layout's size
    at these sizes, in bytes."""
    assert _ws(200_000, 1 << 20, table_slots=1 << 20, candidate_records=1 << 18) == 14_710_784
    assert _ws(1_000_000, 1 << 23, 4, table_slots=1 << 19) == 9_810_432

