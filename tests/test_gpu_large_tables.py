"""Pass-2 tables beyond 256 MB, which are probed slot by slot, against pass 2 on the ordered
records (a table of its own) and against the smaller tables' sectors."""
import functools

import numpy as np
import pytest

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


@functools.lru_cache(maxsize=None)
def _input():
    """Two strings of 14 Mbp at 1%: 17 M distinct k-mers, 0.3 M junctions."""
    anc = G.random_strings(88, 1, 14_000_000, 14_000_000)[0]
    rng = np.random.Generator(np.random.PCG64(8))
    return G.concat([anc, G.substitute(rng, anc, 0.01), np.frombuffer(b"ACGT" * 50, np.uint8)])


@pytest.mark.parametrize("k,extra", [
    (25, {}), (31, {}), (24, {"candidate_records": 1000}), (31, {"wide_layout": 2}), (27, {"wide_layout": 2}),
    (30, {"both_strands": False}),
])
def test_a_table_beyond_l2(k, extra):
    bases, off = _input()
    wide = k > 27
    one = {x: y for x, y in extra.items() if x == "both_strands"}
    records = T().DeviceBuild(bases, off, k, 1 << 16, 1, T().Options(bucket_inserts=1, **one))
    records.run()
    assert records.stats()["ordered_rounds"] == 1
    # the estimate's 40 M slots (k <= 27) or 35 M of 16 bytes; then a reserve that holds them to
    # 256 MB (slots by sectors), nearly full
    for reserve in (0, 1 << 25) if not wide else (0,):
        run = T().DeviceBuild(bases, off, k, 1 << 16, 1, T().Options(table_slots=reserve, **extra))
        run.run()
        st = run.stats()
        assert st["ordered_rounds"] == 0 and st["pass1_marks"] == st["positions"]
        assert (st["table_slots"] * (16 if wide else 8) > 256 << 20) == (reserve == 0)
        assert st["pass2_marks"] == records.stats()["pass2_marks"] > 200_000
        for a, b in zip(run.result(), records.result()):
            assert np.array_equal(a, b)
