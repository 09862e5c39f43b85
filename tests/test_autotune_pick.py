"""The tuner's choice among timed schedules, and that the committed table is made of them."""
import pytest

from paper_2509_26581_gb300 import autotune


def _t(chunk, variant, s):
    return dict(knobs=dict(chunk_edges=chunk, spmv_variant=variant), s_per_iter=s)


@pytest.mark.parametrize("timings,chunk,want", [
    ([_t(256, 2, 1.0), _t(512, 0, 2.0)], None, (256, 2)),
    ([_t(256, 2, 1.0), _t(256, 0, 1.009)], None, (256, 0)),      # within 1 %: the library's choice
    ([_t(256, 2, 1.0), _t(256, 0, 1.011)], None, (256, 2)),
    ([_t(256, 0, 1.0), _t(512, 0, 0.5), _t(512, 3, 0.4)], 256, (256, 0)),   # a table's chunk size is kept
    ([_t(256, 0, 1.0), _t(512, 0, 0.5), _t(512, 3, 0.4)], 512, (512, 3)),
])
def test_pick(timings, chunk, want):
    assert autotune.pick(timings, chunk) == dict(chunk_edges=want[0], spmv_variant=want[1])


def test_every_entry_of_the_table_is_what_its_timings_give():
    table = autotune.load_table()
    assert table
    for key, e in table.items():
        assert e["best"] in [t["knobs"] for t in e["timings"]], key
        assert e["best"] == autotune.pick(e["timings"], e["best"]["chunk_edges"]), key
