"""The work counts that bench.py holds the longest stage against: every stage name that the library can report has one, no
entry is left over, and the counts follow the form of the pass (tables, pooled chunk states, fp32 long-range rows)."""
import os
import re

import pytest

from paper_2609_36062_b200 import binding, roofline

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _geometry(d, T, chunk):
    return binding.SmatPlan(1, 1, T, 128, 128, d, chunk, "bf16").geometry()


def test_every_stage_of_the_library_has_an_entry_and_every_entry_a_stage():
    with open(os.path.join(ROOT, "paper_2609_36062_b200", "csrc", "smat_api.cu")) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    text = text[:text.index("const char* smat_status_string")]
    names = set(re.findall(r'"([a-z]+(?:_[a-z0-9]+)*)"', text))
    assert {"pool", "tiles", "bwd_reads", "segment_output_tc"} <= names
    for d in (1, 3):
        table = roofline.stage_table(2048, 64, 128, 128, 2, _geometry(d, 2048, 64))
        assert set(table) == names
        for work in table.values():
            assert min(work.flops, work.adds, work.bytes) >= 0


def test_an_unknown_stage_is_an_error():
    with pytest.raises(KeyError):
        roofline.stage_work("no_such_stage", 2048, 64, 128, 128, 2, _geometry(3, 2048, 64))


def test_pooling_on_the_alus_includes_the_chunk_states():
    g = _geometry(3, 2048, 64)
    args = (2048, 64, 128, 128, 4, g)
    tables, both = roofline.stage_work("pool", *args), roofline.stage_work("pool", *args, alu_path=True)
    states = 2048 // 64
    assert both.flops - tables.flops == 2 * 2048 * 128 * 128
    assert both.bytes - tables.bytes == (2048 - g.n) * 256 * 4 + states * 128 * 128 * 4   # distant rows are read once


def test_long_range_rows_are_charged_as_they_travel():
    whole, part = _geometry(3, 2048, 64), _geometry(3, 1600, 64)
    assert whole.n % 128 == whole.m % 128 == 0 and part.m % 128 != 0
    for g, size in ((whole, 2), (part, 4)):
        w = roofline.stage_work("segment_output_tc", g.T, 64, 128, 128, 2, g)
        assert w.bytes - g.T * 512 * 2 == g.m * 128 * size
