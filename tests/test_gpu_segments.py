"""The two-level causal branch where its blocks are one segment (no totals), two (the second entered with the first one's
total, no scan) and more (scan), with whole and with partial last tiles, against the dense definition's fp32-ALU form."""
import pytest

from paper_2609_36062_b200 import binding, synth
from tests.helpers import device_inputs, rel_err, to_numpy64

pytestmark = pytest.mark.gpu


# batch x heads and tokens decide the cut into segments per block; d = 1: one block
@pytest.mark.parametrize("d,heads,T,cut", [(2, 64, 2048, (1, 1)), (2, 32, 4096, (2, 2)), (2, 8, 2048, (4, 4)), (1, 128, 2048, (1, 0)),
                                           (1, 64, 4096, (2, 0)), (1, 96, 2112, (3, 0)), (2, 64, 2112, (3, 3)), (2, 32, 3968, (2, 2)),
                                           (2, 32, 2112, (1, 2)), (2, 24, 3136, (2, 3))])
def test_cut_into_one_two_and_more_segments(d, heads, T, cut):
    w = synth.Workload("segments", d, 1, heads, T, 128, 128, 64, "bf16", "normalised", 700 + T)
    _, dev = device_inputs(w)
    got, ref = (binding.SmatPlan(1, heads, T, 128, 128, d, 64, "bf16", flags=f) for f in (0, binding.FLAG_SIMT_ONLY))
    got.profile_enable(True)
    O, R = (p.forward(dev["q"], dev["k"], dev["v"]) for p in (got, ref))
    got.check_status()
    stages = [name for name, _ in got.profile_read()]
    assert ("segment_state_tc" in stages, "segment_scan" in stages) == (max(cut) > 1, max(cut) > 2)
    assert rel_err(to_numpy64(O), to_numpy64(R)) <= 2e-2     # the stated bound of bf16 plans
