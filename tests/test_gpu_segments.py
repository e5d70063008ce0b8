"""The two-level causal branch where its blocks are one segment (no totals), two (the second entered with the first one's
total, no scan) and more (scan), with whole and with partial last tiles, against the dense definition's fp32-ALU form."""
import pytest

from paper_2609_36062_b200 import binding, synth
from tests.helpers import device_inputs, rel_err, to_numpy64

pytestmark = pytest.mark.gpu


# batch x heads and tokens decide the cut: blocks of (1, 1), (2, 2), (4, 4) segments, and d = 1 (one block) with one and two
@pytest.mark.parametrize("d,heads,T", [(2, 64, 2048), (2, 32, 4096), (2, 8, 2048), (1, 128, 2048), (1, 64, 4096), (1, 96, 2112),
                                       (2, 64, 2112), (2, 32, 3968)])
def test_cut_into_one_two_and_more_segments(d, heads, T):
    w = synth.Workload("segments", d, 1, heads, T, 128, 128, 64, "bf16", "normalised", 700 + T)
    _, dev = device_inputs(w)
    got, ref = (binding.SmatPlan(1, heads, T, 128, 128, d, 64, "bf16", flags=f) for f in (0, binding.FLAG_SIMT_ONLY))
    O, R = (p.forward(dev["q"], dev["k"], dev["v"]) for p in (got, ref))
    got.check_status()
    assert rel_err(to_numpy64(O), to_numpy64(R)) <= 2e-2     # the stated bound of bf16 plans
