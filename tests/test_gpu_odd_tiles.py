"""Forward passes whose blocks are odd numbers of 128-token tiles: the two-level causal branch with long-range rows in fp32, against
the per-tile form and, after it, a backward on what it has kept."""
import pytest

from paper_2609_36062_b200 import binding, synth
from tests.helpers import device_inputs, rel_err, to_numpy64

pytestmark = pytest.mark.gpu


# one tile to a block, one and two, three, many with the odd one in either block; d = 1: one block
@pytest.mark.parametrize("d,heads,T", [(2, 4, 256), (2, 4, 384), (3, 4, 768), (3, 16, 2176), (2, 40, 3456), (1, 4, 128), (1, 16, 3200)])
def test_blocks_of_odd_numbers_of_tiles(d, heads, T):
    w = synth.Workload("odd", d, 1, heads, T, 128, 128, 128, "bf16", "normalised", 800 + T)
    _, dev = device_inputs(w, ("q", "k", "v", "do"))
    plans = [binding.SmatPlan(1, heads, T, 128, 128, d, 128, "bf16", flags=f)
             for f in (binding.FLAG_KEEP_FORWARD_TABLES, binding.FLAG_PER_TILE_STATES)]
    got = []
    for plan in plans:
        ws = plan.workspace(for_backward=True)
        plan.profile_enable(True)
        O = plan.forward(dev["q"], dev["k"], dev["v"], workspace=ws)
        stages = [name for name, _ in plan.profile_read()]
        plan.profile_enable(False)
        assert ("segment_output_tc" in stages) == (plan is plans[0])
        got.append([O, *plan.backward(dev["q"], dev["k"], dev["v"], dev["do"], workspace=ws)])
        plan.check_status(ws)
    # The same sums in another order.  Either side's value is rounded to bf16 when it is stored, half a unit in the last place,
    # 2^-8 of the largest at most; operands (state, scores) on a rounding boundary may fall to different sides, another 2^-8.
    for a, b in zip(*got):
        assert rel_err(to_numpy64(a), to_numpy64(b)) <= 3 * 2.0 ** -8
