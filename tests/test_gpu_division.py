"""The division of the normalised output by the output kernel, against the fp64 oracle: blocks of one tile, of even and odd numbers
of tiles, partial last tiles, several segments; and by its own kernel, where O is an operand's array."""
import pytest

from oracle import smat_oracle as so
from paper_2609_36062_b200 import binding, synth
from tests.helpers import device_inputs, rel_err, to_numpy64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,heads,T,c", [(1, 2, 128, 128), (2, 2, 384, 128), (2, 2, 512, 128), (3, 3, 1472, 64), (1, 2, 2624, 64),
                                         (3, 16, 2176, 128)])
def test_rows_leave_divided_by_their_normaliser(d, heads, T, c):
    w = synth.Workload("div", d, 1, heads, T, 128, 128, c, "bf16", "positive", 60 + T)
    host, dev = device_inputs(w)
    plan = binding.SmatPlan(1, heads, T, 128, 128, d, c, "bf16", flags=binding.FLAG_NORMALIZED)
    O = plan.forward_normalized(dev["q"], dev["k"], dev["v"])
    plan.check_status()
    M = so.dense_mask(T, c, d)
    for h in (0, heads - 1):
        Q64, K64, V64 = (synth.as_float64(w, host[x][h]) for x in ("q", "k", "v"))
        ref, den = so.normalized_forward_dense(Q64, K64, V64[:, :-1], M)
        got = to_numpy64(O[0, h])
        assert rel_err(got[:, :-1], ref) <= 2e-2 and rel_err(got[:, -1], den) <= 2e-2   # the stated bound of bf16 plans
    # into Q's array: the row kernel divides what has been rounded, so another half unit in the last place (2^-8) for the sum and
    # one for the normaliser
    into = plan.forward_normalized(dev["q"], dev["k"], dev["v"], O=dev["q"])
    assert into.data_ptr() == dev["q"].data_ptr()
    assert rel_err(to_numpy64(into), to_numpy64(O)) <= 3 * 2.0 ** -8
