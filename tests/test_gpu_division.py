"""The division of the normalised output by the output kernel, and V's ones column set where V is consumed, against the fp64 oracle:
blocks of one tile, of even and odd numbers of tiles, partial last tiles, several segments, with tables and without; and by
kernels of their own, where O is an operand's array."""
import pytest
import torch

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
    # what the caller left in the normaliser column does not matter, to the exported tables either
    tables = plan.debug_tables() if d > 1 else ()
    v = dev["v"].clone()
    v[..., -1] = float("nan")
    assert torch.equal(plan.forward_normalized(dev["q"], dev["k"], v), O)
    for a, b in zip(tables[:2], plan.debug_tables() if d > 1 else ()):
        assert torch.equal(a, b)
    # into an operand's array: the row kernel divides what has been rounded, so another half unit in the last place (2^-8) for the sum and
    # one for the normaliser
    for place in ("q", "v"):
        x = {name: t.clone() for name, t in dev.items()}
        into = plan.forward_normalized(x["q"], x["k"], x["v"], O=x[place])
        assert into.data_ptr() == x[place].data_ptr()
        assert rel_err(to_numpy64(into), to_numpy64(O)) <= 3 * 2.0 ** -8
