"""The d = 4 tabulation that keeps a slab's intermediate table in shared memory (q = 11): every type state, from a profile
table without empty states, with one or two slabs a CTA and with many rounds of the rings; and that the rows of one entry do
not reach another's."""
import numpy as np
import pytest
import torch

from oracle import smat_oracle as so
from paper_2609_36062_b200 import binding, synth
from tests.helpers import device_inputs

pytestmark = pytest.mark.gpu


# slabs of 64 entries: 256 a head; 1331 points, so that every profile state needs a distant block of as many tokens
@pytest.mark.parametrize("heads,T", [(1, 2816), (4, 4096), (5, 2816)])
def test_every_type_state_is_the_incidence_sum_of_the_profile_table(heads, T):
    w = synth.Workload("slab", 4, 1, heads, T, 128, 128, 128, "bf16", "normalised", 700 + heads)
    _, dev = device_inputs(w)
    plan = binding.SmatPlan(1, heads, T, 128, 128, 4, 128, "bf16", q_override=11)
    plan.forward(dev["q"], dev["k"], dev["v"])
    plan.check_status()
    F, U, _ = plan.debug_tables()
    geo = so.geometry(T, 128, 4, 11)
    assert geo.n >= geo.P
    points = np.array([so.prof(v, geo) for v in range(geo.P)])
    pairs = [so.type_pair(h, geo) for h in range(geo.B)]
    on = np.stack([(points @ np.asarray(a)) % 11 == b for a, b in pairs])
    on = torch.as_tensor(on, device=F.device, dtype=torch.float32)
    for head in (0, heads - 1):
        F64 = F[head].double().reshape(geo.P, -1)
        ref, size = on.double() @ F64, on.double() @ F64.abs()
        # two roundings to bf16, which has eight significant bits: u = 2^-8 of the value rounded.  Of the eleven
        # intermediate sums, together at most u of the sum of magnitudes, and of the result, u (|ref| + u size); the fp32
        # accumulation of 2 x 11 terms adds less than 2^-19 of the sum of magnitudes
        u = 2.0 ** -8
        bound = u * (ref.abs() + u * size) + (u + 2.0 ** -19) * size + 1e-30
        assert bool(((U[head].double().reshape(geo.B, -1) - ref).abs() <= bound).all())


@pytest.mark.parametrize("value", [3.0, float("nan")])
def test_an_entry_does_not_reach_another(value):
    """One column of V changes one column of every state; all other entries of the type table stay bit for bit."""
    w = synth.Workload("slab1", 4, 1, 2, 2816, 128, 128, 128, "bf16", "normalised", 77)
    _, dev = device_inputs(w)
    plan = binding.SmatPlan(1, 2, w.T, 128, 128, 4, 128, "bf16", q_override=11)
    plan.forward(dev["q"], dev["k"], dev["v"])
    _, U, _ = plan.debug_tables()
    for column in (0, 63, 64, 127):
        v = dev["v"].clone()
        v[..., column] = value
        plan.forward(dev["q"], dev["k"], v)
        plan.check_status()
        _, V, _ = plan.debug_tables()
        rest = [j for j in range(128) if j != column]
        assert torch.equal(U[..., rest], V[..., rest]) and not torch.equal(U[..., column], V[..., column])
