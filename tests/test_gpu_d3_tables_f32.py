"""The d = 3 tabulation that keeps its sums in registers (fp32 tables): every type state of the last head, for each prime it
is made for, with fewer slabs than CTAs, as many as fill the buffers once, and many rounds of the ring."""
import numpy as np
import pytest
import torch

from oracle import smat_oracle as so
from paper_2609_36062_b200 import binding, synth
from tests.helpers import device_inputs

pytestmark = pytest.mark.gpu


# heads, d_k, d_v: 64, 512 and 6144 slabs of 64 entries
@pytest.mark.parametrize("heads,dk,dv", [(1, 64, 64), (2, 128, 128), (24, 128, 128)])
@pytest.mark.parametrize("q", [11, 13, 17, 19, 23])
def test_every_type_state_is_the_incidence_sum_of_the_profile_table(q, heads, dk, dv):
    w = synth.Workload("d3f32", 3, 1, heads, 1024, dk, dv, 64, "f32", "normalised", 500 + q)
    _, dev = device_inputs(w)
    plan = binding.SmatPlan(1, heads, 1024, dk, dv, 3, 64, "f32", q_override=q)
    plan.forward(dev["q"], dev["k"], dev["v"])
    plan.check_status()
    F, U, _ = plan.debug_tables()
    geo = so.geometry(1024, 64, 3, q)
    assert geo.B == U.shape[1] and geo.P == F.shape[1]
    points = np.array([so.prof(v, geo) for v in range(geo.P)])
    pairs = [so.type_pair(h, geo) for h in range(geo.B)]
    on = np.stack([(points @ np.asarray(a)) % q == b for a, b in pairs])
    on = torch.as_tensor(on, device=F.device, dtype=torch.float64)
    F64 = F[heads - 1].double().reshape(geo.P, -1)
    ref, size = on @ F64, on @ F64.abs()
    # q terms added one by one in fp32: q - 1 roundings of at most 2^-24 of the sum of magnitudes
    assert bool(((U[heads - 1].double().reshape(geo.B, -1) - ref).abs() <= (q - 1) * 2.0 ** -24 * size + 1e-30).all())
