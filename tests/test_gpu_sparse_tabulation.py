"""The tabulation with the incidence matrix as a sparse operand (q = 17): types on the dense tile and on its border, types
through the last point (added outside the matrix product), one head and several, both stages of d = 4, and the
transposed stages with and without the extra class."""
import numpy as np
import pytest
import torch

from oracle import smat_oracle as so
from paper_2609_36062_b200 import binding, synth
from tests.helpers import device_inputs, rel_err, to_numpy64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,T,q,heads", [(3, 512, 17, 1), (3, 1280, 17, 3), (4, 768, 17, 1)])
def test_types_of_both_kinds_of_tiles_and_through_the_last_point(d, T, q, heads):
    w = synth.Workload("sparse", d, 1, heads, T, 128, 128, 128, "bf16", "normalised", 500 + q)
    _, dev = device_inputs(w)
    plan = binding.SmatPlan(1, heads, T, 128, 128, d, 128, "bf16", q_override=q)
    plan.forward(dev["q"], dev["k"], dev["v"])
    plan.check_status()
    F, U, _ = plan.debug_tables()
    geo = so.geometry(T, 128, d, q)
    points = np.array([so.prof(v, geo) for v in range(geo.P)])
    pairs = [so.type_pair(h, geo) for h in range(geo.B)]
    last = [h for h, (a, b) in enumerate(pairs) if int(points[geo.P - 1] @ np.asarray(a)) % q == b]
    edges = [0, 127, 128, 255, 256, q * q - 1, q * q, q * q + q - 1, geo.B - 1]
    F64 = F[heads - 1].double()
    for h in sorted(set(last[:40] + [e for e in edges if e < geo.B])):
        a, b = pairs[h]
        on = torch.as_tensor((points @ np.asarray(a)) % q == b, device=F.device)
        ref, size = F64[on].sum(0), F64[on].abs().sum(0)
        # one bf16 rounding of an fp32 sum (d = 4: and of its q intermediate sums), as for the generated matrix
        bound = 2.0 ** -8 * ref.abs() + (2.0 ** -20 if d == 3 else 2.0 ** -8) * size + 1e-30
        assert bool(((U[heads - 1, h].double() - ref).abs() <= bound).all()), h


def test_transposed_stages_of_d4_match_the_alu_path():
    q, T = 17, 1024
    w = synth.Workload("sparset", 4, 1, 2, T, 128, 128, 128, "bf16", "normalised", 600)
    _, dev = device_inputs(w, ("q", "k", "v", "do"))
    got, ref = (binding.SmatPlan(1, 2, T, 128, 128, 4, 128, "bf16", q_override=q, flags=f).backward(
        dev["q"], dev["k"], dev["v"], dev["do"]) for f in (0, binding.FLAG_SIMT_ONLY))
    for g, r in zip(got, ref):
        assert rel_err(to_numpy64(g), to_numpy64(r)) <= 2e-2     # the stated bound of bf16 plans
