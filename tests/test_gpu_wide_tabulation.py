"""The tensor-core tabulation that generates its incidence tiles: type tables (and their transposes, through the gradients)
at the edges of its range — primes whose last tile of outputs holds a few rows or nearly all, one to eight groups of tiles,
slots cut by rows and by lines, fewer items than CTAs and more."""
import numpy as np
import pytest
import torch

from oracle import smat_oracle as so
from paper_2609_36062_b200 import binding, synth
from tests.helpers import device_inputs, positional_arrays, rel_err, stages, to_numpy64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,T,q,heads", [(3, 512, 13, 1), (3, 4096, 13, 5), (4, 768, 13, 1), (3, 768, 17, 2), (3, 512, 19, 1),
                                         (3, 1024, 23, 3), (3, 1024, 47, 1), (3, 768, 53, 2)])
def test_type_table_is_the_incidence_sum_of_the_stored_profile_table(d, T, q, heads):
    w = synth.Workload("wide", d, 1, heads, T, 128, 128, 128, "bf16", "normalised", 300 + q)
    _, dev = device_inputs(w)
    plan = binding.SmatPlan(1, heads, T, 128, 128, d, 128, "bf16", q_override=q)
    _, ran = stages(plan, lambda: plan.forward(dev["q"], dev["k"], dev["v"], **positional_arrays(plan)))   # (forms tables)
    plan.check_status()
    assert ("tabulate_wide" if d == 3 and q > 17 else "tabulate_tc") in ran
    F, U, _ = plan.debug_tables()
    geo = so.geometry(T, 128, d, q)
    types = np.unique(np.concatenate([[0, q - 1, q, geo.B - q - 1, geo.B - q, geo.B - 1],
                                      np.random.default_rng(q).integers(0, geo.B, 40)]))
    points = np.array([so.prof(v, geo) for v in range(geo.P)])
    F64 = F[heads - 1].double()
    for h in types:
        a, b = so.type_pair(int(h), geo)
        on = torch.as_tensor((points @ np.asarray(a)) % q == b, device=F.device)
        ref = F64[on].sum(0)
        # the sum is exact but for fp32 accumulation (2^-24 of the sum of magnitudes per term) and one bf16 rounding;
        # d = 4 rounds its intermediate sums to bf16 too (2^-9 of each, q of them)
        size = F64[on].abs().sum(0)
        bound = 2.0 ** -8 * ref.abs() + (2.0 ** -20 if d == 3 else 2.0 ** -8) * size + 1e-30
        assert bool(((U[heads - 1, int(h)].double() - ref).abs() <= bound).all()), int(h)


@pytest.mark.parametrize("d,T,q", [(3, 512, 13), (4, 1024, 13), (3, 1280, 17)])
def test_transposed_stages_match_the_alu_path(d, T, q):
    w = synth.Workload("widet", d, 1, 3, T, 128, 128, 128, "bf16", "normalised", 400 + q)
    _, dev = device_inputs(w, ("q", "k", "v", "do"))
    plan = binding.SmatPlan(1, 3, T, 128, 128, d, 128, "bf16", q_override=q)
    alu = binding.SmatPlan(1, 3, T, 128, 128, d, 128, "bf16", q_override=q, flags=binding.FLAG_SIMT_ONLY)
    got, ran = stages(plan, lambda: plan.backward(dev["q"], dev["k"], dev["v"], dev["do"], **positional_arrays(plan)))
    plan.check_status()
    assert "bwd_tabulate_t_tc" in ran
    for g, r in zip(got, alu.backward(dev["q"], dev["k"], dev["v"], dev["do"])):
        assert rel_err(to_numpy64(g), to_numpy64(r)) <= 2e-2     # the stated bound of bf16 plans
