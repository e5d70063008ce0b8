"""The persistent tile-adjoint kernel: one tile, fewer tiles than SMs, one more than a multiple of the SM count, several
rounds — gradients against the fp32-ALU path, gated and ungated, and the same bits on every repetition."""
import numpy as np
import pytest
import torch

from paper_2609_36062_b200 import binding, synth
from tests.helpers import device_inputs, positional_arrays, rel_err, stages, to_numpy64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gated", [False, True])
@pytest.mark.parametrize("d,T,heads", [(1, 128, 1), (2, 256, 2), (3, 512, 37), (1, 19072, 1), (2, 2560, 23)])
def test_gradients_match_the_alu_path(d, T, heads, gated):
    w = synth.Workload("tiles", d, 1, heads, T, 128, 128, 128, "bf16", "normalised", 700 + T)
    _, dev = device_inputs(w, ("q", "k", "v", "do"))
    base = binding.FLAG_GATED if gated else 0
    plan = binding.SmatPlan(1, heads, T, 128, 128, d, 128, "bf16", flags=base)
    alu = binding.SmatPlan(1, heads, T, 128, 128, d, 128, "bf16", flags=base | binding.FLAG_SIMT_ONLY)
    args = [dev[x] for x in ("q", "k", "v")]
    if gated:
        la = np.log(np.random.default_rng(T).uniform(0.97, 1.0, (heads, T))).astype(np.float32)
        args.append(torch.from_numpy(la).cuda())
    call = (lambda p: p.backward_gated(*args, dev["do"])) if gated else (lambda p: p.backward(*args, dev["do"]))
    got = [x.clone() for x in call(plan)]
    plan.check_status()
    for _ in range(3):
        for x, y in zip(got, call(plan)):
            assert torch.equal(x, y)
    for i, (x, y) in enumerate(zip(got, call(alu))):
        # the stated bounds of bf16 plans: 2e-2 of the largest gradient, 5e-2 for the gate gradient (a suffix sum of
        # differences of two rounded products)
        assert rel_err(x.double().cpu().numpy(), y.double().cpu().numpy()) <= (5e-2 if i == 3 else 2e-2), i


@pytest.mark.parametrize("d,T,heads", [(3, 512, 37), (2, 2560, 23)])
def test_gradients_through_tables_match_the_alu_path(d, T, heads):
    """The same with long-range rows from the adjoint tables, where the positional call forms none."""
    w = synth.Workload("tiles", d, 1, heads, T, 128, 128, 128, "bf16", "normalised", 700 + T)
    _, dev = device_inputs(w, ("q", "k", "v", "do"))
    plan = binding.SmatPlan(1, heads, T, 128, 128, d, 128, "bf16")
    alu = binding.SmatPlan(1, heads, T, 128, 128, d, 128, "bf16", flags=binding.FLAG_SIMT_ONLY)
    args = [dev[x] for x in ("q", "k", "v", "do")]
    got, ran = stages(plan, lambda: plan.backward(*args, **positional_arrays(plan)))
    plan.check_status()
    assert {"pool_tc", "bwd_pool_type_tc", "bwd_dkdv_profile_tc", "bwd_tiles_fused_tc"} <= set(ran)
    for x, y in zip(got, alu.backward(*args)):
        assert rel_err(to_numpy64(x), to_numpy64(y)) <= 2e-2     # the stated bound of bf16 plans
