"""Within-chunk tiles, merged pooling and merged routed reads of the fp32-ALU path (other head widths, fp32 inputs)
against the fp64 dense-mask oracle: 32-row blocks of every chunk width, one and two score-column steps, both operand
orders of unequal head widths, groups longer than a staging pass, with and without gates."""
import numpy as np
import pytest
import torch

from oracle import smat_oracle as so
from paper_2609_36062_b200 import binding, synth
from tests.helpers import device_inputs, rel_err, to_numpy64

pytestmark = pytest.mark.gpu

# fp32: sums of a few thousand products of order one, 2^-24 each; bf16: the rounding of the stored result (2^-8)
TOL = {"f32": 1e-5, "bf16": 2.0 ** -8}
# d, T, d_k, d_v, chunk, dtype
CASES = [(2, 512, 128, 128, 128, "f32"), (3, 768, 64, 128, 128, "f32"), (2, 96, 128, 64, 16, "f32"), (1, 640, 64, 64, 128, "f32"),
         (2, 1024, 64, 64, 128, "bf16"), (3, 384, 128, 64, 64, "bf16"), (4, 320, 64, 128, 32, "bf16"), (2, 2048, 64, 64, 64, "f32")]


@pytest.mark.parametrize("gated", [False, True])
@pytest.mark.parametrize("d,T,dk,dv,c,dtype", CASES)
def test_forward_and_gradients(d, T, dk, dv, c, dtype, gated):
    w = synth.Workload("alu", d, 1, 2, T, dk, dv, c, dtype, "scaled", 5 + T + c)
    host, dev = device_inputs(w, ("q", "k", "v", "do"))
    plan = binding.SmatPlan(1, 2, T, dk, dv, d, c, dtype, flags=binding.FLAG_GATED if gated else 0)
    M = so.dense_mask(T, c, d)
    args = (dev["q"], dev["k"], dev["v"])
    if gated:
        la = np.log(np.random.default_rng(1).uniform(0.98, 1.0, (2, T))).astype(np.float32)
        la_dev = torch.from_numpy(la).cuda()
        O = plan.forward_gated(*args, la_dev)
        grads = plan.backward_gated(*args, la_dev, dev["do"])[:3]
    else:
        O = plan.forward(*args)
        grads = plan.backward(*args, dev["do"])
    plan.check_status()
    for h in range(2):
        Q, K, V, G = (synth.as_float64(w, host[x][h]) for x in ("q", "k", "v", "do"))
        if gated:
            lah = la[h].astype(np.float64)
            refs = (so.gated_forward_dense(Q, K, V, M, lah),) + tuple(so.gated_backward_dense(Q, K, V, G, M, lah)[:3])
        else:
            refs = (so.forward_dense(Q, K, V, M),) + tuple(so.backward_dense(Q, K, V, G, M))
        # gated bf16 plans round the rescaled copies of the inputs once more: two roundings per product on the state path
        tol = TOL[dtype] * (2 if gated and dtype == "bf16" else 1)
        for name, got, ref in zip(("O", "dQ", "dK", "dV"), (O,) + tuple(grads), refs):
            e = rel_err(to_numpy64(got[0, h]), ref)
            assert e <= tol, (name, h, e)


@pytest.mark.parametrize("d,T,dim,c,dtype", [(2, 2048, 64, 64, "f32"), (1, 2048, 128, 128, "f32"), (3, 1536, 64, 128, "bf16")])
def test_outputs_in_the_place_of_operands(d, T, dim, c, dtype):
    """O may be written over Q, K or V, dK over V and dV over any operand: the row blocks of a chunk share K's and V's
    rows, so none may store before all have read."""
    g = torch.Generator(device="cuda").manual_seed(8)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    x = {n: (torch.randn(1, 8, T, dim, generator=g, device="cuda") / dim ** 0.25).to(dt) for n in ("q", "k", "v", "do")}
    plan = binding.SmatPlan(1, 8, T, dim, dim, d, c, dtype)
    O = plan.forward(x["q"], x["k"], x["v"])
    grads = plan.backward(x["q"], x["k"], x["v"], x["do"])
    for place in ("q", "k", "v"):
        y = {n: t.clone() for n, t in x.items()}
        assert torch.equal(plan.forward(y["q"], y["k"], y["v"], O=y[place]), O), place
    for dk_place, dv_place in ((None, "do"), (None, "v"), (None, "k"), (None, "q"), ("v", "do")):
        y = {n: t.clone() for n, t in x.items()}
        got = plan.backward(y["q"], y["k"], y["v"], y["do"], dK=y.get(dk_place), dV=y[dv_place])
        plan.check_status()
        for name, a, b in zip(("dQ", "dK", "dV"), got, grads):
            assert torch.equal(a, b), (name, dk_place, dv_place)
