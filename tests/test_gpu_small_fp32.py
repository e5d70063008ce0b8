"""The fp32 path where its launches have an SM for every piece of work (16-row tiles, 64 tokens to a pooling pass, the status
word cleared by the pooling launch) against the same head among enough copies of itself that none of that applies: every sum
has the same terms in the same order, so the results are equal bit for bit."""
import pytest
import torch

from paper_2609_36062_b200 import binding
from tests.helpers import rel_err, to_numpy64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,T,chunk,dk,dv,many", [(1, 256, 32, 64, 64, 48), (2, 512, 64, 64, 128, 32), (3, 288, 16, 128, 64, 24),
                                                  (2, 640, 128, 128, 128, 40)])
def test_one_head_equals_one_of_many(d, T, chunk, dk, dv, many):
    g = torch.Generator(device="cuda")
    g.manual_seed(T)
    q, k, v, do = (torch.randn(1, 1, T, n, generator=g, device="cuda") / n ** 0.5 for n in (dk, dk, dv, dv))
    results = []
    for heads in (1, many):
        x = [t.expand(1, heads, T, t.shape[-1]).contiguous() for t in (q, k, v, do)]
        plan = binding.SmatPlan(1, heads, T, dk, dv, d, chunk, "f32")
        ws = plan.workspace(for_backward=True)
        ws.fill_(0x55)                                            # the status word starts as anything
        out = [plan.forward(*x[:3], workspace=ws)]
        plan.check_status(ws)
        ws.fill_(0x55)                                            # (an fp32 backward makes its own tables)
        out += plan.backward(*x, workspace=ws)
        plan.check_status(ws)
        results.append([o[:, -1].clone() for o in out])
    for a, b in zip(*results):
        assert torch.equal(a, b)


@pytest.mark.parametrize("d,T", [(2, 320), (3, 576), (1, 320)])   # blocks of 128 + 192, 256 + 320 and 320 tokens
def test_short_bf16_head_with_partial_tiles_equals_one_of_many(d, T):
    """fp32 tables of a bf16 plan: at most 148 pooled states (64 tokens to a pass, the status word cleared there) and more."""
    g = torch.Generator(device="cuda")
    g.manual_seed(T)
    x = [torch.randn(1, 1, T, 128, generator=g, device="cuda").div(128 ** 0.5).bfloat16() for _ in range(4)]
    results = []
    for heads in (1, 24):
        plan = binding.SmatPlan(1, heads, T, 128, 128, d, 64, "bf16")
        assert plan.uses_tensor_cores() and not (T // 64 // 2 * 64) % 128 == (T - T // 64 // 2 * 64) % 128 == 0
        ws = plan.workspace(for_backward=True)
        many = [t.expand(1, heads, T, 128).contiguous() for t in x]
        ws.fill_(0x55)
        out = [plan.forward(*many[:3], workspace=ws)]
        plan.check_status(ws)
        ws.fill_(0x55)
        out += plan.backward(*many, workspace=ws)
        plan.check_status(ws)
        results.append([o[:, -1].clone() for o in out])
    (O, *grads), (O_many, *grads_many) = results
    assert rel_err(to_numpy64(O), to_numpy64(O_many)) <= 2e-2    # (another cut of the causal branch: the stated bound)
    for a, b in zip(grads, grads_many):                          # fp32 ALUs
        assert torch.equal(a, b)


@pytest.mark.parametrize("d,heads,T,width,apart", [(2, 1, 512, 64, False), (2, 9, 512, 128, False), (2, 10, 512, 128, True),
                                                   (2, 37, 512, 64, False), (2, 38, 512, 64, True), (2, 128, 512, 128, True),
                                                   (3, 8, 1024, 128, False), (3, 8, 2048, 128, True), (1, 1, 512, 64, True)])
def test_where_the_chunk_scan_runs(d, heads, T, width, apart):
    """A launch of its own from the size on where its CTAs would hold up the routed read (148 SMs); results do not depend on it."""
    g = torch.Generator(device="cuda")
    g.manual_seed(heads)
    x = [torch.randn(1, heads, T, width, generator=g, device="cuda") / width ** 0.5 for _ in range(4)]
    plan = binding.SmatPlan(1, heads, T, width, width, d, 64, "f32")
    ref = binding.SmatPlan(1, 1, T, width, width, d, 64, "f32")   # one head: beside the read
    plan.profile_enable(True)
    stages = []
    O = plan.forward(*x[:3])
    torch.cuda.synchronize()
    stages += [name for name, _ in plan.profile_read()]
    grads = plan.backward(*x)
    torch.cuda.synchronize()
    stages += [name for name, _ in plan.profile_read()]
    plan.profile_enable(False)
    assert ("scan" in stages, "bwd_scan" in stages) == (apart, apart)
    last = [t[:, -1:].contiguous() for t in x]
    for a, b in zip((O, *grads), (ref.forward(*last[:3]), *ref.backward(*last))):
        assert torch.equal(a[:, -1:], b)
