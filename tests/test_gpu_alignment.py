"""Operands and outputs at an odd multiple of 16 bytes, the alignment the C boundary promises to accept (slices of larger
buffers): every pass gives bit for bit what it gives on freshly allocated tensors, and writes nothing beside its rows."""
import pytest
import torch

from paper_2609_36062_b200 import binding

pytestmark = pytest.mark.gpu

GUARD = -7.0


def _shifted(x):
    """A contiguous copy of x that starts 16 bytes behind an allocation, and the whole buffer."""
    step = 16 // x.element_size()
    buf = torch.full((x.numel() + 2 * step,), GUARD, dtype=x.dtype, device=x.device)
    view = buf[step:-step].view(x.shape)
    view.copy_(x)
    assert view.data_ptr() % 32 == 16
    return view, buf


CASES = [   # name, d, T, chunk, d_k, d_v, dtype, flags
    ("two_level", 3, 2048, 128, 128, 128, "bf16", 0),
    ("causal", 1, 1024, 128, 128, 128, "bf16", 0),
    ("per_tile", 3, 2048, 128, 128, 128, "bf16", binding.FLAG_PER_TILE_STATES),
    ("separate_adjoints", 3, 2048, 128, 128, 128, "bf16", binding.FLAG_SEPARATE_TILE_ADJOINTS),
    ("partial_tiles", 3, 1600, 64, 128, 128, "bf16", 0),
    ("partial_tiles_tables", 2, 1600, 64, 128, 128, "bf16", 0),
    ("no_tables", 4, 5120, 128, 128, 128, "bf16", 0),
    ("no_tables_gated", 4, 5120, 128, 128, 128, "bf16", binding.FLAG_GATED),
    ("partial_tiles_causal", 1, 1088, 64, 128, 128, "bf16", 0),
    ("alu_bf16", 2, 512, 32, 64, 128, "bf16", 0),
    ("alu_f32", 3, 512, 64, 128, 64, "f32", 0),
    ("gated", 3, 2048, 128, 128, 128, "bf16", binding.FLAG_GATED),
    ("gated_f32", 2, 512, 32, 64, 64, "f32", binding.FLAG_GATED),
    ("normalized", 3, 2048, 128, 128, 128, "bf16", binding.FLAG_NORMALIZED),
    ("normalized_partial_tiles", 2, 1600, 64, 128, 128, "bf16", binding.FLAG_NORMALIZED),
]


@pytest.mark.parametrize("name,d,T,chunk,dk,dv,dtype,flags", CASES, ids=[c[0] for c in CASES])
def test_passes_on_sixteen_byte_aligned_tensors(name, d, T, chunk, dk, dv, dtype, flags):
    g = torch.Generator(device="cuda").manual_seed(31)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    rows = lambda dim: torch.randn(1, 2, T, dim, generator=g, device="cuda").to(dt)
    q, k, v, do = rows(dk) / dk ** 0.5, rows(dk) / dk ** 0.5, rows(dv), rows(dv)
    if flags & binding.FLAG_NORMALIZED:
        q, k = q.abs(), k.abs()
    plan = binding.SmatPlan(1, 2, T, dk, dv, d, chunk, dtype, flags=flags)
    ws = plan.workspace(for_backward=True)
    gates = torch.log(torch.rand(2, T, generator=g, device="cuda") * 0.02 + 0.98)

    def both(q, k, v, do, O, dQ, dK, dV):
        if flags & binding.FLAG_GATED:
            plan.forward_gated(q, k, v, gates, O=O, workspace=ws)
            plan.check_status(ws)
            plan.backward_gated(q, k, v, gates, do, dQ=dQ, dK=dK, dV=dV, workspace=ws)
        elif flags & binding.FLAG_NORMALIZED:
            plan.forward_normalized(q, k, v, O=O, workspace=ws)
            plan.check_status(ws)
            for dst, src in zip((dQ, dK, dV), plan.backward_normalized(q, k, v, O, do, workspace=ws)):
                dst.copy_(src)      # (its gradients are always its own)
        else:
            plan.forward(q, k, v, O=O, workspace=ws)
            plan.check_status(ws)
            plan.backward(q, k, v, do, dQ=dQ, dK=dK, dV=dV, workspace=ws)
        plan.check_status(ws)

    ref = [torch.zeros_like(x) for x in (v, q, k, v)]
    both(q, k, v, do, *ref)
    ins = [_shifted(x)[0] for x in (q, k, v, do)]
    outs, bufs = zip(*[_shifted(torch.zeros_like(x)) for x in ref])
    both(*ins, *outs)
    step = 16 // v.element_size()
    for r, o, b in zip(ref, outs, bufs):
        assert torch.equal(r, o)
        assert (b[:step] == GUARD).all() and (b[-step:] == GUARD).all()
