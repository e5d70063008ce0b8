"""Forward passes whose blocks are odd numbers of 128-token tiles: the two-level causal branch with long-range rows in fp32, against
the per-tile form and, after it, a backward on what it has kept."""
import pytest
import torch

from oracle import chunkwise_ref as cw
from oracle import smat_oracle as so
from paper_2609_36062_b200 import binding, synth
from tests.helpers import device_inputs, rel_err, to_numpy64

pytestmark = pytest.mark.gpu


# one tile to a block, one and two, three, many with the odd one in either block; d = 1: one block
@pytest.mark.parametrize("d,heads,T", [(2, 4, 256), (2, 4, 384), (3, 4, 768), (3, 16, 2176), (2, 40, 3456), (1, 4, 128), (1, 16, 3200)])
def test_blocks_of_odd_numbers_of_tiles(d, heads, T):
    w = synth.Workload("odd", d, 1, heads, T, 128, 128, 128, "bf16", "normalised", 800 + T)
    _, dev = device_inputs(w, ("q", "k", "v", "do"))
    plans = [binding.SmatPlan(1, heads, T, 128, 128, d, 128, "bf16", flags=f)
             for f in (binding.FLAG_KEEP_FORWARD_TABLES, binding.FLAG_PER_TILE_STATES)]
    got = []
    for plan in plans:
        ws = plan.workspace(for_backward=True)
        plan.profile_enable(True)
        O = plan.forward(dev["q"], dev["k"], dev["v"], workspace=ws)
        stages = [name for name, _ in plan.profile_read()]
        plan.profile_enable(False)
        assert ("segment_output_tc" in stages) == (plan is plans[0])
        got.append([O, *plan.backward(dev["q"], dev["k"], dev["v"], dev["do"], workspace=ws)])
        plan.check_status(ws)
    # The same sums in another order.  Either side's value is rounded to bf16 when it is stored, half a unit in the last place,
    # 2^-8 of the largest at most; operands (state, scores) on a rounding boundary may fall to different sides, another 2^-8.
    for a, b in zip(*got):
        assert rel_err(to_numpy64(a), to_numpy64(b)) <= 3 * 2.0 ** -8


def _export(plan, ws, geo, want):
    """smat_debug_tables itself (the binding asks for states only under PER_TILE_STATES); want: of "F", "U", "S"."""
    b, h, T, _, _ = plan.shape
    size = {"F": geo.P, "U": geo.B, "S": T // 128}
    out = {x: torch.full((b * h, size[x], 128, 128), float("nan"), device="cuda") for x in want}
    code = binding.load_library().smat_debug_tables(plan.handle, ws.data_ptr(), *(out[x].data_ptr() if x in out else None for x in "FUS"), None)
    return code, out


# After a forward of the default flags: odd tiles (with tables, without, d = 1) and an fp32 type table (d = 2, 16 and 31 tiles,
# one state for 8 tokens); after a backward on kept states, blocks of even numbers of tiles too
@pytest.mark.parametrize("d,heads,T,q,flags,step", [
    (2, 4, 384, 0, 0, "forward"), (3, 2, 2304, 0, 0, "forward"), (3, 8, 2304, 0, 0, "forward"), (1, 2, 3200, 0, 0, "forward"),
    (2, 2, 2048, 127, 0, "forward"), (2, 9, 3968, 241, 0, "forward"), (3, 2, 2304, 0, binding.FLAG_KEEP_FORWARD_TABLES, "forward"),
    (3, 2, 2304, 0, binding.FLAG_KEEP_FORWARD_TABLES, "backward"), (2, 2, 2048, 0, binding.FLAG_KEEP_FORWARD_TABLES, "backward"),
    (1, 2, 3200, 0, binding.FLAG_KEEP_FORWARD_TABLES, "backward"), (1, 2, 2048, 0, binding.FLAG_KEEP_FORWARD_TABLES, "backward"),
])
def test_states_entering_the_tiles_are_exported(d, heads, T, q, flags, step):
    w = synth.Workload("left", d, 1, heads, T, 128, 128, 128, "bf16", "normalised", 700 + T)
    host, dev = device_inputs(w, ("q", "k", "v", "do"))
    plan = binding.SmatPlan(1, heads, T, 128, 128, d, 128, "bf16", q_override=q, flags=flags)
    ws = plan.workspace(for_backward=True)
    plan.forward(dev["q"], dev["k"], dev["v"], workspace=ws)
    if step == "backward":
        plan.backward(dev["q"], dev["k"], dev["v"], dev["do"], workspace=ws)
    plan.check_status(ws)
    geo = so.geometry(T, 128, d, q or None)
    code, out = _export(plan, ws, geo, "FUS" if d == 1 else "S")
    assert code == 0
    Q64, K64, V64 = (synth.as_float64(w, host[x][heads - 1]) for x in ("q", "k", "v"))
    _, tab = cw.forward(Q64, K64, V64, geo, return_tables=True)
    ref = tab["Sin"].copy()
    if d == 1:                                                   # the scan carries U_0 = F_0 through the boundary
        ref[geo.n // 128:] += tab["U"][0]
        for x in "FU":
            assert rel_err(to_numpy64(out[x][heads - 1]), tab["U"]) <= 8e-3
    assert rel_err(to_numpy64(out["S"][heads - 1]), ref) <= 8e-3


def test_a_large_causal_batch_leaves_the_state_at_the_boundary():
    w = synth.Workload("boundary", 1, 1, 16, 3200, 128, 128, 128, "bf16", "normalised", 710)
    host, dev = device_inputs(w)
    plan = binding.SmatPlan(1, 16, 3200, 128, 128, 1, 128, "bf16")
    ws = plan.workspace()
    plan.forward(dev["q"], dev["k"], dev["v"], workspace=ws)
    plan.check_status(ws)
    geo = so.geometry(3200, 128, 1)
    code, out = _export(plan, ws, geo, "FU")
    assert code == 0 and _export(plan, ws, geo, "S")[0] == binding.SMAT_ERR_UNSUPPORTED
    for h in (0, 15):
        Q64, K64, V64 = (synth.as_float64(w, host[x][h]) for x in ("q", "k", "v"))
        _, tab = cw.forward(Q64, K64, V64, geo, return_tables=True)
        for x in "FU":
            assert rel_err(to_numpy64(out[x][h]), tab["U"]) <= 8e-3
