"""Long-range rows formed without tables (smat_lines.cu) at its edges, against the fp64 dense-mask oracle: 16- and 32-row tiles
with one row missing, full and one row over, several row blocks, last steps of 1 to 16 slots, every class of direction, blocks
that are not whole tiles, gates; and the export of tables that the pass has not formed."""
import numpy as np
import pytest
import torch

from oracle import chunkwise_ref as cw
from oracle import smat_oracle as so
from paper_2609_36062_b200 import binding, synth
from tests.helpers import TOL, device_inputs, positional_arrays, rel_err, sample_tokens, to_numpy64

pytestmark = pytest.mark.gpu


def _plan(w, flags=0, q=0):
    return binding.SmatPlan(w.batch, w.heads, w.T, w.d_k, w.d_v, w.d, w.chunk, w.dtype, flags=flags, q_override=q)


def _stages(plan, call):
    plan.profile_enable(True)
    out = call()
    names = [name for name, _ in plan.profile_read()]
    plan.profile_enable(False)
    plan.check_status()
    return out, names


# d, heads, tokens, chunk, field size (0: the default); rows of a type / of a cell, slots of a type / of a cell
CASES = [
    (3, 8, 2048, 128, 0),      # q = 11: 7 or 8 / 8 or 9 rows, 99 / 96 slots
    (3, 20, 2048, 128, 7),     # q = 7: 19 / 21 rows (two tiles, two blocks of one), 147 / 152 slots
    (4, 4, 2048, 64, 0),       # q = 7: 2 or 3 rows, three classes of direction
    (4, 32, 1024, 128, 3),     # q = 3: 13 or 14 / 18 or 19 rows
    (3, 8, 2304, 64, 0),       # odd numbers of tiles: rows in fp32
    (3, 8, 2240, 64, 0),       # blocks that are not whole tiles (forward alone)
    (2, 32, 2112, 64, 0),      # ... d = 2: one cell to a type, 32 rows
    (4, 4, 2240, 64, 0),
]


@pytest.mark.parametrize("d,heads,T,c,q", CASES)
def test_rows_without_tables_match_the_dense_oracle(d, heads, T, c, q):
    w = synth.Workload("lines", d, 1, heads, T, 128, 128, c, "bf16", "normalised", 300 + T + d)
    host, dev = device_inputs(w, ("q", "k", "v", "do"))
    plan = _plan(w, q=q)
    O, names = _stages(plan, lambda: plan.forward(dev["q"], dev["k"], dev["v"]))
    assert "read_lines" in names and "pool_tc" not in names
    F, U, _ = plan.debug_tables()
    grads, names = _stages(plan, lambda: plan.backward(dev["q"], dev["k"], dev["v"], dev["do"]))
    geo = so.geometry(T, c, d, q or None)
    assert ("bwd_dkdv_lines" in names) == (geo.n % 128 == 0 and (T - geo.n) % 128 == 0)
    F2, U2, _ = plan.debug_tables()
    M = so.dense_mask(T, c, d, q or None)
    tables = 1.0 if plan.profile_table_element_bytes() == 2 else 1e-3   # bf16 tables, or fp32: bounds of test_gpu_parity.py
    for h in (0, heads - 1):
        Q64, K64, V64, G64 = (synth.as_float64(w, host[x][h]) for x in ("q", "k", "v", "do"))
        for got, ref in zip((O, *grads), (so.forward_dense(Q64, K64, V64, M), *so.backward_dense(Q64, K64, V64, G64, M))):
            assert rel_err(to_numpy64(got[0, h]), ref) <= TOL["bf16"]
        _, tab = cw.forward(Q64, K64, V64, geo, return_tables=True)
        for got in (F, F2):
            assert rel_err(to_numpy64(got[h]), tab["F"]) <= 8e-3 * tables
        for got in (U, U2):
            assert rel_err(to_numpy64(got[h]), tab["U"]) <= 1.2e-2 * tables


@pytest.mark.parametrize("d,heads,T", [(3, 8, 2048), (4, 4, 2304)])
def test_gated_rows_without_tables_match_the_dense_oracle(d, heads, T):
    w = synth.Workload("glines", d, 1, heads, T, 128, 128, 128, "bf16", "normalised", 400 + T)
    host, dev = device_inputs(w, ("q", "k", "v", "do"))
    rng = np.random.default_rng(T)
    la = np.log(rng.uniform(0.99, 1.0, (heads, T))).astype(np.float32)     # the boundary is within reach
    la_dev = torch.from_numpy(la).cuda()
    plan = _plan(w, binding.FLAG_GATED | binding.FLAG_KEEP_FORWARD_TABLES)
    ws = plan.workspace(for_backward=True)
    plan.profile_enable(True)
    O = plan.forward_gated(dev["q"], dev["k"], dev["v"], la_dev, workspace=ws)
    assert "read_lines" in [name for name, _ in plan.profile_read()]
    grads = plan.backward_gated(dev["q"], dev["k"], dev["v"], la_dev, dev["do"], workspace=ws)
    assert {"bwd_dq_lines", "bwd_dkdv_lines"} <= {name for name, _ in plan.profile_read()}
    plan.profile_enable(False)
    plan.check_status(ws)
    M = so.dense_mask(T, 128, d)
    for h in (0, heads - 1):
        Q64, K64, V64, G64 = (synth.as_float64(w, host[x][h]) for x in ("q", "k", "v", "do"))
        lah = la[h].astype(np.float64)
        assert rel_err(to_numpy64(O[0, h]), so.gated_forward_dense(Q64, K64, V64, M, lah)) <= TOL["bf16"]
        rq, rk, rv, rla = so.gated_backward_dense(Q64, K64, V64, G64, M, lah)
        for got, ref in zip(grads[:3], (rq, rk, rv)):
            assert rel_err(to_numpy64(got[0, h]), ref) <= TOL["bf16"]
        assert rel_err(to_numpy64(grads[3].reshape(heads, T)[h]), rla) <= 5e-2   # (the stated bound of the gate gradient)


def test_two_tiles_of_rows_at_full_length():
    """q = 23, 16 or 17 rows to a type, in two tiles of 16: sampled rows of a long forward pass."""
    w = synth.Workload("long", 3, 1, 4, 18432, 128, 128, 128, "bf16", "normalised", 77)
    host, dev = device_inputs(w)
    plan = _plan(w)
    O, names = _stages(plan, lambda: plan.forward(dev["q"], dev["k"], dev["v"]))
    assert "read_lines" in names
    geo = so.geometry(w.T, w.chunk, w.d)
    rows = sample_tokens(geo, 64, seed=5)
    Q64, K64, V64 = (synth.as_float64(w, host[x][3]) for x in ("q", "k", "v"))
    assert rel_err(to_numpy64(O[0, 3][rows]), so.forward_rows(Q64, K64, V64, geo, rows)) <= TOL["bf16"]


def test_non_finite_tokens_reach_no_row_that_does_not_see_them():
    """An unseen token is never gathered, and a slot without a token gathers one that its rows see: rows whose hyperplane misses
    the cell keep their bits."""
    w = synth.Workload("nan", 3, 1, 8, 2048, 128, 128, 128, "bf16", "normalised", 91)
    _, dev = device_inputs(w)
    plan = _plan(w)
    clean = plan.forward(dev["q"], dev["k"], dev["v"])
    s = 5
    k, v = dev["k"].clone(), dev["v"].clone()
    k[0, 3, s], v[0, 3, s] = float("nan"), float("inf")
    dirty = plan.forward(dev["q"], k, v)
    plan.check_status()
    geo = so.geometry(w.T, w.chunk, w.d)
    unseen = torch.from_numpy(so.mask_col(s, geo)[geo.n:] == 0).cuda()
    assert unseen.any() and not unseen.all()
    assert torch.equal(dirty[0, 3, geo.n:][unseen], clean[0, 3, geo.n:][unseen])
    assert not torch.isfinite(dirty[0, 3, geo.n:][~unseen].float()).any(dim=-1).any()
    others = [h for h in range(8) if h != 3]
    assert torch.equal(dirty[0, others], clean[0, others])


# (d = 3: 2 heads, 31 rows; d = 2: two tiles of 16 rows; d = 4)
@pytest.mark.parametrize("d,heads,T", [(3, 2, 2240), (2, 32, 2112), (4, 4, 2240)])
def test_scores_keep_all_bits_where_tables_would_be_fp32(d, heads, T):
    """Two tokens of a cell whose scores are 1 + 2^-10 + 2^-20 and 1 + 2^-10 and whose values are opposite: what a row gets is
    2^-20, exactly, as from an fp32 table (every sum on the way has at most 21 bits).  16 bits of a score would leave nothing."""
    plan = binding.SmatPlan(1, heads, T, 128, 128, d, 64, "bf16")
    assert plan.profile_table_element_bytes() == 4
    geo = so.geometry(T, 64, d)
    q, k, v = (torch.zeros(1, heads, T, 128, device="cuda", dtype=torch.bfloat16) for _ in range(3))
    signs = torch.randint(0, 2, (heads, 128), generator=torch.Generator().manual_seed(T)).mul_(2).sub_(1).cuda().bfloat16()
    first, second = 3, 3 + geo.P
    assert second < geo.n
    q[..., :3] = 1
    k[0, :, (first, second), :2] = torch.tensor([1.0, 2.0 ** -10], device="cuda", dtype=torch.bfloat16)
    k[0, :, first, 2] = 2.0 ** -20
    v[0, :, first], v[0, :, second] = signs, -signs
    O, names = _stages(plan, lambda: plan.forward(q, k, v))
    assert "read_lines" in names
    seen = torch.from_numpy(so.mask_col(first, geo)[geo.n:] != 0).cuda()
    assert seen.any() and not seen.all()
    assert torch.equal(O[0, :, geo.n:][:, seen], (signs * 2.0 ** -20)[:, None].expand(-1, int(seen.sum()), -1))
    assert not O[0, :, geo.n:][:, ~seen].any()


# even and odd numbers of tiles, row tiles of 16 and 32, several row blocks, partial tiles (forward alone)
@pytest.mark.parametrize("d,heads,T,c,q", [(3, 8, 2048, 128, 0), (3, 16, 2176, 128, 0), (2, 40, 3456, 128, 0), (3, 20, 2048, 128, 7),
                                           (4, 8, 4096, 64, 0), (3, 8, 2240, 64, 0)])
def test_rows_without_tables_agree_with_rows_from_tables(d, heads, T, c, q):
    """The positional call against the routed one with the same assignment.  Stored values are rounded on both sides (2^-9 of the
    largest each), tables twice (F, U), scores once, all to eight bits: five times 2^-9 in all."""
    w = synth.Workload("both", d, 1, heads, T, 128, 128, c, "bf16", "normalised", 500 + T)
    _, dev = device_inputs(w, ("q", "k", "v", "do"))
    plan = _plan(w, q=q)
    arrays = positional_arrays(plan)
    args = [dev[x] for x in ("q", "k", "v")]
    a, ran = _stages(plan, lambda: plan.forward(*args))
    b, ran_tables = _stages(plan, lambda: plan.forward(*args, **arrays))
    assert "read_lines" in ran and "read_lines" not in ran_tables
    assert torch.equal(a, plan.forward(*args)) and torch.equal(b, plan.forward(*args, **arrays))   # (each repeats itself)
    got = [(a, b)]
    if plan.geometry().n % 128 == 0:
        got += zip(plan.backward(*args, dev["do"]), plan.backward(*args, dev["do"], **arrays))
    plan.check_status()
    for x, y in got:
        assert rel_err(to_numpy64(x), to_numpy64(y)) <= 5 * 2.0 ** -9


@pytest.mark.parametrize("forward,backward", [("positions", "positions"), ("positions", "arrays"), ("arrays", "positions"), ("arrays", "arrays")])
@pytest.mark.parametrize("between", [None, "positions", "arrays"])
def test_kept_passes_in_any_order_of_routed_and_positional(forward, backward, between):
    """KEEP_FORWARD_TABLES on a plan whose positional passes form no tables: a backward builds what the forward of its workspace
    has not left, whichever forward the plan has run last (`between`: one of other inputs on a workspace of its own)."""
    w = synth.Workload("orders", 3, 1, 8, 2048, 128, 128, 128, "bf16", "normalised", 97)
    host, dev = device_inputs(w, ("q", "k", "v", "do"))
    plan = _plan(w, binding.FLAG_KEEP_FORWARD_TABLES)
    arrays = positional_arrays(plan)
    pick = {"positions": {}, "arrays": arrays}
    args = [dev[x] for x in ("q", "k", "v")]
    ws = plan.workspace(for_backward=True).fill_(255)             # (nothing of another run's tables)
    plan.forward(*args, workspace=ws, **pick[forward])
    if between:
        plan.forward(dev["k"], dev["q"], dev["do"], workspace=torch.empty_like(ws), **pick[between])
    grads = plan.backward(*args, dev["do"], workspace=ws, **pick[backward])
    plan.check_status(ws)
    F, U, _ = plan.debug_tables(workspace=ws)
    M = so.dense_mask(w.T, w.chunk, w.d)
    for h in (0, 7):
        Q64, K64, V64, G64 = (synth.as_float64(w, host[x][h]) for x in ("q", "k", "v", "do"))
        for got, ref in zip(grads, so.backward_dense(Q64, K64, V64, G64, M)):
            assert rel_err(to_numpy64(got[0, h]), ref) <= TOL["bf16"]
        _, tab = cw.forward(Q64, K64, V64, so.geometry(w.T, w.chunk, w.d), return_tables=True)
        assert rel_err(to_numpy64(F[h]), tab["F"]) <= 8e-3 and rel_err(to_numpy64(U[h]), tab["U"]) <= 1.2e-2   # (bf16 tables)


@pytest.mark.parametrize("d,heads,T", [(4, 1, 704), (3, 5, 192), (3, 8, 2240)])   # few states (no memset in front), and many
def test_a_pass_without_tables_begins_with_a_clean_status_word(d, heads, T):
    w = synth.Workload("clean", d, 1, heads, T, 128, 128, 64, "bf16", "normalised", 98)
    host, dev = device_inputs(w)
    plan = _plan(w)
    plan.workspace().fill_(255)                                   # as a pass whose waits ran out would leave it
    O, names = _stages(plan, lambda: plan.forward(dev["q"], dev["k"], dev["v"]))   # (checks the status)
    assert names[0] == "read_lines"
    M = so.dense_mask(T, 64, d)
    Q64, K64, V64 = (synth.as_float64(w, host[x][0]) for x in ("q", "k", "v"))
    assert rel_err(to_numpy64(O[0, 0]), so.forward_dense(Q64, K64, V64, M)) <= 2.0 ** -8   # (rounding of the stored rows)
    F, U, _ = plan.debug_tables()
    _, tab = cw.forward(Q64, K64, V64, so.geometry(T, 64, d), return_tables=True)
    assert rel_err(to_numpy64(F[0]), tab["F"]) <= 1e-5 and rel_err(to_numpy64(U[0]), tab["U"]) <= 1e-5
