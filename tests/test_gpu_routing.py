"""User-supplied routing on the GPU (smat_forward_routed / smat_backward_routed) against the fp64 oracle with the same
explicit prof / type arrays: positional arrays must reproduce the positional call bit for bit, a seeded random hash
(uniform, heavily skewed, with empty cells and out-of-range entries) must match the dense-mask products."""
import numpy as np
import pytest
import torch

from oracle import smat_oracle as so
from paper_2609_36062_b200 import binding, synth
from tests.helpers import TOL, device_inputs, rel_err, sample_tokens, to_numpy64

pytestmark = pytest.mark.gpu


def _assignment(w, geo, skew, drop=False):
    cells, types = [], []
    for h in range(w.bh):
        c = synth.hashed_cells(w, h, geo.n, geo.P, skew)
        qcell, qdir = synth.hashed_query_draws(w, h, geo.m, geo.P, geo.A)
        t = np.array([so.type_through_cell(geo, int(a), int(u)) for a, u in zip(qdir, qcell)], dtype=np.int32)
        if drop:                                                 # a few tokens that belong to no cell / no type
            c[3], c[geo.n // 2], t[1], t[geo.m - 1] = -1, geo.P, geo.B + 5, -2
        cells.append(c); types.append(t)
    return np.stack(cells), np.stack(types)


@pytest.mark.parametrize("d,T,c,dtype,q", [(2, 2048, 128, "bf16", 0), (3, 4096, 128, "bf16", 0), (4, 4096, 128, "bf16", 0),
                                           (3, 512, 32, "f32", 0), (4, 1024, 16, "f32", 3), (3, 4096, 128, "bf16", 37)])
def test_positional_arrays_reproduce_the_positional_call(d, T, c, dtype, q):
    dk = 128 if dtype == "bf16" else 64
    w = synth.Workload("pos", d, 1, 2, T, dk, dk, c, dtype, "normalised", 33)
    host, dev = device_inputs(w, ("q", "k", "v", "do"))
    geo = so.geometry(T, c, d, q or None)
    cells, types = so.positional_assignment(geo)
    prof = torch.from_numpy(np.tile(cells, (w.bh, 1))).int().cuda()
    typ = torch.from_numpy(np.tile(types, (w.bh, 1))).int().cuda()
    plan = binding.SmatPlan(w.batch, w.heads, w.T, w.d_k, w.d_v, w.d, w.chunk, w.dtype, q_override=q)
    a = plan.forward(dev["q"], dev["k"], dev["v"]).clone()
    ga = [x.clone() for x in plan.backward(dev["q"], dev["k"], dev["v"], dev["do"])]
    b = plan.forward(dev["q"], dev["k"], dev["v"], prof=prof, type=typ)
    gb = plan.backward(dev["q"], dev["k"], dev["v"], dev["do"], prof=prof, type=typ)
    plan.check_status()
    assert torch.equal(a, b)                                     # same groups, same token order inside every group
    for x, y in zip(ga, gb):
        assert torch.equal(x, y)


@pytest.mark.parametrize("d,T,c,dtype,q,skew,drop", [
    (2, 2048, 128, "bf16", 0, 0.0, False), (3, 4096, 128, "bf16", 0, 0.0, True), (4, 4096, 128, "bf16", 0, 0.0, False),
    (3, 4096, 128, "bf16", 0, 1.2, False),      # heavy cells (hundreds of tokens) and many empty ones
    (4, 8192, 128, "bf16", 0, 1.0, True), (3, 4096, 128, "bf16", 37, 0.0, False),
    (3, 512, 32, "f32", 0, 0.8, True), (2, 384, 16, "f32", 0, 0.0, False), (4, 1024, 16, "f32", 3, 0.0, False),
])
def test_hashed_routing_matches_the_dense_oracle(d, T, c, dtype, q, skew, drop):
    dk = 128 if dtype == "bf16" else 64
    w = synth.Workload("hash", d, 1, 2, T, dk, dk, c, dtype, "normalised", 55 + d)
    host, dev = device_inputs(w, ("q", "k", "v", "do"))
    geo = so.geometry(T, c, d, q or None)
    cells, types = _assignment(w, geo, skew, drop)
    prof, typ = torch.from_numpy(cells).cuda(), torch.from_numpy(types).cuda()
    plan = binding.SmatPlan(w.batch, w.heads, w.T, w.d_k, w.d_v, w.d, w.chunk, w.dtype, q_override=q)
    O = plan.forward(dev["q"], dev["k"], dev["v"], prof=prof, type=typ)
    dQ, dK, dV = plan.backward(dev["q"], dev["k"], dev["v"], dev["do"], prof=prof, type=typ)
    plan.check_status()
    tol = TOL[dtype]
    for h in range(w.bh):
        Q64, K64, V64, G64 = (synth.as_float64(w, host[x][h]) for x in ("q", "k", "v", "do"))
        if T <= 1024:
            M = so.routed_dense_mask(geo, cells[h], types[h])
            assert rel_err(to_numpy64(O[0, h]), so.forward_dense(Q64, K64, V64, M)) <= tol
            for got, ref in zip((dQ, dK, dV), so.backward_dense(Q64, K64, V64, G64, M)):
                assert rel_err(to_numpy64(got[0, h]), ref) <= tol
        else:
            rows = sample_tokens(geo, 72, seed=h)
            heavy = np.bincount(cells[h][(cells[h] >= 0) & (cells[h] < geo.P)], minlength=geo.P).argmax()
            rows = sorted(set(rows) | set(np.nonzero(cells[h] == heavy)[0][:6].tolist()))   # keys of the heaviest cell
            assert rel_err(to_numpy64(O[0, h][rows]), so.routed_forward_rows(Q64, K64, V64, geo, cells[h], types[h], rows)) <= tol
            assert rel_err(to_numpy64(dQ[0, h][rows]), so.routed_dq_rows(Q64, K64, V64, G64, geo, cells[h], types[h], rows)) <= tol
            rk, rv = so.routed_dkdv_cols(Q64, K64, V64, G64, geo, cells[h], types[h], rows)
            assert rel_err(to_numpy64(dK[0, h][rows]), rk) <= tol
            assert rel_err(to_numpy64(dV[0, h][rows]), rv) <= tol


def test_routed_call_is_reproducible_and_validates_its_arguments():
    w = synth.Workload("rep", 3, 1, 2, 2048, 128, 128, 128, "bf16", "normalised", 5)
    host, dev = device_inputs(w)
    geo = so.geometry(w.T, w.chunk, w.d)
    cells, types = _assignment(w, geo, 1.0)
    prof, typ = torch.from_numpy(cells).cuda(), torch.from_numpy(types).cuda()
    plan = binding.SmatPlan(w.batch, w.heads, w.T, w.d_k, w.d_v, w.d, w.chunk, w.dtype)
    first = plan.forward(dev["q"], dev["k"], dev["v"], prof=prof, type=typ).clone()
    for _ in range(20):
        assert torch.equal(plan.forward(dev["q"], dev["k"], dev["v"], prof=prof, type=typ), first)
    plan.check_status()
    lib = binding.load_library()
    ws = plan.workspace()
    args = [dev[x].data_ptr() for x in ("q", "k", "v")] + [first.data_ptr()]
    assert lib.smat_forward_routed(plan.handle, *args, None, typ.data_ptr(), ws.data_ptr(), ws.numel(), None) == 1
    assert lib.smat_forward_routed(plan.handle, *args, prof.data_ptr() + 2, typ.data_ptr(), ws.data_ptr(), ws.numel(), None) == 6
    with pytest.raises(ValueError):
        plan.forward(dev["q"], dev["k"], dev["v"], prof=prof[:, :-1].contiguous(), type=typ)


def test_one_type_takes_every_query_of_a_short_batch():
    """One segment per block: the launch of the segment totals has nothing to do, and one CTA of the typed read works
    through all queries of a head.  The output kernel must not start on rows the read has yet to write (NaN before)."""
    w = synth.Workload("one_type", 3, 4, 32, 2048, 128, 128, 128, "bf16", "normalised", 71)
    host, dev = device_inputs(w, ("q", "k", "v"))
    geo = so.geometry(w.T, w.chunk, w.d)
    cells, _ = so.positional_assignment(geo)
    types = np.full(geo.m, 5, dtype=np.int32)
    prof = torch.from_numpy(np.tile(cells, (w.bh, 1))).int().cuda()
    typ = torch.from_numpy(np.tile(types, (w.bh, 1))).int().cuda()
    plan = binding.SmatPlan(w.batch, w.heads, w.T, w.d_k, w.d_v, w.d, w.chunk, w.dtype)
    ws = plan.workspace()
    ws.fill_(0xFF)
    O = plan.forward(dev["q"], dev["k"], dev["v"], workspace=ws, prof=prof, type=typ)
    plan.check_status(ws)
    assert torch.isfinite(O).all()
    M = so.routed_dense_mask(geo, cells, types)
    for h in (0, 77, w.bh - 1):
        Q64, K64, V64 = (synth.as_float64(w, host[x][h]) for x in ("q", "k", "v"))
        assert rel_err(to_numpy64(O.reshape(w.bh, w.T, -1)[h]), so.forward_dense(Q64, K64, V64, M)) <= TOL["bf16"]


def _sizes_to_keys(sizes, count, groups, rng):
    """`count` keys in random order: group g gets sizes[g] of them, the groups behind those what is left, one each in turn."""
    keys = [g for g, s in enumerate(sizes) for _ in range(s)]
    rest = np.arange(count - len(keys)) % (groups - len(sizes)) + len(sizes)
    return rng.permutation(np.concatenate([np.array(keys, dtype=np.int64), rest])).astype(np.int32)


# Group sizes at the edges of the passes and of the parts that a heavy group is handed out in: fp32 passes of 8 with
# remainders of 2, 4 and 8; bf16 query tiles of 32 rows, parts of 128
@pytest.mark.parametrize("dtype,d,T,c,sizes", [
    ("f32", 2, 512, 32, (0, 1, 2, 3, 4, 5, 7, 8, 9, 10, 12, 15, 16, 17, 33)),
    ("bf16", 3, 2048, 128, (0, 1, 31, 32, 33, 127, 128, 129, 160, 257)),
    ("bf16", 3, 2048, 64, (0, 640, 5, 256)),
    ("bf16", 3, 1088, 64, (0, 1, 7, 8, 9, 140)),                 # blocks that are not whole tiles: fp32 tables and reads
])
def test_group_sizes_at_the_edges_of_passes_and_parts(dtype, d, T, c, sizes):
    dk = 128 if dtype == "bf16" else 64
    w = synth.Workload("edges", d, 1, 2, T, dk, dk, c, dtype, "normalised", 91)
    host, dev = device_inputs(w, ("q", "k", "v", "do"))
    geo = so.geometry(T, c, d)
    rng = np.random.default_rng(T)
    cells = np.stack([_sizes_to_keys(sizes[::s], geo.n, geo.P, rng) for s in (1, -1)])   # (the heads differ)
    types = np.stack([_sizes_to_keys(sizes[::s], geo.m, geo.B, rng) for s in (-1, 1)])
    prof, typ = torch.from_numpy(cells).cuda(), torch.from_numpy(types).cuda()
    plan = binding.SmatPlan(w.batch, w.heads, w.T, w.d_k, w.d_v, w.d, w.chunk, w.dtype)
    for _ in range(2):                                           # the second pass starts from what the first one left
        O = plan.forward(dev["q"], dev["k"], dev["v"], prof=prof, type=typ)
        grads = plan.backward(dev["q"], dev["k"], dev["v"], dev["do"], prof=prof, type=typ)
    plan.check_status()
    for h in range(w.bh):
        Q64, K64, V64, G64 = (synth.as_float64(w, host[x][h]) for x in ("q", "k", "v", "do"))
        M = so.routed_dense_mask(geo, cells[h], types[h])
        for got, ref in zip((O, *grads), (so.forward_dense(Q64, K64, V64, M), *so.backward_dense(Q64, K64, V64, G64, M))):
            assert rel_err(to_numpy64(got[0, h]), ref) <= TOL[dtype]


def test_a_heavy_type_is_read_by_many_ctas():
    """All queries of a head share one type: the read takes no longer than a uniform one (twice: the slack), where one CTA per
    head walking all of them takes several times as long."""
    w = synth.Workload("heavy", 3, 1, 16, 16384, 128, 128, 128, "bf16", "normalised", 17)
    _, dev = device_inputs(w)
    plan = binding.SmatPlan(w.batch, w.heads, w.T, w.d_k, w.d_v, w.d, w.chunk, w.dtype)
    geo = plan.geometry()
    prof = torch.randint(geo.P, (w.bh, geo.n), device="cuda", dtype=torch.int32)
    uniform = torch.randint(geo.B, (w.bh, geo.m), device="cuda", dtype=torch.int32)
    plan.profile_enable(True)
    took = []
    for typ in (uniform, torch.full_like(uniform, 5)):
        times = []
        for _ in range(9):
            plan.forward(dev["q"], dev["k"], dev["v"], prof=prof, type=typ)
            torch.cuda.synchronize()
            times.append(dict(plan.profile_read())["read_type_tc"])
        took.append(sorted(times)[4])
    plan.profile_enable(False)
    assert took[1] <= 2 * took[0], took


def test_the_list_builder_takes_no_longer_where_tokens_share_a_cell():
    """The warps rank equal keys a key at a time, not a token at a time (all tokens in one group then take twice as long as a
    uniform hash; half as much again is the slack)."""
    w = synth.Workload("lists", 3, 1, 16, 16384, 128, 128, 128, "bf16", "normalised", 18)
    _, dev = device_inputs(w)
    plan = binding.SmatPlan(w.batch, w.heads, w.T, w.d_k, w.d_v, w.d, w.chunk, w.dtype)
    geo = plan.geometry()
    prof = torch.randint(geo.P, (w.bh, geo.n), device="cuda", dtype=torch.int32)
    typ = torch.randint(geo.B, (w.bh, geo.m), device="cuda", dtype=torch.int32)
    plan.profile_enable(True)
    took = []
    for p, t in ((prof, typ), (torch.full_like(prof, 3), torch.full_like(typ, 5)), (prof % 8, typ % 8)):
        times = []
        for _ in range(9):
            plan.forward(dev["q"], dev["k"], dev["v"], prof=p, type=t)
            torch.cuda.synchronize()
            times.append(dict(plan.profile_read())["routing_lists"])
        took.append(sorted(times)[4])
    plan.profile_enable(False)
    assert max(took) <= 1.5 * took[0], took


# Keys that the 32 lanes of a warp meet: one, two in turn, sixteen twice, four neighbours each, and keys out of range among them
@pytest.mark.parametrize("pattern", ["one", "two", "sixteen", "fours", "dropped"])
def test_lists_of_tokens_whose_neighbours_share_cells(pattern):
    w = synth.Workload("shared", 3, 1, 2, 2048, 128, 128, 128, "bf16", "normalised", 92)
    host, dev = device_inputs(w, ("q", "k", "v", "do"))
    geo = so.geometry(w.T, w.chunk, w.d)

    def keys(count, groups, h):
        t = np.arange(count)
        k = {"one": 0 * t + 7 + h, "two": 3 + t % 2, "sixteen": t % 16 + 5 * (t // 32), "fours": 11 * (t // 4) + h,
             "dropped": np.where(t % 3 == h, groups + t % 2, t % 5)}[pattern]
        return (k if pattern == "dropped" else k % groups).astype(np.int32)

    cells = np.stack([keys(geo.n, geo.P, h) for h in range(2)])
    types = np.stack([keys(geo.m, geo.B, 1 - h) for h in range(2)])
    prof, typ = torch.from_numpy(cells).cuda(), torch.from_numpy(types).cuda()
    plan = binding.SmatPlan(w.batch, w.heads, w.T, w.d_k, w.d_v, w.d, w.chunk, w.dtype)
    O = plan.forward(dev["q"], dev["k"], dev["v"], prof=prof, type=typ)
    grads = plan.backward(dev["q"], dev["k"], dev["v"], dev["do"], prof=prof, type=typ)
    plan.check_status()
    for h in range(2):
        Q64, K64, V64, G64 = (synth.as_float64(w, host[x][h]) for x in ("q", "k", "v", "do"))
        M = so.routed_dense_mask(geo, cells[h], types[h])
        for got, ref in zip((O, *grads), (so.forward_dense(Q64, K64, V64, M), *so.backward_dense(Q64, K64, V64, G64, M))):
            assert rel_err(to_numpy64(got[0, h]), ref) <= TOL["bf16"]
