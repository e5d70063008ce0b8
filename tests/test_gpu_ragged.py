"""Forward passes whose blocks are not whole 128-token tiles (bf16, 128-wide heads): tensor-core causal branch with
partial last tiles and fp32 tables, against the fp64 dense-mask oracle."""
import numpy as np
import pytest
import torch

from oracle import chunkwise_ref as cw
from oracle import smat_oracle as so
from paper_2609_36062_b200 import binding, synth
from tests.helpers import device_inputs, positional_arrays, rel_err, stages, to_numpy64

pytestmark = pytest.mark.gpu

# (d, T, chunk): last tiles of 16, 32, 48, 64, 80 and 112 rows, one-tile blocks, blocks longer and shorter than a tile,
# a whole first block with a partial second one and the other way round, several segments per block, d = 1 with a partial
# last tile
CASES = [(2, 32, 16), (1, 16, 16), (2, 128, 64), (3, 224, 16), (3, 320, 32), (1, 336, 16), (2, 320, 64), (4, 1120, 16),
         (3, 1472, 64), (2, 2368, 64), (1, 2624, 64), (3, 4288, 64)]


def _case(d, T, c):
    w = synth.Workload("ragged", d, 1, 3, T, 128, 128, c, "bf16", "normalised", 17 + T)
    host, dev = device_inputs(w)
    return w, host, dev


@pytest.mark.parametrize("d,T,c", CASES)
def test_partial_tiles_match_the_dense_oracle(d, T, c):
    w, host, dev = _case(d, T, c)
    plan = binding.SmatPlan(1, 3, T, 128, 128, d, c, "bf16")
    assert plan.uses_tensor_cores() and plan.type_table_element_bytes() == 4
    O = plan.forward(dev["q"], dev["k"], dev["v"])
    plan.check_status()
    alu = binding.SmatPlan(1, 3, T, 128, 128, d, c, "bf16", flags=binding.FLAG_SIMT_ONLY)
    A = alu.forward(dev["q"], dev["k"], dev["v"])
    M = so.dense_mask(T, c, d)
    for h in range(w.bh):
        Q64, K64, V64 = (synth.as_float64(w, host[x][h]) for x in ("q", "k", "v"))
        ref = so.forward_dense(Q64, K64, V64, M)
        # the fp32 tables and the split operands leave the rounding of the stored output, half a bf16 ulp: 2^-8 of the
        # largest value and no more
        assert rel_err(to_numpy64(O[0, h]), ref) <= 2.0 ** -8
        assert np.linalg.norm(to_numpy64(O[0, h]) - ref) <= 1.02 * np.linalg.norm(to_numpy64(A[0, h]) - ref)


# ... and through fp32 tables, where the positional call forms none: the cases of several tiles to a block
@pytest.mark.parametrize("d,T,c", [(3, 320, 32), (4, 1120, 16), (3, 1472, 64), (2, 2368, 64), (3, 4288, 64)])
def test_partial_tiles_through_tables_match_the_dense_oracle(d, T, c):
    w, host, dev = _case(d, T, c)
    plan = binding.SmatPlan(1, 3, T, 128, 128, d, c, "bf16")
    O, ran = stages(plan, lambda: plan.forward(dev["q"], dev["k"], dev["v"], **positional_arrays(plan)))
    plan.check_status()
    assert {"pool", "read_type", "segment_output_tc"} <= set(ran)
    F, U, _ = plan.debug_tables()
    geo = so.geometry(T, c, d)
    M = so.dense_mask(T, c, d)
    for h in range(w.bh):
        Q64, K64, V64 = (synth.as_float64(w, host[x][h]) for x in ("q", "k", "v"))
        assert rel_err(to_numpy64(O[0, h]), so.forward_dense(Q64, K64, V64, M)) <= 2.0 ** -8   # (as above)
        _, tab = cw.forward(Q64, K64, V64, geo, return_tables=True)
        assert rel_err(to_numpy64(F[h]), tab["F"]) <= 1e-5 and rel_err(to_numpy64(U[h]), tab["U"]) <= 1e-5   # fp32 sums


@pytest.mark.parametrize("tables", [False, True])
def test_rows_past_a_block_do_not_reach_it(tables):
    """Non-finite keys and values behind a block's end (of the recent block, of the next head) stay out of its rows."""
    w, _, dev = _case(3, 1472, 64)
    plan = binding.SmatPlan(1, 3, w.T, 128, 128, 3, 64, "bf16")
    n = plan.geometry().n
    arrays = positional_arrays(plan) if tables else {}
    clean = plan.forward(dev["q"], dev["k"], dev["v"], **arrays)
    k, v = dev["k"].clone(), dev["v"].clone()
    k[0, 0, n:], v[0, 0, n:] = float("inf"), float("nan")
    k[0, 2], v[0, 2] = float("nan"), float("inf")
    dirty, ran = stages(plan, lambda: plan.forward(dev["q"], k, v, **arrays))
    plan.check_status()
    assert ("pool" in ran) == tables
    assert torch.equal(dirty[0, 0, :n], clean[0, 0, :n]) and torch.equal(dirty[0, 1], clean[0, 1])


def test_routed_tokens_of_no_group_add_nothing():
    w, host, dev = _case(3, 1120, 16)
    plan = binding.SmatPlan(1, 3, w.T, 128, 128, 3, 16, "bf16")
    geo = so.geometry(w.T, 16, 3)
    rng = np.random.default_rng(2)
    prof = rng.integers(-2, geo.P, (3, geo.n)).astype(np.int32)
    typ = rng.integers(0, geo.B + 3, (3, geo.m)).astype(np.int32)
    O = plan.forward(dev["q"], dev["k"], dev["v"], prof=torch.from_numpy(prof).cuda(), type=torch.from_numpy(typ).cuda())
    plan.check_status()
    rows = np.arange(w.T)
    for h in range(3):
        Q64, K64, V64 = (synth.as_float64(w, host[x][h]) for x in ("q", "k", "v"))
        ref = so.routed_forward_rows(Q64, K64, V64, geo, prof[h], typ[h], rows)
        assert rel_err(to_numpy64(O[0, h]), ref) <= 2.0 ** -8


@pytest.mark.parametrize("d", [3, 1])
def test_chunk_states_are_exported_where_a_pass_leaves_them(d):
    """The two-level forward keeps no state per chunk; a backward does, and so does the forward under PER_TILE_STATES."""
    w, host, dev = _case(d, 1472, 64)
    plain = binding.SmatPlan(1, 3, w.T, 128, 128, d, 64, "bf16")
    plain.forward(dev["q"], dev["k"], dev["v"])
    F, U, Sin = plain.debug_tables()
    assert Sin is None and (F is None) == (U is None) == (d == 1)
    plain.backward(dev["q"], dev["k"], dev["v"], dev["v"])
    states = binding.SmatPlan(1, 3, w.T, 128, 128, d, 64, "bf16", flags=binding.FLAG_PER_TILE_STATES)
    states.forward(dev["q"], dev["k"], dev["v"])
    n = plain.geometry().n
    tables = [p.debug_tables() for p in (plain, states)]
    for h in range(3):
        K64, V64 = (synth.as_float64(w, host[x][h]) for x in ("k", "v"))
        for chunk in (0, 1, n // 64 - 1, n // 64, n // 64 + 1, w.T // 64 - 1):
            lo = 0 if chunk * 64 < n or d == 1 else n
            ref = K64[lo:chunk * 64].T @ V64[lo:chunk * 64]
            for F, U, Sin in tables:
                e = np.abs(to_numpy64(Sin[h, chunk]) - ref).max()
                assert e <= 1e-5 * np.abs(ref).max(), (h, chunk, e)
                if d == 1 and chunk == n // 64:
                    assert torch.equal(F[h, 0], Sin[h, chunk]) and torch.equal(U[h, 0], Sin[h, chunk])
