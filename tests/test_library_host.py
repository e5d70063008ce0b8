"""CPU-side checks of the C boundary: the library loads, exports every declared symbol, validates its
arguments, and its integer routing matches the oracle bit for bit.  No kernel is launched here."""
import ctypes
import os
import re

import numpy as np
import pytest

from oracle import smat_oracle as so
from paper_2609_36062_b200 import binding, synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared_symbols():
    names = set()
    for fn in os.listdir(os.path.join(ROOT, "include")):
        if fn.endswith(".h"):
            text = open(os.path.join(ROOT, "include", fn)).read()
            text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
            names |= set(re.findall(r"\b(smat_[a-z0-9_]+)\s*\(", text))
    return names


def test_library_exports_every_declared_symbol():
    lib = binding.load_library()
    declared = _declared_symbols()
    assert declared, "no declarations found"
    for name in declared:
        assert hasattr(lib, name), name
    assert set(binding.EXPORTS) <= declared


@pytest.mark.parametrize("name", list(synth.WORKLOADS))
def test_plan_geometry_matches_the_oracle(name):
    w = synth.WORKLOADS[name]
    plan = binding.SmatPlan(w.batch, w.heads, w.T, w.d_k, w.d_v, w.d, w.chunk, w.dtype)
    g = plan.geometry()
    o = so.geometry(w.T, w.chunk, w.d)
    assert (g.n, g.m, g.q, g.P, g.A, g.B, g.nnzC) == (o.n, o.m, o.q, o.P, o.A, o.B, o.nnzC)
    assert g.vc_conditions_met == o.conditions_met
    assert plan.workspace_bytes(True) >= plan.workspace_bytes(False) > 0


@pytest.mark.parametrize("T,c,d,q", [(512, 64, 2, 0), (512, 64, 1, 0), (4096, 64, 3, 0), (2048, 32, 4, 0), (256, 16, 3, 5),
                                     (256, 16, 4, 3), (512, 16, 5, 3), (16384, 128, 4, 0), (8192, 64, 3, 0)])
def test_routing_indices_are_bit_exact(T, c, d, q):
    plan = binding.SmatPlan(1, 1, T, 64, 64, d, c, "f32", q_override=q)
    geo = so.geometry(T, c, d, q or None)
    prof, typ, ab = plan.routing_indices()
    o_prof, o_typ, o_ab = so.routing_tables(geo)
    assert np.array_equal(prof.numpy(), o_prof.reshape(prof.shape))
    assert np.array_equal(typ.numpy(), o_typ)
    assert np.array_equal(ab.numpy(), o_ab)


def test_argument_errors_are_reported_before_any_launch():
    lib = binding.load_library()
    h = ctypes.c_void_p()
    mk = lambda *a: lib.smat_plan_create(ctypes.byref(h), *a)
    assert lib.smat_plan_create(None, 1, 1, 512, 64, 64, 2, 64, 0, 0, 0) == 1          # null
    assert mk(1, 1, 512, 64, 64, 2, 64, 0, 7, 0) == 3                                   # dtype
    assert mk(1, 1, 512, 48, 64, 2, 64, 0, 0, 0) == 2                                   # d_k
    assert mk(1, 1, 500, 64, 64, 2, 64, 0, 0, 0) == 2                                   # T % chunk
    assert mk(1, 1, 512, 64, 64, 2, 48, 0, 0, 0) == 2                                   # chunk
    assert mk(1, 1, 512, 64, 64, 0, 64, 0, 0, 0) == 4                                   # d
    assert mk(1, 1, 512, 64, 64, 9, 64, 0, 0, 0) == 4
    assert mk(1, 1, 512, 64, 64, 2, 64, 15, 0, 0) == 4                                  # q not prime
    assert mk(1, 1, 64, 64, 64, 2, 64, 0, 0, 0) == 4                                    # T < 2c with d >= 2
    assert mk(1, 1, 64, 64, 64, 1, 64, 0, 0, 0) == 0                                    # ... but fine for d = 1
    plan = h.value
    # forward with null / short / misaligned buffers never launches
    assert lib.smat_forward(plan, None, 256, 256, 256, 256, 1 << 40, None) == 1
    assert lib.smat_forward(plan, 256, 256, 256, 256, None, 1 << 40, None) == 1
    assert lib.smat_forward(plan, 256, 256, 256, 256, 256, 16, None) == 5
    assert lib.smat_forward(plan, 256, 256, 256, 256, 264, 1 << 40, None) == 6
    assert lib.smat_forward(plan, 260, 256, 256, 256, 256, 1 << 40, None) == 6
    assert lib.smat_backward(plan, 256, 256, 256, None, 256, 256, 256, 256, 1 << 40, None) == 1
    assert lib.smat_workspace_bytes(None, 0) == 0
    lib.smat_plan_destroy(h)
    assert binding.status_string(5) == "workspace too small"


def test_binding_rejects_wrong_tensors():
    import torch
    plan = binding.SmatPlan(1, 1, 512, 64, 64, 2, 64, "f32")
    x = torch.zeros(1, 1, 512, 64)
    with pytest.raises(ValueError):
        plan.forward(x, x, x)          # CPU tensors: no fallback


def test_non_default_geometry_flags():
    g = binding.SmatPlan(1, 1, 256, 64, 64, 4, 16, "f32").geometry()   # default q too large for this T
    assert not g.vc_conditions_met
    g = binding.SmatPlan(1, 1, 256, 64, 64, 4, 16, "f32", q_override=2).geometry()
    assert g.vc_conditions_met and (g.P, g.B) == (8, 14)


def test_workspace_regions_follow_the_stored_element_types():
    """The bf16 tables and per-tile states of a tensor-core plan take half the bytes of their fp32 forms, and such a
    plan reserves no score-tile buffers; the plan is a function of the shape alone (no device is needed to size it)."""
    w = synth.WORKLOADS["t64k_d4"]
    plan = binding.SmatPlan(w.batch, w.heads, w.T, w.d_k, w.d_v, w.d, w.chunk, w.dtype)
    assert plan.uses_tensor_cores() and plan.profile_table_element_bytes() == 2 and plan.type_table_element_bytes() == 2
    g = plan.geometry()
    state = w.d_k * w.d_v
    tables = w.bh * (g.P + g.B) * state * 2                      # F and U in bf16
    exchange = w.bh * (g.q ** 3 + g.q ** 2) * state * 2          # intermediate of the two d = 4 tabulation stages
    causal = w.bh * (w.T // 128) * state * 2
    rows = w.bh * w.T * 128 * 4                                  # long-range rows
    lists = w.bh * (w.T + g.P + g.B + 2) * 4                     # token lists of user-supplied routing (int32)
    need = tables + exchange + causal + rows + lists
    got = plan.workspace_bytes(False)
    assert need <= got <= need + 64 * 1024, (got, need)
    assert got < 9.0e9                                           # 15 GB with every region at 4 bytes per entry
    simt = binding.SmatPlan(w.batch, w.heads, w.T, w.d_k, w.d_v, w.d, w.chunk, w.dtype, flags=binding.FLAG_SIMT_ONLY)
    assert simt.workspace_bytes(False) > got
    # backward: adjoint tables in bf16 too, per-tile adjoint states
    back = plan.workspace_bytes(True)
    lr3 = w.bh * w.T * 128 * 2                                   # third buffer of bf16 long-range rows
    assert got + tables + causal + lr3 <= back <= got + tables + causal + lr3 + 64 * 1024


def test_launching_calls_report_a_missing_sm100_device():
    import torch
    if torch.cuda.is_available():
        pytest.skip("a device is present: the calls below would launch")
    lib = binding.load_library()
    h = ctypes.c_void_p()
    assert lib.smat_plan_create(ctypes.byref(h), 1, 1, 512, 64, 64, 2, 64, 0, 0, 0) == 0
    # all arguments are acceptable; what is missing is a compute capability 10.x device
    assert lib.smat_forward(h, 256, 256, 256, 256, 256, 1 << 40, None) == 7
    assert lib.smat_backward(h, 256, 256, 256, 256, 256, 256, 256, 256, 1 << 40, None) == 7
    assert lib.smat_forward_causal_static(256, 256, 256, 256, 1, 1, 128, None) == 7
    assert lib.smat_debug_timeout_probe(256, 1000, None) == 7
    assert "sm_100" in binding.status_string(7)
    lib.smat_plan_destroy(h)


@pytest.mark.parametrize("q", [2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31, 37, 41, 43, 47, 53])
def test_tabulation_kernel_shared_memory_map_is_disjoint(q):
    """Ring slots, per-slot extra rows, the output-row table, masks and the barrier words of the tensor-core tabulation
    kernels never overlap and no load box or staged tile leaves its slot, for every stage of every prime they take."""
    assert binding.load_library().smat_debug_tabulation_layout_ok(q) == 1


@pytest.mark.parametrize("q", [59, 61, 241])
def test_no_tabulation_kernel_claims_a_prime_that_does_not_fit(q):
    """Their masks leave no room for a ring of image slots: the sums are formed on the fp32 ALUs."""
    assert binding.load_library().smat_debug_tabulation_layout_ok(q) == 0


def test_gated_plans_size_their_inner_plan_and_decode_cache():
    """A gated plan on a tensor-core shape carries an ungated plan of its own for both passes: its workspace holds that
    plan's backward workspace as a region, its decode cache the bf16 type table, the running state and one word per
    head; other shapes, and SIMT_ONLY, have no inner plan and keep fp32 tables."""
    shape = (2, 4, 4096, 128, 128, 3, 64, "bf16")
    gated = binding.SmatPlan(*shape, flags=binding.FLAG_GATED)
    plain = binding.SmatPlan(*shape, flags=binding.FLAG_PER_TILE_STATES)
    alu = binding.SmatPlan(*shape, flags=binding.FLAG_GATED | binding.FLAG_SIMT_ONLY)
    assert not gated.uses_tensor_cores()                        # the gated plan itself keeps the fp32-ALU layout
    assert gated.gated_forward_uses_tensor_cores() and gated.gated_backward_uses_tensor_cores()
    assert not alu.gated_forward_uses_tensor_cores() and not alu.gated_backward_uses_tensor_cores()
    assert not plain.gated_forward_uses_tensor_cores()
    inner = plain.workspace_bytes(True)
    assert alu.workspace_bytes(False) + inner <= gated.workspace_bytes(False) <= alu.workspace_bytes(False) + inner + 4096
    assert gated.workspace_bytes(True) - gated.workspace_bytes(False) == alu.workspace_bytes(True) - alu.workspace_bytes(False)
    g = gated.geometry()
    bh, state = 8, 128 * 128
    lib = binding.load_library()
    assert lib.smat_decode_cache_bytes(gated.handle) == bh * g.B * state * 2 + bh * state * 4 + 256
    assert lib.smat_decode_cache_bytes(alu.handle) == bh * g.B * state * 4 + bh * state * 4 + 256
    assert lib.smat_decode_cache_bytes(plain.handle) == bh * g.B * state * 2 + bh * state * 4
    # the tabulation flags reach the inner plan: fp32 tables there (the literal Algorithm 2) mean an fp32-ALU gated backward
    odd = binding.SmatPlan(*shape, flags=binding.FLAG_GATED | binding.FLAG_ALG2_TABULATION)
    assert odd.gated_forward_uses_tensor_cores() and not odd.gated_backward_uses_tensor_cores()
    # a block boundary that is not a whole tile: no inner plan
    ragged = binding.SmatPlan(1, 2, 640, 128, 128, 3, 32, "bf16", flags=binding.FLAG_GATED)
    assert not ragged.gated_forward_uses_tensor_cores()


def test_tensors_without_storage_raise_an_error():
    """Under vmap the operands carry no storage: asking for their data pointer raises (and used to do so with the
    interpreter lock released, which ended the process)."""
    import types

    import torch
    from torch._subclasses import FakeTensorMode

    plan = binding.SmatPlan(1, 1, 256, 64, 64, 2, 32, "f32")
    cache_plan = binding.SmatPlan(1, 1, 256, 64, 64, 2, 32, "f32", flags=binding.FLAG_GATED)
    stream = types.SimpleNamespace(cuda_stream=0)
    with FakeTensorMode():
        x, row = torch.empty(3, 1, 1, 256, 64, device="cuda"), torch.empty(3, 1, 1, 64, device="cuda")
        ws, o = torch.empty(1024, dtype=torch.uint8, device="cuda"), torch.empty(1, 1, 256, 64, device="cuda")
        orow, gate = torch.empty(1, 1, 64, device="cuda"), torch.empty(1, device="cuda")
        calls = (lambda t, r: plan.forward(t, t, t, O=o, workspace=ws, stream=stream),
                 lambda t, r: plan.backward(t, t, t, t, dQ=o, dK=o, dV=o, workspace=ws, stream=stream)[0],
                 lambda t, r: plan.decode_step(r, r, r, 200, ws, o=orow, stream=stream),
                 lambda t, r: plan.decode_step(r, r, r, 200.0, ws, o=orow, stream=stream),      # any t that int() takes
                 lambda t, r: plan.decode_step(r, r, r, np.int32(200), ws, o=orow, stream=stream),
                 lambda t, r: cache_plan.decode_step_gated(r, r, r, gate, 200, ws, o=orow, stream=stream))
        for call in calls:
            with pytest.raises(RuntimeError, match="storage"):
                torch.func.vmap(call)(x, row)


def test_output_buffers_may_be_larger_but_not_smaller_or_strided():
    """Outputs other than forward's O: the first elements of a larger buffer are written; anything a call would write
    out of, or in another order than the tensor shows, is refused."""
    import types

    import torch
    from torch._subclasses import FakeTensorMode

    plan = binding.SmatPlan(1, 1, 256, 64, 64, 2, 32, "f32")
    stream = types.SimpleNamespace(cuda_stream=0)
    with FakeTensorMode():
        x, row = torch.empty(3, 1, 1, 256, 64, device="cuda"), torch.empty(3, 1, 1, 64, device="cuda")
        ws = torch.empty(1024, dtype=torch.uint8, device="cuda")
        big, small = torch.empty(2, 256, 64, device="cuda"), torch.empty(1, 1, 255, 64, device="cuda")
        flat, strided = torch.empty(256 * 64, device="cuda"), torch.empty(1, 1, 64, 256, device="cuda").transpose(2, 3)

        def backward(out):
            return torch.func.vmap(lambda t: plan.backward(t, t, t, t, dQ=out, dK=out, dV=out, workspace=ws, stream=stream)[0])(x)

        def decode(out):
            return torch.func.vmap(lambda r: plan.decode_step(r, r, r, 200, ws, o=out, stream=stream))(row)

        for ok in (big, flat):
            with pytest.raises(RuntimeError, match="storage"):      # past the checks
                backward(ok)
        with pytest.raises(RuntimeError, match="storage"):
            decode(big)
        for bad in (small, strided, big.to(torch.bfloat16)):
            with pytest.raises(ValueError):
                backward(bad)
        with pytest.raises(ValueError):
            decode(small[..., :63])


class _SmatGeo(ctypes.Structure):   # csrc/smat_geometry.h
    _fields_ = [(f, ctypes.c_int64) for f in ("T", "c", "n", "m")] + [(f, ctypes.c_int32) for f in ("d", "q", "D")] + \
               [(f, ctypes.c_int64) for f in ("P", "A", "B", "nnzC")] + [("dense_G", ctypes.c_int32)] + \
               [("qpow", ctypes.c_int64 * 8), ("dir_group_start", ctypes.c_int64 * 8)]


@pytest.mark.parametrize("q,bh,fits", [(32749, 1, True), (32771, 1, False), (1009, 1054, True), (1009, 1055, False)])
def test_rows_without_tables_keep_every_launch_inside_its_quotients(q, bh, fits):
    """d = 2, 17 or 18 tokens to a cell and to a type: one row block to a group in the single products, two in the launch that
    forms dK and dV.  The kernel divides an item's number by the items of a head with one multiplication, which is exact
    while items x (items of a head) stays below 2^32; beyond it an item would address another head."""
    n = -(-17 * q // 128) * 128
    plan = binding.SmatPlan(1, bh, 2 * n, 128, 128, 2, 128, "bf16", q_override=q)   # (sizes that a plan accepts)
    g = plan.geometry()
    geo = _SmatGeo(T=g.T, c=g.c, n=g.n, m=g.m, d=2, q=q, D=1, P=g.P, A=g.A, B=g.B, nnzC=g.nnzC)
    geo.qpow[:2] = (1, q)
    assert -(-g.n // g.P) in (17, 18)
    supported = binding.load_library()["_Z20smat_lines_supportedRK7SmatGeoi"]
    supported.restype, supported.argtypes = ctypes.c_bool, [ctypes.c_void_p, ctypes.c_int]
    assert supported(ctypes.byref(geo), bh) == fits
    per = 2 * q
    items = bh * per
    inverse = (2 ** 32 + per - 1) // per
    last_of_a_head = np.arange(per - 1, items, per, dtype=np.uint64)
    exact = bool(np.all(last_of_a_head * np.uint64(inverse) >> np.uint64(32) == last_of_a_head // np.uint64(per)))
    assert exact or not fits


class _LineArgs(ctypes.Structure):   # SmatLineArgs of csrc/smat_internal.h
    _fields_ = [(f, ctypes.c_void_p) for f in ("x1", "x2", "y", "z", "out1", "out2")] + \
               [(f, ctypes.c_int) for f in ("out_f32", "rows_are_types", "ones", "parts")] + \
               [("lam", ctypes.c_void_p), ("copy", ctypes.c_void_p), ("copy_head", ctypes.c_int64), ("copy_swap", ctypes.c_int),
                ("mark", ctypes.c_void_p), ("mark_value", ctypes.c_int), ("clear", ctypes.c_void_p)]


@pytest.mark.parametrize("args", [dict(parts=0), dict(parts=4), dict(parts=2, out2=256), dict(parts=3, lam=256),
                                  dict(parts=1, ones=1, out2=256), dict(parts=1, ones=1, lam=256)])
def test_rows_without_tables_refuse_what_their_kernels_would_ignore(args):
    """Several score parts and the ones column exist in the single ungated product only; the launcher says so before it
    reaches a device (cudaErrorInvalidValue is 1)."""
    import torch
    if torch.cuda.is_available():
        pytest.skip("a device is present: a launcher without the check would launch")
    g = binding.SmatPlan(1, 2, 2048, 128, 128, 3, 128, "bf16").geometry()
    geo = _SmatGeo(T=g.T, c=g.c, n=g.n, m=g.m, d=3, q=g.q, D=2, P=g.P, A=g.A, B=g.B, nnzC=g.nnzC)
    geo.qpow[:3], geo.dir_group_start[:2] = (1, g.q, g.q ** 2), (0, g.q)
    launch = binding.load_library()["_Z25smat_launch_line_productsRK12SmatLineArgsRK7SmatGeoiP11CUstream_st"]
    launch.restype, launch.argtypes = ctypes.c_int, [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]
    assert launch(ctypes.byref(_LineArgs(rows_are_types=1, **args)), ctypes.byref(geo), 2, None) == 1


@pytest.mark.parametrize("d,heads,T,without", [(2, 16, 34880, True), (3, 8, 58240, True), (4, 8, 16448, True), (4, 8, 19520, False),
                                               (4, 8, 22592, False), (5, 8, 3136, True), (5, 8, 14400, True)])
def test_which_partial_tile_plans_form_no_tables(d, heads, T, without):
    """Both sides of the rule's lines for fp32 tables: d = 4 gives up sooner than d = 3 (whose tables take longer) and than
    d = 5 (whose tables are summed by the literal Algorithm 2)."""
    plan = binding.SmatPlan(1, heads, T, 128, 128, d, 64, "bf16")
    assert plan.type_table_element_bytes() == 4
    g = plan.geometry()
    geo = _SmatGeo(T=g.T, c=g.c, n=g.n, m=g.m, d=d, q=g.q, D=d - 1, P=g.P, A=g.A, B=g.B, nnzC=g.nnzC)
    geo.qpow[:d] = [g.q ** k for k in range(d)]
    geo.dir_group_start[:d - 1] = [sum(g.q ** (d - 2 - i) for i in range(k)) for k in range(d - 1)]
    pay = binding.load_library()["_Z14smat_lines_payRK7SmatGeoiib"]
    pay.restype, pay.argtypes = ctypes.c_bool, [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_bool]
    assert pay(ctypes.byref(geo), heads, 4, False) == without
