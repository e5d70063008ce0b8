"""Passes away from the default stream: launches of two plans interleaved on two streams, and passes inside a captured graph.
Every kernel starts early under programmatic dependent launch, so a missing wait, or a conflict over tensor memory or shared
state, would show as a difference from the same calls made one after the other."""
import pytest
import torch

from paper_2609_36062_b200 import binding
from tests.helpers import stages

pytestmark = pytest.mark.gpu

KEEP = binding.FLAG_KEEP_FORWARD_TABLES
# name, d, batch, heads, T, chunk, width, dtype, variant, flags
PASSES = [
    ("train_d3", 3, 1, 8, 4096, 64, 128, "bf16", "train", KEEP),
    ("prefill_d4", 4, 1, 4, 4096, 128, 128, "bf16", "prefill", 0),
    ("prefill_d3_q37", 3, 1, 1, 65536, 128, 128, "bf16", "prefill", 0),
    ("prefill_short", 3, 4, 32, 1024, 128, 128, "bf16", "prefill", 0),
    ("partial_tiles", 3, 1, 8, 3008, 64, 128, "bf16", "prefill", 0),
    ("gated", 3, 1, 8, 4096, 64, 128, "bf16", "gated", KEEP | binding.FLAG_GATED),
    # the same through tables, which batches of so few heads form
    ("train_d3_tables", 3, 1, 4, 4096, 64, 128, "bf16", "train", KEEP),
    ("prefill_d4_tables", 4, 1, 2, 4096, 128, 128, "bf16", "prefill", 0),
    ("partial_tiles_tables", 3, 1, 1, 1984, 64, 128, "bf16", "prefill", 0),
    ("gated_tables", 3, 1, 4, 4096, 64, 128, "bf16", "gated", KEEP | binding.FLAG_GATED),
    ("f32", 2, 1, 4, 1024, 64, 64, "f32", "train", 0),
    ("decode", 3, 4, 16, 2048, 64, 128, "bf16", "decode", 0),
    ("decode_gated", 2, 4, 16, 1024, 64, 64, "f32", "decode", binding.FLAG_GATED),
]
BY_NAME = {p[0]: p for p in PASSES}
STEPS = 6


class Pass:
    """One plan with its inputs and workspace; call() runs a pass (a decoding pass: a few tokens) into fixed outputs."""

    def __init__(self, name, seed):
        _, d, b, h, T, c, dim, dtype, self.kind, flags = BY_NAME[name]
        g = torch.Generator(device="cuda").manual_seed(seed)
        dt = torch.bfloat16 if dtype == "bf16" else torch.float32
        rows = lambda n: (torch.randn(b, h, n, dim, generator=g, device="cuda") / dim ** 0.25).to(dt)
        self.plan = binding.SmatPlan(b, h, T, dim, dim, d, c, dtype, flags=flags)
        self.gated = bool(flags & binding.FLAG_GATED)
        self.q, self.k, self.v, self.do = rows(T), rows(T), rows(T), rows(T)
        self.la = torch.log(torch.rand(b * h, T, generator=g, device="cuda") * 0.01 + 0.99)
        if self.kind == "decode":
            self.begun = self.plan.decode_cache()
            args = (self.k, self.v) + ((self.la,) if self.gated else ())
            (self.plan.decode_begin_gated if self.gated else self.plan.decode_begin)(*args, self.begun)
            self.cache, self.first = self.begun.clone(), self.plan.geometry().n
            self.rows = [tuple(x[:, :, t].contiguous() for x in (self.q, self.k, self.v)) + (self.la[:, t].contiguous(),)
                         for t in range(STEPS)]
            self.out = [torch.zeros_like(self.rows[0][2]) for _ in range(STEPS)] + [self.cache]
        else:
            self.ws = self.plan.workspace(for_backward=True)
            self.out = [torch.zeros_like(x) for x in (self.v, self.q, self.k, self.v, self.la)]
        self.check = self.ws if self.kind != "decode" else self.plan._ws

    def call(self, stream=None):
        p, o = self.plan, self.out
        if self.kind == "decode":
            self.cache.copy_(self.begun)
            for i, (q, k, v, la) in enumerate(self.rows):
                if self.gated:
                    p.decode_step_gated(q, k, v, la, self.first + i, self.cache, o=o[i], stream=stream)
                else:
                    p.decode_step(q, k, v, self.first + i, self.cache, o=o[i], stream=stream)
        elif self.gated:
            p.forward_gated(self.q, self.k, self.v, self.la, O=o[0], workspace=self.ws, stream=stream)
            p.backward_gated(self.q, self.k, self.v, self.la, self.do, dQ=o[1], dK=o[2], dV=o[3], dlog_a=o[4],
                             workspace=self.ws, stream=stream)
        else:
            p.forward(self.q, self.k, self.v, O=o[0], workspace=self.ws, stream=stream)
            if self.kind == "train":
                p.backward(self.q, self.k, self.v, self.do, dQ=o[1], dK=o[2], dV=o[3], workspace=self.ws, stream=stream)

    def expect(self):
        """The outputs of the call made alone."""
        self.call()
        torch.cuda.synchronize()
        self.plan.check_status(self.check)
        want = [x.clone() for x in self.out]
        for x in self.out:
            x.zero_()
        torch.cuda.synchronize()
        return want

    def verify(self, want):
        self.plan.check_status(self.check)
        for a, b in zip(self.out, want):
            assert torch.equal(a, b)


@pytest.mark.parametrize("name", [n for n in BY_NAME if n.startswith(("train_d3", "prefill_d4", "partial_tiles", "gated"))])
def test_the_passes_form_tables_or_not_as_their_names_say(name):
    p = Pass(name, 5)
    _, ran = stages(p.plan, p.call)
    tables = {"pool", "pool_tc", "bwd_pool_type_tc"} & set(ran)
    lines = {"read_lines", "bwd_dkdv_lines"} & set(ran)
    assert (bool(tables), bool(lines)) == ((True, False) if name.endswith("_tables") else (False, True))


@pytest.mark.parametrize("one,other", [("train_d3", "prefill_d4"), ("prefill_d4", "decode"), ("prefill_short", "prefill_d3_q37"),
                                       ("gated", "partial_tiles"), ("f32", "decode_gated"), ("train_d3", "train_d3"),
                                       ("train_d3_tables", "prefill_d4_tables"), ("gated_tables", "partial_tiles_tables"),
                                       ("train_d3_tables", "train_d3_tables"), ("train_d3_tables", "train_d3")])
def test_two_plans_on_two_streams(one, other):
    passes = [Pass(one, 1), Pass(other, 2)]
    want = [p.expect() for p in passes]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(5):
        for p, s in zip(passes, streams):
            with torch.cuda.stream(s):
                p.call()
    torch.cuda.synchronize()
    for p, w in zip(passes, want):
        p.verify(w)


@pytest.mark.parametrize("name", list(BY_NAME))
def test_a_captured_pass_replays_on_new_inputs(name):
    p = Pass(name, 3)
    p.expect()                                    # (and the first launch of every kernel, outside the capture)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        p.call()
    fresh = Pass(name, 4)
    want = fresh.expect()
    for mine, new in zip([p.q, p.k, p.v, p.do, p.la] + ([p.begun] if p.kind == "decode" else []),
                         [fresh.q, fresh.k, fresh.v, fresh.do, fresh.la] + ([fresh.begun] if p.kind == "decode" else [])):
        mine.copy_(new)
    if p.kind == "decode":
        for mine, new in zip(p.rows, fresh.rows):
            for a, b in zip(mine, new):
                a.copy_(b)
    for x in p.out:
        x.zero_()
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    p.verify(want)
