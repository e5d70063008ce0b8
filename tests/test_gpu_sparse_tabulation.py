"""The tabulation with the incidence matrix as a sparse operand (q = 17) on tables that are filled where its kernels differ:
tokens are routed to the last point of every image (added outside the matrix product), to the last points of the table and to
types of the extra class (leading coordinate 0), of one head and of several, both directions, one stage (d = 3) and two."""
import numpy as np
import pytest
import torch

from oracle import smat_oracle as so
from paper_2609_36062_b200 import binding, synth
from tests.helpers import device_inputs, rel_err, to_numpy64

pytestmark = pytest.mark.gpu

Q = 17
TAIL_SCALE = 64.0      # V of the tokens on an image's last point: what is left out there stands out among 289 points


def _routed_workload(d, T, heads, tensors):
    w = synth.Workload("sparse", d, 1, heads, T, 128, 128, 128, "bf16", "normalised", 500 + d)
    host, dev = device_inputs(w, tensors)
    geo = so.geometry(T, 128, d, Q)
    rng = np.random.default_rng(d)
    tails = np.arange(Q * Q - 1, geo.P, Q * Q)
    extra = np.array([h for h in range(geo.B) if so.type_pair(h, geo)[0][0] == 0])
    cells, types = rng.integers(geo.P, size=(heads, geo.n)), rng.integers(geo.B, size=(heads, geo.m))
    fixed = np.concatenate([tails, np.arange(geo.P - 60, geo.P)])
    for h in range(heads):
        cells[h, rng.permutation(geo.n)[:fixed.size]] = fixed
        at = rng.permutation(geo.m)[:geo.m // 2]                        # every extra-class type, then repeats
        types[h, at] = extra[np.arange(at.size) % extra.size]
        on = np.isin(cells[h], tails)
        dev["v"][0, h, :geo.n][torch.as_tensor(on)] *= TAIL_SCALE        # (a power of two: exact)
    arrays = {"prof": torch.from_numpy(cells.astype(np.int32)).cuda(), "type": torch.from_numpy(types.astype(np.int32)).cuda()}
    plan = binding.SmatPlan(1, heads, T, 128, 128, d, 128, "bf16", q_override=Q)
    return w, host, dev, geo, tails, extra, arrays, plan


@pytest.mark.parametrize("d,T,heads", [(3, 512, 1), (3, 1280, 3), (4, 1024, 1), (4, 2048, 2)])
def test_sums_of_both_kinds_of_tiles_and_through_the_last_points(d, T, heads):
    _, _, dev, geo, tails, extra, arrays, plan = _routed_workload(d, T, heads, ("q", "k", "v"))
    plan.forward(dev["q"], dev["k"], dev["v"], **arrays)
    plan.check_status()
    F, U, _ = plan.debug_tables()
    points = np.array([so.prof(v, geo) for v in range(geo.P)])
    pairs = [so.type_pair(h, geo) for h in range(geo.B)]
    through = [h for h, (a, b) in enumerate(pairs) if ((points[tails] @ np.asarray(a)) % Q == b).any()]
    edges = [0, 127, 128, 255, 256, Q * Q - 1, Q * Q, Q * Q + Q - 1, geo.B - 1]
    types = sorted(set(through[::max(1, len(through) // 60)] + extra[::max(1, extra.size // 40)].tolist() + edges))
    for head in {0, heads - 1}:
        F64 = F[head].double()
        assert bool((F64[tails].abs().amax(dim=(1, 2)) > 0).all()) and bool((F64[geo.P - 60:].abs().amax(dim=(1, 2)) > 0).all())
        for h in types:
            a, b = pairs[h]
            on = torch.as_tensor((points @ np.asarray(a)) % Q == b, device=F.device)
            ref, size = F64[on].sum(0), F64[on].abs().sum(0)
            # one bf16 rounding of an fp32 sum (d = 4: and of its q intermediate sums)
            bound = 2.0 ** -8 * ref.abs() + (2.0 ** -20 if d == 3 else 2.0 ** -8) * size + 1e-30
            assert bool(((U[head, h].double() - ref).abs() <= bound).all()), (head, h)


@pytest.mark.parametrize("d,T,heads", [(3, 512, 1), (3, 1280, 2), (4, 1024, 1), (4, 2048, 2)])
def test_gradients_of_the_keys_on_the_last_points(d, T, heads):
    w, host, dev, geo, tails, extra, arrays, plan = _routed_workload(d, T, heads, ("q", "k", "v", "do"))
    _, dK, dV = plan.backward(dev["q"], dev["k"], dev["v"], dev["do"], **arrays)
    plan.check_status()
    for h in range(heads):
        cells, types = (arrays[x][h].cpu().numpy() for x in ("prof", "type"))
        assert np.isin(extra[:types.size // 2], types).all()             # queries on the extra class
        cols = sorted(set(np.nonzero(np.isin(cells, tails))[0][:40].tolist() + np.nonzero(cells >= geo.P - 20)[0][:20].tolist()))
        Q64, K64, G64 = (synth.as_float64(w, host[x][h]) for x in ("q", "k", "do"))
        for got, ref in zip((dK, dV), so.routed_dkdv_cols(Q64, K64, to_numpy64(dev["v"][0, h]), G64, geo, cells, types, cols)):
            for i, c in enumerate(cols):
                # adjoint state, its image sums, the transposed state, the row, the gradient: five bf16 roundings of 2^-9 on
                # sums of many terms, twice that for what cancels
                assert rel_err(to_numpy64(got[0, h, c]), ref[i]) <= 2e-2, (h, c)
