"""The tile form of the FP32 pair sum (pair_split 2048): 8 atoms per warp
against a shared candidate list, packed FP32 arithmetic.

Tolerances: those of the FP32 path (tests/test_gpu_parity.py): its rounding
bound is per pair term and per summation, and the tile form rounds each term
as the per-atom kernel does and adds fewer of them in a row.  Two FP32 forms
differ from each other by at most twice that.
"""
import zlib

import numpy as np
import pytest

from paper_1308_4005_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = dict(E=2e-6, F=1e-4, W=2e-5)
TILE = 2048

CASES = [
    # name, N, box, a, h, levels, least separation
    ("ragged_last_warp", 1001, (13.0, 11.0, 10.0), 2.5, 0.9, 2, 0.8),
    ("slab_empty_rows", 3000, (26.0, 12.0, 30.0), 3.0, 1.0, 3, 0.8),
    ("images_both_sides", 700, (30.0, 6.0, 5.5), 2.0, 0.6, 2, 0.8),
    ("box_below_2a", 600, (9.0, 5.0, 20.0), 3.0, 0.9, 2, 0.8),
    ("five_cells_in_x", 500, (7.4, 9.0, 9.0), 2.8, 0.9, 2, 0.8),
    ("lists_filled_repeatedly", 5000, (12.0, 12.0, 12.0), 3.0, 1.0, 2, 0.4),
    ("sparse_rows", 400, (40.0, 20.0, 20.0), 3.0, 1.5, 2, 0.8),
]


def _run(plan, pos, virial):
    import torch

    r = plan.evaluate(pos, virial=virial)
    torch.cuda.synchronize()
    return r["out"].cpu().numpy(), r["F"].cpu().double().numpy(), r


@pytest.mark.parametrize("name,N,box,a,h,l,dmin", CASES, ids=[c[0] for c in CASES])
def test_tile_form_vs_oracle(gpu_lib, orc, name, N, box, a, h, l, dmin):
    import torch

    region = ((0, box[0]), (0, box[1]), (0.35 * box[2], 0.65 * box[2])) if "slab" in name else None
    x, c = I.uniform_atoms(zlib.crc32(name.encode()) % 10000, N, box, dmin=dmin, region=region)
    x, c = (v.astype(np.float32).astype(np.float64) for v in (x, c))
    o = orc.evaluate(box, a, orc.grid_dims(box, h, l), l, x, c)
    rms = np.sqrt(np.mean(np.sum(o["F"] ** 2, axis=1)))
    plan = gpu_lib.Plan(box, N, a, h, l, precision="fp32")
    gpu_lib.mls6_set_tuning(plan.handle, TILE, 0)
    assert gpu_lib.mls6_get_tuning(plan.handle)[0] == TILE
    pos = torch.tensor(np.c_[x, c], dtype=torch.float32, device="cuda")
    for virial in (True, False):
        out, F, r = _run(plan, pos, virial)
        assert abs(out[0] - o["E"]) <= TOL["E"] * abs(o["E"])
        assert np.abs(F - o["F"]).max() <= TOL["F"] * rms
        if virial:
            assert np.abs(out[1:] - o["W"]).max() <= TOL["W"] * np.abs(o["W"]).max()
        again = _run(plan, pos, virial)[2]
        assert torch.equal(r["F"], again["F"]) and torch.equal(r["out"], again["out"])


@pytest.mark.parametrize("N", [1, 2, 7, 8, 9, 31, 33])
def test_tile_form_few_atoms(gpu_lib, N):
    """Fewer atoms than a warp or a block takes, two of them at one place
    (excluded, as in every form), against the per-atom kernel."""
    import torch

    box = (12.0, 11.0, 10.0)
    x, c = I.uniform_atoms(50 + N, N, box)
    if N > 2:
        x[1] = x[0]
    plan = gpu_lib.Plan(box, N, 2.5, 1.0, 2, precision="fp32")
    pos = torch.tensor(np.c_[x, c], dtype=torch.float32, device="cuda")
    got = {}
    for split in (1, TILE):
        gpu_lib.mls6_set_tuning(plan.handle, split, 0)
        got[split] = _run(plan, pos, True)[:2]
    scale = max(np.abs(got[1][1]).max(), 1e-3)  # a lone atom: the grid's own force of rounding size
    assert np.abs(got[1][1] - got[TILE][1]).max() <= 2 * TOL["F"] * scale
    assert np.abs(got[1][0] - got[TILE][0]).max() <= 2 * TOL["W"] * max(
        np.abs(got[1][0]).max(), 1e-3)


def test_tile_form_lorentz_berthelot(gpu_lib):
    """Exact pair coefficients in the tile form against one lane per atom."""
    import torch

    N, box = 3001, (24.0, 14.0, 13.0)
    x, _ = I.uniform_atoms(77, N, box)
    rng = np.random.default_rng(78)
    arrs = [torch.tensor(v, dtype=torch.float32, device="cuda")
            for v in (x, rng.uniform(0.85, 1.15, N), rng.uniform(0.5, 1.5, N))]
    plan = gpu_lib.Plan(box, N, 2.5, 1.0, 2, precision="fp32")
    got = {}
    for split in (1, TILE):
        gpu_lib.mls6_set_tuning(plan.handle, split, 0)
        F = torch.empty((N, 3), dtype=torch.float32, device="cuda")
        E = torch.zeros(1, dtype=torch.float64, device="cuda")
        rc = gpu_lib.mls6_eval_lb(plan.handle, *[v.data_ptr() for v in arrs], F.data_ptr(),
                                  E.data_ptr())
        assert rc == 0
        torch.cuda.synchronize()
        got[split] = E.item(), F.cpu().double().numpy()
    rms = np.sqrt(np.mean(np.sum(got[1][1] ** 2, axis=1)))
    assert abs(got[1][0] - got[TILE][0]) <= 2 * TOL["E"] * abs(got[1][0])
    assert np.abs(got[1][1] - got[TILE][1]).max() <= 2 * TOL["F"] * rms


def test_tile_form_default_and_refusals(gpu_lib):
    """Default from 8,192 atoms and half an atom per cell on; refused in FP64
    and where a row of cells is shorter than the neighbour range."""
    L = I.cube_side(8192, 0.85)
    tuning = lambda *a, **k: gpu_lib.mls6_get_tuning(gpu_lib.Plan(*a, **k).handle)[0]  # noqa: E731
    assert tuning((L, L, L), 8192, 3.0, 1.5, 0, precision="fp32") == TILE
    assert tuning((L, L, L), 8192, 3.0, 1.5, 0, precision="mixed") == TILE
    assert tuning((L, L, L), 8191, 3.0, 1.5, 0, precision="fp32") <= 8
    assert tuning((3 * L, L, L), 8192, 3.0, 1.5, 0, precision="fp32") == TILE
    assert tuning((6 * L, L, L), 8192, 3.0, 1.5, 0, precision="fp32") <= 8
    assert tuning((L, L, L), 8192, 3.0, 1.5, 0, precision="fp32", continuity=3) <= 8
    for kw in (dict(box=(L, L, L), precision="fp64"), dict(box=(5.0, L, L), precision="fp32")):
        plan = gpu_lib.Plan(kw["box"], 8192, 3.0, 1.5, 0, precision=kw["precision"])
        with pytest.raises(gpu_lib.MLS6Error):
            gpu_lib.mls6_set_tuning(plan.handle, TILE, 0)


def test_tile_form_in_a_batch(gpu_lib):
    """Replicas take their plan's default form in the kernel chains (bit for
    bit the single plan's results); the persistent kernel takes the lanes per
    atom, and stays available."""
    import torch

    Ns = [8300, 2500]
    boxes = [(I.cube_side(n, 0.85),) * 3 for n in Ns]
    parts = [I.uniform_atoms(90 + n, n, b) for n, b in zip(Ns, boxes)]
    pos = torch.tensor(np.concatenate([np.c_[x, c] for x, c in parts]), dtype=torch.float32,
                       device="cuda")
    bt = gpu_lib.Batch(boxes, Ns, 2.5, 1.0, precision="fp32")
    assert bt.info()["pair_split"][0] == TILE and bt.info()["pair_split"][1] <= 8
    for persistent in (False, True):
        gpu_lib.mls6_batch_set_mode(bt.handle, persistent)
        r = bt.evaluate(pos)
        torch.cuda.synchronize()
        info = bt.info()
        assert gpu_lib.mls6_batch_mode(bt.handle) == int(persistent)
        assert (info["pair_split"][0] == TILE) != persistent
        for k in range(2):
            p = gpu_lib.Plan(boxes[k], Ns[k], 2.5, 1.0, 0, precision="fp32")
            gpu_lib.mls6_set_tuning(p.handle, info["pair_split"][k], info["stencil_groups"][k])
            sl = slice(bt.offsets[k], bt.offsets[k + 1])
            one = p.evaluate(pos[sl].contiguous())
            torch.cuda.synchronize()
            assert torch.equal(one["F"], r["F"][sl])
            assert one["out"][0] == r["E"][k] and torch.equal(one["out"][1:], r["W"][k])
