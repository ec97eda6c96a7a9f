"""Batches: the persistent form over the grids that it accepts, and the costs
that the replicas are assigned to chains by."""
import numpy as np
import pytest

from paper_1308_4005_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("box,levels", [((136.0, 180.0, 8.0), 3), ((192.0, 128.0, 16.0), 4)],
                         ids=["136x180", "192x128"])
def test_largest_planes(gpu_lib, box, levels):
    """x-y planes that leave a block of the transforms less than 30 KB of
    shared memory: one persistent launch, equal to the kernel chains bit for
    bit (the same bodies)."""
    import torch

    N = [700, 500]
    boxes = [box, (12.0, 12.0, 12.0)]
    at = [I.uniform_atoms(80 + r, n, b) for r, (n, b) in enumerate(zip(N, boxes))]
    pos = torch.tensor(np.concatenate([np.c_[x, c] for x, c in at]), dtype=torch.float32,
                       device="cuda")
    bt = gpu_lib.Batch(boxes, N, 2.0, 1.0, levels, precision="fp32")
    res = []
    for mode in (True, False):
        gpu_lib.mls6_batch_set_mode(bt.handle, mode)
        r = bt.evaluate(pos)
        torch.cuda.synchronize()
        assert gpu_lib.mls6_batch_mode(bt.handle) == int(mode)
        res.append([r[k].cpu().numpy() for k in ("E", "W", "F")])
    for a, b in zip(*res):
        assert np.array_equal(a, b)


def test_mode_leaves_a_batch_that_cannot_run_it(gpu_lib):
    """A batch with a replica without atoms, or in mixed precision, runs its
    chains whatever the mode: its pair sums stay as they were."""
    for prec, N in (("mixed", [9000, 9000]), ("fp32", [9000, 0])):
        bt = gpu_lib.Batch([(24.0, 24.0, 24.0)] * 2, N, 2.5, 1.0, 3, precision=prec)
        before = bt.info()["pair_split"]
        assert before[0] == 2048  # the tile form
        gpu_lib.mls6_batch_set_mode(bt.handle, True)
        assert gpu_lib.mls6_batch_mode(bt.handle) == 0
        assert bt.info()["pair_split"] == before


def test_cost_of_replicas_by_transforms(gpu_lib):
    """A replica that evaluates by transforms has neither the taps nor the
    coarsest product of the direct kernels: 20,000 atoms on a 44 x 44 x 44 grid
    of two levels (10,648 coarsest nodes) take about 0.1 ms, on a 46 x 46 x 46
    grid (a prime factor 23: direct) the coarsest product alone 40 ms."""
    bt = gpu_lib.Batch([(44.0, 44.0, 44.0), (46.0, 46.0, 46.0)], [20000, 20000], 2.5, 1.0, 2,
                       precision="fp32")
    forms = [gpu_lib.mls6_grid_form(gpu_lib.mls6_batch_replica(bt.handle, r))[0] for r in (0, 1)]
    cost = bt.info()["cost"]
    assert forms == [True, False]
    assert 2e-5 < cost[0] < 5e-4 and cost[1] > 1e-2
