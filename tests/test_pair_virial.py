"""The FP64 pair virial of the queue form (the default) is summed over d (x) d,
which keeps every pair's precision however large its atoms' coordinates are."""
import numpy as np
import pytest

from paper_1308_4005_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [128, 256, 512])
@pytest.mark.parametrize("box", [(8.0, 7.5, 400.0), (400.0, 8.0, 7.5), (8.0, 400.0, 7.5)])
def test_fp64_pair_virial_precision(gpu_lib, box, split):
    """Ten pairs 0.2 apart (more than a/16) far from the origin, whose terms are
    10^4 times the others'.  Against the warp form (32 lanes per atom), which
    sums d (x) d of every pair from both atoms; the grid part is the same, bit
    for bit.  Each form rounds a term a few times (u = 1.1e-16) and adds some
    twenty of them: 10 u of the virial between the two.  Products of forces and
    coordinates lose |x| / r = 2000 of it."""
    import torch

    N = 120
    x, c = I.uniform_atoms(71, N, box, dmin=2.0)
    long = int(np.argmax(box))
    rng = np.random.default_rng(73)
    for k in range(10):
        x[2 * k, long] = 380.0 + 1.5 * k
        d = rng.normal(size=3)
        x[2 * k + 1] = x[2 * k] + 0.2 * d / np.linalg.norm(d)
    pos = torch.tensor(np.c_[x, c], device="cuda")
    plan = gpu_lib.Plan(box, N, 3.0, 1.0, 2, precision="fp64")
    W = []
    for s in (32, split):
        gpu_lib.mls6_set_tuning(plan.handle, s, 0)
        W.append(plan.evaluate(pos)["out"].cpu().numpy()[1:])
    assert np.abs(W[0] - W[1]).max() <= 1.1e-15 * np.abs(W[0]).max()


def test_fp64_pair_virial_self_images(gpu_lib, orc):
    """Axes thinner than the cutoff, where an atom meets its own images: each
    pair of opposite images counts once."""
    import torch

    box, N, a = (12.0, 4.0, 4.5), 40, 4.2
    x, c = I.uniform_atoms(72, N, box)
    n = orc.grid_dims(box, 1.0, 2)
    o = orc.evaluate(box, a, n, 2, x, c)
    plan = gpu_lib.Plan(box, N, a, 1.0, 2, precision="fp64")
    for s in (128, 256, 512):
        gpu_lib.mls6_set_tuning(plan.handle, s, 0)
        w = plan.evaluate(torch.tensor(np.c_[x, c], device="cuda"))["out"].cpu().numpy()[1:]
        assert np.abs(w - o["W"]).max() <= 1e-11 * np.abs(o["W"]).max()
