"""The FP64 queue form of the pair sum (FP32 cutoff test, FP64 evaluation by a
Newton reciprocal) where its FP32 part could go wrong: large coordinates, very
close pairs, images.  Against one lane group per atom, which works in FP64
throughout: every pair term carries a few FP64 roundings (u = 1.1e-16) and a
force sums ~100 of them, so 1e-12 of the atom's largest term bounds both.
"""
import numpy as np
import pytest

from paper_1308_4005_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [128, 256, 512])
@pytest.mark.parametrize("box,a", [((2000.0, 9.0, 8.0), 2.5), ((30.0, 28.0, 26.0), 3.0),
                                   ((8.0, 7.0, 400.0), 3.0)])
def test_queue_form_large_boxes_and_close_pairs(gpu_lib, split, box, a):
    import torch

    N = 900
    x, c = I.uniform_atoms(31, N, box)
    rng = np.random.default_rng(32)
    for k in range(20):  # pairs at distances 1e-6 .. 1e-1, some of them across a face
        d = rng.normal(size=3)
        if k < 6:
            x[2 * k, k % 3] = 0.0
        x[2 * k + 1] = x[2 * k] + d / np.linalg.norm(d) * 10.0 ** -(1 + k % 6)
    pos = torch.tensor(np.c_[x, c], device="cuda")
    plan = gpu_lib.Plan(box, N, a, 1.0, 2, precision="fp64")
    got = {}
    for s in (8, split):
        gpu_lib.mls6_set_tuning(plan.handle, s, 0)
        r = plan.evaluate(pos, virial=True, atom_energy=True)
        torch.cuda.synchronize()
        got[s] = (r["F"].cpu().numpy(), r["out"].cpu().numpy(), r["eatom"].cpu().numpy())
    (f0, o0, e0), (f1, o1, e1) = got[8], got[split]
    # the virial is that of the close pairs, up to 1e-30 of its size: their
    # d (x) d, from the wrapped positions (the one-atom kernel's product with
    # x_i has lost |x_i| / r of it)
    L = np.array(box)
    xw = (x - np.floor(x / L) * L).astype(np.longdouble)
    d = xw[1:40:2] - xw[0:40:2]
    d -= np.round((d / L).astype(np.float64)) * L.astype(np.longdouble)
    r2 = np.sum(d * d, axis=1)
    k = -6.0 * c[0:40:2] * c[1:40:2] / r2 ** 4
    W = np.array([np.sum(k * d[:, p] * d[:, q]) for p, q in
                  ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]).astype(np.float64)
    assert np.abs(o1[1:] - W).max() <= 1e-11 * np.abs(W).max()
    # the largest term of a close pair is its force itself; elsewhere ~30
    scale = np.maximum(np.abs(f0).max(axis=1, keepdims=True), 30.0)
    assert np.all(np.abs(f1 - f0) <= 1e-12 * scale)
    assert np.all(np.abs(e1 - e0) <= 1e-12 * np.maximum(np.abs(e0), 10.0))
    assert abs(o1[0] - o0[0]) <= 1e-12 * abs(o0[0])
