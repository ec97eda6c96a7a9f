"""The order of the atoms within a cell (binning): cells of up to 8 atoms, of 9
to 256 and of more, in blocks of cells and in blocks of atoms (from 6 atoms per
cell on)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BOX, A = (12.0, 12.0, 12.0), 3.0  # 8 x 8 x 8 cells of 1.5


def _system(name):
    """(positions, whether every cell has at most 256 atoms)."""
    rng = np.random.default_rng(61)
    n, crowd = {"small_cells": (900, ()), "one_of_9": (300, (9,)), "one_of_200": (300, (200,)),
                "of_256_and_257": (200, (256, 257)), "of_700": (100, (700, 40)),
                "dense": (5000, ()), "dense_and_300": (5000, (300, 256))}[name]
    x = [rng.uniform(0.0, 12.0, (n, 3))]
    for k, m in enumerate(crowd):  # jittered points of one cell, the others emptied of it
        lo = np.array([1.5 * k, 3.0, 10.5])
        x = [v[np.any((v < lo) | (v >= lo + 1.5), axis=1)] for v in x]
        s = int(np.ceil(m ** (1 / 3)))
        g = np.stack(np.meshgrid(*[np.arange(s)] * 3, indexing="ij"), -1).reshape(-1, 3)
        g = rng.permutation(g)[:m]
        x.append(lo + 1.5 * (g + rng.uniform(0.2, 0.8, g.shape)) / s)
    x = np.concatenate(x).astype(np.float32)
    x = x[rng.permutation(len(x))]
    return x, np.bincount((x // 1.5).astype(int) @ [1, 8, 64], minlength=512).max()


def _forces(lib, x, c, prec):
    import torch

    dt = torch.float64 if prec == "fp64" else torch.float32
    plan = lib.Plan(BOX, len(x), A, 1.0, 2, precision=prec)
    pos = torch.tensor(np.c_[x, c], dtype=dt, device="cuda")
    out = [plan.evaluate(pos) for _ in range(2)]
    torch.cuda.synchronize()
    return [r["F"].cpu().numpy() for r in out]


@pytest.mark.parametrize("name", ["small_cells", "one_of_9", "one_of_200", "of_256_and_257",
                                  "of_700", "dense", "dense_and_300"])
def test_cell_order(gpu_lib, name):
    """FP32 orders a cell by x, FP64 by input index.  Two calls agree bit for
    bit, and in FP32 so do the forces of the same atoms given in another order
    (distinct x), as long as no cell has more than 256 atoms.  All of them agree
    with FP64 at the FP32 tolerance (1e-4 of the RMS force)."""
    x, most = _system(name)
    c = np.sqrt(np.random.default_rng(62).uniform(0.5, 1.5, len(x))).astype(np.float32)
    F, F2 = _forces(gpu_lib, x, c, "fp32")
    p = np.random.default_rng(63).permutation(len(x))
    G, _ = _forces(gpu_lib, x[p], c[p], "fp32")
    D, D2 = _forces(gpu_lib, x.astype(np.float64), c.astype(np.float64), "fp64")
    if most <= 256:
        assert np.array_equal(F, F2) and np.array_equal(F[p], G) and np.array_equal(D, D2)
    rms = np.sqrt(np.mean(np.sum(D ** 2, axis=1)))
    for f in (F, F2):
        assert np.abs(f - D).max() <= 1e-4 * rms
    assert np.abs(F[p] - G).max() <= 1e-4 * rms and np.abs(D - D2).max() <= 1e-11 * rms
