"""The grid part in Fourier space (the default between q^1 and e^{1,tot})
against the FP64 oracle and against the direct kernels.

FP64: the tolerances of the FP64 path (1e-12 of the energy, 1e-11 of the
forces and the virial; the potential to 1e-12 of its maximum, as the direct
grids).  FP32: both forms round each node sum at u = 6e-8 over sums of
~10^3 terms or ~20 transform passes, far inside the FP32 path's 1e-4 of the
RMS force, 2e-6 of the energy and 2e-5 of the virial.
"""
import zlib

import numpy as np
import pytest

from paper_1308_4005_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CASES = [
    # name, box, a, h, levels, order, continuity: grid
    ("radix_4_4_2", (16.0, 8.0, 32.0), 2.5, 1.0, 2, 3, 2),     # 16 x 8 x 32
    ("radix_3_5_7", (12.0, 10.0, 14.0), 2.0, 1.0, 2, 3, 2),
    ("radix_11_13", (22.0, 13.0, 26.0), 2.0, 1.0, 2, 3, 2),    # 13 -> 14 nodes along y
    ("radix_17_19", (34.0, 38.0, 18.0), 2.0, 1.0, 2, 3, 2),
    ("two_nodes", (1.0, 1.0, 2.0), 1.0, 0.5, 2, 3, 2),
    ("quintic", (9.0, 8.0, 16.0), 2.0, 1.0, 3, 5, 2),
    ("smoothing_c3", (12.0, 12.0, 8.0), 2.0, 1.0, 3, 3, 3),
    ("five_levels", (16.0, 16.0, 16.0), 1.2, 0.5, 5, 3, 2),
    ("six_levels_direct", (16.0, 16.0, 16.0), 1.2, 0.5, 6, 3, 2),
]


def _atoms(name, box, prec):
    N = 40
    x, c = I.uniform_atoms(zlib.crc32(name.encode()) % 10000, N, box,
                           dmin=0.1 if min(box) < 4 else 0.8)
    return (x, c) if prec == "fp64" else tuple(v.astype(np.float32).astype(np.float64)
                                               for v in (x, c))


@pytest.mark.parametrize("name,box,a,h,l,order,cont", CASES, ids=[c[0] for c in CASES])
def test_spectral_fp64_vs_oracle(gpu_lib, orc, name, box, a, h, l, order, cont):
    import torch

    x, c = _atoms(name, box, "fp64")
    n = orc.grid_dims(box, h, l)
    p0 = orc.order()
    orc.set_order(order)
    try:
        with orc.smoothing_order(cont):
            o = orc.evaluate(box, a, n, l, x, c)
            G = orc.grids(box, a, n, l, x, c)
    finally:
        orc.set_order(p0)
    plan = gpu_lib.Plan(box, len(c), a, h, l, precision="fp64", order=order, continuity=cont)
    pos = torch.tensor(np.c_[x, c], device="cuda")
    r = plan.evaluate(pos, virial=True)
    torch.cuda.synchronize()
    out, F = r["out"].cpu().numpy(), r["F"].cpu().numpy()
    et = gpu_lib.mls6_debug_grid(plan.handle, 1, 2)
    assert np.abs(et - G[0][2]).max() <= 1e-12 * np.abs(G[0][2]).max()
    # the sums of the large terms that a sparse system's energy is left from
    scale = np.abs(o["E"]) + 0.5 * np.abs(np.sum(c * c)) * 1.875 / a ** 6
    rms = np.sqrt(np.mean(np.sum(o["F"] ** 2, axis=1)))
    assert abs(out[0] - o["E"]) <= 1e-12 * scale
    assert np.abs(F - o["F"]).max() <= 1e-11 * rms
    assert np.abs(out[1:] - o["W"]).max() <= 1e-11 * (np.abs(o["W"]).max() + scale)


@pytest.mark.parametrize("box,a,h,l", [((24.0, 22.0, 26.0), 2.5, 1.0, 2),
                                       ((16.0, 24.0, 40.0), 2.5, 1.0, 4)])
def test_spectral_fp32_vs_direct_kernels(gpu_lib, box, a, h, l):
    """The same FP32 plan with the transforms (automatic) and with the
    CUDA-core stencils (on request), with and without the virial; repeatable."""
    import torch

    N = 4000
    x, c = I.uniform_atoms(11, N, box)
    pos = torch.tensor(np.c_[x, c], dtype=torch.float32, device="cuda")
    got = {}
    for stencil in ("auto", "cuda"):
        plan = gpu_lib.Plan(box, N, a, h, l, precision="mixed", stencil=stencil)
        for vir in (True, False):
            r = plan.evaluate(pos, virial=vir)
            again = plan.evaluate(pos, virial=vir)
            torch.cuda.synchronize()
            assert torch.equal(r["F"], again["F"]) and torch.equal(r["out"], again["out"])
            got[stencil, vir] = r["out"].cpu().numpy(), r["F"].cpu().double().numpy()
        got[stencil] = [gpu_lib.mls6_debug_grid(plan.handle, k, w)
                        for k in range(1, l + 1) for w in range(3)]
    for vir in (True, False):
        (a0, f0), (a1, f1) = got["auto", vir], got["cuda", vir]
        rms = np.sqrt(np.mean(np.sum(f1 ** 2, axis=1)))
        assert abs(a0[0] - a1[0]) <= 2e-6 * abs(a1[0])
        assert np.abs(f0 - f1).max() <= 1e-4 * rms
        if vir:
            assert np.abs(a0[1:] - a1[1:]).max() <= 2e-5 * np.abs(a1[1:]).max()
    for g0, g1 in zip(got["auto"], got["cuda"]):  # every grid of every level
        assert np.abs(g0 - g1).max() <= 2e-5 * np.abs(g1).max()


def test_grids_the_transforms_do_not_take(gpu_lib):
    """A prime factor above 19: the automatic choice is the direct kernels
    (bit for bit the plan that asks for them)."""
    import torch

    box, N = (46.0, 8.0, 8.0), 500
    x, c = I.uniform_atoms(12, N, box)
    pos = torch.tensor(np.c_[x, c], dtype=torch.float32, device="cuda")
    got = []
    for stencil in ("auto", "cuda"):
        plan = gpu_lib.Plan(box, N, 2.0, 1.0, 2, precision="mixed", stencil=stencil)
        r = plan.evaluate(pos, virial=True)
        torch.cuda.synchronize()
        got.append(r)
    assert torch.equal(got[0]["F"], got[1]["F"]) and torch.equal(got[0]["out"], got[1]["out"])
