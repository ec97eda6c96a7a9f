"""The virial of the transformed grid part in FP32: what is kept in FP64, and
its range."""
import numpy as np
import pytest

from paper_1308_4005_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _gamma_d(rho):
    """gamma'(rho)/rho of gamma = 15/8 - 5/4 rho^12 + 3/8 rho^24 (rho < 1), rho^-6."""
    return np.where(rho < 1.0, -15.0 * rho ** 10 + 9.0 * rho ** 22,
                    -6.0 * np.maximum(rho, 1.0) ** -8.0)


def _k1(a):
    """sum over the level-1 taps |m| < 2a (h = 1) of g_1'/r m_x^2."""
    m = np.arange(-2.0, 3.0)
    r = np.stack(np.meshgrid(m, m, m, indexing="ij"), -1)
    d = np.sqrt((r ** 2).sum(-1))
    G = (_gamma_d(d / a) / a ** 8 - _gamma_d(d / (2 * a)) / (2 * a) ** 8) * (d < 2 * a)
    return (G * r[..., 0] ** 2).sum()


@pytest.mark.parametrize("a", [0.95, 0.9, 0.8, 0.7])
def test_coarsest_virial_is_kept_in_fp64(gpu_lib, a):
    """An atom of c = 1 on every node of a 4 x 4 x 4 grid of spacing 1, none
    within the cutoff of another: only the zero frequency is present, and every
    step of the FP32 plan up to it is exact.  Level 1 contributes 1/2 64^2 / 64
    = 32 times its FP32 table entry, exactly; the coarsest level its FP64
    product.  What remains is the rounding of FP64 sums: 1e-13 of the virial."""
    import torch

    g = np.stack(np.meshgrid(*[np.arange(4.0)] * 3, indexing="ij"), -1).reshape(-1, 3)
    W = {}
    for prec, dt in (("fp64", torch.float64), ("fp32", torch.float32)):
        plan = gpu_lib.Plan((4.0, 4.0, 4.0), 64, a, 1.0, 2, precision=prec)
        assert plan.info()["n_grid"][0] == (4, 4, 4)
        pos = torch.tensor(np.c_[g, np.ones(64)], dtype=dt, device="cuda")
        W[prec] = plan.evaluate(pos)["out"].cpu().numpy()[1:4]
    k = _k1(a)
    want = W["fp64"] + 32.0 * (float(np.float32(k)) - k)
    assert np.abs(W["fp32"] - want).max() <= 1e-13 * np.abs(W["fp64"]).max()


@pytest.mark.parametrize("shift", [56, -32])
def test_virial_scales_with_large_and_small_coefficients(gpu_lib, shift):
    """c 2^s gives the virial times 2^(2s), bit for bit: every operation on the
    way is exact under powers of two as long as none leaves the FP32 range.
    c^2 times the sums of a system of 400 atoms, 2^112 x 10^3, is inside it; the
    square of a transform's entry, (N c)^2 times the nodes, is not."""
    import torch

    box = (8.0, 8.0, 16.0)
    x, c = I.uniform_atoms(41, 400, box)
    plan = gpu_lib.Plan(box, 400, 2.0, 1.0, 2, precision="fp32")
    W = []
    for s in (0, shift):
        pos = torch.tensor(np.c_[x, c], dtype=torch.float32, device="cuda")
        pos[:, 3] *= 2.0 ** s
        W.append(plan.evaluate(pos)["out"].cpu().numpy()[1:])
    assert np.all(np.isfinite(W[1])) and np.array_equal(W[1], W[0] * 2.0 ** (2 * shift))
