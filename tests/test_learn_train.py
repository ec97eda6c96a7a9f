"""The one-pass training kernel at the edges of its 128-atom tiles and of its
152-block grid.

Tolerances: against the FP64 reference those of test_learn.py (BF16
activations and tanh.approx: loss 3e-2, gradient 5e-2 relative L2).  The last
row's target is 30 times the others', so that losing or repeating it shows.
Between a batch and its quarters the row terms are the same numbers (2 / N
differs by a power of two), only FP32 sums are split differently: chains of at
most 32 products' sums, 32 * 2^-23 of the terms' absolute sum, which random
signs leave at most sqrt(N) = 128 times the gradient's norm: 1e-3.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mlp_ref(orc):
    from oracle import mlp

    return mlp


def _params(mlp_ref, seed):
    p = np.random.default_rng(seed).normal(0, 0.15, mlp_ref.n_params())
    for W, b in [mlp_ref.unpack(p)[3]]:
        W[:, 3:] = 0.0
        b[3:] = 0.0
    return p.astype(np.float32)


def _batch(N, seed):
    """N rows in front of NaN rows that must not be read."""
    rng = np.random.default_rng(seed)
    X = np.full((N + 200, 128), np.nan)
    T = np.full((N + 200, 3), np.nan)
    X[:N], T[:N] = rng.normal(0, 1, (N, 128)), rng.normal(0, 0.5, (N, 3))
    T[N - 1] *= 30.0
    return (torch.tensor(X, dtype=torch.float32).to(torch.bfloat16).cuda()[:N],
            torch.tensor(T, dtype=torch.float32).cuda()[:N])


@pytest.mark.parametrize("N", [1, 16, 127, 128, 129, 152 * 128, 152 * 128 + 1])
def test_gradient_at_tile_edges(gpu_lib, mlp_ref, N):
    p = _params(mlp_ref, N)
    X, T = _batch(N, N + 1)
    m = gpu_lib.MLP(0)
    m.set_params(p)
    loss, g = m.grad(X, T)
    lr, gr = mlp_ref.loss_grad(p.astype(np.float64), X.double().cpu().numpy(),
                               T.double().cpu().numpy())
    g = g.double().cpu().numpy()
    assert loss == pytest.approx(lr, rel=3e-2)
    assert np.linalg.norm(g - gr) <= 5e-2 * np.linalg.norm(gr)


def test_gradient_of_quarters(gpu_lib, mlp_ref):
    N = 16384
    X, T = _batch(N, 7)
    m = gpu_lib.MLP(0)
    m.set_params(_params(mlp_ref, 8))
    loss, g = m.grad(X, T)
    parts = [m.grad(x.contiguous(), t.contiguous()) for x, t in zip(X.chunk(4), T.chunk(4))]
    gq = sum(q[1].double() for q in parts) / 4
    assert loss == pytest.approx(sum(q[0] for q in parts) / 4, rel=1e-12)
    assert (g.double() - gq).norm() <= 1e-3 * gq.norm()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("N", [1, 31, 33, 1000])
def test_apply_is_forward_of_the_features(gpu_lib, mlp_ref, N, prec):
    """F + c s y with y from the stored features: one product and one sum
    apart (2 u of the larger operand)."""
    dt = torch.float64 if prec == "fp64" else torch.float32
    rng = np.random.default_rng(N)
    pos = torch.tensor(np.c_[rng.uniform(0, 9, (N, 3)), rng.uniform(0.5, 1.5, N)], dtype=dt,
                       device="cuda")
    plan = gpu_lib.Plan((9.0, 9.0, 9.0), N, 2.2, 0.75, 3, precision=prec)
    plan.evaluate(pos, virial=False)
    m = gpu_lib.MLP(0)
    m.set_params(_params(mlp_ref, 3))
    m.set_norm(np.zeros(128), np.full(128, 0.1), 0.7)
    y = m.forward(m.features(plan, fmt="bf16"))[:, :3].to(dt)
    F = torch.ones((N, 3), dtype=dt, device="cuda")
    torch.cuda.synchronize()
    m.apply(plan, F)
    torch.cuda.synchronize()
    add = pos[:, 3:] * torch.tensor(0.7, dtype=torch.float32).to(dt) * y
    u = 2.0**-24 if prec == "fp32" else 2.0**-53
    assert (F - (1 + add)).abs().max() <= 4 * u * (1 + add.abs().max())


def test_forward_of_rows_off_16_bytes(gpu_lib, mlp_ref):
    """Rows that start on a 4-byte boundary give what aligned rows give."""
    m = gpu_lib.MLP(0)
    m.set_params(_params(mlp_ref, 4))
    X = torch.randn(300 * 128 + 2, device="cuda").to(torch.bfloat16)
    off = X[2:].view(300, 128)
    assert off.data_ptr() % 16 == 4
    assert torch.equal(m.forward(off), m.forward(off.clone()))
