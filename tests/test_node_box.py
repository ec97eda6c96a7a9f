"""Node boxes of a block's atoms (anterpolation, interpolation, features): the
box that fits in shared memory, the one that does not, and grids of the fewest
nodes, whose boxes wrap around several times.

Tolerances: energies and forces those of test_gpu_parity.py and test_lb.py;
features those of test_learn.py.  The interpolation of several waves of blocks
is compared with the same FP32 basis arguments in FP64: the chain of at most 12
rounded sums and 4-operation weights stays below 64 u of the largest potential
over h (the weights' absolute sums are below 4), u = 2^-24.
"""
import numpy as np
import pytest

from paper_1308_4005_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# name, atoms, box, a, h, levels: 300 atoms on 40^3 nodes (a block's box holds
# most of them: too large), 550 on 12^3 (fits), 4 nodes per axis
SYSTEMS = [
    ("sparse", 300, (24.0, 24.0, 24.0), 2.0, 0.6, 3),
    ("dense", 550, (9.0, 9.0, 9.0), 2.2, 0.75, 3),
    ("four_nodes", 257, (6.0, 6.0, 6.0), 2.0, 1.5, 1),
]
TOL = {"fp64": (1e-12, 1e-11), "fp32": (2e-6, 1e-4)}


def _check(E, F, r, prec):
    rms = np.sqrt(np.mean(np.sum(r["F"] ** 2, axis=1)))
    assert abs(E - r["E"]) <= TOL[prec][0] * abs(r["E"])
    assert np.abs(F - r["F"]).max() <= TOL[prec][1] * rms


@pytest.mark.parametrize("order", [3, 5])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name,N,box,a,h,l", SYSTEMS)
def test_evaluation(gpu_lib, orc, name, N, box, a, h, l, prec, order):
    import torch

    if order == 5 and name == "four_nodes":
        h = 1.0  # the quintic's support is six nodes
    dt = torch.float64 if prec == "fp64" else torch.float32
    x, c = I.uniform_atoms(17 + N, N, box)
    pos = torch.tensor(np.c_[x, c], dtype=dt, device="cuda")
    q = pos.double().cpu().numpy()
    n = orc.grid_dims(box, h, l)
    with orc.interp_order(order):
        r = orc.evaluate(box, a, n, l, q[:, :3], q[:, 3])
    plan = gpu_lib.Plan(box, N, a, h, l, precision=prec, order=order)
    g = plan.evaluate(pos, virial=True)
    _check(float(g["out"][0]), g["F"].double().cpu().numpy(), r, prec)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name,N,box,a,h,l", SYSTEMS)
def test_lorentz_berthelot(gpu_lib, orc, name, N, box, a, h, l, prec):
    import torch
    from oracle import lb

    dt = torch.float64 if prec == "fp64" else torch.float32
    x, _ = I.uniform_atoms(19 + N, N, box)
    rng = np.random.default_rng(N)
    pos, s, e = (torch.tensor(v, dtype=dt, device="cuda").contiguous()
                 for v in (x, rng.uniform(0.85, 1.15, N), rng.uniform(0.5, 1.5, N)))
    n = orc.grid_dims(box, h, l)
    r = lb.evaluate_lb(box, a, n, l, *(v.double().cpu().numpy() for v in (pos, s, e)))
    plan = gpu_lib.Plan(box, N, a, h, l, precision=prec)
    F = torch.empty((N, 3), dtype=dt, device="cuda")
    E = torch.zeros(1, dtype=torch.float64, device="cuda")
    rc = gpu_lib.mls6_eval_lb(plan.handle, pos.data_ptr(), s.data_ptr(), e.data_ptr(),
                              F.data_ptr(), E.data_ptr())
    assert rc == 0
    torch.cuda.synchronize()
    _check(float(E), F.double().cpu().numpy(), r, prec)


@pytest.mark.parametrize("name,N,box,a,h,l", SYSTEMS)
def test_features(gpu_lib, orc, name, N, box, a, h, l):
    import torch
    from oracle import mlp

    x, c = I.uniform_atoms(23 + N, N, box)
    plan = gpu_lib.Plan(box, N, a, h, l, precision="fp64")
    plan.evaluate(torch.tensor(np.c_[x, c], dtype=torch.float64, device="cuda"), virial=False)
    m = gpu_lib.MLP(1)
    X = m.features(plan, fmt="f32").double().cpu().numpy()
    n = orc.grid_dims(box, h, l)
    E1 = orc.grids(box, a, n, l, x, c)[0][2]
    ref = mlp.features(E1, np.array(box) / np.array(n), np.mod(x, np.array(box)))
    assert np.abs(X - ref).max() <= 1e-6 * np.abs(ref).max()


@pytest.mark.parametrize("h", [4.0, 1.0])  # the box fits, and does not
def test_interpolation_of_several_waves(gpu_lib, h):
    """157,464 atoms of which no two lie within the cutoff: the force is the
    grid's alone."""
    import torch

    m, s, a = 54, 4.0, 3.0
    L = m * s
    rng = np.random.default_rng(5)
    at = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)
    x = ((at + 0.5) * s + rng.uniform(-0.49, 0.49, at.shape)).astype(np.float32)
    c = rng.uniform(0.5, 1.5, len(x)).astype(np.float32)
    plan = gpu_lib.Plan((L, L, L), len(x), a, h, 2, precision="fp32")
    F = plan.evaluate(torch.tensor(np.c_[x, c], device="cuda"), virial=False)["F"]
    e = gpu_lib.mls6_debug_grid(plan.handle, 1, 2)
    n = round(L / h)
    e = np.asarray(e, dtype=np.float64).reshape(n, n, n)
    u = x * np.float32(1.0 / h)
    base = np.floor(u)
    t = (u - base).astype(np.float64)
    k = base.astype(int)

    def phi(t):
        v = np.abs(t)
        w = np.where(v < 1, 1 - 2.5 * v**2 + 1.5 * v**3, 0.5 * (1 - v) * (2 - v) ** 2)
        d = np.where(v < 1, -5 * v + 4.5 * v**2, -0.5 * (2 - v) ** 2 - (1 - v) * (2 - v))
        return w, d * np.sign(t)

    g = np.zeros(x.shape)
    for dz in range(-1, 3):
        wz, gz = phi(t[:, 2] - dz)
        for dy in range(-1, 3):
            wy, gy = phi(t[:, 1] - dy)
            for dx in range(-1, 3):
                wx, gx = phi(t[:, 0] - dx)
                v = e[(k[:, 2] + dz) % n, (k[:, 1] + dy) % n, (k[:, 0] + dx) % n]
                g += np.stack([gx * wy * wz, wx * gy * wz, wx * wy * gz], 1) * v[:, None]
    ref = c[:, None].astype(np.float64) * g / h
    err = np.abs(F.double().cpu().numpy() - ref).max()
    assert err <= 64 * 2.0**-24 * np.abs(e).max() * c.max() / h, err


def test_fp64_block_size_rule(gpu_lib):
    """152 blocks of 256 atoms are the first that keep the larger block; atoms
    of coefficient zero, there or left out, change nothing but the block size."""
    import torch

    N, L = 152 * 256, 36.0
    rng = np.random.default_rng(3)
    m = 34  # jittered lattice, no two atoms close
    at = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)[:N]
    x = (at + 0.5 + rng.uniform(-0.1, 0.1, at.shape)) * (L / m)
    q = np.c_[x, rng.uniform(0.5, 1.5, N)]
    q = np.concatenate([q, [[0.0, 0.0, 0.0, 0.0]]])
    r = []
    for n in (N - 256, N, N + 1):
        p = np.concatenate([q[:N], q[N:]])[:n] if n >= N else q[:n]
        plan = gpu_lib.Plan((L, L, L), n, 2.5, 1.0, 3, precision="fp64")
        g = plan.evaluate(torch.tensor(p, device="cuda"), virial=True)
        r.append((g["out"].cpu().numpy(), g["F"].cpu().numpy()))
    assert np.abs(r[1][0] - r[2][0]).max() <= 1e-12 * np.abs(r[1][0]).max()
    assert np.abs(r[1][1] - r[2][1][:N]).max() <= 1e-11 * np.abs(r[1][1]).max()
    # the 128-thread blocks: the last 256 atoms' coefficients zero against left out
    plan = gpu_lib.Plan((L, L, L), N, 2.5, 1.0, 3, precision="fp64")
    z = q[:N].copy()
    z[N - 256:, 3] = 0.0
    g = plan.evaluate(torch.tensor(z, device="cuda"), virial=True)
    assert np.abs(g["out"].cpu().numpy() - r[0][0]).max() <= 1e-12 * np.abs(r[0][0]).max()
    assert np.abs(g["F"].cpu().numpy()[: N - 256] - r[0][1]).max() <= 1e-11 * np.abs(r[0][1]).max()
