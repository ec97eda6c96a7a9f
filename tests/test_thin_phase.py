"""Thin phases beside dense ones (a vapour around a droplet or a slab): the grid
part runs by the direct kernels there, whose rounding is relative to each
node's own potential, and by transforms otherwise."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1308_4005_gb300 import build as B
from paper_1308_4005_gb300 import inputs as I

# ---------------------------------------------------------------- on the CPU

COUNT = r"""
#include <cstdio>
#include <set>
#include <vector>
#include "mls6_internal.h"

int main() {
  unsigned s = 1;
  const int dims[][3] = {{1, 1, 1}, {2, 1, 3}, {3, 2, 1}, {4, 3, 2}, {1, 5, 4}, {2, 6, 5},
                         {5, 4, 3}, {7, 5, 6}, {16, 1, 2}, {3, 3, 3}, {4, 4, 4}};
  for (auto& d : dims) {
    const int nc[3] = {d[0], d[1], d[2]};
    const long n = (long)nc[0] * nc[1] * nc[2];
    std::vector<int> start(n + 1, 0);  // exactly ncell + 1 entries: reads beyond are seen by ASAN
    for (long c = 0; c < n; ++c) start[c + 1] = start[c] + (int)((s = s * 1664525u + 1013904223u) >> 29);
    for (long c = 0; c < n; ++c) {
      std::set<long> cells;
      const int x = c % nc[0], y = c / nc[0] % nc[1], z = c / ((long)nc[0] * nc[1]);
      for (int k = 0; k < 27; ++k)
        cells.insert((x + k % 3 - 1 + nc[0]) % nc[0] +
                     nc[0] * ((y + k / 3 % 3 - 1 + nc[1]) % nc[1] +
                              (long)nc[1] * ((z + k / 9 - 1 + nc[2]) % nc[2])));
      int want = 0;
      for (long k : cells) want += start[k + 1] - start[k];
      const int got = mls6::atoms_around(start.data(), nc, x, y, z);
      if (got != want) printf("%d %d %d cell %ld: %d, not %d\n", nc[0], nc[1], nc[2], c, got, want);
    }
  }
  printf("done\n");
}
"""


def test_atoms_around_counts_each_cell_once(tmp_path):
    """Every cell's periodic 3 x 3 x 3 surroundings, each cell once, also where
    an axis has one or two cells; no read outside the ncell + 1 starts."""
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(B._nvcc())))
    src = tmp_path / "t.cpp"
    src.write_text(COUNT)
    exe = str(tmp_path / "t")
    subprocess.run([shutil.which("g++") or "g++", "-std=c++17", "-O1", "-fsanitize=address",
                    str(src), "-o", exe, "-I", os.path.join(cuda, "include"), "-I", B.CSRC],
                   check=True)
    assert subprocess.run([exe], capture_output=True, text=True, check=True).stdout == "done\n"


# ---------------------------------------------------------------- on the GPU

A = 3.0


def _droplet(cv=1.0):
    """A droplet and 40 atoms far from it and from each other, of coefficient cv."""
    box = (48.0, 40.0, 48.0)
    rng = np.random.default_rng(31)
    mid = np.array(box) / 2
    x = I.rsa_positions(rng, 2200, tuple((m - 8.0, m + 8.0) for m in mid), box, 0.8)
    x = x[np.linalg.norm(x - mid, axis=1) < 8.0]
    v = I.rsa_positions(rng, 120, tuple((0.0, b) for b in box), box, 5.0)
    v = v[np.linalg.norm(v - mid, axis=1) > 13.0][:40]
    c = np.concatenate([np.sqrt(rng.uniform(0.5, 1.5, len(x))), np.full(len(v), cv)])
    return box, np.concatenate([x, v]), c, len(x)


def _slab():
    """A liquid slab: surfaces, no thin phase."""
    box = (12.0, 12.0, 36.0)
    rng = np.random.default_rng(32)
    x = I.rsa_positions(rng, 1500, ((0.0, 12.0), (0.0, 12.0), (11.0, 25.0)), box, 0.8)
    return box, x, np.sqrt(rng.uniform(0.5, 1.5, len(x))), len(x)


def _run(lib, box, x, c, prec, order=3, stencil="auto", virial=True, levels=3, h=1.0, groups=2):
    import torch

    dt = torch.float64 if prec == "fp64" else torch.float32
    plan = lib.Plan(box, len(c), A, h, levels, precision=prec, order=order, stencil=stencil)
    lib.mls6_set_tuning(plan.handle, 0, groups)
    pos = torch.tensor(np.c_[x, c], dtype=dt, device="cuda")
    r = plan.evaluate(pos, virial=virial, atom_energy=True)
    torch.cuda.synchronize()
    return (r["F"].cpu().numpy(), r["eatom"].cpu().numpy(), r["out"].cpu().numpy(), plan, pos)


@pytest.mark.gpu
@pytest.mark.parametrize("prec,order,virial,h,groups",
                         [("fp32", 3, True, 1.0, 2), ("fp32", 3, True, 1.0, 4),
                          ("fp32", 5, False, 1.0, 4), ("fp32", 5, True, 1.0, 2),
                          ("mixed", 3, False, 1.0, 2), ("fp32", 3, True, 0.4, 2),
                          ("fp32", 3, False, 0.4, 4)])
def test_thin_phase_takes_the_direct_kernels(gpu_lib, prec, order, virial, h, groups):
    """Bit for bit the direct kernels that a mixed plan can ask for, with two
    and four thread groups per tile: forces and energies; the virial to the
    rounding of its FP64 sum over records in another order.  At h = 0.4 the
    stencil's tile does not fit in shared memory."""
    box, x, c, nd = _droplet()
    if h < 1.0:  # its own, smaller box
        box = (24.0, 22.0, 20.0)
        rng = np.random.default_rng(33)
        mid = np.array(box) / 2
        x = np.concatenate([I.rsa_positions(rng, 150, tuple((m - 2.5, m + 2.5) for m in mid), box,
                                            0.8), [[2.0, 2.0, 2.0], [22.0, 20.0, 3.0]]])
        c = np.ones(len(x))
    F, e, o, _, _ = _run(gpu_lib, box, x, c, prec, order, "auto", virial, h=h, groups=groups)
    F1, e1, o1, _, _ = _run(gpu_lib, box, x, c, "mixed", order, "cuda", virial, h=h, groups=groups)
    assert np.array_equal(F, F1) and np.array_equal(e, e1) and o[0] == o1[0]
    assert np.abs(o[1:] - o1[1:]).max() <= 1e-13 * max(np.abs(o1[1:]).max(), 1e-300)


@pytest.mark.gpu
@pytest.mark.parametrize("case", ["slab", "coefficients"])
def test_dense_phases_take_the_transforms(gpu_lib, case):
    """Surfaces alone do not count as a thin phase (the forces differ from the
    direct kernels' in rounding); a light species beside a heavy one does, by
    its coefficients."""
    box, x, c, _ = _slab()
    if case == "coefficients":
        c = np.where(np.arange(len(c)) % 2, c, 0.02 * c)
    F, _, _, _, _ = _run(gpu_lib, box, x, c, "fp32")
    F1, _, _, _, _ = _run(gpu_lib, box, x, c, "mixed", stencil="cuda")
    assert np.array_equal(F, F1) == (case == "coefficients")


@pytest.mark.gpu
@pytest.mark.parametrize("cv", [1.0, 0.01])
def test_thin_phase_vapour_precision(gpu_lib, cv):
    """The vapour's FP32 forces against FP64 on the same inputs: the direct
    kernels round at u = 6e-8 relative to each node's own potential, which is
    the atom's own (about 2e-3 c) plus the droplet's; the force is the
    potential's gradient over 1/h with at most ~10^3 terms of one sign, and
    the fixed-point sums round at 2^-30 of a bound about 10^3 above them:
    1e-8 cv at most.  (Transforms: 4e-9 x the droplet's scale on every atom.)"""
    box, x, c, nd = _droplet(cv)
    x, c = (v.astype(np.float32).astype(np.float64) for v in (x, c))
    F, e, _, _, _ = _run(gpu_lib, box, x, c, "fp32")
    F0, e0, _, _, _ = _run(gpu_lib, box, x, c, "fp64")
    assert np.abs(F - F0)[nd:].max() <= 1e-8 * cv


@pytest.mark.gpu
def test_thin_phase_fp64_vs_oracle(gpu_lib, orc):
    """FP64 at its tolerances, grids included (a small droplet and two atoms)."""
    box = (16.0, 14.0, 12.0)
    rng = np.random.default_rng(34)
    x = np.concatenate([I.rsa_positions(rng, 60, ((6.0, 10.0), (5.0, 9.0), (4.0, 8.0)), box, 0.8),
                        [[1.0, 1.0, 1.0], [15.0, 13.0, 2.0]]])
    c = np.sqrt(rng.uniform(0.5, 1.5, len(x)))
    F, e, out, plan, _ = _run(gpu_lib, box, x, c, "fp64", levels=2)
    n = orc.grid_dims(box, 1.0, 2)
    o = orc.evaluate(box, A, n, 2, x, c)
    G = orc.grids(box, A, n, 2, x, c)
    rms = np.sqrt(np.mean(np.sum(o["F"] ** 2, axis=1)))
    assert abs(out[0] - o["E"]) <= 1e-12 * abs(o["E"])
    assert np.abs(F - o["F"]).max() <= 1e-11 * rms
    assert np.abs(out[1:] - o["W"]).max() <= 1e-11 * np.abs(o["W"]).max()
    for w in range(3):
        for k in (1, 2):
            got = gpu_lib.mls6_debug_grid(plan.handle, k, w)
            assert np.abs(got - G[k - 1][w]).max() <= 1e-12 * np.abs(G[k - 1][w]).max(), (k, w)


@pytest.mark.gpu
@pytest.mark.parametrize("mode", [False, True], ids=["chains", "persistent"])
def test_thin_phase_in_a_batch(gpu_lib, mode):
    """A replica with a thin phase beside one without: each as its own plan."""
    import torch

    sys_ = [_droplet(), _slab()]
    pos = torch.tensor(np.concatenate([np.c_[x, c] for _, x, c, _ in sys_]), dtype=torch.float32,
                       device="cuda")
    bt = gpu_lib.Batch([s[0] for s in sys_], [len(s[2]) for s in sys_], A, 1.0, 3,
                       precision="fp32")
    gpu_lib.mls6_batch_set_mode(bt.handle, mode)
    for _ in range(2):  # the queues start from zero again
        r = bt.evaluate(pos)
        torch.cuda.synchronize()
    info = bt.info()
    E, W, F = (r[k].cpu().numpy() for k in ("E", "W", "F"))
    for k, (box, x, c, _) in enumerate(sys_):
        plan = gpu_lib.Plan(box, len(c), A, 1.0, 3, precision="fp32")
        gpu_lib.mls6_set_tuning(plan.handle, info["pair_split"][k], info["stencil_groups"][k])
        q = plan.evaluate(torch.tensor(np.c_[x, c], dtype=torch.float32, device="cuda"))
        torch.cuda.synchronize()
        o = q["out"].cpu().numpy()
        sl = slice(bt.offsets[k], bt.offsets[k + 1])
        assert E[k] == o[0] and np.array_equal(W[k], o[1:])
        assert np.array_equal(F[sl], q["F"].cpu().numpy())


@pytest.mark.gpu
@pytest.mark.parametrize("groups", [2, 4])
def test_thin_phase_lorentz_berthelot(gpu_lib, groups):
    """Bit for bit the direct kernels of a mixed plan that asks for them; twice,
    as the workspace is allocated by the first call."""
    import torch

    box, x, _, nd = _droplet()
    rng = np.random.default_rng(35)
    s, ep = rng.uniform(0.95, 1.05, len(x)), rng.uniform(0.8, 1.2, len(x))
    out = []
    for prec, st in (("fp32", "auto"), ("mixed", "cuda")):
        plan = gpu_lib.Plan(box, len(x), A, 1.0, 3, precision=prec, stencil=st)
        gpu_lib.mls6_set_tuning(plan.handle, 0, groups)
        p, sg, e = (torch.tensor(v, dtype=torch.float32, device="cuda").contiguous()
                    for v in (x, s, ep))
        for _ in range(2):
            F = torch.empty_like(p)
            E = torch.zeros(1, dtype=torch.float64, device="cuda")
            assert gpu_lib.mls6_eval_lb(plan.handle, p.data_ptr(), sg.data_ptr(), e.data_ptr(),
                                        F.data_ptr(), E.data_ptr()) == 0
            torch.cuda.synchronize()
            out.append((F.cpu().numpy(), float(E[0])))
    for F, E in out[1:]:
        assert np.array_equal(F, out[0][0]) and E == out[0][1]


@pytest.mark.gpu
def test_grid_form_query(gpu_lib):
    """Which form the plan has and which the last evaluation ran."""
    import torch

    box, x, _, nd = _droplet()
    y = x.copy()  # the vapour's atoms moved into the droplet
    y[nd:] = np.array(box) / 2 + np.random.default_rng(36).uniform(-4.0, 4.0, (len(x) - nd, 3))
    for prec in ("fp32", "fp64", "mixed"):
        plan = gpu_lib.Plan(box, len(x), A, 1.0, 3, precision=prec)
        for at, last in ((x, False), (y, True), (x, False)):
            plan.evaluate(torch.tensor(np.c_[at, np.ones(len(x))], device="cuda",
                                       dtype=torch.float64 if prec == "fp64" else torch.float32))
            assert gpu_lib.mls6_grid_form(plan.handle) == (True, last)
        assert plan.info()["transforms"]
    for kw in (dict(levels=3, precision="mixed", stencil="cuda"), dict(levels=1)):
        plan = gpu_lib.Plan((16.0, 16.0, 16.0), 10, A, 1.0, **kw)
        assert gpu_lib.mls6_grid_form(plan.handle) == (False, False)
