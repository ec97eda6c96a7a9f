"""Energies and virials into a new buffer on every call: the evaluation is the
same, and an earlier call's buffer keeps what it got."""
import pytest

from paper_1308_4005_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_new_result_buffers(gpu_lib, prec):
    import numpy as np
    import torch

    box, N = (9.0, 9.0, 9.0), 500
    dt = torch.float64 if prec == "fp64" else torch.float32
    x, c = I.uniform_atoms(7, N, box)
    pos = torch.tensor(np.c_[x, c], dtype=dt, device="cuda")
    plan = gpu_lib.Plan(box, N, 2.2, 0.75, 3, precision=prec)
    F = torch.empty((N, 3), dtype=dt, device="cuda")
    buf = torch.full((6, 16), -1.0, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()

    def call(energy, virial):
        rc = gpu_lib.mls6_eval(plan.handle, pos.data_ptr(), 0, F.data_ptr(), energy, virial)
        assert rc == 0
        torch.cuda.synchronize()

    at = lambda r, k: buf[r, k:].data_ptr()  # noqa: E731
    call(at(0, 0), at(0, 1))   # one copy
    call(at(1, 0), at(1, 1))   # the same into another buffer
    call(at(2, 0), at(2, 8))   # two copies
    call(at(3, 4), at(3, 8))   # two copies into another buffer
    call(0, at(4, 1))          # the virial alone, twice
    call(0, at(5, 1))
    b = buf.cpu().numpy()
    E, W = b[0, 0], b[0, 1:7]
    assert E < 0 and np.all(W != -1.0) and np.all(b[0, 7:] == -1.0)
    assert np.array_equal(b[1], b[0])
    assert b[2, 0] == E and np.array_equal(b[2, 8:14], W) and np.all(b[2, 1:8] == -1.0)
    assert b[3, 4] == E and np.array_equal(b[3, 8:14], W) and np.all(b[3, :4] == -1.0)
    for r in (4, 5):
        assert b[r, 0] == -1.0 and np.array_equal(b[r, 1:7], W)
