"""Calls of different kinds on one plan: what a call reads of the plan's state
belongs to the evaluation before it, whichever kind that was and whether it
captured its graph or replayed one."""
import numpy as np
import pytest

from paper_1308_4005_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BOX, A, H, LEVELS, N = (12.0, 10.0, 8.0), 2.0, 1.0, 3, 150


def _system():
    x, c = I.uniform_atoms(515, N, BOX)
    rng = np.random.default_rng(516)
    return x, c, rng.uniform(0.85, 1.15, N), rng.uniform(0.5, 1.5, N)


def _dev(v, prec="fp64"):
    import torch

    return torch.tensor(np.ascontiguousarray(v),
                        dtype=torch.float64 if prec == "fp64" else torch.float32, device="cuda")


def _grids(lib, plan):
    import torch

    torch.cuda.synchronize()
    return {(k, w): lib.mls6_debug_grid(plan.handle, k, w)
            for w in range(3) for k in range(1, LEVELS + 1)}


def _lb(lib, plan, pos, sg, ep):
    import torch

    F = torch.empty_like(pos)
    E = torch.zeros(1, dtype=torch.float64, device="cuda")
    assert lib.mls6_eval_lb(plan.handle, pos.data_ptr(), sg.data_ptr(), ep.data_ptr(),
                            F.data_ptr(), E.data_ptr()) == 0


@pytest.mark.parametrize("form", ["plan", "batch"])
def test_grids_after_a_replay_behind_lorentz_berthelot(gpu_lib, form):
    """evaluate (captures), mls6_eval_lb, evaluate with the same arrays
    (replays): the grids are those of the last evaluation, bit for bit those
    of a plan that has seen no other call."""
    x, c, s, e = _system()
    pos4, pos, sg, ep = _dev(np.c_[x, c]), _dev(x), _dev(s), _dev(e)
    F = _dev(np.zeros((N, 3)))
    fresh = gpu_lib.Plan(BOX, N, A, H, LEVELS)
    fresh.evaluate(pos4)
    ref = _grids(gpu_lib, fresh)
    if form == "plan":
        plan = gpu_lib.Plan(BOX, N, A, H, LEVELS)
        call = lambda: plan.evaluate(pos4, forces=F)  # noqa: E731
    else:
        bt = gpu_lib.Batch([BOX], [N], A, H, LEVELS)

        class plan:  # noqa: N801
            handle = gpu_lib.mls6_batch_replica(bt.handle, 0)
        call = lambda: bt.evaluate(pos4, forces=F)  # noqa: E731
    call()
    _lb(gpu_lib, plan, pos, sg, ep)
    call()
    got = _grids(gpu_lib, plan)
    for k in ref:
        assert np.array_equal(got[k], ref[k]), k


@pytest.mark.parametrize("before", [False, True], ids=["first_call", "behind_evaluate"])
def test_grids_and_features_after_lorentz_berthelot(gpu_lib, orc, before):
    """After mls6_eval_lb the grids and the features are those of channel
    xi_6, also as the plan's first call.  FP64 grids: 1e-12 of the maximum,
    as for the other grids; features in FP32: u = 6e-8 of the values (a
    potential and its gradient, |.| <= 4 max |e|) through the FP32 output."""
    import torch

    from oracle import lb

    x, c, s, e = _system()
    xi6 = lb.xi(s, e)[6]
    plan = gpu_lib.Plan(BOX, N, A, H, LEVELS)
    if before:
        plan.evaluate(_dev(np.c_[x, c]))
    _lb(gpu_lib, plan, _dev(x), _dev(s), _dev(e))
    G = orc.grids(BOX, A, orc.grid_dims(BOX, H, LEVELS), LEVELS, x, xi6)
    for (k, w), got in _grids(gpu_lib, plan).items():
        assert np.abs(got - G[k - 1][w]).max() <= 1e-12 * np.abs(G[k - 1][w]).max(), (k, w)
    net = gpu_lib.MLP(seed=1)
    X = net.features(plan, "f32")
    other = gpu_lib.Plan(BOX, N, A, H, LEVELS)
    other.evaluate(_dev(np.c_[x, xi6]))
    Y = net.features(other, "f32")
    torch.cuda.synchronize()
    assert float((X - Y).abs().max()) <= 6e-8 * 4 * G[0][2].max()
