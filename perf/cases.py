"""The calls that a user of this framework has it do, over the range of sizes,
precisions and options that they are made with: how each is prepared, one pass
of it, the work that it cannot do without, and its results in 64 bits.

Kinds of case (``kind``):

``eval``     one energy/force evaluation of N atoms (``Plan.evaluate``), with
             or without the virial: the step of a molecular-dynamics program
``lb``       the same with Lorentz-Berthelot mixing (``mls6_eval_lb``)
``batch``    independent replicas of uneven size in one call (``Batch.evaluate``)
``learned``  an evaluation on a coarse grid and the learned correction of its
             forces (``Plan.evaluate``, ``MLP.apply``)
``train``    loss and gradient of that network on a training batch (``MLP.grad``)

Systems are liquids of hard-sphere separation 0.8 at density ``rho``: periodic
cubes (``aspect`` = Lz/Lx = 1, ``fill`` = 1) or slabs that fill the part
``fill`` of the box along z.  Energies and virials of the FP32 and mixed plans
are kept in FP32, the precision that they carry.
"""
import math

import numpy as np
import torch

from paper_1308_4005_gb300 import mls6

DMIN = 0.8        # least separation of two atoms
F64 = torch.float64


# ------------------------------------------------------------------- the cases

def _system(n, rho=0.85, aspect=1.0, fill=1.0, a=3.0, h=1.0, levels=0, precision="fp32", order=3,
            virial=True):
    return dict(n=n, rho=rho, aspect=aspect, fill=fill, a=a, h=h, levels=levels,
                precision=precision, order=order, virial=virial)


SLAB = dict(rho=0.8, aspect=3.0, fill=51.2 / 120.0)    # 40 x 40 x 120 box, 51.2 thick
WIDE = dict(rho=0.8, aspect=1.5, fill=204.8 / 240.0)   # 160 x 160 x 240 box, 204.8 thick


def listed():
    return [
        # the smallest system in use, in full precision: latency and launches
        dict(name="cube1000_fp64", kind="eval",
             **_system(1000, rho=1.0, a=2.5, h=0.99, levels=3, precision="fp64")),
        # a small replica of odd size, one step of a short simulation
        dict(name="slab3001_fp32", kind="eval", **_system(3001, a=2.5, **SLAB)),
        # the ordinary liquid slab with its virial (pressure coupling)
        dict(name="slab65536_fp32", kind="eval", **_system(65536, h=1.25, levels=4, **SLAB)),
        # a reference evaluation: full precision on an ordinary system, ragged size
        dict(name="cube98765_fp64", kind="eval", **_system(98765, precision="fp64")),
        # the quintic basis on an ordinary system
        dict(name="cube131072_order5", kind="eval", **_system(131072, h=1.5, order=5)),
        # forces at the equal-accuracy setting (a = 3.5, h = 1.5), no virial, odd size
        dict(name="cube349983_forces", kind="eval", **_system(349983, a=3.5, h=1.5, virial=False)),
        # the headline: a million atoms, tensor-core stencils, energy, forces, virial
        dict(name="cube1m_mixed", kind="eval",
             **_system(1 << 20, levels=5, precision="mixed")),
        # the largest: four million atoms on a coarse grid
        dict(name="slab4m_fp32", kind="eval", **_system(1 << 22, h=2.0, levels=5, **WIDE)),
        # mixtures: sizes and depths per atom, seven grid channels
        dict(name="lb_cube262144", kind="lb", **_system(262144, virial=False)),
        # replicas of uneven size, cubes and slabs in turn, in one call
        dict(name="batch40", kind="batch", replicas=40, n_min=2048, n_max=65536, sizes=13084008,
             rho=0.8, a=2.5, h=1.0, precision="fp32", virial=True),
        # a coarse evaluation corrected by the network
        dict(name="learned262144", kind="learned",
             **_system(262144, h=2.0, virial=False, **WIDE)),
        # the network's training: forward and backward over one batch
        dict(name="train65536", kind="train", n=65536),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval"] * 7 + ["lb", "batch", "learned", "train"])
    if kind == "train":
        return dict(kind=kind, n=_log_int(rng, 4096, 262144))
    if kind == "batch":
        return dict(kind=kind, replicas=rng.randint(4, 48), n_min=2048,
                    n_max=_log_int(rng, 8192, 65536), sizes=rng.randrange(1 << 30), rho=0.8,
                    a=round(rng.uniform(2.5, 3.5), 2), h=round(rng.uniform(1.0, 1.5), 2),
                    precision="fp32", virial=rng.random() < 0.5)
    precision = rng.choice(["fp64", "fp32", "fp32", "mixed", "mixed"]) if kind == "eval" else "fp32"
    order = 5 if precision == "fp32" and kind == "eval" and rng.random() < 0.2 else 3
    top = {"fp64": 131072, "mixed": 1 << 20}.get(precision, 1 << 20)
    top = 262144 if kind in ("lb", "learned") or order == 5 else top
    shape = rng.choice([{}, {}, SLAB, WIDE])
    h = 2.0 if kind == "learned" else round(rng.uniform(1.0, 2.0), 2)
    a = round(rng.uniform(2.5, 3.5), 2)
    if precision == "fp64":
        a, h = round(rng.uniform(2.5, 3.0), 2), max(h, 1.0)
    virial = kind == "eval" and rng.random() < 0.6
    return dict(kind=kind, **_system(_log_int(rng, 1000, top), a=a, h=h, precision=precision,
                                     order=order, virial=virial, **shape))


# ------------------------------------------------------------------ the systems

def _box(n, rho, aspect, fill):
    lx = (n / (rho * aspect * fill)) ** (1.0 / 3.0)
    return lx, lx, aspect * lx


def _replicas(case):
    """(n, aspect, fill) of a batch's replicas: sizes uniform in their
    logarithm, cubes and slabs in turn."""
    rng = np.random.default_rng(case["sizes"])
    n = np.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"]), case["replicas"]))
    return [(int(v), 1.0, 1.0) if r % 2 == 0 else (int(v), SLAB["aspect"], SLAB["fill"])
            for r, v in enumerate(n)]


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(gen, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, dtype=F64, device="cuda", generator=gen)


def _fluid(gen, n, size):
    """n random points of pairwise periodic separation >= DMIN in a box of the
    given size: trial points are drawn in batches and kept where no earlier
    point lies closer.  A grid of cells that hold at most one point each finds
    a point's neighbours."""
    size = torch.tensor(size, dtype=F64, device="cuda")
    cells = torch.ceil(size * (math.sqrt(3.0) / DMIN)).long()
    nx, ny, nz = cells.tolist()
    key_of = lambda c: c[..., 0] + nx * (c[..., 1] + ny * c[..., 2])  # noqa: E731
    grid = torch.full((nx * ny * nz,), -1, dtype=torch.long, device="cuda")
    reach = torch.arange(-2, 3, device="cuda")
    offsets = torch.cartesian_prod(reach, reach, reach)
    points = torch.empty((0, 3), dtype=F64, device="cuda")
    while points.shape[0] < n:
        have = points.shape[0]
        trial = size * torch.rand(2 * (n - have) + 1024, 3, dtype=F64, device="cuda", generator=gen)
        cell = torch.minimum((trial / size * cells).long(), cells - 1)
        free = grid[key_of(cell)] < 0
        trial, cell = trial[free], cell[free]
        ids = torch.arange(have, have + trial.shape[0], device="cuda")
        key = key_of(cell)
        grid.scatter_reduce_(0, key, ids, "amin", include_self=False)
        everyone = torch.cat([points, trial])
        good = grid[key] == ids
        for at in good.nonzero().squeeze(1).split(1 << 17):
            near = grid[key_of((cell[at, None] + offsets) % cells)]
            d = everyone[near.clamp(min=0)] - trial[at, None]
            d -= size * torch.round(d / size)
            close = (d.square().sum(-1) < DMIN * DMIN) & (near >= 0) & (near < ids[at, None])
            good[at[close.any(1)]] = False
        grid[key] = -1
        kept = good.nonzero().squeeze(1)[: n - have]
        grid[key[kept]] = torch.arange(have, have + kept.shape[0], device="cuda")
        points = torch.cat([points, trial[kept]])
    return points


def _atoms(gen, n, rho, aspect, fill):
    """Box, positions and C6-type coefficients c = sqrt(C6), C6 in [0.5, 1.5]."""
    box = _box(n, rho, aspect, fill)
    x = _fluid(gen, n, (box[0], box[1], fill * box[2]))
    x[:, 2] += 0.5 * (1.0 - fill) * box[2]
    return box, x, torch.sqrt(_uniform(gen, 0.5, 1.5, n))


def _dtype(case):
    return F64 if case["precision"] == "fp64" else torch.float32


def _inputs(case, seed):
    """(box, arrays of the plan's precision) that a pass reads."""
    gen, dt = _generator(seed), _dtype(case)
    box, x, c = _atoms(gen, case["n"], case["rho"], case["aspect"], case["fill"])
    if case["kind"] == "lb":
        return box, x.to(dt), _uniform(gen, 0.85, 1.15, case["n"]).to(dt), _uniform(
            gen, 0.5, 1.5, case["n"]).to(dt)
    return box, torch.cat([x, c[:, None]], 1).to(dt)


def _batch_inputs(case, seed):
    gen, boxes, rows, counts = _generator(seed), [], [], []
    for n, aspect, fill in _replicas(case):
        box, x, c = _atoms(gen, n, case["rho"], aspect, fill)
        boxes.append(box)
        counts.append(n)
        rows.append(torch.cat([x, c[:, None]], 1))
    return boxes, counts, torch.cat(rows).to(_dtype(case))


def _network(seed):
    """Weights of the 128-64-64-64-8 network as one vector (Glorot uniform,
    zero biases), its feature scale and its output scale."""
    rng = np.random.default_rng(seed)
    parts = []
    for i, o in ((128, 64), (64, 64), (64, 64), (64, 8)):
        lim = math.sqrt(6.0 / (i + o))
        parts += [rng.uniform(-lim, lim, i * o), np.zeros(o)]
    scale = np.ones(128)
    scale[0:108:4] = 0.2    # potentials are a few units, gradients and angles about one
    return np.concatenate(parts).astype(np.float32), scale.astype(np.float32), 0.05


def _training_batch(case, seed):
    gen = _generator(seed)
    X = torch.randn(case["n"], 128, device="cuda", generator=gen).to(torch.bfloat16)
    return X, torch.randn(case["n"], 3, device="cuda", generator=gen)


# --------------------------------------------------------------- the measured pass

def _plan(case, box):
    return mls6.Plan(box, case["n"], case["a"], case["h"], case["levels"],
                     precision=case["precision"], order=case["order"])


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "train":
        s["X"], s["T"] = _training_batch(case, seed)
    elif kind == "batch":
        boxes, counts, s["pos"] = _batch_inputs(case, seed)
        s["batch"] = mls6.Batch(boxes, counts, case["a"], case["h"], precision=case["precision"])
        s["F"] = torch.empty((sum(counts), 3), dtype=_dtype(case), device="cuda")
    else:
        box, s["pos"], *s["species"] = _inputs(case, seed)
        s["plan"] = _plan(case, box)
        s["F"] = torch.empty((case["n"], 3), dtype=_dtype(case), device="cuda")
        s["E"] = torch.zeros(1, dtype=F64, device="cuda")
    if kind in ("learned", "train"):
        weights, scale, out_scale = _network(seed)
        s["mlp"] = mls6.MLP(0)
        s["mlp"].set_params(weights)
        s["mlp"].set_norm(np.zeros(128), scale, out_scale)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "train":
        loss, grad = s["mlp"].grad(s["X"], s["T"])
        return {"loss": loss, "grad": grad}
    if kind == "batch":
        r = s["batch"].evaluate(s["pos"], virial=case["virial"], forces=s["F"])
        dt = s["F"].dtype
        out = {"E": r["E"].to(dt), "F": r["F"]}
        if case["virial"]:
            out["W"] = r["W"].to(dt)
        return out
    if kind == "lb":
        sigma, eps = s["species"]
        rc = mls6.mls6_eval_lb(s["plan"].handle, s["pos"].data_ptr(), sigma.data_ptr(),
                               eps.data_ptr(), s["F"].data_ptr(), s["E"].data_ptr())
        if rc:
            raise mls6.MLS6Error(rc, "mls6_eval_lb")
        return {"E": s["E"].to(s["F"].dtype), "F": s["F"]}
    r = s["plan"].evaluate(s["pos"], virial=case["virial"], forces=s["F"])
    if kind == "learned":
        s["mlp"].apply(s["plan"], r["F"])
    ew = r["out"].to(s["F"].dtype)
    out = {"E": ew[:1], "F": r["F"]}
    if case["virial"]:
        out["W"] = ew[1:]
    return out


# ------------------------------------------------------------------------- the work

def _work_atoms(case, n, aspect, fill):
    """One evaluation: atoms in, forces out; each pair inside the cutoff once
    (separation, g_0 and its derivative, both atoms' sums), the basis sums of
    the transfers, and the level stencils (the grids stay on the chip or in
    cache)."""
    box = _box(n, case["rho"], aspect, fill)
    a, h, order = case["a"], case["h"], case.get("order", 3)
    word = 8 if case["precision"] == "fp64" else 4
    virial = case["virial"]
    pairs = 0.5 * n * case["rho"] * 4.0 / 3.0 * math.pi * a ** 3
    nodes = box[0] * box[1] * box[2] / h ** 3
    taps = 4.0 / 3.0 * math.pi * (2.0 * a / h) ** 3
    per_node = 8.0 / 7.0 * taps * (14.0 if virial else 2.0)
    transfer = n * (order + 1) ** 3 * (2.0 + 8.0)
    return {"bytes": n * 7.0 * word,
            "flops": pairs * (60.0 if virial else 48.0) + nodes * per_node + transfer}


def work(case):
    if case["kind"] == "train":
        macs = 128 * 64 + 2 * 64 * 64 + 64 * 8
        return {"bytes": case["n"] * (256.0 + 12.0), "flops": case["n"] * macs * 6.0}
    if case["kind"] == "batch":
        each = [_work_atoms(case, *r) for r in _replicas(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    w = _work_atoms(case, case["n"], case["aspect"], case["fill"])
    n = case["n"]
    if case["kind"] == "lb":  # seven grid channels
        pairs = 0.5 * n * case["rho"] * 4.0 / 3.0 * math.pi * case["a"] ** 3 * 48.0
        return {"bytes": n * 8.0 * 4, "flops": pairs + 7.0 * (w["flops"] - pairs)}
    if case["kind"] == "learned":  # 27 interpolations (separable) and the network
        macs = 128 * 64 + 2 * 64 * 64 + 64 * 8
        return {"bytes": w["bytes"], "flops": w["flops"] + n * (2.0 * macs + 4.0 * 1500)}
    return w


# ------------------------------------------------------- the same results in 64 bits

def _grid_dims(box, h, levels):
    """Finest grid: per axis the multiple of 2^(levels-1) nearest to L/h (ties
    to the finer grid); levels = 0: the most that leave >= 4 coarsest nodes."""
    def dims(l):
        m = 1 << (l - 1)
        out = []
        for L in box:
            u = L / h / m
            lo = math.floor(u)
            out.append(max(1, lo if u - lo < lo + 1 - u else lo + 1) * m)
        return out
    if levels == 0:
        levels = 1
        while levels < 12 and min(dims(levels + 1)) >> levels >= 4:
            levels += 1
    return dims(levels), levels


def _gamma(s, r):
    """s^-6 gamma(r/s) and its derivative over r, gamma = 15/8 - 5/4 p^12 +
    3/8 p^24 inside, p^-6 outside."""
    p2 = (r / s).square()
    q2 = p2.clamp(min=1.0)
    u = p2.clamp(max=1.0) ** 6
    g = torch.where(p2 < 1.0, 1.875 - 1.25 * u + 0.375 * u * u, q2 ** -3)
    d = torch.where(p2 < 1.0, p2.clamp(max=1.0) ** 5 * (-15.0 + 9.0 * u), -6.0 * q2 ** -4)
    return g / s ** 6, d / s ** 8


def _pairs(box, a, x, w, species):
    """Local part: per atom sum_j C_ij g_0, sum_j C_ij g_0'/r d, and the six
    virial sums.  species: C_ij = w_i w_j ((s_i + s_j)/2)^6, else w_i w_j."""
    n = x.shape[0]
    L = torch.tensor(box, dtype=F64, device="cuda")
    nc = [max(1, int(l // a)) for l in box]
    reach = [math.ceil(a / (l / m) - 1e-12) for l, m in zip(box, nc)]
    ncell = nc[0] * nc[1] * nc[2]
    count = torch.tensor(nc, device="cuda")
    cell = torch.minimum((x / L * count).long().clamp(min=0), count - 1)
    key = cell[:, 0] + nc[0] * (cell[:, 1] + nc[1] * cell[:, 2])
    order = torch.argsort(key, stable=True)
    pop = torch.bincount(key, minlength=ncell)
    cap = int(pop.max())
    slot = torch.arange(n, device="cuda") - (pop.cumsum(0) - pop)[key[order]]
    row = key[order] * cap + slot
    rec = torch.cat([x, w[:, None], (species if species is not None else w)[:, None]], 1)
    P = torch.zeros(ncell * cap, 5, dtype=F64, device="cuda")
    P[:, :3] = math.inf
    P[row] = rec[order]
    P = P.reshape(ncell, cap, 5)
    ids = torch.arange(ncell, device="cuda")
    at = torch.stack([ids % nc[0], ids // nc[0] % nc[1], ids // (nc[0] * nc[1])], 1)
    S = torch.zeros(ncell, cap, 4, dtype=F64, device="cuda")
    W = torch.zeros(6, dtype=F64, device="cuda")
    for part in ids.split(max(1, (1 << 24) // (cap * cap))):
        A = P[part][:, :, None, :]
        for oz in range(-reach[2], reach[2] + 1):
            for oy in range(-reach[1], reach[1] + 1):
                for ox in range(-reach[0], reach[0] + 1):
                    to = at[part] + torch.tensor([ox, oy, oz], device="cuda")
                    image = torch.div(to, count, rounding_mode="floor")
                    to = to - image * count
                    B = P[to[:, 0] + nc[0] * (to[:, 1] + nc[1] * to[:, 2])][:, None, :, :]
                    d = (B[..., :3] - A[..., :3]) + (image * L)[:, None, None, :]
                    r2 = d.square().sum(-1)
                    hit = (r2 < a * a) & (r2 > 0.0)
                    r2 = torch.where(hit, r2, a * a)
                    C = A[..., 3] * B[..., 3]
                    if species is not None:
                        C = C * (0.5 * (A[..., 4] + B[..., 4])) ** 6
                    C = torch.where(hit, C, 0.0)
                    g, dg = _gamma(a, r2.sqrt())
                    d = torch.where(hit[..., None], d, 0.0)
                    cg = C * (-6.0 * r2 ** -4 - dg)
                    S[part, :, 0] += (C * (r2 ** -3 - g)).sum(2)
                    S[part, :, 1:] += (cg[..., None] * d).sum(2)
                    for k, (p, q) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
                        W[k] += 0.5 * (cg * d[..., p] * d[..., q]).sum()
    out = torch.empty(n, 4, dtype=F64, device="cuda")
    out[order] = S.reshape(-1, 4)[row]
    return out[:, 0], out[:, 1:], W


def _basis(t, order):
    """Nodal basis Phi and its derivative at t: the cubic Hermite interpolant
    or the C^1 quintic."""
    u, s = t.abs(), torch.sign(t)
    if order == 3:
        pieces = [np.poly1d([1.5, -2.5, 0.0, 1.0]),
                  -0.5 * np.poly1d([1, -1.0]) * np.poly1d([-1, 2.0]) ** 2]
    else:
        f = [np.poly1d([1, -float(r)]) for r in range(5)]
        pieces = [np.poly1d([-1, 0, 1.0]) * np.poly1d([-1, 2.0]) * np.poly1d([-5, 3.0, 6.0]) / 12.0,
                  f[1] * f[2] * f[3] * np.poly1d([5, -9.0, -4.0]) / 24.0,
                  -1.0 * f[1] * f[2] * f[3] * f[3] * f[4] / 24.0]
    v, dv = torch.zeros_like(u), torch.zeros_like(u)
    for k, p in enumerate(pieces):
        inside = (u >= k) & (u < k + 1)
        for out, q in ((v, p), (dv, p.deriv())):
            acc = torch.zeros_like(u)
            for c in q.coeffs:
                acc = acc * u + float(c)
            out += torch.where(inside, acc, 0.0)
    return v, dv * s


class _Support:
    """Weights, derivatives and node indices of the atoms' supports."""

    def __init__(self, box, n, x, order):
        half, axes = (order + 1) // 2, []
        for d in range(3):
            h = box[d] / n[d]
            u = x[:, d] / h
            base = torch.floor(u)
            ax = []
            for k in range(1 - half, half + 1):
                v, dv = _basis(u - (base + k), order)
                ax.append((torch.remainder(base.long() + k, n[d]), v, dv / h, base.long() + k))
            axes.append(ax)
        self.n, self.axes = n, axes

    def spread(self, w):
        q = torch.zeros(self.n[0] * self.n[1] * self.n[2], dtype=F64, device="cuda")
        for iz, vz, _, _ in self.axes[2]:
            for iy, vy, _, _ in self.axes[1]:
                for ix, vx, _, _ in self.axes[0]:
                    q.index_add_(0, ix + self.n[0] * (iy + self.n[1] * iz), w * vx * vy * vz)
        return q.reshape(self.n[2], self.n[1], self.n[0])

    def gather(self, e, shift=(0, 0, 0)):
        """Potential and gradient at the atoms (moved by whole nodes)."""
        e, n = e.reshape(-1), self.n
        out = torch.zeros(self.axes[0][0][0].shape[0], 4, dtype=F64, device="cuda")
        for jz, vz, dz, rz in self.axes[2]:
            for jy, vy, dy, ry in self.axes[1]:
                for jx, vx, dx, rx in self.axes[0]:
                    i = [torch.remainder(r + s, m) for r, s, m in zip((rx, ry, rz), shift, n)]
                    v = e[i[0] + n[0] * (i[1] + n[1] * i[2])]
                    out[:, 0] += vx * vy * vz * v
                    out[:, 1] += dx * vy * vz * v
                    out[:, 2] += vx * dy * vz * v
                    out[:, 3] += vx * vy * dz * v
        return out


def _half_weights(order):
    t = torch.arange(-order, order + 1, dtype=F64, device="cuda") / 2
    return list(zip(range(-order, order + 1), _basis(t, order)[0].tolist()))


def _restrict(q, order):
    for axis in range(3):
        q = sum(v * torch.roll(q, -o, axis) for o, v in _half_weights(order) if v)
        q = q.index_select(axis, torch.arange(0, q.shape[axis], 2, device="cuda"))
    return q


def _prolong(e, order):
    for axis in range(3):
        shape = list(e.shape)
        shape[axis] *= 2
        up = torch.zeros(shape, dtype=F64, device="cuda")
        up.index_copy_(axis, torch.arange(0, shape[axis], 2, device="cuda"), e)
        e = sum(v * torch.roll(up, o, axis) for o, v in _half_weights(order) if v)
    return e


def _mesh(counts):
    r = [torch.arange(-m, m + 1, device="cuda") for m in counts]
    return torch.cartesian_prod(*r)


def _level_kernels(n, h, a):
    """g_1 and the six G r_p r_q of the taps inside 2a, folded onto the grid."""
    m = _mesh([math.ceil(2.0 * a / v) for v in h])
    r3 = m * torch.tensor(h, dtype=F64, device="cuda")
    r = r3.square().sum(1).sqrt()
    m, r3, r = m[r < 2.0 * a], r3[r < 2.0 * a], r[r < 2.0 * a]
    (g1, d1), (g2, d2) = _gamma(a, r), _gamma(2.0 * a, r)
    G = torch.where(r > 0, d1 - d2, 0.0)
    at = torch.remainder(m, torch.tensor(n, device="cuda"))
    at = at[:, 0] + n[0] * (at[:, 1] + n[1] * at[:, 2])
    fold = lambda v: torch.zeros(n[0] * n[1] * n[2], dtype=F64, device="cuda").index_add_(  # noqa: E731
        0, at, v).reshape(n[2], n[1], n[0])
    return [fold(g1 - g2)] + [fold(G * r3[:, p] * r3[:, q])
                              for p, q in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]


def _coarsest_kernels(box, n, s):
    """Lattice sums over all images of s^-6 gamma(r/s) and of its virial terms
    at the coarsest grid's offsets: Ewald summation of r^-6 (a Gaussian-damped
    sum over images, the smooth remainder over reciprocal vectors)."""
    V = box[0] * box[1] * box[2]
    cut = max(3.8 * V ** (1.0 / 3.0), s)
    beta = 7.5 / cut
    L = torch.tensor(box, dtype=F64, device="cuda")
    X = torch.cartesian_prod(*[torch.arange(m, device="cuda", dtype=F64) * l / m
                               for m, l in zip(n[::-1], box[::-1])]).flip(1)
    out = torch.zeros(7, X.shape[0], dtype=F64, device="cuda")
    six = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))
    for image in _mesh([math.ceil(cut / l) + 1 for l in box]).split(512):
        d = X[None] + (image * L)[:, None]
        r = d.square().sum(2).sqrt()
        x = beta * beta * r * r
        far = r >= s
        rf = torch.where(far, r, s)
        xf = beta * beta * rf * rf
        Q = torch.exp(-xf) * (1.0 + xf + 0.5 * xf * xf)
        f_far, p_far = Q / rf ** 6, -6.0 * Q / rf ** 8 - beta ** 2 * xf ** 2 * torch.exp(-xf) / rf ** 6
        # inside: s^-6 gamma minus r^-6 P(3, x), the latter by its series in x
        xn, rn = torch.where(far, 0.0, x), torch.where(far, 0.0, r)
        s3, s4, power = torch.zeros_like(xn), torch.zeros_like(xn), torch.ones_like(xn)
        for k in range(60):
            s3 = s3 + power / float(math.factorial(k + 3))
            s4 = s4 + power / float(math.factorial(k + 4))
            power = power * xn
        g, dg = _gamma(s, rn)
        f_near = g - beta ** 6 * torch.exp(-xn) * s3
        p_near = dg + 6.0 * beta ** 8 * torch.exp(-xn) * s4
        f = torch.where(r < cut, torch.where(far, f_far, f_near), 0.0)
        p = torch.where(r < cut, torch.where(far, p_far, p_near), 0.0)
        out[0] += f.sum(0)
        for k, (i, j) in enumerate(six):
            out[1 + k] += (p * d[..., i] * d[..., j]).sum(0)
    top = 13.0 * beta
    k3 = _mesh([math.ceil(top * l / (2.0 * math.pi)) for l in box]) * (2.0 * math.pi / L)
    k3 = k3[k3.square().sum(1).sqrt() <= top]
    k = k3.square().sum(1).sqrt()
    b = k / (2.0 * beta)
    unit = math.pi ** 1.5 * beta ** 3 / 3.0
    S = unit * ((1.0 - 2.0 * b * b) * torch.exp(-b * b) + 2.0 * math.sqrt(math.pi) * b ** 3 * torch.erfc(b))
    dS = unit * 6.0 * b * (math.sqrt(math.pi) * b * torch.erfc(b) - torch.exp(-b * b)) / (2.0 * beta)
    dS = torch.where(k > 0, dS / k.clamp(min=1e-300), 0.0)
    cos = torch.cos(X @ k3.T)
    out[0] += cos @ S / V
    for c, (i, j) in enumerate(six):
        out[1 + c] += cos @ ((-S if i == j else torch.zeros_like(S)) - dS * k3[:, i] * k3[:, j]) / V
    return [v.reshape(n[2], n[1], n[0]) for v in out]


def _potential(q, kernels, scale):
    """Circular convolution with the first kernel, and half the bilinear forms
    of the others with q."""
    fq = torch.fft.rfftn(q)
    conv = lambda K: torch.fft.irfftn(fq * torch.fft.rfftn(K), s=q.shape) * scale  # noqa: E731
    return conv(kernels[0]), torch.stack([0.5 * (q * conv(K)).sum() for K in kernels[1:]])


class _Method:
    """The multilevel method in 64 bits on one system."""

    def __init__(self, case, box, x):
        self.case, self.box = case, box
        L = torch.tensor(box, dtype=F64, device="cuda")
        self.x = x - torch.floor(x / L) * L
        self.n, self.levels = _grid_dims(box, case["h"], case["levels"] if "levels" in case else 0)
        self.order = case.get("order", 3)
        self.support = _Support(box, self.n, self.x, self.order)
        h = [l / m for l, m in zip(box, self.n)]
        a, top = case["a"], self.levels - 1
        self.kernels = [_level_kernels([m >> k for m in self.n], h, a) for k in range(top)]
        self.kernels.append(_coarsest_kernels(box, [m >> top for m in self.n], a * 2.0 ** top))
        self.self_term = 1.875 / a ** 6

    def grid(self, w):
        """Total potential on the finest grid and the grid part of the virial."""
        q, W, parts = self.support.spread(w), 0.0, []
        for k, kernels in enumerate(self.kernels):
            if k:
                q = _restrict(q, self.order)
            e, v = _potential(q, kernels, 1.0 if k == self.levels - 1 else 2.0 ** (-6 * k))
            parts.append(e)
            W = W + v
        e = parts[-1]
        for finer in parts[-2::-1]:
            e = finer + _prolong(e, self.order)
        return e, W

    def evaluate(self, c):
        """E, F, W with C_ij = c_i c_j, and the finest grid's potential."""
        e0, f0, W0 = _pairs(self.box, self.case["a"], self.x, c, None)
        e, W = self.grid(c)
        at = self.support.gather(e)
        E = -0.5 * (e0 + c * at[:, 0]).sum() + 0.5 * self.self_term * c.square().sum()
        return E, -f0 + c[:, None] * at[:, 1:], W0 + W, e

    def evaluate_lb(self, sigma, eps):
        root = torch.sqrt(2.0 * eps)
        e0, f0, _ = _pairs(self.box, self.case["a"], self.x, root, sigma)
        xi = [math.sqrt(math.comb(6, m)) / 8.0 * sigma ** m * root for m in range(7)]
        E, F = -0.5 * e0.sum(), -f0
        for m in range(7):
            at = self.support.gather(self.grid(xi[m])[0])
            E = E - 0.5 * (xi[6 - m] * at[:, 0]).sum()
            F = F + xi[6 - m][:, None] * at[:, 1:]
        return E + 0.5 * self.self_term * (2.0 * eps * sigma ** 6).sum(), F


def _layers(weights):
    at, out = 0, []
    for i, o in ((128, 64), (64, 64), (64, 64), (64, 8)):
        out.append((weights[at:at + i * o].reshape(i, o), weights[at + i * o:at + i * o + o]))
        at += i * o + o
    return out


def _forward(weights, X):
    for k, (W, b) in enumerate(_layers(weights)):
        X = X @ W + b
        X = torch.tanh(X) if k < 3 else X
    return X


def exact(case, seed):
    kind = case["kind"]
    if kind in ("learned", "train"):
        weights, scale, out_scale = _network(seed)
        weights = torch.tensor(weights, dtype=F64, device="cuda")
    if kind == "train":
        X, T = _training_batch(case, seed)
        weights.requires_grad_()
        loss = (_forward(weights, X.double())[:, :3] - T.double()).square().sum() / case["n"]
        loss.backward()
        return {"loss": float(loss.detach()), "grad": weights.grad}
    if kind == "batch":
        boxes, counts, pos = _batch_inputs(case, seed)
        each = [_Method(case, box, p[:, :3].double()).evaluate(p[:, 3].double())
                for box, p in zip(boxes, pos.split(counts))]
        out = {"E": torch.stack([e[0] for e in each]), "F": torch.cat([e[1] for e in each])}
        if case["virial"]:
            out["W"] = torch.stack([e[2] for e in each])
        return out
    box, pos, *species = _inputs(case, seed)
    method = _Method(case, box, pos[:, :3].double())
    if kind == "lb":
        E, F = method.evaluate_lb(*[v.double() for v in species])
        return {"E": E.reshape(1), "F": F}
    c = pos[:, 3].double()
    E, F, W, e1 = method.evaluate(c)
    if kind == "learned":
        cols = []
        for dz in (-1, 0, 1):
            for dy in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    cols.append(method.support.gather(e1, (dx, dy, dz)))
        for d in range(3):
            t = 2.0 * math.pi * torch.frac(method.x[:, d] * (method.n[d] / box[d]))
            cols += [torch.sin(t)[:, None], torch.cos(t)[:, None]]
        X = torch.nn.functional.pad(torch.cat(cols, 1), (0, 14))
        X = X * torch.tensor(scale, dtype=F64, device="cuda")
        F = F + c[:, None] * out_scale * _forward(weights, X)[:, :3]
    out = {"E": E.reshape(1), "F": F}
    if case["virial"]:
        out["W"] = W
    return out
