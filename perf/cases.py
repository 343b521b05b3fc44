"""Performance cases of the QLA framework: what its users run, as callables.

Each case is one call sequence through the public entry points (``Grid``,
``Batch``, ``Grid3``, ``Surrogate``, ``features``), from the 256^2 lattices of
the parity workload and the surrogate to the 16384^2 bubble.  ``prepare``
builds what a program holds before the call, ``run`` makes the call,
``work`` states what it cannot do without and ``exact`` computes the same
outputs with plain torch operations in 64 bits.

``work``: a lattice whose two buffers of state exceed the 126 MB L2 is read
and written once per step; a smaller one once per call.  Operations count six
per 2 x 2 rotation (four products, two sums).
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2604_21128_gb300 import qla, surrogate

L2_BYTES = 126e6
EXACT_SITE_STEPS = 8e9      # more than this takes plain torch too long


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # The parity workload, whole: a packet is launched at the 256^2
        # ellipse, 400 FP64 steps, energy and state read back on the host.
        dict(name="scatter_256_fp64", kind="lattice", nx=256, ny=256, precision="fp64", te=True,
             steps=400, out="state"),
        # One window of the surrogate's data and of its fallback: K = 32 FP32
        # steps of a 256^2 lattice, the energy check and the features.
        dict(name="window_256_fp32", kind="lattice", nx=256, ny=256, precision="fp32", te=True,
             steps=32, out="features"),
        # A lattice whose sides are no multiple of anything.
        dict(name="odd_1023x769_fp32", kind="lattice", nx=1023, ny=769, precision="fp32", te=True,
             steps=20, out="box"),
        # All six amplitudes, for fields that are not E_z polarised.
        dict(name="six_2048_fp32", kind="lattice", nx=2048, ny=2048, precision="fp32", te=False,
             steps=50, out="box"),
        # A diagonal index tensor, six amplitudes.
        dict(name="tensor_1024_fp32", kind="lattice", nx=1024, ny=1024, precision="fp32", te=False,
             tensor=True, steps=50, out="box"),
        # FP64 accuracy on a production lattice: double-single steps.
        dict(name="ds_4096_fp64", kind="lattice", nx=4096, ny=4096, precision="fp64", te=True,
             double_single=True, steps=20, out="box"),
        # The two large workloads, 100 steps between energy readings.
        dict(name="ellipse_8192_fp32", kind="lattice", nx=8192, ny=8192, precision="fp32", te=True,
             steps=100, out="box"),
        dict(name="bubble_16384_fp32", kind="lattice", nx=16384, ny=16384, precision="fp32",
             te=True, bubble=True, steps=100, out="box"),
        # A sweep of uneven lattices in one batch, energies on the way.
        dict(name="batch_24_fp32", kind="batch", count=24, lo=512, hi=2048, steps=100, every=50),
        # Three dimensions: a run between two checkpoints.
        dict(name="cube_192_fp32", kind="cube", nx=192, ny=160, nz=128, precision="fp32",
             steps=500),
        # The surrogate's network: inference on a batch, and its training.
        dict(name="forward_256_b8", kind="forward", h=256, w=256, batch=8),
        dict(name="train_256_b8", kind="train", h=256, w=256, batch=8, steps=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice"] * 6 + ["batch", "cube", "forward", "train"])
    if kind == "lattice":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        te = rng.random() < 0.7
        tensor = not te and rng.random() < 0.3
        ds = precision == "fp64" and not tensor and rng.random() < 0.5
        top = (8192 if te else 4096) if precision == "fp32" else 4096 if ds else 2048
        top = 2048 if tensor else top
        nx, ny = _log(rng, 128, top), _log(rng, 96, top)
        if rng.random() < 0.6 and not ds:
            nx += -nx % 4
        elif ds:
            nx += nx % 2
        elif nx * ny > 1 << 21:       # odd sides occur on small lattices
            nx += -nx % 4
        steps = max(4, min(200, _log(rng, 10, 200), int(2e9 / (nx * ny))))
        return dict(kind="lattice", nx=nx, ny=ny, precision=precision, te=te, tensor=tensor,
                    double_single=ds, bubble=rng.random() < 0.3, steps=steps, out="box")
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(2, 32), lo=128, hi=_log(rng, 256, 2048),
                    steps=5 * rng.randint(2, 16), every=5)
    if kind == "cube":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        ds = precision == "fp64" and rng.random() < 0.5
        top = 192 if precision == "fp32" else 128
        nx, ny, nz = (_log(rng, 64, top) for _ in range(3))
        return dict(kind="cube", nx=nx + nx % 2, ny=ny, nz=nz, precision=precision,
                    double_single=ds, steps=rng.randint(20, 200))
    h, w = 16 * rng.randint(4, 16), 16 * rng.randint(4, 16)
    if kind == "forward":
        return dict(kind="forward", h=h, w=w, batch=rng.randint(1, 8))
    return dict(kind="train", h=h, w=w, batch=rng.randint(1, 8), steps=rng.randint(1, 4))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _min_image(d, L):
    return torch.remainder(d + 0.5 * L, L) - 0.5 * L


def _axis(n, centre):
    return _min_image(torch.arange(n, dtype=torch.float64, device="cuda") - centre, n)


def _ellipsoid(shape, semi, centre, angle, n_in, n_out, edge):
    """Index map of a smooth ellipse or ellipsoid, rotated by ``angle`` in the
    (x, y) plane; shape (ny, nx) or (nz, ny, nx), the other tuples x first."""
    out = torch.empty(shape, dtype=torch.float64, device="cuda")
    ca, sa = math.cos(angle), math.sin(angle)
    dims = len(shape)
    d = [_axis(shape[dims - 1 - k], centre[k]) for k in range(dims)]
    block = max(1, (1 << 25) // (out[0].numel()))
    for r0 in range(0, shape[0], block):          # blocks of the slowest axis
        d_slow = d[-1][r0:r0 + block]
        x = d[0].view([1] * (dims - 1) + [-1])
        y = d_slow.view(-1, 1) if dims == 2 else d[1].view(1, -1, 1)
        part = [x * ca + y * sa, y * ca - x * sa] + ([d_slow.view(-1, 1, 1)] if dims == 3 else [])
        r2 = sum((p / s) ** 2 for p, s in zip(part, semi))
        g2 = sum((p / s ** 2) ** 2 for p, s in zip(part, semi))
        rho = r2.sqrt()
        dist = torch.where(r2 > 0, (rho - 1) * rho / g2.clamp_min(1e-30).sqrt(),
                           torch.full_like(rho, -min(semi)))
        out[r0:r0 + block] = n_out + (n_in - n_out) * 0.5 * (1 - torch.tanh(dist / edge))
    return out


def _scene(rng, nx, ny, bubble):
    """Medium and packet of a 2D scattering run: an ellipse of 5 to 25% of the
    side in vacuum, or a vacuum bubble in n = 2, and a packet aimed at it."""
    side = min(nx, ny)
    angle, phi = rng.uniform(0, math.pi), rng.uniform(0, 2 * math.pi)
    medium = dict(semi=(rng.uniform(0.05, 0.25) * side, rng.uniform(0.05, 0.25) * side),
                  centre=(nx / 2 + rng.uniform(-0.05, 0.05) * nx,
                          ny / 2 + rng.uniform(-0.05, 0.05) * ny),
                  angle=angle, n_in=1.0 if bubble else rng.uniform(1.5, 4.0),
                  n_out=2.0 if bubble else 1.0, edge=3.0 if side < 4096 else 8.0)
    packet = dict(x0=nx / 2 - 0.3 * side * math.cos(phi), y0=ny / 2 - 0.3 * side * math.sin(phi),
                  angle=phi, k0=rng.uniform(0.1, 0.4), width=side / 16,
                  transverse_width=side / 8)
    return medium, packet


def _lattice_inputs(case, seed):
    rng = np.random.default_rng(seed)
    nx, ny = case["nx"], case["ny"]
    medium, packet = _scene(rng, nx, ny, case.get("bubble", False))
    indices = [medium["n_in"]]
    if case.get("tensor"):
        indices = [rng.uniform(1.5, 4.0) for _ in range(3)]
    n = [_ellipsoid((ny, nx), **dict(medium, n_in=v)) for v in indices]
    return (torch.stack(n) if case.get("tensor") else n[0]), packet


def _lattice_state(case, n, packet):
    return _six(n[2], n[0], n[1], packet) if case.get("tensor") else _six(n, n, n, packet)


def _batch_inputs(case, seed):
    sides = np.random.default_rng(case["count"] * 7919 + case["hi"])
    rng = np.random.default_rng(seed)
    grids = []
    for _ in range(case["count"]):
        side = int(round(sides.uniform(case["lo"], case["hi"]) / 4)) * 4
        medium, packet = _scene(rng, side, side, False)
        grids.append((side, medium, packet))
    return grids


def _cube_inputs(case, seed):
    rng = np.random.default_rng(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    side = min(nx, ny, nz)
    n = _ellipsoid((nz, ny, nx), semi=tuple(rng.uniform(0.1, 0.25) * side for _ in range(3)),
                   centre=(nx / 2, ny / 2, nz / 2), angle=rng.uniform(0, math.pi),
                   n_in=rng.uniform(1.5, 3.0), n_out=1.0, edge=3.0)
    phi = rng.uniform(0, 2 * math.pi)
    packet = dict(x0=nx / 2 - 0.3 * side * math.cos(phi), y0=ny / 2 - 0.3 * side * math.sin(phi),
                  angle=phi, k0=rng.uniform(0.2, 0.4), width=side / 10,
                  transverse_width=side / 6)
    return n, packet


def _packet(n, x0, y0, angle, k0, width, transverse_width):
    """(q2, q3, q4) of the Gaussian E_z packet on the medium n (ny, nx)."""
    ny, nx = n.shape[-2:]
    dx, dy = _axis(nx, x0).view(1, -1), _axis(ny, y0).view(-1, 1)
    c, s = math.cos(angle), math.sin(angle)
    xi, eta = dx * c + dy * s, dy * c - dx * s
    ez = torch.exp(-(xi / width) ** 2 - (eta / transverse_width) ** 2) * torch.cos(k0 * xi)
    q2 = n * ez
    return q2, s * q2, -c * q2


def _six(n, n_x, n_y, packet):
    """All six amplitudes: the E_z packet and, polarised in the plane, a B_z
    packet of the same shape (E perpendicular to the direction of travel)."""
    q2, q3, q4 = _packet(n, **packet)
    if n.dim() == 3:
        q2, q3, q4 = (v.expand(n.shape) for v in (q2, q3, q4))
    ez, c, s = q2 / n, math.cos(packet["angle"]), math.sin(packet["angle"])
    return torch.stack([-s * n_x * ez, c * n_y * ez, q2, q3, q4, q2])


def _gradient(n, dim):
    return 0.5 * (torch.roll(n, -1, dim) - torch.roll(n, 1, dim))


def _features(q, n):
    return torch.stack([*q, n - 1.5, 4 * _gradient(n, 1), 4 * _gradient(n, 0)], dim=-1)


CONVS = [(6, 32), (32, 64), (64, 128), (128, 256), (256, 256), (256, 256), (256, 128), (128, 64),
         (64, 32), (32, 3)]


def _network_inputs(case, seed):
    """Weights (He scaled, flat, FP32), features and targets of a batch."""
    gen = torch.Generator().manual_seed(seed)
    flat = []
    for cin, cout in CONVS:
        w = torch.randn(cout * cin * 9, generator=gen) * math.sqrt(2.0 / (9 * cin))
        flat += [w * (0.1 if cout == 3 else 0.7), 0.01 * torch.randn(cout, generator=gen)]
    rng = np.random.default_rng(seed)
    x, t = [], []
    for _ in range(case["batch"]):
        medium, packet = _scene(rng, case["w"], case["h"], True)
        n = _ellipsoid((case["h"], case["w"]), **medium)
        q = _packet(n, **packet)
        later = dict(packet, x0=packet["x0"] + 8 * math.cos(packet["angle"]),
                     y0=packet["y0"] + 8 * math.sin(packet["angle"]))
        x.append(_features(q, n))
        t.append(torch.stack([b - a for a, b in zip(q, _packet(n, **later))], dim=-1))
    return torch.cat(flat), torch.stack(x).float(), torch.stack(t).float()


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case)
    if kind == "lattice":
        n, s["packet"] = _lattice_inputs(case, seed)
        g = qla.Grid(case["nx"], case["ny"], 1.0, case["precision"], te_only=case["te"],
                     tensor=case.get("tensor", False),
                     double_single=case.get("double_single", False))
        g.set_medium(n.cpu().numpy())
        if case["te"]:
            g.set_packet(**s["packet"])
        else:
            g.set_state(_lattice_state(case, n, s["packet"]).cpu().numpy())
        s["grid"] = g
    elif kind == "batch":
        grids = _batch_inputs(case, seed)
        b = qla.Batch([(side, side) for side, _, _ in grids], 1.0, "fp32", te_only=True)
        s["grids"] = [b.instance(k) for k in range(case["count"])]
        for g, (side, medium, packet) in zip(s["grids"], grids):
            g.set_medium(_ellipsoid((side, side), **medium).cpu().numpy())
            g.set_packet(**packet)
        s["batch_handle"] = b
    elif kind == "cube":
        n, packet = _cube_inputs(case, seed)
        g = qla.Grid3(case["nx"], case["ny"], case["nz"], 1.0, case["precision"],
                      double_single=case.get("double_single", False))
        g.set_medium(n.cpu().numpy())
        g.set_state(_six(n, n, n, packet).cpu().numpy())
        s["grid"] = g
    else:
        flat, s["x"], s["t"] = _network_inputs(case, seed)
        s["net"] = surrogate.Surrogate(case["h"], case["w"], max_batch=case["batch"])
        s["net"].set_params(flat.numpy())
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def run(s):
    kind = s["kind"]
    if kind == "lattice":
        g = s["grid"]
        if s["out"] == "state":
            g.set_packet(**s["packet"])
        g.step(s["steps"])
        energy = g.energy()
        if s["out"] == "state":
            return {"energy": energy, "state": g.get_state()}
        if s["out"] == "features":
            return {"energy": energy, "features": surrogate.features(g)}
        return {"energy": energy, "state": g.pack_box(0, 0, s["nx"], s["ny"])}
    if kind == "batch":
        energies = s["batch_handle"].run(s["steps"], s["every"])
        return {"energies": energies, "features": [surrogate.features(g) for g in s["grids"]]}
    if kind == "cube":
        g = s["grid"]
        g.step(s["steps"])
        return {"energy": g.energy(), "state": g.get_state()}
    if kind == "forward":
        return s["net"].forward(s["x"])
    losses = [s["net"].train_step(s["x"], s["t"], 3e-4) for _ in range(s["steps"])]
    return {"losses": losses, "params": s["net"].params()}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def _lattice_work(sites, planes, size, steps, rotations):
    state = float(sites) * planes * size
    passes = steps if 2 * state > L2_BYTES else 1
    return 2 * state * passes, 6.0 * rotations * sites * steps


def work(case):
    kind = case["kind"]
    if kind == "lattice":
        size = 8 if case["precision"] == "fp64" else 4
        planes = 3 if case["te"] else 6
        sites = case["nx"] * case["ny"]
        b, f = _lattice_work(sites, planes, size, case["steps"], 16 if case["te"] else 32)
        out = {"state": 48.0, "features": 24.0, "box": float(planes * size)}[case["out"]]
        return {"bytes": b + out * sites, "flops": f}
    if kind == "batch":
        sites = sum(side * side for side, _, _ in _batch_inputs(case, 0))
        b, f = _lattice_work(sites, 3, 4, case["steps"], 16)
        return {"bytes": b + 24.0 * sites, "flops": f}
    if kind == "cube":
        sites = case["nx"] * case["ny"] * case["nz"]
        b, f = _lattice_work(sites, 6, 8 if case["precision"] == "fp64" else 4, case["steps"], 48)
        return {"bytes": b + 48.0 * sites, "flops": f}
    levels = [0, 1, 2, 3, 4, 3, 2, 1, 0, 0]
    pixels = case["batch"] * case["h"] * case["w"]
    flops = sum(18.0 * ci * co * pixels / 4 ** k for (ci, co), k in zip(CONVS, levels))
    weights = sum(9 * ci * co + co for ci, co in CONVS)
    # every layer's BF16 output is written once and read by the next layer
    # (and by the skips); the FP32 features and outputs once
    acts = sum(co * pixels / 4 ** k for (_, co), k in zip(CONVS[:-1], levels))
    forward = 2 * 2 * acts + 4 * (6 + 3) * pixels + 2 * weights
    if kind == "forward":
        return {"bytes": forward, "flops": flops}
    # backward: two contractions per layer, activations read again, their
    # gradients written and read; Adam reads and writes three FP32 values
    first = 18.0 * CONVS[0][0] * CONVS[0][1] * pixels
    train = forward + 3 * 2 * acts + 4 * (4 * 2) * weights
    return {"bytes": case["steps"] * train, "flops": case["steps"] * (3 * flops - first)}


# ---------------------------------------------------------------------------
# The same outputs in 64 bits
# ---------------------------------------------------------------------------

# pairs of each axis, with the sine's sign, and the two streamed pairs
PAIRS = {"x": [(1, 5, 1), (2, 4, 1)], "y": [(0, 5, -1), (2, 3, -1)], "z": [(0, 4, 1), (1, 3, 1)]}
MOVERS = {"x": [(1, 4), (2, 5)], "y": [(0, 3), (2, 5)], "z": [(0, 3), (1, 4)]}
POTENTIAL = {"x": [(2, 4, -1), (1, 5, 1)], "y": [(2, 3, 1), (0, 5, -1)],
             "z": [(1, 3, -1), (0, 4, 1)]}
# the sixteen factors of U in the order they act: collision (adjoint: -1) or
# (streamed pair, shift)
FACTORS = [-1, (0, -1), 1, (0, 1), -1, (1, 1), 1, (1, -1),
           1, (0, 1), -1, (0, -1), 1, (1, -1), -1, (1, 1)]
DIM = {"x": -1, "y": -2, "z": -3}


def _rotate(q, a, b, c, s, sign):
    if a in q and b in q:
        x, y = q[a], q[b]
        q[a] = torch.addcmul(c * x, s, y, value=-sign)
        q[b] = torch.addcmul(c * y, s, x, value=sign)


class _Exact:
    """The QLA step with plain periodic arrays: q maps an amplitude to its
    array, index(a, b) is the refractive index that sets a pair's angles."""

    def __init__(self, axes, index):
        self.axes = axes
        self.theta, self.beta = {}, {}
        cache = {}
        for ax in axes:
            for a, b, _ in PAIRS[ax] + POTENTIAL[ax]:
                n = index(a, b, ax)
                key = (ax, n.data_ptr())
                if key not in cache:
                    t = 0.25 / n
                    h = 0.5 * _gradient(n, DIM[ax]) / (n * n)
                    cache[key] = (torch.cos(t), torch.sin(t)), (torch.cos(h), torch.sin(h))
                self.theta[ax, a, b], self.beta[ax, a, b] = cache[key]

    def evolve(self, q):
        for ax in self.axes:
            for f in FACTORS:
                if isinstance(f, tuple):
                    for m in MOVERS[ax][f[0]]:
                        if m in q:
                            q[m] = torch.roll(q[m], -f[1], DIM[ax])
                else:
                    for a, b, sign in PAIRS[ax]:
                        _rotate(q, a, b, *self.theta[ax, a, b], f * sign)

    def potential(self, q):
        for ax in self.axes:
            for a, b, sign in POTENTIAL[ax]:
                _rotate(q, a, b, *self.beta[ax, a, b], sign)

    def run(self, q, steps):
        """Steps q; returns the state before the last potential step."""
        for k in range(steps):
            if k:
                self.potential(q)
            self.evolve(q)
        before = dict(q)
        self.potential(q)
        return before


def _energy(q):
    return float(sum((v * v).sum() for v in q.values()))


def _exact_lattice(case, seed):
    n, packet = _lattice_inputs(case, seed)
    if case.get("tensor"):
        n_of = {"x": n[1], "y": n[0]}      # (q1, q5): n_y; (q0, q5): n_x; with q2: n_z
        n_z, index = n[2], lambda a, b, ax: n_of[ax] if b == 5 else n[2]
    else:
        n_z, index = n, lambda a, b, ax: n
    if case["te"]:
        q = dict(zip((2, 3, 4), _packet(n_z, **packet)))
    else:
        q = dict(enumerate(_lattice_state(case, n, packet)))
    stored = _Exact("xy", index).run(q, case["steps"])
    if case.get("tensor"):                 # these contexts store the state after V
        stored = q
    if case["out"] == "features":
        return {"energy": _energy(q), "features": _features([q[2], q[3], q[4]], n)}
    if case["out"] == "state":
        zero = torch.zeros_like(n_z)
        return {"energy": _energy(q), "state": torch.stack([q.get(c, zero) for c in range(6)])}
    return {"energy": _energy(q), "state": torch.stack([stored[c] for c in sorted(stored)])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        cost = case["nx"] * case["ny"] * case["steps"] * (1 if case["te"] else 2)
        return _exact_lattice(case, seed) if cost < EXACT_SITE_STEPS else None
    if kind == "batch":
        energies, feats = [], []
        for side, medium, packet in _batch_inputs(case, seed):
            n = _ellipsoid((side, side), **medium)
            q = dict(zip((2, 3, 4), _packet(n, **packet)))
            step, e = _Exact("xy", lambda a, b, ax: n), []
            for _ in range(case["steps"] // case["every"]):
                step.run(q, case["every"])
                e.append(_energy(q))
            energies.append(e)
            feats.append(_features([q[2], q[3], q[4]], n).cpu())
        return {"energies": np.array(energies).T.copy(), "features": feats}
    if kind == "cube":
        if case["nx"] * case["ny"] * case["nz"] * case["steps"] * 3 > EXACT_SITE_STEPS:
            return None
        n, packet = _cube_inputs(case, seed)
        q = dict(enumerate(_six(n, n, n, packet)))
        _Exact("xyz", lambda a, b, ax: n).run(q, case["steps"])
        return {"energy": _energy(q), "state": torch.stack([q[c] for c in range(6)])}
    flat, x, t = _network_inputs(case, seed)
    p = flat.double().cuda().requires_grad_(kind == "train")
    if kind == "forward":
        with torch.no_grad():
            return _network(p, x.double())
    m, v, losses = torch.zeros_like(p), torch.zeros_like(p), []
    for k in range(1, case["steps"] + 1):
        loss = ((_network(p, x.double()) - t.double()) ** 2).mean()
        g, = torch.autograd.grad(loss, p)
        losses.append(float(loss))
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        with torch.no_grad():
            p -= 3e-4 * (m / (1 - 0.9 ** k)) / ((v / (1 - 0.999 ** k)).sqrt() + 1e-8)
    return {"losses": losses, "params": p.detach()}


def _conv(x, w, b):
    """3 x 3 periodic convolution as nine products (the FP64 convolutions of
    libraries need large workspaces)."""
    B, C, H, W = x.shape
    out = b.view(1, -1, 1, 1)
    for ky in range(3):
        for kx in range(3):
            shifted = torch.roll(x, (1 - ky, 1 - kx), (2, 3)).reshape(B, C, H * W)
            out = out + torch.matmul(w[:, :, ky, kx], shifted).view(B, -1, H, W)
    return out


def _network(p, x):
    layers, at = [], 0
    for ci, co in CONVS:
        w = p[at:at + co * ci * 9].view(co, ci, 3, 3)
        at += co * ci * 9
        layers.append((w, p[at:at + co]))
        at += co
    h, skips = x.permute(0, 3, 1, 2), []
    for k in range(5):
        h = F.leaky_relu(_conv(F.avg_pool2d(h, 2) if k else h, *layers[k]), 0.1)
        skips.append(h)
    for k, level in enumerate((3, 2, 1, 0)):
        up = F.interpolate(h, scale_factor=2, mode="nearest")
        h = F.leaky_relu(_conv(up, *layers[5 + k]) + skips[level], 0.1)
    return _conv(h, *layers[9]).permute(0, 2, 3, 1).contiguous()
