"""Workloads of the multi-field VoF library that its speed is measured on.

Every case goes through the public entry points (``paper_2407_07463_gb300.vof``)
the way a program that embeds the library does: time steps in the three
precisions with and without recolouring, the batch of independent boxes, the
statistics and drop tables, the surface-tension source and the training
gradient.  Grids, drop radii, volume fractions, field counts and CFL numbers
come from this repository's configurations (``synth.config_*``), its tests
and its benchmark.

Inputs are made on the GPU from the seed: spheres placed by random sequential
addition, cell fractions by quadrature of the analytic chord, a discretely
solenoidal face velocity from a vector potential of Fourier modes.  ``exact``
restates the method in 64 bits with plain torch operations.
"""
import math

import numpy as np
import torch

from paper_2407_07463_gb300 import synth, vof

DEVICE = "cuda"
TAU = 1e-6       # the library's default occupancy threshold
TOL = 1e-3       # the learned normal's default fallback tolerance
PRECISION = {"fp64": vof.VOF_FP64, "mixed": vof.VOF_MIXED, "learned": vof.VOF_MIXED_LEARNED}


# --------------------------------------------------------------------------- cases


def listed():
    return [
        # the smallest validation box (32^3, one field, 8 drops, 20 steps per
        # call, double precision): what every user runs first, and what a
        # parameter study runs thousands of times; launches count here
        _step("step_fp64_small", "fp64", 32, 32, 32, 1, 4.0, 0.065, 0.25, nsteps=20),
        # the paper-like run in double precision with recolouring every step
        # (128^3, K = 4, phi = 0.1)
        _step("step_fp64_recolour", "fp64", 128, 128, 128, 4, 8.0, 0.1, 0.3, recolour=True, nsteps=2),
        # a production-size box in double precision (256^3, K = 8, phi = 0.3)
        _step("step_fp64_large", "fp64", 256, 256, 256, 8, 8.0, 0.3, 0.3),
        # mixed precision with MYC normals on an elongated channel
        _step("step_mixed", "mixed", 192, 160, 224, 6, 8.0, 0.2, 0.3, nsteps=2),
        # mixed precision on a box whose rows are not whole 16-byte lanes
        _step("step_mixed_ragged", "mixed", 101, 90, 75, 3, 6.0, 0.15, 0.3, nsteps=2),
        # the learned normal on a modest box, several steps per call
        _step("step_learned_small", "learned", 64, 64, 64, 3, 5.0, 0.15, 0.25, nsteps=4),
        # the benchmark's step: 256^3, K = 8, phi = 0.3, learned normal,
        # recolouring every step
        _step("step_learned_large", "learned", 256, 256, 256, 8, 8.0, 0.3, 0.3, recolour=True, nsteps=2),
        # an ensemble of independent boxes of uneven sizes advanced together:
        # a job of four steps
        {"name": "batch_learned", "kind": "batch", "precision": "learned", "boxes": 32, "draw": 5, "nsteps": 4},
        # one statistics event of the large box (nearest-particle histograms,
        # moments, drop shapes)
        {"name": "stats_large", "kind": "stats", "precision": "mixed", "nx": 256, "ny": 256, "nz": 256, "k": 8,
         "radius": 8.0, "phi": 0.3},
        # tags, drop table and drop shapes of every field of a double
        # precision box (post-processing of a snapshot)
        {"name": "tags_fp64", "kind": "tags", "precision": "fp64", "nx": 128, "ny": 128, "nz": 128, "k": 4,
         "radius": 8.0, "phi": 0.1},
        # the capillary force of all fields, once per step of a flow solver
        {"name": "tension_mixed", "kind": "tension", "precision": "mixed", "nx": 192, "ny": 192, "nz": 192, "k": 7,
         "radius": 8.0, "phi": 0.25},
        # the gradient of one training batch of the normal estimator (the
        # default batch)
        {"name": "train_gradient", "kind": "grad", "n": 16384},
    ]


def draw(rng):
    """One more case of the ranges above; its cost stays under the largest listed one's."""
    kind = rng.choice(["step", "step", "step", "step", "batch", "stats", "tags", "tension", "grad"])
    if kind == "grad":
        return {"kind": "grad", "n": int(round(math.exp(rng.uniform(math.log(1000), math.log(300000)))))}
    if kind == "batch":
        precision = rng.choice(["fp64", "mixed", "learned"])
        return {"kind": "batch", "precision": precision, "boxes": rng.randint(2, 4) if precision == "fp64" else rng.randint(3, 24),
                "draw": rng.randint(100, 100000), "nsteps": 2 if precision == "fp64" else rng.randint(2, 4)}
    precision = rng.choice(["fp64", "mixed", "learned"] if kind == "step" else ["fp64", "mixed"])
    edge = math.exp(rng.uniform(math.log(32), math.log(140 if precision == "fp64" else 208)))
    dims = [max(28, int(round(edge * rng.uniform(0.8, 1.25)))) for _ in range(3)]
    if rng.random() < 0.6:  # most users take whole words per row, some take what their geometry gives
        dims[0] = max(32, dims[0] // 32 * 32)
    radius = round(rng.uniform(3.5, 5.0) if edge < 64 else rng.uniform(5.0, 10.0), 2)
    case = {"kind": kind, "precision": precision, "nx": dims[0], "ny": dims[1], "nz": dims[2],
            "k": rng.randint(1, 8), "radius": radius, "phi": round(rng.uniform(0.05, 0.3), 3)}
    if kind == "step":
        case.update(cfl=round(rng.uniform(0.1, 0.45), 3), recolour=rng.random() < 0.4, nsteps=rng.randint(1, 3))
        if case["recolour"]:  # enough fields that only the drops that have just met have to move
            case.update(k=rng.randint(5, 8), phi=min(case["phi"], 0.2))
    return case


def _step(name, precision, nx, ny, nz, k, radius, phi, cfl, recolour=False, nsteps=1):
    return {"name": name, "kind": "step", "precision": precision, "nx": nx, "ny": ny, "nz": nz, "k": k,
            "radius": radius, "phi": phi, "cfl": cfl, "recolour": recolour, "nsteps": nsteps}


# --------------------------------------------------------------------------- inputs


def _generator(seed, salt):
    return torch.Generator(device=DEVICE).manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFF)


def _drop_count(case):
    return max(1, synth.n_spheres_for_phi((case["nz"], case["ny"], case["nx"]), case["radius"], case["phi"]))


def _centres(gen, shape, radius, phi):
    """Sphere centres (x, y, z) by random sequential addition in a periodic box."""
    L = torch.tensor([shape[2], shape[1], shape[0]], dtype=torch.float64, device=DEVICE)
    n = max(1, synth.n_spheres_for_phi(shape, radius, phi))
    have = torch.zeros((0, 3), dtype=torch.float64, device=DEVICE)
    for _ in range(400):
        p = torch.rand((2048, 3), dtype=torch.float64, device=DEVICE, generator=gen) * L
        if len(have):
            d = p[:, None, :] - have[None]
            d -= L * torch.round(d / L)
            p = p[(d.square().sum(-1) >= 4 * radius * radius).all(1)]
        d = p[:, None, :] - p[None]
        d -= L * torch.round(d / L)
        near = torch.tril(d.square().sum(-1) < 4 * radius * radius, -1)
        have = torch.cat([have, p[~near.any(1)]])[:n]
        if len(have) == n:
            break
    return have


def _colours(shape, centres, radius, k, gen, mixing):
    """Field of every drop: drops within reach of each other in different
    fields where k allows it; a share `mixing` of them is then put into a
    random field, as drops that have just met."""
    cen = centres.cpu().numpy()
    L = np.array([shape[2], shape[1], shape[0]], dtype=np.float64)
    reach = synth.conflict_distance(radius, 2)
    d = cen[:, None, :] - cen[None]
    d -= L * np.round(d / L)
    near = np.einsum("ijk,ijk->ij", d, d) < reach * reach
    np.fill_diagonal(near, False)
    order = np.argsort(-near.sum(1), kind="stable")
    field = -np.ones(len(cen), dtype=np.int64)
    for i in order:
        count = np.bincount(field[near[i] & (field >= 0)], minlength=k)
        field[i] = int(np.argmin(count))
    field = torch.from_numpy(field).to(DEVICE)
    if mixing > 0 and k > 1:
        pick = torch.rand(len(cen), device=DEVICE, generator=gen) < mixing
        other = torch.randint(0, k, (len(cen),), device=DEVICE, generator=gen)
        field = torch.where(pick, other, field)
    return field


def _gauss(sub, order):
    x, w = np.polynomial.legendre.leggauss(order)
    x, w = 0.5 * (x + 1.0), 0.5 * w
    nodes = ((np.arange(sub)[:, None] + x[None]).ravel()) / sub
    return (torch.from_numpy(nodes).to(DEVICE), torch.from_numpy(np.tile(w, sub) / sub).to(DEVICE))


def _chord_fraction(low, radius, sub=2, chunk=200000):
    """Fraction of unit cells with low corners `low` (relative to a sphere's
    centre) inside a sphere of `radius` (a number or one per cell)."""
    x, w = _gauss(sub, 4)
    qx, qy = [t.reshape(-1) for t in torch.meshgrid(x, x, indexing="ij")]
    qw = torch.outer(w, w).reshape(-1)
    r2 = torch.as_tensor(radius, dtype=torch.float64, device=DEVICE).square().expand(len(low))
    out = torch.empty(len(low), dtype=torch.float64, device=DEVICE)
    for s in range(0, len(low), chunk):
        g = low[s:s + chunk]
        h2 = r2[s:s + chunk, None] - (g[:, :1] + qx).square() - (g[:, 1:2] + qy).square()
        half = h2.clamp_min(0.0).sqrt()
        z = g[:, 2:3]
        out[s:s + chunk] = (torch.minimum(z + 1.0, half) - torch.maximum(z, -half)).clamp(0.0, 1.0) @ qw
    return out


def _spheres(shape, centres, radius):
    """(drop, cell, fraction) of every cell a sphere covers wholly or partly."""
    nz, ny, nx = shape
    span = int(math.ceil(2 * radius)) + 2
    o = torch.arange(span, device=DEVICE)
    oz, oy, ox = [t.reshape(-1) for t in torch.meshgrid(o, o, o, indexing="ij")]
    offs = torch.stack([ox, oy, oz], 1)
    drops, cells, fracs = [], [], []
    for s in range(0, len(centres), 256):
        p = centres[s:s + 256]
        ijk = torch.floor(p - radius).long()[:, None, :] + offs[None]
        low = ijk.double() - p[:, None, :]
        nearest = low.clamp_min(0.0) + (low + 1.0).clamp_max(0.0)
        inside = nearest.square().sum(-1) < radius * radius
        which, at = inside.nonzero(as_tuple=True)
        low, ijk = low[which, at], ijk[which, at]
        far = torch.maximum(low.abs(), (low + 1.0).abs()).square().sum(-1)
        f = torch.ones(len(low), dtype=torch.float64, device=DEVICE)
        cut = far > radius * radius
        f[cut] = _chord_fraction(low[cut], radius)
        i, j, k = ijk[:, 0] % nx, ijk[:, 1] % ny, ijk[:, 2] % nz
        drops.append(which + s)
        cells.append((k * ny + j) * nx + i)
        fracs.append(f)
    return torch.cat(drops), torch.cat(cells), torch.cat(fracs)


def _drops(case, seed, mixing=0.0):
    shape = (case["nz"], case["ny"], case["nx"])
    gen = _generator(seed, 11)
    centres = _centres(gen, shape, case["radius"], case["phi"])
    field = _colours(shape, centres, case["radius"], case["k"], gen, mixing)
    return shape, centres, field, _spheres(shape, centres, case["radius"])


def _fields(case, seed, mixing=0.0):
    """c [K][nz][ny][nx] in double."""
    shape, _, field, (drop, cell, frac) = _drops(case, seed, mixing)
    n = shape[0] * shape[1] * shape[2]
    c = torch.zeros(case["k"] * n, dtype=torch.float64, device=DEVICE)
    c.index_add_(0, field[drop] * n + cell, frac)
    return c.clamp_(0.0, 1.0).reshape((case["k"],) + shape)


def _velocity(shape, seed, amplitude, drift, modes=16):
    """Discretely solenoidal face velocity [3][nz][ny][nx] in double: the
    discrete curl of a vector potential of Fourier modes, plus a drift along z."""
    r = np.random.default_rng(int(seed) + 17)
    waves = []
    while len(waves) < modes:
        k = r.integers(-3, 4, size=3)
        if np.any(k):
            waves.append(k.astype(np.float64))
    waves = np.array(waves)
    amp = r.normal(size=(modes, 3))
    unit = waves / np.linalg.norm(waves, axis=1, keepdims=True)
    amp -= np.einsum("ij,ij->i", amp, unit)[:, None] * unit
    amp /= np.linalg.norm(amp, axis=1, keepdims=True)
    phase = r.random(modes) * 2.0 * math.pi
    nz, ny, nx = shape
    wv = torch.from_numpy(waves).to(DEVICE)

    def potential(comp):
        off = [0.5 if a == comp else 0.0 for a in range(3)]
        ex, ey, ez = [torch.exp(2j * math.pi * wv[:, a:a + 1] *
                                ((torch.arange(n, device=DEVICE, dtype=torch.float64) + off[a]) / n))
                      for a, n in enumerate((nx, ny, nz))]
        lead = torch.from_numpy(amp[:, comp] * np.exp(1j * phase)).to(DEVICE)
        zy = (lead[:, None, None] * ez[:, :, None] * ey[:, None, :]).reshape(modes, nz * ny)
        return (zy.T @ ex).imag.reshape(nz, ny, nx)

    X, Y, Z = potential(0), potential(1), potential(2)
    step = lambda a, axis: torch.roll(a, -1, axis) - a  # noqa: E731
    u = torch.stack([step(Z, 1) - step(Y, 0), step(X, 0) - step(Z, 2), step(Y, 2) - step(X, 1)])
    u *= amplitude / u.abs().max()
    u[2] += drift
    return u.contiguous()


def _network(seed, rough=0.02):
    """Flat parameters (the library's order) of a network near the Youngs
    estimate: hidden units 2a and 2a + 1 carry the positive and negative part
    of the Youngs component a, the other units random features that perturb
    the output by a share of about `rough`.  At the default half of the faces
    keep such a normal, as with a trained one; 0.3 stands for a network early
    in its training."""
    r = np.random.default_rng(int(seed) + 29)
    W1, W2, W3 = np.zeros((64, 32)), np.zeros((64, 64)), np.zeros((16, 64))
    b1, b2, b3 = np.zeros(64), np.zeros(64), np.zeros(16)
    W1[6:, :27] = r.normal(scale=0.2, size=(58, 27))
    W2[6:, 6:] = r.normal(scale=0.15, size=(58, 58))
    W3[:3, 6:] = r.normal(scale=rough, size=(3, 58))
    b1[6:], b2[6:] = r.normal(scale=0.1, size=58), r.normal(scale=0.1, size=58)
    w = {-1: 1.0, 0: 2.0, 1: 1.0}
    for a in range(3):
        for o in np.ndindex(3, 3, 3):
            x = (o[2] - 1, o[1] - 1, o[0] - 1)
            rest = [x[q] for q in range(3) if q != a]
            W1[2 * a, o[0] * 9 + o[1] * 3 + o[2]] = -x[a] * w[rest[0]] * w[rest[1]]
        W1[2 * a + 1] = -W1[2 * a]
        W2[2 * a, 2 * a] = W2[2 * a + 1, 2 * a + 1] = 1.0
        W3[a, 2 * a], W3[a, 2 * a + 1] = 1.0, -1.0
    p = np.concatenate([W1.ravel(), W2.ravel(), W3.ravel(), b1, b2, b3]).astype(np.float32)
    return torch.from_numpy(p).to(DEVICE)


def _stencils(n, seed):
    """Stencils [n][27] of spheres of radius 2..32 cells through the centre
    cell (half of them inverted) and their outward unit normals, in double."""
    gen = _generator(seed, 31)
    rand = lambda *s: torch.rand(*s, dtype=torch.float64, device=DEVICE, generator=gen)  # noqa: E731
    radius = torch.exp(math.log(2.0) + rand(n) * math.log(16.0))
    z, ph = 2.0 * rand(n) - 1.0, 2.0 * math.pi * rand(n)
    rho = (1.0 - z * z).sqrt()
    direction = torch.stack([rho * torch.cos(ph), rho * torch.sin(ph), z], 1)
    centre = -(radius + (rand(n) - 0.5) * 0.8)[:, None] * direction
    flip = rand(n) < 0.5
    o = torch.arange(-1, 2, device=DEVICE, dtype=torch.float64)
    oz, oy, ox = [t.reshape(-1) for t in torch.meshgrid(o, o, o, indexing="ij")]
    low = (torch.stack([ox, oy, oz], 1) - 0.5)[None] - centre[:, None, :]
    c = _chord_fraction(low.reshape(-1, 3), radius[:, None].expand(n, 27).reshape(-1)).reshape(n, 27)
    c = torch.where(flip[:, None], 1.0 - c, c)
    return c, torch.where(flip[:, None], -direction, direction)


def _box_specs(case):
    """(edge, field count, phi, radius) of every box of a batch: the ranges of
    the batched configuration."""
    r = np.random.default_rng(case["draw"])
    out = []
    for _ in range(case["boxes"]):
        n = int(r.choice((32, 48, 64, 96, 128)))
        out.append((n, int(r.integers(2, 9)), float(r.uniform(0.05, 0.3)), 4.0 if n < 64 else 8.0))
    return out


def _boxes(case, seed):
    """[(c, u, dt)] in double."""
    out = []
    for b, (n, k, phi, radius) in enumerate(_box_specs(case)):
        box = {"nx": n, "ny": n, "nz": n, "k": k, "radius": radius, "phi": phi}
        u = _velocity((n, n, n), 1000 * int(seed) + b, 0.5, 1.0)
        out.append((_fields(box, 1000 * int(seed) + b), u, 0.3 / float(u.abs().max())))
    return out


def _mixing(case):
    return 0.01 if case.get("recolour") else 0.0


def _step_inputs(case, seed):
    c = _fields(case, seed, _mixing(case))
    u = _velocity((case["nz"], case["ny"], case["nx"]), seed, 0.5, 1.0)
    return c, u, case["cfl"] / float(u.abs().max())


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _context(case, c, u, **kw):
    cfg = vof.make_config(case["nx"], case["ny"], case["nz"], k_capacity=case["k"], k_active=case["k"],
                          precision=PRECISION[case["precision"]], **kw)
    return vof.Context(cfg, c, u)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "grad":
        st, tgt = _stencils(case["n"], seed)
        weights = vof.vof_mlp_params_to_weights(_network(seed, rough=0.3))
        return {"kind": kind, "weights": weights, "stencils": st.float(), "targets": tgt.float()}
    dt_ = _dtype(case)
    if kind == "batch":
        made = _boxes(case, seed)
        c0 = torch.cat([c.to(dt_).reshape(-1) for c, _, _ in made])
        c = torch.empty_like(c0)
        parts = torch.split(c, [q.numel() for q, _, _ in made])
        boxes = [(part.view(q.shape), u.to(dt_).contiguous(), dt) for part, (q, u, dt) in zip(parts, made)]
        weights = vof.vof_mlp_params_to_weights(_network(seed)) if case["precision"] == "learned" else None
        return {"kind": kind, "boxes": boxes, "c": c, "c0": c0, "weights": weights, "nsteps": case["nsteps"],
                "precision": PRECISION[case["precision"]]}
    if kind == "step":
        c, u, dt = _step_inputs(case, seed)
        c0 = c.to(dt_)
        c = c0.clone()
        ctx = _context(case, c, u.to(dt_).contiguous(), recolour=int(case["recolour"]))
        if case["precision"] == "learned":
            ctx.vof_set_mlp(vof.vof_mlp_params_to_weights(_network(seed)), TOL)
        return {"kind": kind, "ctx": ctx, "c": c, "c0": c0, "dt": dt, "nsteps": case["nsteps"]}
    c = _fields(case, seed).to(dt_).contiguous()
    u = torch.zeros((3,) + tuple(c.shape[1:]), dtype=dt_, device=DEVICE)
    return {"kind": kind, "ctx": _context(case, c, u), "k": case["k"], "shape": tuple(c.shape[1:]),
            "drops": _drop_count(case)}


# --------------------------------------------------------------------------- one pass


def run(s):
    kind = s["kind"]
    if kind == "step":
        # the fields of this pass arrive in the context's buffer (from a
        # checkpoint, or from the solver that owns them)
        s["c"].copy_(s["c0"])
        rep = s["ctx"].vof_step(s["dt"], s["nsteps"])
        return {"c": s["c"], "n_active": rep["n_active"], "n_moved": rep["n_moved"]}
    if kind == "batch":
        # one job of an ensemble: new initial fields, a batch for them (a
        # batch keeps no face list across a change of its fields), its steps
        s["c"].copy_(s["c0"])
        batch = vof.Batch(s["boxes"], precision=s["precision"], autotune=False)
        if s["weights"] is not None:
            batch.set_mlp(s["weights"], TOL)
        batch.step(s["nsteps"])
        batch.close()
        return [b[0] for b in s["boxes"]]
    if kind == "stats":
        r = s["ctx"].vof_stats(reset=True)
        return {q: r[q] for q in ("n_drops", "d", "n_p", "volume", "events", "M", "R", "A", "chi_mean", "chi_max",
                                  "hist_r", "hist_rt")}
    if kind == "tags":
        # the snapshot's record: the tags of every field, one table of all drops
        labels = torch.empty((s["k"],) + s["shape"], dtype=torch.int32, device=DEVICE)
        tables = []
        for f in range(s["k"]):
            _, n = s["ctx"].vof_label(f, out=labels[f])
            volume, centre = s["ctx"].vof_drop_table(f, labels[f], n)
            tables.append((volume, centre) + s["ctx"].vof_drop_shape(f, labels[f], n, centre))
        return _record(labels, [torch.cat(t) for t in zip(*tables)], s["drops"])
    if kind == "tension":
        return s["ctx"].vof_surface_tension(0.05)
    grad, loss = vof.vof_mlp_grad(s["weights"], s["stencils"], s["targets"])
    return {"grad": grad, "loss": loss}


def _record(labels, columns, rows):
    """Tags and drop columns, the columns cut or filled up with zeros to `rows` drops."""
    out = {"labels": labels}
    for name, t in zip(("volume", "centre", "inertia", "chi"), columns):
        out[name] = t.new_zeros((rows,) + tuple(t.shape[1:]))
        out[name][:len(t)] = t[:rows]
    return out


def work(case):
    kind = case["kind"]
    if kind == "grad":
        # forward, backward through the activations and the weight gradients
        macs = 27 * 64 + 64 * 64 + 64 * 3
        return {"bytes": case["n"] * 30 * 4 + 2 * 7312 * 4, "flops": 6.0 * macs * case["n"]}
    es = 8 if case["precision"] == "fp64" else 4
    if kind == "batch":
        bytes_, flops = 0.0, 0.0
        for n, k, phi, radius in _box_specs(case):
            box = {"nx": n, "ny": n, "nz": n, "radius": radius, "phi": phi}
            bytes_ += (2 * k + 3) * n ** 3 * es * case["nsteps"]
            flops += _step_flops(box, case["precision"], case["nsteps"])
        return {"bytes": bytes_, "flops": flops}
    n = case["nx"] * case["ny"] * case["nz"]
    if kind == "step":
        return {"bytes": (2 * case["k"] + 3) * n * es * case["nsteps"],
                "flops": _step_flops(case, case["precision"], case["nsteps"])}
    if kind == "stats":
        return {"bytes": case["k"] * n * es + 1025 * 151 * 8, "flops": case["k"] * n * case["phi"]}
    if kind == "tags":
        return {"bytes": case["k"] * n * (es + 4), "flops": 30.0 * n * case["phi"]}
    return {"bytes": (case["k"] + 3) * n * es, "flops": 200.0 * _interface_cells(case)}


def _interface_cells(case):
    n = case["nx"] * case["ny"] * case["nz"]
    drops = case["phi"] * n / (4.0 / 3.0 * math.pi * case["radius"] ** 3)
    return drops * 1.5 * 4.0 * math.pi * case["radius"] ** 2


def _step_flops(case, precision, nsteps):
    """Normal, plane constant and swept volume of one face per interface cell
    and sweep; with the learned normal also the network and the two residuals."""
    per_face = 300.0 + (2.0 * (27 * 64 + 64 * 64 + 64 * 3) + 2 * 27 * 20.0 if precision == "learned" else 0.0)
    return 3.0 * nsteps * _interface_cells(case) * per_face


# --------------------------------------------------------------------------- 64-bit restatement


def exact(case, seed):
    kind = case["kind"]
    if kind == "grad":
        return _exact_grad(case, seed)
    if kind == "batch":
        net = _network(seed) if case["precision"] == "learned" else None
        out = []
        for c, u, dt in _boxes(case, seed):
            c, u = c.to(_dtype(case)).double(), u.to(_dtype(case)).double()
            out.append(_advance(c, u, dt, case["nsteps"], net))
        return out
    if kind == "step":
        if case["recolour"]:
            return None  # the moves between fields are decisions, compared as whole numbers
        c, u, dt = _step_inputs(case, seed)
        c, u = c.to(_dtype(case)).double(), u.to(_dtype(case)).double()
        net = _network(seed) if case["precision"] == "learned" else None
        return {"c": _advance(c, u, dt, case["nsteps"], net), "n_active": None, "n_moved": None}
    if kind == "tension":
        return _exact_tension(_fields(case, seed).to(_dtype(case)).double(), 0.05)
    return _exact_drops(case, seed)


def _place(cells, shape):
    """(i, j, k, base) of flat indices into fields of `shape` = (nz, ny, nx)."""
    nz, ny, nx = shape
    return cells % nx, cells // nx % ny, cells // (nx * ny) % nz, cells // (nx * ny * nz) * (nx * ny * nz)


def _gather(c, cells):
    """3x3x3 stencils [n][27] (x fastest) of flat cell indices of c [..][nz][ny][nx]."""
    nz, ny, nx = c.shape[-3:]
    i, j, k, base = _place(cells, (nz, ny, nx))
    st = []
    for dk in (-1, 0, 1):
        for dj in (-1, 0, 1):
            for di in (-1, 0, 1):
                at = base + (((k + dk) % nz) * ny + (j + dj) % ny) * nx + (i + di) % nx
                st.append(c.reshape(-1)[at])
    return torch.stack(st, 1)


def _youngs(st):
    s = st.reshape(-1, 3, 3, 3)
    w = torch.tensor([1.0, 2.0, 1.0], dtype=st.dtype, device=st.device)
    w2 = torch.outer(w, w)
    return torch.stack([((s[..., 0] - s[..., 2]) * w2).sum((1, 2)),
                        ((s[:, :, 0, :] - s[:, :, 2, :]) * w2).sum((1, 2)),
                        ((s[:, 0] - s[:, 2]) * w2).sum((1, 2))], 1)


def _myc(st):
    """Mixed-Youngs-Centred normals, L1-normalised."""
    y = _youngs(st)
    s = st.reshape(-1, 3, 3, 3)
    best, own = None, None
    for a in range(3):
        H = s.sum(3 - a)  # columns along axis a; the other axes stay ordered (high, low)
        lo, hi = [q for q in range(3) if q != a]
        m = torch.empty_like(y)
        m[:, lo] = 0.5 * (H[:, 1, 0] - H[:, 1, 2])
        m[:, hi] = 0.5 * (H[:, 0, 1] - H[:, 2, 1])
        m[:, a] = torch.where(y[:, a] < 0, -1.0, 1.0)
        o = m[:, a].abs() / m.abs().sum(1)
        if best is None:
            best, own = m, o
        else:
            take = o > own
            best, own = torch.where(take[:, None], m, best), torch.where(take, o, own)
    ny = y.abs().sum(1)
    use = (ny >= 1e-30) & (y.abs().amax(1) / ny < own)
    m = torch.where(use[:, None], y, best)
    return m / m.abs().sum(1, keepdim=True)


def _lower_half(a, b, c, x):
    """(volume, its slope) under the plane a x + b y + c z < x for sorted
    0 <= a <= b <= c and 0 <= x <= (a + b + c) / 2: inclusion-exclusion over
    the vertices (Scardovelli & Zaleski 2000), its terms paired so that none
    cancels."""
    bc6 = 6.0 * b * c
    thin = a < 1e-90
    abc6 = torch.where(thin, 1.0, bc6 * a)
    bc6 = bc6.clamp_min(1e-290)
    tb, tc = (x - b).clamp_min(0.0), (x - c).clamp_min(0.0)
    corner, area = (tb * tb * tb + tc * tc * tc) / abc6, 3.0 * (tb * tb + tc * tc) / abc6
    v = (3.0 * x * (x - a) + a * a) / bc6 - torch.where(thin, 0.0, corner)
    g = (6.0 * x - 3.0 * a) / bc6 - torch.where(thin, 0.0, area)
    first = (x <= a) & ~thin
    v, g = torch.where(first, x * x * x / abc6, v), torch.where(first, 3.0 * x * x / abc6, g)
    prism = x > a + b
    return torch.where(prism, (2.0 * x - a - b) / (2.0 * c), v), torch.where(prism, 1.0 / c, g)


def _half_volume(m, alpha):
    """Volume of {x in the unit cube: m.x < alpha}."""
    s, _ = m.abs().sort(1)
    a, b, c = s[:, 0], s[:, 1], s[:, 2]
    x = alpha + (-m).clamp_min(0.0).sum(1)
    S = a + b + c
    flip = 2.0 * x > S
    v, _ = _lower_half(a, b, c, torch.where(flip, S - x, x).clamp_min(0.0))
    v = torch.where(flip, 1.0 - v, v)
    return torch.where(x <= 0, 0.0, torch.where(x >= S, 1.0, v))


def _alpha(m, cv):
    """Plane constant with volume cv in (0, 1): Newton on the lower half from
    the root of its first or second piece."""
    s, _ = m.abs().sort(1)
    a, b, c = s[:, 0], s[:, 1], s[:, 2]
    S = a + b + c
    flip = cv > 0.5
    v = torch.where(flip, 1.0 - cv, cv)
    bc = b * c
    tip = v * 6.0 * bc <= a * a
    x = torch.where(tip, (6.0 * a * bc * v).pow(1.0 / 3.0), 0.5 * a + (2.0 * bc * v - a * a / 12.0).clamp_min(0.0).sqrt())
    x = torch.minimum(x, 0.5 * S)
    for _ in range(40):
        f, g = _lower_half(a, b, c, x)
        y = torch.minimum(x - (f - v) / g.clamp_min(1e-290), 0.5 * S)
        y = torch.where((g > 0) & (y > 0), y, x)
        done = bool(((y - x).abs() <= 4e-16 * y).all())
        x = y
        if done:
            break
    x = torch.where(flip, S - x, x)
    return x - (-m).clamp_min(0.0).sum(1)


def _frame(st):
    y = _youngs(st)
    sign = torch.where(y < 0, -1.0, 1.0).double()
    perm = y.abs().argsort(dim=1, stable=True)
    return sign, perm


def _canonical(st):
    """Stencils in the frame with Youngs components >= 0 and increasing, and the frame."""
    sign, perm = _frame(st)
    steps = torch.tensor([1, 3, 9], device=st.device)
    s = torch.gather(sign.long() * steps, 1, perm)
    o = torch.arange(-1, 2, device=st.device)
    kc, jc, ic = [t.reshape(-1) for t in torch.meshgrid(o, o, o, indexing="ij")]
    at = 13 + ic * s[:, :1] + jc * s[:, 1:2] + kc * s[:, 2:3]
    return torch.gather(st, 1, at), sign, perm


def _split_network(params):
    p = params.double()
    w = params.bfloat16().double()
    return (w[:2048].reshape(64, 32)[:, :27], w[2048:6144].reshape(64, 64), w[6144:7168].reshape(16, 64)[:3],
            p[7168:7232], p[7232:7296], p[7296:7299])


def _network_normal(st, params):
    W1, W2, W3, b1, b2, b3 = _split_network(params)
    x, sign, perm = _canonical(st)
    h = torch.relu((x - 0.5) @ W1.T + b1)
    h = torch.relu(h @ W2.T + b2)
    out = h @ W3.T + b3
    n = torch.zeros_like(out).scatter_(1, perm, out) * sign
    return n / n.abs().sum(1, keepdim=True)


def _residual(st, m):
    """Mean over the 27 cells of |extended plane's fraction - c|."""
    A = _alpha(m, st[:, 13])
    e = torch.zeros_like(A)
    for q in range(27):
        o = torch.tensor([q % 3 - 1.0, q // 3 % 3 - 1.0, q // 9 - 1.0], dtype=st.dtype, device=st.device)
        e += (_half_volume(m, A - m @ o) - st[:, q]).abs()
    return e / 27.0


def _normals(st, params):
    m = _myc(st)
    if params is None:
        return m
    n = _network_normal(st, params)
    e = _residual(st, n)
    keep = ((e <= TOL) | (e <= _residual(st, m))) & torch.isfinite(n).all(1)
    return torch.where(keep[:, None], n, m)


def _advance(c, u, dt, nsteps, params, chunk=1000000):
    """nsteps split steps of every field of c [K][nz][ny][nx] from step index 0, in double."""
    x = c
    nz, ny, nx = c.shape[1:]
    for step in range(nsteps):
        cc = (x > 0.5).double()
        for sweep in range(3):
            d = (step + sweep) % 3
            axis = 2 - d
            s = u[d] * dt
            cells = ((x > 0) & (x < 1)).reshape(-1).nonzero().reshape(-1)
            # fluxes through the low faces: full donors first
            full = (x >= 1).double()
            F = s * torch.where(s > 0, torch.roll(full, 1, axis + 1), full)
            del full
            for q in range(0, len(cells), chunk):
                at = cells[q:q + chunk]
                st = _gather(x, at)
                m = _normals(st, params)
                alpha = _alpha(m, st[:, 13])
                *ijk, base = _place(at, (nz, ny, nx))
                ijk[d] = (ijk[d] + 1) % (nx, ny, nz)[d]
                high = base + (ijk[2] * ny + ijk[1]) * nx + ijk[0]
                for face, out in ((at, -1.0), (high, 1.0)):
                    sf = s.reshape(-1)[face % (nx * ny * nz)]
                    go = sf * out > 0
                    sg, mg, ag = sf[go], m[go].clone(), alpha[go]
                    md = mg[:, d].clone()
                    x0 = torch.where(sg > 0, 1.0 - sg, 0.0)
                    mg[:, d] = md * sg.abs()
                    F.reshape(-1)[face[go]] = sg * _half_volume(mg, ag - md * x0)
            x = x - (torch.roll(F, -1, axis + 1) - F) + cc * (torch.roll(s, -1, axis) - s)
        x = x.clamp(0.0, 1.0)
    return x


def _exact_tension(c, gamma):
    """Sum over the fields of gamma kappa grad c on the low faces (h = 1)."""
    K, nz, ny, nx = c.shape
    out = torch.zeros((3, nz, ny, nx), dtype=c.dtype, device=c.device)
    for f in range(K):
        x = c[f]
        cells = ((x > 0) & (x < 1)).reshape(-1).nonzero().reshape(-1)
        m = _myc(_gather(x, cells))
        size = m.abs()
        axis = torch.zeros(len(cells), dtype=torch.long, device=c.device)
        axis = torch.where(size[:, 1] > size[:, 0], 1, axis)
        axis = torch.where(size[:, 2] > torch.gather(size, 1, axis[:, None])[:, 0], 2, axis)
        kappa = torch.full((nz * ny * nx,), math.nan, dtype=c.dtype, device=c.device)
        for a in range(3):
            sel = axis == a
            at = cells[sel]
            s = torch.where(m[sel, a] < 0, -1, 1)
            b, e = [q for q in range(3) if q != a]
            pos = [at % nx, at // nx % ny, at // (nx * ny)]
            ok = torch.ones(len(at), dtype=torch.bool, device=c.device)
            H = {}
            for p in (-1, 0, 1):
                for q in (-1, 0, 1):
                    col = []
                    for t in range(-3, 4):
                        o = list(pos)
                        o[a], o[b], o[e] = pos[a] + t, pos[b] + p, pos[e] + q
                        col.append(x.reshape(-1)[((o[2] % nz) * ny + o[1] % ny) * nx + o[0] % nx])
                    lo, hi = torch.where(s > 0, col[0], col[6]), torch.where(s > 0, col[6], col[0])
                    ok &= (lo > 0.5) & (hi < 0.5)
                    H[p, q] = sum(col)
            fx, fy = 0.5 * (H[1, 0] - H[-1, 0]), 0.5 * (H[0, 1] - H[0, -1])
            fxx, fyy = H[1, 0] - 2 * H[0, 0] + H[-1, 0], H[0, 1] - 2 * H[0, 0] + H[0, -1]
            fxy = 0.25 * (H[1, 1] - H[1, -1] - H[-1, 1] + H[-1, -1])
            k = -(fxx * (1 + fy * fy) + fyy * (1 + fx * fx) - 2 * fxy * fx * fy) / (1 + fx * fx + fy * fy) ** 1.5
            kappa[at] = torch.where(ok, k, math.nan)
        kappa = kappa.reshape(nz, ny, nx)
        for d in range(3):
            low = torch.roll(kappa, 1, 2 - d)
            kf = torch.where(torch.isnan(low), kappa, torch.where(torch.isnan(kappa), low, 0.5 * (low + kappa)))
            out[d] += gamma * torch.nan_to_num(kf) * (x - torch.roll(x, 1, 2 - d))
    return out


def _exact_drops(case, seed):
    """Drop tables and statistics from the drops the spheres make (every
    sphere is one connected drop: same-field spheres do not touch)."""
    shape, centres, field, (drop, cell, frac) = _drops(case, seed)
    nz, ny, nx = shape
    n, D = nz * ny * nx, len(centres)
    L = torch.tensor([nx, ny, nz], dtype=torch.float64, device=DEVICE)
    c = torch.zeros(case["k"] * n, dtype=torch.float64, device=DEVICE)
    c.index_add_(0, field[drop] * n + cell, frac)
    at = field[drop] * n + cell
    # a cell that two same-field spheres share would join them: no value then
    shared = torch.zeros(case["k"] * n, dtype=torch.int32, device=DEVICE)
    shared.index_add_(0, at, torch.ones_like(at, dtype=torch.int32))
    if bool((shared > 1).any()) or _touching(c.clamp(0.0, 1.0).reshape((case["k"],) + shape), at, drop, D):
        return None
    v = c.clamp(0.0, 1.0).to(_dtype(case)).double()[at]
    tau = TAU
    keep = v > tau
    drop, cell, v = drop[keep], cell[keep], v[keep]
    root = torch.full((D,), n, dtype=torch.long, device=DEVICE).scatter_reduce_(0, drop, cell, "amin")
    pos = torch.stack([cell % nx, cell // nx % ny, cell // (nx * ny)], 1).double() + 0.5
    rel = pos - centres[drop]
    rel -= L * torch.round(rel / L)
    zero = torch.zeros(D, dtype=torch.float64, device=DEVICE)
    vol = zero.index_add(0, drop, v)
    cen = torch.stack([zero.index_add(0, drop, v * rel[:, a]) for a in range(3)], 1) / vol[:, None] + centres
    cen = cen % L
    r = pos - cen[drop]
    r -= L * torch.round(r / L)
    rr = r.square().sum(1)
    terms = [v * (rr - r[:, a] * r[:, a] + 1.0 / 6.0) for a in range(3)]
    terms += [-v * r[:, a] * r[:, b] for a, b in ((0, 1), (0, 2), (1, 2))]
    inertia = torch.stack([zero.index_add(0, drop, t) for t in terms], 1)
    full = inertia[:, [0, 3, 4, 3, 1, 5, 4, 5, 2]].reshape(D, 3, 3)
    eig = torch.linalg.eigvalsh(full.cpu()).to(DEVICE)
    chi = (eig[:, 2] / eig[:, 0]).sqrt()
    if case["kind"] == "tags":
        rows = (field * n + root).argsort()
        return _record(None, [vol[rows], cen[rows], inertia[rows], chi[rows]], _drop_count(case))
    total = float(vol.sum())
    d = torch.cat([(lambda q: q - L * torch.round(q / L))(cen[None] - cen[i:i + 256, None]).square().sum(-1)
                   for i in range(0, D, 256)])
    d.fill_diagonal_(math.inf)
    j = d.argmin(1)
    rv = cen[j] - cen
    rv -= L * torch.round(rv / L)
    rv, dist = rv.cpu().numpy(), rv.square().sum(1).sqrt().cpu().numpy()
    hist_r, hist_rt = np.zeros(1025), np.zeros((1025, 150))
    kr = np.minimum(np.floor(dist / 0.2).astype(int), 1024)
    kt = np.minimum(np.floor(np.arccos(np.clip(rv[:, 2] / dist, -1, 1)) / (math.pi / 150)).astype(int), 149)
    np.add.at(hist_r, kr, 1.0)
    np.add.at(hist_rt, (kr, kt), 1.0)
    M, R = rv.mean(0), np.einsum("ia,ib->ab", rv, rv) / D
    return {"n_drops": None, "d": (6.0 * total / D / math.pi) ** (1.0 / 3.0), "n_p": D / n, "volume": total,
            "events": float(D), "M": M, "R": R, "A": R - np.trace(R) / 3.0 * np.eye(3),
            "chi_mean": float(chi.mean()), "chi_max": float(chi.max()), "hist_r": hist_r, "hist_rt": hist_rt}


def _touching(c, at, drop, D):
    """Whether two drops of one field hold cells with a common face."""
    owner = torch.full((c.numel(),), -1, dtype=torch.long, device=c.device)
    owner[at] = drop
    owner = torch.where(c.reshape(-1) > TAU, owner, -1).reshape(c.shape)
    for axis in (1, 2, 3):
        other = torch.roll(owner, 1, axis)
        if bool(((owner >= 0) & (other >= 0) & (owner != other)).any()):
            return True
    return False


def _exact_grad(case, seed):
    st, tgt = _stencils(case["n"], seed)
    st, tgt = st.float().double(), tgt.float().double()
    params = _network(seed, rough=0.3)
    leaves = [w.clone().requires_grad_() for w in _split_network(params)]
    W1, W2, W3, b1, b2, b3 = leaves
    loss = 0.0
    for q in range(0, case["n"], 65536):
        x, sign, perm = _canonical(st[q:q + 65536])
        t = torch.gather(tgt[q:q + 65536] * sign, 1, perm)
        h = torch.relu((x - 0.5) @ W1.T + b1)
        h = torch.relu(h @ W2.T + b2)
        out = h @ W3.T + b3
        part = (1.0 - (out * t).sum(1) / out.square().sum(1).sqrt()).sum()
        (part / case["n"]).backward()
        loss += float(part.detach())
    g = torch.zeros(7312, dtype=torch.float64, device=DEVICE)
    g[:2048].reshape(64, 32)[:, :27] = W1.grad
    g[2048:6144] = W2.grad.reshape(-1)
    g[6144:7168].reshape(16, 64)[:3] = W3.grad
    g[7168:7232], g[7232:7296], g[7296:7299] = b1.grad, b2.grad, b3.grad
    return {"grad": g, "loss": loss}
