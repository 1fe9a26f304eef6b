"""Measured cases: what a user's program has this framework do, through its public entry points.

Each case is one pass of a kind of program:
  fit     one step of a structure fit against a scattering curve: fused forward (density generated in
          the plane pass), log-I(Q) loss gradient, adjoint to the cell and (mask) to the mask weights
  grad    a step through torch.autograd (autograd.binned_intensity) with a weighted least-squares loss
          in torch: the cell alone behind an analytic particle shape, or the cell and voxel weights
  stored  the curve of a density that the program already has on the device (float32 or float16)
  stream  the same with the density in pinned host memory
  merge   the three-level wide-range curve: ED-1, its two block-summed zooms, three forwards, merge
  batch   a fit step over a polydisperse set of particles of uneven sizes (one ur_batch)
  image   forward of a crystallite on a rotated lattice with its half spectrum kept, and the
          Ewald-sphere detector image read from it
  binq    Q binning of a half-spectrum intensity that the program has already

Inputs follow the package's synthetic workloads (inputs.py): cells of Gaussian atoms at seeded
positions, a particle shape, log or linear Q bins up to the grid's Nyquist limit.
"""
import math

import numpy as np
import torch

from paper_2303_13435_gb300 import api, autograd, inputs

SHAPES = {"sphere": inputs.SHAPE_SPHERE, "cube": inputs.SHAPE_CUBE, "octahedron": inputs.SHAPE_OCTAHEDRON,
          "all": inputs.SHAPE_ALL}
DTYPES = {"f32": torch.float32, "f16": torch.float16}


def listed():
    return [
        # the smallest workload of the package (64^3, simple-cubic cell, linear bins): launches and latency
        dict(name="fit64", kind="fit", n=64, ucell=16, dx=1.0 / 16, natoms=1, shape="sphere", frac=0.9, rot=0, org=0,
             nbins=128, log=False, mask=True),
        # a small particle whose occupancy is fitted voxel by voxel; cell edge not a power of two
        dict(name="weights128", kind="grad", n=128, ucell=50, dx=0.05, natoms=60, shape="sphere", frac=0.8, rot=0,
             org=0, nbins=200, log=True, weights=True),
        # a rotated crystallite on a mixed-radix grid (2 5^3), cell alone
        dict(name="cell250", kind="grad", n=250, ucell=64, dx=0.040625, natoms=60, shape="octahedron", frac=0.8,
             rot=1, org=0, nbins=256, log=True, weights=False),
        # the package's flagship: 512^3, 10 nm sphere of a MOF-like cell, 512 log bins
        dict(name="fit512", kind="fit", n=512, ucell=64, dx=0.040625, natoms=60, shape="sphere", frac=0.480769,
             rot=0, org=0, nbins=512, log=True, mask=True),
        # the same at twice the edge
        dict(name="fit1024", kind="fit", n=1024, ucell=64, dx=0.040625, natoms=60, shape="sphere", frac=0.480769,
             rot=0, org=0, nbins=512, log=True, mask=True),
        # a mixed-radix grid (2 3^3 7), tiling origin off the corner, particle of ragged extent
        dict(name="fit378", kind="fit", n=378, ucell=64, dx=0.040625, natoms=60, shape="sphere", frac=0.8, rot=0,
             org=1, nbins=256, log=True, mask=True),
        # a large mixed-radix box (2^4 3^2 5) full of stored float16 density
        dict(name="stored720", kind="stored", n=720, ucell=90, dx=0.04, natoms=60, shape="all", frac=1.0, rot=0, org=0,
             nbins=700, log=True, dtype="f16", sinc=False),
        # the wide-range curve: 20 nm cube filling 1024^3 in float16, 4x and 16x zooms in 512^3 boxes, 1000 bins
        dict(name="merge3", kind="merge", n=1024, low=512, f1=4, f2=16, ucell=128, dx=20.0 / 1024, natoms=60,
             nbins=1000, mode="windows"),
        # the polydisperse set: 64 particles on even smooth grids of 96 to 384
        dict(name="batch64", kind="batch", count=64, lo=96, hi=384, ucell=64, dx=0.040625, natoms=60, nbins=256),
        # a crystallite's detector image
        dict(name="image256", kind="image", n=256, ucell=64, dx=0.040625, natoms=60, shape="cube", frac=0.5, rot=1,
             nbins=300, log=True, det=1024, nlambda=3),
        # a density that is held on the host
        dict(name="stream1024", kind="stream", n=1024, ucell=64, dx=0.040625, natoms=60, shape="sphere", frac=0.38,
             rot=0, org=0, nbins=512, log=True, dtype="f16"),
        # a stored intensity averaged into a curve
        dict(name="binq512", kind="binq", n=512, dx=0.040625, nbins=512, log=True, sinc=False),
    ]


def _size(rng, lo, hi):
    """An even smooth edge, uniform over the logarithm of the range."""
    t = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(inputs.smooth_even_sizes(lo, hi), key=lambda v: abs(v - t))


def draw(rng):
    kind = rng.choice(["fit", "fit", "fit", "grad", "grad", "stored", "stored", "stream", "merge", "batch", "image",
                       "binq"])
    c = dict(kind=kind, ucell=rng.choice([16, 25, 37, 48, 64, 81, 96]), dx=round(rng.uniform(0.035, 0.055), 5),
             natoms=rng.randint(5, 80), nbins=rng.randint(40, 1000), log=rng.random() < 0.7)
    if kind == "merge":
        n = rng.choice([256, 320, 384, 512, 640, 768, 1024])
        c.update(n=n, low=_size(rng, max(n // 4, 64), n // 2), f1=4, f2=16, ucell=rng.choice([64, 100, 128]),
                 dx=round(20.0 / n, 6), mode=rng.choice(["windows", "invvar"]))
        return c
    if kind == "batch":
        c.update(count=rng.randint(3, 63), lo=rng.choice([64, 96, 128]), hi=rng.choice([160, 250, 320, 384]))
        return c
    if kind == "binq":
        c.update(n=_size(rng, 48, 640), sinc=rng.random() < 0.3)
        return c
    c.update(n=_size(rng, 48, 800) if kind != "fit" or rng.random() < 0.6 else rng.choice([64, 128, 256, 512, 1024]),
             shape=rng.choice(["sphere", "sphere", "cube", "octahedron"]), frac=round(rng.uniform(0.2, 0.95), 4),
             rot=rng.randint(0, 1))
    if kind == "image":
        c.update(n=_size(rng, 64, 512), det=rng.randint(200, 1500), nlambda=rng.randint(1, 7))
        return c
    c.update(org=rng.randint(0, 1))
    if kind == "fit":
        c.update(mask=rng.random() < 0.6)
    elif kind == "grad":
        c.update(n=_size(rng, 48, 512), weights=rng.random() < 0.4)
    elif kind == "stored":
        c.update(dtype=rng.choice(["f32", "f16"]), sinc=rng.random() < 0.3)
        if rng.random() < 0.3:
            c.update(shape="all", frac=1.0)
    else:
        c.update(dtype=rng.choice(["f32", "f16"]))
    return c


# ----------------------------------------------------------------------------
# Inputs
# ----------------------------------------------------------------------------

def _cell(case, seed):
    """Periodic cell of Gaussian atoms (inputs.gaussian_cell's recipe, on the GPU), as sharp as the grid
    resolves; float32 [U][U][U]."""
    u, dx = case["ucell"], case["dx"]
    a = u * dx
    if case["natoms"] == 1:
        r = inputs.SplitMix64(seed)
        atoms = [inputs.Atom((0.0, 0.0, 0.0), r.uniform_range(18.0, 22.0), r.uniform_range(0.07, 0.09))]
    else:
        atoms = inputs.mof_like_atoms(seed, case["natoms"], sigma_range=(dx, 2 * dx))
    pos = torch.tensor([t.frac for t in atoms], dtype=torch.float64, device="cuda") * a
    sig = torch.tensor([t.sigma for t in atoms], dtype=torch.float64, device="cuda")
    z = torch.tensor([t.z for t in atoms], dtype=torch.float64, device="cuda")
    x = torch.arange(u, dtype=torch.float64, device="cuda") * dx
    d = x[None, None, :] - pos[:, :, None]
    g = sum(torch.exp(-(d - k * a) ** 2 / (2 * sig * sig)[:, None, None]) for k in (-1, 0, 1))
    norm = z * (2 * math.pi * sig * sig) ** -1.5 * dx ** 3
    gzy = (norm[:, None, None] * g[:, 2, :, None] * g[:, 1, None, :]).reshape(len(atoms), u * u)
    return (gzy.T @ g[:, 0, :]).reshape(u, u, u).float().contiguous()


def _shape(case, seed):
    n = case["n"]
    r = inputs.SplitMix64(seed * 7 + 3)
    rc = 0.5 * case["frac"] * n  # circumscribed radius
    c = (float(n // 2),) * 3
    if case.get("org"):  # a particle that is not on the grid's centre
        c = tuple(n // 2 + round(r.uniform_range(-0.02, 0.02) * n, 2) for _ in range(3))
    rot = inputs.random_rotation(r) if case["rot"] else np.eye(3, dtype=np.float32)
    size = rc / math.sqrt(3.0) if case["shape"] == "cube" else rc
    return inputs.Shape(SHAPES[case["shape"]], c, float(np.float32(size)), rot)


def _planes(case, shape):
    """First plane and number of planes that the particle can reach."""
    n = case["n"]
    if shape.kind == inputs.SHAPE_ALL:
        return 0, n
    rc = 0.5 * case["frac"] * n + 1
    z0 = max(0, math.floor(shape.center[2] - rc))
    return z0, min(n - 1, math.ceil(shape.center[2] + rc)) - z0 + 1


def _edges(case):
    n, dx = case["n"], case["dx"]
    top = inputs.nyquist_q(dx)
    return inputs.log_edges(2 * math.pi / (n * dx), top, case["nbins"]) if case["log"] else inputs.linear_edges(top, case["nbins"])


def _origin(case, seed):
    r = inputs.SplitMix64(seed * 5 + 1)
    return tuple(r.randint(case["ucell"]) for _ in range(3)) if case.get("org") else (0, 0, 0)


def _lattice(case, seed):
    r = inputs.SplitMix64(seed * 3 + 2)
    return inputs.random_rotation(r), np.array([r.uniform() * case["ucell"] for _ in range(3)], dtype=np.float32)


def _weights(case, seed, shape):
    """Occupancies in [0, 1] inside the particle, zero outside."""
    n = case["n"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.rand((n, n, n), generator=g, device="cuda")
    return w * _mask(n, shape)


def _target(edges, radius_nm, electrons, n):
    """The curve that is fitted: a homogeneous sphere's, in Eq. 1 units, on a flat background."""
    q = np.sqrt(np.maximum(edges[:-1], 0.25 * edges[1]) * edges[1:])
    i = inputs.sphere_target_curve(q, radius_nm, electrons) / float(n) ** 6
    return torch.from_numpy(i + 1e-6 * i.max()).cuda()


def _scaled(target):
    """(1 / sigma, target / sigma) of a least-squares fit with errors in proportion to the curve."""
    return 1.0 / target, torch.ones_like(target)


def _detector(case, seed):
    """A detector whose corners reach the grid's Nyquist limit."""
    m, r = case["det"], inputs.SplitMix64(seed * 11 + 5)
    lam, dist = 0.1, 0.3
    two_theta = 2 * math.asin(min(0.9, inputs.nyquist_q(case["dx"]) * lam / (4 * math.pi)))
    return dict(nx=m, ny=m - m // 5, pixel_m=2 * dist * math.tan(two_theta) / (m * 1.28), distance_m=dist,
                beam=(0.5 * m + r.uniform(), 0.4 * m + r.uniform()), wavelength_nm=lam, bandwidth=0.02,
                nlambda=case["nlambda"], rot=inputs.random_rotation(r))


def _plan(case, shape, dtype="f32"):
    z0, nz = _planes(case, shape)
    return api.Plan(case["n"], case["dx"], _edges(case), z0=z0, nz=nz, ed_dtype=dtype)


def _particles(case, seed):
    """(Particle, case of its own) for each member of a polydisperse set."""
    out = []
    for p in inputs.batch_particles(case["count"], seed + 7, case["lo"], case["hi"]):
        size = float(p.shape.size) * (math.sqrt(3.0) if p.shape.kind == inputs.SHAPE_CUBE else 1.0)
        out.append((p, dict(case, n=p.n, frac=2 * size / p.n)))
    return out


def _batch_edges(case):
    return inputs.log_edges(2 * math.pi / (case["hi"] * case["dx"]), inputs.nyquist_q(case["dx"]), case["nbins"])


def _levels(case):
    """(factor, edge, voxel edge, first plane, planes) of the three zoom levels."""
    n, low, dx = case["n"], case["low"], case["dx"]
    out = [(1, n, dx, 0, n)]
    for f in (case["f1"], case["f2"]):
        out.append((f, low, dx * f, (low - n // f) // 2, n // f))
    return out


def _merge_edges(case):
    return inputs.log_edges(0.01, 0.95 * inputs.nyquist_q(case["dx"]), case["nbins"])


def _electrons(case, cell, shape):
    vol = {"sphere": 4.18879, "cube": 1.5396, "octahedron": 1.33333}[case["shape"]] * (0.5 * case["frac"] * case["n"]) ** 3
    return float(cell.double().mean()) * vol


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, kind=kind)
    if kind == "binq":
        n = case["n"]
        s["plan"] = api.Plan(n, case["dx"], _edges(case))
        s["plan"].set_voxel_sinc(case["sinc"])
        s["intensity"] = _intensity(case, seed)
        s["bins"] = api.new_bins(s["plan"])
        return s
    s["cell"] = cell = _cell(case, seed)
    if kind == "merge":
        s["shape"] = inputs.Shape(inputs.SHAPE_CUBE, (float(case["n"] // 2),) * 3, float(case["n"] // 2))
        edges = _merge_edges(case)
        s["edges"] = torch.from_numpy(edges).cuda()
        s["levels"] = []
        for f, n, dx, z0, nz in _levels(case):
            plan = api.Plan(n, dx, edges, z0=z0, nz=nz, ed_dtype="f16")
            s["levels"].append((f, n, dx, z0, nz, plan, torch.empty((n, n, n), dtype=torch.float16, device="cuda"),
                                api.new_bins(plan), plan.workspace(api.UR_WS_FORWARD)))
        s["out"] = torch.empty((5, case["nbins"]), dtype=torch.float64, device="cuda")
        return s
    if kind == "batch":
        edges = _batch_edges(case)
        plans, targets, shapes = [], [], []
        for p, c in _particles(case, seed):
            z0, nz = _planes(c, p.shape)
            plans.append(api.Plan(p.n, case["dx"], edges, z0=z0, nz=nz))
            r = 0.35 * c["frac"] * p.n * case["dx"]
            targets.append(_target(edges, r, float(cell.double().mean()) * 4.19 * (r / case["dx"]) ** 3, p.n))
            shapes.append(p.shape)
        s["targets"] = targets
        s["batch"] = api.Batch(plans, cell, shapes)
        return s
    s["shape"] = shape = _shape(case, seed)
    s["origin"] = _origin(case, seed)
    n = case["n"]
    s["plan"] = plan = _plan(case, shape, case.get("dtype", "f32"))
    if kind in ("fit", "grad"):
        s["target"] = _target(plan.edges, 0.4 * case["frac"] * n * case["dx"], _electrons(case, cell, shape), n)
    if kind == "grad":
        s["scale"], s["fitted"] = _scaled(s["target"])
    if kind == "fit":
        s["ws"] = plan.workspace(api.UR_WS_FORWARD | api.UR_WS_BACKWARD)
        s["bins"] = api.new_bins(plan)
        s["g"] = torch.empty(plan.nbins, dtype=torch.float64, device="cuda")
        s["dcell"] = torch.empty_like(cell)
        s["dmask"] = torch.empty((n, n, n), device="cuda") if case["mask"] else None
    elif kind == "grad":
        cell.requires_grad_()
        s["weights"] = _weights(case, seed, shape).requires_grad_() if case["weights"] else None
    elif kind == "image":
        s["lattice"] = _lattice(case, seed)
        s["detector"] = _detector(case, seed)
        s["ws"] = plan.workspace(api.UR_WS_FORWARD)
        s["bins"] = api.new_bins(plan)
        s["F"] = torch.empty((n, n, n // 2 + 1), dtype=torch.complex64, device="cuda")
    else:
        if kind == "stored":
            plan.set_voxel_sinc(case["sinc"])
        ed = api.build_density(n, cell, shape, origin=s["origin"], z_begin=plan.z0, z_count=plan.nz,
                               out_dtype=case["dtype"])
        what = api.UR_WS_FORWARD
        if kind == "stream":
            ed = torch.empty(ed.shape, dtype=ed.dtype, pin_memory=True).copy_(ed)
            what |= api.UR_WS_HOST_SLABS
        s["ed"] = ed
        s["ws"] = plan.workspace(what)
        s["bins"] = api.new_bins(plan)
    return s


def _intensity(case, seed):
    """|F|^2 as a disordered particle's: exponential speckle on a falling envelope; float32 half spectrum."""
    n = case["n"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    i = torch.empty((n, n, n // 2 + 1), device="cuda").exponential_(generator=g)
    k = torch.fft.fftfreq(n, 1.0 / n, device="cuda") ** 2
    kx = torch.arange(n // 2 + 1, device="cuda", dtype=torch.float32) ** 2
    return i.div_((1.0 + 0.01 * (k[:, None, None] + k[None, :, None] + kx)).square_())


def _curve(bins):
    """The mean intensities, as the float32 array that a plot or a comparison takes."""
    return bins[api.BIN_MEAN].float()


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "fit":
        api.fft_intensity_tiled(s["plan"], s["cell"], s["shape"], origin=s["origin"], bins=s["bins"], ws=s["ws"])
        api.log_mse_grad(s["bins"], s["target"], s["g"])
        api.backward(s["plan"], s["g"], s["bins"], s["cell"], s["shape"], s["ws"], origin=s["origin"],
                     dl_dcell=s["dcell"], dl_dmask=s["dmask"], want_mask=case["mask"])
        out = {"bins": s["bins"], "curve": _curve(s["bins"]), "dcell": s["dcell"]}
        if case["mask"]:
            out["dmask"] = s["dmask"]
        return out
    if kind == "grad":
        s["cell"].grad = None
        if case["weights"]:
            s["weights"].grad = None
        mean = autograd.binned_intensity(s["cell"], s["plan"], s["shape"], weights=s["weights"], origin=s["origin"])
        loss = torch.nn.functional.mse_loss(mean.nan_to_num() * s["scale"], s["fitted"])
        loss.backward()
        out = {"curve": mean.detach().float(), "loss": loss.detach().float(), "dcell": s["cell"].grad}
        if case["weights"]:
            out["dweights"] = s["weights"].grad
        return out
    if kind in ("stored", "stream"):
        api.fft_intensity(s["plan"], s["ed"], bins=s["bins"], ws=s["ws"])
        return {"bins": s["bins"], "curve": _curve(s["bins"])}
    if kind == "merge":
        ed1 = s["levels"][0][6]
        api.build_density(case["n"], s["cell"], s["shape"], out_dtype="f16", out=ed1)
        for f, n, dx, z0, nz, plan, ed, bins, ws in s["levels"]:
            if f > 1:
                api.zoom_density(ed1, f, n, out_dtype="f16", out=ed)
            api.fft_intensity(plan, ed[z0:z0 + nz], bins=bins, ws=ws)
        lv = s["levels"]
        api.merge([t[7] for t in lv], [t[1] for t in lv], [t[2] for t in lv], s["edges"], out=s["out"],
                  mode=case["mode"])
        return {"merged": s["out"].float(), "bins": [t[7] for t in lv], "zooms": [t[6] for t in lv[1:]]}
    if kind == "batch":
        b = s["batch"]
        b.forward()
        for bins, target, g in zip(b.bins, s["targets"], b.dl_dmean):
            api.log_mse_grad(bins, target, g)
        b.backward()
        return {"curves": torch.stack([t[api.BIN_MEAN] for t in b.bins]).float(), "dcell": torch.stack(b.dl_dcell)}
    if kind == "image":
        api.fft_intensity_tiled(s["plan"], s["cell"], s["shape"], bins=s["bins"], F_out=s["F"], ws=s["ws"],
                                lattice=s["lattice"])
        return {"bins": s["bins"], "curve": _curve(s["bins"]), "F": s["F"],
                "image": api.ewald_image(s["plan"], s["F"], s["detector"])}
    api.bin_q(s["plan"], s["intensity"], bins=s["bins"])
    return {"bins": s["bins"], "curve": _curve(s["bins"])}


# ----------------------------------------------------------------------------
# What a pass cannot do without
# ----------------------------------------------------------------------------

def _forward_flops(n, nz):
    h = n // 2 + 1
    return 2.5 * n * math.log2(n) * n * nz + 5.0 * n * math.log2(n) * (nz * h + n * h)


def work(case):
    kind, b = case["kind"], 48.0 * case["nbins"]
    if kind == "binq":
        e = case["n"] ** 2 * (case["n"] // 2 + 1)
        return {"bytes": 4.0 * e + b, "flops": 4.0 * e}
    u3 = 4.0 * case["ucell"] ** 3
    if kind == "merge":
        n, low = case["n"], case["low"]
        return {"bytes": u3 + 2.0 * (n ** 3 + 2 * low ** 3) + 3 * b + 40.0 * case["nbins"],
                "flops": 2.0 * n ** 3 + sum(_forward_flops(n, nz) for _, n, _, _, nz in _levels(case))}
    if kind == "batch":
        flops = 0.0
        for p, c in _particles(case, 0):
            nz = _planes(c, p.shape)[1]
            flops += _forward_flops(p.n, nz) * 2 + 5.0 * p.n * math.log2(p.n) * p.n * (p.n // 2 + 1)
        return {"bytes": (u3 + 2 * b) * case["count"], "flops": flops}
    n = case["n"]
    nz = n if case["shape"] == "all" else min(n, int(case["frac"] * n) + 1)
    fwd = _forward_flops(n, nz)
    adj = _forward_flops(n, n) + 5.0 * n * math.log2(n) * n * (n // 2 + 1)
    if kind == "fit":
        return {"bytes": 2 * u3 + 2 * b + (4.0 * n ** 3 if case["mask"] else 0.0), "flops": fwd + adj}
    if kind == "grad":
        return {"bytes": 2 * u3 + b + (12.0 * n ** 3 if case["weights"] else 0.0), "flops": fwd + adj}
    if kind == "image":
        return {"bytes": u3 + b + 8.0 * n * n * (n // 2 + 1) + 4.0 * case["det"] ** 2, "flops": fwd}
    return {"bytes": nz * n * n * (2.0 if case["dtype"] == "f16" else 4.0) + b, "flops": fwd}


# ----------------------------------------------------------------------------
# The same results in float64, with plain torch
# ----------------------------------------------------------------------------

def _mask(n, shape, z0=0, nz=None):
    """The particle's 0/1 mask; the decision is defined in float32 (ur.h)."""
    nz = n - z0 if nz is None else nz
    if shape.kind == inputs.SHAPE_ALL:
        return torch.ones((nz, n, n), device="cuda")
    c, size, rot = shape.f32()
    ax = torch.arange(n, dtype=torch.float32, device="cuda")
    x, y, z = (ax - float(c[0]))[None, None, :], (ax - float(c[1]))[None, :, None], (ax[z0:z0 + nz] - float(c[2]))[:, None, None]
    if shape.kind == inputs.SHAPE_SPHERE:
        return ((x * x + y * y) + z * z <= float(size * size)).float()
    p = [torch.abs((float(rot[0, a]) * x + float(rot[1, a]) * y) + float(rot[2, a]) * z) for a in range(3)]
    if shape.kind == inputs.SHAPE_CUBE:
        return ((p[0] <= float(size)) & (p[1] <= float(size)) & (p[2] <= float(size))).float()
    return ((p[0] + p[1]) + p[2] <= float(size)).float()


def _tiled(n, cell, origin):
    u = cell.shape[0]
    ix, iy, iz = ((torch.arange(n, device="cuda") + o) % u for o in origin)
    return cell[iz[:, None, None], iy[None, :, None], ix[None, None, :]]


def _rotated(n, cell, lattice, shape):
    """The cell on a rotated lattice: trilinear, float32 with every step rounded (ur.h)."""
    u, (r, q) = cell.shape[0], lattice
    ax = torch.arange(n, dtype=torch.float32, device="cuda")
    c = shape.f32()[0]
    d = [(ax - float(c[0]))[None, None, :], (ax - float(c[1]))[None, :, None], (ax - float(c[2]))[:, None, None]]
    p = [((float(r[a, 0]) * d[0] + float(r[a, 1]) * d[1]) + float(r[a, 2]) * d[2]) + float(q[a]) for a in range(3)]
    lo = [torch.floor(t) for t in p]
    f = [t - i for t, i in zip(p, lo)]
    i = [t.long() % u for t in lo]
    j = [(t + 1) % u for t in i]
    lerp = lambda a, b, t: a + t * (b - a)  # noqa: E731
    line = lambda iz, iy: lerp(cell[iz, iy, i[0]], cell[iz, iy, j[0]], f[0])  # noqa: E731
    return lerp(lerp(line(i[2], i[1]), line(i[2], j[1]), f[1]), lerp(line(j[2], i[1]), line(j[2], j[1]), f[1]), f[2])


def _spectrum(rho):
    """Eq. 1, half axis along x."""
    return torch.fft.rfftn(rho.double()).div_(float(rho.numel()))


def _k2_bins(n, dx, edges):
    """Bin of every k^2 (-1: none) and its |Q|."""
    dq = 2.0 * math.pi / (n * dx)
    q = dq * np.sqrt(np.arange(3 * (n // 2) ** 2 + 1, dtype=np.float64))
    j = np.searchsorted(edges, q, side="right") - 1
    j = np.where(q == edges[-1], len(edges) - 2, j)
    j = np.where((j >= 0) & (j < len(edges) - 1), j, -1)
    return torch.from_numpy(j).cuda(), torch.from_numpy(q).cuda()


def _k2_planes(n):
    k = torch.arange(n, device="cuda")
    k = torch.where(k < n // 2, k, k - n)
    kx = torch.arange(n // 2 + 1, device="cuda")
    kk = (k * k)[:, None] + (kx * kx)[None, :]
    w = torch.full((n // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
    w[0] = w[-1] = 1.0
    w = w.expand(n, -1)
    for z in range(n):
        yield z, int(k[z]) ** 2 + kk, w


def _sinc2(n, dims):
    k = torch.fft.fftfreq(n, 1.0, dtype=torch.float64, device="cuda") if dims == "full" else torch.arange(n // 2 + 1, dtype=torch.float64, device="cuda") / n
    return torch.sinc(k).square()


def _binned(n, dx, edges, plane, sinc=False):
    """[6][B] statistics of the intensities plane(z) of a half spectrum."""
    nb = len(edges) - 1
    lut, qs = _k2_bins(n, dx, edges)
    acc = torch.zeros((4, nb + 1), dtype=torch.float64, device="cuda")
    m2 = torch.zeros(nb + 1, dtype=torch.float64, device="cuda")
    s = _sinc2(n, "full") if sinc else None
    sxy = s[:, None] * _sinc2(n, "half")[None, :] if sinc else None

    def add(out, j, v):
        out += torch.bincount(j, weights=v, minlength=nb + 1)

    for sweep in (0, 1):
        for z, k2, w in _k2_planes(n):
            j = lut[k2] + 1
            v = plane(z) * (sxy * s[z]) if sinc else plane(z)
            j, w, v = j.reshape(-1), w.reshape(-1), v.reshape(-1)
            if sweep == 0:
                add(acc[0], j, w)
                add(acc[1], j, w * v)
                add(acc[2], j, w * v * v)
                add(acc[3], j, w * qs[k2].reshape(-1))
            else:
                add(m2, j, w * (v - mean[j]).square())
        if sweep == 0:
            mean = acc[1] / acc[0]
    a, m2, mean = acc[:, 1:], m2[1:], mean[1:]
    cnt = a[0]
    sem = torch.where(cnt > 1, torch.sqrt(m2 / (cnt * (cnt - 1))), math.nan)
    return torch.stack([cnt, a[1], a[2], a[3], mean, sem])


def _bins_of(F, dx, edges, sinc=False):
    n = F.shape[0]
    return _binned(n, dx, edges, lambda z: F[z].real.square() + F[z].imag.square(), sinc)


def _loss(bins, target, kind):
    mean = bins[4]
    if kind == "grad":
        scale, fitted = _scaled(target)
        d = mean.nan_to_num() * scale - fitted
        return d.square().mean(), 2.0 * d * scale / len(d)
    ok = mean > 0
    d = torch.where(ok, torch.log(torch.where(ok, mean, 1.0) / target), 0.0)
    return d.square().sum() / ok.sum(), torch.where(ok, 2.0 * d / (torch.where(ok, mean, 1.0) * ok.sum()), 0.0)


def _grad_rho(F, dx, edges, bins, g):
    """dL/drho of a loss on the bin means; F is overwritten."""
    n = F.shape[0]
    lut, _ = _k2_bins(n, dx, edges)
    per = torch.cat([torch.zeros(1, dtype=torch.float64, device="cuda"), torch.where(bins[0] > 0, g / bins[0], 0.0)])
    for z, k2, _ in _k2_planes(n):
        F[z] *= per[lut[k2] + 1]
    return torch.fft.irfftn(F, s=(n, n, n)).mul_(2.0)


def _fold(grho, mask, u, origin):
    """dL/du: the voxels of every repeat of the cell, summed."""
    v = grho * mask
    n = v.shape[0]
    for a, o in enumerate(origin[::-1]):  # axes z, y, x
        i = (torch.arange(n, device="cuda") + o) % u
        shape = list(v.shape)
        shape[a] = u
        v = torch.zeros(shape, dtype=torch.float64, device="cuda").index_add_(a, i, v)
    return v


def _zoomed(ed, f, low):
    n = ed.shape[0]
    m = n // f
    o = (low - m) // 2
    out = torch.zeros((low, low, low), dtype=torch.float64, device="cuda")
    for z in range(m):
        t = ed[z * f:(z + 1) * f].double().sum(0)
        out[o + z, o:o + m, o:o + m] = t.reshape(m, f, m, f).sum((1, 3))
    return out.half()


def _merged(levels, bins, edges, mode):
    c = np.sqrt(edges[:-1] * edges[1:])
    out = np.full((5, len(c)), np.nan)
    out[2], out[4] = 0.0, -1.0
    order = sorted(range(len(levels)), key=lambda i: inputs.nyquist_q(levels[i][2]))
    top = [inputs.nyquist_q(levels[i][2]) for i in range(len(levels))]
    b = [t.cpu().numpy() for t in bins]
    scale = [float(t[1]) ** 6 for t in levels]
    for j in range(len(c)):
        use = [i for i in range(len(levels)) if c[j] <= top[i] and b[i][0, j] > 0 and np.isfinite(b[i][5, j]) and b[i][5, j] > 0]
        if mode == "invvar" and use:
            w = np.array([1.0 / (b[i][5, j] * scale[i]) ** 2 for i in use])
            cnt = sum(b[i][0, j] for i in use)
            out[:, j] = (sum(w[t] * b[i][4, j] * scale[i] for t, i in enumerate(use)) / w.sum(), w.sum() ** -0.5, cnt,
                         sum(b[i][3, j] for i in use) / cnt, use[int(np.argmax(w))])
            continue
        lo = 0.0
        for t, i in enumerate(order):
            if lo <= c[j] < top[i] or (t == len(order) - 1 and c[j] == top[i]):
                if b[i][0, j] > 0:
                    out[:, j] = (b[i][4, j] * scale[i], b[i][5, j] * scale[i], b[i][0, j], b[i][3, j] / b[i][0, j], i)
                break
            lo = top[i]
    return torch.from_numpy(out)


def _ewald(F, dx, det):
    n = F.shape[0]
    iy, ix = torch.meshgrid(torch.arange(det["ny"], device="cuda"), torch.arange(det["nx"], device="cuda"), indexing="ij")
    x, y = (ix - det["beam"][0]).double() * det["pixel_m"], (iy - det["beam"][1]).double() * det["pixel_m"]
    r = torch.sqrt(x * x + y * y + det["distance_m"] ** 2)
    s = torch.stack([x / r, y / r, -(x * x + y * y) / (r * (r + det["distance_m"]))], -1)
    s = s @ torch.from_numpy(np.asarray(det["rot"], dtype=np.float64)).cuda()
    total = torch.zeros_like(x)
    count = torch.zeros_like(x)
    for t in range(det["nlambda"]):
        lam = det["wavelength_nm"] * (1.0 + det["bandwidth"] * ((t + 0.5) / det["nlambda"] - 0.5))
        k = s * (n * dx / lam)
        i0 = torch.floor(k)
        f = k - i0
        i0 = i0.long()
        ok = ((i0 >= -(n // 2)) & (i0 + 1 <= n // 2 - 1)).all(-1)
        v = torch.zeros_like(x)
        for c in range(8):
            bit = [(c >> a) & 1 for a in range(3)]
            w = torch.ones_like(x)
            for a in range(3):
                w = w * (f[..., a] if bit[a] else 1.0 - f[..., a])
            kx, ky, kz = (i0[..., a] + bit[a] for a in range(3))
            flip = torch.where(kx < 0, -1, 1)
            h = F[(kz * flip) % n, (ky * flip) % n, (kx * flip).clamp(max=n // 2)]
            v += w * (h.real.square() + h.imag.square())
        total += torch.where(ok, v, 0.0)
        count += ok
    return total / torch.where(count > 0, count, math.nan)


def _particle(case, cell, shape, edges, target, origin=(0, 0, 0), weights=None):
    """(bins, loss, dL/du, dL/drho) of one particle."""
    n = case["n"]
    mask = weights if weights is not None else _mask(n, shape)
    F = _spectrum(_tiled(n, cell, origin) * mask)
    bins = _bins_of(F, case["dx"], edges)
    loss, g = _loss(bins, target, case["kind"])
    grho = _grad_rho(F, case["dx"], edges, bins, g)
    return bins, loss, _fold(grho, mask, case["ucell"], origin), grho


def exact(case, seed):
    kind, dx = case["kind"], case["dx"]
    if kind == "binq":
        i = _intensity(case, seed)
        bins = _binned(case["n"], dx, _edges(case), lambda z: i[z].double(), case["sinc"])
        return {"bins": bins, "curve": bins[4]}
    cell = _cell(case, seed)
    if kind == "merge":
        n = case["n"]
        ed1 = _tiled(n, cell, (0, 0, 0)).half()
        shape = inputs.Shape(inputs.SHAPE_CUBE, (float(n // 2),) * 3, float(n // 2))
        ed1 *= _mask(n, shape).half()
        eds = [ed1] + [_zoomed(ed1, f, case["low"]) for f in (case["f1"], case["f2"])]
        edges, levels = _merge_edges(case), _levels(case)
        bins = [_bins_of(_spectrum(ed), lv[2], edges) for ed, lv in zip(eds, levels)]
        return {"merged": _merged(levels, bins, edges, case["mode"]), "bins": bins, "zooms": eds[1:]}
    if kind == "batch":
        edges, curves, grads = _batch_edges(case), [], []
        for p, c in _particles(case, seed):
            r = 0.35 * c["frac"] * p.n * dx
            target = _target(edges, r, float(cell.double().mean()) * 4.19 * (r / dx) ** 3, p.n)
            bins, _, du, _ = _particle(c, cell, p.shape, edges, target)
            curves.append(bins[4])
            grads.append(du)
        return {"curves": torch.stack(curves), "dcell": torch.stack(grads)}
    shape, n = _shape(case, seed), case["n"]
    edges, origin = _edges(case), _origin(case, seed)
    if kind in ("fit", "grad"):
        target = _target(edges, 0.4 * case["frac"] * n * dx, _electrons(case, cell, shape), n)
        w = _weights(case, seed, shape) if case.get("weights") else None
        bins, loss, du, grho = _particle(case, cell, shape, edges, target, origin, w)
        if kind == "fit":
            out = {"bins": bins, "curve": bins[4], "dcell": du}
        else:
            out = {"curve": bins[4], "loss": loss, "dcell": du}
        if case.get("mask") or case.get("weights"):
            out["dmask" if kind == "fit" else "dweights"] = grho.mul_(_tiled(n, cell, origin))
        return out
    if kind == "image":
        F = _spectrum(_rotated(n, cell, _lattice(case, seed), shape) * _mask(n, shape))
        bins = _bins_of(F, dx, edges)
        return {"bins": bins, "curve": bins[4], "F": F, "image": _ewald(F, dx, _detector(case, seed))}
    rho = _tiled(n, cell, origin) * _mask(n, shape)
    F = _spectrum(rho.half() if case["dtype"] == "f16" else rho)
    bins = _bins_of(F, dx, edges, case.get("sinc", False))
    return {"bins": bins, "curve": bins[4]}
