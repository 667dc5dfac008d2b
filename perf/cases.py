"""The work a user of this library has it do, as cases that can be timed: whole closures from the
smallest grids to the largest, both precisions, block edges with and without mirrored kernels, the
trace and its quadratures, ragged batches, the learned closure's training step and inference, point
sources, and the calls an implicit moment solver makes on every step.

A case is a dict of plain values; its "kind" says which entry points one pass calls.  `exact` gives the
same outputs in 64 bits from plain numpy and torch, without the library.
"""
import math

import numpy as np
import torch

from paper_2202_08778_gb300 import vet

FOUR_PI = 4.0 * math.pi


def listed():
    return [
        # the smallest closure: one refined patch (the 32^3 test grid in 8^3 blocks, 48 directions),
        # where launches and the wavefront's latency count
        _closure("closure_patch32", 32, 32, 32, block=8, nside=2),
        # the benchmark's grid
        _closure("closure_lognormal128", 128, 128, 128, block=16, nside=4),
        # the shadow test: the largest grid and direction set, a beam through one face, moments wanted
        _closure("closure_shadow256", 256, 128, 128, block=16, nside=8, field="cloud", boundary="beam", moments=True),
        # the FP64 path, as used to check the FP32 one
        _closure("closure_fp64_64", 64, 64, 64, block=16, nside=4, fp64=True, moments=True),
        # a block edge other than 8 and 16, ragged extents
        _closure("closure_block12", 108, 84, 60, block=12, nside=4, moments=True),
        # intensities of every direction kept, then their quadratures (with E also summed in FP64)
        {"name": "trace_moments", "kind": "trace", "nx": 96, "ny": 64, "nz": 48, "block": 8, "nside": 4, "fp64": False,
         "field": "lognormal", "boundary": "vacuum"},
        # the patches of an adaptive grid at one time step: ragged grids in one call
        {"name": "batch16", "kind": "batch", "grids": 16, "first": 100},
        # one optimiser step of the learned closure on a batch of snapshots
        {"name": "train_4x64", "kind": "train", "volumes": 4, "nx": 64, "ny": 64, "nz": 64, "block": 16},
        # the learned closure's network on one grid
        {"name": "learned_128", "kind": "learned", "nx": 128, "ny": 128, "nz": 128, "block": 16},
        # direct radiation of a star somewhere in the grid
        {"name": "point_source_128", "kind": "point", "nx": 128, "ny": 128, "nz": 128},
        # a moment solver's calls on a step that keeps f: change gate, wavespeeds on the faces of
        # every axis, the local closure for comparison; on a patch (launches count) and on a large
        # grid (memory counts)
        {"name": "solver_step_32", "kind": "solver", "nx": 32, "ny": 32, "nz": 32, "block": 8},
        {"name": "solver_step_256", "kind": "solver", "nx": 256, "ny": 256, "nz": 256, "block": 16},
    ]


def _closure(name, nx, ny, nz, block, nside, fp64=False, field="lognormal", boundary="vacuum", moments=False):
    return {"name": name, "kind": "closure", "nx": nx, "ny": ny, "nz": nz, "block": block, "nside": nside, "fp64": fp64,
            "field": field, "boundary": boundary, "moments": moments}


def draw(rng):
    kind = rng.choice(["closure", "closure", "closure", "closure", "trace", "batch", "train", "learned", "point",
                       "solver"])
    if kind in ("closure", "trace"):
        block = rng.choice([16, 16, 16, 8, 8, 8, 12, 10, 5, 4])
        nside = rng.choice([1, 2, 4, 4, 4, 8])
        fp64 = rng.random() < 0.25
        # cell-angles: as the largest listed case where the mirrored kernels run, less where a cell-angle
        # costs more or its stored faces or intensities take more memory
        most = 5e7 if fp64 else (3e9 if block in (8, 16) else 2e8)
        if kind == "trace":
            most = min(most, 4e8)
        nx, ny, nz = _extents(rng, block, most / (12 * nside * nside))
        field = rng.choice(["lognormal", "lognormal", "cloud"])
        # the cloud does not emit: it is lit from outside
        boundary = rng.choice(["beam", "lit"] if field == "cloud" else ["vacuum", "vacuum", "lit"])
        case = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "block": block, "nside": nside, "fp64": fp64, "field": field,
                "boundary": boundary}
        if kind == "closure":
            case["moments"] = rng.random() < 0.5
        return case
    if kind == "batch":
        return {"kind": kind, "grids": rng.randint(2, 20), "first": rng.randint(100, 1000)}
    if kind == "point":
        nx, ny, nz = _extents(rng, 1, 2e6)
        return {"kind": kind, "nx": nx, "ny": ny, "nz": nz}
    block = rng.choice([16, 16, 8, 8, 4, 6, 10, 12])
    nx, ny, nz = _extents(rng, block, {"train": 1e6, "learned": 4e6, "solver": 16e6}[kind])
    case = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "block": block}
    if kind == "train":
        case["volumes"] = rng.randint(1, max(1, min(6, int(1.2e6 // (nx * ny * nz)))))
    return case


def _extents(rng, block, most_cells):
    """Three multiples of the block edge, their product spread over its logarithm up to most_cells."""
    least = max(block, 16) ** 3
    target = math.exp(rng.uniform(math.log(least), math.log(max(least * 1.01, most_cells))))
    edge = target ** (1.0 / 3.0)
    out = []
    for _ in range(3):
        n = int(edge * rng.uniform(0.7, 1.3) / block)
        out.append(block * max(1, min(n, 320 // block)))
    while out[0] * out[1] * out[2] > max(most_cells, block ** 3):
        k = out.index(max(out))
        if out[k] == block:
            break
        out[k] -= block
    return out


# ---------------------------------------------------------------- inputs

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _gaussian_field(shape, gen, kmin=2.0, kmax=32.0, slope=-2.0):
    """Zero mean, unit variance, power k^slope for kmin <= |k| <= kmax (wavenumbers of the longest axis)."""
    longest = max(shape)
    white = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
    kz, ky = (torch.fft.fftfreq(n, d=1.0 / longest, device="cuda", dtype=torch.float64) for n in shape[:2])
    kx = torch.fft.rfftfreq(shape[2], d=1.0 / longest, device="cuda", dtype=torch.float64)
    k = torch.sqrt(kz[:, None, None] ** 2 + ky[None, :, None] ** 2 + kx[None, None, :] ** 2)
    band = (k >= kmin) & (k <= kmax)
    amp = torch.where(band, k.clamp(min=1.0) ** (0.5 * slope), torch.zeros_like(k))
    g = torch.fft.irfftn(torch.fft.rfftn(white) * amp, s=shape)
    g = g - g.mean()
    return g / g.std().clamp(min=1e-30)


def _lognormal(shape, gen):
    """(kappa, S, h): lognormal optical depths per cell (median 10^-0.5, clipped to [1e-3, 1e2]) and a
    correlated lognormal temperature behind S = T^4 / 4 pi."""
    h = 1.0 / max(shape)
    g1, g2 = _gaussian_field(shape, gen), _gaussian_field(shape, gen)
    dtau = torch.exp(-0.5 * math.log(10.0) + 1.5 * g1).clamp(1e-3, 1e2)
    S = torch.exp(4.0 * 0.5 * (0.5 * g1 + math.sqrt(0.75) * g2)) / FOUR_PI
    return dtau / h, S, h


def _cloud(shape, gen):
    """(kappa, S, h): a thick ellipsoidal cloud (kappa 1e3, two-cell edge) at a drawn place in a thin
    ambient medium, no emission."""
    nz, ny, nx = shape
    h = 1.0 / min(shape)
    c = 0.4 + 0.2 * torch.rand(3, generator=gen, device="cuda", dtype=torch.float64)
    axis = [(torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * h for n in shape]
    z, y, x = torch.meshgrid(*axis, indexing="ij")
    rho = torch.sqrt(((x - c[0] * nx * h) / 0.1) ** 2 + ((y - c[1] * ny * h) / 0.06) ** 2 + ((z - c[2] * nz * h) / 0.06) ** 2)
    kappa = 1e-2 + 1e3 * 0.5 * (1.0 - torch.tanh((rho - 1.0) * 0.06 / (2.0 * h)))
    return kappa, torch.zeros_like(kappa), h


def _quaternion(seed):
    q = np.random.default_rng(seed).standard_normal(4)
    return q / np.linalg.norm(q)


def _directions(nside, q):
    """HEALPix ring-scheme pixel centres, rotated by the unit quaternion q: [N][3]."""
    rows = []
    for ring in range(1, 4 * nside):
        cap = min(ring, 4 * nside - ring)
        if cap < nside:
            z, count, shift = 1.0 - cap * cap / (3.0 * nside * nside), 4 * cap, 0.5
            z = z if ring < nside else -z
        else:
            z, count = 4.0 / 3.0 - 2.0 * ring / (3.0 * nside), 4 * nside
            shift = 0.5 if (ring - nside) % 2 == 0 else 1.0
        phi = (np.arange(count) + shift) * (2.0 * math.pi / count)
        s = math.sqrt((1.0 - z) * (1.0 + z))
        rows.append(np.stack([s * np.cos(phi), s * np.sin(phi), np.full(count, z)], axis=1))
    v = np.concatenate(rows)
    w, u = q[0], np.asarray(q[1:])
    return v + 2.0 * np.cross(u, np.cross(u, v) + w * v)


def _boundary(kind, dirs, gen):
    """Ib [6][N]: none, a beam within 10 degrees of +x through the x = 0 face (within the nearest
    direction where none is that close), or a background that differs by face and direction."""
    if kind == "vacuum":
        return None
    n = dirs.shape[0]
    if kind == "beam":
        Ib = torch.zeros(6, n, device="cuda", dtype=torch.float64)
        lit = dirs[:, 0] >= min(math.cos(math.radians(10.0)), dirs[:, 0].max())
        Ib[0, torch.from_numpy(np.flatnonzero(lit)).cuda()] = 1.0
        return Ib
    return 0.5 + torch.rand(6, n, generator=gen, device="cuda", dtype=torch.float64)


def _transfer_inputs(case, seed):
    """kappa, S, Ib in the case's precision, h, the rotation."""
    gen = _generator(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    kappa, S, h = (_cloud if case["field"] == "cloud" else _lognormal)(shape, gen)
    q = _quaternion(seed)
    Ib = _boundary(case["boundary"], _directions(case["nside"], q), gen)
    real = torch.float64 if case["fp64"] else torch.float32
    return kappa.to(real), S.to(real), None if Ib is None else Ib.to(real), h, q


def _batch_grids(case):
    """Grid edge, block edge and nside of each grid of a ragged batch."""
    out = []
    for g in range(case["grids"]):
        rng = np.random.default_rng(case["first"] + g)
        out.append((int(rng.choice((32, 48, 64, 80, 96))), int(rng.choice((8, 16))), int(rng.choice((2, 4)))))
    return out


def _bf16_values(x):
    return x.to(torch.bfloat16).to(torch.float32)


def _network_params(seed):
    """He-uniform hidden layers, a small last layer, as BF16 values: a network some way into training."""
    gen = torch.Generator().manual_seed(int(seed))
    out = []
    for i, (ci, co) in enumerate(vet.layer_shapes()):
        bound = math.sqrt(6.0 / (27 * ci)) if i < 3 else 0.02
        W = (2.0 * torch.rand(27, co, ci, generator=gen) - 1.0) * bound
        b = 0.1 * torch.randn(co, generator=gen)
        if i == 3:
            b = torch.tensor([0.0] * 6 + [math.log(1e-2)])
        out.append((_bf16_values(W).numpy(), b.numpy()))
    return out


def _network_inputs(case, seed):
    """kappa, S, E (FP32, one or more volumes) and h."""
    gen = _generator(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    k, s, e = [], [], []
    for _ in range(case.get("volumes", 1)):
        kappa, S, h = _lognormal(shape, gen)
        k.append(kappa)
        s.append(S)
        e.append(FOUR_PI * torch.exp(0.7 * _gaussian_field(shape, gen, kmax=6.0)))
    return tuple(torch.stack(x).to(torch.float32) for x in (k, s, e)) + (h,)


def _tensor_field(shape, gen):
    """A symmetric tensor of unit trace per cell, [6][...]: xx, yy, zz, xy, xz, yz (FP64)."""
    d = 0.2 + torch.rand((3,) + tuple(shape), generator=gen, device="cuda", dtype=torch.float64)
    d = d / d.sum(0)
    o = 0.1 * torch.randn((3,) + tuple(shape), generator=gen, device="cuda", dtype=torch.float64)
    return torch.cat([d, o])


def _solver_inputs(case, seed):
    gen = _generator(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    kappa, S, h = _lognormal(shape, gen)
    kappa_ref = kappa * (1.0 + 0.02 * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64))
    S_ref = S * (1.0 + 0.02 * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64))
    E = FOUR_PI * S
    F = torch.randn((3,) + shape, generator=gen, device="cuda", dtype=torch.float64)
    F = E * F / F.norm(dim=0).clamp(min=1e-30) * torch.rand(shape, generator=gen, device="cuda", dtype=torch.float64)
    M = torch.zeros((10,) + shape, device="cuda", dtype=torch.float64)
    M[0], M[1:4] = E, F
    f = _tensor_field(shape, gen)
    return tuple(x.to(torch.float32).contiguous() for x in (kappa, S, kappa_ref, S_ref, M, f)) + (h,)


def _point_inputs(case, seed):
    gen = _generator(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    kappa, _, h = _lognormal(shape, gen)
    u = np.random.default_rng(seed).uniform(0.2, 0.8, 3)
    # the optical depth across the box stays moderate, as for a star that is seen at all
    return (0.1 * kappa).to(torch.float32), h, tuple(float(v) * n * h for v, n in zip(u, shape[::-1])), 1.0


# ---------------------------------------------------------------- one pass

def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        grids, fields = _batch_grids(case), []
        problems = []
        for g, (n, block, nside) in enumerate(grids):
            kappa, S, h = _lognormal((n, n, n), _generator(seed * 1000 + g))
            fields.append((kappa.to(torch.float32), S.to(torch.float32), torch.empty(6, n, n, n, device="cuda")))
            problems.append(((n, n, n), block, h, nside, _quaternion(seed * 1000 + g)))
        batch = vet.Batch(problems)
        return {"kind": kind, "batch": batch, "kappa": [x[0] for x in fields], "S": [x[1] for x in fields],
                "f": [x[2] for x in fields]}
    shape = (case["nz"], case["ny"], case["nx"])
    if kind in ("closure", "trace"):
        kappa, S, Ib, h, q = _transfer_inputs(case, seed)
        ctx = vet.Context(shape, case["block"], h, case["nside"], q, vet.VET_FP64 if case["fp64"] else vet.VET_FP32)
        s = {"kind": kind, "ctx": ctx, "kappa": kappa, "S": S, "Ib": Ib, "E64": None}
        if kind == "closure":
            s["f"] = kappa.new_empty((6,) + shape)
            s["M"] = kappa.new_empty((10,) + shape) if case["moments"] else None
        else:
            s["I"] = kappa.new_empty((ctx.N,) + shape)
            s["M"] = kappa.new_empty((10,) + shape)
            if not case["fp64"]:
                s["E64"] = torch.empty(shape, device="cuda", dtype=torch.float64)
        return s
    if kind == "train":
        kappa, S, E, h = _network_inputs(case, seed)
        f_ref = torch.stack([_tensor_field(shape, _generator(seed * 1000 + v)) for v in range(case["volumes"])])
        model = vet.Model()
        model.set_params(_network_params(seed))
        return {"kind": kind, "model": model, "shape": shape, "block": case["block"], "h": h, "kappa": kappa, "S": S,
                "E": E, "f_ref": f_ref.to(torch.float32), "volumes": case["volumes"],
                "loss": torch.zeros(1, device="cuda", dtype=torch.float64)}
    if kind == "learned":
        kappa, S, E, h = _network_inputs(case, seed)
        # the network needs the grid alone; a small direction set serves a fallback that is not taken
        ctx = vet.Context(shape, case["block"], h, 1, _quaternion(seed))
        model = vet.Model()
        model.set_params(_network_params(seed))
        return {"kind": kind, "ctx": ctx, "model": model, "kappa": kappa[0], "S": S[0], "E": E[0],
                "f": kappa.new_empty((6,) + shape)}
    if kind == "point":
        kappa, h, xs, L = _point_inputs(case, seed)
        return {"kind": kind, "shape": shape, "h": h, "xs": xs, "L": L, "kappa": kappa,
                "Edot": torch.empty_like(kappa), "pdot": kappa.new_empty((3,) + shape)}
    kappa, S, kappa_ref, S_ref, M, f, h = _solver_inputs(case, seed)
    blocks = kappa.numel() // case["block"] ** 3
    speeds = [kappa.new_empty([n + (a == 2 - k) for k, n in enumerate(shape)]) for a in range(3)]
    return {"kind": kind, "shape": shape, "block": case["block"], "h": h, "kappa": kappa, "S": S, "kappa_ref": kappa_ref,
            "S_ref": S_ref, "M": M, "f": f, "change": kappa.new_empty(3 + 3 * blocks), "T": kappa.new_empty((6,) + shape),
            "speeds": speeds}


def run(state):
    s, kind = state, state["kind"]
    if kind == "closure":
        s["ctx"].closure(s["kappa"], s["S"], s["Ib"], s["f"], s["M"])
        return [s["f"]] if s["M"] is None else [s["f"], s["M"]]
    if kind == "trace":
        s["ctx"].trace(s["kappa"], s["S"], s["Ib"], s["I"])
        s["ctx"].moments(s["I"], s["M"], E64_out=s["E64"])
        return [s["I"], s["M"]] if s["E64"] is None else [s["I"], s["M"], s["E64"]]
    if kind == "batch":
        s["batch"].closure(s["kappa"], s["S"], None, s["f"])
        return list(s["f"])
    if kind == "train":
        m = s["model"]
        m.features(s["shape"], s["block"], s["h"], s["kappa"], s["S"], s["E"], nvol=s["volumes"])
        m.forward()
        m.backward(s["f_ref"], lam=2e-3, loss_out=s["loss"])
        grads = m.grads()
        # a rate of zero: the optimiser's work is done and the weights stay, so that a pass can be repeated
        m.step(lr=0.0)
        return [s["loss"], [list(g) for g in grads]]
    if kind == "learned":
        kept = s["model"].closure(s["ctx"], s["kappa"], s["S"], s["E"], s["f"], threshold=float("inf"))
        return [s["f"], kept]
    if kind == "point":
        vet.point_source(s["shape"], s["h"], s["xs"], s["L"], s["kappa"], s["Edot"], s["pdot"])
        return [s["Edot"], s["pdot"]]
    vet.field_change(s["shape"], s["block"], s["h"], s["kappa"], s["S"], s["kappa_ref"], s["S_ref"], s["change"])
    for axis in range(3):
        vet.hlle_wavespeed(s["shape"], s["h"], s["f"], s["kappa"], s["speeds"][axis], axis)
    vet.local_closure(vet.VET_CLOSURE_M1, s["M"], s["T"])
    return [s["change"], s["speeds"], s["T"]]


# ---------------------------------------------------------------- what a pass cannot do without

def _segments(block):
    """Mean number of cell-ray and face-node-ray segments per cell-angle of an isotropic direction set
    (rays end at the first of a block's three upwind faces): a cell ray crosses about 0.7 block edges'
    worth of planes, and a block has 3 (block + 1)^2 nodes for its block^3 cells."""
    per_ray = 0.7 * block
    return per_ray, per_ray * 3.0 * (block + 1) ** 2 / block ** 3


def _transfer_flops(cells, block, nside):
    """Each segment is one exponential and one exact update (10 operations), each cell-angle ten moments."""
    cell, face = _segments(block)
    return cells * 12 * nside * nside * (10.0 * (cell + face) + 20.0)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = {"bytes": 0.0, "flops": 0.0}
        for n, block, nside in _batch_grids(case):
            w["bytes"] += 4.0 * 8 * n ** 3
            w["flops"] += _transfer_flops(n ** 3, block, nside)
        return w
    cells = float(case["nx"] * case["ny"] * case["nz"])
    if kind in ("closure", "trace"):
        real, n = (8.0 if case["fp64"] else 4.0), 12 * case["nside"] ** 2
        flops = _transfer_flops(cells, case["block"], case["nside"])
        if kind == "closure":
            return {"bytes": real * cells * (2 + 6 + (10 if case["moments"] else 0)), "flops": flops}
        return {"bytes": real * cells * (2 + 2 * n + 10) + (0 if case["fp64"] else 8.0 * cells), "flops": flops}
    # multiply-adds of the four convolutions with the real channel counts
    net = 2.0 * 27 * (6 * 32 + 2 * 32 * 32 + 32 * 7)
    if kind == "train":
        return {"bytes": 4.0 * cells * case["volumes"] * (3 + 6), "flops": 3.0 * net * cells * case["volumes"]}
    if kind == "learned":
        return {"bytes": 4.0 * cells * (3 + 6), "flops": net * cells}
    if kind == "point":
        # planes crossed on the way from the source: a quarter of each extent on average
        return {"bytes": 4.0 * cells * 5, "flops": cells * (2.0 * 0.25 * (case["nx"] + case["ny"] + case["nz"]) + 40.0)}
    faces = 3.0 * cells + case["nx"] * case["ny"] + case["ny"] * case["nz"] + case["nx"] * case["nz"]
    # gate: four fields; wavespeeds: three tensor components, the opacity, the faces; M1: four read, six written
    return {"bytes": 4.0 * (4.0 * cells + 3.0 * cells + faces + 10.0 * cells), "flops": 60.0 * cells}


# ---------------------------------------------------------------- the same in 64 bits

def exact(case, seed):
    kind = case["kind"]
    if kind == "closure":
        kappa, S, Ib, h, q = _transfer_inputs(case, seed)
        M, f = _exact_closure(kappa, S, Ib, h, q, case["block"], case["nside"])
        return [f, M] if case["moments"] else [f]
    if kind == "trace":
        kappa, S, Ib, h, q = _transfer_inputs(case, seed)
        dirs = _directions(case["nside"], q)
        I = torch.empty((len(dirs),) + tuple(kappa.shape), device="cuda", dtype=torch.float64)
        for k, Ik in _exact_intensities(kappa, S, Ib, h, dirs, case["block"]):
            I[k] = Ik
        w = FOUR_PI / len(dirs)
        d = torch.from_numpy(dirs).cuda()
        c = w * torch.cat([torch.ones_like(d[:, :1]), d, d * d, d[:, :1] * d[:, 1:], d[:, 1:2] * d[:, 2:]], dim=1)
        M = (c.T @ I.reshape(len(dirs), -1)).reshape((10,) + tuple(kappa.shape))
        return [I, M] if case["fp64"] else [I, M, M[0].clone()]
    if kind == "batch":
        out = []
        for g, (n, block, nside) in enumerate(_batch_grids(case)):
            kappa, S, h = _lognormal((n, n, n), _generator(seed * 1000 + g))
            q = _quaternion(seed * 1000 + g)
            out.append(_exact_closure(kappa.to(torch.float32), S.to(torch.float32), None, h, q, block, nside)[1])
        return out
    if kind == "train":
        return _exact_training(case, seed)
    if kind == "learned":
        kappa, S, E, h = _network_inputs(case, seed)
        params = [(torch.from_numpy(W).cuda().double(), torch.from_numpy(b).cuda().double()) for W, b in _network_params(seed)]
        o = _exact_network(_exact_features(kappa[0], S[0], E[0], h, case["block"])[None], params)[0]
        return [_exact_head(o), None]
    if kind == "point":
        return _exact_point(case, seed)
    return _exact_solver(case, seed)


def _march_events(n, block, half):
    """Plane crossings of a ray from a cell centre (half = 0.5) or lattice point (half = 0) back through a
    block along a direction of components n > 0: segment lengths in cells, the planes of each axis crossed
    before each segment, and the event index at which the ray leaves by axis a from upwind coordinate l."""
    planes = [((m + half) / n[a], a, m) for a in range(3) for m in range(0 if half else 1, block if half else block + 1)]
    planes.sort()
    t = np.array([p[0] for p in planes])
    crossed = np.zeros((len(planes), 3), dtype=np.int64)
    leave = np.full((3, block + 1), -1, dtype=np.int64)
    seen = np.zeros(3, dtype=np.int64)
    for e, (_, a, m) in enumerate(planes):
        crossed[e] = seen
        seen[a] += 1
        leave[a, m] = e
    return np.diff(t, prepend=0.0), crossed, leave


def _entry(n, block, half, leave, l):
    """Where rays from upwind coordinates l [3][rays] enter the block: their last event, and the flat index
    (into the three (block + 1)^2 upwind faces) and weight of the four nodes around the entry point."""
    at = np.stack([leave[a, l[a]] for a in range(3)])
    axis = np.argmin(at, axis=0)
    depth = np.take_along_axis(l, axis[None], 0)[0] + half
    nn = np.asarray(n)
    t = depth / nn[axis]
    b = np.where(axis == 0, 1, 0)
    c = np.where(axis == 2, 1, 2)
    N1 = block + 1
    idx, wgt = 0, []
    pos = [np.clip(np.take_along_axis(l, v[None], 0)[0] + half - t * nn[v], 0.0, float(block)) for v in (b, c)]
    low = [np.minimum(np.floor(p).astype(np.int64), block - 1) for p in pos]
    fb, fc = pos[0] - low[0], pos[1] - low[1]
    idx = axis * N1 * N1 + low[0] * N1 + low[1]
    wgt = np.stack([(1 - fb) * (1 - fc), (1 - fb) * fc, fb * (1 - fc), fb * fc])
    return at.min(axis=0), np.stack([idx, idx + 1, idx + N1, idx + N1 + 1]), wgt


def _exact_intensities(kappa, S, Ib, h, dirs, B):
    """(k, I_k) for every direction: hybrid characteristics (long inside blocks of edge B, bilinear on
    the lattice points of the faces between them), octant by octant."""
    dev, f64 = kappa.device, torch.float64
    shape = tuple(kappa.shape)
    nbz, nby, nbx = (n // B for n in shape)
    N1, NN = B + 1, (B + 1) ** 2
    to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    neg = dirs < 0
    for octant in range(8):
        flip = [bool(octant >> a & 1) for a in range(3)]
        ks = np.flatnonzero((neg == np.array(flip)).all(axis=1))
        if not len(ks):
            continue
        turn = [2 - a for a in range(3) if flip[a]]

        def blocks(x):
            x = x.to(f64).flip(turn) if turn else x.to(f64)
            return x.reshape(nbz, B, nby, B, nbx, B).permute(0, 2, 4, 1, 3, 5).reshape(-1, B, B, B).contiguous()

        kb, Sb = blocks(kappa * 1.0), blocks(S)
        kflat, Sflat = kb.reshape(-1, B ** 3), Sb.reshape(-1, B ** 3)
        # node rays of the three downwind faces
        u, v = np.divmod(np.arange(NN), N1)
        full = np.full(NN, B)
        nodes = np.concatenate([np.stack([full, u, v]), np.stack([u, full, v]), np.stack([u, v, full])], axis=1)
        tabs = []
        for k in ks:
            n = np.abs(dirs[k])
            length, crossed, leave = _march_events(n, B, 0.0)
            last, idx, wgt = _entry(n, B, 0.0, leave, nodes)
            live = last[None] >= np.arange(len(length))[:, None]
            cell = nodes[:, None, :] - 1 - crossed.T[:, :, None]
            cell = np.where(live[None], cell, 0)
            tabs.append((length[:, None] * live * h, (cell[2] * B + cell[1]) * B + cell[0], idx, wgt))
        seg, cell, idx, wgt = (to(np.stack([t[i] for t in tabs])) for i in range(4))
        nD, nE = seg.shape[:2]
        out = torch.zeros(nbz * nby * nbx, nD, 3, NN, device=dev, dtype=f64)
        edge = torch.zeros(3, nD, device=dev, dtype=f64)
        if Ib is not None:
            for a in range(3):
                edge[a] = Ib[2 * a + (1 if flip[a] else 0)].to(f64)[to(ks)]
        bz, by, bx = (to(x.ravel()) for x in np.indices((nbz, nby, nbx)))
        stride = (1, nbx, nbx * nby)

        def incoming(sel, d=slice(None)):
            fin = []
            for a, b in enumerate((bx, by, bz)):
                up = out[(sel - stride[a]).clamp(min=0)][:, d, a]
                fin.append(torch.where((b[sel] > 0)[:, None, None], up, edge[a][d][None, :, None]))
            return torch.cat(fin, dim=2)

        everything = torch.arange(nbx * nby * nbz, device=dev)
        for level in range(nbx + nby + nbz - 2):
            sel = everything[bx + by + bz == level]
            fin = incoming(sel)
            I = sum(fin.gather(2, idx[:, i][None].expand(len(sel), -1, -1)) * wgt[:, i] for i in range(4))
            kl, Sl = kflat[sel], Sflat[sel]
            for e in range(nE - 1, -1, -1):
                at = cell[:, e]
                I = I + (I - Sl[:, at]) * torch.expm1(-kl[:, at] * seg[:, e])
            out[sel] = I.reshape(len(sel), nD, 3, NN)
        # cell rays
        l = np.indices((B, B, B)).reshape(3, -1)[::-1]
        for j, k in enumerate(ks):
            n = np.abs(dirs[k])
            length, crossed, leave = _march_events(n, B, 0.5)
            _, idx_c, wgt_c = _entry(n, B, 0.5, leave, l)
            fin = incoming(everything, slice(j, j + 1))[:, 0]
            idx_c, wgt_c = to(idx_c), to(wgt_c)
            I = sum(fin[:, idx_c[i]] * wgt_c[i] for i in range(4)).reshape(-1, B, B, B)
            for e in range(len(length) - 1, -1, -1):
                x, y, z = (int(c) for c in crossed[e])
                if max(x, y, z) >= B:
                    continue
                part = I[:, z:, y:, x:]
                Su, ku = Sb[:, :B - z, :B - y, :B - x], kb[:, :B - z, :B - y, :B - x]
                part += (part - Su) * torch.expm1(-ku * (length[e] * h))
            I = I.reshape(nbz, nby, nbx, B, B, B).permute(0, 3, 1, 4, 2, 5).reshape(shape)
            yield int(k), I.flip(turn) if turn else I


def _exact_closure(kappa, S, Ib, h, q, B, nside):
    """(M [10], f [6]) of the closure."""
    dirs = _directions(nside, q)
    M = torch.zeros((10,) + tuple(kappa.shape), device=kappa.device, dtype=torch.float64)
    w = FOUR_PI / len(dirs)
    for k, I in _exact_intensities(kappa, S, Ib, h, dirs, B):
        x, y, z = (float(v) for v in dirs[k])
        for m, c in enumerate((1.0, x, y, z, x * x, y * y, z * z, x * y, x * z, y * z)):
            M[m].add_(I, alpha=w * c)
    E = M[0]
    lit = E > 1e-30 * E.max()
    iso = torch.tensor([1 / 3] * 3 + [0.0] * 3, device=E.device, dtype=torch.float64).view(6, 1, 1, 1)
    return M, torch.where(lit, M[4:] / torch.where(lit, E, torch.ones_like(E)), iso)


def _exact_features(kappa, S, E, h, B):
    """[6][cells...] features of one volume."""
    tiny = 1e-30
    lk, ls, le = (torch.log10(x.double().clamp(min=tiny)) for x in (kappa.double() * h, S, E))
    nz, ny, nx = kappa.shape
    t = lk.reshape(nz // B, B, ny // B, B, nx // B, B)
    mean, sd = t.mean((1, 3, 5)), t.var((1, 3, 5), unbiased=False).sqrt()
    spread = lambda v: v.repeat_interleave(B, 0).repeat_interleave(B, 1).repeat_interleave(B, 2)  # noqa: E731
    return torch.stack([torch.ones_like(lk), lk, ls - ls.mean(), le - le.mean(), spread(mean), spread(sd)])


def _exact_network(x, params):
    """x [v][6][z][y][x] -> [v][7][z][y][x]."""
    for i, (W, b) in enumerate(params):
        v, _, nz, ny, nx = x.shape
        pad = torch.nn.functional.pad(x, (1, 1, 1, 1, 1, 1))
        y = b.view(1, -1, 1, 1, 1).expand(v, -1, nz, ny, nx)
        for tap in range(27):
            dz, dy, dx = tap // 9, tap // 3 % 3, tap % 3
            y = y + torch.einsum("oc,vczyx->vozyx", W[tap], pad[:, :, dz:dz + nz, dy:dy + ny, dx:dx + nx])
        x = torch.nn.functional.silu(y) if i < 3 else y
    return x


def _exact_head(o):
    """f [6][...] of raw outputs o [7][...]."""
    tr = o[:3].sum(0) / 3.0
    return torch.cat([1.0 / 3.0 + o[:3] - tr, o[3:6]])


def _exact_training(case, seed):
    kappa, S, E, h = _network_inputs(case, seed)
    shape = (case["nz"], case["ny"], case["nx"])
    n = case["volumes"]
    params = [tuple(torch.from_numpy(p).cuda().double().requires_grad_() for p in layer) for layer in _network_params(seed)]
    loss = 0.0
    for v in range(n):
        o = _exact_network(_exact_features(kappa[v], S[v], E[v], h, case["block"])[None], params)[0]
        f_ref = _tensor_field(shape, _generator(seed * 1000 + v)).to(torch.float32).double()
        d = _exact_head(o) - f_ref
        target = torch.log(d.detach().abs().amax(0) + 1e-4)
        part = ((d * d).mean() + 2e-3 * ((o[6] - target) ** 2).mean()) / n
        part.backward()
        loss += part.detach()
    return [loss.reshape(1), [[W.grad, b.grad] for W, b in params]]


def _exact_point(case, seed):
    kappa, h, xs, L = _point_inputs(case, seed)
    nz, ny, nx = kappa.shape
    dev, f64 = kappa.device, torch.float64
    src = torch.tensor([x / h for x in xs], device=dev, dtype=f64).to(torch.float32).to(f64)
    ext = torch.tensor([nx, ny, nz], device=dev)
    z, y, x = torch.meshgrid(*(torch.arange(n, device=dev) for n in (nz, ny, nx)), indexing="ij")
    target = torch.stack([x, y, z]).reshape(3, -1)
    v = target + 0.5 - src[:, None]
    r = v.norm(dim=0)
    d = v / r
    up = (d > 0).long()
    inv = 1.0 / d
    lo, hi = (target - src[:, None]) * inv, (target + 1 - src[:, None]) * inv
    t_in = torch.minimum(lo, hi).amax(0).clamp(min=0.0)
    dr = torch.maximum(lo, hi).amin(0) - t_in
    at = src.floor().long()[:, None].expand(3, r.numel()).clone()
    kflat = kappa.double().reshape(-1)
    t, tau = torch.zeros_like(r), torch.zeros_like(r)
    for _ in range(nx + ny + nz + 3):
        cross = (at + up - src[:, None]) * inv
        nxt, axis = cross.min(0)
        nxt = torch.minimum(nxt, t_in)
        inside = ((at >= 0) & (at < ext[:, None])).all(0) & (t < t_in)
        if not bool(inside.any()):
            break
        cell = (at[2].clamp(0, nz - 1) * ny + at[1].clamp(0, ny - 1)) * nx + at[0].clamp(0, nx - 1)
        tau += torch.where(inside, kflat[cell] * (nxt - t), torch.zeros_like(t))
        t = torch.maximum(t, nxt)
        at.scatter_add_(0, axis[None], (2 * up - 1).gather(0, axis[None]))
    own = kflat * dr * h
    Edot = L * torch.exp(-tau * h) * -torch.expm1(-own) / (FOUR_PI * (r * h) ** 2 * dr * h)
    return [Edot.reshape(nz, ny, nx), (Edot * d).reshape(3, nz, ny, nx)]


def _exact_solver(case, seed):
    kappa, S, kappa_ref, S_ref, M, f, h = (x.double() if isinstance(x, torch.Tensor) else x for x in _solver_inputs(case, seed))
    B = case["block"]
    nz, ny, nx = kappa.shape
    a, b = kappa * h, kappa_ref * h
    per = torch.stack([(a - b).abs() / ((1 + a / 2) * (1 + b / 2)), (S - S_ref).abs(), S_ref.abs()])
    blk = per.reshape(3, nz // B, B, ny // B, B, nx // B, B).amax((2, 4, 6)).reshape(3, -1)
    change = torch.cat([blk.amax(1), blk.T.reshape(-1)])
    speeds = []
    for axis in range(3):
        dim, fa = 2 - axis, f[axis]
        tau = (10.0 * h * kappa) ** 2 / (2.0 * fa)
        first, end = (lambda t: t.narrow(dim, 0, 1)), (lambda t: t.narrow(dim, t.shape[dim] - 1, 1))
        left, right = (lambda t: torch.cat([first(t), t], dim)), (lambda t: torch.cat([t, end(t)], dim))
        mean = 0.5 * (left(tau) + right(tau))
        speeds.append(torch.maximum(left(fa), right(fa)).sqrt() * (-torch.expm1(-mean) / mean).sqrt())
    E, F = M[0], M[1:4]
    norm = F.norm(dim=0)
    red = (norm / E).clamp(max=1.0)
    chi = (3 + 4 * red ** 2) / (5 + 2 * (4 - 3 * red ** 2).sqrt())
    n = F / norm.clamp(min=1e-300)
    p, s = (1 - chi) / 2, (3 * chi - 1) / 2
    T = torch.stack([p + s * n[0] ** 2, p + s * n[1] ** 2, p + s * n[2] ** 2, s * n[0] * n[1], s * n[0] * n[2], s * n[1] * n[2]])
    return [change, speeds, T]
