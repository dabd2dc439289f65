"""The work that users of the local-Hamiltonian library have it do, as timed cases.

Every case goes through the package's public entry points on device tensors,
as a program that owns its orbitals does.  The sizes are those of the
package's benchmark and tests (orbitals on coarse cells of 16 to 64 points per
axis, one to 512 of them) and ragged ones between them.

Kinds
-----
hpsi       one `hpsi_local` call on the orbitals of one periodic cell
plan       `Plan.hpsi` over cells of different sizes, with preallocated results
           on the program's compute stream (graph replay), the density included
eloc       `ELoc` forward and backward: E, dE/dpsi and dE/dV
products   `overlap` of all orbitals and the per-orbital `dot` with H psi
precond    `precondition`: a fixed number of CG iterations per orbital
region     `hpsi_local_region` on a ball-shaped localisation region
bc         `hpsi_local_bc` with free axes (isolated and surface conditions)
operators  the five 3D operators one after another, as a program that builds
           its own chain calls them

`prec` is f64 (FP64), f32 (FP32 convolutions) or emu (FP64 arrays, convolution
sums on the tensor cores).  Coefficients are uniform and every orbital has unit
norm, potentials are sums of 8 Gaussian wells, occupations are 2.
"""
import math

import numpy as np
import torch

import paper_0904_1543_gb300 as W

# least-asymmetric Daubechies filter with 8 vanishing moments, h_j, j = -7..8;
# the magic filter w_k, k = -7..8; a_l = int phi phi''(x - l) dx, l = 0..14
_H = (0.001889950332767689, -0.0003029205147241331, -0.014952258337062199, 0.0038087520138944896,
      0.04913717967373029, -0.027219029917103486, -0.0519458381078818, 0.36444189483617895,
      0.777185751699628, 0.4813596512590534, -0.061273359067811076, -0.14329423835127267,
      0.007607487324976609, 0.03169508781152599, -0.0005421323318000107, -0.0033824159510050028)
_WF = (8.433424733352934e-07, -1.290557201342061e-05, 8.76298447621056e-05, -0.00030158038132690465,
      0.001747237136729939, -0.009420470302010804, 0.023738214637249424, 0.0612625895831208,
      0.9940415697834004, -0.06048952891969835, -0.021030251609303816, 0.013372634148547948,
      -0.0034412814449349387, 0.0004944322768868992, -5.185986881173433e-05, 2.7273449291197967e-06)
_A = (-3.55369228991319, 2.2191465938911166, -0.615614146557007, 0.23717805821538057,
      -0.08226639997421234, 0.022070291884822554, -0.004097656893426338, 0.00045167920287502236,
      -2.3982285245075998e-05, 2.0904234952920368e-06, -3.7230763047369276e-07,
      -1.0585705549674146e-08, -5.8138798302825403e-11, 2.7080049362631943e-13,
      -6.9244749406392e-18)

_PREC = {"f64": W.WVL_F64, "f32": W.WVL_F32, "emu": W.WVL_F64_EMU}


def listed():
    return [
        # a single call on one orbital of a 32^3 cell in FP64, density and
        # energies included: a structure's last check, or a code that hands
        # over one orbital at a time; latency and launches count
        {"name": "one orbital f64", "kind": "hpsi", "prec": "f64", "n": "32x32x32", "norb": 1,
         "h": "0.25,0.25,0.25", "density": True},
        # the smallest calls: two orbitals of a small cell in FP32
        {"name": "small cell f32", "kind": "hpsi", "prec": "f32", "n": "16x16x16", "norb": 2,
         "h": "0.25,0.25,0.25", "density": True},
        # the batch of an SCF step in FP64: 192 orbitals on three uneven cells
        {"name": "batch f64", "kind": "plan", "prec": "f64", "n": "56x56x56,48x48x48,40x40x40",
         "norb": "64,64,64", "h": "0.25,0.25,0.25"},
        # the same batch with FP64 accuracy from the tensor cores
        {"name": "batch emu", "kind": "plan", "prec": "emu", "n": "56x56x56,48x48x48,40x40x40",
         "norb": "64,64,64", "h": "0.25,0.25,0.25"},
        # the mixed-precision batch: 256 orbitals of one cell, FP64 density
        {"name": "batch f32", "kind": "plan", "prec": "f32", "n": "48x48x48", "norb": "256",
         "h": "0.25,0.25,0.25"},
        # H applied inside an iterative diagonaliser: a cell whose extents are
        # no multiples of anything, uneven spacings, no density
        {"name": "ragged cell f32", "kind": "hpsi", "prec": "f32", "n": "37x45x51", "norb": 48,
         "h": "0.25,0.3,0.2", "density": False},
        # the differentiable energy of 512 orbitals: forward and backward
        {"name": "eloc f32", "kind": "eloc", "prec": "f32", "n": "64x64x64", "norb": 512,
         "h": "0.25,0.25,0.25"},
        # scalar products of all orbitals, as orthogonalisation needs them,
        # and the expectation values <psi|H psi>
        {"name": "products f32", "kind": "products", "prec": "f32", "n": "48x48x48", "norb": 256,
         "h": "0.25,0.25,0.25"},
        # the preconditioner of the residuals: 5 CG iterations per orbital
        {"name": "preconditioner f32", "kind": "precond", "prec": "f32", "n": "48x48x48",
         "norb": 256, "h": "0.25,0.25,0.25", "iterations": 5},
        # localised orbitals: a ball of radius 12 in a 48^3 cell
        {"name": "region f32", "kind": "region", "prec": "f32", "n": "48x48x48", "norb": 64,
         "h": "0.25,0.25,0.25", "radius": 12.0, "fine_radius": 6.0},
        # an isolated molecule: free conditions on a 32^3 box
        {"name": "free f64", "kind": "bc", "prec": "f64", "n": "32x32x32", "norb": 64,
         "h": "0.25,0.25,0.25", "free": "1,1,1"},
        # the operators alone, both directions, on a batch of orbitals
        {"name": "operators f32", "kind": "operators", "prec": "f32", "n": "40x40x40",
         "norb": 64, "h": "0.25,0.25,0.25"},
    ]


# fine points times orbitals of a drawn case, by precision (per CG iteration
# for the preconditioner): no drawn case costs more than the largest listed one
_POINTS = {"f64": 1.2e8, "emu": 1.6e8, "f32": 4e8}


def _loguniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _extents(rng, lo, hi):
    """Half of the cells have extents that are multiples of 4, the others any."""
    base, unit = _loguniform(rng, lo, hi), rng.choice([1, 4])
    return [max(4, min(80, unit * int(round(base * rng.uniform(0.75, 1.3) / unit))))
            for _ in range(3)]


def _orbitals(rng, lo, hi, points, limit):
    return max(1, min(int(round(_loguniform(rng, lo, hi))), int(limit / points)))


def draw(rng):
    kind = rng.choice(["hpsi", "hpsi", "plan", "plan", "eloc", "products", "precond", "region",
                       "bc", "operators"])
    prec = rng.choice(["f64", "f32", "f32", "emu"])
    limit = _POINTS[prec]
    case = {"kind": kind, "prec": prec,
            "h": rng.choice(["0.25,0.25,0.25", "0.25,0.25,0.25", "0.25,0.3,0.2", "0.31,0.22,0.27"])}
    if kind == "plan":
        ns, cnt = [], []
        cells = rng.randint(1, 4)
        for _ in range(cells):
            n = _extents(rng, 10, 60)
            ns.append("x".join(map(str, n)))
            cnt.append(str(_orbitals(rng, 2, 96, 8 * n[0] * n[1] * n[2], limit / cells)))
        case.update(n=",".join(ns), norb=",".join(cnt))
        return case
    n = _extents(rng, *{"hpsi": (6, 64), "eloc": (8, 64), "products": (8, 56), "precond": (8, 56),
                        "region": (24, 48), "bc": (6, 40), "operators": (8, 80)}[kind])
    points = 8 * n[0] * n[1] * n[2]
    if kind == "bc":
        free = rng.choice([(1, 1, 1), (1, 1, 1), (0, 0, 1), (0, 1, 0), (1, 0, 0), (1, 1, 0)])
        case["free"] = ",".join(map(str, free))
        points = 8 * math.prod(v + 16 * f for v, f in zip(n, free))
    case["n"] = "x".join(map(str, n))
    if kind == "hpsi":
        case.update(norb=_orbitals(rng, 1, 96, points, limit), density=rng.random() < 0.5)
    elif kind == "eloc":
        case["norb"] = _orbitals(rng, 2, 512, points, limit / 2)
    elif kind == "products":
        most = int(math.sqrt(2.5e10 / points))
        case["norb"] = max(2, min(most, int(_loguniform(rng, 4, 320))))
    elif kind == "precond":
        case["iterations"] = rng.randint(3, 8)
        case["norb"] = _orbitals(rng, 4, 256, points * case["iterations"], 2 * limit)
    elif kind == "region":
        r = rng.uniform(0.15, 0.45) * min(n)
        case.update(norb=_orbitals(rng, 4, 64, points, limit), radius=round(r, 2),
                    fine_radius=round(r * rng.uniform(0.4, 0.8), 2))
    else:
        case["norb"] = _orbitals(rng, 4, 96, points, limit)
    return case


# ------------------------------------------------------------------ inputs
def _ints(text, sep):
    return [int(v) for v in str(text).split(sep)]


def _cells(case):
    return [tuple(_ints(n, "x")) for n in case["n"].split(",")]


def _counts(case):
    return _ints(case["norb"], ",")


def _spacing(case):
    return tuple(float(v) for v in case["h"].split(","))


def _dtype(case):
    return torch.float32 if case["prec"] == "f32" else torch.float64


def _vectors(gen, norb, length, dtype):
    """Unit-norm vectors of uniform[-1, 1) coefficients."""
    x = torch.rand((norb, length), generator=gen, device="cuda", dtype=dtype)
    x.mul_(2.0).sub_(1.0)
    for o in range(0, norb, 64):
        x[o:o + 64] /= torch.linalg.vector_norm(x[o:o + 64], dim=1, keepdim=True)
    return x


def _potential(rs, shape, origin, periodic):
    """Sum of 8 Gaussian wells on a fine grid of `shape` (N3, N2, N1) whose
    first point sits at -origin, in float64 on the device."""
    inner = [s - 2 * o for s, o in zip(shape, origin)]
    v = torch.zeros(shape, dtype=torch.float64, device="cuda")
    for _ in range(8):
        centre = [rs.uniform(0.0, m) for m in inner]
        sigma, depth = rs.uniform(2.0, 6.0), rs.uniform(-2.0, 0.0)
        f = []
        for s, o, c, p in zip(shape, origin, centre, periodic):
            x = torch.arange(s, dtype=torch.float64, device="cuda") - o - c
            if p:
                x = x - s * torch.round(x / s)
            f.append(torch.exp(-x * x / (2.0 * sigma * sigma)))
        v += depth * f[0][:, None, None] * f[1][None, :, None] * f[2][None, None, :]
    return v


def _masks(case):
    """Coarse and fine masks (n3, n2, n1) of balls around the same centre."""
    n = _cells(case)[0]
    d2 = np.zeros((n[2], n[1], n[0]))
    for axis, v in enumerate((n[2], n[1], n[0])):
        x = np.arange(v) - (0.1 + 0.3 * axis) * v
        x = x - v * np.round(x / v)
        shape = [1, 1, 1]
        shape[axis] = v
        d2 = d2 + (x * x).reshape(shape)
    return d2 <= case["radius"] ** 2, d2 <= case["fine_radius"] ** 2


def _inputs(case, seed):
    """The arrays of a case; `exact` makes the same ones."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rs = np.random.RandomState((seed * 7919 + 17) % (1 << 32))
    kind, dtype = case["kind"], _dtype(case)
    cells, counts = _cells(case), _counts(case)
    total = sum(counts)
    a = {"occ": torch.full((total,), 2.0, dtype=torch.float64, device="cuda")}
    if kind == "plan":
        a["psi"] = torch.cat([_vectors(gen, c, 8 * math.prod(n), dtype).reshape(-1)
                              for n, c in zip(cells, counts)])
        a["V"] = [_potential(rs, (2 * n[2], 2 * n[1], 2 * n[0]), (0, 0, 0), (True,) * 3).to(dtype)
                  for n in cells]
        return a
    n = cells[0]
    length = 8 * math.prod(n)
    if kind == "region":
        a["masks"] = _masks(case)
        length = int(a["masks"][0].sum()) + 7 * int(a["masks"][1].sum())
    a["psi"] = _vectors(gen, total, length, dtype)
    if kind == "products":
        a["hpsi"] = _vectors(gen, total, length, dtype)
    elif kind == "precond":
        a["eps"] = torch.from_numpy(-rs.uniform(0.2, 1.5, total)).cuda()
    elif kind != "operators":
        free = _ints(case.get("free", "0,0,0"), ",")
        pad = [16 * f for f in free][::-1]
        shape = [2 * v + 2 * p for v, p in zip(n[::-1], pad)]
        a["V"] = _potential(rs, tuple(shape), pad, [not f for f in free[::-1]]).to(dtype)
    return a


_compute = None


def _stream():
    """The program's compute stream."""
    global _compute
    if _compute is None:
        _compute = torch.cuda.Stream()
    return _compute


def prepare(case, seed):
    s = _inputs(case, seed)
    kind, h = case["kind"], _spacing(case)
    s["kind"], s["emu"] = kind, case["prec"] == "emu"
    if kind == "plan":
        s["grids"] = [W.Grid(n, h) for n in _cells(case)]
        of = [c for c, m in enumerate(_counts(case)) for _ in range(m)]
        s["plan"] = W.Plan(s["grids"], of, prec=_PREC[case["prec"]], graph=True)
        s["out"] = torch.empty_like(s["psi"])
        s["rho"] = [torch.zeros(g.fine, dtype=torch.float64, device="cuda") for g in s["grids"]]
        s["ekin"] = torch.empty(len(of), dtype=torch.float64, device="cuda")
        s["epot"] = torch.empty_like(s["ekin"])
        _stream().wait_stream(torch.cuda.current_stream())
        return s
    s["grid"] = W.Grid(_cells(case)[0], h)
    if kind == "hpsi":
        s["density"] = bool(case["density"])
    elif kind == "eloc":
        s["psi"].requires_grad_(True)
        s["V"].requires_grad_(True)
    elif kind == "precond":
        s["iterations"] = int(case["iterations"])
    elif kind == "region":
        s["region"] = W.Region(s["grid"], *s["masks"])
    elif kind == "bc":
        s["free"] = tuple(_ints(case["free"], ","))
    return s


def run(s):
    kind, emu = s["kind"], s["emu"]
    if kind == "plan":
        with torch.cuda.stream(_stream()):
            for r in s["rho"]:
                r.zero_()
            s["plan"].hpsi(s["psi"], s["V"], s["occ"], hpsi=s["out"], rho=s["rho"],
                           ekin=s["ekin"], epot=s["epot"])
        return {"hpsi": s["out"], "rho": s["rho"], "ekin": s["ekin"], "epot": s["epot"]}
    g, psi = s["grid"], s["psi"]
    if kind == "hpsi":
        rho = torch.zeros(g.fine, dtype=torch.float64, device="cuda") if s["density"] else None
        hpsi, ekin, epot = W.hpsi_local(psi, s["V"], s["occ"], g, rho=rho, emu=emu)
        return {"hpsi": hpsi, "rho": rho, "ekin": ekin, "epot": epot}
    if kind == "eloc":
        e = W.ELoc.apply(psi, s["V"], s["occ"], g, emu)
        dpsi, dv = torch.autograd.grad(e, (psi, s["V"]))
        return {"energy": e, "dpsi": dpsi, "dV": dv}
    if kind == "products":
        return {"overlap": W.overlap(psi), "dot": W.dot(psi, s["hpsi"])}
    if kind == "precond":
        x, _ = W.precondition(psi, s["eps"], g, ncg=s["iterations"], want_residual=False, emu=emu)
        return {"x": x}
    if kind == "region":
        hpsi, ekin, epot = W.hpsi_local_region(psi, s["V"], s["occ"], g, s["region"], emu=emu)
        return {"hpsi": hpsi, "ekin": ekin, "epot": epot}
    if kind == "bc":
        rho = torch.zeros(W.bc_fine(g, s["free"]), dtype=torch.float64, device="cuda")
        hpsi, ekin, epot = W.hpsi_local_bc(psi, s["V"], s["occ"], g, s["free"], rho=rho, emu=emu)
        return {"hpsi": hpsi, "rho": rho, "ekin": ekin, "epot": epot}
    fine = W.synthesis(psi, g, emu=emu)
    real = W.magicfilter(fine, g, emu=emu)
    back = W.magicfilter_T(real, g, emu=emu)
    z, ekin = W.kinetic(fine, g, k0=back, emu=emu)
    return {"s": fine, "psi_r": real, "y": back, "z": z, "ekin": ekin,
            "c": W.analysis(z, g, emu=emu)}


# multiply-adds per fine point and axis: the 16-tap filters and the 29-tap one
_TAP, _KIN = 16, 29


def work(case):
    kind, cells, counts = case["kind"], _cells(case), _counts(case)
    size = 4 if case["prec"] == "f32" else 8
    pts = [8 * math.prod(n) for n in cells]
    orb = sum(p * c for p, c in zip(pts, counts))
    if kind == "plan" or kind == "hpsi":
        cell = sum(pts)
        density = 16 * cell if kind == "plan" or case["density"] else 0
        return {"bytes": 2 * size * orb + size * cell + density + 24 * sum(counts),
                "flops": 2 * orb * (12 * _TAP + 3 * _KIN + 4)}
    if kind == "eloc":
        forward = 6 * _TAP + 3 * _KIN + 4
        return {"bytes": 2 * size * orb + 2 * size * pts[0] + 8 * sum(counts),
                "flops": 2 * orb * (forward + 12 * _TAP + 3 * _KIN + 1)}
    if kind == "products":
        c = counts[0]
        return {"bytes": 2 * size * orb + 8 * c * c + 8 * c, "flops": orb * (c + 1) + 2 * orb}
    if kind == "precond":
        return {"bytes": 2 * size * orb + 8 * counts[0],
                "flops": 2 * orb * case["iterations"] * (6 * _TAP + 3 * _KIN + 6)}
    if kind == "region":
        # the ball's points and the filters' reach around them
        r = case["radius"]
        ball, fine = (4.0 / 3.0 * math.pi * v ** 3 for v in (r, case["fine_radius"]))
        near = min(8 * (2 * r + 8) ** 3, pts[0])
        return {"bytes": counts[0] * 2 * size * (ball + 7 * fine) + size * near + 8 * math.prod(cells[0]),
                "flops": 2 * counts[0] * near * (12 * _TAP + 3 * _KIN + 4)}
    if kind == "bc":
        free = _ints(case["free"], ",")
        cell = 8 * math.prod(v + 16 * f for v, f in zip(cells[0], free))
        return {"bytes": 2 * size * orb + (size + 16) * cell + 24 * counts[0],
                "flops": 2 * orb * (12 * _TAP + 3 * _KIN + 4)}
    return {"bytes": 6 * size * orb + 8 * counts[0], "flops": 2 * orb * (12 * _TAP + 3 * _KIN)}


# ------------------------------------------------- the same in plain 64 bits
def _line(lo, n, periodic, entries):
    """Matrix rows lo .. lo + n - 1 of a 1D operator: entries(i) gives the
    (column, value) pairs of row i; columns wrap on a periodic line."""
    m = np.zeros((n, n))
    for r in range(n):
        for c, v in entries(r + lo):
            c -= lo
            if periodic:
                m[r, c % n] += v
            elif 0 <= c < n:
                m[r, c] += v
    return m


def _filters(nc, h, free):
    """The 1D operators of an axis of nc coarse points: (S, M, T) and the
    fine points kept of the coarse and of the padded range.  On a free axis the
    line is long enough for every filter, and nothing wraps."""
    lo, n = (-64, 2 * nc + 128) if free else (0, 2 * nc)
    hf = {j: _H[j + 7] for j in range(-7, 9)}
    gf = {j: (-1) ** j * hf[1 - j] for j in range(-7, 9)}

    def synthesis(i):
        for j in range((i - 9) // 2, (i + 9) // 2 + 1):
            yield 2 * j, hf.get(i - 2 * j, 0.0)
            yield 2 * j + 1, gf.get(i - 2 * j, 0.0)

    s = _line(lo, n, not free, synthesis)
    m = _line(lo, n, not free, lambda i: [(i - k, _WF[k + 7]) for k in range(-7, 9)])
    t = _line(lo, n, not free,
              lambda i: [(i - k, -_A[abs(k)] / (2.0 * h * h)) for k in range(-14, 15)])
    box = slice(-lo, -lo + 2 * nc)
    pad = slice(-lo - 16, -lo + 2 * nc + 16) if free else box
    return s, m, t, box, pad


def _dev(m):
    return torch.from_numpy(np.ascontiguousarray(m)).cuda()


def _along(x, m, axis):
    """The matrix m along `axis` (1, 2, 3 = x, y, z) of (orbital, z, y, x) arrays."""
    return torch.movedim(torch.movedim(x, 4 - axis, -1) @ m.T, -1, 4 - axis)


def _three(x, ms):
    for axis in (1, 2, 3):
        x = _along(x, ms[axis - 1], axis)
    return x.contiguous()


def _spread(psi, n, masks=None):
    """Compressed coefficients -> interleaved (orbital, z, y, x) arrays."""
    n1, n2, n3 = n
    m = n1 * n2 * n3
    x = torch.zeros((psi.shape[0], 2 * n3, 2 * n2, 2 * n1), dtype=torch.float64, device="cuda")
    if masks is None:
        scaling = psi[:, :m]
        wavelet = psi[:, m:].reshape(-1, m, 7)
    else:
        coarse, fine = (torch.from_numpy(np.flatnonzero(v)).cuda() for v in masks)
        scaling = torch.zeros((psi.shape[0], m), dtype=torch.float64, device="cuda")
        wavelet = torch.zeros((psi.shape[0], m, 7), dtype=torch.float64, device="cuda")
        scaling[:, coarse] = psi[:, :coarse.numel()]
        wavelet[:, fine] = psi[:, coarse.numel():].reshape(-1, fine.numel(), 7)
    x[:, ::2, ::2, ::2] = scaling.reshape(-1, n3, n2, n1)
    for mu in range(1, 8):
        x[:, mu >> 2::2, mu >> 1 & 1::2, mu & 1::2] = wavelet[..., mu - 1].reshape(-1, n3, n2, n1)
    return x


def _gather(x, n, masks=None):
    m = n[0] * n[1] * n[2]
    scaling = x[:, ::2, ::2, ::2].reshape(-1, m)
    wavelet = torch.stack([x[:, mu >> 2::2, mu >> 1 & 1::2, mu & 1::2].reshape(-1, m)
                           for mu in range(1, 8)], dim=2)
    if masks is not None:
        coarse, fine = (torch.from_numpy(np.flatnonzero(v)).cuda() for v in masks)
        scaling, wavelet = scaling[:, coarse], wavelet[:, fine]
    return torch.cat([scaling, wavelet.reshape(x.shape[0], -1)], dim=1)


def _operators(n, h, free=(0, 0, 0)):
    """Per axis: coefficients -> real-space values, and the kinetic operator
    between coefficients."""
    real, kin = [], []
    for d in range(3):
        s, m, t, box, pad = _filters(n[d], h[d], free[d])
        real.append(_dev((m @ s)[pad, box]))
        kin.append(_dev((s.T @ t @ s)[box, box]))
    return real, kin


def _hamiltonian(psi, v, occ, n, h, free=(0, 0, 0), masks=None):
    """(H psi, density, Ekin, Epot), a few orbitals at a time."""
    real, kin = _operators(n, h, free)
    back = [m.T for m in real]
    v = v.double()
    rho = torch.zeros(v.shape, dtype=torch.float64, device="cuda")
    hpsi, ekin, epot = [], [], []
    step = max(1, int(5e7 / v.numel()))
    for o in range(0, psi.shape[0], step):
        x = _spread(psi[o:o + step].double(), n, masks)
        r = _three(x, real)
        rho += torch.einsum("o,ozyx->zyx", occ[o:o + step], r * r)
        epot.append((v * r * r).sum(dim=(1, 2, 3)))
        k = sum(_along(x, kin[d], d + 1) for d in range(3))
        ekin.append((x * k).sum(dim=(1, 2, 3)))
        hpsi.append(_gather(_three(v * r, back) + k, n, masks))
    return torch.cat(hpsi), rho, torch.cat(ekin), torch.cat(epot)


def _preconditioned(g, eps, n, h, iterations):
    """x after the given number of CG iterations for (K - eps) x = g,
    preconditioned by the operator's diagonal, from x = 0."""
    _, kin = _operators(n, h)
    diag = torch.zeros((2 * n[2], 2 * n[1], 2 * n[0]), dtype=torch.float64, device="cuda")
    for d in range(3):
        shape = [1, 1, 1]
        shape[2 - d] = -1
        diag += torch.diagonal(kin[d]).reshape(shape)
    out = []
    step = max(1, int(5e7 / diag.numel()))
    for o in range(0, g.shape[0], step):
        r = _spread(g[o:o + step].double(), n)
        e = eps[o:o + step, None, None, None]
        x = torch.zeros_like(r)
        z = r / (diag - e)
        p = z.clone()
        rz = (r * z).sum(dim=(1, 2, 3), keepdim=True)
        for _ in range(iterations):
            q = sum(_along(p, kin[d], d + 1) for d in range(3)) - e * p
            alpha = rz / (p * q).sum(dim=(1, 2, 3), keepdim=True)
            x += alpha * p
            r = r - alpha * q
            z = r / (diag - e)
            new = (r * z).sum(dim=(1, 2, 3), keepdim=True)
            p = z + (new / rz) * p
            rz = new
        out.append(_gather(x, n))
    return torch.cat(out)


def exact(case, seed):
    a = _inputs(case, seed)
    kind, cells, counts, h = case["kind"], _cells(case), _counts(case), _spacing(case)
    if kind == "plan":
        res = {"hpsi": [], "rho": [], "ekin": [], "epot": []}
        at = first = 0
        for n, c, v in zip(cells, counts, a["V"]):
            length = 8 * math.prod(n)
            psi = a["psi"][at:at + c * length].reshape(c, length)
            for key, val in zip(res, _hamiltonian(psi, v, a["occ"][first:first + c], n, h)):
                res[key].append(val if key == "rho" else val.reshape(-1))
            at, first = at + c * length, first + c
        return {k: v if k == "rho" else torch.cat(v) for k, v in res.items()}
    n, psi = cells[0], a["psi"]
    if kind in ("hpsi", "region", "bc"):
        free = tuple(_ints(case.get("free", "0,0,0"), ","))
        hpsi, rho, ekin, epot = _hamiltonian(psi, a["V"], a["occ"], n, h, free, a.get("masks"))
        res = {"hpsi": hpsi, "rho": rho, "ekin": ekin, "epot": epot}
        if kind == "region":
            del res["rho"]
        elif kind == "hpsi" and not case["density"]:
            res["rho"] = None
        return res
    if kind == "eloc":
        dpsi, rho, ekin, epot = _hamiltonian(psi, a["V"], a["occ"], n, h)
        for o in range(0, psi.shape[0], 64):
            dpsi[o:o + 64] *= 2.0 * a["occ"][o:o + 64, None]
        return {"energy": (a["occ"] * (ekin + epot)).sum(), "dpsi": dpsi, "dV": rho}
    if kind == "products":
        s = torch.zeros((psi.shape[0],) * 2, dtype=torch.float64, device="cuda")
        d = torch.zeros(psi.shape[0], dtype=torch.float64, device="cuda")
        for k in range(0, psi.shape[1], 8192):
            p = psi[:, k:k + 8192].double()
            s += p @ p.T
            d += (p * a["hpsi"][:, k:k + 8192].double()).sum(dim=1)
        return {"overlap": s, "dot": d}
    if kind == "precond":
        return {"x": _preconditioned(psi, a["eps"], n, h, int(case["iterations"]))}
    ss, ms, ts = [], [], []
    for d in range(3):
        s, m, t, _, _ = _filters(n[d], h[d], 0)
        ss.append(_dev(s))
        ms.append(_dev(m))
        ts.append(_dev(t))
    fine = _three(_spread(psi.double(), n), ss)
    real = _three(fine, ms)
    back = _three(real, [m.T for m in ms])
    k = sum(_along(fine, ts[d], d + 1) for d in range(3))
    z = back + k
    return {"s": fine, "psi_r": real, "y": back, "z": z, "ekin": (fine * k).sum(dim=(1, 2, 3)),
            "c": _gather(_three(z, [s.T for s in ss]), n)}
