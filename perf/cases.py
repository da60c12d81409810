"""The work that a user of this library has it do, as cases that can be timed
and whose outputs can be compared.

A case is a dict of plain values.  ``kind`` says which public call one pass is:

* ``push``  one PSATD step of every box (``Solver.push``), Maxwell's equations;
* ``heat``  one step of the heat equation (``HeatSolver.push``);
* ``yee``   one finite-difference step on a periodic grid (``YeeSolver.step``);
* ``io``    what a particle code moves in a step: J and rho from the global
  grid into the padded boxes, the valid E and B back (``psatd_scatter_global``,
  ``psatd_gather_global``).

``cx``, ``cy``, ``cz`` are the widths of the boxes along each axis, ``ng`` and
``p`` the guard widths and stencil orders that the boxes take in turn.
"""
import math

import torch

from paper_1707_08500_gb300 import fdtd as F
from paper_1707_08500_gb300 import inputs as I
from paper_1707_08500_gb300 import psatd as P

EB = ("Ex", "Ey", "Ez", "Bx", "By", "Bz")
J = ("Jx", "Jy", "Jz")
C_DT = 0.5          # c dt (and D dt of the heat equation) with cells of size 1
DEVICE = "cuda"


def _case(name, kind, cuts, ng=0, p=0, precision="f32", gauss=False, staggered=False, two_d=False, source=False):
    c = {"kind": kind, "cx": cuts[0], "cy": cuts[1], "cz": cuts[2], "ng": str(ng), "p": str(p),
         "precision": precision, "gauss": gauss, "staggered": staggered, "two_d": two_d, "source": source}
    return dict(c, name=name) if name else c


def _same(n, count):
    return " ".join([str(n)] * count)


def listed():
    return [
        # the smallest box in use, one periodic 32^3 in double precision:
        # launches and latency
        _case("box32_f64", "push", ("32", "32", "32"), precision="f64"),
        # a small staggered (Yee-positioned) run in double precision with the
        # Gauss diagnostic: eight local boxes of 48^3
        _case("boxes48_f64_staggered", "push", (_same(32, 2),) * 3, 8, 32, "f64", gauss=True, staggered=True),
        # the same size in single precision: a test problem, or a rank's share
        # of a strongly scaled run
        _case("boxes48_f32", "push", (_same(32, 2),) * 3, 8, 16, gauss=True),
        # a load-balanced decomposition: 48 boxes of unequal sizes, guards and
        # orders
        _case("uneven48_f32", "push", ("56 24 72 40", "48 64 32", "48 32 64 48"), "16 8", "32 16 64", gauss=True),
        # the ordinary run: 64 boxes of 64^3 with 16 guards, no diagnostic
        _case("boxes96_f32", "push", (_same(64, 4),) * 3, 16, 64),
        # the largest: 512 boxes of 64^3 at the paper's order 100, with the
        # Gauss diagnostic
        _case("mirror512_f32", "push", (_same(64, 8),) * 3, 16, 100, gauss=True),
        # a decomposition cut to fit a geometry: local lengths with factors 2,
        # 3, 5, 7, 11 and 13, odd ones among them
        _case("ragged_f32", "push", ("68 50 42", "53 45 89", "44 56 65"), 5, 8),
        # the global solver: one periodic box over the grid
        _case("global256_f32", "push", ("256", "256", "256"), 0, 64),
        # a two-dimensional run
        _case("plane2048_f32", "push", (_same(64, 32), _same(64, 32), "1"), 16, 64, gauss=True, two_d=True),
        # the heat equation with a source on the ordinary decomposition
        _case("heat96_f32", "heat", (_same(64, 4),) * 3, 16, 16, source=True),
        # the finite-difference solver that the method is compared with
        _case("yee_f32", "yee", ("768", "320", "250")),
        # what a particle code moves into and out of the boxes in every step
        _case("io96_f32", "io", (_same(64, 4), _same(64, 4), _same(64, 4)), 16, 64, gauss=True),
    ]


# ---- drawn cases -----------------------------------------------------------------
def _length_ok(n):
    """A transform length: a product of two factors of at most 16."""
    return any(n % a == 0 and n // a <= 16 for a in range(1, 17))


def _widths(rng, count, g, lo, hi, even):
    """`count` valid widths in [lo, hi] whose padded lengths can be transformed."""
    fit = [n for n in range(lo, hi + 1)
           if (_length_ok((n + 2 * g) // 2) and n % 2 == 0 if even else _length_ok(n + 2 * g))]
    return [rng.choice(fit) for _ in range(count)]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["push", "push", "push", "push", "push64", "push64", "plane", "global", "heat", "yee", "io"])
    if what == "yee":
        # at most 134 M cells
        n = [_log(rng, 24, 600), _log(rng, 24, 500), _log(rng, 24, 400)]
        return _case(None, "yee", tuple(str(v) for v in n), precision=rng.choice(["f32", "f32", "f64"]) if max(n) < 300 else "f32")
    if what == "global":
        x, y, z = (_log(rng, 24, 256) for _ in range(3))
        while not _length_ok(x // 2):
            x += 1
        x -= x % 2
        while not _length_ok(y):
            y -= 1
        while not _length_ok(z):
            z -= 1
        return _case(None, "push", (str(x), str(y), str(z)), 0, rng.choice([0, 16, 64]), gauss=rng.random() < 0.5)
    if what == "plane":
        g = rng.choice([8, 16])
        nb = _log(rng, 2, 40)
        if rng.random() < 0.5:
            cut = _same(rng.choice([32, 64]), nb)
            return _case(None, "push", (cut, cut, "1"), g, rng.choice([16, 64]), gauss=rng.random() < 0.5, two_d=True)
        cx = _widths(rng, min(nb, 12), g, 24, 88, True)
        cy = _widths(rng, min(nb, 12), g, 24, 88, False)
        return _case(None, "push", (" ".join(map(str, cx)), " ".join(map(str, cy)), "1"), g, rng.choice([16, 64]), two_d=True)
    # boxes: uniform cubes of the usual sizes, or uneven ones; up to 216 boxes
    # in single precision and 27 in double
    f64 = what == "push64"
    most = 3 if f64 else 6
    nb = [rng.randint(1, most) for _ in range(3)]
    form = rng.random()
    if form < 0.45:
        n, g = rng.choice([(64, 16), (32, 16), (32, 8), (48, 8), (32, 0), (64, 8), (48, 16)])
        if f64 and n == 64:
            n, g = 32, 8
        cuts = tuple(_same(n, k) for k in nb)
        ng, p = g, rng.choice([8, 16, 64, 100])
    elif form < 0.7:
        cuts = tuple(" ".join(str(rng.choice([24, 40, 56, 72][:2 if f64 else 4] if a == 0 else [32, 48, 64][:2 if f64 else 3]))
                              for _ in range(min(k, 4))) for a, k in enumerate(nb))
        ng, p = "8 16", "16 32 64"
    else:
        g = rng.randint(3, 9)
        hi = 44 if f64 else 90
        cuts = tuple(" ".join(map(str, _widths(rng, min(k, 3), g, 16, hi, a == 0))) for a, k in enumerate(nb))
        ng, p = g, rng.choice([2, 8, 32])
    kind = what if what in ("heat", "io") else "push"
    return _case(None, kind, cuts, ng, p, "f64" if f64 else "f32",
                 gauss=kind == "io" or (kind == "push" and rng.random() < 0.5),
                 staggered=kind == "push" and rng.random() < 0.25, source=kind == "heat" and rng.random() < 0.7)


# ---- the decomposition of a case ---------------------------------------------------
def _grid(case):
    cuts = [[int(v) for v in case[k].split()] for k in ("cx", "cy", "cz")]
    return cuts, tuple(sum(c) for c in cuts)


def _boxes(case):
    """[(lo, n, guards (x, y, z), order)], x fastest; guard widths and orders are
    taken in turn from the case's lists."""
    cuts, _ = _grid(case)
    ngs, ps = [int(v) for v in case["ng"].split()], [int(v) for v in case["p"].split()]
    boxes, oz = [], 0
    for iz, wz in enumerate(cuts[2]):
        oy = 0
        for iy, wy in enumerate(cuts[1]):
            ox = 0
            for ix, wx in enumerate(cuts[0]):
                g, p = ngs[(ix + 3 * iy + 5 * iz) % len(ngs)], ps[(2 * ix + iy + 3 * iz) % len(ps)]
                boxes.append(((ox, oy, oz), (wx, wy, wz), (g, g, 0 if case["two_d"] else g), p))
                ox += wx
            oy += wy
        oz += wz
    return boxes


def _workload(case):
    _, gn = _grid(case)
    subs = [I.Sub(lo, n, g[0], p, zguard=not case["two_d"]) for lo, n, g, p in _boxes(case)]
    return I.Workload(case.get("name", "drawn"), gn, subs, "broadband", 1, case["precision"], 1707,
                      c_dt=C_DT, staggered=case["staggered"], two_d=case["two_d"])


def _names(case):
    if case["kind"] == "heat":
        return ("T", "S") if case["source"] else ("T",)
    if case["kind"] == "yee":
        return EB + J
    return EB + J + (("rho",) if case["gauss"] else ())


def _fields(case, seed):
    """Global [Nz][Ny][Nx] fields: a wave packet (eight cells per wavelength)
    over broadband noise for E and B; noise for the currents, the charge and a
    heat source."""
    _, (nx, ny, nz) = _grid(case)
    dt = torch.float64 if case["precision"] == "f64" else torch.float32
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)
    ax = [torch.arange(n, device=DEVICE, dtype=dt) - n / 2 for n in (nx, ny, nz)]
    w = max(6.0, nx / 8)
    ex, ey, ez = (torch.exp(-(a / w) ** 2) for a in ax)
    out = {}
    for name in _names(case):
        t = torch.empty((nz, ny, nx), device=DEVICE, dtype=dt).normal_(0.0, 0.05 if name[0] in "JS" else 0.25, generator=gen)
        if name in ("Ey", "Bz", "T"):
            t += (torch.cos(ax[0] * (2 * math.pi / 8)) * ex)[None, None, :] * ey[None, :, None] * ez[:, None, None]
        out[name] = t
    return out


# ---- one pass -------------------------------------------------------------------------
def prepare(case, seed):
    glob = _fields(case, seed)
    if case["kind"] == "yee":
        _, gn = _grid(case)
        s = F.YeeSolver(gn, C_DT, precision=case["precision"], device=DEVICE)
        s.load(glob)
        return {"case": case, "solver": s}
    wl = _workload(case)
    if case["kind"] == "heat":
        s = P.HeatSolver(wl, C_DT, source=case["source"], device=DEVICE)
    else:
        s = P.Solver(wl, gauss=case["gauss"], device=DEVICE)
    stream = torch.cuda.current_stream().cuda_stream
    names = [n for n in glob if case["kind"] != "io" or n in EB]
    P.psatd_scatter_global(s.plan, [glob[n] for n in names], [s.arenas[n] for n in names], stream)
    state = {"case": case, "solver": s}
    if case["kind"] == "io":
        state["sources"] = [glob[n] for n in J + ("rho",)]
        state["out"] = [torch.empty_like(glob[n]) for n in EB]
    return state


def run(state):
    s, case = state["solver"], state["case"]
    if case["kind"] == "yee":
        s.step()
        f = s.fields
        return {n: f[n] for n in EB}
    if case["kind"] == "io":
        stream = torch.cuda.current_stream().cuda_stream
        arenas = [s.arenas[n] for n in J + ("rho",)]
        P.psatd_scatter_global(s.plan, state["sources"], arenas, stream)
        P.psatd_gather_global(s.plan, [s.arenas[n] for n in EB], state["out"], stream)
        return {"boxes": arenas, "grid": state["out"]}
    s.push()
    out = {n: s.arenas[n] for n in (("T",) if case["kind"] == "heat" else EB)}
    if case["gauss"]:
        out["gauss"] = s.gauss_out
    return out


# ---- what a pass cannot do without ------------------------------------------------------
def work(case):
    """Bytes: each input cell of every padded box read once, each output cell
    written once.  Operations of the push: the real transforms of every input
    field forward (5/2 N log2 N for N cells) and of every output back (only the
    valid planes and rows after the z and y parts), and 250 (Maxwell) or 6
    (heat) per half-spectrum mode."""
    sz = 8 if case["precision"] == "f64" else 4
    _, gn = _grid(case)
    cells = gn[0] * gn[1] * gn[2]
    if case["kind"] == "yee":
        return {"bytes": 15 * sz * cells, "flops": 36 * cells}
    local = [tuple(n[a] + 2 * g[a] for a in range(3)) + n for _, n, g, _ in _boxes(case)]
    padded = sum(b[0] * b[1] * b[2] for b in local)
    if case["kind"] == "io":
        return {"bytes": sz * (4 * (cells + padded) + 6 * 2 * cells), "flops": 0}
    nin = len(_names(case))
    nout, per_mode = (1, 6) if case["kind"] == "heat" else (6, 250)
    flops = 0.0
    for lx, ly, lz, _, vy, vz in local:
        lg = [math.log2(v) for v in (lx, ly, lz)]
        n = lx * ly * lz
        flops += nin * 2.5 * n * sum(lg) + per_mode * (lx // 2 + 1) * ly * lz
        flops += nout * 2.5 * n * (lg[2] + lg[1] * vz / lz + lg[0] * vz / lz * vy / ly)
    return {"bytes": sz * (nin + nout) * padded, "flops": flops}


# Measured against exact(), in the 2-norm: 2.6e-7 at most in single precision,
# 7e-16 in double, and 8e-15 on staggered grids in double (the rounding of the
# high-order staggered weights); the Gauss sums are nearer, since the drawn
# charge is far from the fields' divergence.  Copies are copies.
def tolerance(case):
    if case["kind"] == "io":
        return "exact"
    if case["precision"] == "f32":
        return {"rel": 1e-6}
    return {"rel": 3e-14 if case["staggered"] else 4e-15}


# ---- the same in 64 bits, in plain torch --------------------------------------------------
def _weights(p, staggered):
    m = p // 2
    if not staggered:
        w = [m / (m + 1.0)]
        for j in range(1, m):
            w.append(-w[-1] * j * (m - j) / ((j + 1.0) * (m + j + 1.0)))
        return w
    # c_1 = ((2m-1)!!)^2 / (4^(m-1) m! (m-1)!)
    odd = math.prod(range(1, 2 * m, 2))
    c = [odd * odd / (4 ** (m - 1) * math.factorial(m) * math.factorial(m - 1))]
    for j in range(1, m):
        c.append(-c[-1] * (2 * j - 1) ** 2 * (m - j) / ((2 * j + 1) ** 2 * (m + j)))
    return c


def _freq(n, half):
    f = (torch.fft.rfftfreq if half else torch.fft.fftfreq)(n, dtype=torch.float64, device=DEVICE) * (2 * math.pi)
    if n % 2 == 0:
        f[n // 2] = -math.pi
    return f


def _modified(n, half, p, staggered, keep_nyquist=False):
    k = _freq(n, half)
    if p == 0:
        s = k.clone()
    else:
        s = torch.zeros_like(k)
        for j, w in enumerate(_weights(p, staggered)):
            s += 2 * w * torch.sin((j + 0.5) * k) if staggered else 2 * w * torch.sin((j + 1) * k)
    if n % 2 == 0 and not keep_nyquist:
        s[n // 2] = 0.0
    return s


def _axes(v):
    return v[0][None, None, :], v[1][None, :, None], v[2][:, None, None]


def _maxwell(box, p, staggered, gauss):
    """One step of one padded box (E, B, J and rho in 64 bits): E, B and the two
    Gauss sums."""
    lz, ly, lx = box["Ex"].shape
    kx, ky, kz = _axes([_modified(n, n_ax == 0, p, staggered) for n_ax, n in enumerate((lx, ly, lz))])
    k = torch.sqrt(kx * kx + ky * ky + kz * kz)
    one = torch.ones_like(k)
    ks = torch.where(k > 0, k, one)
    inv = torch.where(k > 0, 1 / ks, 0 * one)
    x = k * C_DT
    c, s = torch.cos(x), torch.sin(x)
    omc = 2 * torch.sin(x / 2) ** 2
    sk = torch.where(k > 0, s / ks, C_DT * one)
    omck = omc * inv
    dk = torch.where(x.abs() < 1e-3, C_DT * (-x * x / 6 + x ** 4 / 120), sk - C_DT)
    h = [kx * inv, ky * inv, kz * inv]
    f = {n: torch.fft.rfftn(box[n]) for n in box}
    shift = {}
    if staggered:
        ph = _axes([torch.exp(-0.5j * _freq(n, a == 0)) for a, n in enumerate((lx, ly, lz))])
        for a, n in enumerate("xyz"):
            shift["E" + n] = shift["J" + n] = ph[a]
            shift["B" + n] = ph[(a + 1) % 3] * ph[(a + 2) % 3]
        for n in shift:
            f[n] = f[n] * shift[n]
    e, b, j = ([f[q + n] for n in "xyz"] for q in "EBJ")

    def cross(u):
        return [h[(a + 1) % 3] * u[(a + 2) % 3] - h[(a + 2) % 3] * u[(a + 1) % 3] for a in range(3)]

    def dot(u):
        return h[0] * u[0] + h[1] * u[1] + h[2] * u[2]

    he, hb, hj, de, dj = cross(e), cross(b), cross(j), dot(e), dot(j)
    e2 = [c * e[a] + 1j * s * hb[a] - sk * j[a] + h[a] * (omc * de + dk * dj) for a in range(3)]
    b2 = [c * b[a] - 1j * s * he[a] + 1j * omck * hj[a] for a in range(3)]
    sums = None
    if gauss:
        wgt = torch.full((lx // 2 + 1,), 2.0, dtype=torch.float64, device=DEVICE)
        wgt[0] = wgt[-1] = 1.0
        res = 1j * (kx * e2[0] + ky * e2[1] + kz * e2[2]) - f["rho"]
        sums = [float((wgt * v.abs() ** 2).sum()) for v in (res, f["rho"])]
    out = {}
    for q, v in (("E", e2), ("B", b2)):
        for a, n in enumerate("xyz"):
            t = v[a] / shift[q + n] if staggered else v[a]
            out[q + n] = torch.fft.irfftn(t, s=(lz, ly, lx))
    return out, sums


def _heat(box, p):
    lz, ly, lx = box["T"].shape
    kx, ky, kz = _axes([_modified(n, a == 0, p, True, True) for a, n in enumerate((lx, ly, lz))])
    x = C_DT * (kx * kx + ky * ky + kz * kz)
    t = torch.exp(-x) * torch.fft.rfftn(box["T"])
    if "S" in box:
        g = torch.where(x > 0, -torch.expm1(-x) / torch.where(x > 0, x, torch.ones_like(x)), torch.ones_like(x))
        t = t + g * torch.fft.rfftn(box["S"])
    return {"T": torch.fft.irfftn(t, s=(lz, ly, lx))}


def _yee(f):
    def d(t, axis, way):     # way +1: t[i+1] - t[i]; -1: t[i] - t[i-1]
        dim = 2 - axis
        return torch.roll(t, -1, dim) - t if way > 0 else t - torch.roll(t, 1, dim)

    def curl(u, way):
        return [d(u[(a + 2) % 3], (a + 1) % 3, way) - d(u[(a + 1) % 3], (a + 2) % 3, way) for a in range(3)]

    e, b, j = ([f[q + n] for n in "xyz"] for q in "EBJ")
    b = [v - C_DT * w for v, w in zip(b, curl(e, +1))]
    e = [v + C_DT * (w - u) for v, w, u in zip(e, curl(b, -1), j)]
    return dict(zip(EB, e + b))


def _padded(g, lo, n, gd):
    """The padded box of a global field, read by periodic index."""
    iz, iy, ix = (((torch.arange(n[a] + 2 * gd[a], device=DEVICE) + lo[a] - gd[a]) % g.shape[2 - a]) for a in (2, 1, 0))
    return g[iz][:, iy][:, :, ix]


def _arena(case, g):
    """A global field spread over the boxes as an arena holds it: dense boxes at
    offsets rounded up to 64 cells, zeros between them."""
    size, at = 0, []
    for _, n, gd, _ in _boxes(case):
        at.append(size)
        cells = 1
        for a in range(3):
            cells *= n[a] + 2 * gd[a]
        size += -(-cells // 64) * 64
    out = torch.zeros(size, dtype=g.dtype, device=DEVICE)
    for off, (lo, n, gd, _) in zip(at, _boxes(case)):
        t = _padded(g, lo, n, gd).reshape(-1)
        out[off:off + t.numel()] = t
    return out


def exact(case, seed):
    glob = {n: t.double() for n, t in _fields(case, seed).items()}
    if case["kind"] == "yee":
        return _yee(glob)
    if case["kind"] == "io":
        return {"boxes": [_arena(case, glob[n]) for n in J + ("rho",)], "grid": [glob[n] for n in EB]}
    names = ("T",) if case["kind"] == "heat" else EB
    new = {n: torch.empty_like(glob[n]) for n in names}
    sums = []
    for lo, n, gd, p in _boxes(case):
        box = {k: _padded(t, lo, n, gd) for k, t in glob.items()}
        if case["kind"] == "heat":
            out = _heat(box, p)
        else:
            out, s = _maxwell(box, p, case["staggered"], case["gauss"])
            sums += s or []
        at = tuple(slice(lo[a], lo[a] + n[a]) for a in (2, 1, 0))
        inner = tuple(slice(gd[a], gd[a] + n[a]) for a in (2, 1, 0))
        for k in names:
            new[k][at] = out[k][inner]
    del glob
    res = {k: _arena(case, new.pop(k)) for k in names}
    if case["gauss"]:
        res["gauss"] = torch.tensor(sums, dtype=torch.float64)
    return res
