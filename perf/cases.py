"""Wakefield solves as a user's program runs them: the geometry of a structure in host memory, one call after another
of the public binding (create, bunch, steps, wakes), the wakes, energies and balance records back on the host.

Every case is a whole solve (or a batch of them): a solver is made for the geometry, the bunch enters, crosses the
structure and leaves its wake window behind, the results are read and the solver is closed. Its device state lives
only inside the pass, so what a pass computes are the wakes, the energies, the balance records and, where a case says
so, the electric field it reads back. Geometry (radii, bunch line, liner) and charge come from the seed; the sizes
from the case.

Kinds:
  "cart"   the Cartesian scheme: "shape" box (the grid's box is the pipe), pipe, cavity or collimator; float32 or
           float64 fields; "liner" adds a dielectric liner as a per-cell eps_r array; "observer" gathers the transverse
           wake; "balance" is the cadence of the energy and charge records (0: none)
  "batch"  uneven pipes and cavities advanced together (run_batch)
  "rz"     the rotationally symmetric scheme on a chain of cavities, modes m_lo..m_hi; "start" cold or scattered
"""
import math

import numpy as np
import torch

from paper_0901_1053_gb300 import tetm
from paper_0901_1053_gb300.batching import run_batch

DZ = 1.0e-3                  # Cartesian mesh: dz = 1 mm, dx = dy = sqrt(2) mm, c dt = dz
DXY = math.sqrt(2.0) * DZ
DR = 0.25e-3                 # (r, z) mesh: dr = dz = 0.25 mm
C0 = 299792458.0
EPS0 = 8.8541878128e-12
MU0 = 1.0 / (EPS0 * C0 * C0)


def _window(nz, sigma):
    """Steps for the bunch to enter, cross nz planes and leave a window of 15 sigma behind (sigma in planes)."""
    return nz + math.ceil(5.0 * sigma - 1e-12) + math.ceil(15.0 * sigma - 1e-12) + 1


def _cart(name, shape, nx, ny, nz, precision, sigma, steps=0, observer=False, balance=0, liner=0.0, fields=False):
    return {"name": name, "kind": "cart", "shape": shape, "nx": nx, "ny": ny, "nz": nz, "precision": precision,
            "sigma": sigma, "steps": steps or _window(nz, sigma), "observer": observer, "balance": balance,
            "liner": liner, "fields": fields}


def _rz(name, nr, nz, m_lo, m_hi, precision, sigma, start):
    return {"name": name, "kind": "rz", "nr": nr, "nz": nz, "m_lo": m_lo, "m_hi": m_hi, "precision": precision,
            "sigma": sigma, "start": start}


def listed():
    return [
        # the plain method in float64 on a small pipe (the smallest solve anyone runs: a check of a set-up, a
        # teaching example, one point of a parameter scan), its electric field read back
        _cart("pipe fp64 24x24x96", "box", 24, 24, 96, "fp64", 4.0, steps=400, observer=True, fields=True),
        # the smallest request of a stream of served solves
        _cart("cavity fp32 48x48x192", "cavity", 48, 48, 192, "fp32", 5.0),
        # a grid that fits no tile: an off-axis bunch in a pipe, its dipole wake, frequent balances
        _cart("pipe fp32 118x131x603", "pipe", 118, 131, 603, "fp32", 3.7, observer=True, balance=100),
        # the largest request of the stream
        _cart("collimator fp32 256x256x1024", "collimator", 256, 256, 1024, "fp32", 6.0),
        # the step collimator of the benchmark, with its balances
        _cart("collimator fp32 256x256x2048", "collimator", 256, 256, 2048, "fp32", 6.0, balance=250),
        # a structure with a dielectric liner (per-cell eps_r)
        _cart("liner fp32 192x192x768", "collimator", 192, 192, 768, "fp32", 6.0, balance=250, liner=3.0),
        # a reference solve in float64
        _cart("collimator fp64 96x96x384", "collimator", 96, 96, 384, "fp64", 6.0, balance=250),
        # a scan: uneven solves in one batch
        {"name": "batch fp32 of 16", "kind": "batch", "count": 16, "n_lo": 32, "n_hi": 192, "precision": "fp32",
         "draw": 9011053},
        # a multi-cell structure, five modes, started inside its ingoing pipe (the float32 form for high modes)
        _rz("chain fp32 512x4096 m0-4", 512, 4096, 0, 4, "fp32", 8.0, "scattered"),
        # monopole and dipole in float64, cold start
        _rz("chain fp64 256x2048 m0-1", 256, 2048, 0, 1, "fp64", 8.0, "cold"),
        # a small on-axis solve on an odd grid
        _rz("chain fp32 93x771 m0", 93, 771, 0, 0, "fp32", 5.0, "cold"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp32", "fp32", "fp64", "liner", "batch", "rz32", "rz64"])
    if kind in ("fp32", "fp64", "liner"):
        top = {"fp32": 256, "fp64": 128, "liner": 192}[kind]
        nx = _log(rng, 24, top)
        ny = min(top, max(24, nx + rng.randint(-nx // 5, nx // 5)))
        nz = min({"fp32": 2048, "fp64": 512, "liner": 768}[kind], int(nx * rng.uniform(2.0, 6.0)))
        shape = rng.choice(["pipe", "cavity", "collimator"] if kind != "liner" else ["collimator"])
        sigma = round(rng.uniform(3.0, 8.0), 2)
        return {k: v for k, v in _cart("", shape, nx, ny, nz, "fp64" if kind == "fp64" else "fp32", sigma,
                                       observer=rng.random() < 0.4, balance=rng.choice([0, 100, 250]),
                                       liner=round(rng.uniform(2.0, 4.0), 2) if kind == "liner" else 0.0,
                                       fields=nx * ny * nz < 100000).items() if k != "name"}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(2, 12), "n_lo": 32, "n_hi": _log(rng, 40, 160),
                "precision": "fp32", "draw": rng.randint(1, 1 << 30)}
    nr = _log(rng, 48, 512 if kind == "rz32" else 256)
    nz = _log(rng, 1024, 4096 if kind == "rz32" else 2048)
    m_lo = rng.choice([0, 0, 1])
    c = _rz("", nr, nz, m_lo, m_lo + rng.randint(0, 4 if kind == "rz32" else 1),
            "fp32" if kind == "rz32" else "fp64", round(rng.uniform(3.0, 8.0), 2),
            rng.choice(["cold", "scattered"]) if kind == "rz32" else "cold")
    return {k: v for k, v in c.items() if k != "name"}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _radii(shape, nx, ny, nz, rs):
    """Radius (in transverse cells) of the vacuum of every plane."""
    n = min(nx, ny)
    k = np.arange(nz)
    if shape == "pipe":
        return np.full(nz, (0.36 + 0.02 * rs.uniform(-1, 1)) * n)
    if shape == "cavity":
        return np.where((k >= (3 * nz) // 8) & (k < (5 * nz) // 8), (0.44 + 0.01 * rs.uniform(-1, 1)) * n,
                        (0.2 + 0.01 * rs.uniform(-1, 1)) * n)
    return np.where((k >= nz // 4) & (k < (3 * nz) // 4), (0.125 + 0.004 * rs.uniform(-1, 1)) * n,
                    (0.375 + 0.004 * rs.uniform(-1, 1)) * n)


def _outside(nx, ny, rad):
    """uint8 (nz, ny, nx): 1 where a cell's centre lies further than rad[k] from the axis."""
    r = np.sqrt((np.arange(nx)[None, :] + 0.5 - nx / 2.0) ** 2 + (np.arange(ny)[:, None] + 0.5 - ny / 2.0) ** 2)
    radii, which = np.unique(rad, return_inverse=True)
    return np.stack([(r > v).astype(np.uint8) for v in radii])[which.reshape(-1)]


def _cart_inputs(c, seed):
    rs = np.random.RandomState(seed % (1 << 31))
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    w = {"nx": nx, "ny": ny, "nz": nz, "sigma": c["sigma"] * DZ, "charge": rs.uniform(0.5, 2.0) * 1e-9,
         "pec": None, "eps": None, "steps": c["steps"], "precision": c["precision"]}
    off = (lambda: int(rs.randint(-2, 3))) if c["observer"] else (lambda: 0)
    w["i0"], w["j0"] = nx // 2 + off(), ny // 2 + off()
    if c["shape"] == "box":
        return w
    rad = _radii(c["shape"], nx, ny, nz, rs)
    w["pec"] = _outside(nx, ny, rad)
    if c["liner"]:
        # cells within 4 of the narrow section's wall
        eps = 1.0 + (c["liner"] + 0.2 * rs.uniform(-1, 1) - 1.0) * (
            _outside(nx, ny, np.where(rad < rad.max(), rad - 4.0, 1e9)) * (1 - w["pec"]))
        w["eps"] = np.ascontiguousarray(eps, dtype=np.float64)
    return w


class _Solve:
    """One solve of a batch, with the attributes run_batch reads."""

    def __init__(self, w):
        self.nx, self.ny, self.nz, self.sigma, self.charge = w["nx"], w["ny"], w["nz"], w["sigma"], w["charge"]
        self.pec, self.i0, self.j0, self.steps = w["pec"], w["i0"], w["j0"], w["steps"]
        self.dx, self.dy, self.dz, self.cdt = DXY, DXY, DZ, DZ


def _batch_cases(c):
    """Uneven solves N x N x 4N, N between n_lo and n_hi, sigma between 3 and 10 planes."""
    rs = np.random.RandomState(c["draw"] % (1 << 31))
    out = []
    for _ in range(c["count"]):
        n = int(rs.randint(c["n_lo"], c["n_hi"] + 1)) & ~1
        out.append(_cart("", ("pipe", "cavity")[int(rs.randint(0, 2))], n, n, 4 * n, c["precision"],
                         round(float(rs.uniform(3.0, 10.0)), 2)))
    return out


def _rz_inputs(c, seed):
    """A chain of 9 cavities (radius 400/512 of nr) between irises and beam pipes (160/512), period 3/32 of nz."""
    rs = np.random.RandomState(seed % (1 << 31))
    nr, nz = c["nr"], c["nz"]
    period = max(4, (3 * nz) // 32)
    gap = (3 * period) // 4
    rel = np.arange(nz) - (nz - 9 * period) // 2 - (period - gap) // 2
    inside = (rel >= 0) & (rel < 9 * period) & (rel % period < gap)
    rad = np.where(inside, (400.0 + 8.0 * rs.uniform(-1, 1)) / 512.0 * nr, (160.0 + 4.0 * rs.uniform(-1, 1)) / 512.0 * nr)
    sigma = c["sigma"] * DR
    c0 = math.ceil(5.0 * c["sigma"] - 1e-12)
    head = 2 * c0 + 2 if c["start"] == "scattered" else 0
    return {"nr": nr, "nz": nz, "pec": (np.arange(nr)[None, :] + 0.5 > rad[:, None]).astype(np.uint8), "sigma": sigma,
            "charge": rs.uniform(0.5, 2.0) * 1e-9, "i0": 0 if c["m_hi"] == 0 else max(1, nr // 64), "head": head,
            "steps": _window(nz, c["sigma"]) - head}


def prepare(case, seed):
    if case["kind"] == "batch":
        return case, [_Solve(_cart_inputs(c, seed + 7919 * i)) for i, c in enumerate(_batch_cases(case))]
    return case, (_rz_inputs if case["kind"] == "rz" else _cart_inputs)(case, seed)


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(state):
    c, w = state
    if c["kind"] == "batch":
        return run_batch(w, c["precision"])[0]
    if c["kind"] == "rz":
        s = tetm.RzSolver(w["nr"], w["nz"], c["m_lo"], c["m_hi"], DR, DR, DR, c["precision"], pec=w["pec"])
        if c["start"] == "scattered":
            s.set_bunch_scattered(w["sigma"], w["charge"], w["i0"], w["head"])
        else:
            s.set_bunch(w["sigma"], w["charge"], w["i0"])
        s.step(w["steps"])
        out = {"m%d" % m: {"wake": s.wake(m)[0], "transverse": s.transverse_wake(m), "energy": s.energy(m)}
               for m in range(c["m_lo"], c["m_hi"] + 1)}
        s.close()
        return out
    s = tetm.Solver(w["nx"], w["ny"], w["nz"], DXY, DXY, DZ, DZ, c["precision"], eps_r=w["eps"], pec=w["pec"])
    s.set_bunch(w["sigma"], w["charge"], w["i0"], w["j0"])
    if c["observer"]:
        s.set_observer(w["i0"] + 1, w["j0"] - 2)
    if c["balance"]:
        s.set_balance_every(c["balance"])
    s.step(w["steps"])
    out = {"wake": s.wake()[0], "energy": s.energy()}
    if c["observer"]:
        out["transverse"] = s.transverse_wake()
    if c["balance"]:
        out["balances"] = s.balance_history()
    if c["fields"]:
        out["fields"] = {comp: s.get(comp) for comp in ("ex", "ey", "ez")}
    s.close()
    return out


def _vacuum_cells(c):
    rad = _radii(c["shape"], c["nx"], c["ny"], c["nz"], _Centre()) if c["shape"] != "box" else None
    return c["nx"] * c["ny"] * c["nz"] if rad is None else float(np.sum(np.pi * rad ** 2))


class _Centre:
    """Stands for the random state where the seed's middle value is wanted."""

    @staticmethod
    def uniform(a, b):
        return 0.5 * (a + b)


def work(case):
    """Each step reads and writes the six components of the cells that carry a field once, with a byte of activity
    (and six coefficients where there is a material array); 48 operations a cell. A solve reads its cell arrays once."""
    if case["kind"] == "batch":
        each = [work(c) for c in _batch_cases(case)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    size = 8 if case["precision"] == "fp64" else 4
    if case["kind"] == "rz":
        w = _rz_inputs(case, 0)
        cells = float((case["m_hi"] - case["m_lo"] + 1) * (w["pec"].size - int(w["pec"].sum())))
        return {"bytes": cells * w["steps"] * (12 * size + 1) + w["pec"].nbytes, "flops": cells * w["steps"] * 47}
    cells = _vacuum_cells(case)
    box = case["nx"] * case["ny"] * case["nz"]
    per = (18 if case["liner"] else 12) * size + 1
    return {"bytes": cells * case["steps"] * per + box * (9 if case["liner"] else 1), "flops": cells * case["steps"] * 48}


# ---------------------------------------------------------------------------
# The same in plain 64-bit torch
# ---------------------------------------------------------------------------
def _phi(x):
    return 0.5 * math.erfc(-x / math.sqrt(2.0))


def _cell_charges(sigma, q, dz, c0):
    """Charge of the truncated Gaussian in [d dz, (d+1) dz], d = -c0 .. c0-1."""
    out = []
    for d in range(-c0, c0):
        lo, hi = max(d * dz, -5.0 * sigma), min((d + 1) * dz, 5.0 * sigma)
        out.append(q * (_phi(hi / sigma) - _phi(lo / sigma)) if hi > lo else 0.0)
    return out


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _cart_coefficients(w, dev):
    """M^-1 of (ex, ey, ez, hx, hy, hz), arrays (nz+1, ny+1, nx+1), 0 on PEC: an edge needs its four cells free of
    PEC and takes the mean of their eps_r, a face its two cells."""
    nx, ny, nz = w["nx"], w["ny"], w["nz"]
    free = torch.zeros((nz + 2, ny + 2, nx + 2), dtype=torch.float64, device=dev)  # cell (i, j, k) at [k+1, j+1, i+1]
    free[1:-1, 1:-1, 1:-1] = 1.0 if w["pec"] is None else 1.0 - torch.from_numpy(w["pec"]).to(dev).double()
    eps = None
    if w["eps"] is not None:
        eps = torch.ones_like(free)
        eps[1:-1, 1:-1, 1:-1] = torch.from_numpy(w["eps"]).to(dev)

    def cells(a, di, dj, dk):  # value of cell (i+di, j+dj, k+dk) for every node
        return a[1 + dk:nz + 2 + dk, 1 + dj:ny + 2 + dj, 1 + di:nx + 2 + di]

    def obj(around, scale, edge):
        on = scale * cells(free, *around[0])
        for o in around[1:]:
            on *= cells(free, *o)
        if edge and eps is not None:
            on /= sum(cells(eps, *o) for o in around) / len(around)
        return on
    x, y, z = (0, -1), (0, -1), (0, -1)
    return [obj([(0, b, c) for b in y for c in z], DXY / (EPS0 * DXY * DZ), True),
            obj([(a, 0, c) for a in x for c in z], DXY / (EPS0 * DXY * DZ), True),
            obj([(a, b, 0) for a in x for b in y], DZ / (EPS0 * DXY * DXY), True),
            obj([(a, 0, 0) for a in x], DXY / (MU0 * DXY * DZ), False),
            obj([(0, b, 0) for b in y], DXY / (MU0 * DXY * DZ), False),
            obj([(0, 0, c) for c in z], DZ / (MU0 * DXY * DXY), False)]


def _cart_exact(c, w):
    dev = _device()
    nx, ny, nz = w["nx"], w["ny"], w["nz"]
    M = _cart_coefficients(w, dev)
    a = 0.5 * DZ / C0
    A = [m * (2 * a if q in (2, 5) else a) for q, m in enumerate(M)]
    ex, ey, ez, hx, hy, hz = (torch.zeros((nz + 1, ny + 1, nx + 1), dtype=torch.float64, device=dev) for _ in range(6))
    t = torch.empty_like(ex)
    up = {0: (slice(1, None),), 1: (slice(None), slice(1, None)), 2: (slice(None), slice(None), slice(1, None))}
    dn = {0: (slice(None, -1),), 1: (slice(None), slice(None, -1)), 2: (slice(None), slice(None), slice(None, -1))}
    cut = {0: (slice(-1, None),), 1: (slice(None), slice(-1, None)), 2: (slice(None), slice(None), slice(-1, None))}
    first = {0: (slice(0, 1),), 1: (slice(None), slice(0, 1)), 2: (slice(None), slice(None), slice(0, 1))}

    def ahead(f, ax, co, out, sign):       # out += sign * co * (f[+1] - f)
        d = torch.sub(f[up[ax]], f[dn[ax]], out=t[dn[ax]])
        t[cut[ax]] = 0.0
        out.addcmul_(co, t, value=sign)

    def behind(f, ax, co, out, sign):      # out += sign * co * (f[-1] - f)
        torch.sub(f[dn[ax]], f[up[ax]], out=t[up[ax]])
        t[first[ax]] = 0.0
        out.addcmul_(co, t, value=sign)
    sp = c["sigma"]
    c0, m_max = math.ceil(5.0 * sp - 1e-12), math.ceil(15.0 * sp - 1e-12)
    m_min = -c0 - 1
    nw = m_max - m_min + 1
    Q = torch.tensor([C0 * v / DZ for v in _cell_charges(w["sigma"], w["charge"], DZ, c0)], dtype=torch.float64, device=dev)
    i0, j0, q = w["i0"], w["j0"], w["charge"]
    io, jo = i0 + 1, j0 - 2
    wake, wx, wy = (torch.zeros(nw, dtype=torch.float64, device=dev) for _ in range(3))
    eta0 = MU0 * C0

    def energy():
        e = sum(float(torch.where(m > 0, f * f / torch.where(m > 0, m, torch.ones_like(m)), torch.zeros_like(m)).sum())
                for m, f in zip(M, (ex, ey, ez, hx, hy, hz))) * 0.5
        r = 0.0
        for m, f, ax, fwd in ((M[3], ez, 1, True), (M[4], ez, 2, True), (M[0], hz, 1, False), (M[1], hz, 2, False)):
            d = f[up[ax]] - f[dn[ax]]
            r += float((m[dn[ax] if fwd else up[ax]] * d * d).sum())
        l = float((hx[:-1] * (ey[1:] - ey[:-1]) - hy[:-1] * (ex[1:] - ex[:-1])).sum())
        return e - 0.5 * a * a * r + a * l
    rows = []
    for n in range(w["steps"]):
        k_lo, k_hi = max(0, n - m_max - c0), min(nz, n - m_min - c0 + 1)   # planes whose sample is in the window
        if c["observer"]:
            ex_o, ey_o = ex[k_lo:k_hi, jo, io].clone(), ey[k_lo:k_hi, jo, io].clone()
        for half in (0, 1):
            ahead(ey, 0, A[3], hx, 1.0)
            ahead(ez, 1, A[3], hx, -1.0)
            ahead(ex, 0, A[4], hy, -1.0)
            ahead(ez, 2, A[4], hy, 1.0)
            if half == 0:
                behind(hx, 1, A[2], ez, 1.0)
                behind(hy, 2, A[2], ez, -1.0)
                lo, hi = max(0, n - 2 * c0), min(nz, n)                    # planes that carry current
                if hi > lo:
                    ez[lo:hi, j0, i0] -= A[2][lo:hi, j0, i0] * Q[lo - n + 2 * c0:hi - n + 2 * c0]
        for half in (0, 1):
            behind(hy, 0, A[0], ex, 1.0)
            behind(hz, 1, A[0], ex, -1.0)
            behind(hx, 0, A[1], ey, -1.0)
            behind(hz, 2, A[1], ey, 1.0)
            if half == 0:
                ahead(ex, 1, A[5], hz, 1.0)
                ahead(ey, 2, A[5], hz, -1.0)
        if k_hi > k_lo:
            at = slice(n - c0 - m_min - (k_hi - 1), n - c0 - m_min - k_lo + 1)  # sample of plane k: n - c0 - k - m_min
            wake[at] -= ez[k_lo:k_hi, j0, i0].flip(0) / q
            if c["observer"]:
                wx[at] += (DZ / q * (ex_o / DXY - eta0 * hy[k_lo:k_hi, jo, io] / DXY)).flip(0)
                wy[at] += (DZ / q * (ey_o / DXY + eta0 * hx[k_lo:k_hi, jo, io] / DXY)).flip(0)
        if c["balance"] and (n + 1) % c["balance"] == 0:
            zc = (n + 0.5 - c0) * DZ
            s5 = 5.0 * w["sigma"]
            qs = 0.0
            for k in range(nz + 1):
                lo, hi = max((k - 0.5) * DZ - zc, -s5), min((k + 0.5) * DZ - zc, s5)
                if hi > lo:
                    qs = max(qs, q * (_phi(hi / w["sigma"]) - _phi(lo / w["sigma"])))
            rows.append([n + 1.0, energy(), 0.0, 0.0, qs])   # the charge laws hold exactly
    out = {"wake": wake, "energy": energy()}
    if c["observer"]:
        out["transverse"] = (wx, wy)
    if c["balance"]:
        out["balances"] = np.array(rows, dtype=np.float64).reshape(-1, 5)
    if c["fields"]:
        out["fields"] = {"ex": ex, "ey": ey, "ez": ez}
    return out


def _rz_exact(c, w):
    dev = _device()
    nr, nz = w["nr"], w["nz"]
    modes = list(range(c["m_lo"], c["m_hi"] + 1))
    new = lambda: torch.zeros((len(modes), nz + 1, nr + 1), dtype=torch.float64, device=dev)  # noqa: E731
    i = torch.arange(nr + 1, dtype=torch.float64, device=dev)
    ri, rh = i * DR, (i + 0.5) * DR
    m = torch.tensor(modes, dtype=torch.float64, device=dev).view(-1, 1, 1)
    free = torch.zeros((nz + 2, nr + 2), dtype=torch.float64, device=dev)           # cell (i, k) at [k+1, i+1]
    free[1:-1, 1:-1] = 1.0 - torch.from_numpy(w["pec"]).to(dev).double()
    cell = lambda di, dk: free[1 + dk:nz + 2 + dk, 1 + di:nr + 2 + di]  # noqa: E731
    zero_axis = torch.ones(nr + 1, dtype=torch.float64, device=dev)
    zero_axis[0] = 0.0
    inv_ri = torch.where(i > 0, 1.0 / torch.where(i > 0, ri, torch.ones_like(ri)), torch.zeros_like(ri))
    CER = (DR / (EPS0 * rh * DR)) * cell(0, -1) * cell(0, 0)
    CEP = (ri / (EPS0 * DR * DR)) * cell(-1, -1) * cell(0, -1) * cell(-1, 0) * cell(0, 0)
    CEZ = (DR / (EPS0 * DR)) * inv_ri * cell(-1, 0) * cell(0, 0)
    CHR = (DR / (MU0 * DR)) * inv_ri * cell(-1, 0) * cell(0, 0)
    CHP = (rh / (MU0 * DR * DR)) * cell(0, 0)
    CHZ = (DR / (MU0 * rh * DR)) * cell(0, -1) * cell(0, 0)
    CEZ = CEZ.expand(len(modes), -1, -1).clone()
    if modes[0] == 0:
        CEZ[0, :, 0] = DR / (EPS0 * DR * DR / 4.0) * cell(0, 0)[:, 0]
    a = 0.5 * DR / C0
    FEZ = 2.0 * a * CEZ / (1.0 + a * a * m * m * CEZ * CHR)
    FHZ = 2.0 * a * CHZ / (1.0 + a * a * m * m * CHZ * CER)
    er, ep, ez, hr, hp, hz = (new() for _ in range(6))
    sp = c["sigma"]
    c0, m_max = math.ceil(5.0 * sp - 1e-12), math.ceil(15.0 * sp - 1e-12)
    m_min = -c0 - 1
    nw = m_max - m_min + 1
    q, i0, K = w["charge"], w["i0"], w["head"]
    share = torch.where(m == 0, torch.ones_like(m), 2.0 * torch.ones_like(m)) / (2.0 * math.pi)
    cells = torch.tensor(_cell_charges(w["sigma"], q, DR, c0), dtype=torch.float64, device=dev)
    J = share.view(-1, 1) * (C0 / DR) * cells.view(1, -1)
    eta0 = MU0 * C0
    if K:  # the bunch's field inside the ingoing pipe: a radial potential times a longitudinal profile
        for mi, mm in enumerate(modes):
            on = (CEZ[mi, 1] != 0).cpu().numpy()
            edge = (CER[1] != 0).cpu().numpy()
            D = np.zeros((nr + 1, nr + 1))
            for x in range(nr + 1):
                if not on[x]:
                    D[x, x] = 1.0
                    continue
                if x < nr and edge[x]:
                    D[x, x] += x + 0.5
                    if on[x + 1]:
                        D[x, x + 1] -= x + 0.5
                if x > 0 and edge[x - 1]:
                    D[x, x] += x - 0.5
                    if on[x - 1]:
                        D[x, x - 1] -= x - 0.5
                if x > 0:
                    D[x, x] += mm * mm / x
            rhs = np.zeros(nr + 1)
            rhs[i0] = 1.0
            psi = np.where(on, np.linalg.solve(D, rhs), 0.0)
            G = np.zeros(nz + 4)                                      # G[u + 1]
            jj = J[mi].cpu().numpy()
            for u in range(K - 1, K - 2 * c0 - 1, -1):
                G[u + 1] = 2.0 * eta0 * jj[u - K + 2 * c0] - G[u + 2]
            G = torch.from_numpy(G).to(dev)
            g0, g1 = G[1:nz + 2].clone(), G[2:nz + 3].clone()
            g0[K + 1:] = 0.0
            g1[K:] = 0.0
            ps = torch.from_numpy(psi).to(dev)
            prp = torch.zeros_like(ps)
            prp[:-1] = ps[1:] - ps[:-1]
            er[mi] = -(CER != 0).double() * g0.view(-1, 1) * prp
            ep[mi] = -(CEP != 0).double() * g0.view(-1, 1) * (mm * ps)
            hp[mi] = (CHP != 0).double() * g1.view(-1, 1) * (rh / (DR * eta0) * prp)
            hr[mi] = -(CHR != 0).double() * g1.view(-1, 1) * (DR * inv_ri / eta0 * mm * ps)
    AER, AEP, AHR, AHP = a * CER, a * CEP, a * CHR, a * CHP
    t = new()

    def tm_half():
        torch.sub(er[:, 1:], er[:, :-1], out=t[:, :-1])
        t[:, -1] = 0.0
        t[:, :, :-1] -= ez[:, :, 1:] - ez[:, :, :-1]
        hp.addcmul_(AHP, t)
        torch.sub(ep[:, :-1], ep[:, 1:], out=t[:, :-1])
        t[:, -1] = 0.0
        t.addcmul_(m, ez)
        hr.addcmul_(AHR, t)

    def te_half():
        torch.sub(hr[:, :-1], hr[:, 1:], out=t[:, 1:])
        t[:, 0] = 0.0
        t[:, :, 1:] -= hz[:, :, :-1] - hz[:, :, 1:]
        ep.addcmul_(AEP, t)
        torch.sub(hp[:, 1:], hp[:, :-1], out=t[:, 1:])
        t[:, 0] = 0.0
        t.addcmul_(m, hz)
        er.addcmul_(AER, t)
    wake, wt = (torch.zeros((len(modes), nw), dtype=torch.float64, device=dev) for _ in range(2))
    for n in range(w["steps"]):
        at_n = n + K
        k_lo, k_hi = max(0, at_n - m_max - c0), min(nz, at_n - m_min - c0 + 1)
        er_o = er[:, k_lo:k_hi, i0].clone()
        tm_half()
        torch.neg(hp, out=t)
        t[:, :, 1:] += hp[:, :, :-1]
        t.addcmul_(m, hr, value=-1.0)
        lo, hi = max(0, at_n - 2 * c0), min(nz, at_n)
        if hi > lo:
            t[:, lo:hi, i0] -= J[:, lo - at_n + 2 * c0:hi - at_n + 2 * c0]
        ez.addcmul_(FEZ, t)
        tm_half()
        te_half()
        torch.sub(ep[:, :, 1:], ep[:, :, :-1], out=t[:, :, :-1])
        t[:, :, -1] = 0.0
        t.addcmul_(m, er, value=-1.0)
        hz.addcmul_(FHZ, t)
        te_half()
        if k_hi > k_lo:
            at = slice(at_n - c0 - m_min - (k_hi - 1), at_n - c0 - m_min - k_lo + 1)
            wake[:, at] -= ez[:, k_lo:k_hi, i0].flip(1) / q
            wt[:, at] += ((er_o / DR + eta0 * hp[:, k_lo:k_hi, i0] / ((i0 + 0.5) * DR)) * DR / q).flip(1)
    out = {}
    for mi, mm in enumerate(modes):
        e = 0.0
        for C, f in ((CER, er), (CEP, ep), (CEZ[mi], ez), (CHR, hr), (CHP, hp), (CHZ, hz)):
            on = C != 0
            e += 0.5 * float((f[mi][on] ** 2 / C[on]).sum())
        d1 = ez[mi][:, 1:] - ez[mi][:, :-1]
        d2 = hz[mi][:, :-1] - hz[mi][:, 1:]
        r = float((CHP[:, :-1] * d1 * d1).sum() + (CEP[:, 1:] * d2 * d2).sum())
        l = float((hp[mi][:-1] * (er[mi][1:] - er[mi][:-1]) - hr[mi][:-1] * (ep[mi][1:] - ep[mi][:-1])).sum())
        out["m%d" % mm] = {"wake": wake[mi], "transverse": wt[mi], "energy": e - 0.5 * a * a * r + a * l}
    return out


def exact(case, seed):
    if case["kind"] == "batch":
        parts = _batch_cases(case)
        if sum(c["nx"] * c["ny"] * c["nz"] * c["steps"] for c in parts) > 4e10:
            return None
        return [_cart_exact(c, _cart_inputs(c, seed + 7919 * i))["wake"] for i, c in enumerate(parts)]
    if case["kind"] == "rz":
        return _rz_exact(case, _rz_inputs(case, seed))
    if case["nx"] * case["ny"] * case["nz"] * case["steps"] > 4e10:
        return None
    return _cart_exact(case, _cart_inputs(case, seed))
