"""The work that users of the framework have it do, as cases that can be timed and compared.

Every case is one pass through the public Python face of the library on a synthetic ultrasound
ring acquisition: transducers on a ring, stepped over some elevations, one traveltime per
unordered pair of elements of an elevation and per frequency band, and a voxel grid in the ring.

* ``listed()`` - the cases by name, smallest calls to the largest acquisition;
* ``draw(rng)`` - another case of the same ranges;
* ``prepare(case, seed)`` - the inputs and the operator handle a program holds before the call;
* ``run(state)`` - the call;
* ``work(case)`` - bytes and operations the call cannot do without;
* ``exact(case, seed)`` - the same outputs by plain torch in 64 bits (none of this library's code).

Lengths in a case are in millimetres; ``bands`` lists "centre/sigma" in MHz.
"""
import math
import random

import numpy as np
import torch

import paper_1908_03302_gb300 as fg

C0 = 1500.0            # water (m/s)
NOISE_S = 5e-9         # standard deviation of a traveltime pick (s)
N_TABLE = 4096         # samples of a band's Phi table
PERIODS = 3.0          # cut-off detour time, in dominant periods of the band
LAMBDA_REL = 1e-3      # relative damping of the least-squares solves
N_BLOBS = 8
OPS_PER_EVAL = 26      # operations of one in-support entry J[p, v] (24 FP32, 2 square roots or reciprocals)

ONE_BAND = "1.0/0.4"
SMALL_BAND = "1.0/0.3"
# the 1.0 and 1.4 MHz bands have not decayed at the cut-off: their truncation is a jump
THREE_BANDS = "0.6/0.2 1.0/0.2 1.4/0.2"


def _case(name, op, n_tx, radius, slices, step, bands, nx, ny, nz, h, **more):
    c = {"name": name, "op": op, "n_tx": n_tx, "radius": radius, "slices": slices, "step": step, "bands": bands,
         "nx": nx, "ny": ny, "nz": nz, "h": h}
    c.update(more)
    return c


def listed():
    ring32 = (32, 50.0, 1, 0.0, SMALL_BAND, 48, 48, 16, 2.0)
    ring256 = (256, 100.0, 1, 0.0, ONE_BAND, 200, 200, 40, 1.0)
    ring256_3band = (256, 100.0, 1, 0.0, THREE_BANDS, 200, 200, 40, 1.0)
    return [
        # predicted traveltimes of a small array and the gradient of their misfit, as an optimiser
        # in PyTorch asks for them at every step: the smallest calls
        _case("grad_ring32", "grad", *ring32),
        # a whole damped least-squares solve of a small slice-by-slice acquisition with three bands
        _case("cg_slices32", "cg", 32, 50.0, 4, 4.0, THREE_BANDS, 48, 48, 24, 2.0, iters=20),
        # predicted traveltimes of the 256-element ring: the forward operator of every solver
        _case("j_ring256", "j", *ring256),
        # backprojection of its residuals: the adjoint of every solver
        _case("jt_ring256", "jt", *ring256),
        # the same array measured in three bands, two of them with a sharp cut-off
        _case("j_ring256_3band", "j", *ring256_3band),
        # the whole volume: sixteen elevations, three bands, 1.6 M rows against 6.3 M voxels
        _case("jt_slices3d", "jt", 256, 100.0, 16, 4.0, THREE_BANDS, 256, 256, 96, 0.75),
        # the Hessian applied to a block of vectors, as block eigensolvers do
        _case("block_ring256", "block", *ring256, cols=8),
        # resolution of the array and of its every 2nd and every 4th element: point-spread
        # functions of many voxels on the tensor cores
        _case("psf_tc_ring256_3band", "psf", *ring256_3band, spikes=128, mode=1, strides="4 2 1"),
        # resolution of a stack of elevations 8 mm apart at a few voxels, in FP32, on an odd grid
        _case("psf_stack8", "psf", 256, 100.0, 7, 8.0, ONE_BAND, 141, 141, 33, 1.0, spikes=4, mode=0, strides="1"),
        # a plane image under a ring, the kernel integrated over the layers that its support reaches
        _case("plane_ring256", "plane", 256, 100.0, 1, 0.0, ONE_BAND, 141, 141, 41, 1.0),
        # Phi kept as the paper keeps it, as a few sine terms
        _case("series_jt_ring256", "jt", *ring256, phi="series"),
        # a new acquisition: table, operator and its first forward product
        _case("setup_ring256", "setup", *ring256),
    ]


def draw(rng):
    """One more case: small solver calls, single-ring calls and slice stacks, over the ranges of the
    listed ones, odd grid sizes included."""

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["grad", "cg", "j", "jt", "j", "jt", "stack_j", "stack_jt", "block", "psf_tc", "psf", "plane",
                     "series", "setup"])
    more = {}
    if op in ("grad", "cg"):
        c = _case("", op, log_int(16, 56), rng.choice([40.0, 50.0, 60.0]), rng.randint(1, 4), 4.0,
                  rng.choice([SMALL_BAND, THREE_BANDS]), rng.randint(25, 64), rng.randint(25, 64), rng.randint(7, 25),
                  rng.choice([1.5, 2.0]))
        if op == "cg":
            more = {"iters": rng.randint(8, 16)}
    else:
        slices, step, bands = 1, 0.0, rng.choice([ONE_BAND, ONE_BAND, THREE_BANDS])
        if op.startswith("stack"):
            slices, step, bands, op = log_int(2, 16), rng.choice([3.0, 4.0, 8.0]), THREE_BANDS, op[6:]
        n_tx = log_int(48, 256)
        if op in ("series", "plane"):
            bands = ONE_BAND
        if op == "psf_tc":
            op, more = "psf", {"spikes": log_int(8, 128), "mode": 1, "strides": "4 2 1"}
            n_tx = 4 * max(12, n_tx // 4)
        elif op == "psf":
            slices, step, bands = rng.randint(2, 11), rng.choice([3.0, 8.0]), ONE_BAND
            more = {"spikes": rng.randint(1, 4), "mode": rng.choice([0, 2]), "strides": rng.choice(["1", "2 1"])}
        elif op == "block":
            more = {"cols": rng.randint(4, 12)}
        elif op == "series":
            op, more = "jt", {"phi": "series"}
        c = _case("", op, n_tx, rng.choice([70.0, 85.0, 100.0]), slices, step, bands, rng.randint(90, 220),
                  rng.randint(90, 220), rng.randint(17, 96 if slices > 2 else 48), rng.choice([0.75, 1.0, 1.0]))
    c.update(more)
    del c["name"]
    return c


# ------------------------------------------------------------------ the acquisition

class _Grid:
    def __init__(self, c):
        self.nx, self.ny, self.nz, self.h = c["nx"], c["ny"], c["nz"], c["h"] * 1e-3
        self.origin = tuple(-(n - 1) * self.h / 2 for n in (self.nx, self.ny, self.nz))
        self.n_vox = self.nx * self.ny * self.nz

    def axes(self, device):
        return [self.origin[a] + torch.arange(n, device=device, dtype=torch.float64) * self.h
                for a, n in enumerate((self.nx, self.ny, self.nz))]


def _bands(c):
    return [tuple(float(x) * 1e6 for x in b.split("/")) for b in c["bands"].split()]


def _acquisition(c, seed=None):
    """Transducers, rows (emitter, receiver) and the rows' bands. With a seed the elements sit up to
    0.2 mm off the ring, as a calibration finds them."""
    n, ns = c["n_tx"], c["slices"]
    ang = 2.0 * np.pi * np.arange(n) / n
    rad = c["radius"] * 1e-3
    z = (np.arange(ns) - (ns - 1) / 2.0) * c["step"] * 1e-3
    tx = np.stack([np.tile(rad * np.cos(ang), ns), np.tile(rad * np.sin(ang), ns), np.repeat(z, n)], axis=1)
    if seed is not None:
        tx = tx + np.random.default_rng(seed).uniform(-2e-4, 2e-4, size=tx.shape)
    a, b = np.triu_indices(n, 1)
    pairs = np.stack([a, b], axis=1).astype(np.int32)
    pairs = (pairs[None] + (n * np.arange(ns, dtype=np.int32))[:, None, None]).reshape(-1, 2)
    nb = len(_bands(c))
    return tx, np.tile(pairs, (nb, 1)), np.repeat(np.arange(nb, dtype=np.int32), len(pairs))


def _subsets(c):
    """Row subsets of a case: the pairs of every k-th element of each ring, for each stride k."""
    a, b = np.triu_indices(c["n_tx"], 1)
    out = []
    for k in (int(s) for s in c["strides"].split()):
        keep = np.flatnonzero((a % k == 0) & (b % k == 0))
        n_rings = c["slices"] * len(_bands(c))
        out.append((keep[None] + len(a) * np.arange(n_rings)[:, None]).reshape(-1).astype(np.int32))
    return out


def _blobs(c, seed):
    """A model of Gaussian inclusions: centres, widths (m) and amplitudes (m/s)."""
    rng = np.random.default_rng(seed)
    g = _Grid(c)
    half = 0.35 * g.h * min(g.nx, g.ny)
    r, phi = half * np.sqrt(rng.uniform(size=N_BLOBS)), rng.uniform(0, 2 * np.pi, size=N_BLOBS)
    zc = rng.uniform(-0.4, 0.4, size=N_BLOBS) * g.h * g.nz
    amp = rng.uniform(10.0, 40.0, size=N_BLOBS) * rng.choice([-1.0, 1.0], size=N_BLOBS)
    return np.stack([r * np.cos(phi), r * np.sin(phi), zc], axis=1), rng.uniform(3e-3, 9e-3, size=N_BLOBS), amp


def _model(c, seed, plane=False):
    """Sound-speed perturbation (m/s) on the grid, or on its mid plane."""
    g, dev = _Grid(c), torch.device("cuda")
    x, y, z = g.axes(dev)
    if plane:
        z = z[:1] * 0.0
    m = torch.zeros((len(z), g.ny, g.nx), device=dev, dtype=torch.float64)
    for ctr, s, amp in zip(*_blobs(c, seed)):
        ex, ey, ez = (torch.exp(-0.5 * ((u - float(o)) / float(s)) ** 2) for u, o in zip((x, y, z), ctr))
        if plane:
            ez = torch.ones_like(ez)
        m += float(amp) * ez[:, None, None] * ey[None, :, None] * ex[None, None, :]
    return m.reshape(-1).float()


def _data(c, seed, tx, rows):
    """Traveltime shifts (s) of the same inclusions along straight rays, with picking noise."""
    dev = torch.device("cuda")
    t, r = torch.as_tensor(tx, device=dev), torch.as_tensor(rows, device=dev).long()
    s, e = t[r[:, 0]], t[r[:, 1]]
    u = (e - s) / (e - s).norm(dim=1, keepdim=True)
    d = torch.zeros(len(rows), device=dev, dtype=torch.float64)
    for ctr, w, amp in zip(*_blobs(c, seed)):
        q = torch.as_tensor(ctr, device=dev) - s
        dist2 = (q * q).sum(1) - (q * u).sum(1) ** 2
        d -= float(amp) * float(w) * math.sqrt(2 * math.pi) / C0 ** 2 * torch.exp(-0.5 * dist2 / float(w) ** 2)
    gen = torch.Generator(device=dev).manual_seed(int(seed) + 1)
    return (d + NOISE_S * torch.randn(len(rows), device=dev, dtype=torch.float64, generator=gen)).float()


def _spikes(c, seed):
    """Distinct voxels in the middle of the grid."""
    g, rng = _Grid(c), np.random.default_rng(seed)
    i, j, k = (np.arange(n) for n in (g.nx, g.ny, g.nz))
    rho2 = ((i - (g.nx - 1) / 2.0)[None, :] ** 2 + (j - (g.ny - 1) / 2.0)[:, None] ** 2)
    plane = np.flatnonzero(rho2.ravel() <= (0.35 * min(g.nx, g.ny)) ** 2)
    layers = k[(k >= g.nz // 5) & (k < g.nz - g.nz // 5)]
    v = rng.choice(len(plane) * len(layers), size=c["spikes"], replace=False)
    return np.sort(layers[v // len(plane)] * (g.nx * g.ny) + plane[v % len(plane)]).astype(np.int64)


def _inputs(c, seed):
    """What the call takes besides the operator."""
    op = c["op"]
    tx, rows, band = _acquisition(c, seed if op == "setup" else None)
    x = {"tx": tx, "rows": rows, "band": band}
    if op in ("j", "grad", "setup"):
        x["m"] = _model(c, seed)
    if op in ("jt", "grad", "cg", "plane"):
        x["d"] = _data(c, seed, tx, rows)
    if op == "plane":
        x["m2"] = _model(c, seed, plane=True)
    if op == "block":
        gen = torch.Generator(device="cuda").manual_seed(int(seed))
        x["X"] = torch.randn((c["cols"], _Grid(c).n_vox), device="cuda", generator=gen)
    if op == "psf":
        x["spikes"], x["subsets"] = _spikes(c, seed), _subsets(c)
    return x


def _operator(c, x, keep_host=False):
    make = (lambda f, s: fg.TrigTable(f, s)) if c.get("phi") == "series" else \
        (lambda f, s: fg.Table(f, s, n=N_TABLE, keep_host=keep_host))
    tables = [make(f, s) for f, s in _bands(c)]
    return tables, fg.Geometry(x["tx"], x["rows"], _Grid(c), C0, tables,
                               band_of_row=x["band"] if len(tables) > 1 else None)


def prepare(case, seed):
    x = _inputs(case, seed)
    if case["op"] == "setup":
        return case, x, None
    if case["op"] == "grad":
        x["m"].requires_grad_(True)
    return case, x, _operator(case, x)[1]


def run(state):
    case, x, geo = state
    op = case["op"]
    if op == "j":
        return geo.J(x["m"])
    if op == "jt":
        return geo.JT(x["d"])
    if op == "grad":
        d = fg.jacobian_apply(x["m"], geo)
        g, = torch.autograd.grad(d, x["m"], grad_outputs=d.detach() - x["d"])
        return d.detach(), g
    if op == "cg":
        return geo.cg_solve(x["d"], LAMBDA_REL, case["iters"])
    if op == "block":
        d = geo.J_batch(x["X"])
        return d, geo.JT_batch(d)
    if op == "psf":
        return geo.psf_batch(x["spikes"], x["subsets"], mode=case["mode"])
    if op == "plane":
        return geo.J2d(x["m2"]), geo.JT2d(x["d"])
    tables, geo = _operator(case, x, keep_host=True)   # a new acquisition
    return [t.host for t in tables], geo.J(x["m"])


# ------------------------------------------------------------------ what a call cannot do without

def _support(c):
    """Estimated in-support entries of J, (rows, voxels) sampled with a fixed seed; for point-spread
    functions the entries of the rows that hold a spike, and those times the spikes each holds."""
    tx, rows, band = _acquisition(c)
    g, rng = _Grid(c), np.random.default_rng(0)
    n_r, n_v = 2048, 4096
    p = rng.integers(0, len(rows), size=n_r)
    s, r = tx[rows[p, 0]], tx[rows[p, 1]]
    U = np.array([C0 * PERIODS / f for f, _ in _bands(c)])[band[p]]

    def inside(ijk):
        v = np.array(g.origin)[None] + ijk * g.h
        R = -np.linalg.norm(s - r, axis=1)[:, None]
        for t in (s, r):
            R = R + np.sqrt(np.maximum((t * t).sum(1)[:, None] + (v * v).sum(1)[None] - 2.0 * t @ v.T, 0.0))
        return R < U[:, None]

    n = inside(rng.uniform(size=(n_v, 3)) * np.array([g.nx, g.ny, g.nz]) - 0.5).mean(1) * g.n_vox
    if c["op"] != "psf":
        return float(n.mean()) * len(rows), 0.0
    v = _spikes(c, 0)
    k = inside(np.stack([v % g.nx, (v // g.nx) % g.ny, v // (g.nx * g.ny)], axis=1)).sum(1)
    return float((n * (k > 0)).mean()) * len(rows), float((n * k).mean()) * len(rows)


def work(case):
    c, op = case, case["op"]
    g = _Grid(c)
    m = len(_bands(c)) * c["slices"] * c["n_tx"] * (c["n_tx"] - 1) // 2
    evals, products = _support(c)
    per = OPS_PER_EVAL * evals
    if op in ("j", "jt"):
        return {"bytes": 4 * (m + g.n_vox), "flops": per}
    if op == "grad":
        return {"bytes": 4 * (3 * m + 2 * g.n_vox), "flops": 2 * per}
    if op == "cg":   # the first residual and every iteration apply J and J^T once
        n = c["iters"] + 1
        return {"bytes": n * 4 * (5 * m + 8 * g.n_vox), "flops": 2 * n * per}
    if op == "block":   # each entry is made once per direction and used for every column
        return {"bytes": 4 * c["cols"] * (2 * m + 2 * g.n_vox), "flops": 2 * (per + 2 * c["cols"] * evals)}
    if op == "psf":
        n_out = len(c["strides"].split()) * c["spikes"]
        return {"bytes": 4 * n_out * g.n_vox + 4 * m, "flops": per + 2 * products}
    if op == "plane":
        return {"bytes": 4 * (2 * m + 2 * g.nx * g.ny), "flops": 2 * per}
    # setup: the table's quadrature (a node's sine and product for each sample, 1024 nodes at least for
    # the accuracy it states), the support, one J
    return {"bytes": 8 * m + 4 * (m + g.n_vox) + 8 * N_TABLE, "flops": per + 2 * 1024 * N_TABLE}


# ------------------------------------------------------------------ 64 bits, by plain torch

def _phi(f_center, f_sigma, dt):
    """Phi(dt) of a Gaussian power spectrum, from the closed form of int w^n W(w) exp(i w t) dw: with
    E(t) = exp(i w0 t - s^2 t^2 / 2) the third derivative of E gives the numerator."""
    w0, s = 2 * math.pi * f_center, 2 * math.pi * f_sigma
    u = w0 + 1j * s * s * dt            # d/dt E = i u E, d/dt u = i s^2
    e = torch.exp(-0.5 * (s * dt) ** 2) * torch.exp(1j * w0 * dt)
    num = ((u ** 3 + 3 * s * s * u) * e).imag
    return num / (w0 * w0 + s * s)


BLK = 4   # culling blocks of 4 x 4 x 4 voxels


def _entries(c, x, keep_rows=None):
    """The in-support entries: yields (block of each of n pairs (ascending), row, J values (n, 64)), and
    the voxels of the blocks (n_blocks, 64) first, -1 outside the grid."""
    dev, g = torch.device("cuda"), _Grid(c)
    ax = g.axes(dev)
    n3 = (g.nx, g.ny, g.nz)
    nb = [-(-n // BLK) for n in n3]
    k = torch.arange(BLK, device=dev)
    idx = [torch.arange(b, device=dev)[:, None] * BLK + k for b in nb]   # (blocks of the axis, 4)
    bx = torch.arange(nb[0] * nb[1] * nb[2], device=dev)
    b3 = [bx % nb[0], (bx // nb[0]) % nb[1], bx // (nb[0] * nb[1])]
    ix, iy, iz = (idx[a][b3[a]] for a in range(3))
    ok = (iz < g.nz)[:, :, None, None] & (iy < g.ny)[:, None, :, None] & (ix < g.nx)[:, None, None, :]
    vox = (iz[:, :, None, None] * g.ny + iy[:, None, :, None]) * g.nx + ix[:, None, None, :]
    vox = torch.where(ok, vox, torch.full_like(vox, -1)).reshape(-1, BLK ** 3)
    yield vox
    full = [g.origin[a] + idx[a].double() * g.h for a in range(3)]
    rows = torch.as_tensor(x["rows"], device=dev).long()
    band = torch.as_tensor(x["band"], device=dev).long()
    ids = torch.arange(len(rows), device=dev) if keep_rows is None else keep_rows
    rows, band = rows[ids], band[ids]
    tx = torch.as_tensor(x["tx"], device=dev)
    s, r = tx[rows[:, 0]], tx[rows[:, 1]]
    L = (r - s).norm(dim=1)
    e, o = (r - s) / L[:, None], 0.5 * (s + r)
    dtm = torch.tensor([PERIODS / f for f, _ in _bands(c)], device=dev, dtype=torch.float64)
    U = (C0 * dtm)[band]
    C = -L * g.h ** 3 / (2 * math.pi * C0 ** 3)
    tabs = torch.stack([_phi(f, w, torch.linspace(0, PERIODS / f, N_TABLE, device=dev, dtype=torch.float64))
                        for f, w in _bands(c)])
    tabs[:, 0] = 0.0
    half = 0.5 * (BLK - 1) * g.h
    ctr = torch.stack([full[a][b3[a]].mean(1) for a in range(3)], dim=1)
    step = max(1, int(4e7 // max(1, len(rows))))
    per = 1 << 17
    for c0 in range(0, len(ctr), step):
        # R(x) is convex: its tangent plane at a block's centre bounds it from below over the block
        q = ctr[c0:c0 + step]
        low, grad = -L[None].expand(len(q), -1), None
        for t in (s, r):
            dl = [q[:, a, None] - t[None, :, a] for a in range(3)]
            dist = (dl[0] ** 2 + dl[1] ** 2 + dl[2] ** 2).sqrt().clamp_min(1e-12)
            u = [v / dist for v in dl]
            low = low + dist
            grad = u if grad is None else [p + v for p, v in zip(grad, u)]
        low = low - half * (grad[0].abs() + grad[1].abs() + grad[2].abs())
        bi, ri = torch.nonzero(low < U[None] * (1 + 1e-9), as_tuple=True)
        del low, grad, dl, dist, u
        bi += c0
        for a0 in range(0, len(bi), per):
            b, p = bi[a0:a0 + per], ri[a0:a0 + per]
            dx, dy, dz = (full[a][b3[a][b]] - o[p, a, None] for a in range(3))   # (n, 4) each
            ex, ey, ez = (e[p, a, None, None, None] for a in range(3))
            dx, dy, dz = dx[:, None, None, :], dy[:, None, :, None], dz[:, :, None, None]
            pp = dx * ex + dy * ey + dz * ez
            q2 = (dy * ez - dz * ey) ** 2 + (dz * ex - dx * ez) ** 2 + (dx * ey - dy * ex) ** 2
            hl = 0.5 * L[p, None, None, None]
            ps, pr = pp + hl, pp - hl
            Rs, Rr = (ps * ps + q2).sqrt(), (pr * pr + q2).sqrt()
            A, B = Rs + ps.abs(), Rr + pr.abs()
            R = q2 * (A + B) / (A * B).clamp_min(1e-300) + ((ps.abs() - ps) + (pr.abs() + pr))
            v = R / U[p, None, None, None]
            if c.get("phi") == "series":
                f, w = _bands(c)[0]
                phi = _phi(f, w, v * float(dtm[0]))
            else:
                t = (v * (N_TABLE - 1)).clamp(0, N_TABLE - 1)
                j = t.floor().clamp(max=N_TABLE - 2).long()
                at = band[p, None, None, None] * N_TABLE + j
                lo = tabs.reshape(-1)[at]
                phi = lo + (t - j) * (tabs.reshape(-1)[at + 1] - lo)
            # a voxel centre on a transducer has no K0 (its limit depends on the direction): 0 there
            off = (Rs > 1e-9) & (Rr > 1e-9)
            val = C[p, None, None, None] * phi / (Rs * Rr).clamp_min(1e-18)
            val = torch.where((R < U[p, None, None, None]) & off, val, torch.zeros_like(val))
            val = val.reshape(len(b), -1) * (vox[b] >= 0)
            yield b, ids[p], val


def _exact_J(c, x, m):
    """J m for the columns of m (n, V)."""
    gen = _entries(c, x)
    vox = next(gen).clamp_min(0)
    m = m.double()
    d = torch.zeros((len(m), len(x["rows"])), device=m.device, dtype=torch.float64)
    for b, p, val in gen:
        for k in range(len(m)):
            d[k].index_add_(0, p, (val * m[k][vox[b]]).sum(1))
    return d


def _gather(c, vox, g):
    out = torch.zeros((len(g), _Grid(c).n_vox), device=g.device, dtype=torch.float64)
    keep = vox >= 0
    out[:, vox[keep]] = g[:, keep]
    return out


def _exact_JT(c, x, d):
    gen = _entries(c, x)
    vox = next(gen)
    d = d.double()
    g = torch.zeros((len(d), *vox.shape), device=d.device, dtype=torch.float64)
    for b, p, val in gen:
        for k in range(len(d)):
            g[k].index_add_(0, b, val * d[k][p][:, None])
    return _gather(c, vox, g)


def _exact_psf(c, x):
    g = _Grid(c)
    dev = torch.device("cuda")
    spikes = torch.as_tensor(x["spikes"], device=dev)
    n_sub, n_row = len(x["subsets"]), len(x["rows"])
    # J at the spikes: the columns of D
    gen = _entries(c, x)
    vox = next(gen)
    where = torch.full((g.n_vox,), -1, device=dev, dtype=torch.long)
    where[spikes] = torch.arange(len(spikes), device=dev)
    at = torch.where(vox >= 0, where[vox.clamp_min(0)], torch.full_like(vox, -1))
    held = (at >= 0).any(1)
    D = torch.zeros((n_row, len(spikes)), device=dev, dtype=torch.float64)
    for b, p, val in gen:
        sel = held[b]
        if sel.any():
            i, j = torch.nonzero(at[b[sel]] >= 0, as_tuple=True)
            D[p[sel][i], at[b[sel]][i, j]] = val[sel][i, j]
    member = torch.zeros((n_row, n_sub), device=dev, dtype=torch.float64)
    for s, rows in enumerate(x["subsets"]):
        member[torch.as_tensor(rows, device=dev).long(), s] = 1.0
    live = torch.nonzero((D != 0).any(1) & (member != 0).any(1)).reshape(-1)
    W = torch.cat([D * member[:, s:s + 1] for s in range(n_sub)], dim=1)   # (rows, subset-major columns)
    out = torch.zeros((*vox.shape, W.shape[1]), device=dev, dtype=torch.float64)
    gen = _entries(c, x, live)
    next(gen)
    for b, p, val in gen:
        blocks, n = torch.unique_consecutive(b, return_counts=True)
        ends = torch.cumsum(n, 0).tolist()
        lo = 0
        for blk, hi in zip(blocks.tolist(), ends):
            out[blk].addmm_(val[lo:hi].T, W[p[lo:hi]])
            lo = hi
    full = torch.zeros((W.shape[1], g.n_vox), device=dev, dtype=torch.float64)
    keep = vox >= 0
    full[:, vox[keep]] = out[keep].T
    return full.reshape(n_sub, len(spikes), g.n_vox)


def _exact_cg(c, x):
    g = _Grid(c)
    gen = _entries(c, x)
    vox = next(gen)
    F = torch.zeros((len(x["rows"]), g.n_vox), device="cuda", dtype=torch.float64)
    for b, p, val in gen:
        ok = vox[b] >= 0
        F[p[:, None].expand_as(ok)[ok], vox[b][ok]] = val[ok]
    lam = LAMBDA_REL * float(sum((f * f).sum() for f in F.split(256))) / g.n_vox
    m = torch.zeros(g.n_vox, device="cuda", dtype=torch.float64)
    r = x["d"].double()
    s = F.T @ r
    p, gam = s.clone(), float(s @ s)
    for _ in range(c["iters"]):
        q = F @ p
        a = gam / (float(q @ q) + lam * float(p @ p))
        m += a * p
        r = r - a * q
        s = F.T @ r - lam * m
        gam, old = float(s @ s), gam
        p = s + (gam / old) * p
    return m


def _pair_estimate(c):
    m = len(_bands(c)) * c["slices"] * c["n_tx"] * (c["n_tx"] - 1) // 2
    return m, _Grid(c).n_vox


def exact(case, seed):
    c, op = case, case["op"]
    m, v = _pair_estimate(c)
    # about 20 s: the full volume's 4e11 entries take minutes, a dense operator has to fit
    if m * v > 4e11 or (op == "cg" and m * v > 6e9):
        return None
    if op == "psf" and m * v * c["spikes"] > 3e13:
        return None
    x = _inputs(c, seed)
    if op == "j":
        return _exact_J(c, x, x["m"][None])[0]
    if op == "jt":
        return _exact_JT(c, x, x["d"][None])[0]
    if op == "grad":
        d = _exact_J(c, x, x["m"][None])
        return d[0], _exact_JT(c, x, d - x["d"].double()[None])[0]
    if op == "cg":
        return _exact_cg(c, x)
    if op == "block":
        d = _exact_J(c, x, x["X"])
        return d, _exact_JT(c, x, d)
    if op == "psf":
        return _exact_psf(c, x)
    if op == "plane":
        g = _Grid(c)
        d = _exact_J(c, x, x["m2"].repeat(g.nz)[None])[0]
        return d, _exact_JT(c, x, x["d"][None])[0].reshape(g.nz, -1).sum(0)
    phi = []
    for f, w in _bands(c):
        t = _phi(f, w, torch.linspace(0, PERIODS / f, N_TABLE, dtype=torch.float64))
        t[0] = 0.0
        phi.append(t)
    return phi, _exact_J(c, x, x["m"][None])[0]


if __name__ == "__main__":
    for case_ in listed() + [draw(random.Random(k)) for k in range(6)]:
        w_ = work(case_)
        print(case_, "%.3g bytes %.3g operations" % (w_["bytes"], w_["flops"]))
