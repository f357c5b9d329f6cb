"""The solver's compensated products over the forms they exist in: tables, sine series as quadratics and by the
recurrence, sharp bands, voxels on transducers, a mirror plane, tiles with one item and with none. The saved
state shows them: p after no iteration is J^T d, and d - r after one is a multiple of J p. Against the plain
products of the same entries: 5e-7 (their FP32 sums are within 2e-7, the saved vectors add a rounding)."""
import numpy as np
import pytest

import workloads as wl
from gpu_common import to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHARP = [(1.0e6, 0.3e6, 3e-6), (1.4e6, 0.2e6, 3 / 1.4e6)]


def case(fg, kind):
    tx, grid, n = wl.ring(24, 36e-3, 0.3e-3), wl.Grid.centred(35, 33, 19, 2e-3), 1
    tabs = [fg.Table(1.0e6, 0.3e6)]
    if kind == "sharp":
        n, tabs = 2, [fg.Table(f, s, 4096, d) for f, s, d in SHARP]
    elif kind == "series":
        n, tabs = 2, [fg.TrigTable(*b) for b in SHARP]
    elif kind == "recurrence":
        n, tabs = 5, [fg.TrigTable(f, 0.3e6, 6 / f) for f in (0.8e6 + 0.1e6 * np.arange(5))]
    elif kind == "on a voxel":
        tx = np.round(tx / 2e-3) * 2e-3
        tx = np.unique(tx, axis=0)
    elif kind == "mirror":
        tx, grid = wl.ring(128, 35e-3), wl.Grid.centred(39, 36, 18, 1.5e-3)
        n, tabs = 2, [fg.Table(f, s, 4096, d) for f, s, d in SHARP]
    elif kind == "few rows":   # tiles with one item or none
        tx, grid = wl.ring(5, 60e-3), wl.Grid.centred(49, 47, 19, 2e-3)
    pairs = wl.unordered_pairs(range(len(tx)))
    return fg.Geometry(tx, np.tile(pairs, (n, 1)).astype(np.int32), grid, 1500.0, tabs,
                       band_of_row=np.repeat(np.arange(n, dtype=np.int32), len(pairs)))


@pytest.mark.parametrize("kind", ["table", "sharp", "series", "recurrence", "on a voxel", "mirror", "few rows"])
def test_products_of_the_solver(kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_03302_gb300 as fg
    fg._lib.load()
    geo = case(fg, kind)
    route = geo.route()
    assert route["solver_comp"] == 1 and (route["mirror"] >= 0) == (kind == "mirror")
    assert (route["segments"] > 0) == (kind == "series")
    d = to_dev(1e-8 * np.random.default_rng(8).normal(size=geo.M))

    def state(n):
        geo.cg_solve(d, 1e-3, n)
        v = geo.cg_save()[64:].view(np.float32)
        return [torch.as_tensor(x.copy(), device="cuda") for x in np.split(v, [geo.V, 2 * geo.V])]

    _, p, r = state(0)
    want = geo.JT(d).double()
    assert torch.equal(r, d)
    assert float((p.double() - want).norm() / want.norm()) <= 5e-7
    assert torch.equal(p == 0, want == 0)
    _, _, r1 = state(1)
    step, q = d.double() - r1.double(), geo.J(p).double()
    a = float(step @ q) / float(q @ q)
    off = float((step - a * q).norm())
    assert off <= 5e-7 * float(step.norm()) + 6e-8 * float(r1.double().norm())
