"""Which evaluation the acquisitions of the mirror, stack, batch, series and solver tests take: those tests compare
it with the general path, which says nothing if both sides took that."""
import numpy as np
import pytest

import test_gpu_mirror
import workloads as wl
from gpu_common import gpu_geometry, to_dev
from test_gpu_stack import BANDS, CASES, H, acquisition

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def fg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_03302_gb300 as m
    m._lib.load()
    return m


MIRRORS = [m for m in test_gpu_mirror.test_mirrored_products.pytestmark if m.name == "parametrize"][0].args[1]


@pytest.mark.parametrize("plane,nz,mirrors", MIRRORS)
def test_mirror_planes(fg, plane, nz, mirrors):
    h = 1.5e-3
    pairs = wl.unordered_pairs(range(128))
    geo = fg.Geometry(wl.ring(128, 35e-3), np.concatenate([pairs, pairs]),
                      wl.Grid(39, 36, nz, h, (-28.5e-3, -26.25e-3, -plane * h)), 1500.0,
                      [fg.Table(f, s, 4096, d) for f, s, d in test_gpu_mirror.BANDS],
                      band_of_row=np.repeat(np.arange(2, dtype=np.int32), len(pairs)))
    assert geo.route()["mirror"] == (int(2 * plane) if mirrors else -1)


@pytest.mark.parametrize("series", [False, True])
@pytest.mark.parametrize("layers,nz,order,odd,stack", CASES)
def test_stacks(fg, layers, nz, order, odd, stack, series):
    tx, rows, bor = acquisition(layers, order, odd)
    far = np.array([[0.5, 0.5, 0.5], [0.51, 0.5, 0.53]])
    grid = wl.Grid(47, 46, nz, H, (-34.5e-3, -33.75e-3, -(nz - 1) * H / 2))
    tabs = [fg.TrigTable(f, s) if series else fg.Table(f, s, 4096, d) for f, s, d in BANDS]
    geo = fg.Geometry(tx, rows, grid, 1500.0, tabs, band_of_row=bor)
    # one class per fraction of a layer; an odd slice is a class of its own beside the others'
    classes = 2 if odd else (len({round((z - layers[0]) % 1.0, 6) % 1.0 for z in layers}) if stack else 0)
    assert geo.route()["stack_classes"] == classes
    assert (geo.route()["segments"] > 0) == series
    gen = fg.Geometry(np.concatenate([tx, far]), np.concatenate([rows, [[len(tx), len(tx) + 1]]]).astype(np.int32), grid,
                      1500.0, tabs, band_of_row=np.append(bor, 0).astype(np.int32))
    assert gen.route()["stack_classes"] == 0 and gen.route()["mirror"] == -1


@pytest.mark.parametrize("n_tx,n,step,grid,classes,psf", [
    (64, 11, 3e-3, (120, 113, 40, 1e-3), 1, 0), (100, 5, 8e-3, (120, 113, 60, 1e-3), 1, 1),
    (128, 2, 3e-3, (180, 173, 40, 1e-3), 1, 3), (96, 9, 2e-3, (100, 93, 30, 1.5e-3), 3, 0)])
def test_sparse_columns_of_stacks(fg, n_tx, n, step, grid, classes, psf):
    """PSFs take the classes where a stack is dense enough in entries, in either mode the values of the general path
    (2e-6: each is within 1e-6 of the exact PSF)."""
    ring, pairs = wl.ring(n_tx, 85e-3), wl.unordered_pairs(range(n_tx))
    tx = np.concatenate([ring + [0.0, 0.0, (k - (n - 1) / 2) * step] for k in range(n)])
    rows = np.concatenate([pairs + n_tx * k for k in range(n)]).astype(np.int32)
    far = np.array([[0.5, 0.5, 0.5], [0.51, 0.5, 0.53]])
    tab = fg.Table(1.0e6, 0.4e6)
    geo = fg.Geometry(tx, rows, wl.Grid.centred(*grid), 1500.0, [tab])
    gen = fg.Geometry(np.concatenate([tx, far]), np.concatenate([rows, [[len(tx), len(tx) + 1]]]).astype(np.int32),
                      wl.Grid.centred(*grid), 1500.0, [tab])
    assert (geo.route()["stack_classes"], geo.route()["stack_psf"]) == (classes, psf)
    nx, ny, nz, _ = grid
    middle = (nz // 2 * ny + ny // 2) * nx + nx // 2
    spikes = np.array([middle, middle + 7], dtype=np.int64)
    subs = [np.arange(geo.M, dtype=np.int32), np.arange(0, geo.M, 2, dtype=np.int32)]
    for mode in (0, 2):
        a, b = (g.psf_batch(spikes, subs, mode=mode).double() for g in (geo, gen))
        assert float((a - b).norm() / b.norm()) <= 2e-6
    one = geo.psf_noalloc(middle, torch.arange(geo.M, device="cuda", dtype=torch.int32)).double()
    assert float((one - b[0, 0]).norm() / b[0, 0].norm()) <= 2e-6


def test_batch_width_grows_once(fg):
    geo, _ = gpu_geometry(wl.slices32())
    rng = np.random.default_rng(4)
    X, D = to_dev(rng.normal(size=(9, geo.V))), to_dev(1e-8 * rng.normal(size=(9, geo.M)))
    assert geo.route()["batch_cols"] == 0 and geo.route()["solver_comp"] == 1 and geo.route()["launches"] == 3
    geo.J_batch(X[:4].contiguous())
    assert geo.route()["batch_cols"] == 4
    want = [(geo.J_batch(X[:n].contiguous()).clone(), geo.JT_batch(D[:n].contiguous()).clone()) for n in (5, 8, 9)]
    assert geo.route()["batch_cols"] == 8
    # a handle that has no memory for eight: the same bits from passes of four, and it is not asked again
    other, _ = gpu_geometry(wl.slices32())
    other.J_batch(X[:4].contiguous())
    try:
        fg._lib.load().fft_fail_alloc(0, 1)
        other.J_batch(X[:5].contiguous())
    finally:
        fg._lib.load().fft_fail_alloc(0, 0)
    for n, (j, jt) in zip((5, 8, 9), want):
        assert torch.equal(other.J_batch(X[:n].contiguous()), j) and torch.equal(other.JT_batch(D[:n].contiguous()), jt)
    assert other.route()["batch_cols"] == 4


def test_large_solves_keep_plain_products(fg):
    geo, _ = gpu_geometry(wl.ring256())
    assert geo.route() == {"mirror": wl.ring256().grid.nz - 1, "stack_classes": 0, "stack_batch": 0, "stack_psf": 0, "batch_cols": 0,
                           "segments": 0, "solver_comp": 0, "launches": 2}
