"""A handle keeps working after another one with smaller tables was made: every product and a solve give
the same bits before and after (the kernels' shared-memory limit is the process's, not the handle's)."""
import numpy as np
import pytest

import workloads as wl
from gpu_common import gpu_geometry, to_dev
from test_gpu_stack import acquisition, layers_of

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BANDS = [(0.6e6, 0.2e6), (1.0e6, 0.3e6), (1.4e6, 0.2e6)]   # the last is sharp


@pytest.mark.parametrize("kind,n_bands", [("table", 2), ("table", 3), ("series", 2), ("stack", 2)])
def test_first_handle_after_a_smaller_one(kind, n_bands):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_03302_gb300 as fg
    fg._lib.load()
    make = fg.TrigTable if kind == "series" else (lambda f, s: fg.Table(f, s, 4096, 3.0 / f))
    tabs = [make(f, s) for f, s in BANDS[1:1 + n_bands] + BANDS[:max(0, n_bands - 2)]]
    if kind == "stack":
        tx, rows, bor = acquisition(layers_of(4, 4), "slices")
        grid = wl.Grid.centred(47, 46, 24, 1.5e-3)
    else:
        tx = wl.ring(32, 36e-3)
        rows = np.tile(wl.unordered_pairs(range(32)), (n_bands, 1)).astype(np.int32)
        bor = np.repeat(np.arange(n_bands, dtype=np.int32), len(rows) // n_bands)
        grid = wl.Grid.centred(33, 31, 17, 2e-3)
    geo = fg.Geometry(tx, rows, grid, 1500.0, tabs, band_of_row=bor)
    rng = np.random.default_rng(3)
    X, D = to_dev(rng.normal(size=(8, geo.V))), to_dev(1e-8 * rng.normal(size=(8, geo.M)))
    spikes = np.array([geo.V // 2], dtype=np.int64)
    subs = [np.arange(geo.M, dtype=np.int32)]

    def calls():
        out = [geo.J(X[0]), geo.JT(D[0]), geo.J_batch(X), geo.JT_batch(D), geo.J_batch(X[:4].contiguous()),
               geo.JT_batch(D[:4].contiguous()), geo.coverage(), geo.cg_solve(D[0], 1e-3, 3)]
        return out if kind == "series" else out + [geo.psf_batch(spikes, subs, mode=k) for k in (0, 1, 2)]

    before = [t.clone() for t in calls()]
    small, _ = gpu_geometry(wl.tiny())
    small.J(to_dev(rng.normal(size=small.V)))
    for a, b in zip(before, calls()):
        assert torch.equal(a, b)
