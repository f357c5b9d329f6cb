"""Passes of one to eight columns (the batch kernels with columns missing, their remainders, and the
partial buffers grown from four columns to eight) against the single-column products: 2e-6 relative
L2 per column, the bound of the four-column kernels (each is within 1e-6 of the exact product)."""
import numpy as np
import pytest

import workloads as wl
from gpu_common import gpu_geometry, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sharp", [False, True])
@pytest.mark.parametrize("order", [(4, 5, 8, 9, 13), (8, 7, 4, 6, 11)])
def test_columns(sharp, order):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_03302_gb300 as fg
    fg._lib.load()
    if sharp:   # slices32's bands; an odd grid that cuts tiles and sub-bricks
        w = wl.slices32()
        tabs = [fg.Table(b.f_center_hz, b.f_sigma_hz, b.n_samples, b.dt_max) for b in w.bands]
        geo = fg.Geometry(w.tx, w.row_pairs(), wl.Grid.centred(45, 43, 19, 2e-3), w.c0, tabs, band_of_row=w.band_of_row)
    else:
        geo, _ = gpu_geometry(wl.ring32())
    rng = np.random.default_rng(7)
    for n in order:
        X, D = to_dev(rng.normal(size=(n, geo.V))), to_dev(rng.normal(size=(n, geo.M)))
        JX, JTD = geo.J_batch(X), geo.JT_batch(D)
        assert torch.equal(JX, geo.J_batch(X)) and torch.equal(JTD, geo.JT_batch(D))
        for c in range(n):
            assert rel_l2(to_np(JX[c]), to_np(geo.J(X[c].contiguous()))) <= 2e-6
            assert rel_l2(to_np(JTD[c]), to_np(geo.JT(D[c].contiguous()))) <= 2e-6
