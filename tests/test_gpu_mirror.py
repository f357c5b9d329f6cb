"""Acquisitions whose transducers lie in a mirror plane of the voxel lattice: one evaluation serves a
layer and its image. Against the general path (the same rows plus one out-of-plane row far outside
the grid, which switches the mirroring off) to 2e-6 relative L2 (each is within 1e-6 of the exact
product) and, for two of them, against the FP64 oracle to 1e-5; planes on a layer, between layers,
off the middle in both directions, at the first layers, and planes that mirror nothing."""
import numpy as np
import pytest

import oracle
import workloads as wl
from gpu_common import rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BANDS = [(1.0e6, 0.3e6, 3e-6), (1.4e6, 0.2e6, 3 / 1.4e6)]   # the second is sharp


# plane position in layers (K = 2 x that), layers, is there anything to mirror?
@pytest.mark.parametrize("plane,nz,mirrors", [
    (8.5, 18, True), (9.0, 19, True), (4.0, 19, True), (13.5, 17, True), (0.5, 17, True), (15.0, 17, True), (20.0, 24, True),
    (2.25, 9, False), (0.0, 9, False), (8.0, 9, False), (-1.0, 9, False)])
def test_mirrored_products(plane, nz, mirrors):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_03302_gb300 as fg
    h = 1.5e-3
    grid = wl.Grid(39, 36, nz, h, (-28.5e-3, -26.25e-3, -plane * h))
    tx = wl.ring(128, 35e-3)
    pairs = wl.unordered_pairs(range(128))
    rows = np.concatenate([pairs, pairs])
    bor = np.repeat(np.arange(2, dtype=np.int32), len(pairs))
    far = np.array([[0.5, 0.5, 0.5], [0.51, 0.5, 0.53]])
    tabs = [fg.Table(f, s, 4096, d) for f, s, d in BANDS]
    geo = fg.Geometry(tx, rows, grid, 1500.0, tabs, band_of_row=bor)
    gen = fg.Geometry(np.concatenate([tx, far]), np.concatenate([rows, [[128, 129]]]).astype(np.int32), grid, 1500.0,
                      tabs, band_of_row=np.append(bor, 0).astype(np.int32))
    assert geo.info().n_entries == gen.info().n_entries >= (65536 if mirrors else 0)
    rng = np.random.default_rng(3)
    m, d, w = (to_dev(rng.normal(size=n)) for n in (geo.V, geo.M, geo.M))
    more = lambda x: torch.cat([x, torch.zeros_like(x[..., :1])], dim=-1).contiguous()   # noqa: E731
    J, JT = to_np(geo.J(m)), to_np(geo.JT(d))
    if mirrors:   # a layer and its image come from the same evaluation
        K = int(2 * plane)
        k = [k for k in range(nz) if 0 <= K - k < nz]
        layers = JT.reshape(nz, -1)
        assert np.array_equal(layers[k], layers[[K - i for i in k]])
    assert rel_l2(J, to_np(gen.J(m))[:-1]) <= 2e-6
    assert rel_l2(JT, to_np(gen.JT(more(d)))) <= 2e-6
    assert rel_l2(to_np(geo.coverage(w)), to_np(gen.coverage(more(w)))) <= 2e-6
    assert geo.frob2() == pytest.approx(gen.frob2(), rel=2e-6)
    # (a plain band counts by its FP32 detour: the bound that the support counts are tested to elsewhere)
    assert abs(geo.support_evals - gen.support_evals) <= 1e-4 * gen.support_evals
    X, D = to_dev(rng.normal(size=(4, geo.V))), to_dev(rng.normal(size=(4, geo.M)))
    assert rel_l2(to_np(geo.J_batch(X)), to_np(gen.J_batch(X))[:, :-1]) <= 2e-6
    assert rel_l2(to_np(geo.JT_batch(D)), to_np(gen.JT_batch(more(D)))) <= 2e-6
    spikes = rng.choice(geo.V, size=3, replace=False).astype(np.int64)
    subs = [np.arange(0, geo.M, 2, dtype=np.int32), np.arange(geo.M, dtype=np.int32)]
    for mode in (0, 1, 2):
        a, b = to_np(geo.psf_batch(spikes, subs, mode=mode)), to_np(gen.psf_batch(spikes, subs, mode=mode))
        assert rel_l2(a, b) <= 2e-6
    if (plane, nz) in ((8.5, 18), (4.0, 19)):
        og = oracle.Geometry(tx, rows, bor, [oracle.phi_table_gauss(f, s, 4096, t) for f, s, t in BANDS],
                             [b[2] for b in BANDS], grid, 1500.0)
        assert rel_l2(J, og.J(to_np(m))) <= 1e-5
        assert rel_l2(JT, og.JT(to_np(d))) <= 1e-5
