"""Elevation stacks: slices a whole number of layers apart share one evaluation. Against the general
path (the same rows plus one out-of-plane row far outside the grid, which is no stack) to 2e-6
relative L2 (each is within 1e-6 of the exact product) and, for one of them, against the FP64 oracle
to 1e-5; 2 to 9 slices (every remainder of the four-column passes), one and several classes, planes on
layers and between them, slices outside the grid, rows in slice, interleaved and descending order,
tables and sine series, and slices that are not alike."""
import numpy as np
import pytest

import oracle
import workloads as wl
from gpu_common import rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

BANDS = [(1.0e6, 0.3e6, 3e-6), (1.4e6, 0.2e6, 3 / 1.4e6)]   # the second is sharp
H = 1.5e-3


def acquisition(layers, order, odd=None, n=256):
    """One ring per entry of `layers` (in voxel layers from the middle); rows of both bands."""
    ring = wl.ring(n, 36e-3)
    tx = np.concatenate([ring + [0.0, 0.0, z * H] for z in layers])
    pairs = wl.unordered_pairs(range(n))
    rows = np.concatenate([pairs + n * s for s in range(len(layers))])
    if odd == "radius":      # one slice of another radius
        tx[:n, :2] *= 0.97
    if odd == "missing":     # one slice without its last row
        rows = rows[:-1]
    rows, bor = np.concatenate([rows, rows]), np.repeat(np.arange(2, dtype=np.int32), len(rows))
    if order == "interleaved":   # pair by pair, all slices of a pair together
        k = np.arange(len(rows)).reshape(2, len(layers), -1).transpose(0, 2, 1).reshape(-1)
    elif order == "descending":
        k = np.arange(len(rows)).reshape(2, len(layers), -1)[:, ::-1].reshape(-1)
    else:
        k = np.arange(len(rows))
    return tx, np.ascontiguousarray(rows[k].astype(np.int32)), np.ascontiguousarray(bor[k])


def layers_of(n, step, start=None):
    z = np.arange(n) * float(step)
    return z - (z[-1] / 2 if start is None else -start)


CASES = [  # layers of the slices, layers of the grid, order, oddity, a stack?
    (layers_of(2, 6), 24, "slices", None, True),
    (layers_of(3, 4), 23, "descending", None, True),
    (layers_of(4, 5), 24, "interleaved", None, True),
    (layers_of(5, 3), 24, "slices", None, True),
    (layers_of(6, 16 / 3, -13.0), 24, "slices", None, False),          # three classes of two, one of them mirrored
    (layers_of(9, 8 / 3), 25, "slices", None, True),                   # three classes of three
    (layers_of(5, 8, -14.25), 24, "slices", None, True),               # a plane that mirrors nothing
    (layers_of(4, 9, -9.0), 17, "slices", None, True),                 # the highest slice above the grid
    (layers_of(4, 5), 24, "slices", "radius", False),
    (layers_of(4, 5), 24, "slices", "missing", False),
    (layers_of(4, 5.3), 24, "slices", None, False),
]


@pytest.mark.parametrize("series", [False, True])
@pytest.mark.parametrize("layers,nz,order,odd,stack", CASES)
def test_stacked_products(layers, nz, order, odd, stack, series):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_03302_gb300 as fg
    if series and (odd or order != "slices"):
        pytest.skip("Phi does not matter to how rows are grouped")
    grid = wl.Grid(47, 46, nz, H, (-34.5e-3, -33.75e-3, -(nz - 1) * H / 2))
    tx, rows, bor = acquisition(layers, order, odd)
    far = np.array([[0.5, 0.5, 0.5], [0.51, 0.5, 0.53]])
    tabs = [fg.TrigTable(f, s) if series else fg.Table(f, s, 4096, d) for f, s, d in BANDS]
    geo = fg.Geometry(tx, rows, grid, 1500.0, tabs, band_of_row=bor)
    gen = fg.Geometry(np.concatenate([tx, far]), np.concatenate([rows, [[len(tx), len(tx) + 1]]]).astype(np.int32), grid,
                      1500.0, tabs, band_of_row=np.append(bor, 0).astype(np.int32))
    assert geo.info().n_entries == gen.info().n_entries > 1 << 20
    rng = np.random.default_rng(5)
    m, d, w = (to_dev(rng.normal(size=n)) for n in (geo.V, geo.M, geo.M))
    more = lambda x: torch.cat([x, torch.zeros_like(x[..., :1])], dim=-1).contiguous()   # noqa: E731
    J, JT = to_np(geo.J(m)), to_np(geo.JT(d))
    assert rel_l2(J, to_np(gen.J(m))[:-1]) <= 2e-6
    assert rel_l2(JT, to_np(gen.JT(more(d)))) <= 2e-6
    if stack and order == "slices" and abs(layers[-1] - layers[0]) < nz:
        # the same data on two slices that one four-column pass serves: the same image, shifted (a single
        # column left over goes through the single-column kernel, whose units are larger)
        per = len(rows) // (2 * len(layers))
        off = (layers - layers[0]) - np.round(layers - layers[0])
        same = [s for s in range(len(layers)) if abs(off[s]) < 1e-9][:4]
        k = int(round(layers[same[-1]] - layers[0]))
        one = rng.normal(size=2 * per)
        img = []
        for s in (0, same[-1]):
            x = np.zeros((2, len(layers), per))
            x[:, s] = one.reshape(2, per)
            img.append(to_np(geo.JT(to_dev(x.reshape(-1)))).reshape(nz, -1))
        assert np.array_equal(img[0][:nz - k], img[1][k:])
    assert rel_l2(to_np(geo.coverage(w)), to_np(gen.coverage(more(w)))) <= 2e-6
    assert geo.frob2() == pytest.approx(gen.frob2(), rel=2e-6)
    # (a plain band counts by its FP32 detour: the bound that the support counts are tested to elsewhere)
    assert abs(geo.support_evals - gen.support_evals) <= 1e-4 * gen.support_evals
    for n in (2, 4, 6):
        X, D = to_dev(rng.normal(size=(n, geo.V))), to_dev(rng.normal(size=(n, geo.M)))
        assert rel_l2(to_np(geo.J_batch(X)), to_np(gen.J_batch(X))[:, :-1]) <= 2e-6
        assert rel_l2(to_np(geo.JT_batch(D)), to_np(gen.JT_batch(more(D)))) <= 2e-6
    if not series:
        spikes = rng.choice(geo.V, size=3, replace=False).astype(np.int64)
        subs = [np.arange(0, geo.M, 2, dtype=np.int32), np.arange(geo.M, dtype=np.int32)]
        for mode in (0, 2):
            a, b = to_np(geo.psf_batch(spikes, subs, mode=mode)), to_np(gen.psf_batch(spikes, subs, mode=mode))
            assert rel_l2(a, b) <= 2e-6
        if len(layers) == 2:
            og = oracle.Geometry(tx, rows, bor, [oracle.phi_table_gauss(f, s, 4096, t) for f, s, t in BANDS],
                                 [b[2] for b in BANDS], grid, 1500.0)
            assert rel_l2(J, og.J(to_np(m))) <= 1e-5
            assert rel_l2(JT, og.JT(to_np(d))) <= 1e-5


def test_solves_tuning_and_capture_of_a_stack():
    """A captured solve, a retuned operator and the solve captured anew agree; J is the same bits."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_03302_gb300 as fg
    tx, rows, bor = acquisition(layers_of(5, 3), "slices")
    grid = wl.Grid(47, 46, 24, H, (-34.5e-3, -33.75e-3, -23 * H / 2))
    geo = fg.Geometry(tx, rows, grid, 1500.0, [fg.Table(f, s, 4096, d) for f, s, d in BANDS], band_of_row=bor)
    m = to_dev(np.random.default_rng(1).normal(size=geo.V))
    d = geo.J(m)
    x0 = to_np(geo.cg_solve(d, 1e-3, 5))
    t = geo.autotune()
    assert t["ms_J"] > 0 and t["ms_JT"] > 0
    assert torch.equal(geo.J(m), d)
    assert rel_l2(to_np(geo.cg_solve(d, 1e-3, 5)), x0) <= 1e-5
