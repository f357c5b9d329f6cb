"""The two evaluations of a sine series inside the products: piecewise quadratics in shared memory
where they fit, the Clenshaw recurrence where they do not (five bands cut after six periods need
4096 segments each, 246 KB). Both against the FP64 oracle's series, 1e-5 relative L2 as for every
J / J^T path: the quadratics add 5e-8 of max |Phi|, the FP32 detour (1e-7 of the cut-off) times
the phase of six periods 4e-6 per entry."""
import numpy as np
import pytest

import oracle
import workloads as wl
from gpu_common import rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_bands,periods", [(1, 3.0), (2, 6.0), (5, 6.0)])
def test_series_evaluations_match_oracle(n_bands, periods):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_03302_gb300 as fg
    w = wl.tiny()
    rows = w.row_pairs()
    bor = (np.arange(len(rows)) % n_bands).astype(np.int32)
    bands = [(0.8e6 + 0.1e6 * k, 0.3e6, periods / (0.8e6 + 0.1e6 * k)) for k in range(n_bands)]
    geo = fg.Geometry(w.tx, rows, w.grid, w.c0, [fg.TrigTable(*b) for b in bands], band_of_row=bor)
    series = [oracle.trig_coefs(*b) for b in bands]
    og = oracle.Geometry(w.tx, rows, bor, [a for a, _ in series], [b[2] for b in bands], w.grid, w.c0,
                         trig_dw=[dw for _, dw in series])
    m = np.random.default_rng(1).normal(size=og.V)
    d = np.random.default_rng(2).normal(size=og.M)
    assert rel_l2(to_np(geo.J(to_dev(m))), og.J(m)) <= 1e-5
    assert rel_l2(to_np(geo.JT(to_dev(d))), og.JT(d)) <= 1e-5
    X = np.random.default_rng(3).normal(size=(4, og.V))
    JX = to_np(geo.J_batch(to_dev(X)))
    assert rel_l2(JX[3], og.J(X[3])) <= 1e-5
