"""Infinite data in J^T: a voxel inside the support of a row with infinite weight gets that infinity with
the sign of its entry, however many partial sums its tile has (0 x infinity outside the support, inside
an evaluated brick, is NaN as ever)."""
import numpy as np
import pytest

import workloads as wl
from gpu_common import gpu_geometry, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("name", ["ring32", "slices32"])
@pytest.mark.parametrize("where", [0.02, 0.5, 0.9])
def test_infinite_weight(name, where):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    geo, _ = gpu_geometry(wl.by_name(name))
    p = int(where * geo.M)
    e = torch.zeros(geo.M, device="cuda")
    e[p] = 1.0
    entry = geo.JT(e)                                  # column p of J^T
    hit = entry != 0
    assert hit.any()
    d = to_dev(1e-8 * np.random.default_rng(1).normal(size=geo.M))
    for v in (float("inf"), float("-inf")):
        d[p] = v
        want = torch.where(entry[hit] > 0, v, -v)
        assert torch.equal(geo.JT(d)[hit], want)
        D = torch.stack([d] * 4 + [e])
        assert all(torch.equal(g[hit], want) for g in geo.JT_batch(D)[:4])
