"""Batch products in CUDA graphs: a captured call replays to the same bits after later, wider calls (its
scratch stays where it was), and passes of four and of eight columns give a column the same bits."""
import numpy as np
import pytest

import workloads as wl
from gpu_common import gpu_geometry, to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("name", ["ring32", "slices32"])
def test_replay_after_a_wider_call(name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    geo, _ = gpu_geometry(wl.by_name(name))
    rng = np.random.default_rng(11)
    X, D = to_dev(rng.normal(size=(13, geo.V))), to_dev(1e-8 * rng.normal(size=(13, geo.M)))
    cols = (4, 5, 7, 8, 9, 13)
    cut = {n: (X[:n].contiguous(), D[:n].contiguous()) for n in cols}
    geo.J_batch(cut[4][0]), geo.JT_batch(cut[4][1])      # four-column scratch
    small = geo.info().scratch_bytes
    out = {n: (torch.zeros(n, geo.M, device="cuda"), torch.zeros(n, geo.V, device="cuda")) for n in cols}
    side = torch.cuda.Stream()
    graphs = {}
    for n in cols:   # captured while there is scratch for four columns only
        graphs[n] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graphs[n], stream=side):
            geo.J_batch(cut[n][0], out=out[n][0])
            geo.JT_batch(cut[n][1], out=out[n][1])
    assert geo.info().scratch_bytes == small
    torch.cuda.synchronize()
    wide = {n: (geo.J_batch(cut[n][0]).clone(), geo.JT_batch(cut[n][1]).clone()) for n in cols}
    assert geo.info().scratch_bytes > small   # the wider one came beside it
    torch.cuda.synchronize()
    # (what was freed would be used again)
    taken = [torch.full((1 << 22,), float("nan"), device="cuda") for _ in range(16)]
    for n in cols:
        for _ in range(2):
            out[n][0].zero_(), out[n][1].zero_()
            torch.cuda.synchronize()
            graphs[n].replay()
            torch.cuda.synchronize()
            assert torch.equal(out[n][0], wide[n][0]) and torch.equal(out[n][1], wide[n][1])
    del taken
