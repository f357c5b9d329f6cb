"""Out of memory while an operator is retuned (allocations made to fail on the host): the call reports
it, the operator keeps working with the decomposition it had, or refuses every call if not even that
one can be had, until a tuning succeeds."""
import numpy as np
import pytest

import workloads as wl
from gpu_common import gpu_geometry, to_dev
from test_gpu_stack import BANDS, acquisition, layers_of

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def operator(fg, stack):
    if not stack:
        return gpu_geometry(wl.slices32())[0]
    tx, rows, bor = acquisition(layers_of(5, 3), "slices")
    return fg.Geometry(tx, rows, wl.Grid.centred(47, 46, 24, 1.5e-3), 1500.0,
                       [fg.Table(f, s, 4096, d) for f, s, d in BANDS], band_of_row=bor)


@pytest.mark.parametrize("stack", [False, True])
# (four allocations a candidate; with a stack three for a class's operator, and the J^T partials' if they grow)
@pytest.mark.parametrize("after", [0, 1, 3, 4, 6, 8, 9])
def test_one_allocation_fails(stack, after):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_03302_gb300 as fg
    L = fg._lib.load()
    geo = operator(fg, stack)
    rng = np.random.default_rng(2)
    m, d = to_dev(rng.normal(size=geo.V)), to_dev(1e-8 * rng.normal(size=geo.M))
    calls = lambda: [geo.J(m), geo.JT(d), geo.cg_solve(d, 1e-3, 3), geo.J_batch(torch.stack([m] * 4))]   # noqa: E731
    before = [t.clone() for t in calls()]
    info = geo.info()
    try:
        L.fft_fail_alloc(after, 1)
        with pytest.raises(fg.FFTError) as ei:
            geo.autotune()
    finally:
        L.fft_fail_alloc(0, 0)
    assert ei.value.status == fg._lib.FFT_ERR_OOM
    assert geo.info().n_items == info.n_items
    for a, b in zip(before, calls()):
        assert torch.equal(a, b)
    if not stack:   # (a stack keeps the larger partial buffer of a candidate)
        assert geo.info().scratch_bytes == info.scratch_bytes


@pytest.mark.parametrize("stack", [False, True])
def test_every_allocation_fails(stack):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_03302_gb300 as fg
    L = fg._lib.load()
    geo = operator(fg, stack)
    rng = np.random.default_rng(2)
    m, d = to_dev(rng.normal(size=geo.V)), to_dev(1e-8 * rng.normal(size=geo.M))
    want = geo.J(m).clone()
    geo.cg_solve(d, 1e-3, 3)
    try:
        L.fft_fail_alloc(6, 1 << 30)
        with pytest.raises(fg.FFTError) as ei:
            geo.autotune()
    finally:
        L.fft_fail_alloc(0, 0)
    assert ei.value.status == fg._lib.FFT_ERR_OOM
    for call in (lambda: geo.J(m), lambda: geo.JT(d), lambda: geo.cg_solve(d, 1e-3, 3), lambda: geo.coverage(),
                 lambda: geo.J_batch(torch.stack([m] * 5)), lambda: geo.J2d(m[:geo.V2].contiguous())):
        with pytest.raises(fg.FFTError) as ei:
            call()
        assert ei.value.status == fg._lib.FFT_ERR_STATE
    geo.autotune()
    assert torch.equal(geo.J(m), want)


@pytest.mark.parametrize("after", [0, 10, 20, 30, 40, 60])
def test_a_stack_that_does_not_fit_is_left_out(after):
    """Creation with one allocation failing: refused, or an operator that agrees with the whole one."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1908_03302_gb300 as fg
    L = fg._lib.load()
    whole = operator(fg, True)
    m = to_dev(np.random.default_rng(2).normal(size=whole.V))
    want = whole.J(m)
    try:
        L.fft_fail_alloc(after, 1)
        geo = operator(fg, True)
    except fg.FFTError as e:
        assert e.status == fg._lib.FFT_ERR_OOM
        return
    finally:
        L.fft_fail_alloc(0, 0)
    assert float((geo.J(m) - want).norm() / want.norm()) <= 2e-6
