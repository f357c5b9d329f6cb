"""The solver's own rounding: how far fft_cg_solve is from CGLS in FP64 on the same operator.

The operator's entries are read off the device (J of unit models), so what is compared is the solver
and its products' sums, not the entries. A solve of the small slice-by-slice acquisition amplifies
rounding, by a factor that depends on the data; the yardstick is the least that the saved state's
FP32 vectors allow: FP64 CGLS with m, p and r rounded to FP32 in every iteration and nothing else. Over 24
data sets the geometric mean of the distance has to stay within 1.6 times the yardstick's (the two are
draws of the same amplification: the logarithm of one distance scatters by about 0.8 around its mean, the
mean of 24 differences by 0.23, and 1.6 is two of those). Products with plain FP32 sums are at 2 to 2.5."""
import numpy as np
import pytest

import workloads as wl
from gpu_common import gpu_geometry

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def cgls(F, lam, d, iters, rnd):
    m, r = torch.zeros_like(F[0]), d.clone()
    s = F.T @ r
    p, gam = rnd(s), float(s @ s)
    for _ in range(iters):
        q = F @ p
        a = gam / (float(q @ q) + lam * float(p @ p))
        m, r = rnd(m + a * p), rnd(r - a * q)
        s = F.T @ r - lam * m
        gam, old = float(s @ s), gam
        p = rnd(s + (gam / old) * p)
    return m


def test_solution_is_limited_by_the_states_fp32():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = wl.slices32()
    geo, _ = gpu_geometry(w)
    F = torch.zeros((geo.M, geo.V), device="cuda", dtype=torch.float64)
    e = torch.zeros(geo.V, device="cuda")
    for v in range(geo.V):
        e[v] = 1.0
        F[:, v] = geo.J(e)
        e[v] = 0.0
    lam = w.lambda_rel * float(sum((b * b).sum() for b in F.split(512))) / geo.V
    m_true = torch.as_tensor(wl.model_for(w), device="cuda", dtype=torch.float64)
    clean = F @ m_true
    here, least = [], []
    for seed in range(24):
        d = (clean + torch.as_tensor(wl.noise(geo.M, 100 + seed), device="cuda")).float()
        exact = cgls(F, lam, d.double(), w.cg_iters, lambda x: x)
        far = lambda m: float((m.double() - exact).norm() / exact.norm())   # noqa: E731
        here.append(far(geo.cg_solve(d, w.lambda_rel, w.cg_iters)))
        least.append(far(cgls(F, lam, d.double(), w.cg_iters, lambda x: x.float().double())))
    ratio = float(np.exp(np.mean(np.log(here)) - np.mean(np.log(least))))
    print("distance to FP64: here %.2e (max %.2e), FP32 state alone %.2e (max %.2e), ratio %.2f" % (
        np.exp(np.mean(np.log(here))), max(here), np.exp(np.mean(np.log(least))), max(least), ratio))
    assert ratio <= 1.6
