"""The FP64 path's rounding: the density of isolated pairs, f(r) of each, against
the same spline in extended precision.  Its error is mostly that of r / h, of
which the interval, up to thousands, is taken off; the bound is the error of
sqrt(r^2) * (1 / h) with correctly rounded operations in plain NumPy, over the
same 20,000 pairs, summed over five numbers of knots (1 / h happens to be nearly
exact for some)."""
import numpy as np
import pytest

import oracle as O
from paper_2201_04622_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2201_04622_gb300 import ne  # noqa: E402


def errors(nk):
    par = dict(W.EAM_FE_LIKE, n_knots=nk)
    th = np.array(O.eam_theta(O.eam(**par))).reshape(3, -1, 2)
    g = np.random.Generator(np.random.PCG64(1))
    n = 20000
    d = g.normal(size=(n, 3))
    d *= (g.uniform(2.0, 5.2, n) / np.linalg.norm(d, axis=1))[:, None]
    d = np.round(d * 2**20) / 2**20  # differences of positions are exact
    side = 28
    site = 16.0 * np.stack(np.unravel_index(np.arange(n), (side,) * 3), -1) + 8.0
    x = np.stack([site, site + d], 1).reshape(-1, 3)
    box = (16.0 * side,) * 3

    def spline(t, k, dt):
        h = dt(par["r_c"] / (nk - 1))
        y, m = th[1, :, 0].astype(dt), th[1, :, 1].astype(dt) * h
        u = t - k.astype(dt)
        c2 = dt(3) * (y[k + 1] - y[k]) - dt(2) * m[k] - m[k + 1]
        c3 = dt(2) * (y[k] - y[k + 1]) + m[k] + m[k + 1]
        return ((c3 * u + c2) * u + m[k]) * u + y[k]

    ld = np.longdouble
    t = np.sqrt((d.astype(ld) ** 2).sum(1)) * (ld(nk - 1) / ld(par["r_c"]))
    want = spline(t, t.astype(int), ld)
    t = np.sqrt((d[:, 0] ** 2 + d[:, 1] ** 2) + d[:, 2] ** 2) * ((nk - 1) / par["r_c"])
    plain = spline(t, t.astype(int), np.float64)

    ctx = ne.ne_ctx_create(ne.eam_params(**par), 8 * len(x), 1)
    try:
        rho = torch.zeros(len(x), dtype=torch.float64, device="cuda")
        ne.ne_eam_energy_forces(ctx, ne.NE_FP64, torch.tensor(x, dtype=torch.float64, device="cuda"), box, rho=rho)
        got = rho.cpu().numpy().reshape(n, 2)
    finally:
        ne.ne_ctx_destroy(ctx)

    def rms(f):
        return float(np.sqrt((((f - want) / want).astype(np.float64) ** 2).mean()))

    return rms(got[:, 0]), rms(got[:, 1]), rms(plain)


def test_density_of_single_pairs():
    a, b, plain = np.sum([errors(nk) for nk in (5000, 1024, 337, 64, 9999)], axis=0)
    assert a <= plain and b <= plain
