"""The mixed parameter gradient's fixed-point bins against what they must not
depend on or cut off: the unit of the density, densities below zero, and the
small weights of F's knots."""
import numpy as np
import pytest

import oracle as O
from paper_2201_04622_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2201_04622_gb300 import ne  # noqa: E402


def T(a):
    return torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")


def crystal():
    x0, box = O.create_crystal(O.BCC, W.A_BCC, 6, 6, 6)
    return T(W.displaced(x0, 0.1, 5)), box


def gradient(prec, par, theta, x, box, with_rho=False):
    ctx = ne.ne_ctx_create(ne.eam_params(**par), len(x), 1)
    try:
        ne.ne_ctx_set_theta(ctx, T(theta))
        g = torch.zeros((3, par["n_knots"], 2), dtype=torch.float64, device="cuda")
        ne.ne_eam_backward(ctx, prec, x, box, 1.0, None, g)
        rho = T(np.zeros(len(x)))
        if with_rho:
            ne.ne_eam_energy_forces(ctx, prec, x, box, rho=rho)
        return g.cpu().numpy(), rho.cpu().numpy()
    finally:
        ne.ne_ctx_destroy(ctx)


@pytest.mark.parametrize("log2c", [13, 30, -13, -34])
def test_gradient_does_not_depend_on_the_unit_of_the_density(log2c):
    """f -> c f and F(rho) -> F(rho / c) leave every energy as it is.  With c a
    power of two every rounding of the forward pass is the same, so dU/df is
    1 / c times the plain one and dU/dphi and dU/dF (by its values) the same,
    all bit for bit."""
    par = W.EAM_FE_LIKE
    x, box = crystal()
    th = np.array(O.eam_theta(O.eam(**par))).reshape(3, -1, 2)
    g, _ = gradient(ne.NE_MIXED, par, th, x, box)
    c = 2.0 ** log2c
    ths = th.copy()
    ths[1] *= c
    ths[2, :, 1] /= c
    gs, _ = gradient(ne.NE_MIXED, dict(par, rho_max=par["rho_max"] * c), ths, x, box)
    assert np.array_equal(gs[0], g[0])
    assert np.array_equal(gs[1] * c, g[1])
    assert np.array_equal(gs[2, :, 0], g[2, :, 0]) and np.array_equal(gs[2, :, 1] / c, g[2, :, 1])


def test_a_few_atoms_of_large_slope_leave_the_others_precise():
    """An atom next to nothing has F' a thousand times its fellows': its own
    weights are kept, and so are theirs (3e-3 as for the other mixed gradients,
    over all of f's knots and over those that no pair of such an atom touches)."""
    par = W.EAM_FE_LIKE
    x0, box = O.create_crystal(O.BCC, W.A_BCC, 6, 6, 6)
    x = T(W.displaced(x0, 0.1, 5))
    th = np.array(O.eam_theta(O.eam(**par))).reshape(3, -1, 2)
    _, rho = gradient(ne.NE_MIXED, par, th, x, box, with_rho=True)
    # F with slope -1000 below the second lowest density, -1e-3 above
    nk, h = par["n_knots"], par["rho_max"] / (par["n_knots"] - 1)
    r = np.arange(nk) * h
    cut = 0.5 * (np.sort(rho)[1] + np.sort(rho)[2])
    th[2, :, 1] = np.where(r < cut, -1e3, -1e-3)
    th[2, 1:, 0] = np.cumsum(0.5 * (th[2, 1:, 1] + th[2, :-1, 1]) * h)
    gm, _ = gradient(ne.NE_MIXED, par, th, x, box)
    gd, _ = gradient(ne.NE_FP64, par, th, x, box)
    assert np.linalg.norm(gm[1] - gd[1]) < 3e-3 * np.linalg.norm(gd[1])
    pi, pj = O.pairs_brute(x.cpu().numpy(), box, par["r_c"])
    hot = (rho < cut)[pi] | (rho < cut)[pj]
    d = (x[pj] - x[pi]).cpu().numpy()[hot]
    d -= np.asarray(box) * np.round(d / np.asarray(box))
    k = (np.linalg.norm(d, axis=1) * ((nk - 1) / par["r_c"])).astype(int)
    small = np.ones(nk, bool)
    for q in (-1, 0, 1, 2):
        small[np.clip(k + q, 0, nk - 1)] = False
    assert hot.any() and np.abs(gd[1][small]).max() > 0
    assert np.linalg.norm(gm[1][small] - gd[1][small]) < 3e-3 * np.linalg.norm(gd[1][small])


@pytest.mark.parametrize("nk", [5000, 8000, 12000])
def test_gradient_with_densities_below_zero(nk):
    """A negative density takes F's first interval's cubic at u < 0, whose
    weights grow like 2 |u|^3: none may be cut off."""
    par = dict(W.EAM_FE_LIKE, n_knots=nk)
    x, box = crystal()
    th = np.array(O.eam_theta(O.eam(**par))).reshape(3, -1, 2)
    h = par["rho_max"] / (nk - 1)
    # densities of about -20 h; F quadratic
    _, rho = gradient(ne.NE_MIXED, par, th, x, box, with_rho=True)
    th[1] *= -20.0 * h / rho.mean()
    r = np.arange(nk) * h
    th[2, :, 0] = 0.3 * r + 0.05 * r * r
    th[2, :, 1] = 0.3 + 0.1 * r
    gm, rm = gradient(ne.NE_MIXED, par, th, x, box, with_rho=True)
    gd, _ = gradient(ne.NE_FP64, par, th, x, box)
    assert rm.max() < -3 * h
    for w in range(3):
        assert np.linalg.norm(gm[w] - gd[w]) < 3e-3 * np.linalg.norm(gd[w])


@pytest.mark.parametrize("nk", [5000, 8000, 12000])
def test_small_weights_of_the_embedding_knots(nk):
    """dU/dF against the basis weights at the kernel's own densities, knot by
    knot: FP32 weights (three roundings, 2e-7 relative of the largest term) in
    units of 2^-32 (2^-33 an add)."""
    par = dict(W.EAM_FE_LIKE, n_knots=nk)
    x, box = crystal()
    th = np.array(O.eam_theta(O.eam(**par))).reshape(3, -1, 2)
    g, rho = gradient(ne.NE_MIXED, par, th, x, box, with_rho=True)
    h = par["rho_max"] / (nk - 1)
    t = rho * ((nk - 1) / par["rho_max"])
    k = np.clip(t.astype(int), 0, nk - 2)
    u = t - k
    want, adds, scale = np.zeros((nk, 2)), np.zeros((nk, 2)), np.zeros((nk, 2))
    for c, d, w, s in ((0, 0, 2 * u**3 - 3 * u**2 + 1, 6.0), (0, 1, u**3 - 2 * u**2 + u, 4 * u),
                       (1, 0, -2 * u**3 + 3 * u**2, 5 * u * u), (1, 1, u**3 - u**2, 2 * u * u)):
        np.add.at(want, (k + c, d), w * (h if d else 1.0))
        np.add.at(adds, (k + c, d), 1.0 * (h if d else 1.0))
        np.add.at(scale, (k + c, d), s * (h if d else 1.0))
    assert np.all(np.abs(g[2] - want) <= 2.0**-33 * adds + 2e-7 * scale)
