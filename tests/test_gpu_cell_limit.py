"""Boxes whose cells are hardly wider than r_c + skin, where an atom binned a
millionth of an Angstrom off would be one cell away from a neighbour: a dense
disordered box of three such cells an axis, and a barostatted crystal contracted
to within 4e-4 A of its limit, one step before it is refused (NE_ERANGE)."""
import numpy as np
import pytest

import oracle as O
from paper_2201_04622_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2201_04622_gb300 import ne  # noqa: E402

MASS = W.MASS_FE_AMU / 9648.5332
R_C = W.EAM_FE_LIKE["r_c"]


def T(a):
    return torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("wider", [1e-9, 1e-6, 0.9e-3, 1.1e-3])
def test_cells_of_the_cutoff(wider):
    """Atoms within 1e-6 A of every cell face, with partners at r_c less 1e-5 to
    1e-2 A along the axis, shifted by boxes: the oracle's rho (1e-11 of the
    largest), in both forms of the call."""
    p = O.eam(**W.EAM_FE_LIKE)
    edge = R_C + wider
    L = 3 * edge
    g = np.random.Generator(np.random.PCG64(4))
    ctx = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), 512, 1)
    try:
        for _ in range(8):
            x = []
            for axis in range(3):
                for face in range(3):
                    for side in (-1, 1):
                        for q in range(8):
                            r0 = g.uniform(0, L, 3)
                            r0[axis] = face * edge + g.uniform(-1e-6, 1e-6)
                            r1 = r0.copy()
                            r1[axis] += side * (R_C - 10.0 ** g.uniform(-5, -2))
                            x += [r0, r1]
            x = np.array(x)
            # drop atoms closer than 1 A to an earlier one
            keep = []
            for i in range(len(x)):
                d = x[keep] - x[i]
                d -= L * np.round(d / L)
                if not len(keep) or (d * d).sum(1).min() > 1.0:
                    keep.append(i)
            x = x[keep]
            Eo, _, rho_o = O.eam_energy_forces(p, O.eam_theta(p), x, (L, L, L))
            far = x + np.array([L, L, L]) * g.integers(-3, 4, x.shape)
            rho, e = T(np.zeros(len(x))), T([0.0])
            ne.ne_eam_energy_forces(ctx, ne.NE_FP64, T(x), (L, L, L), e=e, rho=rho)
            assert np.abs(rho.cpu().numpy() - rho_o).max() < 1e-11 * rho_o.max()
            assert float(e) == pytest.approx(Eo, rel=1e-10)
            ne.ne_eam_energy_forces(ctx, ne.NE_FP64, T(far), (L, L, L), e=e)
            assert float(e) == pytest.approx(Eo, rel=1e-10)
            ne.ne_eam_energy_forces_noalloc(ne.eam_params(**W.EAM_FE_LIKE), ne.NE_FP64, T(x), (L, L, L), e=e)
            assert float(e) == pytest.approx(Eo, rel=1e-10)
    finally:
        ne.ne_ctx_destroy(ctx)


@pytest.mark.parametrize("prec", [ne.NE_FP64, ne.NE_MIXED])
def test_a_barostatted_box_at_its_limit(prec):
    """Three cells of r_c + skin = 5.7 A hold down to 17.1 A: after 36 steps at
    8 eV/A^3 the oracle's box is 17.10034 A, after 37 17.0551 A."""
    a, steps = 2.7156279063560085, 36
    kw = dict(path=O.PATH_RS, T=300.0, t_eq=40, t_s=40, lambda_f=0.5, npt=1, P0=8.0, beta_T=1.2, tau_p=1.0, damp=0.1,
              dt=1e-3, k_spring=1.0, lambda_fn=2, fix_cm=1, seed=11, replica=2)
    mo, mg = O.md(mass=MASS, **kw), ne.md_params(mass=MASS, skin=0.4, prec=prec, **kw)
    x0, box = O.create_crystal(O.BCC, a, 7, 7, 7)
    p = O.eam(**W.EAM_FE_LIKE)
    v0 = O.init_velocities(mo, len(x0))
    ro = O.switch_run_prefix(p, O.eam_theta(p), mo, x0, v0, x0, box, steps)
    assert 17.1 < ro["box"][0] < 17.1 + 3e-3
    ctx = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), len(x0), 1)
    try:
        x, v, Wd = T(x0), T(v0), torch.zeros((1, 2), dtype=torch.float64, device="cuda")
        ne.ne_switch_run_segment(ctx, [mg], [0, len(x0)], x, v, T(x0), [box], Wd, 0, steps)
        tol = 1e-9 if prec == ne.NE_FP64 else 2e-6
        assert np.allclose(ne.ne_ctx_boxes(ctx, 1)[0], ro["box"], rtol=tol, atol=0)
        assert np.abs(x.cpu().numpy() - ro["x"]).max() < (1e-7 if prec == ne.NE_FP64 else 2e-4)
        x, v = T(x0), T(v0)
        with pytest.raises(ne.NeError, match="NE_ERANGE"):
            ne.ne_switch_run_segment(ctx, [mg], [0, len(x0)], x, v, T(x0), [box], Wd, 0, steps + 1)
    finally:
        ne.ne_ctx_destroy(ctx)
