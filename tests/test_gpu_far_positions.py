"""Unwrapped positions far from the origin: atoms shifted by whole box lengths (up
to 10^3 .. 10^9 A) give the densities, forces and energies that the oracle gives
for the same positions taken into the box in exact arithmetic.

The box holds exactly three cells of an edge a hair above r_c an axis, so an
atom binned a hundredth of an Angstrom off loses pairs along an axis.  The
tolerances are those of the list test (1e-12 relative in rho with its factor ten,
1e-10 in forces and energy)."""
from fractions import Fraction

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


def T(a):
    return torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")


def gas(edge, seed, far):
    """7^3 atoms on a disordered simple cubic grid, each shifted by whole boxes up to `far` A."""
    g = np.random.Generator(np.random.PCG64(seed))
    i = np.arange(7) + 0.5
    x = np.stack(np.meshgrid(i, i, i, indexing="ij"), -1).reshape(-1, 3) * (edge / 7)
    x += g.uniform(-0.4, 0.4, x.shape)
    return x + np.round(g.uniform(-far, far, x.shape) / edge) * edge


def in_box(x, edge):
    """x less whole boxes, exact but for the last rounding."""
    e = Fraction(edge)
    return np.array([float(Fraction(c) - (Fraction(c) // e) * e) for c in x.ravel()]).reshape(x.shape)


@pytest.mark.parametrize("far", [1e3, 1e6, 1e8, 1e9])
def test_far_positions_keep_every_pair(far):
    p = O.eam(**W.EAM_FE_LIKE)
    th = O.eam_theta(p)
    edge = 3 * (W.EAM_FE_LIKE["r_c"] + 1.1e-3)
    box = (edge, edge, edge)
    ctx = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), 343, 1)
    try:
        for seed in range(8):
            x = gas(edge, seed, far)
            Eo, fo, rho_o = O.eam_energy_forces(p, th, in_box(x, edge), box)
            f, e, rho = T(np.zeros_like(x)), T([0.0]), T(np.zeros(len(x)))
            ne.ne_eam_energy_forces(ctx, ne.NE_FP64, T(x), box, f=f, e=e, rho=rho)
            assert np.abs(rho.cpu().numpy() - rho_o).max() < 1e-11 * np.abs(rho_o).max()
            assert float(e) == pytest.approx(Eo, rel=1e-10)
            assert np.linalg.norm(f.cpu().numpy() - fo) < 1e-10 * np.linalg.norm(fo)
            ne.ne_eam_energy_forces(ctx, ne.NE_MIXED, T(x), box, f=f, e=e, rho=rho)
            assert float(e) == pytest.approx(Eo, rel=1e-6)
            assert np.linalg.norm(f.cpu().numpy() - fo) < 5e-5 * np.linalg.norm(fo)
    finally:
        ne.ne_ctx_destroy(ctx)


@pytest.mark.parametrize("prec", [ne.NE_FP64, ne.NE_MIXED])
def test_a_run_far_from_the_origin(prec):
    """A 24-step switch of a crystal whose atoms and sites lie up to 10^6 A off
    (a box edge of 20.5 A, exact in FP32, so that shifts by it are exact)
    follows the unshifted one: positions of 10^6 A are rounded to 6e-11 A at
    every step, which 24 steps of ~10 fs of motion amplify less than a
    hundredfold."""
    a, cells = 20.5 / 7, 7
    x0, _ = O.create_crystal(O.BCC, a, cells, cells, cells)
    x0 = np.round(x0 * 2.0**20) / 2.0**20
    box = (20.5, 20.5, 20.5)
    g = np.random.Generator(np.random.PCG64(2))
    shift = g.integers(-48000, 48000, x0.shape) * 20.5
    ctx = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), len(x0), 1)
    md = ne.md_params(T=300.0, mass=MASS, k_spring=5.0, skin=0.4, prec=prec, t_eq=4, t_s=8, seed=3, replica=0, fix_cm=1)
    try:
        v0 = T(np.zeros_like(x0))
        ne.ne_init_velocities(ctx, md, v0)
        out = []
        for sh in (0.0 * shift, shift):
            X0 = T(x0 + sh)
            x, v, Wd = X0.clone(), v0.clone(), torch.zeros((1, 2), dtype=torch.float64, device="cuda")
            ne.ne_switch_run_segment(ctx, [md], [0, len(x0)], x, v, X0, [box], Wd, 0, 24)
            out.append((x.cpu().numpy() - sh, Wd.cpu().numpy()))
        assert np.abs(out[1][0] - out[0][0]).max() < (24 * 6e-11 * 100 if prec == ne.NE_FP64 else 2e-6)
        assert np.allclose(out[1][1], out[0][1], rtol=1e-7, atol=1e-6 if prec == ne.NE_FP64 else 2e-4)
    finally:
        ne.ne_ctx_destroy(ctx)


@pytest.mark.parametrize("lat,cells", [(O.BCC, 4), (O.BCC, 7)])  # all pairs; cells
@pytest.mark.parametrize("prec", [ne.NE_FP64, ne.NE_MIXED])
@pytest.mark.parametrize("at", [2.0**100, 1e30, 3e38, 1e60])
def test_a_position_beyond_any_box_stays_inside_the_tables(lat, cells, prec, at):
    """One atom at a finite coordinate that FP32 cannot wrap: single-point calls
    and runs return (with an error or without: the coordinate has no meaning),
    and the context then gives the oracle's energy of the plain crystal."""
    x0, box = O.create_crystal(lat, W.A_BCC, cells, cells, cells)
    p = O.eam(**W.EAM_FE_LIKE)
    Eo, _, _ = O.eam_energy_forces(p, O.eam_theta(p), x0, box)
    ctx = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), len(x0), 1)
    md = ne.md_params(T=300.0, mass=MASS, k_spring=5.0, skin=0.4, prec=prec, t_eq=4, t_s=8, seed=3, replica=0, fix_cm=0)
    far = x0.copy()
    far[5] = (at, -at, at)
    try:
        e = T([0.0])
        for _ in range(2):
            try:
                ne.ne_eam_energy_forces(ctx, prec, T(far), box, e=e)
            except ne.NeError:
                pass
            for sites in (x0, far):
                try:
                    ne.ne_switch_run_segment(ctx, [md], [0, len(x0)], T(far), T(np.zeros_like(x0)), T(sites), [box],
                                             torch.zeros((1, 2), dtype=torch.float64, device="cuda"), 0, 12)
                except ne.NeError:
                    pass
            ne.ne_eam_energy_forces(ctx, prec, T(x0), box, e=e)
            assert float(e) == pytest.approx(Eo, rel=1e-10 if prec == ne.NE_FP64 else 1e-6)
    finally:
        ne.ne_ctx_destroy(ctx)
