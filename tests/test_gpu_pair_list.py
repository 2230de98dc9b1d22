"""The neighbour-list build against the oracle at the sizes where it takes
another route: all pairs (fewer than three cells an axis), exactly three
cells, long thin boxes, the change of lanes per atom (8192 atoms) and of the
cell sort (16,384 atoms in one replica), ragged last tiles, with atoms moved by
whole box lengths.

A missed or doubled pair changes an atom's density by f(r) ~ 0.01 to 1 of ~10;
the FP64 path's sums otherwise agree with the oracle's to rounding (1e-12
relative in rho and 1e-10 in forces and energy, as in the parity tests).
"""
import numpy as np
import pytest

import oracle as O
from paper_2201_04622_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2201_04622_gb300 import ne  # noqa: E402

CELLS = [(O.BCC, 4, 4, 4), (O.BCC, 5, 6, 7), (O.FCC, 5, 5, 5), (O.BCC, 6, 9, 40), (O.BCC, 16, 16, 16),
         (O.BCC, 16, 16, 17), (O.BCC, 16, 16, 32), (O.BCC, 16, 16, 33), (O.FCC, 13, 19, 17)]


@pytest.mark.parametrize("cell", CELLS)
def test_list_finds_every_pair_once(cell):
    lat, nx, ny, nz = cell
    x0, box = O.create_crystal(lat, W.A_BCC if lat == O.BCC else W.A_FCC, nx, ny, nz)
    p = O.eam(**W.EAM_FE_LIKE)
    x = W.displaced(x0, 0.25, 7)
    g = np.random.Generator(np.random.PCG64(3))
    moved = x + g.integers(-2, 3, size=x.shape) * np.asarray(box)
    Eo, fo, rho_o = O.eam_energy_forces(p, O.eam_theta(p), moved, box)
    ctx = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), len(x), 1)
    try:
        xt = torch.tensor(moved, dtype=torch.float64, device="cuda")
        f, e = torch.zeros_like(xt), torch.zeros(1, dtype=torch.float64, device="cuda")
        rho = torch.zeros(len(x), dtype=torch.float64, device="cuda")
        for _ in range(2):  # the second build starts from what the first left
            ne.ne_eam_energy_forces(ctx, ne.NE_FP64, xt, box, f=f, e=e, rho=rho)
            assert float(e) == pytest.approx(Eo, rel=1e-10)
            assert np.abs(rho.cpu().numpy() - rho_o).max() < 1e-12 * np.abs(rho_o).max() * 10
            assert np.linalg.norm(f.cpu().numpy() - fo) < 1e-10 * np.linalg.norm(fo)
    finally:
        ne.ne_ctx_destroy(ctx)
