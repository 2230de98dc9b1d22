"""Pairs just outside r_c do not count against the 128 pairs an atom may have:
a compressed bcc crystal with 112 neighbours inside r_c and the next shell, 24
more, 5e-5 A beyond it runs in both precisions and gives the oracle's energy
and forces (1e-10, mixed 1e-6 and 5e-5 as in the parity tests)."""
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


@pytest.mark.parametrize("cells", [6, 9, 17])  # 32, 32 and 16 lanes an atom
def test_a_shell_just_beyond_the_cutoff(cells):
    par = W.EAM_FE_LIKE
    # ninth shell of bcc: (a/2) sqrt(24) from each atom; 112 atoms are nearer
    a = (par["r_c"] + 5e-5) / (0.5 * np.sqrt(24.0))
    x, box = O.create_crystal(O.BCC, a, cells, cells, cells)
    x = W.displaced(x, 5e-6, 1)
    p = O.eam(**par)
    Eo, fo, rho_o = O.eam_energy_forces(p, O.eam_theta(p), x, box)
    ctx = ne.ne_ctx_create(ne.eam_params(**par), len(x), 1)
    try:
        f, e, rho = T(np.zeros_like(x)), T([0.0]), T(np.zeros(len(x)))
        ne.ne_eam_energy_forces(ctx, ne.NE_FP64, T(x), box, f=f, e=e, rho=rho)
        assert float(e) == pytest.approx(Eo, rel=1e-10)
        assert np.abs(rho.cpu().numpy() - rho_o).max() < 1e-11 * rho_o.max()
        # the forces of a near-perfect crystal are small differences: against the
        # largest pair force, not their own norm
        assert np.abs(f.cpu().numpy() - fo).max() < 1e-10 * np.abs(Eo) / len(x)
        ne.ne_eam_energy_forces(ctx, ne.NE_MIXED, T(x), box, f=f, e=e)
        assert float(e) == pytest.approx(Eo, rel=1e-6)
    finally:
        ne.ne_ctx_destroy(ctx)
