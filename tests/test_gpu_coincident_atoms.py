"""Two atoms at one place, or closer than 0.2 A: NE_ERANGE from every form of the
evaluation and in a run, not the NE_ENAN of a position that is not finite."""
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


@pytest.mark.parametrize("prec", [ne.NE_FP64, ne.NE_MIXED])
@pytest.mark.parametrize("apart", [0.0, 1e-30, 1e-9, 0.1])
@pytest.mark.parametrize("cells", [4, 7])
def test_coincident_atoms_are_out_of_range(prec, apart, cells):
    x, box = O.create_crystal(O.BCC, W.A_BCC, cells, cells, cells)
    x[9] = x[8] + [apart, 0.0, 0.0]
    ctx = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), len(x), 1)
    par = ne.eam_params(**W.EAM_FE_LIKE)
    try:
        e, g = T([0.0]), T(np.zeros((3, W.EAM_FE_LIKE["n_knots"], 2)))
        with pytest.raises(ne.NeError, match="NE_ERANGE"):
            ne.ne_eam_energy_forces(ctx, prec, T(x), box, e=e)
        with pytest.raises(ne.NeError, match="NE_ERANGE"):
            ne.ne_eam_energy_forces_noalloc(par, prec, T(x), box, e=e)
        with pytest.raises(ne.NeError, match="NE_ERANGE"):
            ne.ne_eam_backward(ctx, prec, T(x), box, 1.0, None, g)
        md = ne.md_params(T=10.0, mass=MASS, k_spring=5.0, skin=0.4, prec=prec, t_eq=1, t_s=1, seed=3, replica=0, fix_cm=1)
        Wd = torch.zeros((1, 2), dtype=torch.float64, device="cuda")
        y = x.copy()
        y[10] = [np.nan, 0.0, 0.0]
        with pytest.raises(ne.NeError, match="NE_ENAN"):
            ne.ne_eam_energy_forces(ctx, prec, T(y), box, e=e)
        if apart > 1e-3:  # (forces of nearer atoms leave the range of a step)
            with pytest.raises(ne.NeError, match="NE_ERANGE"):
                ne.ne_switch_run_segment(ctx, [md], [0, len(x)], T(x), T(np.zeros_like(x)), T(x), [box], Wd, 0, 1)
    finally:
        ne.ne_ctx_destroy(ctx)
