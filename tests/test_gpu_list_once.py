"""A run's first step does not build the list of the sites a second time: with
65,536 atoms the list kernels of that step take as long as those of a step without
a build (~9 us between events; a build takes 60 to 90 more)."""
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


def test_the_first_step_lists_nothing():
    x0, box = O.create_crystal(O.BCC, W.A_BCC, 32, 32, 32)
    n = len(x0)
    ctx = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), n, 1)
    md = ne.md_params(T=100.0, mass=MASS, k_spring=5.0, skin=0.4, prec=ne.NE_MIXED, t_eq=4, t_s=8, seed=3, replica=0,
                      fix_cm=1)
    X0 = torch.tensor(x0, dtype=torch.float64, device="cuda")

    def list_ms(steps):
        """Time of the list kernels of a run's first `steps` steps, the least of seven runs."""
        best = np.inf
        for _ in range(7):
            x, v = X0.clone(), torch.zeros_like(X0)
            Wd = torch.zeros((1, 2), dtype=torch.float64, device="cuda")
            ms, _ = ne.ne_profile_segment(ctx, [md], [0, n], x, v, X0, [box], Wd, 0, steps)
            best = min(best, ms[0] * steps)
        return best

    try:
        one, two = list_ms(1), list_ms(2)
        assert two - one > 0.0
        assert one < 3.0 * (two - one)
    finally:
        ne.ne_ctx_destroy(ctx)
