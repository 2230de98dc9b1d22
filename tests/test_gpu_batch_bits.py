"""A replica in batches on either side of a change of lanes per atom (25 and 40
replicas of 128 atoms: 3200 and 5120 atoms): the same bits with the threads per
atom fixed by ne_ctx_set_tuning, and to rounding without.  24 steps of a crystal
amplify the last bit (1e-16 of forces of ~1 eV/A, or 6e-8 of them in FP32) less than
a thousandfold."""
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


@pytest.mark.parametrize("prec,tol", [(ne.NE_FP64, 1e-11), (ne.NE_MIXED, 1e-5)])
@pytest.mark.parametrize("lanes", [0, 8])
def test_a_replica_in_batches_of_other_lanes(prec, tol, lanes):
    x0, box = O.create_crystal(O.BCC, W.A_BCC, 4, 4, 4)
    n, most = len(x0), 40
    ctx = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), most * n, most)
    if lanes:
        ne.ne_ctx_set_tuning(ctx, lanes)
    mds = [ne.md_params(T=300.0, mass=MASS, k_spring=5.0, skin=0.4, prec=prec, t_eq=4, t_s=8, seed=r, replica=r, fix_cm=1)
           for r in range(most)]
    try:
        v0 = []
        for m in mds:
            v = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
            ne.ne_init_velocities(ctx, m, v)
            v0.append(v)
        out = []
        for R in (most, 25):
            X0 = torch.tensor(np.concatenate([x0] * R), dtype=torch.float64, device="cuda")
            x, v, Wd = X0.clone(), torch.cat(v0[:R]), torch.zeros((R, 2), dtype=torch.float64, device="cuda")
            ne.ne_switch_run_segment(ctx, mds[:R], [n * r for r in range(R + 1)], x, v, X0, [box] * R, Wd, 0, 24)
            out.append((x[:25 * n], v[:25 * n], Wd[:25]))
    finally:
        ne.ne_ctx_destroy(ctx)
    if lanes:
        assert all(torch.equal(a, b) for a, b in zip(*out))
    else:
        assert torch.abs(out[0][0] - out[1][0]).max().item() < tol
        assert torch.allclose(out[0][2], out[1][2], rtol=tol, atol=100 * tol)
