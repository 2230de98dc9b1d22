"""One context used in turn for batches of many replicas and for single-point
calls: the single-point calls' first kernel follows the one that writes the
replica and tile tables, so it must not see the batch's.  The outputs are those
of a context of their own, bit for bit (the sums' order is fixed; FP64 gradients
go through atomics, so only the mixed ones are compared)."""
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


def single_point(ctx, prec, x, box):
    f, e, rho = torch.zeros_like(x), T([0.0]), T(np.zeros(len(x)))
    ne.ne_eam_energy_forces(ctx, prec, x, box, f=f, e=e, rho=rho)
    out = [f, e, rho]
    if prec == ne.NE_FP64:
        w = T([0.0])
        ne.ne_eam_virial(ctx, x, box, w)
        out.append(w)
    if prec == ne.NE_MIXED:
        gx, gt = torch.zeros_like(x), T(np.zeros((3, W.EAM_FE_LIKE["n_knots"], 2)))
        ne.ne_eam_backward(ctx, prec, x, box, 1.0, gx, gt)
        out += [gx, gt]
    return out


@pytest.mark.parametrize("replicas", [2, 24])
def test_single_point_calls_between_batched_runs(replicas):
    small, sbox = O.create_crystal(O.BCC, W.A_BCC, 4, 4, 4)
    big, box = O.create_crystal(O.BCC, W.A_BCC, 12, 12, 12)
    x = T(W.displaced(big, 0.1, 3))
    n = len(small)
    mds = [ne.md_params(T=300.0, mass=MASS, k_spring=5.0, skin=0.4, prec=ne.NE_MIXED, t_eq=4, t_s=8, seed=r, replica=r,
                        fix_cm=1) for r in range(replicas)]
    size = max(len(big), replicas * n)
    fresh = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), size, replicas)
    ctx = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), size, replicas)
    try:
        X0 = T(np.concatenate([small] * replicas))
        for prec in (ne.NE_FP64, ne.NE_MIXED):
            want = single_point(fresh, prec, x, box)
            for _ in range(10):
                xr, v, Wd = X0.clone(), torch.zeros_like(X0), torch.zeros((replicas, 2), dtype=torch.float64, device="cuda")
                ne.ne_switch_run_segment(ctx, mds, [n * r for r in range(replicas + 1)], xr, v, X0, [sbox] * replicas, Wd,
                                         0, 3)
                got = single_point(ctx, prec, x, box)
                assert all(torch.equal(a, b) for a, b in zip(got, want))
    finally:
        ne.ne_ctx_destroy(ctx)
        ne.ne_ctx_destroy(fresh)
