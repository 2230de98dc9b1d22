"""The multi-kernel path where it changes its form: the lanes per atom of the
pair passes (32 up to 4096 atoms, 16 up to 16,384, 8 above) with the replica
totals in groups (above 4096 atoms), the replica table as a launch argument
(up to 24 replicas, six a launch) or copied, and the mixed parameter gradient
with the bins of all three functions in shared memory or F's in global memory
(above ~9,600 knots).

Tolerances are those of the parity tests for the same quantities: FP64 1e-10
(energy, forces) and 1e-12 (rho); mixed 1e-6 (energy, rho), 5e-5 (forces) and
1e-3 (gradient by knots); replicas of one batch do not see each other, so
their bits do not depend on the batch's size."""
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


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


@pytest.mark.parametrize("cell", [(16, 16, 8), (15, 12, 12), (16, 16, 32), (16, 16, 33)])
def test_pair_passes_at_the_edges_of_the_lane_rule(cell):
    x0, box = O.create_crystal(O.BCC, W.A_BCC, *cell)
    p = O.eam(**W.EAM_FE_LIKE)
    x = W.displaced(x0, 0.12, 5)
    Eo, fo, rho_o = O.eam_energy_forces(p, O.eam_theta(p), x, box)
    ctx = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), len(x), 1)
    try:
        f, e, rho = torch.zeros_like(T(x)), torch.zeros(1, dtype=torch.float64, device="cuda"), T(np.zeros(len(x)))
        for prec, te, tf, tr in ((ne.NE_FP64, 1e-10, 1e-10, 1e-12), (ne.NE_MIXED, 1e-6, 5e-5, 1e-6)):
            ne.ne_eam_energy_forces(ctx, prec, T(x), box, f=f, e=e, rho=rho)
            assert float(e) == pytest.approx(Eo, rel=te)
            assert rel(f.cpu().numpy(), fo) < tf
            assert rel(rho.cpu().numpy(), rho_o) < tr
    finally:
        ne.ne_ctx_destroy(ctx)


@pytest.mark.parametrize("prec", [ne.NE_FP64, ne.NE_MIXED])
def test_a_replica_does_not_depend_on_the_size_of_its_batch(prec):
    x0, box = O.create_crystal(O.BCC, W.A_BCC, 4, 4, 4)
    n, most = len(x0), 25
    ctx = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), most * n, most)
    mds = [ne.md_params(T=100.0 + 20 * r, mass=MASS, k_spring=5.0 + 0.1 * r, skin=0.4, prec=prec, t_eq=4, t_s=8, seed=r,
                        replica=r, fix_cm=1) for r in range(most)]
    v0 = []
    for m in mds:
        v = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
        ne.ne_init_velocities(ctx, m, v)
        v0.append(v)
    outs = []
    try:
        for R in (most, 24, 7, 6, 1):
            X0 = T(np.concatenate([x0] * R))
            x, v, Wd = X0.clone(), torch.cat(v0[:R]), torch.zeros((R, 2), dtype=torch.float64, device="cuda")
            ne.ne_switch_run_segment(ctx, mds[:R], [n * r for r in range(R + 1)], x, v, X0, [box] * R, Wd, 0, 24)
            outs.append((R, x, v, Wd))
    finally:
        ne.ne_ctx_destroy(ctx)
    _, xa, va, Wa = outs[0]
    assert float(Wa.abs().min()) > 0.0
    for R, x, v, Wd in outs[1:]:
        assert torch.equal(x, xa[:R * n]) and torch.equal(v, va[:R * n]) and torch.equal(Wd, Wa[:R])


@pytest.mark.parametrize("nk", [9600, 12000, 14000])
def test_mixed_gradient_with_many_knots(nk):
    par = dict(W.EAM_FE_LIKE, n_knots=nk)
    p = O.eam(**par)
    x0, box = O.create_crystal(O.BCC, W.A_BCC, 6, 6, 6)
    x = W.displaced(x0, 0.1, 5)
    go = O.eam_grad_theta(p, O.eam_theta(p), x, box)
    ctx = ne.ne_ctx_create(ne.eam_params(**par), len(x), 1)
    try:
        for gE in (2.0, -0.5):  # the second call starts from the bins that the first left
            g = torch.zeros((3, nk, 2), dtype=torch.float64, device="cuda")
            ne.ne_eam_backward(ctx, ne.NE_MIXED, T(x), box, gE, None, g)
            for w in range(3):
                assert rel(g[w].cpu().numpy(), gE * go[w]) < 3e-3
            assert rel(g.cpu().numpy(), gE * go) < 1e-3
    finally:
        ne.ne_ctx_destroy(ctx)
