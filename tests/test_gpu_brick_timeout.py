"""A wait of the brick runner that gives up (its limit set to a few polls) gives
NE_ETIMEOUT and leaves every replica as it was, whatever the others had reached;
the same context then runs the batch as if nothing had been.

One poll runs out at the first barrier; higher limits run out somewhere in the
run, or in none of its waits.  Replicas of unlike sizes end at unlike times."""
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
SIZES = [(5, 5, 5), (12, 12, 12), (6, 5, 7), (9, 8, 8)]


def T(a):
    return torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("npt", [0, 1])
def test_a_wait_that_gives_up_changes_nothing(npt):
    sizes = SIZES
    x0s, _ = zip(*(O.create_crystal(O.BCC, W.A_BCC, *c) for c in sizes))
    n, R, steps = sum(len(q) for q in x0s), len(sizes), 40
    ctx = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), n, R)
    ne.ne_ctx_set_runner(ctx, 2)
    kw = dict(path=O.PATH_RS, lambda_f=0.5, npt=1, P0=0.0, beta_T=1.2, tau_p=0.05) if npt else {}
    mds = [ne.md_params(T=300.0, mass=MASS, k_spring=2.4, skin=1.0, prec=ne.NE_MIXED, t_eq=8, t_s=12, seed=r + 1,
                        replica=r, fix_cm=1, **kw) for r in range(R)]
    cr = [(O.BCC, W.A_BCC) + c for c in sizes]
    X0 = T(np.concatenate(x0s))
    g = torch.Generator(device="cuda").manual_seed(1)
    V0 = 0.5 * torch.randn(X0.shape, dtype=torch.float64, device="cuda", generator=g)
    W0 = T(np.arange(2.0 * R).reshape(R, 2))

    def go(limit):
        ne.ne_ctx_set_wait_limit(ctx, limit)
        x, v, Wd = X0.clone(), V0.clone(), W0.clone()
        try:
            ne.ne_crystal_run_segment(ctx, mds, cr, x, v, Wd, 0, steps)
            late = False
        except ne.NeError as e:
            assert "NE_ETIMEOUT" in str(e)
            late = True
        return late, x, v, Wd, list(ne.ne_ctx_replica_status(ctx, R))

    try:
        late, xr, vr, Wr, st = go(0)
        assert not late and st == [ne.NE_OK] * R and not torch.equal(xr, X0)
        assert go(1)[0]
        for limit in [1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64] * 4 + [0]:
            late, x, v, Wd, st = go(limit)
            want = (X0, V0, W0) if late else (xr, vr, Wr)
            assert st == [ne.NE_ETIMEOUT if late else ne.NE_OK] * R
            assert torch.equal(x, want[0]) and torch.equal(v, want[1]) and torch.equal(Wd, want[2])
        assert not late
    finally:
        ne.ne_ctx_destroy(ctx)
