"""How many CTAs the brick runner takes: as many as its atoms need, so that
launches of other contexts fit beside it, and more only at one thread per atom,
where it leaves 24 SMs free.  The spread over an uneven batch against the
multi-kernel path (the tolerances of the other brick tests)."""
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
SMS = torch.cuda.get_device_properties(0).multi_processor_count


def T(a):
    return torch.tensor(np.asarray(a), dtype=torch.float64, device="cuda")


def run(sizes, steps, general=False):
    x0s, boxes = zip(*(O.create_crystal(O.BCC, W.A_BCC, *c) for c in sizes))
    off = np.concatenate([[0], np.cumsum([len(q) for q in x0s])]).astype(int)
    ctx = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), int(off[-1]), len(sizes))
    mds = [ne.md_params(T=300.0, mass=MASS, k_spring=2.4, skin=1.0, prec=ne.NE_MIXED, t_eq=2, t_s=4, seed=r + 1,
                        replica=r, fix_cm=1) for r in range(len(sizes))]
    try:
        X0 = T(np.concatenate(x0s))
        x, v, Wd = X0.clone(), torch.zeros_like(X0), torch.zeros((len(sizes), 2), dtype=torch.float64, device="cuda")
        if general:
            ne.ne_switch_run_segment(ctx, mds, list(off), x, v, X0, list(boxes), Wd, 0, steps)
            return x, v, Wd
        ne.ne_ctx_set_runner(ctx, 2)
        ne.ne_crystal_run_segment(ctx, mds, [(O.BCC, W.A_BCC) + tuple(c) for c in sizes], x, v, Wd, 0, steps)
        return x, v, Wd, ne.ne_ctx_crystal_plan(ctx)
    finally:
        ne.ne_ctx_destroy(ctx)


@pytest.mark.skipif(SMS < 144, reason="plans of a device of at least 144 SMs")
@pytest.mark.parametrize("cells,tpa,ctas", [((8, 8, 8), 8, 11), ((13, 13, 13), 8, 46), ((16, 16, 16), 8, 86),
                                            ((20, 20, 20), 4, 84)])
def test_a_small_batch_takes_the_ctas_its_atoms_need(cells, tpa, ctas):
    """ceil(atoms / (768 / threads per atom)) CTAs."""
    plan = run([cells], 2)[3]
    assert (plan["threads_per_atom"], plan["ctas"]) == (tpa, ctas)


@pytest.mark.parametrize("sizes", [[(32, 32, 32)], [(24, 24, 24), (26, 26, 26)], [(30, 30, 31), (9, 9, 9), (12, 11, 10)]])
def test_the_spread_of_a_large_batch(sizes):
    x, v, Wd, plan = run(sizes, 12)
    if SMS == 152:
        assert plan["threads_per_atom"] == 1 and plan["ctas"] <= SMS - 24
        assert plan["ctas"] > sum(-(-2 * a * b * c // 768) for a, b, c in sizes)
    xg, vg, Wg = run(sizes, 12, general=True)
    assert torch.abs(x - xg).max().item() < 2e-5
    assert torch.allclose(Wd, Wg, rtol=1e-5, atol=1e-2)
