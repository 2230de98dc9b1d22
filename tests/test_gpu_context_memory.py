"""A context's device memory: the lists of pairs of the two precisions share one
buffer, so an atom takes 1024 + 512 + 1024 B of lists and ~230 B besides."""
import pytest

from paper_2201_04622_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2201_04622_gb300 import ne  # noqa: E402


def test_bytes_an_atom():
    n = 4_000_000
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx = ne.ne_ctx_create(ne.eam_params(**W.EAM_FE_LIKE), n, 1)
    try:
        assert (before - torch.cuda.mem_get_info()[0]) / n < 2900.0
    finally:
        ne.ne_ctx_destroy(ctx)
