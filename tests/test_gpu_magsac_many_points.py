"""GPU MAGSAC++ at the edges of its work division: hypotheses that fill the last
warp of the fit (four per warp) only in part, and correspondences on both sides
of the count from which several blocks mark the inliers (8,192 points, at least
two per hypothesis). Against the FP64 oracle, with the bounds derived in
test_gpu_magsac.py."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2605_17869_gb300 as pkg  # noqa: E402
from test_gpu_magsac import _check, _planted  # noqa: E402


@pytest.mark.parametrize("n,n_hyp", [(64, 1), (64, 3), (64, 5), (8191, 33), (8192, 33), (20011, 64)])
def test_magsac_partial_warps_and_many_points(n, n_hyp):
    n_out = n // 8
    _, xa, xb = _planted(n + n_hyp, n - n_out, n_out)
    _check(xa, xb, pkg.draw_samples(n, n_hyp, seed=n))
