"""The matcher at the edges of its work division: 128-row halves, 256-row tiles
and blocks, runs of several tiles, the last one cut anywhere; NaN descriptors."""
import numpy as np
import pytest

from oracle import matcher as om

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2605_17869_gb300 as pkg  # noqa: E402
from test_gpu_match import _planted  # noqa: E402


@pytest.mark.parametrize("na,nb", [(2, 2), (127, 33), (129, 255), (256, 257), (257, 31), (385, 1025),
                                   (40, 6000), (6000, 300), (8192, 4609)])
def test_match_edges(na, nb):
    a, b = _planted(na * 3 + nb, na, nb, min(na, nb) // 2)
    ex = pkg.Extractor()
    got = ex.match(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()).cpu().numpy()
    want, info = om.match(a, b, 0.8)
    assert np.array_equal(got[info["robust"]], want[info["robust"]])
    ex.close()


def test_nan_descriptors_never_match():
    """A NaN similarity is never larger than another: the sets match as if the
    NaN descriptors were not there."""
    a, b = _planted(11, 300, 520, 200)
    ia, ib = np.array([0, 5, 128, 299]), np.array([3, 255, 256, 519])
    ka, kb = np.setdiff1d(np.arange(300), ia), np.setdiff1d(np.arange(520), ib)
    an, bn = a.copy(), b.copy()
    an[ia], bn[ib, 7] = np.nan, np.nan
    ex = pkg.Extractor()
    got = ex.match(torch.from_numpy(an).cuda(), torch.from_numpy(bn).cuda()).cpu().numpy()
    ref = ex.match(torch.from_numpy(a[ka].copy()).cuda(), torch.from_numpy(b[kb].copy()).cuda()).cpu().numpy()
    assert (got[ia] == -1).all()
    assert np.array_equal(got[ka], np.where(ref >= 0, kb[ref], -1))
    ex.close()
