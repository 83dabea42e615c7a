"""Descriptors with components beyond fp16's range: they become infinite as the tensor
core's operands, and similarities infinite or NaN. A NaN or minus-infinite similarity is
never larger than another, an infinite one is the nearest; worked out in 64 bits from the
operands rounded to fp16."""
import numpy as np
import pytest

from oracle import matcher as om

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2605_17869_gb300 as pkg  # noqa: E402
from test_gpu_match import _planted  # noqa: E402

RATIO = 0.8


def _best_two(S):
    S = np.where(np.isnan(S), -np.inf, S)
    j = np.argmax(S, axis=1)
    s1 = S.max(axis=1)
    T = S.copy()
    T[np.arange(len(S)), j] = -np.inf
    return np.where(s1 > -np.inf, j, -1), s1, T.max(axis=1)


def _distance(s):
    return np.sqrt(np.maximum(0.0, 2.0 - 2.0 * s))


@pytest.mark.parametrize("value", [7e4, -7e4, 1e30, np.inf, -np.inf])
@pytest.mark.parametrize("na,nb", [(300, 520), (40, 3000)])
def test_operands_beyond_fp16(value, na, nb):
    a, b = _planted(na + 5, na, nb, min(na, nb) * 2 // 3)
    a[3, 5] = value       # one component of a matched row
    a[na - 1] = value     # a whole row
    b[7, 100] = value
    b[nb - 1, :64] = value
    with np.errstate(all="ignore"):
        a16, b16 = (om.round_fp16(x) for x in (a, b))
        S = np.stack([(r * b16).sum(axis=1) for r in a16])
        ja, sa1, sa2 = _best_two(S)
        ib, sb1, sb2 = _best_two(S.T)
        da1, da2, db1, db2 = (_distance(s) for s in (sa1, sa2, sb1, sb2))
        ok_a, ok_b = da1 < RATIO * da2, db1 < RATIO * db2
        # Decisions that the FP32 sums (off by less than 1e-5) leave as they are; equal infinities are.
        sure = lambda s1, s2, d1, d2: ((s1 == s2) & np.isinf(s1)) | (  # noqa: E731
            (s1 - s2 > 2e-5) & (np.isinf(s1) | np.isinf(s2) | (np.abs(d1 - RATIO * d2) > 2e-3)))
        sa, sb = sure(sa1, sa2, da1, da2), sure(sb1, sb2, db1, db2)
    want = np.array([j if j >= 0 and ib[j] == i and ok_a[i] and ok_b[j] else -1 for i, j in enumerate(ja)])
    robust = np.array([j < 0 or (sa[i] and sb[j]) for i, j in enumerate(ja)])
    ex = pkg.Extractor()
    got = ex.match(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), RATIO).cpu().numpy()
    assert robust.mean() > 0.7 and robust[[3, na - 1]].all()
    assert np.array_equal(got[robust], want[robust])
    ex.close()
