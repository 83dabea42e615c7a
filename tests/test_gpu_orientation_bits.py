"""Orientation angles bit for bit: the histogram bins come from a polynomial with an exact
fallback, and each vote is to be the one that atan2f gave, weight and bin. The golden
angles (tests/golden/orientation_angles.json: the bits of the first 400 keypoints'
angles) were written by the kernel that took every bin from atan2f; the image is exact in
FP32, so that it is the same on every host."""
import json
from pathlib import Path

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2605_17869_gb300 as pkg  # noqa: E402

GOLDEN = Path(__file__).parent / "golden" / "orientation_angles.json"


def image():
    """Random 6 x 6 blocks of k / 256, smoothed by 5 x 5 and 3 x 3 sums: integers over a power of two."""
    a = np.kron(np.random.default_rng(11).integers(0, 256, (60, 80)), np.ones((6, 6), np.int64))
    for n in (5, 3):
        for axis in (0, 1):
            a = sum(np.roll(a, k, axis) for k in range(n))
    return (a / 2.0 ** 16).astype(np.float32)  # at most 256 * 225 / 2^16


def angle_bits():
    ex = pkg.Extractor()
    f = ex.extract(torch.from_numpy(image()).cuda())
    bits = f.angle[:400].cpu().numpy().view(np.uint32).tolist()
    ex.close()
    return bits


def test_angles_are_those_of_atan2f_bins():
    want = json.loads(GOLDEN.read_text())["angle_bits"]
    got = angle_bits()
    assert len(got) == len(want) == 400
    assert [i for i in range(400) if got[i] != want[i]] == []
