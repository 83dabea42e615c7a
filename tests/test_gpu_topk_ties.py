"""The output cap on long lists and ties: the kept keypoints of a capped extraction
against a stable sort of the uncapped one's responses."""
import numpy as np
import pytest

from workloads import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2605_17869_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("cap", [1, 2, 31, 33, 500, 1023, 2049])
@pytest.mark.parametrize("fp16", (0, 1))
def test_cap_keeps_the_largest_in_canonical_order(cap, fp16):
    # A pattern repeated 6 x 6 times: most responses occur many times over, bit for bit.
    tile = synth.make_image(synth.rng_for(82, 0), 128, 128, n_blobs=30, n_rects=4, n_gratings=0, fractal_std=0.1)
    imgs = [torch.from_numpy(np.tile(tile, (6, 6))).cuda(),
            torch.from_numpy(synth.make_image(synth.rng_for(82, 1), 300, 400, n_blobs=60, fractal_std=0.1)).cuda()]
    full = pkg.Extractor(max_kpts=65536, fp16_pyramid=fp16).extract_batch(imgs)
    assert full[0].count > 2049  # the largest cap cuts the list
    r = full[0].response.cpu().numpy()
    assert len(np.unique(r)) < 0.6 * len(r)
    got = pkg.Extractor(max_kpts=cap, fp16_pyramid=fp16).extract_batch(imgs)
    for f, g in zip(full, got):
        keep = np.sort(np.argsort(-f.response.cpu().numpy(), kind="stable")[:cap])
        assert g.count == len(keep)
        for k in ("x", "y", "sigma", "angle", "response", "octave", "layer", "desc"):
            assert np.array_equal(getattr(g, k).cpu().numpy(), getattr(f, k).cpu().numpy()[keep]), k
