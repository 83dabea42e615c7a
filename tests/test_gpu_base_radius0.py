"""A base blur of radius 0: the input already has at least the blur of level 0, so
level 0 is the input itself, or its 2x bilinear magnification."""
import numpy as np
import pytest

from oracle import compare
from oracle import sift_oracle as so
from workloads import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2605_17869_gb300 as pkg  # noqa: E402

# (upsample, init_blur) with init_blur >= sigma0 = 1.6, or >= sigma0 / 2 where the input is magnified.
MODES = [(0, 1.6), (0, 2.5), (1, 0.8), (1, 1.0)]


@pytest.mark.parametrize("up,init", MODES)
@pytest.mark.parametrize("h,w", [(16, 17), (33, 129), (64, 200), (97, 131)])
def test_level_0_is_the_input(up, init, h, w):
    kw = dict(upsample=up, init_blur=init)
    img = synth.make_image(synth.rng_for(82, h), h, w, n_blobs=10, n_rects=3, n_gratings=1, fractal_std=0.05)
    ex = pkg.Extractor(**kw)
    got = ex.pyramid(torch.from_numpy(img).cuda())
    ref = so.build_pyramid(img, so.Params(**kw))
    base = got[0][0].cpu().numpy().astype(np.float64)
    if up:  # means of two and of four FP32 values in [0, 1]: two roundings of half an ulp of 1 at most
        assert np.abs(base - ref[0][0]).max() <= 2.0 ** -24
    else:
        assert np.array_equal(base, img.astype(np.float64))
    # The levels above, as in the test of every radius: 2R + 3 roundings in each of two passes per level.
    tol = sum(2 * (2 * r + 3) for r in (5, 7, 8, 10, 13)) * 2.0 ** -25
    assert len(got) == len(ref)
    for o, (g, r) in enumerate(zip(got, ref)):
        assert np.abs(g.cpu().numpy().astype(np.float64) - r).max() <= tol * (o + 1), o
    ex.close()


@pytest.mark.parametrize("up,init", MODES[::2])
def test_keypoints_match_the_oracle(up, init):
    kw = dict(upsample=up, init_blur=init, max_kpts=4096)
    img = synth.make_image(synth.rng_for(82, 1), 120, 161)
    ex = pkg.Extractor(**kw)
    f = ex.extract(torch.from_numpy(img).cuda())
    ref = so.extract(img, so.Params(**kw))
    m = compare.match(ref, f.as_numpy())
    assert f.count > 0 and len(ref) > 0
    assert m.found_frac >= 0.99 and m.desc_max_l2 <= compare.DESC_TOL, m
    ex.close()
