"""The level blur at every radius and at the sizes where its tiles end: 128
columns x 20 or 40 rows, steps of 8 outputs per lane, the reflected border."""
import math

import numpy as np
import pytest

from oracle import sift_oracle as so
from workloads import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2605_17869_gb300 as pkg  # noqa: E402

# (n_scales, sigma0, init_blur, min_octave_side) -> radii of the level blurs (base blur in front).
SETS = {
    (6, 0.3, 0.0, 16): (2, 1, 1, 1, 1, 1, 2, 2, 2),
    (6, 0.8, 0.5, 16): (3, 2, 2, 3, 3, 3, 3, 4, 4),
    (4, 1.6, 0.5, 16): (7, 5, 5, 6, 7, 9, 10),
    (2, 1.3, 0.5, 16): (5, 6, 8, 11, 15),
    (3, 1.8, 0.5, 16): (7, 6, 7, 9, 12, 14),
    (3, 2.0, 0.5, 24): (8, 7, 8, 10, 13, 16),
}
SIZES = [(41, 129), (40, 128), (39, 257), (20, 131), (61, 25), (100, 391)]


def _radii(S, s0, init, _):
    sig = [s0 * 2 ** (i / S) for i in range(S + 3)]
    steps = [math.sqrt(s0 ** 2 - init ** 2)] + [math.sqrt(b * b - a * a) for a, b in zip(sig, sig[1:])]
    return tuple(math.ceil(4 * k) for k in steps)


@pytest.mark.parametrize("rows", (32, 64))
@pytest.mark.parametrize("cfg", list(SETS))
def test_pyramid_every_radius(cfg, rows):
    S, s0, init, side = cfg
    assert _radii(*cfg) == SETS[cfg]
    kw = dict(n_scales=S, sigma0=s0, init_blur=init, min_octave_side=side)
    ex = pkg.Extractor(**kw)
    ex.set_tuning('{"blur_tile_rows": [%s]}' % ", ".join([str([rows] * (S + 2))] * 2))
    # A level is two sums of 2R + 1 products of values in [0, 1]: at most (2R + 3) roundings of half
    # an ulp of 1 each, carried through every level before it.
    tol = sum(2 * (2 * r + 3) for r in SETS[cfg]) * 2.0 ** -25
    for i, (h, w) in enumerate(SIZES):
        if min(h, w) < side:
            continue
        img = synth.make_image(synth.rng_for(80, i), h, w, n_blobs=10, n_rects=3, n_gratings=1, fractal_std=0.05)
        got = ex.pyramid(torch.from_numpy(img).cuda())
        ref = so.build_pyramid(img, so.Params(**kw))
        assert len(got) == len(ref)
        for o, (g, r) in enumerate(zip(got, ref)):
            assert np.abs(g.cpu().numpy().astype(np.float64) - r).max() <= tol * (o + 1), (cfg, h, w, o)
    ex.close()
