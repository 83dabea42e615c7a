"""Descriptors next to pixels so large that gradient magnitudes overflow FP32. The bins
that such gradients vote for are infinite and take the clip value, all others vanish
beside them: the descriptor is 1 / sqrt(n) in its n hit bins. A gradient that is itself
NaN (infinity less infinity) makes the descriptor zero. The hit bins are worked out in
64 bits from the exported pyramid."""
import numpy as np
import pytest

from workloads import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2605_17869_gb300 as pkg  # noqa: E402

OVERFLOW = 2.0 ** 64  # a magnitude above it has a square beyond the largest FP32 value
EDGE = 1e-3           # samples nearer than this to a cell's or a bin's border leave it open which is hit


def _expected(level, x, y, sigma, angle):
    """The descriptor of a keypoint at (x, y) of its octave's level; None where no gradient
    overflows (an ordinary descriptor) or where a sample lies too near a border."""
    H, W = level.shape
    wbin = 3.0 * sigma
    R = int(np.floor(wbin * np.sqrt(2.0) * 2.5 + 0.5))
    px, py = int(np.rint(x)), int(np.rint(y))
    X, Y = np.meshgrid(np.arange(max(1, px - R), min(W - 2, px + R) + 1),
                       np.arange(max(1, py - R), min(H - 2, py + R) + 1))
    th = np.deg2rad(angle)
    ox, oy = X - x, Y - y
    u = (np.cos(th) * ox + np.sin(th) * oy) / wbin + 1.5
    v = (-np.sin(th) * ox + np.cos(th) * oy) / wbin + 1.5
    with np.errstate(all="ignore"):
        gx = (level[Y, X + 1] - level[Y, X - 1]).astype(np.float64)
        gy = (level[Y + 1, X] - level[Y - 1, X]).astype(np.float64)
        mag = np.hypot(gx, gy)
    inside = (u > -1) & (u < 4) & (v > -1) & (v < 4)
    large = ~(mag < OVERFLOW * (1 - EDGE))  # NaN as well
    near = (u > -1 - EDGE) & (u < 4 + EDGE) & (v > -1 - EDGE) & (v < 4 + EDGE)
    if not (near & large).any():
        return None
    nan = np.isnan(gx) | np.isnan(gy)
    ob = np.mod(np.arctan2(gy, gx) - th, 2 * np.pi) * 8 / (2 * np.pi)
    frac = np.stack([u, v, np.where(nan, 0.5, ob)])[:, near & large]
    odd = (np.abs(frac - np.rint(frac)) < EDGE).any() or (near != inside)[large].any()
    odd |= (np.maximum(np.abs(X - px), np.abs(Y - py)) >= R)[near & large].any()
    odd |= (mag[near & large] < OVERFLOW * (1 + EDGE)).any()
    if odd:
        return None
    if (inside & nan).any():
        return np.zeros(128)
    hit = np.zeros((4, 4, 8), bool)
    for a, b, o in zip(*(np.floor(q[inside & large]).astype(int) for q in (u, v, ob))):
        for da, db, do in np.ndindex(2, 2, 2):
            if 0 <= a + da < 4 and 0 <= b + db < 4:
                hit[b + db, a + da, (o + do) % 8] = True
    return hit.reshape(128) / np.sqrt(hit.sum())


@pytest.mark.parametrize("kw", [dict(), dict(upsample=1)])
@pytest.mark.parametrize("value", [1e25, 1e30, 3e38, np.inf])
def test_bins_hit_by_overflowing_gradients(kw, value):
    ex = pkg.Extractor(**kw)
    up = 0.5 if kw else 1.0
    checked = 0
    for seed in range(6):
        img = torch.from_numpy(synth.make_image(synth.rng_for(90, seed), 160, 200, n_blobs=12, n_rects=4,
                                                n_gratings=1, fractal_std=0.07)).cuda()
        rng = np.random.default_rng(seed)
        for _ in range(6):
            img[int(rng.integers(10, 150)), int(rng.integers(10, 190))] = value
        pyr = [o.cpu().numpy() for o in ex.pyramid(img)]
        f = ex.extract(img).as_numpy()
        for k in range(len(f["x"])):
            o = int(f["octave"][k])
            sc = up * 2.0 ** o
            want = _expected(pyr[o][f["layer"][k]], *(f[n][k].astype(np.float64) / sc for n in ("x", "y", "sigma")),
                             float(f["angle"][k]))
            if want is not None:
                checked += 1
                assert np.abs(f["desc"][k] - want).max() < 1e-6, (seed, k)
    assert checked >= 3
    ex.close()
