"""The extrema scan at the edges of its strips: 60 columns in two words of 30, strips
of 30, 15, 6 and 3 rows, borders of 1 to 7 pixels, every number of layers."""
import numpy as np
import pytest

from workloads import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2605_17869_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("S,border", [(2, 1), (3, 5), (3, 7), (4, 2), (5, 1), (6, 3)])
@pytest.mark.parametrize("fp16", (0, 1))
def test_candidate_count_from_the_exported_pyramid(S, border, fp16):
    """The candidates are exact comparisons of the FP32 pyramid: their number per image equals
    that of the plain definition on the pyramid as exported, with no tolerance."""
    sig0 = 1.2 if S == 2 else 1.6
    ex = pkg.Extractor(n_scales=S, border=border, sigma0=sig0, fp16_pyramid=fp16, contrast_thr=0.004)
    gate = np.float32(0.5 * np.float32(0.004))
    sizes = [(41, 61), (31, 59), (60, 60), (97, 119), (64, 121), (16, 33), (700, 900)]
    imgs = [torch.from_numpy(synth.make_image(synth.rng_for(81, i), h, w, n_blobs=12, n_rects=4,
                                              n_gratings=1, fractal_std=0.08)).cuda()
            for i, (h, w) in enumerate(sizes)]
    want = []
    for im in imgs:
        n = 0
        for G in ex.pyramid(im):
            D = (G[1:] - G[:-1]).cpu().numpy()
            _, H, W = D.shape
            b = border
            if H <= 2 * b or W <= 2 * b:
                continue
            c = D[1:S + 1, b:H - b, b:W - b]
            near = np.stack([D[1 + k:S + 1 + k, b + j:H - b + j, b + i:W - b + i] for k in (-1, 0, 1)
                             for j in (-1, 0, 1) for i in (-1, 0, 1) if (k, j, i) != (0, 0, 0)])
            n += int(((np.abs(c) > gate) & ((c > near.max(0)) | (c < near.min(0)))).sum())
        want.append(n)
    assert sum(want) > 100
    for batch in (imgs, imgs[:1], imgs[5:]):
        ex.extract_batch(batch)
        got = [s[0] for s in ex.stats(len(batch))[1]]
        assert got == [want[next(i for i, x in enumerate(imgs) if x is im)] for im in batch]
    ex.close()
