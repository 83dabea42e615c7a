"""The extrema scan's longest strips (30 rows), which only images and batches with more
15-row strips than the GPU holds warps take, and warps that take several strips in turn:
exact candidate counts, as for the shorter strips, on one large image whose sides end
inside a strip."""
import pytest

from workloads import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2605_17869_gb300 as pkg  # noqa: E402

H, W = 2159, 3833
ROWS = (30, 15, 6, 3)


def _strip_rows(h, w, ctas):
    """The plan's rule for one image: per octave the shortest strips (60 columns) that the
    resident warps (4 per block) take all at once, else the longest."""
    warps = torch.cuda.get_device_properties(0).multi_processor_count * ctas * 4
    out = []
    while min(h, w) >= 16:
        strips = lambda rows: -(-(-(-w // 30)) // 2) * -(-h // rows)  # noqa: B023,E731
        out.append(next((r for r in reversed(ROWS[1:]) if all(strips(q) <= warps for q in ROWS[1:] if q >= r)), 30))
        h, w = h // 2, w // 2
    return out


def _count(G, S, border, gate):
    D = G[1:] - G[:-1]
    _, h, w = D.shape
    b = border
    if h <= 2 * b or w <= 2 * b:
        return 0
    c = D[1:S + 1, b:h - b, b:w - b]
    hi, lo = torch.full_like(c, -torch.inf), torch.full_like(c, torch.inf)
    for k in (-1, 0, 1):
        for j in (-1, 0, 1):
            for i in (-1, 0, 1):
                if (k, j, i) != (0, 0, 0):
                    v = D[1 + k:S + 1 + k, b + j:h - b + j, b + i:w - b + i]
                    hi, lo = torch.maximum(hi, v), torch.minimum(lo, v)
    return int(((c.abs() > gate) & ((c > hi) | (c < lo))).sum())


# Blocks per SM that the scan's launch bounds allow for.
@pytest.mark.parametrize("S,border,ctas", [(2, 1, 4), (3, 5, 4), (4, 2, 3), (6, 3, 2)])
@pytest.mark.parametrize("fp16", (0, 1))
def test_candidate_count_of_a_large_image(S, border, ctas, fp16):
    rows = _strip_rows(H, W, ctas)
    assert rows[0] == 30 and rows[-1] == 3
    if ctas == 4:
        assert set(rows) == set(ROWS)
    ex = pkg.Extractor(n_scales=S, border=border, sigma0=1.2 if S == 2 else 1.6, fp16_pyramid=fp16,
                       contrast_thr=0.004)
    img = torch.from_numpy(synth.make_image(synth.rng_for(85, S), 540, 959, n_blobs=60, n_rects=20,
                                            n_gratings=4, fractal_std=0.08)).cuda()
    img = img.repeat(4, 4)[:H, :W].contiguous()
    assert img.shape == (H, W)
    gate = torch.tensor(0.5, dtype=torch.float32) * torch.tensor(0.004, dtype=torch.float32)
    want = sum(_count(G, S, border, gate.item()) for G in ex.pyramid(img))
    ex.extract(img)
    assert want > 1000 and ex.stats(1)[1][0][0] == want
    ex.close()
