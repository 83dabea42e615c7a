"""The pyramid export against the handle's next call on another stream: that call
uploads a new geometry and reuses the workspace, so it has to wait for the copy too.
A large export and small ones take turns on two streams; every output equals its own
serial export, and nothing is written outside the packed planes."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2605_17869_gb300 as pkg  # noqa: E402

PAD = 1024


@pytest.mark.parametrize("small", [(64, 64), (67, 129), (480, 640)])
def test_next_call_on_another_stream_waits_for_the_export(small):
    ex = pkg.Extractor()
    gen = torch.Generator().manual_seed(small[1])
    imgs = [torch.rand(h, w, generator=gen).cuda() for h, w in ((1080, 1920), small)]
    totals = [pkg.sift_pyramid_size(ex.handle, *im.shape)[1] for im in imgs]

    def export(k, buf, stream):
        h, w = imgs[k].shape
        pkg.sift_build_pyramid(ex.handle, imgs[k].data_ptr(), h, w, w, stream.cuda_stream,
                               buf.data_ptr() + 4 * PAD, totals[k])

    bufs = lambda: [torch.full((t + 2 * PAD,), -7.0, device="cuda") for t in totals]  # noqa: E731
    want = bufs()
    for k in (0, 1):
        export(k, want[k], torch.cuda.current_stream())
        torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(10):
        got = bufs()
        torch.cuda.synchronize()
        for k in (0, 1):
            export(k, got[k], streams[k])
        torch.cuda.synchronize()
        for k in (0, 1):
            assert torch.equal(got[k], want[k]), k
            assert (got[k][:PAD] == -7).all() and (got[k][-PAD:] == -7).all()
    ex.close()
