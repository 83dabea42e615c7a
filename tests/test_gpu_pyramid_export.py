"""The pyramid export's copy kernel: rows whose width or whose place in the output
does not allow 16-byte stores, FP32 and binary16 octaves, and an output buffer that
starts at any element. Element by element against the same planes exported to an
aligned buffer, and nothing outside the packed planes is written."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2605_17869_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("fp16", [0, 1])
@pytest.mark.parametrize("h,w", [(64, 64), (67, 129), (130, 66)])
def test_export_to_any_element(h, w, fp16):
    img = torch.rand(h, w, generator=torch.Generator().manual_seed(h + w)).cuda()
    ex = pkg.Extractor(fp16_pyramid=fp16)
    _, total = pkg.sift_pyramid_size(ex.handle, h, w)
    stream = torch.cuda.current_stream().cuda_stream
    ref = None
    for shift in range(4):
        buf = torch.full((total + 8,), -7.0, device="cuda")
        pkg.sift_build_pyramid(ex.handle, img.data_ptr(), h, w, w, stream,
                               buf.data_ptr() + 4 * shift, total)
        torch.cuda.synchronize()
        got = buf[shift:shift + total]
        ref = got.clone() if ref is None else ref
        assert torch.equal(got, ref) and (got > -1).all()
        assert (buf[:shift] == -7).all() and (buf[shift + total:] == -7).all()
    ex.close()
