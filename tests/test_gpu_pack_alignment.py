"""Packing reads the descriptors by 16-byte loads, while an extraction writes them to any
buffer of floats: after an extraction into a buffer that starts elsewhere, packing is
refused on the host, and nothing is launched."""
import ctypes

import pytest

from workloads import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2605_17869_gb300 as pkg  # noqa: E402
from paper_2605_17869_gb300 import _abi  # noqa: E402

K = 512


@pytest.mark.parametrize("off,status", [(0, pkg.SIFT_OK), (1, pkg.SIFT_E_INVALID),
                                        (2, pkg.SIFT_E_INVALID), (4, pkg.SIFT_OK)])
def test_pack_after_an_extraction_into_an_offset_buffer(off, status):
    ex = pkg.Extractor(max_kpts=K)
    img = torch.from_numpy(synth.make_image(synth.rng_for(83, 0), 200, 300)).cuda()
    ref = ex.extract(img)
    buf = pkg.OutputBuffers(K, img.device)
    desc = torch.zeros(K * 128 + 4, device="cuda")
    count = torch.zeros(1, dtype=torch.int32, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    pkg.sift_extract(ex.handle, img.data_ptr(), 200, 300, 300, stream, buf.kpts(),
                     desc.data_ptr() + 4 * off, count.data_ptr())
    n = int(count.item())
    assert n == ref.count > 0
    assert torch.equal(desc[off:off + n * 128].view(n, 128), ref.desc)
    dst = torch.zeros(K * 540, dtype=torch.uint8, device="cuda")
    st = _abi.load().sift_pack_outputs(ex.handle, ctypes.c_void_p(stream), ctypes.c_void_p(dst.data_ptr()),
                                       ctypes.c_size_t(dst.numel()))
    assert st == status
    if st == pkg.SIFT_OK:
        assert torch.equal(dst[:n * 512].view(torch.float32).view(n, 128), ref.desc)
    ex.close()
