"""The matcher reads descriptors by 16-byte loads: sets that start elsewhere are
refused on the host (the header asks for 16-byte alignment), and nothing is launched."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2605_17869_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("off_a,off_b", [(1, 0), (0, 2), (3, 3)])
def test_misaligned_sets_are_refused(off_a, off_b):
    ex = pkg.Extractor()
    buf = torch.zeros(40 * 128 + 4, device="cuda")
    a = buf[off_a:off_a + 20 * 128].view(20, 128)
    b = buf[20 * 128 + off_b:40 * 128 + off_b].view(20, 128)
    with pytest.raises(pkg.SiftError) as e:
        ex.match(a, b)
    assert e.value.status == pkg.SIFT_E_INVALID and "aligned" in str(e.value)
    # Sets of four elements further on are aligned again; an empty set may lie anywhere.
    assert ex.match(buf[4:4 + 20 * 128].view(20, 128), buf[:20 * 128].view(20, 128)).shape == (20,)
    assert (ex.match(buf[:20 * 128].view(20, 128), buf[1:1].view(0, 128)) == -1).all()
    ex.close()
