"""A tuning cache written with other kernels: its entries were timed for other tile
heights, so a batch tuned then is tuned again and its new entry stored beside the old."""
import json

import pytest

from workloads import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2605_17869_gb300 as pkg  # noqa: E402


def test_entries_of_other_kernels_are_not_applied(tmp_path):
    path = str(tmp_path / "tuning.json")
    img = torch.from_numpy(synth.make_image(synth.rng_for(84, 0), 96, 128)).cuda()
    ex = pkg.Extractor()
    prop = torch.cuda.get_device_properties(0)
    device = f"sm{prop.major}{prop.minor}x{prop.multi_processor_count};"
    sig = pkg.sift_batch_signature(ex.params, [96], [128])
    old = '{"blur_tile_rows": [[64, 64, 64, 64, 64]], "extrema_ctas_per_sm": 1}'
    pkg.sift_tuning_cache_put(path, device + sig, old)  # the key before kernels were numbered
    _, hit = ex.autotune_batch([img], cache=path)
    assert not hit
    with open(path) as f:
        entries = json.load(f)["entries"]
    assert entries[device + sig] == json.loads(old) and len(entries) == 2
    js, hit = ex.autotune_batch([img], cache=path)  # the new entry is found
    assert hit
    new = next(v for k, v in entries.items() if k != device + sig)
    assert json.loads(js) == new
    ex.close()
