"""Where the level blur's kernels are compiled: every radius 1 .. 16 once, and those of
the default scale space in the unit that a handle loads anyway (pyramid.cu), since each
further unit costs a handle's creation some 0.4 ms and more."""
import math
import re
from pathlib import Path

import pytest

from oracle import sift_oracle as so

CSRC = Path(__file__).resolve().parent.parent / "paper_2605_17869_gb300" / "csrc"


def _instances(name):
    """Radii of the unit's instances, and of its 40-row ones, in the order of its switch."""
    text = (CSRC / name).read_text()
    radii = lambda fn: [int(r) for r in re.findall(fn + r"<(\d+)>\(variant\)", text)]  # noqa: E731
    return radii("blur_instance"), radii("blur_instance64")


def test_every_radius_has_one_unit():
    main, main64 = _instances("pyramid.cu")
    rest, none = _instances("blur_rest.cu")
    none64, rest64 = _instances("blur_rest64.cu")
    assert main == main64 and rest == rest64 and not none and not none64
    assert sorted(main + rest) == list(range(1, 17))


@pytest.mark.parametrize("up", (False, True))
def test_the_default_radii_are_in_the_pyramids_unit(up):
    p = so.Params(upsample=up)
    sigmas = [so.base_sigma(p)] + [float(k) for k in so.increment_sigmas(p)]
    assert {math.ceil(4 * s) for s in sigmas} <= set(_instances("pyramid.cu")[0])
