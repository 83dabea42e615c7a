"""The two arctangent polynomials of the keypoint stages, restated in FP32 from the
coefficients in the source, against the 64-bit arctangent: their error bounds, and that
the orientation's margin leaves every doubtful vote to the exact way."""
import re
from pathlib import Path

import numpy as np
import pytest

SRC = (Path(__file__).resolve().parent.parent / "paper_2605_17869_gb300" / "csrc" / "describe.cu").read_text()
F = np.float32


def _body(name):
    return SRC[SRC.index(name):].split("\n}\n")[0]


def _coefficients(name):
    """Highest power first: the start value and the addends of the chain of FMAs."""
    body = _body(name)
    return [F(v) for v in re.findall(r"float r = (-?[\d.]+)f;", body) + re.findall(r"fmaf\(r, u, (-?[\d.]+)f\)", body)]


def _fma(a, b, c):  # the product of two FP32 values is exact in 64 bits
    return (a.astype(np.float64) * b.astype(np.float64) + np.float64(c)).astype(F)


def _poly(coef, t):
    u = t * t
    r = np.full_like(t, coef[0])
    for c in coef[1:]:
        r = _fma(r, u, c)
    return r * t


def _gradients():
    """Gradient pairs whose magnitude does not vanish in FP32: random ones over all
    magnitudes, and directions on and next to the axes, the diagonals and the borders of the
    36 bins and the 8 bins."""
    rng = np.random.default_rng(5)
    scale = 10.0 ** rng.uniform(-20, 18, 400_000)
    th = rng.uniform(0, 2 * np.pi, scale.size)
    near = np.deg2rad(np.repeat(np.arange(0, 360, 5), 3000)) + rng.normal(0, 3e-5, 72 * 3000)
    th = np.concatenate([th, near, np.deg2rad(np.arange(0, 360, 2.5))])
    scale = np.concatenate([scale, 10.0 ** rng.uniform(-10, 3, near.size), np.ones(144)])
    dx, dy = (scale * np.cos(th)).astype(F), (scale * np.sin(th)).astype(F)
    axis = np.array([[1, 0], [-1, 0], [0, 1], [0, -1], [1, 1], [-1, 1], [1, -1], [-1, -1]], F)
    return np.concatenate([dx, 0.25 * axis[:, 0]]), np.concatenate([dy, 0.25 * axis[:, 1]])


def _quotient(dx, dy, ulps):
    """min / max by an approximate reciprocal that is off by so many units in the last place."""
    ax, ay = np.abs(dx), np.abs(dy)
    rcp = F(1) / np.maximum(ax, ay)
    for _ in range(abs(ulps)):
        rcp = np.nextafter(rcp, F(np.inf) if ulps > 0 else F(0))
    return np.minimum(ax, ay) * rcp


@pytest.mark.parametrize("ulps", (-1, 0, 1))
def test_orientation_bins(ulps):
    margin = float(re.search(r"kVoteMargin = ([\d.e-]+)f", SRC).group(1))
    dx, dy = _gradients()
    coef = _coefficients("int ori_bin(")
    assert len(coef) == 6
    r = _poly(coef, _quotient(dx, dy, ulps))
    r = np.where(np.abs(dy) > np.abs(dx), F(9) - r, r)
    r = np.where(dx < 0, F(18) - r, r)
    r = np.where(dy < 0, F(36) - r, r).astype(F)
    exact = np.mod(np.arctan2(dy.astype(np.float64), dx.astype(np.float64)), 2 * np.pi) * (18 / np.pi)
    err = np.abs(r - exact)
    err = np.minimum(err, 36 - err)
    # The fit is 2.8e-5 bins off at most; the quotient (1.5 ulp), the chain and the three
    # differences up to 36 round by less than 6e-6 together.
    assert err.max() < 3.4e-5
    assert err.max() < margin / 4
    # Away from the borders by the margin, the nearest integer is the exact bin.
    m = (r + F(12582912)).astype(F)
    bins = (m.view(np.int32) & 63) % 36
    sure = np.abs(r - (m - F(12582912))) < F(0.5) - F(margin)
    want = np.floor(exact + 0.5).astype(int) % 36
    assert sure.mean() > 0.6 and (bins[sure] == want[sure]).all()
    # The diagonals lie on a border: left to the exact way.
    assert not sure[np.abs(dx) == np.abs(dy)].any()


@pytest.mark.parametrize("ulps", (-1, 0, 1))
def test_descriptor_angles(ulps):
    dx, dy = _gradients()
    coef = _coefficients("float atan2_eighths(")
    assert len(coef) == 9
    r = _poly(coef, _quotient(dx, dy, ulps))
    r = np.where(np.abs(dy) > np.abs(dx), F(2) - r, r)
    r = np.where(dx < 0, F(4) - r, r)
    r = np.where(dy < 0, F(8) - r, r)
    exact = np.mod(np.arctan2(dy.astype(np.float64), dx.astype(np.float64)), 2 * np.pi) * (4 / np.pi)
    err = np.abs(r - exact)
    err = np.minimum(err, 8 - err)
    # Chain and quotient: 1.5e-7 + 1.5 ulp of 1, relative to values up to 1; the differences:
    # half a unit in the last place of 2, 4 and 8. atan2f's 3 ulp of pi are 9e-7 in these units.
    assert err.max() < 1.5e-7 + 1.8e-7 + 0.6e-7 + 1.2e-7 + 2.4e-7
    # A quotient of two infinities is taken as 1, and no reciprocal is flushed to 0.
    assert re.search(r"fminf\(fminf\(ax, ay\), 0x1p126f\) \* rcp_approx\(fminf\(.*, 0x1p126f\)\)",
                     _body("float atan2_eighths("))
