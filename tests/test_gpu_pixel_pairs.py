"""The two-pixels-per-thread ray loop against the one-pixel form, bit for bit.

MIXED_FF offers every launch configuration with the float-float re-traces in
the trace block (one pixel per thread) and as a second pass, whose first pass
traces two pixels per thread.  Every ray takes the same operations with the
same roundings in both, so the results are equal whatever the image size (one
pixel, fewer than a warp's or a block's pixels, one more than that), the
number of nodes per row (chunks of 1 to 4 rays, odd rows, guarded rows beyond
8) and the components.
"""
import numpy as np
import pytest

import workloads as W
from workloads import component, fixed, free

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

RULES = [("point", 1), ("sub", 2), ("gl", 3), ("gl", 4), ("gl", 5), ("gl", 6), ("gl", 7), ("gl", 8),
         ("gl", 9), ("gk", 5), ("sub", 16)]
SIZES = [(1, 1), (5, 3), (9, 7), (8, 8), (13, 5), (127, 1), (16, 8), (43, 3), (67, 41)]


@pytest.fixture(scope="module", autouse=True)
def built():
    import paper_1505_07674_gb300 as pkg
    pkg.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _components(which):
    sie = component("sie", "lens", [free(0), fixed(0.0), free(1), free(2), free(3), fixed(0.01)])
    shear = component("shear", "lens", [free(0), fixed(0.0), fixed(0.04), fixed(25.0)])
    src = component("sersic", "source", [free(4), fixed(0.03), fixed(0.25), fixed(0.0), free(5),
                                         fixed(0.6), fixed(70.0)])
    if which == "plain":
        return [sie, shear, src]
    if which == "bare":  # no lens: every pixel of the source's centre is near it
        return [src]
    return [component("sky", "foreground", [free(4)]),
            component("pointmass", "lens", [fixed(0.313), fixed(-0.217), fixed(0.1)]),
            component("sersic", "foreground", [fixed(0.1), fixed(0.2), fixed(0.4), fixed(1.0), free(5),
                                               fixed(0.8), free(3)]),
            sie, component("sie", "lens", [fixed(0.4), fixed(0.3), fixed(0.2), fixed(1.0), fixed(0.0),
                                           fixed(0.0)]),
            shear, component("gauss", "source", [free(4), fixed(0.0), fixed(0.1), fixed(1.0),
                                                 fixed(0.7), fixed(10.0)]), src]


def _points():
    # x_L, b, q, pa, x_S, n; q = 1 takes the series of atan and atanh
    rng = np.random.default_rng(5)
    lo, hi = np.array([-0.05, 0.3, 0.45, 0.0, -0.1, 0.5]), np.array([0.05, 0.9, 0.99, 180.0, 0.1, 4.0])
    p = lo + (hi - lo) * rng.random((7, 6))
    p[5, 2] = 1.0
    p[6, 0] = 0.0  # the lens centre on the middle ray of odd images
    return p


@pytest.mark.parametrize("which", ["plain", "bare", "all"])
@pytest.mark.parametrize("rule", RULES, ids=lambda r: f"{r[0]}{r[1]}")
def test_pixel_pairs_equal_single_pixels(rule, which):
    from paper_1505_07674_gb300 import lensed as LZ
    sizes = SIZES if rule[1] <= 5 else SIZES[1::3]
    specs, obs = [], []
    for nx, ny in sizes:
        rng = np.random.default_rng(nx * 100 + ny)
        specs.append({"nx": nx, "ny": ny, "h": 0.05, "rule": rule, "psf": None, "mask": None,
                      "zeropoint": 0.0, "components": _components(which), "n_params": 6})
        obs.append({"data": rng.standard_normal((ny, nx)), "variance": np.ones((ny, nx))})
    m = LZ.Model(specs, obs, precision="mixed_ff")
    pts = np.repeat(_points()[None], len(sizes), 0)
    for blk in (0, 2):  # trace blocks of 128 and 64 pixels
        m.set_config(blk)
        ref = m.loglike_batch(pts).cpu().numpy()
        assert np.isfinite(ref).all()
        for cfg in (blk + 12, blk + 18):  # second pass; the same, work-queued
            m.set_config(cfg)
            got = m.loglike_batch(pts).cpu().numpy()
            assert np.array_equal(got, ref), (cfg, np.abs(got - ref).max())
    m.close()
