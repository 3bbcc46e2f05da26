"""The guarded two-pixel ray loop (rules of more than 8 nodes per row) against the
one-pixel form, bit for bit.

FP32 models trace two pixels per thread; MIXED_FF ones with more than 8 nodes
per row trace one.  With Gaussian and flat lights MIXED_FF re-traces nothing,
and with coreless lenses of e >= 0.05 its fix-up recomputes nothing, so both
modes do the same FP32 operations with the same roundings.
"""
import numpy as np
import pytest

from workloads import component, fixed, free

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES = [(1, 1), (5, 3), (8, 8), (43, 3), (67, 41)]


def _components(lenses):
    out = [component("gauss", "source", [free(4), fixed(0.0), fixed(0.2), fixed(0.0), free(5), fixed(10.0)])]
    if lenses == 0:
        return out
    sie = component("sie", "lens", [free(0), fixed(0.01), free(1), free(2), free(3), fixed(0.0)])
    if lenses == 1:
        return [sie] + out
    return [component("sky", "foreground", [free(1)]),
            component("pointmass", "lens", [fixed(0.313), fixed(-0.217), fixed(0.1)]),
            component("gauss", "foreground", [fixed(0.1), fixed(0.2), fixed(0.4), fixed(1.0), free(5), free(3)]),
            sie, component("sie", "lens", [fixed(0.4), fixed(0.3), fixed(0.2), free(2), fixed(0.0), fixed(0.0)]),
            component("shear", "lens", [free(0), fixed(0.0), fixed(0.04), fixed(25.0)])] + out


@pytest.mark.parametrize("lenses", [0, 1, 2])
@pytest.mark.parametrize("rule", [("gl", 9), ("gl", 10), ("gk", 5), ("sub", 12), ("gk", 7), ("sub", 16)],
                         ids=lambda r: f"{r[0]}{r[1]}")
def test_guarded_pixel_pairs_equal_single_pixels(rule, lenses):
    import paper_1505_07674_gb300 as pkg
    pkg.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1505_07674_gb300 import lensed as LZ
    specs, obs = [], []
    for nx, ny in SIZES:
        rng = np.random.default_rng(nx * 100 + ny)
        specs.append({"nx": nx, "ny": ny, "h": 0.05, "rule": rule, "psf": None, "mask": None,
                      "zeropoint": 0.0, "components": _components(lenses), "n_params": 6})
        obs.append({"data": rng.standard_normal((ny, nx)), "variance": np.ones((ny, nx))})
    # x_L, b, q, pa, x_S, q_S
    rng = np.random.default_rng(5)
    lo, hi = np.array([-0.05, 0.3, 0.45, 0.0, -0.1, 0.5]), np.array([0.05, 0.9, 0.99, 180.0, 0.1, 0.9])
    pts = np.repeat((lo + (hi - lo) * rng.random((9, 6)))[None], len(SIZES), 0)
    pairs = LZ.Model(specs, obs, precision="fp32")
    single = LZ.Model(specs, obs, precision="mixed_ff")
    for cfg in (0, 2, 6):  # blocks of 128 and 64 pixels, work-queued
        single.set_config(cfg)
        ref = single.loglike_batch(pts).cpu().numpy()
        assert np.isfinite(ref).all()
        pairs.set_config(cfg)
        got = pairs.loglike_batch(pts).cpu().numpy()
        assert np.array_equal(got, ref), (cfg, np.abs(got - ref).max())
    pairs.close()
    single.close()
