"""The work-queued trace against the plain grid, bit for bit, with one, two and four
items taken at a time and with numbers of items that leave remainders."""
import numpy as np
import pytest

from workloads import component, fixed, free

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision,plain,queued", [("fp32", 0, 6), ("fp32", 2, 8), ("mixed_ff", 0, 6),
                                                    ("mixed_ff", 12, 18)])
def test_work_queue_equals_the_plain_grid(precision, plain, queued):
    import paper_1505_07674_gb300 as pkg
    pkg.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1505_07674_gb300 import lensed as LZ
    comps = [component("sie", "lens", [free(0), fixed(0.0), fixed(0.8), free(1), fixed(20.0), fixed(0.01)]),
             component("sersic", "source", [free(2), fixed(0.0), fixed(0.2), fixed(0.0), fixed(1.5), fixed(0.7),
                                            fixed(20.0)])]
    # two systems, so that a turn of the queue crosses from one to the other;
    # 131 + 33 blocks of 128 pixels a point: 164 to 49,200 items
    specs, obs = [], []
    for nx, ny in ((129, 130), (65, 64)):
        specs.append({"nx": nx, "ny": ny, "h": 0.05, "rule": ("gl", 2), "psf": None, "mask": None,
                      "zeropoint": 0.0, "components": comps, "n_params": 3})
        obs.append({"data": np.zeros((ny, nx)), "variance": np.ones((ny, nx))})
    rng = np.random.default_rng(9)
    m = LZ.Model(specs, obs, precision=precision)
    for P in (1, 3, 37, 61, 97, 131, 300):
        pts = np.stack([rng.uniform(-0.1, 0.1, P), rng.uniform(0.5, 0.95, P), rng.uniform(-0.2, 0.2, P)], 1)
        pts[::5, 1] = 1.5  # an invalid point now and then
        pts = np.repeat(pts[None], 2, 0)
        m.set_config(plain)
        ref = m.loglike_batch(pts).cpu().numpy()
        m.set_config(queued)
        got = m.loglike_batch(pts).cpu().numpy()
        assert np.array_equal(got, ref), P
    m.close()
