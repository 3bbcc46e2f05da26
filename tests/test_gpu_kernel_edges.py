"""Kernels at the edges of their tiles, ranges and launch rules.

Each check compares a kernel with another path of the library or with a plain
64-bit evaluation; the tolerance is stated with its reason where it is not
bit equality.
"""
import numpy as np
import pytest

import workloads as W
from workloads import component, fixed, free

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    import paper_1505_07674_gb300 as pkg
    pkg.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _spec(nx, ny, comps, n_params, rule=("gl", 2), psf=None, mask=None):
    return {"nx": nx, "ny": ny, "h": 0.05, "rule": rule, "psf": psf, "mask": mask,
            "zeropoint": 0.0, "components": comps, "n_params": n_params}


def _psf(shape, rank):
    rng = np.random.default_rng(shape[0] * 100 + shape[1])
    if rank:  # a sum of `rank` outer products
        return sum(np.outer(rng.random(shape[0]) + 0.2, rng.random(shape[1]) + 0.2) for _ in range(rank))
    return rng.random(shape) + 0.1


@pytest.mark.parametrize("shape", [(1, 1), (1, 5), (5, 1), (3, 3), (3, 31), (31, 3), (9, 7), (21, 21), (31, 31)])
@pytest.mark.parametrize("rank", [0, 1, 3])
def test_psf_kernels_at_tile_edges(shape, rank):
    # chi^2 against zero data is the weighted square sum of the convolved
    # image: float sums of at most 31 + 31 terms per output (direct) or two of
    # 31 (separable) are off by < 62 x 2^-24 = 4e-6 of it, its square by twice
    # that, whatever the signs; the 64-bit mode is the reference
    from paper_1505_07674_gb300 import lensed as LZ
    comps = [component("gauss", "source", [free(0), free(1), fixed(0.3), fixed(0.0), fixed(0.7), fixed(30.0)])]
    sizes = [(1, 1), (3, 40), (64, 32), (65, 33), (130, 17), (16, 70)]
    specs, obs = [], []
    for k, (nx, ny) in enumerate(sizes):
        mask = (np.random.default_rng(k).random((ny, nx)) < 0.4).astype(np.uint8) if k % 2 else None
        if mask is not None:
            mask[0, 0] = 0
        specs.append(_spec(nx, ny, comps, 2, psf=_psf(shape, rank), mask=mask))
        obs.append({"data": np.zeros((ny, nx)), "variance": np.full((ny, nx), 0.01)})
    pts = np.tile(np.array([[0.0, 0.0], [0.4, -0.3], [-0.7, 0.2]]), (len(sizes), 1, 1))
    ref = LZ.Model(specs, obs, precision="fp64").loglike_batch(pts).cpu().numpy()
    m = LZ.Model(specs, obs, precision="fp32")
    for cfg in (0, 3):  # direct, separable
        m.set_config(cfg)
        got = m.loglike_batch(pts).cpu().numpy()
        assert np.all(np.abs(got - ref) <= 1e-5 * np.abs(ref)), (cfg, np.abs(got / ref - 1).max())


@pytest.mark.parametrize("n", [0.15, 0.2, 0.21, 0.5, 1.0, 2.7, 4.0, 11.9, 12.0, 12.5])
def test_sersic_constants_inside_and_outside_the_tables(n):
    # the 64-bit mode against the oracle's own b_n (bisection) and gamma
    # function: a few hundred operations at 2^-53 and the tables' 3e-15
    # relative error, times ln-scale factors of up to 2n ~ 25: 1e-12
    from oracle import oracle as O
    from paper_1505_07674_gb300 import lensed as LZ
    comps = [component("sersic", "source", [fixed(0.02), fixed(-0.03), free(0), free(1), free(2), fixed(0.6),
                                            fixed(40.0)])]
    spec = _spec(24, 20, comps, 3)
    obs = {"data": np.zeros((20, 24)), "variance": np.ones((20, 24))}
    pts = np.array([[0.3, -1.0, n], [0.5, 2.0, n]])
    got = LZ.Model(spec, obs, precision="fp64").loglike_batch(pts).cpu().numpy()[0]
    ref = O.OracleSystem(spec, obs).loglike(pts)
    assert np.all(np.abs(got - ref) <= 1e-12 * np.abs(ref)), got / ref - 1


@pytest.mark.parametrize("precision", ["mixed", "mixed_ff"])
@pytest.mark.parametrize("core,q", [(0.0, 0.8), (0.01, 0.8), (0.3, 0.5), (0.01, 0.999), (0.05, 1.0)])
def test_fix_up_of_one_point_equals_its_place_in_a_batch(precision, core, q):
    # a launch of few points splits each point's FP64 pixels over several
    # blocks; a large one gives a point one block: the same bits
    from paper_1505_07674_gb300 import lensed as LZ
    comps = [component("sie", "lens", [free(0), fixed(0.0), fixed(0.8), fixed(q), free(1), fixed(core)]),
             component("sie", "lens", [fixed(0.5), fixed(0.4), fixed(0.2), fixed(0.7), fixed(0.0), fixed(0.02)]),
             component("sersic", "source", [free(2), fixed(0.0), fixed(0.2), fixed(0.0), fixed(1.5), fixed(0.7),
                                            fixed(20.0)])]
    spec = _spec(37, 41, comps, 3, rule=("gl", 5))
    rng = np.random.default_rng(3)
    obs = {"data": rng.standard_normal((41, 37)), "variance": np.ones((41, 37))}
    pts = np.stack([rng.uniform(-0.1, 0.1, 200), rng.uniform(0, 180, 200), rng.uniform(-0.2, 0.2, 200)], 1)
    m = LZ.Model(spec, obs, precision=precision)
    whole = m.loglike_batch(pts).cpu().numpy()[0]
    for k in (0, 57, 199):
        assert m.loglike_batch(pts[k:k + 1]).cpu().numpy()[0, 0] == whole[k]
    assert np.array_equal(m.loglike_batch(pts[:9]).cpu().numpy()[0], whole[:9])


@pytest.mark.parametrize("H,d", [(64, 1), (64, 64), (128, 32), (192, 33), (256, 18), (320, 18)])
@pytest.mark.parametrize("B", [1, 127, 128, 129, 1000])
def test_network_forward_at_tile_edges(H, d, B):
    # both forward paths (one kernel up to 256 wide, layer by layer in a
    # gradient call): the loss of the gradient call is that of the forward
    # outputs (float sums of B terms: 1e-5), and the outputs agree with a
    # 64-bit evaluation to the BF16 roundings of three layers (2^-8 each,
    # averaged over the width: 2e-2 in the 2-norm)
    from paper_1505_07674_gb300.surrogate import Surrogate
    rng = np.random.default_rng(H + d)
    shapes = ((H, d), (H,), (H, H), (H,), (H, H), (H,), (H,), (1,))
    parts = [rng.standard_normal(s) * (np.sqrt(2.0 / s[1]) if len(s) == 2 else 0.1) for s in shapes]
    theta = np.concatenate([p.ravel() for p in parts]).astype(np.float32)
    X = rng.standard_normal((B, d)).astype(np.float32)
    t = rng.standard_normal(B).astype(np.float32)
    net = Surrogate(d, H, 1024)
    net.set_params(theta)
    y = net.forward(X).cpu().numpy().astype(np.float64)
    loss, _ = net.gradient(X, t)
    assert abs(loss.item() - 0.5 * np.mean((y - t) ** 2)) <= 1e-5 * 0.5 * np.mean((y - t) ** 2)
    W1, b1, W2, b2, W3, b3, w4, b4 = [p.astype(np.float32).astype(np.float64) for p in parts]
    h = X.astype(np.float64)
    for Wl, bl in ((W1, b1), (W2, b2), (W3, b3)):
        z = h @ Wl.T + bl
        h = z / (1.0 + np.exp(-z))
    ref = h @ w4 + b4
    scale = np.sqrt(np.mean((np.abs(h) @ np.abs(w4)) ** 2))
    assert np.sqrt(np.mean((y - ref) ** 2)) <= 2e-2 * scale
    net.close()


def test_network_activations_at_the_ends_of_their_range():
    # one hidden unit of each layer passes its input on: activations far out on
    # both sides stay finite and exact (silu(z) = z for large z), and an
    # infinite activation gives an infinite output
    from paper_1505_07674_gb300.surrogate import Surrogate
    H = 64
    for x, want in ((2048.0, 2048.0), (-2048.0, 0.0), (0.0, 0.0), (3e38, np.inf)):
        parts = [np.zeros(s) for s in ((H, 1), (H,), (H, H), (H,), (H, H), (H,), (H,), (1,))]
        parts[0][0, 0] = parts[2][0, 0] = parts[4][0, 0] = parts[6][0] = 1.0
        if np.isinf(want):
            parts[2][0, 0] = 4.0
        net = Surrogate(1, H, 64)
        net.set_params(np.concatenate([p.ravel() for p in parts]))
        y = net.forward(np.full((3, 1), x, np.float32)).cpu().numpy()
        net.close()
        if np.isinf(want):
            # (0 x inf in the other units' products is NaN in any evaluation)
            assert not np.isfinite(y).any()
        else:
            # (silu(-2048) is -1e-32 at most, whatever the form of the exponential)
            assert np.all(np.abs(y - want) <= 1e-30), (x, y)
