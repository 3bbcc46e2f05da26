"""Values far out: activations, fluxes and pixel values at the ends of the range
that the entry points take, against plain 64-bit evaluations.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    import paper_1505_07674_gb300 as pkg
    pkg.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _unit_path(H, w1=1.0, w2=-1.0, w3=-1.0, b2=0.0):
    """A network whose first unit of each layer passes its input on."""
    parts = [np.zeros(s) for s in ((H, 1), (H,), (H, H), (H,), (H, H), (H,), (H,), (1,))]
    parts[0][0, 0], parts[2][0, 0], parts[4][0, 0], parts[6][0] = w1, w2, w3, 1.0
    parts[3][0] = b2
    return np.concatenate([p.ravel() for p in parts])


FAR = (-60.0, -79.0, -81.0, -86.0, -88.5, -100.0, -2048.0, -1e10, -1e28, -1e30, -1e35, -3e38)


@pytest.mark.parametrize("H", [64, 256, 320])
def test_silu_of_very_negative_values_vanishes(H):
    # silu(z) is z exp(z) to within 1e-25 of itself below -60: at most 6e-25 in
    # size, and the weights of -1 that follow would carry anything larger on.
    # One hidden width above the single forward kernel's limit
    from paper_1505_07674_gb300.surrogate import Surrogate
    net = Surrogate(1, H, 64)
    net.set_params(_unit_path(H))
    y = net.forward(np.array(FAR, np.float32)[:, None]).cpu().numpy()
    net.close()
    assert np.all(np.abs(y) <= 1e-24), y


@pytest.mark.parametrize("x", FAR)
def test_silu_derivative_of_very_negative_values_vanishes(x):
    # layer 1's activation and derivative vanish; a bias of 1 in layer 2 keeps
    # the rest of the path alive, so its gradients are those of x = -infinity
    from paper_1505_07674_gb300.surrogate import Surrogate
    H, B = 64, 3
    net = Surrogate(1, H, 64)
    net.set_params(_unit_path(H, w2=1.0, w3=1.0, b2=1.0))
    loss, g = net.gradient(np.full((B, 1), x, np.float32), np.zeros(B, np.float32))
    g = g.cpu().numpy().astype(np.float64)
    loss = loss.item()
    net.close()

    def silu(z):
        return z / (1.0 + np.exp(-z))

    def grad(z):
        s = 1.0 / (1.0 + np.exp(-z))
        return s * (1.0 + z * (1.0 - s))
    h2 = silu(1.0)
    y = silu(h2)
    # BF16 roundings of two activations and of the layers' gradients: 2^-8 each
    assert abs(loss - 0.5 * y * y) <= 3e-2 * 0.5 * y * y
    o_b1, o_b2 = H, 2 * H + H * H
    assert abs(g[o_b2] - y * grad(h2) * grad(1.0)) <= 3e-2 * abs(y * grad(h2) * grad(1.0))
    # silu'(z) ~ z exp(z): at most 6e-25 in size
    assert abs(g[o_b1]) <= 1e-24, g[o_b1]
    assert abs(g[0]) <= 1e-24 * max(1.0, abs(x)) and np.isfinite(g).all()


@pytest.mark.parametrize("precision,config", [("fp32", 0), ("fp32", 3), ("mixed_ff", 0), ("mixed_ff", 12),
                                              ("fp64", 0)])
def test_chi2_beyond_the_largest_float(precision, config):
    # every pixel's squared residual fits a float, the sum of a warp's does not.
    # The source is too faint for a float; per term the rounding of the data and
    # of two products (4 x 2^-24), the sum in FP64: 1e-6
    from paper_1505_07674_gb300 import lensed as LZ
    from workloads import component, fixed, free
    comps = [component("gauss", "source", [free(0), fixed(0.0), fixed(0.3), fixed(1000.0), fixed(0.7),
                                           fixed(30.0)])]
    ny, nx = 40, 70
    psf = np.outer([1.0, 2.0, 1.0], [1.0, 3.0, 1.0])
    spec = {"nx": nx, "ny": ny, "h": 0.05, "rule": ("gl", 2), "psf": psf, "mask": None, "zeropoint": 0.0,
            "components": comps, "n_params": 1}
    rng = np.random.default_rng(2)
    data = rng.uniform(0.9e19, 1.8e19, (ny, nx))
    m = LZ.Model(spec, {"data": data, "variance": np.ones((ny, nx))}, precision=precision)
    m.set_config(config)
    got = m.loglike_batch(np.array([[0.0], [0.1]])).cpu().numpy()
    m.close()
    want = -0.5 * np.sum(data * data)
    assert np.all(np.abs(got - want) <= 1e-6 * abs(want)), got


def test_gaussian_flux_keeps_its_precision():
    # one pixel of side 1 with one ray at the centre of a Gaussian: in 64 bits
    # -2 loglike is the square of F / (2 pi sigma^2), so the ratio to magnitude
    # 0 is F^2 = 10^(-0.8 mag).  With u = 2^-53 the exponent -0.4 mag of the
    # power carries 1.5 u (the constant and the product), ln 10 |0.4 mag| times
    # that in F; the power itself 2 ulp (4 u), the quotient u; F squared doubles
    # it, and the two squares, the reference's square and the ratio add 5 u
    from decimal import Decimal, getcontext
    from paper_1505_07674_gb300 import lensed as LZ
    from workloads import component, fixed, free
    getcontext().prec = 40
    comps = [component("gauss", "source", [fixed(0.0), fixed(0.0), fixed(0.8), free(0), fixed(0.7), fixed(0.0)])]
    spec = {"nx": 1, "ny": 1, "h": 1.0, "rule": ("point", 1), "psf": None, "mask": None, "zeropoint": 0.0,
            "components": comps, "n_params": 1}
    mag = np.concatenate([[0.0], np.arange(-25.0, 26.0), np.random.default_rng(4).uniform(-25, 25, 1500)])
    m = LZ.Model(spec, {"data": np.zeros((1, 1)), "variance": np.ones((1, 1))}, precision="fp64")
    ll = m.loglike_batch(mag[:, None]).cpu().numpy()[0]
    m.close()
    u = 2.0 ** -53
    for v, got in zip(mag, ll / ll[0]):
        want = Decimal(10) ** (Decimal(-8) / Decimal(10) * Decimal(float(v)))
        err = abs(float(Decimal(float(got)) / want - 1))
        assert err <= u * (2 * (1.5 * np.log(10.0) * 0.4 * abs(v) + 5) + 5), (v, err / u)
