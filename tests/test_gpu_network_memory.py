"""Device memory a network holds."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_a_network_holds_no_more_than_its_training_step_needs():
    # per row and hidden unit: five BF16 and three FP32 activations, 22 bytes
    # (the backward pass works in their place); the inputs (two BF16 copies of
    # 32 columns), two floats per row, and the weights, their copies and the
    # split-K slabs (below 64 MB at this width) on top
    import paper_1505_07674_gb300 as pkg
    pkg.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1505_07674_gb300.surrogate import Surrogate
    rows, H = 262144, 256
    Surrogate(18, 64, 64).close()  # the library's modules are loaded
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    net = Surrogate(18, H, rows)
    held = before - torch.cuda.mem_get_info()[0]
    rng = np.random.default_rng(1)
    net.set_params((rng.standard_normal(net.n_params) * 0.05).astype(np.float32))
    X = rng.standard_normal((rows, 18)).astype(np.float32)
    loss, g = net.gradient(X, X[:, 0].copy())
    assert np.isfinite(loss.item()) and bool(torch.isfinite(g).all())
    net.close()
    assert held <= rows * (22 * H + 2 * 2 * 32 + 8) + (64 << 20), held
