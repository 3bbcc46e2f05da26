"""The order of the likelihood's chained kernels (programmatic dependent launch).

A chained kernel may start while the one before it still runs; what earlier
kernels wrote is visible to it only after its own griddepcontrol.wait.  So
every kernel that is launched by chain() waits before it does anything else
(read from the source, no GPU), and calls in quick succession with very
different parameters give what each of them gives by itself.
"""
import os
import re

import numpy as np
import pytest

from paper_1505_07674_gb300 import _build as B


def _source():
    with open(os.path.join(B.CSRC, "lensed_kernels.cu")) as f:
        s = f.read()
    return re.sub(r"//[^\n]*", "", s)


CHAINED = sorted(set(re.findall(r"\bchain\(\s*(k_\w+)", _source())))


def test_the_chained_kernels_are_found():
    assert {"k_prologue_comp", "k_prologue_valid", "k_trace_rows", "k_trace_rows_pq", "k_trace_fix64",
            "k_psf", "k_psf_sep", "k_finalize"} <= set(CHAINED)


@pytest.mark.parametrize("kernel", CHAINED)
def test_a_chained_kernel_waits_before_anything_else(kernel):
    s = _source()
    bodies = [s[m.end():] for m in re.finditer(
        r"__global__\s+void\s+(?:__launch_bounds__\([^;{}]*?\)\s+)?" + kernel + r"\s*\([^;{}]*\)\s*\{", s)]
    assert len(bodies) == 1, (kernel, len(bodies))
    assert re.match(r"\s*chain_wait\(\);", bodies[0]), bodies[0][:200]


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["mixed", "mixed_ff"])
def test_calls_in_quick_succession_do_not_mix(precision):
    # the lens moves, grows a core and becomes round from call to call, and
    # some points are invalid: every pixel that the fix-up takes over differs
    torch = pytest.importorskip("torch")
    import paper_1505_07674_gb300 as pkg
    pkg.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1505_07674_gb300 import lensed as LZ
    from workloads import component, fixed, free
    comps = [component("sie", "lens", [free(0), free(1), fixed(0.8), free(2), fixed(20.0), free(3)]),
             component("sersic", "source", [free(4), fixed(0.0), fixed(0.2), fixed(0.0), fixed(1.5),
                                            fixed(0.7), fixed(20.0)])]
    spec = {"nx": 37, "ny": 41, "h": 0.05, "rule": ("gl", 5), "psf": np.ones((3, 3)), "mask": None,
            "zeropoint": 0.0, "components": comps, "n_params": 5}
    rng = np.random.default_rng(11)
    obs = {"data": rng.standard_normal((41, 37)), "variance": np.ones((41, 37))}
    m = LZ.Model(spec, obs, precision=precision)
    calls = []
    for k in range(24):
        n = (1, 3, 40, 160)[k % 4]
        q = (0.5, 0.9995, 0.8)[k % 3]
        p = np.stack([rng.uniform(-0.8, 0.8, n), rng.uniform(-0.8, 0.8, n), np.full(n, q),
                      rng.uniform(0.0, 0.3, n), rng.uniform(-0.2, 0.2, n)], 1)
        p[::7, 2] = 1.5 if k % 2 else q  # an axis ratio out of its domain
        calls.append(torch.as_tensor(p, device="cuda"))
    alone = []
    for p in calls:
        alone.append(m.loglike_batch(p).clone())
        torch.cuda.synchronize()
    for _ in range(5):
        got = [m.loglike_batch(p).clone() for p in calls]
        torch.cuda.synchronize()
        for a, b in zip(alone, got):
            assert torch.equal(a, b)
