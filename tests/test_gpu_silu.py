"""quotient2 and SiLU (lensed_silu.cuh) against CUDA's division operator.

A probe kernel, compiled here from the library's header with its flags, puts
the header's quotients beside those of the operator.  They are the same bits
over the range the header states, but for divisors whose significand is all
ones, where one unit in the last place may differ.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_1505_07674_gb300 import _build as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PROBE = r"""
#include "lensed_silu.cuh"
using namespace lensed;
// out: [6][count]: n / d both ways; silu and its derivative both ways (of n)
__global__ void k(const float *n, const float *d, int count, float *out)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        const float z = n[i], e = 1.f + __expf(-z);
        const float2 q = quotient2(make_float2(z, 1.f), make_float2(d[i], d[i]));
        float2 v[1] = {make_float2(z, z)}, h[1], g[1];
        silu<false>(v, h);
        silu<true>(v, g);
        const float s = 1.f / e;
        out[i] = q.x;
        out[count + i] = z / d[i];
        out[2 * count + i] = h[0].y;
        out[3 * count + i] = z / e;
        out[4 * count + i] = g[0].x;
        out[5 * count + i] = s * (1.f + z * (1.f - s));
        out[6 * count + i] = e;
    }
}
extern "C" int probe(const float *n, const float *d, int count, float *out)
{
    k<<<512, 256>>>(n, d, count, out);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    tmp = tmp_path_factory.mktemp("probe")
    src, lib = os.path.join(tmp, "p.cu"), os.path.join(tmp, "p.so")
    with open(src, "w") as f:
        f.write(PROBE)
    subprocess.run([B.nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-shared", src, "-o", lib], check=True)
    fn = C.CDLL(lib).probe

    def run(n, d):
        n, d = np.ascontiguousarray(n, np.float32), np.ascontiguousarray(d, np.float32)
        tn, td = torch.from_numpy(n).cuda(), torch.from_numpy(d).cuda()
        out = torch.empty((7, len(n)), dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        assert fn(C.c_void_p(tn.data_ptr()), C.c_void_p(td.data_ptr()), len(n),
                  C.c_void_p(out.data_ptr())) == 0
        return out.cpu().numpy()
    return run


def _ordered(a):
    """Floats as integers in their order (neighbours differ by 1)."""
    i = a.view(np.int32).astype(np.int64)
    return np.where(i < 0, -(i & 0x7fffffff), i)


def _same(a, b, d):
    ones = (d.view(np.uint32) & 0x7fffff) == 0x7fffff
    off = np.abs(_ordered(a) - _ordered(b))
    bad = np.where(ones, off > 1, off > 0)
    assert not bad.any(), (bad.sum(), a[bad][:5], b[bad][:5], d[bad][:5])


def test_quotients_over_the_stated_range(probe):
    rng = np.random.default_rng(7)
    count = 4_000_000
    d = np.ldexp(rng.uniform(1, 2, count), rng.integers(0, 126, count)).astype(np.float32)
    d[:4] = [1.0, 2.0, np.nextafter(np.float32(2), np.float32(1)), np.float32(2.0 ** 125)]
    q = np.ldexp(rng.uniform(1, 2, count), rng.integers(-60, 60, count))
    with np.errstate(over="ignore"):
        n = (q * d.astype(np.float64) * rng.choice([-1, 1], count)).astype(np.float32)
    ok = np.isfinite(n) & (np.abs(n) >= 2.0 ** -100) & (np.abs(n) < 3e38)
    n, d = n[ok], d[ok]
    out = probe(n, d)
    _same(out[0], out[1], d)


def test_silu_takes_the_quotients_of_the_division_operator(probe):
    rng = np.random.default_rng(8)
    # every size of float of both signs, and the range activations lie in
    bits = rng.integers(0, 0x7f800000, 2_000_000).astype(np.uint32)
    z = np.concatenate([bits.view(np.float32), -bits.view(np.float32),
                        rng.uniform(-100, 100, 2_000_000).astype(np.float32),
                        rng.standard_normal(2_000_000).astype(np.float32),
                        np.float32([0.0, -0.0, -80.0, np.nextafter(np.float32(-80), np.float32(-90)), 1e-45,
                                    -1e-45, 3.4e38, -3.4e38])])
    out = probe(z, np.ones_like(z))
    _same(out[2], out[3], out[6])
    # the derivative is two further operations on the quotient 1 / d: where
    # that is the same, so are they
    exact = (out[6].view(np.uint32) & 0x7fffff) != 0x7fffff
    assert np.array_equal(out[4][exact].view(np.uint32), out[5][exact].view(np.uint32))
