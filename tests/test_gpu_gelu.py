"""GPU test of the network's activation and its derivative against FP64, with the
functions compiled from their header."""
import ctypes
import math
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SOURCE = """
#include "gelu.cuh"
__global__ void k(const float *h, float *g, float *d, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        g[i] = gbfd::cnn::gelu(h[i]);
        d[i] = gbfd::cnn::gelu_grad(h[i]);
    }
}
extern "C" int run(const float *h, float *g, float *d, int n)
{
    k<<<(n + 255) / 256, 256>>>(h, g, d, n);
    return (int)cudaDeviceSynchronize();
}
"""

# Units of 2^-24.  Phi = (1 + erf) / 2: erff is within 2 ulps (2 units below 1), the
# sum rounds by 1, halved: 1.5; the argument's rounding moves it by 0.3.
# h phi(h) <= 0.242: expf within 2 ulps (4 units, relative), its argument
# and three products 2.5 more: 1.6.  The last sum, up to 1.13, rounds by 1.
GRAD_ERR = 4.4 * 2.0 ** -24


def test_activation_against_fp64(tmp_path):
    from paper_1707_08900_gb300 import build
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    src, lib = tmp_path / "gelu_test.cu", tmp_path / "gelu_test.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I" + build.SRC_DIR, "-shared",
                    str(src), "-o", str(lib)], check=True)
    h = torch.cat([torch.linspace(-14.0, 14.0, 2 ** 20), torch.linspace(-1.5, 1.5, 2 ** 20),
                   torch.tensor([0.0, -0.0, 1e-30, -1e-30, 40.0, -40.0])]).float().cuda()
    g, d = torch.empty_like(h), torch.empty_like(h)
    fn = ctypes.CDLL(str(lib)).run
    fn.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]
    assert fn(h.data_ptr(), g.data_ptr(), d.data_ptr(), h.numel()) == 0
    x = h.double()
    phi = 0.5 * torch.special.erfc(-x / math.sqrt(2.0))
    want_g = x * phi
    want_d = phi + x * torch.exp(-0.5 * x * x) / math.sqrt(2.0 * math.pi)
    err = float((d.double() - want_d).abs().max())
    assert err <= GRAD_ERR, err * 2.0 ** 24
    # |h| times the error of Phi, and two roundings of the result
    bound = x.abs() * 1.8 * 2.0 ** -24 + want_g.abs() * 2.0 ** -23 + 2.0 ** -149
    assert bool(((g.double() - want_g).abs() <= bound).all())
    assert float(np.float32(d[-2].item())) == 1.0 and float(d[-1].item()) == 0.0
