"""GPU test of the library in a second CUDA context of the same device: function
attributes belong to the context, so kernels with more than 48 KB of shared
memory must run there too, after they have run in the first one."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CHILD = r"""
import ctypes
import numpy as np
import torch
from paper_1707_08900_gb300 import gbfd, inputs

shape = (16, 16, 32)
st = inputs.random_state(shape, 3, scale=0.02)
torch.zeros(1, device="cuda")
cu = ctypes.CDLL("libcuda.so.1")


def run(precision, first):
    if first:
        s = gbfd.Solver(shape, precision=precision)
        s.set_state(st)
        s.rk3_step(0.01, 1)
        s.sync()
        out = s.get_state()
        s.close()
        return out
    p = gbfd.make_params(shape, precision=precision)
    nbytes = gbfd.gbfd_workspace_bytes(p)
    ws = ctypes.c_uint64()
    assert cu.cuMemAlloc_v2(ctypes.byref(ws), ctypes.c_size_t(nbytes)) == 0
    ctx = gbfd.gbfd_init(p, ws.value, nbytes, 0)
    gbfd.gbfd_set_state(ctx, st.ctypes.data, 0, 1)
    gbfd.gbfd_rk3_step(ctx, 0.01, 1)
    gbfd.gbfd_sync(ctx)
    out = np.empty_like(st)
    gbfd.gbfd_get_state(ctx, out.ctypes.data, 0, 1)
    gbfd.gbfd_destroy(ctx)
    assert cu.cuMemFree_v2(ws) == 0
    return out


KINDS = ("fp32", "fp64", "fp32_acc64", "fp32_accff")
want = [run(k, True) for k in KINDS]
dev, ctx = ctypes.c_int(), ctypes.c_void_p()
assert cu.cuDeviceGet(ctypes.byref(dev), 0) == 0
assert cu.cuCtxCreate_v2(ctypes.byref(ctx), 0, dev) == 0  # and makes it current
for k, w in zip(KINDS, want):
    assert np.array_equal(run(k, False), w), k
assert cu.cuCtxDestroy_v2(ctx) == 0
print("second context ok")
"""


def test_solver_in_a_second_context():
    from paper_1707_08900_gb300 import build
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=root, capture_output=True, text=True,
                       timeout=300, env=dict(os.environ, PYTHONPATH=root))
    assert r.returncode == 0 and "second context ok" in r.stdout, r.stdout + r.stderr
