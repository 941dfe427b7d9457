"""GPU test of the kernel path option for the FP64 19-point form: path 0 asked for
launches the tiled kernel, path 1 and the unset default the simple one (told apart
by the kernel names of a captured step)."""
import ctypes

import numpy as np
import pytest

from paper_1707_08900_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPE = (20, 44, 36)


def _run(st, options, dot):
    """State after two steps, and whether the first pass is the simple kernel."""
    from paper_1707_08900_gb300 import gbfd
    stream = torch.cuda.Stream()
    s = gbfd.Solver(SHAPE, lengths=(3.0, 4.5, 2.5), precision="fp64", form="19p", nu=0.02,
                    stream=stream)
    for k, v in options:
        s.set_option(k, v)
    s.set_state(st)
    s.rk3_step(0.01, 2)
    s.sync()
    out = s.get_state()
    cu, graph = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p()
    handle = ctypes.c_void_p(stream.cuda_stream)
    assert cu.cuStreamBeginCapture_v2(handle, 1) == 0  # thread-local
    s.substep(0, 0.01)
    assert cu.cuStreamEndCapture(handle, ctypes.byref(graph)) == 0
    assert cu.cuGraphDebugDotPrint(graph, str(dot).encode(), 1) == 0  # verbose: kernel names
    assert cu.cuGraphDestroy(graph) == 0
    text = dot.read_text()
    s.close()
    assert ("k_substep_simple" in text) != ("k_substep_tiled" in text), text
    return out, "k_substep_simple" in text


def test_path_zero_runs_the_tiled_kernels(tmp_path):
    from paper_1707_08900_gb300 import build, gbfd
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    st = inputs.random_state(SHAPE, 7, scale=0.02)
    path, cfg = gbfd.GBFD_OPT_KERNEL_PATH, gbfd.GBFD_OPT_TILE_CONFIG
    want, simple = _run(st, [], tmp_path / "unset.dot")
    assert simple
    for i, (options, expect) in enumerate([([(path, 0)], False), ([(path, 1)], True),
                                           ([(path, 1), (path, 0)], False),
                                           ([(cfg, 5)], False), ([(path, 1), (cfg, 5)], True)]):
        out, simple = _run(st, options, tmp_path / ("%d.dot" % i))
        assert simple == expect, options
        assert np.abs(out - want).max() < 1e-13
