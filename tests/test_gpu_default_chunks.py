"""GPU test of the z-chunk length that the default kernels take from the grid:
chunks of one plane, of the whole column, with short and odd last chunks, give
the bits of the fixed 40-plane table entry of the same kernel (a chunk
boundary changes no point's arithmetic)."""
import numpy as np
import pytest

from paper_1707_08900_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision,entry", [("fp32", 20), ("fp64", 25), ("fp32_accff", 0)])
@pytest.mark.parametrize("shape", [(9, 8, 8), (16, 16, 16), (33, 40, 96), (48, 48, 48),
                                   (61, 72, 100), (200, 24, 32)])
def test_default_chunk_changes_no_bit(precision, entry, shape):
    from paper_1707_08900_gb300 import build, gbfd
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    nz, ny, nx = shape
    st = inputs.random_state(shape, 7, scale=0.02)
    outs = []
    for cfg in (-1, entry):
        s = gbfd.Solver(shape, lengths=(nx * 0.1, ny * 0.1, nz * 0.1), precision=precision, nu=5e-3)
        s.set_option(gbfd.GBFD_OPT_TILE_CONFIG, cfg)
        s.set_state(st)
        s.rk3_step(0.01, 2)
        s.sync()
        outs.append(s.get_state())
        s.close()
    assert np.all(np.isfinite(outs[0]))
    assert np.array_equal(outs[0], outs[1])
