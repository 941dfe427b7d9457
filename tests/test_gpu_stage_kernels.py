"""GPU test of the FP32 default kernel's instantiations per RK3 substep, which
large grids (2^21 points and more) run: on whole and on ragged tiles, four and
five fields, equal and unequal spacings, they give the bits of the kernel that
takes the substep at run time and keeps its pending values in registers."""
import numpy as np
import pytest

from paper_1707_08900_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _step(gbfd, shape, lengths, nf, st, cfg, forced):
    s = gbfd.Solver(shape, lengths=lengths, precision="fp32", nu=5e-3, entropy_mode=nf - 4)
    s.set_option(gbfd.GBFD_OPT_TILE_CONFIG, cfg)
    s.set_state(st)
    if forced:  # a zero force: the forced instantiations, the unforced result
        s.rk3_step_forced(0.005, 0.0, [[1, 1, 0]], [0.3], [[0.0, 0.0, 1.0]])
    else:
        s.rk3_step(0.005, 1)
    s.sync()
    out = s.get_state(fp64=False)
    s.close()
    return out


@pytest.mark.parametrize("nf", [5, 4])
@pytest.mark.parametrize("even", [True, False])
@pytest.mark.parametrize("shape", [(128, 128, 128), (125, 131, 132)])
def test_stage_kernels_match_the_general_one(shape, even, nf):
    from paper_1707_08900_gb300 import build, gbfd
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    nz, ny, nx = shape
    assert nx * ny * nz >= 2 ** 21
    lengths = (nx * 0.05, ny * 0.05, nz * 0.05) if even else (6.0, 5.0, 4.5)
    st = inputs.random_state(shape, 11, scale=0.02, nfields=nf).astype(np.float32)
    want = _step(gbfd, shape, lengths, nf, st, 10, False)
    assert np.all(np.isfinite(want))
    for forced in (False, True):
        assert np.array_equal(_step(gbfd, shape, lengths, nf, st, -1, forced), want), forced
