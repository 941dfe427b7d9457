"""GPU test of a launch that CUDA refuses (more chunks along z than a grid may have):
the call reports it, and the calls after it do not."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision,entry", [("fp32", 24), ("fp64", 29)])  # 8-plane chunks
def test_refused_launch_leaves_no_error_behind(precision, entry):
    from paper_1707_08900_gb300 import build, gbfd
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    shape = (8 * 65535 + 8, 8, 8)
    s = gbfd.Solver(shape, lengths=(1.0, 1.0, 1.0 * shape[0] / 8), precision=precision, nu=0.0,
                    entropy_mode=0)
    s.set_option(gbfd.GBFD_OPT_TILE_CONFIG, entry)
    with pytest.raises(gbfd.GbfdError):
        s.rk3_step(1e-3, 1)
    s.set_option(gbfd.GBFD_OPT_TILE_CONFIG, -1)
    s.rk3_step(1e-3, 1)
    s.sync()
    d = s.diagnostics()  # its launches ask CUDA for the last error
    assert not d["nonfinite"] and d["umax"] == 0.0
    assert float(torch.ones(4, device="cuda").sum()) == 4.0
    s.close()
