"""GPU test of the training loss over the range of FP32 residuals: squares that
overflow, vanish or lose bits in FP32 are summed in FP64."""
import numpy as np
import pytest

from oracle import cnn as ocnn

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# 2560 squares, exact in FP64, added there (2560 x 2^-53 = 2.8e-13) or first in
# float-float by 20 (2^-45 each)
TOL = 1e-12


@pytest.mark.parametrize("scales", [(1.0, 1.0), (1e25, 1e25), (1e30, 1.0), (3e18, 2.5e19), (1e-25, 1e-25),
                                    (1e-12, 3e-17), (1e-18, 1e-20), (1.0, 1e-30), (0.0, 0.0)])
def test_loss_of_residuals_of_any_size(scales):
    from paper_1707_08900_gb300 import build, gbfd
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    n = 8
    p = {k: np.zeros_like(v) for k, v in ocnn.init_params(1).items()}  # the prediction is zero
    rng = np.random.default_rng(3)
    t = rng.standard_normal((1, 5, n, n, n))
    t[:, :, : n // 2] *= scales[0]
    t[:, :, n // 2:] *= scales[1]
    t = t.astype(np.float32)
    net = gbfd.CNN(n, batch=1)
    net.set_params(p)
    net.set_norm(np.zeros(5), np.ones(5), np.ones(5))
    ts = torch.from_numpy(t).cuda()
    _, loss = net.gradients(torch.zeros_like(ts), ts)
    net.close()
    want = float((t.astype(np.float64) ** 2).sum() / t.size)
    assert np.isfinite(loss)
    assert abs(loss - want) <= TOL * want, (loss, want)
