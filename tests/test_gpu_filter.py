"""GPU test of the box filter's float-float kernel (ratios 2, 4, 8) and the
general one (6) against the FP64 oracle: periodic wraps on every side, coarse
rows shorter and longer than a warp, a constant, and non-finite values."""
import numpy as np
import pytest

from oracle import fd
from paper_1707_08900_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,r", [(8, 2), (8, 8), (12, 4), (24, 6), (48, 8), (72, 2), (136, 4)])
def test_box_filter_ratios(n, r):
    from paper_1707_08900_gb300 import build, gbfd
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    st = inputs.random_state((n, n, n), 5).astype(np.float32)
    st[4] = np.float32(1.0 / 3.0)
    s = gbfd.Solver((n, n, n), precision="fp32")
    s.set_state(st)
    got = gbfd.box_filter(s, r).cpu().numpy()
    ref = fd.box_filter(st.astype(np.float64), r)
    # one FP32 rounding of a sum known to 46 bits of its largest terms (|st| < 1)
    assert np.abs(got - ref).max() <= 2.0 ** -24 * np.abs(ref).max() + (r + 1) ** 3 * 2.0 ** -46
    assert np.array_equal(got[4], np.full_like(got[4], np.float32(1.0 / 3.0)))
    st[0, 0, 0, 0] = np.inf
    st[1, 1, 1, 1] = np.nan
    s.set_state(st)
    got = gbfd.box_filter(s, r).cpu().numpy()
    assert got[0, 0, 0, 0] == np.inf and np.isnan(got[1]).any()
    assert np.isfinite(got[2:]).all()
    s.close()
