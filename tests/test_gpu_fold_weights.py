"""GPU test of the folded weights of the batch's lagged routine: on boxes with a mean
flow they must not add a multiple of it (the second-derivative weights cancel on a
constant), for time steps where rounding the centre weight alone leaves most."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

N, NU, STEPS = 32, 0.19, 10
U = (0.7, -0.9, 0.6)


def _left_over(dt, h):
    """Centre + arms when each weight is rounded by itself."""
    d2 = np.array([1.5, -0.15, 1.0 / 90.0])
    v = (dt * NU * d2 / h ** 2).astype(np.float32).astype(float)
    x = (dt * NU * 4.0 / 3.0 * d2 / h ** 2).astype(np.float32).astype(float)
    s = 2.0 * (x + 2.0 * v).sum()
    return abs(float(np.float32(-s)) + s)


def test_second_derivative_weights_cancel_on_a_mean_flow():
    from paper_1707_08900_gb300 import build, gbfd
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    length = 2 * np.pi
    rng = np.random.default_rng(5)
    st = 0.01 * rng.standard_normal((5, N, N, N))
    for i in range(3):
        st[1 + i] += U[i]
    st = st.astype(np.float32).astype(np.float64)
    dts = sorted(np.linspace(0.012, 0.02, 200), key=lambda d: -_left_over(d, length / N))[:2]
    b = gbfd.Batch([N], [length], [NU])
    b.set_option(gbfd.GBFD_BATCH_OPT_KERNEL, 1)
    for dt in dts:
        assert _left_over(dt, length / N) > 2e-8
        s = gbfd.Solver((N,) * 3, lengths=(length,) * 3, precision="fp64", nu=NU)
        s.set_state(st)
        s.rk3_step(dt, STEPS)
        s.sync()
        want = s.get_state(fp64=True)
        s.close()
        b.set_state(0, st)
        b.step([dt], STEPS)
        b.sync()
        d = np.asarray(b.get_state(0), dtype=np.float64) - want
        # rounding errors of either sign average out over the points; a left-over of
        # 2e-8 would be 2e-7 of the mean flow after ten steps
        assert max(abs(d[1 + i].mean() / U[i]) for i in range(3)) < 5e-8, dt
    b.close()
