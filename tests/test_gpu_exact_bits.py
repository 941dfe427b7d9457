"""GPU test of the FP64-update precision form's bits, through two runs whose FP64
updates are the same up to a power of two.

A shear flow u_x(y) without pressure and viscosity moves only lnrho and s, at
the rate u_x d/dx.  With u_x scaled by 2^110 and the time step by 2^-110 every
product dt x rhs is the same number, so the FP64 update gives the same lnrho and
s; but that time step has no exact float-float form, so there every value
takes the FP64 update, where the unscaled run takes it for the few values that
float-float arithmetic might round differently."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SCALE = 2.0 ** 110


def _run(precision, shape, entropy, st, dt, steps):
    from paper_1707_08900_gb300 import gbfd
    nz, ny, nx = shape
    s = gbfd.Solver(shape, lengths=(0.3 * nx, 0.3 * ny, 0.3 * nz), cs=0.0, nu=0.0,
                    precision=precision, entropy_mode=entropy)
    s.set_state(st)
    s.rk3_step(dt, steps)
    s.sync()
    out = s.get_state(fp64=False)
    s.close()
    return out


@pytest.mark.parametrize("shape,entropy,steps", [((128, 128, 128), 1, 10), ((33, 21, 36), 1, 3),
                                                 ((9, 8, 8), 0, 3), ((125, 131, 132), 0, 2)])
def test_update_has_the_fp64_bits(shape, entropy, steps):
    from paper_1707_08900_gb300 import build
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    nz, ny, nx = shape
    rng = np.random.default_rng(nx)
    st = np.zeros((4 + entropy,) + shape, dtype=np.float32)
    st[0] = rng.standard_normal(shape)
    st[1] = rng.standard_normal(ny)[None, :, None]
    if entropy:
        st[4] = rng.standard_normal(shape)
    big = st.copy()
    big[1] *= np.float32(SCALE)
    assert np.all(np.isfinite(big))
    dt = 0.0123
    a = _run("fp32_acc64", shape, entropy, st, dt, steps)
    b = _run("fp32_acc64", shape, entropy, big, dt / SCALE, steps)
    assert np.array_equal(b[1], big[1]) and np.array_equal(a[1], st[1])
    moved = [0] + ([4] if entropy else [])
    for f in moved:
        assert np.abs(a[f] - st[f]).max() > 1e-3
        assert np.array_equal(a[f], b[f]), f
    if shape == (128, 128, 128):  # large enough for float-float to round otherwise
        c = _run("fp32_accff", shape, entropy, st, dt, steps)
        assert any((a[f] != c[f]).any() for f in moved)
