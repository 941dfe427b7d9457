"""GPU test of gbfd_cfl_dt's own reduction: the largest |u| must be the full
diagnostics' value bit for bit, whatever the FP32 look ahead of it sees."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision,bc", [("fp32", "periodic"), ("fp32", "wall"),
                                          ("fp64", "periodic")])
@pytest.mark.parametrize("kind", ["random", "smooth", "close", "zero", "tiny", "huge", "nan"])
def test_cfl_dt_uses_the_diagnostics_maximum(precision, bc, kind):
    from paper_1707_08900_gb300 import build, gbfd
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    shape = (13, 22, 36)
    rng = np.random.default_rng(3)
    st = np.zeros((5,) + shape)
    if kind == "random":
        st[1:4] = rng.standard_normal((3,) + shape)
    elif kind == "smooth":  # the maximum grows along the scan
        st[1:4] = np.linspace(0.1, 1.0, st[1].size).reshape(shape)
    elif kind == "close":  # values one FP32 ulp apart, equal in FP32 |u|^2
        st[1:4] = np.float32(0.7) + rng.integers(0, 3, (3,) + shape) * 2.0 ** -24
    elif kind == "tiny":
        st[1:4] = 1e-25 * rng.standard_normal((3,) + shape)
    elif kind == "huge":  # |u|^2 leaves the FP32 range
        st[1:4] = 1e25 * rng.standard_normal((3,) + shape)
    elif kind == "nan":
        st[1:4] = rng.standard_normal((3,) + shape)
        st[2, 3, 4, 5] = np.nan
        st[3, 0, 0, 0] = -np.inf
    s = gbfd.Solver(shape, precision=precision, nu=0.0, cs=0.5, bc_z=bc)
    s.set_state(st if precision == "fp64" else st.astype(np.float32))
    umax = s.diagnostics()["umax"]
    nz, ny, nx = shape
    h = min(2 * np.pi / nx, 2 * np.pi / ny, 2 * np.pi / (nz - (bc == "wall")))
    assert s.cfl_dt(0.4) == 0.4 * h / (umax + 0.5)
    s.close()
