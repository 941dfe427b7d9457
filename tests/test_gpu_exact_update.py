"""GPU test of the FP64-update precision form's default kernel, whose update runs
in float-float arithmetic with every result checked to be the FP64 one."""
import numpy as np
import pytest

from bars import FP32_TOL, TERM_NU, inc_bar, inc_err, rel_l2, term_exposing_state
from oracle import fd
from paper_1707_08900_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _run(precision, st, shape, lengths, dt, entropy, cfg=-1):
    from paper_1707_08900_gb300 import gbfd
    s = gbfd.Solver(shape, lengths=lengths, precision=precision, nu=TERM_NU, entropy_mode=entropy)
    s.set_option(gbfd.GBFD_OPT_TILE_CONFIG, cfg)
    s.set_state(st.astype(np.float32))
    s.rk3_step(dt, 1)
    s.sync()
    out = s.get_state(fp64=False)
    s.close()
    return out


@pytest.mark.parametrize("shape,even,entropy", [((24, 32, 64), True, 1), ((19, 21, 36), False, 1),
                                                ((9, 8, 8), True, 0), ((40, 24, 100), False, 0)])
def test_exact_update_matches_oracle_and_float_float(shape, even, entropy):
    """One step within the FP32 bars of the oracle, and the float-float form's
    result (the same right-hand sides) except where a value of 48 and one of
    53 bits round differently: below 1e-3 of the values, two ulps of the
    field's magnitude (the bars of the simple kernels' comparison)."""
    from paper_1707_08900_gb300 import build
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    nz, ny, nx = shape
    lengths = (nx * 0.2, ny * 0.2, nz * 0.2) if even else (2 * np.pi,) * 3
    st = term_exposing_state(shape, 3, inputs)[:4 + entropy]
    g = fd.Grid(nx, ny, nz, *lengths)
    ph = fd.Physics(cs=1.0, nu=TERM_NU, entropy_mode=entropy)
    dt = fd.cfl_dt(st, g, ph, 0.4)
    ref = fd.rk3_step(st, dt, g, ph)
    a = _run("fp32_acc64", st, shape, lengths, dt, entropy)
    assert np.all(rel_l2(a, ref) <= FP32_TOL)
    assert np.all(inc_err(a, ref, st) <= inc_bar(ref, st))
    b = _run("fp32_accff", st, shape, lengths, dt, entropy)
    scale = np.array([np.spacing(np.float32(np.abs(x).max())) for x in a], dtype=np.float64)
    d = np.abs(a.astype(np.float64) - b.astype(np.float64)).reshape(a.shape[0], -1).max(axis=1)
    assert (a != b).mean() < 1e-3
    assert np.all(d <= 2.0 * scale)


def test_exact_update_keeps_extreme_values():
    """Zeros, subnormals, ties and values near the FP32 limits on a field whose
    right-hand side vanishes (the velocity is zero, so the passive scalar does
    not move): every value comes back as it went in."""
    from paper_1707_08900_gb300 import build
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    shape = (12, 16, 32)
    st = np.zeros((5,) + shape, dtype=np.float32)
    special = np.array([0.0, 1e-40, -3e-39, 1.1754944e-38, 1.0e37, -1.0e37, 1e-30,
                        1.0 + 2.0 ** -23, -(1.0 + 2.0 ** -22), 7.0], dtype=np.float32)
    st[4] = np.resize(special, shape[0] * shape[1] * shape[2]).reshape(shape)
    out = _run("fp32_acc64", st, shape, (2 * np.pi,) * 3, 1e-3, 1)
    assert np.array_equal(out, st)
