"""GPU test of tile table entries that no default runs: the FP64 and FP64-update
forms with explicit entries (every kernel, 40- and 8-plane chunks), 55- and
19-point, unforced, forced and between walls, one step against the oracle."""
import numpy as np
import pytest

from bars import FP32_TOL, FP64_TOL, rel_l2
from oracle import fd
from paper_1707_08900_gb300 import inputs
from test_gpu_walls import wall_state

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

VARIANTS = {"fp64": 6, "fp32_acc64": 3, "fp32_acc64_w64": 3}
SHAPE = (20, 44, 36)


@pytest.mark.parametrize("what", ["plain", "forced", "wall"])
@pytest.mark.parametrize("form", ["55p", "19p"])
@pytest.mark.parametrize("precision", sorted(VARIANTS))
def test_explicit_entries(precision, form, what):
    from paper_1707_08900_gb300 import build, gbfd
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    nz, ny, nx = SHAPE
    lengths = (3.0, 4.5, 2.5)
    g = fd.Grid(nx, ny, nz, *lengths)
    ph = fd.Physics(cs=1.0, nu=0.02, entropy_mode=1)
    fm = fd.FORM_55P if form == "55p" else fd.FORM_19P
    wall = what == "wall"
    st = wall_state(SHAPE, 4, amp=0.1) if wall else inputs.spectrum(SHAPE, 21, mach=0.2, lnrho_rms=1e-2)
    if precision != "fp64":
        st = st.astype(np.float32).astype(np.float64)
    dt = (fd.cfl_dt_wall if wall else fd.cfl_dt)(st, g, ph, 0.4)
    forcing = inputs.forcing_sequence(11, 1, kmin=1.0, kmax=3.0)
    if wall:
        ref = fd.rk3_step_wall(st, dt, g, ph, fm)
    elif what == "forced":
        ref = fd.rk3_step_forced(st, dt, g, ph, 0.2, *forcing, form=fm)
    else:
        ref = fd.rk3_step(st, dt, g, ph, fm)
    tol = FP64_TOL if precision == "fp64" else FP32_TOL
    for v in range(VARIANTS[precision]):
        for zi in (0, 4):
            s = gbfd.Solver(SHAPE, lengths=lengths, nu=0.02, precision=precision, form=form,
                            bc_z="wall" if wall else "periodic")
            s.set_option(gbfd.GBFD_OPT_TILE_CONFIG, 5 * v + zi)
            s.set_state(st)
            if what == "forced":
                s.rk3_step_forced(dt, 0.2, *forcing)
            else:
                s.rk3_step(dt, 1)
            got = s.get_state()
            s.close()
            assert np.all(rel_l2(got, ref) <= tol), (v, zi, rel_l2(got, ref))
