"""GPU test of the state copies at the edges of their row groups (8, 16 and 32
lanes per row, one and two rows at once, aligned and unaligned buffers, all pairs
of types): a round trip keeps every bit, and the ghost columns and rows are the
periodic images (a step of a shifted state is the shifted step)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [(8, 9, nx) for nx in (8, 12, 28, 32, 36, 60, 64, 68, 124, 132, 200, 1024, 2048)]
SHAPES += [(50, 33, 72), (50, 32, 72), (64, 32, 68), (8, 8, 4096)]  # either side of the two-row rule


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_round_trip_and_ghosts(shape, precision):
    from paper_1707_08900_gb300 import build, gbfd
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    nz, ny, nx = shape
    rng = np.random.default_rng(nx + nz)
    st = 0.01 * rng.standard_normal((5,) + shape).astype(np.float32)
    s = gbfd.Solver(shape, lengths=(0.1 * nx, 0.1 * ny, 0.1 * nz), precision=precision, nu=1e-3)
    for dtype in (torch.float32, torch.float64):
        for off in (0, 1):
            def buf():
                b = torch.full((st.size + off,), float("nan"), device="cuda", dtype=dtype)
                return b[off:].view(st.shape)
            src, dst = buf(), buf()
            src.copy_(torch.from_numpy(st))
            s.set_state(src)
            s.get_state(out=dst)
            s.sync()
            assert np.array_equal(dst.cpu().numpy(), st.astype(dst.cpu().numpy().dtype))
            outs = []
            for roll in ((0, 0, 0), (3, 4, 5)):
                src.copy_(torch.from_numpy(np.roll(st, roll, axis=(1, 2, 3))))
                s.set_state(src)
                s.rk3_step(0.01, 1)
                s.sync()
                outs.append(np.roll(s.get_state(), [-r for r in roll], axis=(1, 2, 3)))
            assert np.array_equal(outs[0], outs[1])
            assert np.abs(outs[0] - st).max() > 1e-6
    s.close()
