"""GPU test of the batch's default column routine when the caller sets the chunk
length alone: the lagged one for five fields with 64-plane items, else the
two-plane one; a routine that the caller set stays."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("entropy", [1, 0])
def test_default_routine_follows_the_chunk(entropy):
    from paper_1707_08900_gb300 import build, gbfd
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()
    Z, K = gbfd.GBFD_BATCH_OPT_ZCHUNK, gbfd.GBFD_BATCH_OPT_KERNEL
    b = gbfd.Batch([16, 24], [1.0, 1.0], [1e-3, 1e-3], entropy_mode=entropy)
    for zc in (64, 32, 16, 8, 64):
        b.set_option(Z, zc)
        assert (b.get_option(Z), b.get_option(K)) == (zc, 1 if zc == 64 and entropy else 0)
    b.set_option(K, 2)
    for zc in (8, 64):
        b.set_option(Z, zc)
        assert (b.get_option(Z), b.get_option(K)) == (zc, 2)
    b.close()
