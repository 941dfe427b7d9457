"""GPU test of the autotuner's candidates: the built-in default is one of them (no
table entry runs its kernel or chunk length here), is kept when it is the
fastest, is cached, and can be selected by the reported index."""
import numpy as np
import pytest

from paper_1707_08900_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _gpu():
    from paper_1707_08900_gb300 import build
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    build.build()


def _step(s, st):
    s.set_state(st)
    s.rk3_step(0.005, 1)
    s.sync()
    return s.get_state(fp64=False)


# precision, side, table length: the default of each is at least 1.5 times as fast
# as any table entry (the update's FP64 operations; chunks of at least 8 planes)
@pytest.mark.parametrize("precision,n,count", [("fp32_acc64", 96, 35), ("fp64", 16, 30)])
def test_the_default_is_kept_when_it_is_fastest(precision, n, count, tmp_path):
    from paper_1707_08900_gb300 import gbfd
    _gpu()
    shape = (n,) * 3
    st = inputs.random_state(shape, 5, scale=0.02).astype(np.float32)
    path = str(tmp_path / "tune.json")
    out = []
    for tune in (False, True, True, None):
        s = gbfd.Solver(shape, precision=precision)
        s.set_state(st)
        if tune:
            cfg, ms = s.autotune(reps=20, cache_path=path)
            assert cfg == count
            assert (ms == 0.0) == (len(out) == 2)  # the second time from the cache
        elif tune is None:
            s.set_option(gbfd.GBFD_OPT_TILE_CONFIG, 1)
            s.set_option(gbfd.GBFD_OPT_TILE_CONFIG, count)
        out.append(_step(s, st))
        with pytest.raises(gbfd.GbfdError):
            s.set_option(gbfd.GBFD_OPT_TILE_CONFIG, count + 1)
        s.close()
    for o in out[1:]:
        assert np.array_equal(o, out[0])


def test_choices_of_another_table_are_not_taken(tmp_path):
    from paper_1707_08900_gb300 import gbfd
    _gpu()
    shape = (16, 16, 32)
    name = torch.cuda.get_device_name(0)
    path = tmp_path / "tune.json"
    path.write_text('{\n  "%s|32x16x16|precision1|form0|fields5": {"cfg": 3, "ms": 0.5}\n}\n' % name)
    s = gbfd.Solver(shape, precision="fp32")
    _, ms = s.autotune(reps=1, cache_path=str(path))
    assert ms > 0.0
    s.close()
