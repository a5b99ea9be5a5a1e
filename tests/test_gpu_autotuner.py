"""The autotuner's choice holds for a model shape and a class of sizes."""
import pytest

from workloads import make_model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_timed_per_shape_and_size(ed, prec):
    """One orbital, twelve bath levels (no other test has this shape): the first sector of a
    size times both kernels, a second one of that size none; in FP32 a much larger sector
    times its own, in FP64 none."""
    m = make_model(1, 12, U=2.0, seed=8)
    timed = []
    for nup, ndw in ((3, 4), (4, 3), (7, 6), (6, 7)):  # 2.0e5, 2.0e5, 2.9e6, 2.9e6 elements
        s = ed.Sector(m, nup, ndw)
        kernel, ms = s.tune_info(prec)
        timed.append(min(ms.values()) > 0)
        if timed[-1]:
            assert (kernel == "elementwise") == (ms["elementwise"] < ms["tiled"])
        s.free()
    assert timed == [True, False, prec == "fp32", False]
