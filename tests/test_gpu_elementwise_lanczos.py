"""Lanczos on the element-parallel product over the sizes where its form changes:
a CTA takes several chunks of 256 elements above 2^21 elements in the Lanczos
mode, and FP32 sectors take four rows per thread above 2^22."""
import pytest

from workloads import make_model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nup,ndw", [(4, 5), (4, 6), (5, 6)])
@pytest.mark.parametrize("prec,tol", [("fp32", 1e-6), ("fp64", 1e-10)])
def test_ground_state_by_kernel(ed, nup, ndw, prec, tol):
    """Two orbitals, Ns=14: D = 2,004,002 (one chunk), 3,006,003 (chunks), 6,012,006 (rows
    in FP32).  Each kernel's E0 against FP64 on the other family: FP64 converges to 1e-10,
    raw FP32 carries the rounding of its products (2^-24 of |H| a few times |E0|)."""
    m = make_model(2, 6, U=2.0, Jh=0.2, seed=3)
    ref = ed.Sector(m, nup, ndw)
    ref.set_kernel("tiled", "fp64")
    e0 = ed.lanczos_ground(ref, "fp64")["e0"]
    ref.free()
    s = ed.Sector(m, nup, ndw)
    s.set_kernel("elementwise", prec)
    r = ed.lanczos_ground(s, prec)
    assert abs(r["e0"] - e0) <= tol * abs(e0)
    s.free()
