"""All phonon slices of a coupled sector in one launch of the electronic
product: the kernel that serves it, and the factorised pass over slices."""
import pytest
import torch

from workloads import make_model

pytestmark = pytest.mark.gpu


def test_sliced_products_by_kernel(ed):
    """A two-orbital FP32 coupled ground state of 2^22 elements and more (71 slices of
    63,504 elements).  The element-parallel product is one launch, the orbital-factorised
    one two (one CTA shape, then the H_dw pass): a pinned kernel serves every product, no
    pin takes the tiled family; psi and E0 are the same bit for bit."""
    m = make_model(2, 4, U=2.0, Jh=0.3, seed=5)
    ph = ed.phonon(0.5, [0.1, 0.1], 70)
    out = {}
    for kernel in ("elementwise", "tiled", None):
        s = ed.Sector(m, 5, 5)
        if kernel:
            s.set_kernel(kernel, "fp32")
        psi = torch.zeros(s.dim * 71, device="cuda")
        ed.eph_lanczos_ground(s, ph, "fp32", tol=1e-3, psi=psi)  # every table exists
        before = ed.kernel_launches()
        r = ed.eph_lanczos_ground(s, ph, "fp32", tol=1e-3, psi=psi)
        out[kernel] = r, psi, ed.kernel_launches() - before
        s.free()
    products = out["tiled"][0]["matvecs"] - out["tiled"][0]["matvecs_fp64"]
    assert products > 4
    assert out["tiled"][2] - out["elementwise"][2] == products
    assert out[None][2] == out["tiled"][2]
    for kernel in ("tiled", None):
        assert out[kernel][0]["e0"] == out["elementwise"][0]["e0"]
        assert torch.equal(out[kernel][1], out["elementwise"][1])


def test_one_slice_follows_the_tuner(ed):
    """Cut-off 0 is one slice: the electronic product on the kernel the tuner chose or
    the caller pinned, whatever the number of elements (6.9e6)."""
    m = make_model(2, 6, U=2.0, Jh=0.3, seed=5)
    ph = ed.phonon(0.5, [0.1, 0.1], 0)
    s = ed.Sector(m, 7, 5)
    tuned = s.blocked_kernel("fp32")
    psi = torch.zeros(s.dim, device="cuda")
    ed.eph_lanczos_ground(s, ph, "fp32", tol=1e-3, psi=psi)
    n = {}
    for k in (None, "elementwise", "tiled"):
        if k:
            s.set_kernel(k, "fp32")
        before = ed.kernel_launches()
        ed.eph_lanczos_ground(s, ph, "fp32", tol=1e-3, psi=psi)
        n[k] = ed.kernel_launches() - before
    assert n["elementwise"] < n["tiled"]
    assert n[None] == n[tuned]
    s.free()
