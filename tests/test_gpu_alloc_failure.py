"""Failed device allocations (injected on the host, one at a time): the call
either reports ED_ERR_OOM or does without the memory, and the sector works as
if nothing had happened once memory is there again."""
import pytest
import torch

from workloads import make_model

pytestmark = pytest.mark.gpu

DT = {"fp32": torch.float32, "fp64": torch.float64}


def _vec(n, dt, seed=1):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand(n, device="cuda", dtype=dt, generator=g) - 0.5


def _failures(ed, call, most=40):
    """Runs `call(n)` (which makes its n-th allocation fail) for n = 1, 2, .. until
    one needs fewer allocations; returns the number of calls that met a failure."""
    for n in range(1, most):
        try:
            met = call(n)
        finally:
            ed.inject_alloc_failure(0)
        if not met:
            return n - 1
    raise AssertionError("a call allocates more than expected")


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("case", [(2, 6, 5, 4), (1, 11, 6, 5), (2, 3, 4, 4)])
def test_product_after_a_failed_allocation(ed, case, prec):
    """Every allocation of a sector's first block-major product fails once; the
    next product on the same sector gives w bit for bit."""
    norb, nbath, nup, ndw = case
    m = make_model(norb, nbath, U=2.0, Jh=0.3 * (norb > 1), seed=4)
    ref = ed.Sector(m, nup, ndw)
    v = torch.empty(ref.blocked_dim, device="cuda", dtype=DT[prec])
    ed.permute(ref, _vec(ref.dim, DT[prec]), v, True, prec)
    want = torch.zeros_like(v)
    ed.matvec_blocked(ref, v, want, prec)
    ref.free()

    def call(n):
        s = ed.Sector(m, nup, ndw)
        ed.inject_alloc_failure(n)
        failed = False
        try:
            ed.matvec_blocked(s, v, torch.zeros_like(v), prec)
        except ed.EDError as e:
            assert e.status == ed.ED_ERR_OOM
            failed = True
        ed.inject_alloc_failure(0)
        w = torch.zeros_like(v)
        ed.matvec_blocked(s, v, w, prec)
        assert torch.equal(w, want)
        s.free()
        return failed

    assert _failures(ed, call) >= 2


def test_sector_order_product_needs_only_its_own_list(ed):
    """A sector-order FP32 product that goes through block-major order (Norb=2 Ns=16) does
    without it where an allocation of that way fails: only the sector-order list itself,
    the first allocation, is needed.  Against the product with all memory there, both ways
    within FP32 rounding (2 eps per term of rows of at most 32 terms of size below 10 |v|
    with |v| <= 1/2)."""
    m = make_model(2, 7, U=3.0, Jh=0.5, seed=12)
    s = ed.Sector(m, 6, 6)
    v = _vec(s.dim, torch.float32)
    want = torch.empty_like(v)
    ed.matvec(s, v, want, "fp32")
    s.free()
    tol = 2 * 2.0 ** -24 * 32 * 5.0

    def call(n):
        s = ed.Sector(m, 6, 6)
        before = ed.kernel_launches()
        ed.inject_alloc_failure(n)
        w = torch.empty_like(v)
        if n == 1:
            with pytest.raises(ed.EDError) as e:
                ed.matvec(s, v, w, "fp32")
            assert e.value.status == ed.ED_ERR_OOM
        else:
            ed.matvec(s, v, w, "fp32")
            launches = ed.kernel_launches() - before
            assert float((w - want).abs().max()) <= tol
        ed.inject_alloc_failure(0)
        s.free()
        return n == 1 or launches == 1  # one launch: the sector-order kernel

    assert _failures(ed, call) >= 4
