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


@pytest.mark.parametrize("nph", [None, 3])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_one_orbital_product_needs_only_its_own_list(ed, prec, nph):
    """Sector-order vectors of one orbital that are block-major as they are (D_up = 924)
    take that layout's kernels; where an allocation for those fails the call runs on the
    sector-order list, its first allocation: the same w bit for bit.  nph: the coupled
    product."""
    m = make_model(1, 11, U=2.0, seed=4)
    ph = ed.phonon(0.5, [0.3], nph or 0)

    def product(s, v, w):
        if nph is None:
            ed.matvec(s, v, w, prec)
        else:
            ed.eph_matvec(s, ph, v, w, prec)

    s = ed.Sector(m, 6, 5)
    v = _vec(s.dim * ((nph or 0) + 1), DT[prec])
    want = torch.empty_like(v)
    product(s, v, want)
    # both lists exist now: vectors at an odd element allocate nothing
    off = [torch.empty(v.numel() + 1, device="cuda", dtype=DT[prec])[1:] for _ in range(2)]
    off[0].copy_(v)
    ed.inject_alloc_failure(1)
    product(s, off[0], off[1])
    ed.inject_alloc_failure(0)
    assert torch.equal(off[1], want)
    s.free()

    def call(n):
        s = ed.Sector(m, 6, 5)
        ed.inject_alloc_failure(n)
        w = torch.empty_like(v)
        if n == 1:
            with pytest.raises(ed.EDError) as e:
                product(s, v, w)
            assert e.value.status == ed.ED_ERR_OOM
        else:
            product(s, v, w)
            assert torch.equal(w, want)
        ed.inject_alloc_failure(0)
        s.free()

    for n in range(1, 10):
        call(n)


def test_one_orbital_product_under_capture(ed):
    """Captured before the block-major tables exist (an earlier call on vectors at an odd
    element built the sector-order list): nothing is built under capture, and the replayed
    product is the same w bit for bit."""
    s = ed.Sector(make_model(1, 11, U=2.0, seed=4), 6, 5)
    x = _vec(s.dim + 1, torch.float32)
    v, w = x[:-1], torch.empty(s.dim, device="cuda")
    off = torch.empty(s.dim + 1, device="cuda")[1:]
    y = torch.empty(s.dim + 1, device="cuda")[1:]
    off.copy_(v)
    ed.matvec(s, off, y, "fp32")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        ed.inject_alloc_failure(1)
        ed.matvec(s, v, w, "fp32")
        ed.inject_alloc_failure(0)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(w, y)
    s.free()


def test_unknown_precision_builds_nothing(ed):
    """Refused before the first allocation, as an argument error."""
    s = ed.Sector(make_model(1, 11, U=2.0, seed=4), 6, 5)
    v, w = _vec(s.dim, torch.float64), torch.empty(s.dim, device="cuda", dtype=torch.float64)
    ed.inject_alloc_failure(1)
    for product in (lambda: ed.matvec(s, v, w, 7),
                    lambda: ed.eph_matvec(s, ed.phonon(0.5, [0.3], 0), v, w, 7)):
        with pytest.raises(ed.EDError) as e:
            product()
        assert e.value.status == ed.ED_ERR_ARG
    ed.inject_alloc_failure(0)
    s.free()
