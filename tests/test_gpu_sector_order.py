"""Which way a sector-order FP32 product of several orbitals takes (counted in
kernel launches: the sector-order kernel is one, the way through block-major
order has both permutations around the product's)."""
import pytest
import torch

from workloads import make_model

pytestmark = pytest.mark.gpu


def _vec(n, dt, seed=1):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand(n, device="cuda", dtype=dt, generator=g) - 0.5


def test_sector_order_product_below_the_crossover_stays_in_its_layout(ed):
    """Norb=2 Ns=14 (7,7): the sector-order kernel, one launch (no
    block-major lists, nothing timed); with the tiled family pinned, through block-major
    order."""
    s = ed.Sector(make_model(2, 6, U=3.0, Jh=0.5, seed=12), 7, 7)
    v = _vec(s.dim, torch.float32)
    w = torch.empty_like(v)
    before = ed.kernel_launches()
    ed.matvec(s, v, w, "fp32")
    assert ed.kernel_launches() - before == 1
    s.set_kernel("tiled", "fp32")
    before = ed.kernel_launches()
    ed.matvec(s, v, w, "fp32")
    assert ed.kernel_launches() - before >= 4
    s.free()


def test_first_call_through_block_major_order_times_nothing(ed):
    """Norb=2 Ns=16 (6,6): both permutations, the H_up pass (one launch: no block is
    wider than 4912 columns) and the H_dw pass, also on the shape's first call: no ELL
    table is built and no kernel is timed for it."""
    s = ed.Sector(make_model(2, 7, U=3.0, Jh=0.5, seed=12), 6, 6)
    v = _vec(s.dim, torch.float32)
    w = torch.empty_like(v)
    for _ in range(2):
        before = ed.kernel_launches()
        ed.matvec(s, v, w, "fp32")
        assert ed.kernel_launches() - before == 4
    s.free()
