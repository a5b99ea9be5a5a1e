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
    """Norb=2 Ns=14 (7,7): the sector-order kernel, one launch; with the
    tiled family pinned, through block-major order."""
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
