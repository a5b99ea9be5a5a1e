"""The orbital-factorised FP32 product (two and more orbitals, groups of 2 to
8 levels): every group size, both CTA shapes, blocks of one column, empty and
full spins, items that end inside a dw block.  Bit for bit against the
element-parallel product, which takes the same operations per element in the
same order and is checked against the oracle in test_gpu_matvec.py."""
import pytest
import torch

from workloads import make_model

pytestmark = pytest.mark.gpu

CASES = [  # norb, nbath, nup, ndw
    (2, 1, 2, 2), (3, 1, 3, 2), (5, 1, 4, 5),    # G = 2
    (2, 2, 3, 0), (5, 2, 3, 4), (4, 2, 5, 3),    # G = 3
    (4, 3, 4, 2), (2, 3, 8, 3),                  # G = 4, a full up string
    (2, 4, 5, 3), (3, 4, 6, 2),                  # G = 5
    (2, 5, 6, 4), (3, 5, 5, 2),                  # G = 6
    (3, 5, 9, 1),                                # G = 6, blocks of 8000 columns
    (2, 6, 7, 2), (3, 6, 4, 1),                  # G = 7
    (2, 7, 8, 2), (2, 7, 3, 4),                  # G = 8
]


@pytest.mark.parametrize("case", CASES)
def test_orbital_factorised_product(ed, case):
    norb, nbath, nup, ndw = case
    m = make_model(norb, nbath, U=2.5, Jh=0.4, seed=sum(case))
    s = ed.Sector(m, nup, ndw)
    g = torch.Generator(device="cuda").manual_seed(7)
    v = torch.rand(s.dim, device="cuda", generator=g) * 2 - 1
    vb = torch.empty(s.blocked_dim, device="cuda")
    ed.permute(s, v, vb, True, "fp32")
    out = {}
    for kernel in ("tiled", "elementwise"):
        s.set_kernel(kernel, "fp32")
        wb = torch.full_like(vb, float("nan"))
        ed.matvec_blocked(s, vb, wb, "fp32")
        assert int(torch.isnan(wb).sum()) == s.blocked_dim - s.dim  # padding is not written
        out[kernel] = wb.nan_to_num()
    assert torch.equal(out["tiled"], out["elementwise"])
    s.free()
