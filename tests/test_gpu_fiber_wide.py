"""The wide CTA shape of the orbital-factorised FP32 product for groups of 4 and
5 levels (blocks of 5,000 and 7,776 columns), beside the narrow one in the same
sector: bit for bit the element-parallel product, see test_gpu_fiber.py."""
import pytest
import torch

from workloads import make_model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", [(4, 4, 7, 1), (4, 4, 7, 2), (5, 3, 10, 1)])
def test_wide_blocks(ed, case):
    norb, nbath, nup, ndw = case
    s = ed.Sector(make_model(norb, nbath, U=2.5, Jh=0.4, seed=sum(case)), nup, ndw)
    g = torch.Generator(device="cuda").manual_seed(7)
    v = torch.rand(s.dim, device="cuda", generator=g) * 2 - 1
    vb = torch.empty(s.blocked_dim, device="cuda")
    ed.permute(s, v, vb, True, "fp32")
    out, launches = {}, {}
    for kernel in ("tiled", "elementwise"):
        s.set_kernel(kernel, "fp32")
        wb = torch.full_like(vb, float("nan"))
        before = ed.kernel_launches()
        ed.matvec_blocked(s, vb, wb, "fp32")
        launches[kernel] = ed.kernel_launches() - before
        assert int(torch.isnan(wb).sum()) == s.blocked_dim - s.dim  # padding is not written
        out[kernel] = wb.nan_to_num()
    assert launches == {"tiled": 3, "elementwise": 1}  # both CTA shapes, then the H_dw pass
    assert torch.equal(out["tiled"], out["elementwise"])
    s.free()
