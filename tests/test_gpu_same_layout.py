"""Sector-order products of one-orbital sectors, whose vectors are block-major
vectors as they are: 16-byte aligned ones take the block-major kernels, others
the general path.  The same w bit for bit, for the electronic product and for
the electron-phonon product (whose phonon pass has 16-byte and element forms,
and launches all slices at once)."""
import pytest
import torch

from workloads import make_model

pytestmark = pytest.mark.gpu


def _vec(n, dt, off, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand(n, device="cuda", dtype=dt, generator=g) - 0.5
    y = torch.empty(n + off, device="cuda", dtype=dt)[off:]
    y.copy_(x)
    return y


@pytest.mark.parametrize("prec,dt", [("fp32", torch.float32), ("fp64", torch.float64)])
@pytest.mark.parametrize("nbath,nup,ndw", [(7, 3, 4), (11, 6, 5), (9, 5, 0)])
def test_matvec_aligned_and_offset_vectors(ed, nbath, nup, ndw, prec, dt):
    s = ed.Sector(make_model(1, nbath, U=2.0, seed=5), nup, ndw)
    w = [_vec(s.dim, dt, off, 2) for off in (0, 1)]
    for off in (0, 1):
        ed.matvec(s, _vec(s.dim, dt, off, 1), w[off], prec)
    assert torch.equal(w[0], w[1])
    s.free()


@pytest.mark.parametrize("prec,dt", [("fp32", torch.float32), ("fp64", torch.float64)])
@pytest.mark.parametrize("norb,nbath,nup,ndw,nph", [
    (1, 11, 6, 6, 10), (1, 7, 4, 3, 1), (1, 9, 5, 5, 0), (1, 8, 4, 5, 7), (2, 4, 5, 4, 3)])
def test_phonon_product_aligned_and_offset_vectors(ed, norb, nbath, nup, ndw, nph, prec, dt):
    s = ed.Sector(make_model(norb, nbath, U=2.0, Jh=0.1 * (norb - 1), seed=6), nup, ndw)
    ph = ed.phonon(0.5, [0.3] * norb, nph)
    n = s.dim * (nph + 1)
    w = [_vec(n, dt, off, 2) for off in (0, 1)]
    for off in (0, 1):
        ed.eph_matvec(s, ph, _vec(n, dt, off, 1), w[off], prec)
    assert torch.equal(w[0], w[1])
    s.free()


@pytest.mark.parametrize("norb,nbath,nup,ndw", [(2, 6, 5, 6), (3, 4, 5, 4)])
def test_sector_order_product_through_block_major_order(ed, norb, nbath, nup, ndw):
    """FP32 sector-order products of more than 2^20 elements on the tiled family
    go through block-major order: the same w as the three calls, bit for bit,
    also for vectors at an odd element; with the element-parallel kernel
    pinned, and under stream capture, the sector-order kernel gives the same w
    up to FP32 rounding (2 eps per term of rows of at most 30 terms of size
    below 10 |v| with |v| <= 1/2)."""
    s = ed.Sector(make_model(norb, nbath, U=3.0, Jh=0.5, seed=12), nup, ndw)
    v = _vec(s.dim, torch.float32, 0, 1)
    vb, wb = (torch.zeros(s.blocked_dim, device="cuda") for _ in range(2))
    want, w = torch.empty_like(v), torch.empty_like(v)
    s.set_kernel("tiled", "fp32")
    ed.permute(s, v, vb, True, "fp32")
    ed.matvec_blocked(s, vb, wb, "fp32")
    ed.permute(s, wb, want, False, "fp32")
    for off in (0, 1):
        w = torch.empty(s.dim + off, device="cuda")[off:]
        ed.matvec(s, _vec(s.dim, torch.float32, off, 1), w, "fp32")
        assert torch.equal(w, want)
    tol = 2 * 2.0 ** -24 * 30 * 5.0
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        ed.matvec(s, v, w, "fp32")
    w.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert float((w - want).abs().max()) <= tol
    s.set_kernel("elementwise", "fp32")
    ed.matvec(s, v, w, "fp32")
    assert float((w - want).abs().max()) <= tol
    s.free()
