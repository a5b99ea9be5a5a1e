"""The batched chains of small solves (one cluster of CTAs per chain) against
the graph-driven chain of the same ground state: sectors of a few elements
(most CTAs of the cluster hold none), odd sizes, the largest sector the batch
takes (16,128 padded elements: 160 KB of shared memory in FP64), spin exchange
and pair hopping.

FP64; tolerance: the bound of G against the oracle, 1e-8, which both paths
satisfy on their own."""
import numpy as np
import pytest
import torch

from workloads import make_model, with_exchange

pytestmark = pytest.mark.gpu

CASES = [(1, 1, 1, 1), (1, 2, 1, 2), (2, 1, 2, 2), (1, 5, 3, 2), (2, 2, 3, 3), (3, 1, 3, 2),
         (1, 8, 4, 4)]


@pytest.mark.parametrize("exchange", [False, True])
@pytest.mark.parametrize("case", CASES)
def test_cluster_chains_against_graph_chains(ed, case, exchange):
    norb, nbath, nup, ndw = case
    if exchange and norb == 1:
        pytest.skip("one orbital has no exchange terms")
    m = make_model(norb, nbath, U=2.0, Jh=0.3 * (norb > 1), seed=sum(case))
    if exchange:
        m = with_exchange(m)
    before = ed.batch_stats()["chains"]
    s = ed.Sector(m, nup, ndw)
    psi = torch.empty(s.dim, dtype=torch.float64, device="cuda")
    res, G = ed.solve(m, nup, ndw, precision="fp64", psi=psi, nmats=32, beta=20.0, gf_steps=60)
    assert ed.batch_stats()["chains"] > before
    for orb in range(norb):
        g, _ = ed.gf_lanczos(s, psi, res["e0"], orb, 0, "fp64", nsteps=60, beta=20.0, nmats=32)
        assert np.abs(G[0, orb] - g).max() <= 1e-8
    s.free()
