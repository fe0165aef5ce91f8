"""Sweeps shared by several thread blocks, repeated: the blocks pass solved rows and
partial sums through slots that are cleared and filled again every few links, so a
value lost between a clear and a fill would show as a timeout or another result.
All sums run in a fixed order: the results are the same bits."""
import numpy as np
import pytest

from gpu_helpers import run_gpu
from test_gpu_sweeps import _problem

pytestmark = pytest.mark.gpu


# eight boxes: clusters of eight, four and two thread blocks by half width; one box
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nel,parts,overlap", [((26, 23, 22), (2, 2, 2), 2), ((18, 16, 15), (2, 2, 2), 1),
                                               ((64, 62), (2, 2), 1), ((60, 30, 6), (1, 1, 1), 0)])
def test_repeated_sweeps_give_the_same_bits(nel, parts, overlap, precision):
    import torch
    prob = _problem(nel, parts, overlap)
    sol, _ = run_gpu(prob, nev_max=0, precision=precision)
    try:
        rng = np.random.default_rng(8)
        r = torch.from_numpy(rng.standard_normal(prob.n)).cuda()
        b = torch.from_numpy(rng.standard_normal((3, prob.n))).cuda()
        first = None
        for _ in range(60):
            z, x = torch.full_like(r, 7.0), torch.full_like(b, 7.0)
            sol.apply(r, z)
            sol.solve(b, x, tol=1e-14, maxit=2, nrhs=3, raise_on_error=False)
            if first is None:
                first = (z.clone(), x.clone())
            assert torch.equal(z, first[0]) and torch.equal(x, first[1])
        from paper_1906_10944_gb300 import geneo as G
        assert G.geneo_last_error(sol.h)[0] == 0
    finally:
        sol.close()
