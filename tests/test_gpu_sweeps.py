"""Edges of the band sweeps, the batched factorisations, the block PCG kernels
and the restriction, through the public entry points against the oracle.

The block height of a sweep depends on the half bandwidth (15, 31 and 63 are its
thresholds), the thread blocks per matrix on the number of subdomains, the
columns per block on the right-hand sides, the restriction on the number of
subdomains (304).  Tolerances: FP64 one-level applies 1e-10 relative (banded
against sparse LU, as in the parity tests); one-level applies with FP32 factors
4 u kappa relative, u = 2^-24 and kappa the largest condition number of the
equilibrated A_j (a Cholesky factorisation and two triangular solves perturb A_j
by a small multiple of u); two-level applies 1e-6 (coarse vectors of an iterative
eigensolve at residual 1e-9); solves: the true residual at tol, evaluated again
here (1.01 tol).
"""
import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spla

import gen
import oracle
from gpu_helpers import run_gpu

pytestmark = pytest.mark.gpu

# (elements, parts, overlap): local half bandwidths about 5, 12, 16, 33, 64, 68, 90
# and 190, orders with every kind of remainder, 2 to 144 subdomains; the last two,
# flat boxes of half bandwidth about 930 and 1840, take the 16- and 8-row blocks of
# FP64 and the 32- and 16-row blocks of FP32
GEOMETRIES = [
    ((12, 10), (4, 3), 1),
    ((96, 90), (12, 12), 1),
    ((50, 45), (4, 3), 1),
    ((64, 62), (2, 2), 1),
    ((61, 124), (1, 2), 1),
    ((134, 66), (2, 1), 1),
    ((18, 16, 15), (2, 2, 2), 1),
    ((26, 23, 22), (2, 2, 2), 2),
    ((60, 30, 6), (2, 1, 1), 1),
    ((90, 40, 5), (2, 1, 1), 1),
]


def _problem(nel, parts, overlap, contrast=1e2):
    if len(nel) == 2:
        k = gen.kappa_channels_2d(nel, seed=2, contrast=contrast)
    else:
        k = gen.kappa_grf_layers_3d(nel, seed=4, corr_len=0.2, variance=1.0, contrast=contrast,
                                    slab_z=(30, 80), slab_thickness=1)
    return gen.darcy_problem(nel, k, parts, overlap)


def _kappa(orc, prob):
    """Largest condition number of the equilibrated local matrices."""
    worst = 1.0
    for st in orc.sets:
        a = prob.A[st["D"]][:, st["D"]].tocsc()
        d = sp.diags(1.0 / np.sqrt(a.diagonal()))
        a = (d @ a @ d).tocsc()
        v = np.random.default_rng(0).standard_normal(a.shape[0])
        big = spla.eigsh(a, k=1, which="LA", v0=v, return_eigenvectors=False, tol=1e-2)[0]
        small = spla.eigsh(a, k=1, sigma=0.0, which="LM", v0=v, return_eigenvectors=False, tol=1e-2)[0]
        worst = max(worst, big / small)
    return worst


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nel,parts,overlap", GEOMETRIES)
def test_one_level_apply(nel, parts, overlap, precision):
    import torch
    prob = _problem(nel, parts, overlap)
    orc = oracle.GenEOOracle(prob, oracle.OracleOptions(nev_max=0))
    tol = 1e-10 if precision == 0 else 4 * 2.0 ** -24 * _kappa(orc, prob)
    sol, _ = run_gpu(prob, nev_max=0, precision=precision)
    try:
        rng = np.random.default_rng(1)
        for _ in range(2):
            r = rng.standard_normal(prob.n)
            z = torch.zeros(prob.n, dtype=torch.float64, device="cuda")
            sol.apply(torch.from_numpy(r).cuda(), z)
            zo = orc.apply(r)
            assert np.linalg.norm(z.cpu().numpy() - zo) <= tol * np.linalg.norm(zo)
    finally:
        sol.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nrhs", [2, 3, 4, 5, 8])
def test_block_solve_columns(nrhs, precision):
    import torch
    prob = _problem((50, 45), (4, 3), 1)
    sol, _ = run_gpu(prob, nev_max=4, precision=precision)
    try:
        B = np.random.default_rng(3).standard_normal((nrhs, prob.n))
        b = torch.from_numpy(B).cuda()
        x = torch.zeros_like(b)
        sol.solve(b, x, tol=1e-8, maxit=2000, nrhs=nrhs)
        X = x.cpu().numpy()
        for c in range(nrhs):
            assert np.linalg.norm(B[c] - prob.A @ X[c]) <= 1.01e-8 * np.linalg.norm(B[c]), c
    finally:
        sol.close()


@pytest.mark.parametrize("parts", [(18, 16), (18, 17)])
def test_restriction_below_and_above_304_subdomains(parts):
    import torch
    prob = _problem((54, 51), parts, 1)
    orc = oracle.GenEOOracle(prob, oracle.OracleOptions(nev_max=3))
    sol, _ = run_gpu(prob, nev_max=3, eig_tol=1e-9)
    try:
        r = np.random.default_rng(2).standard_normal(prob.n)
        z = torch.zeros(prob.n, dtype=torch.float64, device="cuda")
        sol.apply(torch.from_numpy(r).cuda(), z)
        zo = orc.apply(r)
        assert np.linalg.norm(z.cpu().numpy() - zo) <= 1e-6 * np.linalg.norm(zo)
    finally:
        sol.close()
