"""The sweeps of several right-hand sides, and the routes of very wide bands.

A solve of several right-hand sides stopped after one iteration returns, column by
column, x = alpha M^{-1} b with alpha = b.z / z.Az, z = M^{-1} b.  So its direction
is one multi-column apply, compared here with the oracle's apply of every column,
and b.x = x.Ax holds to rounding.  One level (no coarse space): the local solves
are all of M^{-1}.

Tolerances (of the direction, relative): FP64 1e-10 (banded against sparse LU, as
in the parity tests); FP32 factors 16 u kappa, u = 2^-24 and kappa the largest
condition number of the equilibrated A_j (the factorisation and the sweeps perturb
A_j by a small multiple of u, the three TF32 passes of a product by 3 * 2^-22 =
12 u); FP64 factors in double-single arithmetic 4 * 2^-44 kappa + 1e-10.  b.x and
x.Ax: 1e-10 (two FP64 sums of at most 10^5 terms).
"""
import functools

import numpy as np
import pytest

import gen
import oracle
from gpu_helpers import run_gpu
from test_gpu_sweeps import GEOMETRIES, _kappa, _problem

pytestmark = pytest.mark.gpu

# Boxes cut along x at the given element indices, overlap 1: half widths 461, 281
# and 281, which share a size class and its thread blocks per matrix; then 2538 (8
# rows per block in FP32, the streamed kernel in FP64) and 4801 (the streamed
# kernel in FP32 as well)
MIXED = ((50, 20, 13), (0, 23, 36, 50))
WIDE = ((118, 43, 4), (0, 59, 118))
WIDEST = ((120, 80, 3), (0, 60, 120))


@functools.lru_cache(maxsize=2)
def _setup(geometry):
    nel, second = geometry[0], geometry[1]
    if len(geometry) == 3:
        prob = _problem(*geometry)
    else:
        k = gen.kappa_grf_layers_3d(nel, seed=4, corr_len=0.2, variance=1.0, contrast=1e2,
                                    slab_z=(30, 80), slab_thickness=1)
        cores = [((a, 0, 0), (b, nel[1], nel[2])) for a, b in zip(second[:-1], second[1:])]
        prob = gen.darcy_problem(nel, k, None, None, cores=cores, overlaps=[1] * len(cores))
    orc = oracle.GenEOOracle(prob, oracle.OracleOptions(nev_max=0))
    return prob, orc, _kappa(orc, prob)


OPTIONS = {"fp64": {"precision": 0}, "fp32": {"precision": 1}, "ds": {"precision": 1, "fp32_pivot_tol": 0.99}}


def _tol(kind, kappa):
    return {"fp64": 1e-10, "fp32": 16 * 2.0 ** -24 * kappa, "ds": 4 * 2.0 ** -44 * kappa + 1e-10}[kind]


def _half_widths(prob, orc):
    out = []
    for st in orc.sets:
        a = prob.A[st["D"]][:, st["D"]].tocoo()
        out.append(int(np.abs(a.row - a.col)[a.data != 0].max()))
    return out


def _check_columns(geometry, kind, counts):
    import torch
    prob, orc, kappa = _setup(geometry)
    tol = _tol(kind, kappa)
    sol, _ = run_gpu(prob, nev_max=0, **OPTIONS[kind])
    try:
        assert sol.query()["fp64_factors_A"] == (prob.n_sub if kind == "ds" else 0)
        B = np.random.default_rng(5).standard_normal((max(counts), prob.n))
        Z = np.stack([orc.apply(r) for r in B])
        for nrhs in counts:
            b = torch.from_numpy(B[:nrhs].copy()).cuda()
            x = torch.zeros_like(b)
            info = sol.solve(b, x, tol=1e-14, maxit=1, nrhs=nrhs, raise_on_error=False)
            assert info["iterations"] == 1 and info["status"] == 5
            X = x.cpu().numpy()
            for c in range(nrhs):
                s = X[c] @ Z[c] / (Z[c] @ Z[c])
                err = np.linalg.norm(X[c] - s * Z[c]) / np.linalg.norm(X[c])
                assert err <= tol, (nrhs, c, err, tol)
                bx, xax = B[c] @ X[c], X[c] @ (prob.A @ X[c])
                assert abs(bx - xax) <= 1e-10 * abs(bx), (nrhs, c, bx, xax)
    finally:
        sol.close()


@pytest.mark.parametrize("kind", ["fp64", "fp32", "ds"])
@pytest.mark.parametrize("geometry", GEOMETRIES + [MIXED, WIDE], ids=str)
def test_one_iteration_of_several_columns(geometry, kind):
    _check_columns(geometry, kind, (2, 3, 4, 5, 8))


def test_one_iteration_of_several_columns_widest():
    _check_columns(WIDEST, "fp32", (2, 3, 8))


def test_mixed_widths_share_a_class():
    """The narrow boxes lie further left of their band than the mbarriers and the
    padding before the row slots are long (512 bytes) when eight thread blocks of 64
    rows share a matrix: what the class of MIXED is for."""
    prob, orc, _ = _setup(MIXED)
    w = _half_widths(prob, orc)
    assert max(w) >= 449 and 0.6 * max(w) <= min(w) < 7 * 64 - 128, w


@pytest.mark.parametrize("geometry,kind", [(MIXED, "fp64"), (MIXED, "fp32"), (WIDE, "fp64"), (WIDE, "fp32"),
                                           (WIDEST, "fp32")], ids=str)
def test_one_level_apply_of_wide_and_mixed_bands(geometry, kind):
    import torch
    prob, orc, kappa = _setup(geometry)
    sol, _ = run_gpu(prob, nev_max=0, **OPTIONS[kind])
    try:
        r = np.random.default_rng(6).standard_normal(prob.n)
        z = torch.zeros(prob.n, dtype=torch.float64, device="cuda")
        sol.apply(torch.from_numpy(r).cuda(), z)
        zo = orc.apply(r)
        assert np.linalg.norm(z.cpu().numpy() - zo) <= _tol(kind, kappa) * np.linalg.norm(zo)
    finally:
        sol.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_block_solve_iterations_as_alone(precision):
    """A column takes as many iterations in a block as alone (within two: sums in
    another order)."""
    import torch
    prob = _problem((50, 45), (4, 3), 1)
    sol, _ = run_gpu(prob, nev_max=4, precision=precision)
    try:
        B = np.random.default_rng(3).standard_normal((4, prob.n))
        for c in range(4):
            order = [(c + 1 + i) % 4 for i in range(4)]   # column c last: the one reported
            b = torch.from_numpy(B[order].copy()).cuda()
            its = sol.solve(b, torch.zeros_like(b), tol=1e-8, nrhs=4)["iterations"]
            one = torch.from_numpy(B[c].copy()).cuda()
            alone = sol.solve(one, torch.zeros_like(one), tol=1e-8)["iterations"]
            assert abs(its - alone) <= 2, (c, its, alone)
    finally:
        sol.close()


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("kind", ["fp64", "fp32"])
def test_apply_with_a_value_that_is_not_finite(kind, value):
    """Values of the solved rows are their own arrival flags, and the flag's pattern
    is a NaN: an input that is not finite spreads over the subdomains that hold it,
    stalls no wait and leaves the others as they are."""
    import torch
    prob, orc, kappa = _setup(MIXED)
    sol, _ = run_gpu(prob, nev_max=0, **OPTIONS[kind])
    try:
        r = np.random.default_rng(7).standard_normal(prob.n)
        only = np.setdiff1d(orc.sets[0]["D"], np.concatenate([s["D"] for s in orc.sets[1:]]))
        zo = orc.apply(r)
        r[only[only.size // 2]] = value
        z = torch.zeros(prob.n, dtype=torch.float64, device="cuda")
        sol.apply(torch.from_numpy(r).cuda(), z)
        z = z.cpu().numpy()
        clean = np.setdiff1d(np.arange(prob.n), orc.sets[0]["D"])
        assert np.all(np.isfinite(z[clean])) and not np.all(np.isfinite(z[only]))
        assert np.linalg.norm(z[clean] - zo[clean]) <= _tol(kind, kappa) * np.linalg.norm(zo)
        b = torch.from_numpy(np.stack([prob.b, prob.b])).cuda()
        sol.solve(b, torch.zeros_like(b), tol=1e-6, nrhs=2)   # no timeout on record
    finally:
        sol.close()
