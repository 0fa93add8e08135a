"""The FP64 LU by itself: pivots, factors, error bounds.  Graded matrices: rows of L that rise over a panel's
columns while the columns of U fall by as much.  The digit-split update loses relative to a row's and a
column's largest entry, which such products do not reach; FP64 arithmetic relative to the products
themselves.  Bound: Gaussian elimination computes |P A - L U| <= g |L||U| entrywise, g a complex product's
and its sum's roundings, (n + 3) 2 sqrt(2) eps with eps = 2^-53 (Higham, Accuracy and Stability of
Numerical Algorithms, ch. 3 and 9).  The residual is formed with 64-bit mantissas or more.  The
factorisation is called below the C entry points, which take meshes."""
import ctypes
import re
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _factor_device(sol, d, info=None):
    """(LU, pivots) of d [batch][n][n], which LU overwrites"""
    import torch
    from paper_1706_07919_gb300 import binding as B

    lib = B.load()
    names = subprocess.run(["nm", "-D", "--defined-only", lib._name], capture_output=True, text=True, check=True).stdout
    f = getattr(lib, re.search(r"\sT\s(_ZN3bie11lu_factor64\S+)", names).group(1))
    f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_int64,
                  ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]
    nb, n, _ = d.shape
    piv = torch.zeros((nb, n), dtype=torch.int32, device="cuda:0")
    info = torch.zeros(nb, dtype=torch.int32, device="cuda:0") if info is None else info
    err = torch.zeros(1, dtype=torch.int32, device="cuda:0")
    torch.cuda.synchronize()
    assert f(sol.ctx, d.data_ptr(), nb, n, n, n * n, piv.data_ptr(), info.data_ptr(), err.data_ptr()) == B.BIE_OK
    torch.cuda.synchronize()
    assert int(err) == 0
    return d, piv


def _factor(sol, A):
    """(LU, row order, zero-pivot words) of A [batch][n][n]"""
    import torch

    nb, n, _ = A.shape
    info = torch.zeros(nb, dtype=torch.int32, device="cuda:0")
    LU, piv = _factor_device(sol, torch.tensor(A, device="cuda:0").contiguous(), info)
    order = np.tile(np.arange(n), (nb, 1))
    for z, p in enumerate(piv.cpu().numpy()):
        for c in range(n):
            order[z, [c, p[c]]] = order[z, [p[c], c]]
    return LU.cpu().numpy(), order, info.cpu().numpy()


def _check(A, LU, order, cols=None):
    """the residual of the first `cols` columns (all) against its bound"""
    n = len(A)
    cols = n if cols is None else cols
    wide = np.clongdouble
    L, U = (np.tril(LU, -1) + np.eye(n))[:, :cols], np.triu(LU)[:cols, :cols]
    bound = (n + 3) * 2 * np.sqrt(2.0) * 2.0 ** -53 * (np.abs(L) @ np.abs(U))
    res = np.abs(A[order][:, :cols].astype(wide) - L.astype(wide) @ U.astype(wide)).astype(float)
    assert np.all(res <= bound), np.max(res / bound)


@pytest.mark.parametrize("n", [193, 320])
@pytest.mark.parametrize("grading", [0, 10, 30, 60])
def test_graded_rows(n, grading):
    from paper_1706_07919_gb300 import Solver

    rng = np.random.default_rng(100 * n + grading)
    A = rng.standard_normal((2, n, n)) + 1j * rng.standard_normal((2, n, n)) + 8 * np.eye(n)
    d = 2.0 ** (-grading * np.minimum(np.arange(n), 63) / 63.0)
    A[0] *= d[:, None]                                   # the panel's pivots fall
    A[1] *= rng.permutation(d)[:, None] * rng.permutation(2.0 ** (rng.uniform(-40, 40, n)))[None, :]
    sol = Solver(0)
    LU, order, info = _factor(sol, A)
    assert not info.any()
    for z in range(2):
        _check(A[z], LU[z], order[z])
    sol.close()


def test_entries_that_are_not_finite():
    """A NaN spreads as it does in an elimination of the rows in their final order; the columns before it,
    zero and subnormal-scale rows and columns factor."""
    from paper_1706_07919_gb300 import Solver

    n = 320
    rng = np.random.default_rng(5)
    A = rng.standard_normal((3, n, n)) + 1j * rng.standard_normal((3, n, n)) + 8 * np.eye(n)
    A[0, 300, 100] = np.nan
    A[1, 70:90, :64] = 0.0
    A[1, :64, 200:210] = 0.0
    A[2, :, 250] *= 2.0 ** -1030
    sol = Solver(0)
    LU, order, _ = _factor(sol, A)
    ref = A[0][order[0]].copy()
    with np.errstate(invalid="ignore"):
        for c in range(n):
            ref[c + 1:, c] /= ref[c, c]
            ref[c + 1:, c + 1:] -= np.outer(ref[c + 1:, c], ref[c, c + 1:])
    assert np.array_equal(np.isnan(LU[0]), np.isnan(ref))
    lu0 = LU[0].copy()
    lu0[:, 100:] = 0.0
    _check(A[0], lu0, order[0], 100)
    _check(A[1], LU[1], order[1])
    cols = np.arange(n) != 250  # (its own products are below the normal numbers)
    assert np.isfinite(LU[2]).all()
    L, U = np.tril(LU[2], -1) + np.eye(n), np.triu(LU[2])
    res = np.abs(A[2][order[2]] - L @ U)[:, cols]
    assert np.all(res <= 2 * (n + 3) * 2 * np.sqrt(2.0) * 2.0 ** -53 * (np.abs(L) @ np.abs(U))[:, cols])
    sol.close()


def test_pivots_are_the_largest_entries():
    """Entries of a column that differ by 1e-9: the pivot is the largest one, wherever it lies."""
    from paper_1706_07919_gb300 import Solver

    n = 700
    rng = np.random.default_rng(11)
    A = 1e-3 * (rng.standard_normal((2, n, n)) + 1j * rng.standard_normal((2, n, n)))
    for z in range(2):
        A[z, :, 0] = (1 + 1e-9 * rng.permutation(n)) * np.exp(2j * np.pi * rng.uniform(size=n))
    sol = Solver(0)
    LU, order, info = _factor(sol, A)
    assert not info.any()
    for z in range(2):
        assert order[z][0] == np.argmax(np.abs(A[z, :, 0]))
        assert np.max(np.abs(np.tril(LU[z], -1))) <= 1 + 4 * 2.0 ** -53
    sol.close()


@pytest.mark.parametrize("n", [1030, 1480])
def test_factor_does_not_depend_on_the_cluster(n):
    """The systems of a batch (which decide the CTAs of a cluster: 16 to 2, sizes between the powers of two
    among them) have one system's factor, bit for bit; a cluster of few CTAs gives a thread several rows."""
    import torch
    from paper_1706_07919_gb300 import Solver

    sol = Solver(0)
    torch.manual_seed(n)
    A = torch.randn((64, n, n), dtype=torch.complex128, device="cuda:0")
    A[:, torch.arange(n), torch.arange(n)] += 8
    one = {}
    for batch in (1, 3, 10, 14, 20, 28, 40, 64):
        LU, piv = _factor_device(sol, A[:batch].clone())
        for z in range(batch):
            if z not in one:
                one[z] = (LU[z].clone(), piv[z].clone()) if batch == 1 else tuple(t[0] for t in _factor_device(sol, A[z:z + 1].clone()))
            assert torch.equal(piv[z], one[z][1]) and torch.equal(torch.view_as_real(LU[z]), torch.view_as_real(one[z][0]))
    sol.close()
