"""Rows and columns of very different scale (weighted least squares, blocks of different units): FP64 Householder
transformations keep each row to its own scale, so fixed point relative to whole columns must not be used on them.

Tolerances: against an 80-bit run of the oracle on these inputs its FP64 run is off by at most 1.4e-12 of a row's or
column's norm of the band, and Q (Q^T C) - C by at most 5.7e-15 of a row's norm of C; seven and seventeen times that are
allowed for another order of summation.
"""
import numpy as np
import pytest

import paper_1611_06892_gb300 as G
from oracle import bidiag as OB
from paper_1611_06892_gb300 import inputs

pytestmark = pytest.mark.gpu
TOL_BAND, TOL_Q = 1e-11, 1e-13


@pytest.fixture(scope="module")
def handle():
    import torch  # noqa: F401
    h = G.Handle()
    yield h
    h.close()


def graded(m, n, kind, decades):
    A = inputs.gaussian(m, n, seed=m + n)
    if kind == "rows":
        A *= (10.0 ** (-decades * np.arange(m) / (m - 1)))[:, None]
    elif kind == "columns":
        A *= (10.0 ** (-decades * np.arange(n) / (n - 1)))[None, :]
    else:
        A *= np.where(np.arange(m) >= m // 3, 10.0 ** -decades, 1.0)[:, None]
    return np.asfortranarray(A)


def worst(D, R, axis):
    return (np.linalg.norm(D, axis=axis) / np.linalg.norm(R, axis=axis)).max()


SIZES = [(256, 256, 256, 32, "flatts", "rbidiag"), (600, 250, 256, 32, "flatts", "rbidiag"),
         (600, 250, 128, 32, "greedy", "rbidiag"), (600, 400, 128, 32, "greedy", "bidiag"),
         (500, 300, 64, 16, "flatts", "bidiag")]


@pytest.mark.parametrize("decades", [3, 8, 16])
@pytest.mark.parametrize("kind", ["rows", "columns", "blocks"])
@pytest.mark.parametrize("m,n,nb,ib,tree,variant", SIZES)
def test_band_keeps_each_rows_scale(handle, m, n, nb, ib, tree, variant, kind, decades):
    import torch
    A = graded(m, n, kind, decades)
    res = handle.band(torch.from_numpy(A).cuda(), nb, ib, tree, variant)
    handle.sync()
    B = OB.band_to_dense(res.band().cpu().numpy(), n)
    R = OB.band_to_dense(OB.bidiag_band(A, nb, ib, G.TREES[tree], G.VARIANTS[variant])["ab"], n)
    assert worst(B - R, R, 1) <= TOL_BAND
    assert worst(B - R, R, 0) <= TOL_BAND


@pytest.mark.parametrize("decades", [3, 8, 16])
@pytest.mark.parametrize("kind", ["rows", "blocks"])
@pytest.mark.parametrize("m,n,nb,ib,tree,variant", SIZES)
def test_back_transformation_keeps_each_rows_scale(handle, m, n, nb, ib, tree, variant, kind, decades):
    import torch
    A = graded(m, n, kind, decades)
    res = handle.band(torch.from_numpy(A).cuda(), nb, ib, tree, variant)
    C = np.asfortranarray(A[:, :40])
    Y = torch.from_numpy(C.copy(order="F")).cuda()
    res.apply_q(Y, 1)
    res.apply_q(Y, 0)
    handle.sync()
    assert worst(Y.cpu().numpy() - C, C, 1) <= TOL_Q


@pytest.mark.parametrize("kind", ["rows", "columns", "blocks"])
@pytest.mark.parametrize("nb,ib,tree,variant", [(64, 16, "greedy", "bidiag"), (128, 32, "flatts", "rbidiag")])
def test_same_rows_refused_without_published_blocks(handle, nb, ib, tree, variant, kind):
    """bidiag_band_noalloc reads V and T as stored, bidiag_band the published blocks: the same bits."""
    import ctypes

    import torch
    m, n = 400, 289                       # (a last strip of one column)
    A = torch.from_numpy(graded(m, n, kind, 8)).cuda()
    ref = handle.band(A, nb, ib, tree, variant).band()
    ab = torch.zeros((n, nb + 1), dtype=torch.float64, device="cuda").t()
    handle.sync()
    rc = G.bidiag_band_noalloc(m, n, ctypes.c_void_p(A.data_ptr()), m, nb, ib, G.TREES[tree], G.VARIANTS[variant],
                               ctypes.c_void_p(ab.data_ptr()), nb + 1, None)
    torch.cuda.synchronize()
    assert rc == G.OK
    assert torch.equal(ab, ref)
