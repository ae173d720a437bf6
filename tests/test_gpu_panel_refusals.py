"""Panel factors from Gram matrices at their limits of refusal: just inside they run on the tensor cores, just outside
the block is factored column by column and published from there; either way the reduction matches the FP64 oracle and
Q stays orthogonal.  Also inner blocks of 24 reflectors, which no power of two covers.

Tolerance: the parity tests' 1e-12 ||A||_F.  The inputs are conditioned to about 1e4 at worst, so the band is determined
to a few 1e-12 / 1e4 of that.
"""
import numpy as np
import pytest

import paper_1611_06892_gb300 as G
from oracle import bidiag as OB
from paper_1611_06892_gb300 import inputs

pytestmark = pytest.mark.gpu
TOL = 1e-12
PF = 7


@pytest.fixture(scope="module")
def handle():
    import torch  # noqa: F401
    h = G.Handle()
    h.set_option(G.OPT_TRACE, 1)
    yield h
    h.close()


def check(handle, A, nb, ib, tree, variant):
    """Reduces A, compares with the oracle; {(kind, block): number of factors not on the tensor cores}."""
    import torch
    m, n = A.shape
    res = handle.band(torch.from_numpy(np.asfortranarray(A)).cuda(), nb, ib, tree, variant)
    handle.sync()
    ref = OB.bidiag_band(A, nb, ib, G.TREES[tree], G.VARIANTS[variant])
    assert np.abs(res.band().cpu().numpy() - ref["ab"]).max() <= TOL * np.linalg.norm(A)
    off = {}
    for op, fl in zip(handle.trace_program()[0][:, 0], handle.trace()[:, 3]):
        if int(op) & 15 == PF and not (int(fl) >> 32) & 1:
            key = (("GE", "TS", "TT")[int(op) >> 24 & 3], int(op) >> 16 & 255)
            off[key] = off.get(key, 0) + 1
    X = torch.from_numpy(np.asfortranarray(inputs.gaussian(m, 5, seed=3))).cuda()
    Y = X.clone()
    res.apply_q(Y, 1)
    handle.sync()
    assert abs(torch.linalg.norm(Y).item() / torch.linalg.norm(X).item() - 1.0) <= TOL
    res.apply_q(Y, 0)
    handle.sync()
    assert torch.linalg.norm(Y - X).item() <= TOL * torch.linalg.norm(X).item()
    return off


def correlated(A, d):            # column 37 keeps d of its norm under the reflectors before it
    A[:, 37] = A[:, 36] + d * A[:, 37]


def large_entry(A, k):           # no short tail: the 37 reflectors before spread it over the column
    A[37, 37] = k * np.sqrt(A.shape[0])


def short_tail(A, k):            # column 0's pivot is k times its tail
    A[0, 0] = k * np.sqrt(A.shape[0])


def zero_column(A, _):
    A[:, 37] = 0.0


def weak_row(A, s):              # a row of every tile s times the others
    A[50::128, :] *= s


# (a column's scale is a power of two 1.03 to 2.06 times its norm: the limits are hit within a factor of two)
@pytest.mark.parametrize("change,arg,refused", [
    (correlated, 0.5, False), (correlated, 0.04, True), (large_entry, 2.0 ** 5, False), (large_entry, 2.0 ** 12, False),
    (short_tail, 2.0 ** 4, False), (short_tail, 2.0 ** 12, True), (zero_column, 0.0, True), (weak_row, 2.0 ** -1, False), (weak_row, 2.0 ** -9, True)])
@pytest.mark.parametrize("tree", ["flatts", "flattt"])
def test_at_the_limits(handle, change, arg, refused, tree):
    A = inputs.gaussian(384, 128, seed=12)
    change(A, arg)
    off = check(handle, A, 128, 32, tree, "rbidiag")
    ge = 1 if tree == "flatts" else 3          # GE panels; their last, square block is always column by column
    assert off.pop(("GE", 3)) == ge
    off.pop(("TT", 3), None)                   # (its last row has one entry, small by chance)
    if not refused:
        assert not off
    else:
        blk = 0 if change is short_tail else 1
        assert off.get(("GE", blk)) == (1 if change is short_tail else ge)      # (its tile alone has the large pivot)
        if tree == "flatts":
            assert off.get(("TS", blk)) == 2


@pytest.mark.parametrize("change,arg", [(correlated, 0.04), (short_tail, 2.0 ** 12), (large_entry, 2.0 ** 12), (weak_row, 2.0 ** -9)])
@pytest.mark.parametrize("tree,variant", [("greedy", "bidiag"), ("flatts", "rbidiag")])
def test_refused_blocks_are_published(handle, change, arg, tree, variant):
    A = inputs.gaussian(420, 300, seed=13)
    change(A, arg)
    assert check(handle, A, 128, 32, tree, variant)


@pytest.mark.parametrize("nb", [48, 72, 96, 144, 192, 240])
@pytest.mark.parametrize("tree,variant", [("greedy", "bidiag"), ("flatts", "rbidiag")])
def test_inner_blocks_of_24(handle, nb, tree, variant):
    off = check(handle, inputs.gaussian(2 * nb + 53, nb + 61, seed=nb), nb, 24, tree, variant)
    assert sum(off.values()) < sum(int(op) & 15 == PF for op in handle.trace_program()[0][:, 0])
