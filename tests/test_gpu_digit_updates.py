"""FP64 block updates as digit products on tcgen05 (nb x ib >= 1024, ib <= 32, multiples of 8) against the FP64
oracle, at the sizes where they can go wrong: tiles below, at and above one 128-row half, inner blocks of 8, 16
and 32 reflectors, ragged edges, both orientations, and columns of very different or extreme scale.

Tolerance: the parity tests' 1e-12 ||A||_F.  Scaling the input by a power of two only shifts exponents, so in
range it must scale the band exactly.
"""
import numpy as np
import pytest

import paper_1611_06892_gb300 as G
from oracle import bidiag as OB
from oracle import trees as T
from paper_1611_06892_gb300 import inputs

pytestmark = pytest.mark.gpu
TOL = 1e-12
TREES = {"flatts": T.FLATTS, "greedy": T.GREEDY}


@pytest.fixture(scope="module")
def handle():
    import torch  # noqa: F401
    h = G.Handle()
    h.set_option(G.OPT_TRACE, 1)
    yield h
    h.close()


def band(handle, A, nb, ib, tree, variant):
    import torch
    res = handle.band(torch.from_numpy(np.asfortranarray(A)).cuda(), nb, ib, tree, variant)
    handle.sync()
    return res


def on_tensor_cores(handle):
    return int(((handle.trace()[:, 3] >> 32) & 1).sum())


@pytest.mark.parametrize("m,n,nb,ib", [(150, 130, 64, 16), (150, 97, 64, 32), (300, 200, 96, 32), (260, 257, 128, 8),
                                       (400, 290, 128, 32), (330, 170, 136, 8), (500, 330, 160, 32),
                                       (600, 400, 256, 32), (513, 300, 256, 16)])
@pytest.mark.parametrize("tree,variant", [("greedy", "bidiag"), ("flatts", "rbidiag")])
def test_against_oracle(handle, m, n, nb, ib, tree, variant):
    import torch
    A = inputs.gaussian(m, n, seed=m + n)
    A *= 2.0 ** (np.arange(n) % 40 - 20)[None, :]          # columns over twelve decades
    A[:, n // 3] = 0.0
    res = band(handle, A, nb, ib, tree, variant)
    assert on_tensor_cores(handle) > 0
    ref = OB.bidiag_band(A, nb, ib, TREES[tree], G.VARIANTS[variant])
    assert np.abs(res.band().cpu().numpy() - ref["ab"]).max() <= TOL * np.linalg.norm(A)
    X = torch.from_numpy(np.asfortranarray(inputs.gaussian(m, 7, seed=3))).cuda()
    Y = X.clone()
    res.apply_q(Y, 0)
    res.apply_q(Y, 1)           # (the columns span 1e12: Q itself is not comparable entry by entry)
    handle.sync()
    assert torch.linalg.norm(Y - X).item() <= TOL * torch.linalg.norm(X).item()
    res.free()


@pytest.mark.parametrize("shift", [-900, -600, 300, 900])
def test_scaling_by_powers_of_two(handle, shift):
    A = inputs.gaussian(300, 200, seed=8)
    b0 = band(handle, A, 96, 32, "greedy", "bidiag").band().cpu().numpy()
    b1 = band(handle, np.ldexp(A, shift), 96, 32, "greedy", "bidiag").band().cpu().numpy()
    if abs(shift) <= 300:       # beyond, squared norms of the panel factor leave the range of FP64
        assert np.array_equal(np.ldexp(b0, shift), b1)
    assert b1.shape == b0.shape


@pytest.mark.parametrize("bad", [np.inf, np.nan, 1e308])
def test_values_out_of_range_take_the_fp64_units(handle, bad):
    A = inputs.gaussian(300, 200, seed=9)
    A[250, 150] = bad
    ab = band(handle, A, 96, 32, "greedy", "bidiag").band().cpu().numpy()
    assert not np.isfinite(ab).all()
    A[250, 150] = 0.0           # the handle goes on
    ref = OB.bidiag_band(A, 96, 32, T.GREEDY, T.BIDIAG)
    ab = band(handle, A, 96, 32, "greedy", "bidiag").band().cpu().numpy()
    assert np.abs(ab - ref["ab"]).max() <= TOL * np.linalg.norm(A)


@pytest.mark.parametrize("dtype", ["float64", "float32"])
def test_batch_with_odd_tiles_beside(handle, dtype):
    """Tiles whose sizes leave the next matrix's storage unaligned (nb 7, 9, 33) beside ones that take the tensor-core
    paths: each result is bitwise that of the matrix alone."""
    import torch
    cfg = [(7, 7), (96, 32), (9, 3), (64, 32), (33, 11), (128, 32), (64, 16)]
    As = [torch.from_numpy(np.asfortranarray(inputs.gaussian(90 + 41 * i, 61 + 29 * i, seed=i)).astype(dtype, order="F")).cuda()
          for i in range(len(cfg))]
    res = handle.band_batched(As, [c[0] for c in cfg], [c[1] for c in cfg], ["greedy"] * 7, ["bidiag"] * 7)
    handle.sync()
    for A, (nb, ib), r in zip(As, cfg, res):
        single = handle.band(A, nb, ib, "greedy", "bidiag")
        handle.sync()
        assert torch.equal(r.band(), single.band()), (nb, ib)
