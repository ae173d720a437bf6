"""Measured cases of the band bidiagonalization: what a program that uses this package has it do.

A case is one of four kinds:

  band     B = Q^T A P of one matrix (``Handle.band``), the band copied out
  batch    many small uneven matrices in one call (``Handle.band_batched``)
  grad     band and dL/dA through torch's autograd (``autograd.band_bidiag``), forward and backward
  vectors  singular-vector back-transformation with a reduction made before: Q C and D P^T
           (``Result.apply_q`` / ``Result.apply_p``)

Options of a case: ``dtype`` (f64 / f32 storage), ``m``, ``n``, tile size ``nb``, inner blocking ``ib``,
reduction ``tree``, ``variant`` (bidiag / rbidiag / auto) and the ``input``: i.i.d. N(0, 1), or U diag(s) V^T
with singular values falling geometrically from 1 to 1e-8.  A program keeps one handle per GPU.
"""
import math

import numpy as np
import torch

import paper_1611_06892_gb300 as G
from paper_1611_06892_gb300.autograd import band_bidiag

_handle = None


def _get_handle():
    global _handle
    if _handle is None:
        _handle = G.Handle()
    return _handle


# ---- the cases -----------------------------------------------------------------------------------

def _band(name, m, n, nb, ib, tree, variant="bidiag", dtype="f64", data="gauss"):
    c = dict(kind="band", m=m, n=n, nb=nb, ib=ib, tree=tree, variant=variant, dtype=dtype, input=data)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call, a matrix of a few tiles: launches, queue latency and the panel chain
        _band("tiny-192x160", 192, 160, 32, 8, "greedy"),
        # one small dense matrix
        _band("square-512", 512, 512, 64, 16, "flatts"),
        # sizes that no tile divides, as a caller with arbitrary data has it
        _band("ragged-3001x1537", 3001, 1537, 192, 32, "greedy"),
        # a middle-sized square matrix with a decaying spectrum, as in an SVD
        _band("square-4096", 4096, 4096, 256, 32, "auto", data="geometric"),
        # the headline size
        _band("square-8192", 8192, 8192, 256, 32, "auto"),
        # tall and skinny, through the preliminary QR: least squares, PCA
        _band("tall-65536x1024", 65536, 1024, 256, 32, "auto", "rbidiag"),
        # the single-precision forms of the last two
        _band("f32-square-8192", 8192, 8192, 256, 32, "auto", dtype="f32"),
        _band("f32-tall-65536x1024", 65536, 1024, 256, 32, "auto", "rbidiag", dtype="f32"),
        # a batch of small uneven matrices, its configuration left to the autotuner
        dict(name="batch-64", kind="batch", count=64, m=1024, nb=0, ib=0, tree="", dtype="f64"),
        # a single-precision batch with one configuration for all
        dict(name="f32-batch-64", kind="batch", count=64, m=1024, nb=128, ib=32, tree="flatts", dtype="f32"),
        # differentiation: a spectral loss on a layer's matrix, forward and backward
        dict(name="grad-4096x1024", kind="grad", m=4096, n=1024, nb=256, ib=32, tree="greedy", variant="bidiag",
             dtype="f64", input="gauss"),
        # left and right singular vectors of B taken back to those of A
        dict(name="vectors-4096x2048", kind="vectors", m=4096, n=2048, cols=128, nb=256, ib=32, tree="auto",
             variant="bidiag", dtype="f64", input="gauss"),
    ]


_BLOCKINGS = [(32, 8), (32, 16), (64, 16), (64, 32), (96, 32), (128, 16), (128, 32), (160, 32), (192, 32), (256, 32)]
_MAX_FLOPS = 2.0e11     # a drawn case stays well under the largest listed one


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_shape(rng, kind):
    top_m, top_n = {"band": (65536, 8192), "grad": (8192, 2048), "vectors": (16384, 4096)}[kind]
    while True:
        n = _log_int(rng, 96, top_n)
        m = _log_int(rng, n, max(n, min(top_m, 64 * n)))
        if _flops(m, n) > _MAX_FLOPS / (4 if kind == "grad" else 1):
            continue
        # tiles as callers size them: up to 24 tile columns, 256 tile rows, no tile wider than the matrix
        fit = [b for b in _BLOCKINGS if b[0] <= n and -(-n // b[0]) <= 24 and -(-m // b[0]) <= 256]
        if fit:
            return (m, n) + rng.choice(fit)


def draw(rng):
    kind = rng.choice(["band"] * 5 + ["batch", "grad", "vectors"])
    dtype = rng.choice(["f64", "f64", "f32"])
    if kind == "batch":
        tuned = rng.random() < 0.5
        nb, ib = (0, 0) if tuned else rng.choice([(32, 16), (64, 32), (128, 32)])
        return dict(kind="batch", count=rng.randint(8, 64), m=_log_int(rng, 128, 1024), nb=nb, ib=ib,
                    tree="" if tuned else rng.choice(["flatts", "greedy", "auto"]), dtype=dtype)
    m, n, nb, ib = _draw_shape(rng, kind)
    tree = rng.choice(["auto", "auto", "greedy", "flatts", "flattt"])
    variant = rng.choice(["bidiag", "auto"] if m < 2 * n else ["bidiag", "auto", "rbidiag"])
    if kind == "band":
        # (in single precision a spectrum of eight decades is below the roundings)
        data = "geometric" if dtype == "f64" and n <= 2048 and rng.random() < 0.25 else "gauss"
        return _band("", m, n, nb, ib, tree, variant, dtype, data)
    c = dict(kind=kind, m=m, n=n, nb=nb, ib=ib, tree=tree, variant="bidiag" if kind == "grad" else variant,
             dtype=dtype, input="gauss")
    if kind == "vectors":
        c["cols"] = rng.choice([1, 32, 100, 256])
    return c


# ---- inputs --------------------------------------------------------------------------------------

def _dtype(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _randn(rows, cols, seed, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(cols, rows, dtype=torch.float64, device="cuda", generator=g).to(dtype).t()   # column-major


def _matrix(case, seed):
    m, n, dt = case["m"], case["n"], _dtype(case)
    if case.get("input", "gauss") == "gauss":
        return _randn(m, n, 1000 * seed + 1, dt)
    U = torch.linalg.qr(_randn(m, n, 1000 * seed + 1, torch.float64))[0]
    V = torch.linalg.qr(_randn(n, n, 1000 * seed + 2, torch.float64))[0]
    s = 10.0 ** (-8.0 * torch.arange(n, dtype=torch.float64, device="cuda") / max(1, n - 1))
    return (V @ (U * s).t()).to(dt).t()


def _batch_shapes(case, seed):
    """m uniform in [64, case m], n uniform in [32, m]; the shapes belong to the case, not to the seed, as in
    a program that reduces batches of the same layers again and again."""
    rng = np.random.default_rng(6)
    ms = rng.integers(64, case["m"] + 1, case["count"])
    return [(int(m), int(rng.integers(32, m + 1))) for m in ms]


def _batch(case, seed):
    return [_randn(m, n, 1000 * seed + b, _dtype(case)) for b, (m, n) in enumerate(_batch_shapes(case, seed))]


def prepare(case, seed):
    s = dict(case=case, h=_get_handle())
    if case["kind"] == "batch":
        s["As"] = _batch(case, seed)
        return s
    s["A"] = _matrix(case, seed)
    if case["kind"] == "grad":
        s["W"] = _randn(case["nb"] + 1, case["n"], 1000 * seed + 3, _dtype(case))
        s["A"] = s["A"].requires_grad_()
    if case["kind"] == "vectors":
        s["C"] = _randn(case["m"], case["cols"], 1000 * seed + 4, _dtype(case))
        s["D"] = _randn(case["cols"], case["n"], 1000 * seed + 5, _dtype(case))
        s["res"] = s["h"].band(s["A"], case["nb"], case["ib"], case["tree"], case["variant"])
    return s


def run(state):
    c, h = state["case"], state["h"]
    if c["kind"] == "band":
        return h.band(state["A"], c["nb"], c["ib"], c["tree"], c["variant"]).band()
    if c["kind"] == "batch":
        As, k = state["As"], len(state["As"])
        if c["nb"]:
            res = h.band_batched(As, [c["nb"]] * k, [c["ib"]] * k, [c["tree"]] * k, ["bidiag"] * k)
        else:
            res = h.band_batched(As)
        return [r.band() for r in res]
    if c["kind"] == "grad":
        ab = band_bidiag(state["A"], c["nb"], c["ib"], c["tree"], c["variant"], handle=h)
        (grad,) = torch.autograd.grad(ab, state["A"], state["W"])
        return {"band": ab.detach(), "grad": grad}
    Q = state["res"].apply_q(state["C"].t().clone().t(), 0)
    P = state["res"].apply_p(state["D"].t().clone().t(), 1)
    return {"QC": Q, "DPt": P}


# ---- what a pass cannot do without ---------------------------------------------------------------

def _flops(m, n):
    """The cheaper of the direct reduction and the one through a QR factorization."""
    return min(4.0 * n * n * (m - n / 3.0), 2.0 * n * n * (m + n))


def work(case):
    e = 8 if case["dtype"] == "f64" else 4
    if case["kind"] == "batch":
        sh = _batch_shapes(case, 0)
        return {"bytes": e * sum(m * n + ((case["nb"] or 64) + 1) * n for m, n in sh),
                "flops": sum(_flops(m, n) for m, n in sh)}
    m, n, nb = case["m"], case["n"], case["nb"]
    if case["kind"] == "band":
        return {"bytes": e * (m * n + (nb + 1) * n), "flops": _flops(m, n)}
    if case["kind"] == "grad":
        return {"bytes": e * (2 * m * n + 2 * (nb + 1) * n), "flops": 3 * _flops(m, n)}
    k = case["cols"]
    return {"bytes": e * (m * n + 2 * k * (m + n)), "flops": 4.0 * k * (m * n - n * n / 2.0) + 2.0 * k * n * n}


# ---- the same results in 64 bits -----------------------------------------------------------------
# The tile algorithm in dense torch.linalg calls: eliminating a tile is LAPACK's QR of the two stacked
# tiles, whose reflectors and signs are those of the tile kernels (zeros below the pivot's triangle stay
# zeros), applied to the tiles right of it.  LQ steps are QR steps of the transpose.

def _halving(rows):
    out = []
    while len(rows) > 1:
        z, h = len(rows), len(rows) // 2
        out += [(rows[z - h + t], rows[z - 2 * h + t]) for t in range(h)]
        rows = rows[:z - h]
    return out


def _eliminations(rows, v, tree, R):
    """(row, pivot, is TS) of one step with v trailing tile columns."""
    if tree in ("flatts", "flattt"):
        return [(r, rows[0], tree == "flatts") for r in rows[1:]]
    a = 1
    if tree == "auto":
        a = next((a for a in range(len(rows), 0, -1) if -(-len(rows) // a) * v >= 2 * R), 1)
    heads, out = rows[::a], []
    for s in range(0, len(rows), a):
        out += [(r, rows[s], True) for r in rows[s + 1:s + a]]
    return out + [(i, p, False) for i, p in _halving(heads)]


def _qr_step(M, k, rows, v, tree, R, nb, ops):
    """One QR step of tile column k of M (in place) over the given tile rows."""
    done = set()

    def factor(tiles):
        r = torch.cat([torch.arange(t * nb, (t + 1) * nb, device=M.device) for t in tiles])
        a, tau = torch.geqrf(M[r, k * nb:(k + 1) * nb])
        ops.append((r, a, tau))
        M[r, k * nb:(k + 1) * nb] = torch.triu(a)
        if (k + 1) * nb < M.shape[1]:
            M[r, (k + 1) * nb:] = torch.ormqr(a, tau, M[r, (k + 1) * nb:], left=True, transpose=True)

    def triangle(t):
        if t not in done:
            done.add(t)
            factor([t])

    el = _eliminations(rows, v, tree, R)
    if not el:
        triangle(rows[0])
    for i, piv, ts in el:
        triangle(piv)
        if not ts:
            triangle(i)
        factor([piv, i])


def _reduce(A, nb, tree, variant, R):
    """(band-bidiagonal matrix padded to whole tiles, QR operations, LQ operations) of the tile algorithm."""
    m, n = A.shape
    p, q = -(-m // nb), -(-n // nb)
    M = torch.zeros((p * nb, q * nb), dtype=torch.float64, device="cuda")
    M[:m, :n] = A
    left, right = [], []
    if variant == "rbidiag":
        for k in range(q):
            _qr_step(M, k, list(range(k, p)), q - k - 1, tree, R, nb, left)
        M = M[:q * nb].clone()
        p = q
    for k in range(q):
        if variant != "rbidiag" or k > 0:
            _qr_step(M, k, list(range(k, p)), q - k - 1, tree, R, nb, left)
        if k + 1 < q:
            _qr_step(M.t(), k, list(range(k + 1, q)), p - k - 1, tree, R, nb, right)
    return M, left, right


def _band_of(M, n, nb):
    ab = torch.zeros((nb + 1, n), dtype=torch.float64, device="cuda")
    for d in range(nb + 1):            # ab[nb - s, j] = M[j - s, j], s the superdiagonal
        s = nb - d
        if s < n:
            ab[d, s:] = torch.diagonal(M[:n, :n], s)
    return ab


def _apply(ops, C):
    """Q C for the product Q of the operations in the order they were made."""
    for r, a, tau in reversed(ops):
        C[r] = torch.ormqr(a, tau, C[r], left=True, transpose=False)
    return C


def _dense_reflectors(M, nb, record):
    """Band bidiagonalization of M (in place), one reflector at a time on the whole matrix."""
    m, n = M.shape
    order = []
    for k in range(0, n, nb):
        order += [(False, j, j) for j in range(k, min(k + nb, n))]
        order += [(True, i, i + nb) for i in range(k, min(k + nb, n)) if i + nb < n]
    for lq, col, row in order:         # in the orientation of the step: column `col`, rows from `row` on
        X = M.t() if lq else M
        if row + 1 >= X.shape[0]:      # nothing below: H = I
            continue
        x = X[row:, col].clone()
        sigma = torch.linalg.vector_norm(x)
        beta = torch.where(x[0] < 0, sigma, -sigma)
        v = x / (x[0] - beta)
        v[0] = 1.0
        tau = (beta - x[0]) / beta
        X[row:, col:] -= torch.outer(tau * v, v @ X[row:, col:])
        X[row + 1:, col] = 0.0
        record.append((lq, col, row, v, tau, beta))


def _dense_gradient(M, S, record):
    """dL/dA from S = dL/dB, undoing the recorded reflectors on the state M = B and on the gradient."""
    for lq, col, row, v, tau, beta in reversed(record):
        X, Y = (M.t(), S.t()) if lq else (M, S)
        Xs, Ys = X[row:, col:], Y[row:, col:]
        Ys[1:, 0] = 0.0                                  # the eliminated entries are constants
        b = v @ Ys
        Xs -= torch.outer(tau * v, v @ Xs)               # the state before the step
        a = v @ Xs
        v_bar = -tau * (Ys @ a + Xs @ b)
        tau_bar = -(a @ b)
        Ys -= torch.outer(tau * v, b)
        x = Xs[:, 0].clone()
        d = x[0] - beta
        d_bar = -(v_bar[1:] @ v[1:]) / d
        x_bar = torch.cat([(d_bar - tau_bar / beta)[None], v_bar[1:] / d])
        x_bar += (tau_bar * x[0] / beta ** 2 - d_bar) * x / beta
        Ys[:, 0] += x_bar
    return S


def _exact_grad(A, W, nb, Bt):
    m, n = A.shape
    M, record = A.clone(), []
    _dense_reflectors(M, nb, record)
    # the tree's band differs from the dense one by signs of rows and columns
    t, d = Bt[:n, :n].cpu().numpy(), M[:n].cpu().numpy()
    s1, s2 = np.ones(n), np.ones(n)
    s2[:nb + 1] = np.sign(t[0, :nb + 1] * d[0, :nb + 1])
    for i in range(1, n):
        s1[i] = np.sign(t[i, i] * d[i, i]) * s2[i]
        if i + nb < n:
            s2[i + nb] = np.sign(t[i, i + nb] * d[i, i + nb]) * s1[i]
    S = torch.zeros_like(M)
    sign = torch.from_numpy(np.outer(s1, s2)).cuda()
    for e in range(nb + 1):
        s = nb - e
        if s < n:
            torch.diagonal(S[:n], s).copy_(W[e, s:].double())
    S[:n] *= sign
    return _dense_gradient(M, S, record)


def _resources(nb, dtype):
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    return max(1, nsm * (64 if dtype == "f32" else 32) // nb)


def exact(case, seed):
    c = case
    R = _resources(c["nb"], c["dtype"]) if c["nb"] else 1
    if c["kind"] == "batch":
        if not c["nb"]:                # the autotuner's choice decides the form of the band
            return None
        tiles = sum((-(-m // c["nb"]) * -(-n // c["nb"])) for m, n in _batch_shapes(c, seed))
        if tiles > 1500:
            return None
        out = []
        for A in _batch(c, seed):
            M, _, _ = _reduce(A.double(), c["nb"], c["tree"], "bidiag", R)
            out.append(_band_of(M, A.shape[1], c["nb"]))
        return out
    m, n, nb = c["m"], c["n"], c["nb"]
    p, q = -(-m // nb), -(-n // nb)
    if c["variant"] == "auto" or (c["variant"] == "rbidiag" and c["tree"] == "greedy") or p * q > 1100:
        return None
    if c["dtype"] == "f32" and n > 2048:   # among so many pivots some are near zero, where FP32 turns a row's sign
        return None
    A = _matrix(c, seed).double()
    M, left, right = _reduce(A, nb, c["tree"], c["variant"], R)
    if c["kind"] == "band":
        return _band_of(M, n, nb)
    if c["kind"] == "grad":
        if n > 1024:
            return None
        W = _randn(nb + 1, n, 1000 * seed + 3, _dtype(c))
        return {"band": _band_of(M, n, nb), "grad": _exact_grad(A, W, nb, M)}
    C = torch.zeros((p * nb, c["cols"]), dtype=torch.float64, device="cuda")
    C[:m] = _randn(m, c["cols"], 1000 * seed + 4, _dtype(c)).double()
    D = torch.zeros((q * nb, c["cols"]), dtype=torch.float64, device="cuda")
    D[:n] = _randn(c["cols"], n, 1000 * seed + 5, _dtype(c)).double().t()
    return {"QC": _apply(left, C)[:m], "DPt": _apply(right, D)[:n].t()}
