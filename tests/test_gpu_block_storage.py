"""Device memory a handle keeps for published panel blocks: given up when the handle's own allocations need it, not
kept above 2 GiB, returned with the handle."""
import numpy as np
import pytest

import paper_1611_06892_gb300 as G

pytestmark = pytest.mark.gpu
MB = 1 << 20


def gaussian(m, n):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(m + n)
    return torch.randn(n, m, dtype=torch.float64, device="cuda", generator=g).t()


def free_memory():
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_given_up_when_memory_is_short():
    import torch
    A = gaussian(8192, 8192)
    h = G.Handle()
    fill = None
    try:
        res = h.band(A, 256, 32, "auto", "bidiag")
        ref = res.band().clone()
        h.sync()
        res.free()
        # the tiles (512 MB) no longer fit beside the kept blocks, and the blocks (1.15 GB) not beside the tiles
        fill = torch.empty(free_memory() - 300 * MB, dtype=torch.uint8, device="cuda")
        res = h.band(A, 256, 32, "auto", "bidiag")
        h.sync()
        got = res.band()
        torch.cuda.synchronize()
        assert torch.equal(got, ref)
        res.free()
    finally:
        del fill
        h.close()
        torch.cuda.empty_cache()


def test_bounded_and_returned():
    import torch
    h = G.Handle()
    before = free_memory()
    try:
        A = gaussian(131072, 1024)            # 2.7 GB of blocks
        res = h.band(A, 256, 32, "auto", "rbidiag")
        h.sync()
        res.free()
        del A, res
        h.sync()
        assert before - free_memory() < 256 * MB       # (the plan)
        A = gaussian(4096, 4096)                       # 0.35 GB
        res = h.band(A, 256, 32, "auto", "bidiag")
        h.sync()
        res.free()
        del A, res
        assert before - free_memory() < 768 * MB
    finally:
        h.close()
    assert before - free_memory() < 64 * MB
