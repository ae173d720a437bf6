"""A matrix of an FP64 batch gets the bits it gets alone, also when only others of the batch take the tensor cores:
with strips of 64 columns tiles of 64 to 192 stay on the FP64 units, tiles of 32 do not."""
import numpy as np
import pytest

import paper_1611_06892_gb300 as G
from paper_1611_06892_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("strip", [16, 32, 64])
def test_batch_beside_other_strip_widths(strip):
    import torch
    cfg = [(32, 32), (64, 32), (96, 32), (128, 32), (64, 16), (48, 24), (128, 8), (32, 8)]
    As = [torch.from_numpy(np.asfortranarray(inputs.gaussian(140 + 37 * i, 101 + 23 * i, seed=i))).cuda()
          for i in range(len(cfg))]
    h = G.Handle()
    try:
        h.set_option(G.OPT_STRIP, strip)
        res = h.band_batched(As, [c[0] for c in cfg], [c[1] for c in cfg], ["greedy"] * len(cfg), ["bidiag"] * len(cfg))
        h.sync()
        for A, (nb, ib), r in zip(As, cfg, res):
            alone = h.band(A, nb, ib, "greedy", "bidiag")
            h.sync()
            assert torch.equal(r.band(), alone.band()), (nb, ib)
    finally:
        h.close()
