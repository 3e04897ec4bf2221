"""The block-wide sums and maxima of the screen and the best at sizes around a
warp and a block, with values that need all 64 bits.  Integer results: the
tolerance is zero."""
import numpy as np
import pytest
import torch

from paper_1706_00037_gb300 import ubqp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [1, 2, 31, 32, 33, 1023, 1024, 1025, 2600])
@pytest.mark.parametrize("kind", ["wide", "low", "high", "ties"])
def test_block_reductions(S, kind):
    rng = np.random.default_rng(S)
    top = 2 ** 62 // S  # any sum of S such values fits
    v = {"wide": rng.integers(-top, top, S), "low": -rng.integers(1, top, S),
         "high": rng.integers(2 ** 33, 2 ** 33 + 3, S) * 2 ** 16,
         "ties": rng.integers(0, 2, S) * (2 ** 32) - 2 ** 32}[kind].astype(np.int64)
    f = torch.from_numpy(v).cuda()
    st = ubqp.screen_stats(f, 5).cpu().tolist()
    assert st == [sum(int(a) for a in v), int(v.max()), int(v.argmax()) + 5]
    X = torch.arange(S * 3, dtype=torch.int64, device="cuda").view(S, 3)
    bx, bf = ubqp.best(f, X)
    assert bf.cpu().tolist() == [int(v.max()), int(v.argmax())]
    assert torch.equal(bx, X[int(v.argmax())])
