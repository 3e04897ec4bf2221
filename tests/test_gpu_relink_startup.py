"""The relinking's start-up without a tensor-core workspace, which adds the rows
of the set bits several at a time: initiating solutions with from 0 to n bits set,
so that the rows of a word come in full groups and remainders, against the
tensor-core start-up and the oracle.  Integer results: the tolerance is zero."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_1706_00037_gb300 import synth, ubqp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [500, 1000, 2561, 3072, 4096, 4500, 8192, 8300])
def test_startup_rows_in_flight(n):
    Q = synth.make_instance(n, 0.2, n)
    inst = ubqp.Instance(torch.from_numpy(Q).cuda())
    bits = [0, 1, 2, 7, 8, 9, 15, 16, 17, 31, 63, 64, 65, 100, 300, n]
    rng = np.random.default_rng(n)
    x = np.zeros((len(bits), (n + 63) // 64 * 64), np.uint8)
    for p, k in enumerate(bits):
        # the first pairs' bits crowd into one word, the others lie anywhere
        x[p, rng.permutation(min(n, 64) if k <= 64 else n)[:k]] = 1
    Xh = np.packbits(x, axis=1, bitorder="little").view(np.uint64)
    X = torch.from_numpy(Xh.view(np.int64)).cuda()
    G = X.clone()
    G[:, :3] = ubqp.diversify(inst, len(bits), mode=ubqp.RANDOM, seed=n)[:, :3]
    f = ubqp.eval(inst, X)
    got = ubqp.relink(inst, X, f, G, tensor_startup=False)
    want = ubqp.relink(inst, X, f, G)
    inst.sync()
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    Gh = G.cpu().numpy().view(np.uint64)
    for p in (0, 5, 13):
        xb, fb, d, *_ = orc.relink1(Q, Xh[p], Gh[p])
        assert (int(got[1][p]), int(got[2][p])) == (fb, d)
        assert np.array_equal(got[0][p].cpu().numpy().view(np.uint64), xb)
