"""Small instances (n <= 128): the shared-memory evaluation that AUTO launches
and the climb's own start-up, at the edges of their rules; and the block-wide
sums and maxima of the screen and the best at sizes around a warp and a block,
with values that need all 64 bits.  Integer results: the tolerance is zero."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_1706_00037_gb300 import ubqp

pytestmark = pytest.mark.gpu

NS = [1, 2, 31, 33, 63, 64, 65, 100, 127, 128, 129]


def instance(n, kind):
    if kind == "minus":
        return np.full((n, n), -128, np.int8)
    v = np.triu(np.random.default_rng(n).integers(-128, 128, (n, n)).astype(np.int8))
    return v + np.triu(v, 1).T


@pytest.mark.parametrize("kind", ["minus", "any"])
@pytest.mark.parametrize("n", NS)
def test_small_evaluation(n, kind):
    Q = instance(n, kind)
    inst = ubqp.Instance(torch.from_numpy(Q).cuda())
    line = min(2 ** 18 // n, 8192)  # the last S of the rule and the first beyond it
    for S in (1, 7, 8, 9, line, line + 1):
        X = torch.randint(-2 ** 63, 2 ** 63 - 1, (S, (n + 63) // 64), dtype=torch.int64,
                          device="cuda")  # bits above n are set and do not count
        f = torch.full((S,), -1, dtype=torch.int64, device="cuda")
        ubqp.eval(inst, X, out=f)
        plain = ubqp.eval(inst, X, path=ubqp.EVAL_PLAIN)
        assert torch.equal(f, plain)
        j = torch.arange(n, device="cuda")
        bits = ((X[:, j // 64] >> (j % 64)) & 1).double()
        want = ((bits @ torch.from_numpy(Q).cuda().double()) * bits).sum(1).long()
        assert torch.equal(f, want)


@pytest.mark.parametrize("n", NS)
def test_small_startup(n):
    Q = instance(n, "any")
    inst = ubqp.Instance(torch.from_numpy(Q).cuda())
    line = 10 * torch.cuda.get_device_properties(0).multi_processor_count
    S = line + 1
    X0 = ubqp.diversify(inst, S, mode=ubqp.RANDOM, seed=n)
    f0 = ubqp.eval(inst, X0)
    got = []
    for cap in (line, line + 1):  # the climb's own start-up, then the tensor cores'
        X, f = X0.clone(), f0.clone()
        idx = torch.arange(cap, dtype=torch.int32, device="cuda")
        cnt = torch.full((1,), line, dtype=torch.int64, device="cuda")
        flips = torch.full((S,), -1, dtype=torch.int32, device="cuda")
        ubqp.ascent(inst, X, f, idx, cnt, 0, flips)
        got.append((X, f, flips))
    for a, b in zip(*got):
        assert torch.equal(a, b)
    Xh = X0.cpu().numpy().view(np.uint64)
    for s in (0, line - 1):
        x, fv, c, _ = orc.ascent1(Q, Xh[s], int(f0[s]), 0, 0)
        assert (int(got[0][1][s]), int(got[0][2][s])) == (fv, c)
        assert np.array_equal(got[0][0][s].cpu().numpy().view(np.uint64), x)


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
