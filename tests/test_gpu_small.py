"""Small instances (n <= 128): the shared-memory evaluation that AUTO launches
and the climb's own start-up, at the edges of their rules; and the block-wide
sums and maxima of the screen and the best at sizes around a warp and a block,
with values that need all 64 bits; and the preparation of Q from rows at any
alignment, with the start-up product built on it, at the edges of its tiles.
Integer results: the tolerance is zero."""
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


@pytest.mark.parametrize("off", [0, 1, 3])
@pytest.mark.parametrize("n", [1, 2, 3, 63, 64, 65, 68, 127, 130, 197, 257, 322, 515])
def test_prepare_rows_at_any_alignment(n, off):
    Q = instance(n, "any")
    flat = torch.full((n * n + off,), 77, dtype=torch.int8, device="cuda")
    flat[off:] = torch.from_numpy(Q).cuda().flatten()
    inst = ubqp.Instance(flat[off:].view(n, n))
    assert inst.max_abs == int(np.abs(Q.astype(np.int32)).max())
    S = 150
    X = ubqp.diversify(inst, S, mode=ubqp.RANDOM, seed=n)
    j = torch.arange(n, device="cuda")
    bits = ((X[:, j // 64] >> (j % 64)) & 1).double()
    y = bits @ torch.from_numpy(Q).cuda().double()
    want = (y * bits).sum(1).long()
    for path in (ubqp.EVAL_PLAIN, ubqp.EVAL_TC_STAGED, ubqp.EVAL_TC):  # the int8 copy, Q'
        assert torch.equal(ubqp.eval(inst, X, path=path), want)
    # one move from the tensor-core start-up (Q' and its transpose) against one without
    idx = torch.zeros(1600, dtype=torch.int32, device="cuda")
    idx[:S] = torch.arange(S, dtype=torch.int32, device="cuda")
    cnt = torch.full((1,), S, dtype=torch.int64, device="cuda")
    got = []
    for use in (True, False):
        Xa, f = X.clone(), want.clone()
        ubqp.ascent(inst, Xa, f, idx, cnt, 1, use_ws=use)
        got.append((Xa, f))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    x0 = ubqp.first_derivative(inst)
    x0 = ((x0[j // 64] >> (j % 64)) & 1).bool().cpu().numpy()
    assert np.array_equal(x0, Q.astype(np.int64).sum(1) > 0)
    if n > 1:  # one element off the symmetric value, anywhere in a tile
        for r, c in ((0, n - 1), (n - 1, 0), (n // 2, n // 2 - 1)):
            bad = flat.clone()
            bad[off + r * n + c] = (int(Q[r, c]) + 129) % 256 - 128
            with pytest.raises(Exception, match="symmetric"):
                ubqp.Instance(bad[off:].view(n, n))


@pytest.mark.parametrize("count", [0, 1, 31, 32, 33, 127, 128, 129, 160])
def test_startup_product_rows(count):
    """The rows of Y that the start-up product adds to, at the edges of a warp's
    32 rows and of a tile's 128: one move from it against one without."""
    n, S = 515, 200
    inst = ubqp.Instance(torch.from_numpy(instance(n, "any")).cuda())
    X = ubqp.diversify(inst, S, mode=ubqp.RANDOM, seed=count)
    f0 = ubqp.eval(inst, X)
    idx = torch.randperm(S, device="cuda").int()
    cnt = torch.full((1,), count, dtype=torch.int64, device="cuda")
    got = []
    for use in (True, False):
        Xa, f = X.clone(), f0.clone()
        ubqp.ascent(inst, Xa, f, idx, cnt, 1, use_ws=use)
        got.append((Xa, f))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    assert int((got[0][1] != f0).sum()) <= count
