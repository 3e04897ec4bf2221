"""The ascent's launches by count, each to the end of its climbs: for every range
of n one list for each launch of the rule (its lengths follow from the number of
SMs), climbed without a cap, against the same starts climbed 100 at a time and,
for starts of the first wave and far beyond it, against the oracle with its flip
sequence; and lists capped past the moves between two looks at the clock.  Integer
results: the tolerance is zero."""
import numpy as np
import pytest
import torch

import oracle as orc
from oracle_pool import OraclePool
from paper_1706_00037_gb300 import synth, ubqp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pool():
    p = OraclePool()
    yield p
    p.close()


def lengths(n):
    """A list for each launch but the shortest lists' (the chunks of 100 take that):
    the middle launch, where there is one, and the one for long lists."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if n <= 1024:
        return [10 * sms + 80]
    if n <= 4096 or n > 6144:
        return [10 * sms - 20, 10 * sms + 80]
    if n <= 5120:
        return [2 * sms + 80]
    return [2 * sms - 10, 2 * sms + 80]


def climb(inst, X0, f0, lists, cap=0):
    X, f = X0.clone(), f0.clone()
    flips = torch.full((X.shape[0],), -1, dtype=torch.int32, device="cuda")
    ws = torch.empty(ubqp.ascent_workspace_size(inst, X.shape[0]), dtype=torch.uint8,
                     device="cuda")
    for idx in lists:
        cnt = torch.full((1,), idx.numel(), dtype=torch.int64, device="cuda")
        ubqp.ascent(inst, X, f, idx, cnt, cap, flips, ws=ws)
    inst.sync()
    return X, f, flips


@pytest.mark.parametrize("n", [400, 900, 1400, 1900, 2400, 2900, 3900, 4900, 5900, 6500, 8000])
def test_every_launch_to_the_end(pool, n):
    Q = synth.make_instance(n, 0.7, 500 + n)
    ref = pool.put(Q)
    inst = ubqp.Instance(torch.from_numpy(Q).cuda())
    S = max(lengths(n))
    X0 = ubqp.diversify(inst, S, mode=ubqp.RANDOM, seed=n)
    f0 = ubqp.eval(inst, X0)
    every = torch.arange(S, dtype=torch.int32, device="cuda")
    want = climb(inst, X0, f0, every.split(100))
    for m in lengths(n):
        got = climb(inst, X0, f0, [every[:m]])
        for a, b in zip(got, want):
            assert torch.equal(a[:m], b[:m])
    # the traced climb of the longest list
    ldt = 2 * n
    X, f = X0.clone(), f0.clone()
    cnt = torch.full((1,), S, dtype=torch.int64, device="cuda")
    flips, trace = ubqp.ascent_trace(inst, X, f, every, cnt, ldt)
    inst.sync()
    for a, b in zip((X, f, flips), want):
        assert torch.equal(a, b)
    Xh, fh = X0.cpu().numpy().view(np.uint64), f0.cpu().numpy()
    pick = sorted({0, 151, 153, S // 2, S - 2, S - 1} |
                  set(np.random.default_rng(n).integers(0, S, 4).tolist()))
    exact = pool.ascents(ref, Xh, fh, pick, cap=ldt)
    Xg, tr = X.cpu().numpy().view(np.uint64), trace.cpu().numpy().view(np.uint16)
    for s in pick:
        xw, fw, cw, tw = exact[s]
        assert (int(f[s]), int(flips[s])) == (fw, cw) and np.array_equal(Xg[s], xw), s
        assert np.array_equal(tr[s, :cw].astype(np.int64), tw.astype(np.int64)), s


@pytest.mark.parametrize("cap", [1022, 1023, 1024, 1025, 2100])
def test_caps_past_the_looks_at_the_clock(cap):
    n = 6500
    Q = synth.make_instance(n, 0.7, 500 + n)
    inst = ubqp.Instance(torch.from_numpy(Q).cuda())
    S = max(lengths(n))
    X0 = ubqp.diversify(inst, S, mode=ubqp.RANDOM, seed=n)
    f0 = ubqp.eval(inst, X0)
    every = torch.arange(S, dtype=torch.int32, device="cuda")
    want = climb(inst, X0, f0, every.split(100), cap)
    got = climb(inst, X0, f0, [every], cap)
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    assert int(got[2].max()) == cap
    Xh = X0.cpu().numpy().view(np.uint64)
    for s in (0, S - 1):
        x, fv, c, _ = orc.ascent1(Q, Xh[s], int(f0[s]), cap, cap)
        assert (int(got[1][s]), int(got[2][s])) == (fv, c)
        assert np.array_equal(got[0][s].cpu().numpy().view(np.uint64), x)
