"""The ascent's and the relinking's group shapes at the edges of the rule that
picks them: at each n where the shape changes, the same starts climbed in one
long list (the shape for a full chip), in lists of a few hundred and in chunks
of 100 (the shape with the shortest chain) give identical results, and some of
them equal the oracle's.  Two kinds of instance: every coefficient -128 (the
largest gains int8 allows, all of them ties) and coefficients in {-1, 0, 1}
(many equal gains).  Integer results: the tolerance is zero."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_1706_00037_gb300 import ubqp

pytestmark = pytest.mark.gpu

EDGES = [512, 513, 1024, 1025, 1536, 1537, 2048, 2049, 2560, 2561, 3072, 3073, 4096, 4097, 5120,
         5121, 6144, 6145, 7168, 7169, 8192, 8193]


def instance(n, kind):
    if kind == "minus":
        return np.full((n, n), -128, np.int8)
    v = np.triu(np.random.default_rng(n).integers(-1, 2, (n, n), dtype=np.int8))
    return v + np.triu(v, 1).T


def climb(inst, X0, f0, lists, cap, use_ws=True):
    X, f = X0.clone(), f0.clone()
    flips = torch.full((X.shape[0],), -1, dtype=torch.int32, device="cuda")
    for idx in lists:
        cnt = torch.full((1,), idx.numel(), dtype=torch.int64, device="cuda")
        ubqp.ascent(inst, X, f, idx, cnt, cap, flips, use_ws=use_ws)
    inst.sync()
    return X, f, flips


@pytest.mark.parametrize("kind", ["minus", "small"])
@pytest.mark.parametrize("n", EDGES)
def test_shapes_agree(n, kind):
    S, cap = 1700, 20
    Q = instance(n, kind)
    inst = ubqp.Instance(torch.from_numpy(Q).cuda())
    X0 = ubqp.diversify(inst, S, mode=ubqp.RANDOM, seed=n)
    f0 = ubqp.eval(inst, X0)
    every = torch.arange(S, dtype=torch.int32, device="cuda")
    want = climb(inst, X0, f0, every.split(100), cap)
    for lists, ws in (([every], True), (every.split(700), True), (every.split(850), False)):
        if not ws:  # start-up on the CUDA cores: a few starts
            lists = [every[:40]]
        got = climb(inst, X0, f0, lists, cap, use_ws=ws)
        some = slice(None) if ws else slice(0, 40)
        for a, b in zip(got, want):
            assert torch.equal(a[some], b[some])
    Xh = X0.cpu().numpy().view(np.uint64)
    for s in (0, S - 1):
        x, fv, c, _ = orc.ascent1(Q, Xh[s], int(f0[s]), cap, cap)
        assert (int(want[1][s]), int(want[2][s])) == (fv, c)
        assert np.array_equal(want[0][s].cpu().numpy().view(np.uint64), x)


@pytest.mark.parametrize("n", [512, 513, 1025, 2049, 2561, 4097, 5121, 7169])
def test_relink_shapes_agree(n):
    P = 200
    Q = instance(n, "small")
    inst = ubqp.Instance(torch.from_numpy(Q).cuda())
    X = ubqp.diversify(inst, P, mode=ubqp.RANDOM, seed=n)
    G = X.clone()
    G[:, : min(4, X.shape[1])] = torch.roll(X, 1, 0)[:, : min(4, X.shape[1])]
    f = ubqp.eval(inst, X)
    got = ubqp.relink(inst, X, f, G)
    parts = [ubqp.relink(inst, X[a:a + 100], f[a:a + 100], G[a:a + 100]) for a in (0, 100)]
    bare = ubqp.relink(inst, X, f, G, tensor_startup=False)
    inst.sync()
    for k in range(3):
        assert torch.equal(got[k], torch.cat([p[k] for p in parts]))
        assert torch.equal(got[k], bare[k])
    Xh, Gh = (t.cpu().numpy().view(np.uint64) for t in (X, G))
    for p in (0, P - 1):
        xb, fb, d, *_ = orc.relink1(Q, Xh[p], Gh[p])
        assert (int(got[1][p]), int(got[2][p])) == (fb, d)
        assert np.array_equal(got[0][p].cpu().numpy().view(np.uint64), xb)


@pytest.mark.parametrize("S", [64, 400])
def test_packed_classes_equal_single_solves(S):
    """The packed batch climb at the edges of its size classes, with few starts
    in all and with more than ten per SM."""
    insts = [ubqp.Instance(torch.from_numpy(instance(n, "small")).cuda())
             for n in (512, 513, 1024, 1025, 1536, 1537, 2048, 2049, 2560, 2561, 3072, 3073, 4096,
                       4097)]
    p = ubqp.make_params(S, 0.25, seed=5)
    batch = ubqp.Batch(insts, p)
    batch.set(256, 2, packed=True)
    batch.run(5)
    for i, inst in enumerate(insts):
        bx, bf = batch.result(i)
        x, f, _ = ubqp.solve(inst, p, want_stats=False)
        assert torch.equal(bx, x) and torch.equal(bf, f), inst.n
