"""The preparation of large instances: every pair of tiles taken once.  Row sums
(the first-derivative start), the largest coefficient, evaluations that read all
of the int8 copy and of the tensor-core operand, the start-up product that reads
both triangles, and the symmetry check at single elements in the corners and the
middle, at sizes around the largest supported.  Integer results: the tolerance is
zero."""
import pytest
import torch

from paper_1706_00037_gb300 import ubqp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1281, 4097, 7936, 7937, 16129, 16383, 16384])
def test_prepare_large(n):
    g = torch.Generator("cuda").manual_seed(n)
    Q = torch.randint(-100, 101, (n, n), dtype=torch.int8, device="cuda", generator=g)
    Q = torch.triu(Q) + torch.triu(Q, 1).T
    Q[n // 3, n - 2] = Q[n - 2, n // 3] = -128
    inst = ubqp.Instance(Q)
    assert inst.max_abs == 128
    j = torch.arange(n, device="cuda")
    x0 = ubqp.first_derivative(inst)
    assert torch.equal((x0[j // 64] >> (j % 64)) & 1, (Q.sum(1, dtype=torch.int64) > 0).long())
    S = 4
    X = ubqp.diversify(inst, S, mode=ubqp.RANDOM, seed=n)
    X[0] = -1  # every variable set; bits above n do not count
    if n % 64:
        X[0, -1] = (1 << (n % 64)) - 1
    bits = ((X[:, j // 64] >> (j % 64)) & 1).double()
    want = torch.zeros(S, dtype=torch.float64, device="cuda")
    for a in range(0, n, 2048):  # exact in double: |sums| < 2^36
        want += ((bits @ Q[:, a:a + 2048].double()) * bits[:, a:a + 2048]).sum(1)
    for path in (ubqp.EVAL_PLAIN, ubqp.EVAL_TC_STAGED, ubqp.EVAL_TC, ubqp.EVAL_TC_TMEM):
        assert torch.equal(ubqp.eval(inst, X, path=path), want.long())
    # one move from the tensor-core start-up against one without
    idx = torch.arange(S, dtype=torch.int32, device="cuda")
    cnt = torch.full((1,), S, dtype=torch.int64, device="cuda")
    got = []
    for use in (True, False):
        Xa, f = X.clone(), want.long()
        ubqp.ascent(inst, Xa, f, idx, cnt, 1, use_ws=use)
        got.append((Xa, f))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    for r, c in ((0, n - 1), (n - 1, 0), (n // 2, n // 2 - 1), (n - 2, n - 1), (n // 3, n // 2)):
        keep = Q[r, c].clone()
        Q[r, c] = 127 if int(keep) != 127 else 126
        with pytest.raises(ubqp.UbqpError, match="symmetric"):
            ubqp.Instance(Q)
        Q[r, c] = keep
