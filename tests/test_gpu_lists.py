"""Lists of the ascent that are longer than the starts: entries outside [0, S)
are skipped and reported by sync, every valid entry is climbed wherever it
stands, as it is when listed alone.  Integer results: the tolerance is zero."""
import pytest
import torch

from paper_1706_00037_gb300 import synth, ubqp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("use_ws", [True, False])
@pytest.mark.parametrize("length", [130, 700, 1700])
@pytest.mark.parametrize("n", [100, 513, 1500, 2100, 5000])
def test_list_longer_than_the_starts(n, length, use_ws):
    S = 100
    inst = ubqp.Instance(torch.from_numpy(synth.make_instance(n, 0.5, n)).cuda())
    X0 = ubqp.diversify(inst, S, seed=n)
    f0 = ubqp.eval(inst, X0)
    every = torch.arange(S, dtype=torch.int32, device="cuda")
    want = (X0.clone(), f0.clone(), torch.full((S,), -1, dtype=torch.int32, device="cuda"))
    ubqp.ascent(inst, want[0], want[1], every, torch.tensor([S], device="cuda"), 0, want[2],
                use_ws=use_ws)
    inst.sync()
    # outside: -1 and S; the valid ones spread over the list, its end included
    idx = torch.full((length,), -1, dtype=torch.int32, device="cuda")
    idx[::2] = S
    idx[torch.linspace(0, length - 1, S).long().cuda()] = every
    got = (X0.clone(), f0.clone(), torch.full((S,), -1, dtype=torch.int32, device="cuda"))
    ubqp.ascent(inst, got[0], got[1], idx, torch.tensor([length], device="cuda"), 0, got[2],
                use_ws=use_ws)
    with pytest.raises(ubqp.UbqpError) as e:
        inst.sync()
    assert e.value.status == -1  # UBQP_ERR_ARG
    inst.sync()  # reported once
    for a, b in zip(got, want):
        assert torch.equal(a, b)
