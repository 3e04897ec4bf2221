"""The measured rates that the ascent's roofline is made of: the element update is
counted as the two operations per element that the climb makes of it, and a climb
that fills the chip stays below the rate."""
import pytest
import torch

from paper_1706_00037_gb300 import synth, ubqp

pytestmark = pytest.mark.gpu


def test_element_update_bounds_the_climb():
    lib = ubqp.load()
    # per thread and iteration: 8 multiply-adds; 16 elements of 2 operations
    assert lib.ubqp_peak_int32_ops(1, 1000) == 4 * lib.ubqp_peak_int32_ops(0, 1000) > 0
    rate = ubqp.measure_peaks()["ascent_update_tops"] * 1e12
    n, S = 2048, 4000
    inst = ubqp.Instance(torch.from_numpy(synth.make_instance(n, 0.5, 9)).cuda())
    X0 = ubqp.diversify(inst, S, mode=ubqp.RANDOM, seed=1)
    f0 = ubqp.eval(inst, X0)
    every = torch.arange(S, dtype=torch.int32, device="cuda")
    cnt = torch.full((1,), S, dtype=torch.int64, device="cuda")
    flips = torch.zeros(S, dtype=torch.int32, device="cuda")
    best = 0.0
    for _ in range(3):
        X, f = X0.clone(), f0.clone()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        ubqp.ascent(inst, X, f, every, cnt, 0, flips)
        e1.record()
        torch.cuda.synchronize()
        best = max(best, 2 * n * int(flips.sum()) / (e0.elapsed_time(e1) / 1e3))
    assert 0.1 * rate < best < rate
