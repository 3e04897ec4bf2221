"""The unpacked batch climb in each of its shapes: groups much wider than the
instances' rows and groups that every row fills by three quarters or more, with fewer listed starts than
SMs and with more, run and replayed from a graph.  Every instance's result
equals its single solve, exactly."""
import pytest
import torch

from paper_1706_00037_gb300 import synth, ubqp

pytestmark = pytest.mark.gpu

SHAPES = [(64, 1), (64, 2), (128, 1), (128, 2), (256, 1), (256, 2), (512, 1), (512, 2)]


@pytest.mark.parametrize("S,mode", [(60, ubqp.RANDOM), (900, ubqp.DIVERSIFY)])
@pytest.mark.parametrize("rows", ["narrow", "full"])
@pytest.mark.parametrize("shape", SHAPES)
def test_unpacked_shapes_equal_single_solves(shape, rows, S, mode):
    width = 16 * shape[0] * shape[1]
    # narrow: rows from 1024 elements up in a group of `width`; full: rows that
    # fill it (rows are padded to a multiple of 1024)
    sizes = [33, 200, 513, min(width, 1100)] if rows == "narrow" else [width, width * 3 // 4]
    insts = [ubqp.Instance(torch.from_numpy(synth.make_instance(n, 0.3, 40 + n)).cuda())
             for n in sizes]
    p = ubqp.make_params(S, 0.25, max_flips=300, mode=mode, seed=1)
    b = ubqp.Batch(insts, p)
    b.set(*shape)
    for seed, graph in ((3, False), (4, True)):
        if graph:
            b.capture()
        b.run(seed)
        for i, inst in enumerate(insts):
            p1 = ubqp.make_params(S, 0.25, max_flips=300, mode=mode, seed=seed)
            x, f, _ = ubqp.solve(inst, p1, want_stats=False)
            bx, bf = b.result(i)
            assert torch.equal(bf, f) and torch.equal(bx, x), inst.n
