"""Batches of frames around the size from which on the frames of a segmented launch take
their later steps one after another: bit for bit what one call a frame gives (direct, recorded and
replayed, a remainder of one frame, uint8 and float colours), and with large powers not
slower than the frames one by one."""
import numpy as np
import pytest
import torch

from paper_2401_09721_gb300 import build

pytestmark = pytest.mark.gpu

LIMIT = 7 << 17  # mean points


@pytest.fixture(scope="module")
def F():
    build.build()
    from paper_2401_09721_gb300 import fgbd
    return fgbd


def frame(n, sigma, seed, as_float=False, slope=0.002):
    """Points of a sphere, smooth colours and noise."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn(n, 3, generator=g, device="cuda")
    xyz = (511.0 + 500.0 * v / v.norm(dim=1, keepdim=True)).round().to(torch.int32)
    rgb = 128.0 + 60.0 * torch.sin(slope * xyz.float()) + sigma * torch.randn(n, 3, generator=g, device="cuda")
    return xyz.contiguous(), rgb if as_float else rgb.round().clamp(0, 255).to(torch.uint8)


@pytest.mark.parametrize("q_max", [64, 8, 9])
def test_limits_around_the_steps_side_by_side(F, q_max):
    """The search's own limit before, at and behind the step after which it is taken up again."""
    n = LIMIT + 3
    x, y = frame(n, 40.0, 1, slope=0.0003)
    ctxs = [F.Context(n, bits=10, q_max=q_max) for _ in range(3)]
    ref = ctxs[0].run(x, y).clone()
    q, objective = ctxs[0].stats()["q"], ctxs[0].stats()["objective"]
    assert q >= min(q_max, 9)
    for o, c in zip(F.Context.run_batch(ctxs, [x] * 3, [y] * 3), ctxs):
        assert torch.equal(o, ref) and c.stats()["q"] == q and c.stats()["objective"] == objective
        c.close()


@pytest.mark.parametrize("sizes,as_float", [([LIMIT - 9, LIMIT + 9], False), ([LIMIT - 10, LIMIT + 9], False),
                                            ([1000000, 30000, 1900000, 900001, LIMIT + 1], False),
                                            ([LIMIT + 5, LIMIT + 4, LIMIT + 3], True)])
def test_equal_to_single_frames(F, sizes, as_float):
    # powers below, at and above the steps taken side by side
    slopes = [0.002, 0.0003, 0.012, 0.0008, 0.006]
    frames = [frame(n, 20.0 + 6.0 * i, i, as_float, slopes[i]) for i, n in enumerate(sizes)]
    ctxs = [F.Context(n, bits=10) for n in sizes]
    refs = []
    for c, (x, y) in zip(ctxs, frames):
        out = c.run(x, y).clone()
        st = c.stats()
        refs.append((out, st["q"], st["sigma_est"], st["objective"], c.denoise(None, -1).clone()))
    outs = [torch.empty((n, 3), dtype=torch.float32, device="cuda") for n in sizes]
    for _ in range(3):
        for o in outs:
            o.fill_(-1.0)
        F.Context.run_batch(ctxs, [x for x, _ in frames], [y for _, y in frames], outs=outs)
        for c, o, (ref, q, sg, objective, kept) in zip(ctxs, outs, refs):
            st = c.stats()
            assert st["q"] == q and st["sigma_est"] == sg and st["objective"] == objective
            assert torch.equal(o, ref) and torch.equal(c.denoise(None, -1), kept)
    for c in ctxs:
        c.close()


def test_large_powers_cost_what_single_frames_do(F):
    """(Side by side the steps of four frames evict each other's data from L2.)"""
    n, count = 1000000, 8
    x, y = frame(n, 40.0, 1, slope=0.0003)
    ctxs = [F.Context(n, bits=10) for _ in range(count)]
    outs = [torch.empty((n, 3), dtype=torch.uint8, device="cuda") for _ in range(count)]

    def time(run):
        best = 1e9
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            run()
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    def one_by_one():
        for c, o in zip(ctxs, outs):
            c.run(x, y, out=o)

    alone = time(one_by_one)
    assert ctxs[0].stats()["q"] >= 32
    together = time(lambda: F.Context.run_batch(ctxs, [x] * count, [y] * count, outs=outs))
    for c in ctxs:
        c.close()
    assert together < 1.03 * alone
