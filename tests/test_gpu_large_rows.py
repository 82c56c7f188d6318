"""Rows of more points than an item holds, the largest of which are put line by line before
the windows are sorted: planes and boxes along the axes, thick slabs, several large rows side
by side with small ones between, grids of few bits; the three orders of the graph, of a
segmented batch and of the static call must equal a stable sort of the codes.  And what
they cost: a plane of 10^6 points no more than a few times a sphere of as many."""
import numpy as np
import pytest
import torch

from oracle import fgbd_oracle as orc
from paper_2401_09721_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    build.build()
    from paper_2401_09721_gb300 import fgbd
    return fgbd


def plane(axis, u, v, at):
    a, b = np.meshgrid(np.arange(u), np.arange(v), indexing="ij")
    return np.insert(np.stack([a.ravel(), b.ravel()], 1), axis, at, axis=1)


def points(kind, axis, rng):
    if kind == "plane":
        xyz, bits = plane(axis, 400, 250, 300), 10
    elif kind == "slab":  # four rows of 40,000 points of this axis's code, hundreds of the others'
        xyz, bits = np.concatenate([plane(axis, 200, 200, 50 + i) for i in range(4)]), 8
    elif kind == "box":
        xyz, bits = np.concatenate([plane(a, 150, 120, at) for a in range(3) for at in (0, 149)]), 9
    elif kind == "between":  # split rows among large and small ones, and on both sides of the limits
        xyz = np.concatenate([plane(axis, 190, 190, 20), plane(axis, 256, 128, 40), plane(axis, 256, 128, 41)[1:],
                              plane(axis, 129, 255, 42), plane(axis, 85, 85, 43), plane(axis, 84, 84, 44),
                              plane(axis, 190, 190, 45)])
        xyz = np.concatenate([xyz, rng.integers(0, 256, size=(3000, 3))])
        xyz = xyz[~((xyz[:, axis] == 40) | (xyz[:, axis] == 41)) | (np.arange(len(xyz)) < len(xyz) - 3000)]
        bits = 8
    elif kind == "few_bits":
        xyz, bits = rng.integers(0, 4, size=(150000, 3)), 2
    elif kind == "line":  # one line longer than an item, among others of its row
        xyz = np.concatenate([np.insert(rng.integers(0, 2, size=(30000, 2)), axis, 9, axis=1),
                              np.insert(rng.integers(0, 64, size=(9000, 2)), axis, 9, axis=1)])
        bits = 6
    return xyz[rng.permutation(len(xyz))].astype(np.int32), bits


KINDS = ["plane", "slab", "box", "between", "few_bits", "line"]


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("kind", KINDS)
def test_orders(F, kind, axis):
    xyz, bits = points(kind, axis, np.random.default_rng(axis))
    want = orc.scan_orders(orc.scan_line_codes(xyz, bits))
    d = torch.from_numpy(xyz).cuda()
    ctx = F.Context(len(xyz) + 5000, bits=bits)
    for _ in range(2):  # and with the counters of a call before
        ctx.build_graph(d)
        ctx.sync()
        assert np.array_equal(ctx.orders().cpu().numpy(), want)
    ctx.close()


def test_segmented_batch_and_static(F):
    rng = np.random.default_rng(9)
    frames = [points(k, a, rng) for a, k in enumerate(["between", "slab"])]
    frames.append((rng.integers(0, 256, size=(5000, 3)).astype(np.int32), 8))
    frames.append((np.concatenate([plane(2, 85, 86, 7), rng.integers(0, 256, size=(200, 3))]).astype(np.int32), 8))
    ctxs = [F.Context(len(x), bits=8) for x, _ in frames]
    xs = [torch.from_numpy(x).cuda() for x, _ in frames]
    cs = [torch.from_numpy(rng.integers(0, 256, size=x.shape, dtype=np.uint8)).cuda() for x, _ in frames]
    for _ in range(3):
        F.Context.run_batch(ctxs, xs, cs)
        for c, (x, bits) in zip(ctxs, frames):
            c.sync()
            assert np.array_equal(c.orders().cpu().numpy(), orc.scan_orders(orc.scan_line_codes(x, bits)))
    for c in ctxs:
        c.close()
    for axis in range(3):
        xyz = np.concatenate([plane(axis, 150, 150, 200), rng.integers(0, 256, size=(9000, 3))]).astype(np.int32)
        out = torch.empty((3, len(xyz)), dtype=torch.int32, device="cuda")
        d = torch.from_numpy(xyz).cuda()
        F._check(F.lib().fgbd_scan_orders_static(F._ptr(d), len(xyz), 8, F._ptr(out), None, F._stream(None)), "static")
        assert np.array_equal(out.cpu().numpy(), orc.scan_orders(orc.scan_line_codes(xyz, 8)))


def test_a_wait_that_gives_up_is_reported(F):
    p = plane(2, 1000, 1000, 300)
    xyz = p[np.random.default_rng(4).permutation(len(p))].astype(np.int32)
    d = torch.from_numpy(xyz).cuda()
    ctx = F.Context(len(xyz), bits=10)
    ctx.set_wait_limit(0)
    ctx.build_graph(d)
    with pytest.raises(F.FgbdError) as err:
        ctx.sync()
    assert err.value.status == 5  # FGBD_ETIMEOUT
    ctx.set_wait_limit(2_000_000_000)
    ctx.build_graph(d)
    ctx.sync()
    assert np.array_equal(ctx.orders().cpu().numpy(), orc.scan_orders(orc.scan_line_codes(xyz, 10)))
    ctx.close()


def build_time(F, xyz, bits):
    ctx = F.Context(len(xyz), bits=bits)
    d = torch.from_numpy(xyz.astype(np.int32)).cuda()
    times = []
    for _ in range(8):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        ctx.build_graph(d)
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b))
    ctx.close()
    return min(times)


def test_a_plane_costs_like_a_surface(F):
    """Three passes over the points of a row for every 4096 of them cost 6 times as much."""
    rng = np.random.default_rng(1)
    v = rng.normal(size=(1000000, 3))
    v /= np.linalg.norm(v, axis=1)[:, None]
    ball = build_time(F, np.rint(512 + 500 * v), 10)
    for axis in range(3):
        p = plane(axis, 1000, 1000, 300)
        assert build_time(F, p[rng.permutation(len(p))], 10) < 2.5 * ball
