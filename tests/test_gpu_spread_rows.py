"""Orders of points whose rows lie far apart or whose extent is that of a few stray points,
where the buckets of the sort follow the rows: bodies apart along an axis, dense blocks
with points in the corners of the grid, thin rods, on both sides of the frame size that one
launch sorts; alone, in the static call and in a segmented batch.  And what that costs."""
import numpy as np
import pytest
import torch

from oracle import fgbd_oracle as orc
from paper_2401_09721_gb300 import build

pytestmark = pytest.mark.gpu

CORNERS = np.array([[0, 0, 0], [1023, 1023, 1023], [0, 1023, 0], [1023, 0, 1023]])


@pytest.fixture(scope="module")
def F():
    build.build()
    from paper_2401_09721_gb300 import fgbd
    return fgbd


def ball(n, radius, centre, rng):
    out = np.zeros((0, 3), int)
    while len(out) < n:
        v = rng.normal(size=(2 * n, 3))
        v /= np.linalg.norm(v, axis=1)[:, None]
        out = np.unique(np.concatenate([out, np.floor(v * radius + centre).astype(int)]), axis=0)
    return out[rng.permutation(len(out))[:n]]


def block(sides, at):
    return np.stack(np.meshgrid(*[np.arange(s) for s in sides], indexing="ij"), -1).reshape(-1, 3) + at


def points(kind, axis, rng):
    turn = lambda v: np.roll(v, axis, axis=1)
    if kind == "apart":
        return turn(np.concatenate([ball(20000, 50, 100, rng), ball(20000, 50, [900, 100, 100], rng)]))
    if kind == "block":
        return np.concatenate([block([30, 30, 30], 400), CORNERS])
    if kind == "small_block":
        return np.concatenate([block([20, 20, 20], 400), CORNERS])
    if kind == "rods":  # two lines side by side in a row, and as many points far from them
        return turn(np.concatenate([block([500, 2, 8], 300), block([500, 2, 8], [10, 900, 900]), CORNERS]))
    if kind == "wall":  # a row above an item, a split one, corners
        return turn(np.concatenate([block([1, 90, 90], 500), block([1, 190, 190], 600), CORNERS]))
    if kind == "repeats":  # buckets of rows that repeated voxels overfill
        return np.concatenate([np.repeat(block([2, 2, 2], 500), 700, axis=0), block([10, 10, 10], 400), CORNERS])


KINDS = ["apart", "block", "small_block", "rods", "wall", "repeats"]


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("kind", KINDS)
def test_orders(F, kind, axis):
    rng = np.random.default_rng(axis)
    xyz = points(kind, axis, rng)
    xyz = xyz[rng.permutation(len(xyz))].astype(np.int32)
    want = orc.scan_orders(orc.scan_line_codes(xyz, 10))
    d = torch.from_numpy(xyz).cuda()
    ctx = F.Context(len(xyz), bits=10)
    for _ in range(2):
        ctx.build_graph(d)
        ctx.sync()
        assert np.array_equal(ctx.orders().cpu().numpy(), want)
    ctx.close()
    if len(xyz) <= 32768:
        out = torch.empty((3, len(xyz)), dtype=torch.int32, device="cuda")
        F._check(F.lib().fgbd_scan_orders_static(F._ptr(d), len(xyz), 10, F._ptr(out), None, F._stream(None)), "static")
        assert np.array_equal(out.cpu().numpy(), want)


def test_segmented_batch(F):
    rng = np.random.default_rng(5)
    xyz = [points(k, 1, rng).astype(np.int32) for k in KINDS]
    ctxs = [F.Context(len(x), bits=10) for x in xyz]
    cs = [torch.from_numpy(rng.integers(0, 256, size=x.shape, dtype=np.uint8)).cuda() for x in xyz]
    F.Context.run_batch(ctxs, [torch.from_numpy(x).cuda() for x in xyz], cs)
    for c, x in zip(ctxs, xyz):
        c.sync()
        assert np.array_equal(c.orders().cpu().numpy(), orc.scan_orders(orc.scan_line_codes(x, 10)))
        c.close()


def build_time(F, xyz):
    ctx = F.Context(len(xyz), bits=10)
    d = torch.from_numpy(xyz[np.random.default_rng(0).permutation(len(xyz))].astype(np.int32)).cuda()
    times = []
    for _ in range(10):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        ctx.build_graph(d)
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b))
    ctx.close()
    return min(times)


def test_bodies_apart_cost_like_one(F):
    """(Items across the gap by the radix sort: 2.5 times one body of as many points.)"""
    rng = np.random.default_rng(2)
    one = build_time(F, ball(400000, 215, 512, rng))
    for axis in range(3):
        two = np.concatenate([ball(200000, 150, 200, rng), ball(200000, 150, [800, 200, 200], rng)])
        assert build_time(F, np.roll(two, axis, axis=1)) < 1.7 * one
