"""Orders of points that repeat voxels thousands of times, which the sort takes through a
bitonic sort or a bitmap of the input indices: one voxel and a few, among others and alone, in the input's
order and shuffled, in rows that are split by lines and not, more input indices than one
bitmap holds, on both sides of the frame size that one launch sorts, and in a segmented
batch.  Equal codes are ordered by input index (Section 2.2).  And what that costs."""
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


def points(kind, rng):
    others = lambda n, top: rng.integers(0, top, size=(n, 3))
    if kind == "one":
        return np.full((100000, 3), 77), 10
    if kind == "small":        # one launch from the coordinates
        return np.concatenate([np.full((5000, 3), 9), others(3000, 16)]), 4
    if kind == "beside":       # a row that is not split
        return np.concatenate([others(20000, 1024), np.full((20000, 3), 500)]), 10
    if kind == "few":
        return np.array([[3, 5, 9], [4, 5, 9], [4, 6, 9], [4, 6, 8]])[rng.integers(0, 4, size=50000)], 6
    if kind == "runs":         # side by side in the input, in a split row
        return np.concatenate([np.repeat(np.array([[7, 7, 7], [8, 7, 7], [7, 7, 8]]), 15000, axis=0), others(500, 64)]), 6
    if kind == "wide":         # indices of two bitmaps
        return np.concatenate([others(880000, 128), np.full((30000, 3), 3)]), 7
    if kind == "many":         # buckets of equal points
        return np.concatenate([np.repeat(rng.integers(0, 1024, size=(20, 3)), 500 + 2 * np.arange(20), axis=0),
                               others(9000, 1024)]), 10
    if kind == "crowded":      # equal points around what is ranked by comparisons, on a line and not
        spread = np.repeat(rng.integers(0, 1024, size=(100, 3)), np.arange(270, 370), axis=0)
        line = np.repeat(np.stack([np.arange(100), np.full(100, 3), np.full(100, 4)], 1), np.arange(270, 370), axis=0)
        return np.concatenate([spread, line]), 10
    if kind == "pairs":        # an item of the largest size, and a frame of two voxels
        return np.array([[3, 4, 5], [900, 4, 5]])[rng.integers(0, 2, size=11264)], 10


KINDS = ["one", "small", "beside", "few", "runs", "wide", "many", "crowded", "pairs"]


@pytest.mark.parametrize("shuffle", [False, True])
@pytest.mark.parametrize("kind", KINDS)
def test_orders(F, kind, shuffle):
    rng = np.random.default_rng(len(kind))
    xyz, bits = points(kind, rng)
    if shuffle:
        xyz = xyz[rng.permutation(len(xyz))]
    xyz = xyz.astype(np.int32)
    d = torch.from_numpy(xyz).cuda()
    ctx = F.Context(len(xyz), bits=bits)
    ctx.build_graph(d)
    ctx.sync()
    assert np.array_equal(ctx.orders().cpu().numpy(), orc.scan_orders(orc.scan_line_codes(xyz, bits)))
    ctx.close()


def test_segmented_batch(F):
    rng = np.random.default_rng(3)
    xyz = [points(k, rng)[0].astype(np.int32) for k in ("beside", "one", "many")]
    ctxs = [F.Context(len(x), bits=10) for x in xyz]
    cs = [torch.from_numpy(rng.integers(0, 256, size=x.shape, dtype=np.uint8)).cuda() for x in xyz]
    F.Context.run_batch(ctxs, [torch.from_numpy(x).cuda() for x in xyz], cs)
    for c, x in zip(ctxs, xyz):
        c.sync()
        assert np.array_equal(c.orders().cpu().numpy(), orc.scan_orders(orc.scan_line_codes(x, 10)))
        c.close()


def build_time(F, xyz):
    ctx = F.Context(len(xyz), bits=10)
    d = torch.from_numpy(xyz.astype(np.int32)).cuda()
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


def test_what_one_voxel_costs(F):
    """(A radix sort of all digits, a chunk of 1024 points at a time: some 45 times a spread frame.)"""
    rng = np.random.default_rng(2)
    spread = build_time(F, rng.integers(0, 1024, size=(100000, 3)))
    assert build_time(F, np.full((100000, 3), 77)) < 18 * spread
