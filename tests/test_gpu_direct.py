"""Frames of up to 8192 points are sorted by one launch from the coordinates, larger
ones through the row scatter: the three orders on both sides of the line, of points
spread out, on one line, in one voxel or a few (which overfill the buckets), and what a
coordinate out of range does."""
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


def points(kind, n, bits, rng):
    top = 1 << bits
    xyz = rng.integers(0, top, size=(n, 3))
    if kind == "line":
        xyz[:, 1:] = top - 1
    elif kind == "voxel":
        xyz[:] = top // 3
    elif kind == "few":
        xyz = rng.integers(0, 2, size=(n, 3)) * (top - 1)
    elif kind == "corner":
        xyz = np.minimum(xyz, rng.integers(0, top, size=(n, 3)) // 16) + top - top // 16 - 1
    return xyz.astype(np.int32)


@pytest.mark.parametrize("bits", [4, 10])
@pytest.mark.parametrize("kind", ["spread", "line", "voxel", "few", "corner"])
@pytest.mark.parametrize("n", [1, 2, 1023, 1025, 8191, 8192, 8193])
def test_orders_on_both_sides(F, n, kind, bits):
    rng = np.random.default_rng(n + bits)
    xyz = points(kind, n, bits, rng)
    ctx = F.Context(9000, bits=bits)
    want = orc.scan_orders(orc.scan_line_codes(xyz, bits))
    for _ in range(2):  # and with the scalars of a call before
        ctx.build_graph(torch.from_numpy(xyz).cuda())
        assert np.array_equal(ctx.orders().cpu().numpy(), want)
    ctx.close()


@pytest.mark.parametrize("n", [5, 8192, 8193])
def test_a_coordinate_out_of_range_is_an_error(F, n):
    rng = np.random.default_rng(n)
    xyz = rng.integers(0, 64, size=(n, 3)).astype(np.int32)
    bad = xyz.copy()
    bad[n // 2, 1] = 64
    ctx = F.Context(n, bits=6)
    ctx.build_graph(torch.from_numpy(bad).cuda())
    with pytest.raises(F.FgbdError):
        ctx.sync()
    ctx.build_graph(torch.from_numpy(xyz).cuda())
    ctx.sync()
    assert np.array_equal(ctx.orders().cpu().numpy(), orc.scan_orders(orc.scan_line_codes(xyz, 6)))
    ctx.close()
