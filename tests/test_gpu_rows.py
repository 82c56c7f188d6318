"""The three scan orders at the sizes where the row scatter and the bucket sort
can go wrong: frames around a tile, a window and the sizes where the window
changes; rows larger than an item; lines of repeated voxels that overfill an
item or a bucket (the radix sort through global memory).  Orders must equal a
stable sort of the codes exactly (Section 2.2, ties by input index)."""
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


def _check(F, xyz, bits):
    xyz = np.ascontiguousarray(xyz.astype(np.int32))
    ref = orc.scan_orders(orc.scan_line_codes(xyz, bits))
    ctx = F.Context(len(xyz), bits=bits)
    d = torch.from_numpy(xyz).cuda()
    ctx.build_graph(d)
    ctx.sync()
    assert np.array_equal(ctx.orders().cpu().numpy(), ref)
    if len(xyz) <= 32768:
        out = torch.empty((3, len(xyz)), dtype=torch.int32, device="cuda")
        F._check(F.lib().fgbd_scan_orders_static(F._ptr(d), len(xyz), bits, F._ptr(out), None, F._stream(None)), "static")
        assert np.array_equal(out.cpu().numpy(), ref)
    ctx.close()


@pytest.mark.parametrize("bits", [6, 10])
@pytest.mark.parametrize("n", [1, 1023, 1025, 4095, 4097, 32767, 32769, 131071, 131073])
def test_sizes_around_tiles_and_windows(F, n, bits):
    rng = np.random.default_rng(n + bits)
    _check(F, rng.integers(0, 1 << bits, size=(n, 3)), bits)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("side", [84, 85, 256])   # 7056 and 7225 points a row (below and above one item), and a large one
def test_one_dense_plane_and_a_few_others(F, axis, side):
    rng = np.random.default_rng(axis + side)
    a, b = np.meshgrid(np.arange(side), np.arange(side), indexing="ij")
    plane = np.insert(np.stack([a.ravel(), b.ravel()], 1), axis, 77, axis=1)
    xyz = np.concatenate([plane, rng.integers(0, 256, size=(3000, 3))])
    _check(F, xyz[rng.permutation(len(xyz))], 8)


@pytest.mark.parametrize("n,cells", [(513, 1), (20000, 1), (50000, 2), (30000, 40)])
def test_repeated_voxels(F, n, cells):
    """n points on `cells` voxels of a line, among 2000 others."""
    rng = np.random.default_rng(n)
    line = np.stack([rng.integers(0, cells, size=n), np.full(n, 3), np.full(n, 9)], 1)
    xyz = np.concatenate([line, rng.integers(0, 64, size=(2000, 3))])
    _check(F, xyz[rng.permutation(len(xyz))], 6)


@pytest.mark.parametrize("bits", [1, 2])
def test_tiny_grids(F, bits):
    rng = np.random.default_rng(bits)
    _check(F, rng.integers(0, 1 << bits, size=(50000, 3)), bits)
