"""The eigenvalues of the patch covariance where their reduction can go wrong:
grey and constant channels (rank-deficient, whole columns already reduced), one
direction only (every reflection but the first skipped), clusters (white noise) and
two levels; with uint8 colours, whose moments are exact integers, so that only the
eigenvalues differ."""
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


def colours(kind, xyz, rng):
    n = len(xyz)
    c = rng.integers(0, 256, (n, 3))
    if kind == "grey":
        c = np.repeat(c[:, :1], 3, axis=1)
    elif kind == "one_channel":
        c[:, 1:] = 77
    elif kind == "ramp":
        c = np.outer(xyz.sum(1), [1, 2, 3])
    elif kind == "two_levels":
        c = np.repeat(255 * (xyz.sum(1) % 2)[:, None], 3, axis=1)
    elif kind == "faint":
        c = 128 + (rng.random((n, 3)) < 0.01)
    return c.astype(np.uint8)


# Bound: 1e-7 of the largest eigenvalue (float64 quotients of vectors with float32
# errors: second order) and the 1e-9 below which an eigenvalue counts as zero.
@pytest.mark.parametrize("window", [1, 2])
@pytest.mark.parametrize("kind", ["white", "grey", "one_channel", "ramp", "two_levels", "faint"])
def test_eigenvalues(F, kind, window):
    rng = np.random.default_rng(3)
    xyz = np.unique(rng.integers(0, 16, size=(6000, 3)), axis=0).astype(np.int32)
    rgb = colours(kind, xyz, rng)
    res = orc.fgbd(xyz, rgb, orc.Params(bits=4, window=window), q=0)
    ctx = F.Context(len(xyz), bits=4, window=window)
    ctx.build_graph(torch.from_numpy(xyz).cuda())
    ctx.estimate_noise(torch.from_numpy(rgb).cuda())
    ctx.sync()
    st = ctx.stats()
    want = np.array(res.noise["eigenvalues"])
    got = np.array(st["eigenvalues"])
    assert st["n_patches"] == res.noise["n_patches"] > 0
    assert np.isfinite(got).all()
    assert np.allclose(got, want, rtol=0, atol=1e-7 * abs(want[0]) + 1e-9)
    ctx.close()
