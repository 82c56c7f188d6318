"""Colours taken into the C1 order: uint8 arrays that start on any byte (read as
aligned words where they can be) and sizes around the four points a thread takes
must give what the same colours give in an aligned array."""
import numpy as np
import pytest
import torch

from paper_2401_09721_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    build.build()
    from paper_2401_09721_gb300 import fgbd
    return fgbd


@pytest.mark.parametrize("window", [1, 2])
@pytest.mark.parametrize("n", [1, 2, 3, 5, 1021, 4098])
def test_colour_arrays_at_any_byte(F, n, window):
    rng = np.random.default_rng(n)
    xyz = torch.from_numpy(rng.integers(0, 64, size=(n, 3)).astype(np.int32)).cuda()
    rgb = torch.from_numpy(rng.integers(0, 256, size=(n, 3)).astype(np.uint8)).cuda()
    ref = None
    for off in range(4):
        store = torch.zeros(3 * n + 4, dtype=torch.uint8, device="cuda")
        c = store[off:off + 3 * n].view(n, 3)
        c.copy_(rgb)
        assert c.data_ptr() % 4 == off
        ctx = F.Context(n, bits=6, window=window)
        whole = ctx.run(xyz, c).cpu().numpy()
        ctx.sync()
        st = ctx.stats()
        ctx.build_graph(xyz)
        ctx.estimate_noise(c)
        ctx.select_filter(c)
        parts = ctx.denoise(None, -1).cpu().numpy()
        got = (whole, st["sigma_est"], st["q"], ctx.fslr()[0].cpu().numpy())
        assert np.array_equal(whole, parts)
        if ref is None:
            ref = got
        else:
            assert np.array_equal(got[0], ref[0]) and got[1:3] == ref[1:3] and np.array_equal(got[3], ref[3])
        ctx.close()
