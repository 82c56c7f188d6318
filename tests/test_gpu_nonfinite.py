"""Float colours that are not finite: a point with empty slots (no neighbour along
a code) must not let 0 x infinity turn its own infinity into something else, and
points out of reach of the odd colours keep the bits they have without them."""
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


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("variant", [0, 4])   # 4: same-line links, so that many slots are empty
def test_filter_with_a_colour_that_is_not_finite(F, bad, variant):
    rng = np.random.default_rng(3)
    n = 3000
    xyz = torch.from_numpy(np.unique(rng.integers(0, 40, size=(n, 3)), axis=0).astype(np.int32)).cuda()
    n = xyz.shape[0]
    rgb = rng.uniform(0, 255, size=(n, 3)).astype(np.float32)
    i = int(rng.integers(0, n))
    odd = rgb.copy()
    odd[i] = bad
    ctx = F.Context(n, bits=6, variant=variant)
    ctx.build_graph(xyz)
    row_ptr, col, w = (t.cpu().numpy() for t in ctx.graph_csr())
    a = ctx.denoise(torch.from_numpy(rgb).cuda(), 1).cpu().numpy()
    b = ctx.denoise(torch.from_numpy(odd).cuda(), 1).cpu().numpy()
    near = set(col[row_ptr[i]:row_ptr[i + 1]].tolist()) | {i}
    far = np.array([k for k in range(n) if k not in near])
    assert np.array_equal(a[far], b[far]) and np.isfinite(b[far]).all()
    if np.isnan(bad):
        assert np.isnan(b[i]).all()
    else:   # x_i / 2 + a finite sum / 2
        assert (b[i] == bad).all()
    ctx.close()
