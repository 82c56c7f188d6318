"""Float colours are summed in shares of the points, one or two a block: whole-number
float colours, whose sums are exact in any grouping, must give the patch count and the
eigenvalues of the same uint8 colours, from one share to two a block and several turns
a share.  Bound: the covariance's float64 cancellation (255^2 2^-53 and a few times
that) and the eigenvectors' second-order error, both below 1e-9 of the largest."""
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


@pytest.mark.parametrize("n", [255, 257, 116735, 116737, 136193, 155647, 155649, 311297, 400001])
def test_every_point_once(F, n):
    rng = np.random.default_rng(n)
    v = rng.normal(size=(n, 3))
    v /= np.linalg.norm(v, axis=1)[:, None]
    xyz = torch.from_numpy(np.rint(255 + 250 * v).astype(np.int32)).cuda()
    rgb = np.clip(np.rint(128 + 60 * v + rng.normal(0, 20, (n, 3))), 0, 255).astype(np.uint8)
    got = []
    for c in (rgb, rgb.astype(np.float32)):
        ctx = F.Context(n, bits=9)
        ctx.build_graph(xyz)
        ctx.estimate_noise(torch.from_numpy(c).cuda())
        ctx.sync()
        st = ctx.stats()
        got.append((st["n_patches"], np.array(st["eigenvalues"])))
        ctx.close()
    (pa, ea), (pb, eb) = got
    assert pa == pb
    assert np.allclose(ea, eb, rtol=0, atol=1e-9 * abs(ea[0]) + 1e-9)
