"""The differentiable filter where its rows are unusual: one point (no neighbour),
two and three, sizes around a block of threads and past one wave of blocks, points
alone on a scan line in the same-line variant, results written over the input.
Tolerances as for the larger frames: colours 1e-4 on the [0, 1] scale, gradients 1e-4
of their largest magnitude, dL/dalpha and dL/dsigma 1e-4 or what the rounding of their
terms allows, whatever cancels."""
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


@pytest.mark.parametrize("same_line", [False, True])
@pytest.mark.parametrize("n,q,checkpoint", [(n, q, c) for n in (1, 2, 3, 255, 257)
                                            for q, c in ((1, 1), (3, 1), (5, 3))] + [(311297 + 300, 5, 3)])
def test_small_and_ragged_frames(F, n, q, checkpoint, same_line):
    rng = np.random.default_rng(n)
    bits = 6 if n < 1000 else 9
    xyz = rng.integers(0, 1 << bits, size=(n, 3)).astype(np.int32)
    y = rng.uniform(0, 255, size=(n, 3)).astype(np.float32)
    gout = rng.normal(size=(n, 3)).astype(np.float32)
    ctx = F.Context(n, bits=bits, variant=F.VARIANT_SAME_LINE if same_line else 0)
    ctx.build_graph(torch.from_numpy(xyz).cuda())
    codes = orc.scan_line_codes(xyz, bits)
    edges = orc.slg_edges(orc.scan_orders(codes), 1, codes if same_line else None, bits)
    row_ptr, col = orc.adjacency_csr(edges, n)
    sigma = 0.7 * 2.0 ** bits / max(n, 8) ** 0.34
    yt = torch.from_numpy(y).cuda()
    out, g = yt.clone(), torch.from_numpy(gout).cuda()
    gp = torch.full((2,), 7.0, dtype=torch.float64, device="cuda")
    F.fgbd_filter_forward(ctx.handle, out, q, 0.4, sigma, checkpoint, out, n)   # in place
    for _ in range(2):                                                         # the state serves again
        gin = g.clone()
        F.fgbd_filter_backward(ctx.handle, gin, gin, gp, n)
    torch.cuda.synchronize()
    ref = orc.param_filter(xyz, row_ptr, col, y, q, 0.4, sigma)
    gy, da, ds = orc.param_filter_vjp(xyz, row_ptr, col, y, q, 0.4, sigma, gout.astype(np.float64))
    assert np.abs(out.cpu().numpy() - ref[-1]).max() <= 1e-4 * 255
    assert np.abs(gin.cpu().numpy() - gy).max() <= 1e-4 * max(np.abs(gy).max(), 1e-12)
    # a term is a product of u and colours, each after at most q float32 steps of ~8 roundings;
    # R_ij (d_ij^2 - e_i) is at most a few sigma^2
    size = (q + 8) * 2.0 ** -24 * q * 2 * 255.0 * np.abs(gout).sum()
    got = gp.cpu().numpy()
    assert abs(got[0] - da) <= max(1e-4 * abs(da), size)
    assert abs(got[1] - ds) <= max(1e-4 * abs(ds), size * 8 / sigma)
    ctx.close()
