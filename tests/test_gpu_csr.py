"""The CSR export at the edges of its blocks (1024 rows), warps and staged rows, for
every window, with repeated voxels: row pointers and columns as the oracle's, weights
within 1e-6 of max(1, |log w|) in the exponent, and the handle's copy the same."""
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


@pytest.mark.parametrize("window", [1, 2, 3])
@pytest.mark.parametrize("n", [1, 2, 3, 31, 33, 1023, 1024, 1025, 5000])
def test_rows_of_any_frame(F, n, window):
    rng = np.random.default_rng(n)
    xyz = rng.integers(0, 16, size=(n, 3)).astype(np.int32)
    ctx = F.Context(n, bits=4, window=window)
    ctx.build_graph(torch.from_numpy(xyz).cuda())
    edges = orc.slg_edges(orc.scan_orders(orc.scan_line_codes(xyz, 4)), window)
    row_ptr, col = orc.adjacency_csr(edges, n)
    got_ptr, got_col, got_w = (t.cpu().numpy() for t in ctx.graph_csr())
    assert np.array_equal(got_ptr, row_ptr) and np.array_equal(got_col, col)
    if col.size:
        w = orc.edge_weights(xyz, row_ptr, col, orc.sigma_g(xyz, row_ptr, col))
        ok = w > 1e-30
        lw = np.log(w[ok])
        err = np.abs(np.log(got_w.astype(np.float64)[ok]) - lw)
        assert (err <= 1e-6 * np.maximum(1.0, np.abs(lw)) + 1e-6).all()
    g = ctx.export_graph()
    assert np.array_equal(g.row_ptr.cpu().numpy(), got_ptr)
    assert np.array_equal(g.col.cpu().numpy(), got_col) and np.array_equal(g.w.cpu().numpy(), got_w)
    none = ctx.graph_csr(with_weights=False)
    assert none[2] is None and np.array_equal(none[1].cpu().numpy(), got_col)
    del g
    ctx.close()
