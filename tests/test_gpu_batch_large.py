"""Batches of frames of 2^18 points and more that nothing was tuned for (four frames a
launch): bit for bit what one call a frame gives, direct, recorded and replayed, with a
remainder of one frame, uint8 and float colours, the same-line links, and equal to the
same batch on streams."""
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


def _frames(count, as_float):
    xs, cs = [], []
    for f in range(count):
        rng = np.random.default_rng(f)
        n = 262144 + 9001 * f
        v = rng.normal(size=(n, 3))
        v /= np.linalg.norm(v, axis=1)[:, None]
        xyz = np.clip(np.rint(511 + 400 * v), 0, 1023).astype(np.int32)
        rgb = np.clip(128 + 60 * v + rng.normal(0, 15 + 10 * f, (n, 3)), 0, 255)
        xs.append(torch.from_numpy(xyz).cuda())
        cs.append(torch.from_numpy(rgb.astype(np.float32) if as_float else np.rint(rgb).astype(np.uint8)).cuda())
    return xs, cs


@pytest.mark.parametrize("count,as_float,same_line", [(2, False, False), (5, False, False), (5, True, False),
                                                      (3, False, True)])
def test_untuned_large_batch(F, count, as_float, same_line):
    xs, cs = _frames(count, as_float)
    mean = int(np.mean([len(x) for x in xs]))
    dev = torch.cuda.current_device()
    v = F.VARIANT_SAME_LINE if same_line else 0
    ctxs = [F.Context(len(x), bits=10, variant=v) for x in xs]
    refs = []
    for c, x, y in zip(ctxs, xs, cs):
        refs.append((c.run(x, y, out_dtype=torch.float32).cpu().numpy(), c.stats()["q"], c.stats()["sigma_est"]))
    outs = [torch.empty((len(x), 3), dtype=torch.float32, device="cuda") for x in xs]
    streams = dict(seg_frames=0, scatter_threads=512, filter_threads=512, filter_blocks_per_sm=2)
    try:
        for shape in (None, streams):
            F.fgbd_set_batch_shape(dev, mean, shape)
            for _ in range(3):   # direct, recorded, replayed
                for o in outs:
                    o.fill_(-1.0)
                F.Context.run_batch(ctxs, xs, cs, outs=outs)
                torch.cuda.synchronize()
                for c, o, (ref, q, sg) in zip(ctxs, outs, refs):
                    assert np.array_equal(o.cpu().numpy(), ref)
                    assert c.stats()["q"] == q and c.stats()["sigma_est"] == sg
    finally:
        F.fgbd_set_batch_shape(dev, mean, None)
        for c in ctxs:
            c.close()
