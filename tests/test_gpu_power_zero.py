"""Power 0 leaves the colours as they are, whichever buffer the steps would have started
from: the output equals the input bit for bit, for both colour types, in a context whose
buffers hold the iterates of another frame, on every path that can end at q = 0 without
stored steps (a fixed power, q_max = 0, a reused power, batches on streams)."""
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


def frame(n, src, seed):
    rng = np.random.default_rng(seed)
    xyz = torch.from_numpy(rng.integers(0, 128, size=(n, 3)).astype(np.int32)).cuda()
    rgb = rng.uniform(0, 255, size=(n, 3)).astype(np.float32) if src == "f32" else rng.integers(0, 256, size=(n, 3), dtype=np.uint8)
    return xyz, torch.from_numpy(rgb).cuda()


def constant(xyz, src):
    """Colours without noise, for which the search stops at q = 0."""
    c = torch.tensor([10.0, 99.0, 200.0], device="cuda").repeat(len(xyz), 1)
    return c if src == "f32" else c.to(torch.uint8)


def expect(rgb, out):
    """The input in the output's type (rounded half to even, as the output conversion does)."""
    want = rgb.float()
    if out.dtype == torch.uint8:
        want = want.round().clamp(0, 255).to(torch.uint8)
    assert torch.equal(out, want)


OUT = [torch.float32, torch.uint8]


@pytest.mark.parametrize("window", [1, 2])
@pytest.mark.parametrize("src", ["u8", "f32"])
@pytest.mark.parametrize("n", [1001, 4098, 70003])
def test_fixed_power(F, n, src, window):
    xyz, rgb = frame(n, src, n)
    other = frame(n, src, n + 1)
    ctx = F.Context(n, bits=7, window=window)
    for dt in OUT:
        ctx.run(*other)
        ctx.build_graph(xyz)
        expect(rgb, ctx.denoise(rgb, 0, out_dtype=dt))
    ctx.close()


@pytest.mark.parametrize("window", [1, 2])
@pytest.mark.parametrize("src", ["u8", "f32"])
@pytest.mark.parametrize("n", [1001, 4098, 70003])
def test_largest_power_zero(F, n, src, window):
    xyz, rgb = frame(n, src, n)
    other = frame(n, src, n + 1)
    ctx = F.Context(n, bits=7, window=window, q_max=0)
    for dt in OUT:
        out = torch.empty((n, 3), dtype=dt, device="cuda")
        for _ in range(3):  # direct, recorded, replayed
            ctx.build_graph(other[0])
            ctx.denoise(other[1], 3)
            expect(rgb, ctx.run(xyz, rgb, out=out))
            expect(rgb, ctx.denoise(None, -1, out_dtype=dt))
        ctx.denoise(other[1], 3)
        ctx.build_graph(xyz)
        ctx.estimate_noise(rgb)
        assert ctx.select_filter(rgb, host=True) == 0
        expect(rgb, ctx.denoise(None, -1, out_dtype=dt))
    ctx.close()


@pytest.mark.parametrize("src", ["u8", "f32"])
@pytest.mark.parametrize("n", [1002, 70003])
def test_reused_power(F, n, src):
    xyz, rgb = frame(n, src, n)
    other = frame(n, src, n + 1)
    ctx = F.Context(n, bits=7)
    for dt in OUT:
        ctx.build_graph(other[0])
        ctx.denoise(other[1], 3)
        ctx.run(xyz, constant(xyz, src))
        assert ctx.stats()["q"] == 0
        expect(rgb, ctx.run_reuse(xyz, rgb, out_dtype=dt))
    ctx.close()


@pytest.mark.parametrize("kinds", [["f32"], ["f32", "f32", "f32"], ["u8", "f32", "u8", "f32"]])
def test_batches_on_streams(F, kinds):
    dev = torch.cuda.current_device()
    frames = [frame(3001 + 17 * i, k, i) for i, k in enumerate(kinds)]
    others = [frame(3001 + 17 * i, k, 50 + i) for i, k in enumerate(kinds)]
    flat = [constant(x, k) for (x, _), k in zip(frames, kinds)]
    ctxs = [F.Context(len(x), bits=7) for x, _ in frames]
    mean = int(np.mean([len(x) for x, _ in frames]))
    streams = dict(seg_frames=0, scatter_threads=512, filter_threads=512, filter_blocks_per_sm=2)
    try:
        F.fgbd_set_batch_shape(dev, mean, streams)
        for dt in OUT:
            outs = [torch.empty((len(x), 3), dtype=dt, device="cuda") for x, _ in frames]
            for _ in range(3):  # direct, recorded, replayed
                for c, (x, y) in zip(ctxs, others):
                    c.build_graph(x)
                    c.denoise(y, 3)
                F.Context.run_batch(ctxs, [x for x, _ in frames], flat, outs=outs)
                for c, y, o in zip(ctxs, flat, outs):
                    assert c.stats()["q"] == 0
                    expect(y, o)
                    expect(y, c.denoise(None, -1, out_dtype=dt))
    finally:
        F.fgbd_set_batch_shape(dev, mean, None)
        for c in ctxs:
            c.close()
