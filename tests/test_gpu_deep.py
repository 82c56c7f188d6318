"""Contexts of up to 65536 points store up to eight filter steps beside the noise
estimate, larger ones three: the same frame in a context of either kind gives the same
bits, power, objective and keep flags, from frames of a few points to the largest, with
powers below, at and beyond the stored steps."""
import numpy as np
import pytest
import torch

from paper_2401_09721_gb300 import build, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    build.build()
    from paper_2401_09721_gb300 import fgbd
    return fgbd


@pytest.mark.parametrize("variant", ["plain", "global", "all_points"])
@pytest.mark.parametrize("q_max", [1, 2, 5, 64])
@pytest.mark.parametrize("n,noise", [(1, 30.0), (3, 30.0), (129, 60.0), (2051, 4.0), (7001, 60.0), (65536, 30.0)])
def test_either_context_gives_the_same(F, n, noise, q_max, variant):
    rng = np.random.default_rng(n)
    bits = 5 if n < 3000 else 7
    xyz = rng.integers(0, 1 << bits, size=(n, 3)).astype(np.int32)
    base = 128 + 80 * np.sin(xyz / float(1 << bits) * 3.0)
    rgb = np.clip(np.rint(base + rng.normal(0, noise, (n, 3))), 0, 255).astype(np.uint8)
    x, c = torch.from_numpy(xyz).cuda(), torch.from_numpy(rgb).cuda()
    v = {"plain": 0, "global": F.VARIANT_GLOBAL_Q, "all_points": F.VARIANT_NO_FSLR}[variant]
    got = []
    for cap in (65536, 65537):
        ctx = F.Context(cap, bits=bits, q_max=q_max, variant=v)
        whole = ctx.run(x, c, out_dtype=torch.float32).cpu().numpy()
        ctx.sync()
        st = ctx.stats()
        got.append((whole, st["q"], np.array(st["objective"]), ctx.fslr()[1].cpu().numpy()))
        ctx.close()
    (a, qa, ja, ka), (b, qb, jb, kb) = got
    assert qa == qb and np.array_equal(ja, jb) and np.array_equal(ka, kb) and np.array_equal(a, b)
