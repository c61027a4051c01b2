"""vq_decode_weights at the sizes where its tile changes: 8 rows, 16 where the codebooks outweigh a row, 16 and 32 where the grid
would be too tall."""
import numpy as np
import pytest

import vq_synth
from oracle import vq_oracle as orc
from tests.helpers import DeviceLayer, draw, lib_fmt, oracle_fmt

vq = pytest.importorskip("paper_2402_15319_b200")
pytestmark = pytest.mark.gpu

CASES = [
    vq_synth.LayerSpec("rows8_tail", N=300, K=2304, d=2, b=6, Br=4, Bc=256, int8=True),
    vq_synth.LayerSpec("rows8_short_tile", N=24, K=256, d=2, b=5, Br=24, Bc=128, int8=False),
    vq_synth.LayerSpec("rows16", N=4864, K=2048, d=4, b=8, Br=256, Bc=512, int8=False),
    vq_synth.LayerSpec("rows8_4d_few", N=512, K=2048, d=4, b=8, Br=256, Bc=512, int8=True),
]


@pytest.mark.parametrize("spec", CASES, ids=lambda s: s.name)
def test_decode_bit_exact(spec):
    L = draw(spec, 41)
    _, W16 = orc.decode(oracle_fmt(spec), L.idx, L.cb, L.scale, exact=False)
    assert np.array_equal(DeviceLayer(spec, L).decode().view(np.uint16), W16)


@pytest.mark.parametrize("times,d,b", [(8200, 1, 2), (16400, 2, 6)], ids=["16 rows", "32 rows"])   # 524,800 and 1,049,600 rows
def test_more_rows_than_a_grid_of_small_tiles_holds(times, d, b):
    import torch
    K = 256
    part = vq_synth.LayerSpec("part", N=64, K=K, d=d, b=b, Br=64, Bc=256, int8=True)
    L = draw(part, 43)
    dev = DeviceLayer(part, L)
    want = torch.from_numpy(dev.decode().view(np.int16)).cuda()
    tall = vq_synth.LayerSpec("tall", N=64 * times, K=K, d=d, b=b, Br=64, Bc=256, int8=True)
    W = torch.empty((tall.N, K), dtype=torch.float16, device="cuda")
    rep = [t.repeat(times, *[1] * (t.dim() - 1)) for t in (dev.idx, dev.cb, dev.scale)]
    torch.cuda.synchronize()
    vq.vq_decode_weights(lib_fmt(tall), *rep, W)
    torch.cuda.synchronize()
    assert bool((W.view(torch.int16).view(times, 64, K) == want).all())
