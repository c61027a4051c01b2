"""The E-step where the same columns of four rows share their weights: blocks of 4, 8, 16 and more rows, rows and columns that do not fill
a tile, every size class of codebook.  Byte for byte the oracle's stream."""
import numpy as np
import pytest

import vq_synth
from oracle import vq_oracle as orc
from tests.helpers import DeviceLayer, draw, oracle_fmt

vq = pytest.importorskip("paper_2402_15319_b200")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,d,b,Br,Bc,int8", [
    (4, 128, 2, 5, 4, 64, True), (44, 1152, 2, 5, 4, 128, False), (40, 640, 2, 6, 8, 128, True), (48, 576, 2, 7, 16, 64, False),
    (96, 1088, 2, 6, 32, 64, False), (384, 512, 2, 8, 128, 256, True), (40, 1280, 4, 6, 8, 256, False), (256, 2048, 4, 8, 128, 512, True),
])
def test_weighted(N, K, d, b, Br, Bc, int8):
    import torch
    spec = vq_synth.LayerSpec("rows", N=N, K=K, d=d, b=b, Br=Br, Bc=Bc, int8=int8)
    f, L = oracle_fmt(spec), draw(spec, 101)
    W = (0.05 * vq_synth.normal(101, 40, N * K)).astype(np.float16).reshape(N, K)
    h = (0.25 + 2.0 * vq_synth.uniform01(101, 41, K)).astype(np.float32)
    want = orc.pack(f, orc.assign(f, W, L.cb, L.scale, h))
    dev = DeviceLayer(spec, L)
    d_idx = torch.full((N, f.stride), 0x5A, dtype=torch.uint8, device="cuda")
    vq.vq_assign_indices(dev.fmt, torch.from_numpy(W).cuda(), dev.cb, dev.scale, torch.from_numpy(h).cuda(), d_idx)
    torch.cuda.synchronize()
    assert np.array_equal(d_idx.cpu().numpy(), want)
