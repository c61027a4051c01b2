"""Which calls the tcgen05 kernel serves: a call on either side of a line, for every set of lines; row tables at batches below 9, which are not
asked for by name.  Which kernel ran, and its outputs."""
import numpy as np
import pytest

import vq_synth
from oracle import vq_oracle as orc
from tests.helpers import DeviceLayer, assert_outputs_close, draw, kernels_launched, oracle_fmt

vq = pytest.importorskip("paper_2402_15319_b200")
pytestmark = pytest.mark.gpu

# N, K, d, b, Br, Bc, codebook type, [(batch, the tcgen05 kernel?)]
CALLS = {
    "row256_persistent": (8192, 4096, 2, 4, 1, 256, False, [(1, True), (3, True), (5, True), (7, True)]),
    "row256_cluster": (4096, 4096, 2, 4, 1, 256, False, [(1, False), (3, False), (6, True)]),
    "row256_short": (8192, 1024, 2, 4, 4, 256, True, [(2, False), (4, True), (9, True)]),
    "row512_cluster": (1024, 14336, 2, 4, 1, 512, True, [(1, False), (3, True), (5, True), (6, True)]),
    "row512_persistent": (8192, 4096, 2, 4, 4, 512, True, [(3, False), (6, False), (8, True), (9, True)]),
    "row512_5120": (8192, 5120, 2, 4, 1, 512, True, [(1, False), (4, True), (7, True)]),
    "row1024_short": (4096, 1024, 2, 4, 1, 1024, False, [(1, False), (3, True), (8, True)]),
    "row1024_long": (2048, 14336, 2, 4, 1, 1024, False, [(2, False), (5, True)]),
    "row2048_persistent": (8192, 4096, 2, 4, 1, 2048, True, [(6, False), (8, True), (10, True)]),
    "row2048_2048": (4608, 2048, 2, 4, 1, 2048, True, [(7, True), (11, True)]),
    "tall6": (8192, 4096, 2, 6, 128, 128, False, [(1, False), (5, False), (6, True)]),
    "tall6_long": (512, 6144, 2, 6, 128, 128, False, [(1, True)]),
    "tall6_int4": (5120, 4096, 2, 6, 128, 128, 2, [(2, False), (6, True)]),
    "warp6": (5120, 4096, 2, 6, 32, 256, True, [(1, False), (3, False), (8, True)]),
    "warp6_int4": (5120, 2048, 2, 6, 64, 128, 2, [(1, False), (6, True)]),
    "tall5": (5120, 4096, 2, 5, 128, 256, False, [(1, False), (4, True)]),
    "warp5_int4": (5120, 4096, 2, 5, 32, 256, 2, [(1, False), (3, True)]),
    "four_d": (8192, 2048, 4, 8, 256, 512, False, [(2, False), (4, True)]),
    "four_d_128": (1024, 1024, 4, 8, 128, 128, False, [(1, True)]),
    "small4": (4096, 1024, 2, 5, 4, 256, True, [(1, True), (3, False), (9, True)]),
    "small8": (5120, 2048, 2, 5, 8, 256, False, [(1, False), (16, False)]),
    "small16": (10240, 2048, 2, 5, 16, 512, True, [(2, False), (9, True)]),
    "ragged5": (8160, 1024, 2, 5, 32, 256, True, [(1, False), (9, True)]),
    "ragged6": (5024, 1024, 2, 6, 32, 128, False, [(1, False), (9, True)]),
    "ragged6_96": (5184, 4096, 2, 6, 96, 256, True, [(1, True)]),
}


@pytest.mark.parametrize("name", CALLS)
def test_either_side_of_a_line(name):
    import torch
    *shape, calls = CALLS[name]
    spec = vq_synth.LayerSpec(name, **dict(zip(("N", "K", "d", "b", "Br", "Bc", "int8"), shape)))
    L = draw(spec, 121)
    dev = DeviceLayer(spec, L)
    rows = np.unique(np.concatenate([np.arange(16), np.random.default_rng(9).integers(0, spec.N, 64), np.arange(spec.N - 16, spec.N)])).astype(np.int32)
    for batch, tile in calls:
        X = vq_synth.make_x(spec, 122, batch)
        Yg = dev.gemm(X)
        dX, dY = torch.from_numpy(X).cuda(), torch.empty((batch, spec.N), dtype=torch.float16, device="cuda")
        names = kernels_launched(lambda: vq.vq_gemm_small_batch(dev.fmt, dev.idx, dev.cb, dev.scale, dX, dY, batch, dev.ws))
        assert len(names) == 1 and ("tile_kernel" in names[0]) == tile, (batch, names)
        Y, A = orc.gemm(oracle_fmt(spec), L.idx, L.cb, L.scale, X, rows=rows, threads=8)
        assert_outputs_close(Yg[:, rows], Y, A, f"{name} batch {batch}")
        assert np.array_equal(dev.gemm(X).view(np.uint16), Yg.view(np.uint16))
    assert vq.vq_device_wait_failures() == 0


@pytest.mark.parametrize("rows,K,d,b,Br,Bc,cb,batch,tile", [
    ((4096, 1024, 1024), 4096, 2, 4, 1, 2048, True, 6, False),     # 24 x 2^20 weights: the persistent kernel's
    ((4096, 1024, 1024), 4096, 2, 4, 1, 256, False, 1, True),      # ... with blocks of 256 columns
    ((4096, 4096, 4096), 4096, 2, 6, 128, 128, False, 1, False),   # 48: as one layer of as many rows
    ((11008, 11008), 4096, 2, 6, 128, 128, False, 1, True),        # 86
], ids=str)
def test_groups_have_the_lines_of_layers(rows, K, d, b, Br, Bc, cb, batch, tile):
    import torch
    tmpl = dict(K=K, d=d, b=b, Br=Br, Bc=Bc, int8=cb)
    total = vq.VQFormat(sum(rows), K, d, b, Br, Bc, int(cb))
    specs = [vq_synth.LayerSpec(f"g{i}", N=n, **tmpl) for i, n in enumerate(rows)]
    X = vq_synth.make_x(specs[0], 131, batch)
    dX, ws = torch.from_numpy(X).cuda(), torch.zeros(vq.vq_workspace_bytes(total, batch), dtype=torch.uint8, device="cuda")
    layers, members, outs = [], [], []
    for i, spec in enumerate(specs):
        L = draw(spec, 130, i)
        dev = DeviceLayer(spec, L)
        outs.append(torch.full((batch, spec.N), float("nan"), dtype=torch.float16, device="cuda"))
        layers.append((spec, L, dev))
        members.append((dev.idx, dev.cb, dev.scale, outs[-1], spec.N))
    torch.cuda.synchronize()
    vq.vq_gemm_small_batch_grouped(total, members, dX, batch, ws)
    torch.cuda.synchronize()
    got = [y.cpu().numpy() for y in outs]
    names = kernels_launched(lambda: vq.vq_gemm_small_batch_grouped(total, members, dX, batch, ws))
    assert len(names) == vq.vq_grouped_kernel_launches(total, len(rows), batch) == 1 and ("tile_kernel" in names[0]) == tile, names
    if d == 2 and b == 6:   # one layer of the same rows goes the same way
        one = vq.VQFormat(sum(rows), K, d, b, Br, Bc, int(cb))
        info = vq.vq_pack_info(one)
        idx, book = torch.zeros(info.index_bytes, dtype=torch.uint8, device="cuda"), torch.zeros(info.codebook_bytes, dtype=torch.uint8, device="cuda")
        Y1 = torch.empty((batch, sum(rows)), dtype=torch.float16, device="cuda")
        alone = kernels_launched(lambda: vq.vq_gemm_small_batch(one, idx, book, None, dX, Y1, batch, ws))
        assert len(alone) == 1 and ("tile_kernel" in alone[0]) == tile, alone
    pick = np.unique(np.concatenate([np.arange(16), np.arange(500, 540), np.arange(min(rows) - 16, min(rows))])).astype(np.int32)
    for (spec, L, _), y in zip(layers, got):
        Y, A = orc.gemm(oracle_fmt(spec), L.idx, L.cb, L.scale, X, rows=pick, threads=8)
        assert_outputs_close(y[:, pick], Y, A, spec.name)
