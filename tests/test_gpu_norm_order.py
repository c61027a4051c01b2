"""The normalised product is ordered by its stream alone: codes, scale table and indices may be written by kernels directly in front of
it, the scale table even by a product call that lets its successor start early; captured in a graph too."""
import numpy as np
import pytest

import vq_synth
from oracle import vq_oracle as orc
from tests.helpers import DeviceLayer, assert_outputs_close, draw, kernels_launched, oracle_fmt

vq = pytest.importorskip("paper_2402_15319_b200")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,Br,Bc,cols,kernel", [
    (14336, 4096, 32, 256, 32, "tile_kernel"), (16384, 2048, 128, 128, 64, "tile_kernel"), (1024, 1024, 32, 256, 32, "warptab_kernel"),
])
def test_reads_what_the_stream_wrote_before_it(N, K, Br, Bc, cols, kernel):
    import torch
    spec = vq_synth.LayerSpec("order", N=N, K=K, d=2, b=6, Br=Br, Bc=Bc, int8=True)
    L = draw(spec, 111)
    dev = DeviceLayer(spec, L)
    codes, _ = vq_synth.make_norm(spec, cols, seed=112)
    # the scale table is the output of a product: 16 rows a codebook block, 128 columns
    lut_spec = vq_synth.LayerSpec("table", N=spec.n_blocks * 16, K=128, d=2, b=6, Br=128, Bc=128, int8=False)
    table = DeviceLayer(lut_spec, draw(lut_spec, 113), max_batch=1)
    V = 4
    code_masks, index_masks = (0x00, 0xFF, 0x3C, 0xA5), (0x00, 0x5A, 0xFF, 0x0F)
    dX = torch.from_numpy(vq_synth.make_x(spec, 114, 2)).cuda()
    tX = torch.from_numpy(vq_synth.make_x(lut_spec, 115, V)).cuda()
    codes0, idx0 = torch.from_numpy(codes).cuda(), dev.idx.clone()
    d_codes, d_idx = torch.empty_like(codes0), torch.empty_like(idx0)
    d_lut = torch.empty((1, spec.n_blocks * 16), dtype=torch.float16, device="cuda")
    torch.cuda.synchronize()

    def step(v, order, Y, between=lambda: None):
        def index():
            torch.bitwise_xor(idx0, index_masks[v], out=d_idx)

        def code():
            torch.bitwise_xor(codes0, code_masks[v], out=d_codes)

        def lut():   # the tcgen05 kernel, whose dependents may start while it runs
            vq.vq_gemm_small_batch_impl(table.fmt, table.idx, table.cb, table.scale, tX[v:v + 1], d_lut, 1, table.ws, vq.VQ_IMPL_TILE)
        for producer in ((index, code, lut), (lut, index, code), (code, lut, index))[order]:
            producer()
            between()
        vq.vq_gemm_small_batch_normalized(dev.fmt, d_idx, dev.cb, dev.scale, d_codes, d_lut, cols, dX, Y, 2)

    Ys = torch.full((60, 2, N), float("nan"), dtype=torch.float16, device="cuda")
    want = torch.empty((V, 2, N), dtype=torch.float16, device="cuda")
    tables = []
    for v in range(V):   # each variant alone, every producer complete before the next step
        step(v, 0, want[v], torch.cuda.synchronize)
        torch.cuda.synchronize()
        tables.append(d_lut.cpu().numpy().reshape(-1, 16))
    names = kernels_launched(lambda: vq.vq_gemm_small_batch_normalized(dev.fmt, d_idx, dev.cb, dev.scale, d_codes, d_lut, cols, dX, want[0], 2))
    assert len(names) == 1 and kernel in names[0], names
    torch.cuda.synchronize()
    for i, Y in enumerate(Ys):
        step(i % V, i // V % 3, Y)
    torch.cuda.synchronize()
    for i, Y in enumerate(Ys):
        assert torch.equal(Y.view(torch.int16), want[i % V].view(torch.int16)), f"launch {i}"
    graph = torch.cuda.CUDAGraph()   # the same row of calls captured
    with torch.cuda.graph(graph):
        for i, Y in enumerate(Ys):
            step(i % V, i // V % 3, Y)
    for replay in range(3):
        Ys.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        for i, Y in enumerate(Ys):
            assert torch.equal(Y.view(torch.int16), want[i % V].view(torch.int16)), f"captured launch {i}, replay {replay}"

    rows = np.unique(np.concatenate([np.arange(8), np.random.default_rng(7).integers(0, N, 56), np.arange(N - 8, N)])).astype(np.int32)
    for v in range(V):
        W, _ = orc.normalized_decode(oracle_fmt(spec), (L.idx ^ np.uint8(index_masks[v])), L.cb, L.scale, codes ^ np.uint8(code_masks[v]), tables[v], cols)
        Wr, X = W[rows].astype(np.float64), dX.cpu().numpy().astype(np.float64)
        assert_outputs_close(want[v].cpu().numpy()[:, rows], X @ Wr.T, np.abs(X) @ np.abs(Wr).T, f"variant {v}")
    assert vq.vq_device_wait_failures() == 0
