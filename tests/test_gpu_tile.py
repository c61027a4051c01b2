"""The tcgen05 kernel (vq_tile.cu) against the oracle, at sizes just above where it takes over from the other kernels:
row counts that end inside a tile, every table kind, codebook type and batch class."""
import numpy as np
import pytest

import vq_synth
from oracle import vq_oracle as orc
from tests.helpers import DeviceLayer, assert_outputs_close, draw, oracle_fmt

vq = pytest.importorskip("paper_2402_15319_b200")
pytestmark = pytest.mark.gpu


def _rows(N, n=48):
    edge = [r for t in (0, 128, N // 128 * 128, N) for r in range(t - 20, t + 20) if 0 <= r < N]
    return np.unique(np.concatenate([edge, np.random.default_rng(3).integers(0, N, n)])).astype(np.int32)


def _spec(name, N, K, d, b, Br, Bc, cb):
    return vq_synth.LayerSpec(name, N=N, K=K, d=d, b=b, Br=Br, Bc=Bc, int8=cb)


CASES = [
    # row tables (sums scaled per block), one row and four rows per block, a tile of 68 rows at the end
    (_spec("row_i8", 18500, 4096, 2, 4, 1, 2048, True), (13, 16)),
    (_spec("row_fp16", 18500, 4096, 2, 4, 1, 256, False), (13,)),
    (_spec("row4_i8", 18500, 4096, 2, 4, 4, 512, True), (16,)),
    # one table for the four warps
    (_spec("cta6_fp16", 11904, 4096, 2, 6, 128, 128, False), (9, 16)),
    (_spec("cta6_odd_k", 6272, 4224, 2, 6, 128, 128, True), (1, 8, 9)),
    (_spec("cta5_fp16", 20608, 4096, 2, 5, 128, 256, False), (9,)),
    (_spec("cta_4d_fp16", 13312, 5120, 4, 8, 256, 512, False), (9, 16)),
    (_spec("cta_4d_i8", 13312, 5120, 4, 8, 256, 512, True), (9,)),
    # a table per warp: 32-row blocks (rows end 96 short of a tile), INT4 codebooks, small blocks
    (_spec("warp6_i8", 6176, 4352, 2, 6, 32, 256, True), (1, 8, 9, 16)),
    (_spec("warp6_fp16", 6176, 4352, 2, 6, 32, 256, False), (3,)),
    (_spec("warp6_i4", 6176, 4224, 2, 6, 32, 128, 2), (1, 16)),
    (_spec("warp5_i4", 13088, 4352, 2, 5, 32, 256, 2), (5,)),
    (_spec("warp5_4", 13060, 4352, 2, 5, 4, 256, True), (1, 8, 9)),
    (_spec("warp5_8", 13072, 4352, 2, 5, 8, 256, False), (3,)),
    (_spec("warp5_16", 13072, 4352, 2, 5, 16, 256, True), (16,)),
]


@pytest.mark.parametrize("spec,batches", CASES, ids=lambda v: v.name if hasattr(v, "name") else None)
def test_tile_kernel_against_oracle(spec, batches):
    L = draw(spec, 61)
    dev = DeviceLayer(spec, L)
    rows = _rows(spec.N)
    for batch in batches:
        X = vq_synth.make_x(spec, 62, batch)
        Y, A = orc.gemm(oracle_fmt(spec), L.idx, L.cb, L.scale, X, rows=rows, threads=8)
        Yg = dev.gemm(X)
        assert_outputs_close(Yg[:, rows], Y, A, f"{spec.name} batch {batch}")
        assert np.isfinite(Yg.astype(np.float32)).all()
        assert np.array_equal(dev.gemm(X).view(np.uint16), Yg.view(np.uint16))   # bit-identical, whoever draws the last ticket
    assert vq.vq_device_wait_failures() == 0


def test_tile_kernel_group_of_ragged_layers():
    import torch
    rows, K, batch = (3328, 416, 96), 3328, 5
    tmpl = dict(K=K, d=2, b=6, Br=32, Bc=128, int8=2)
    fmt = vq.VQFormat(sum(rows), K, 2, 6, 32, 128, vq.VQ_CB_INT4_G128)
    assert vq.vq_grouped_kernel_launches(fmt, len(rows), batch) == 1
    specs = [vq_synth.LayerSpec(f"grp{i}", N=n, **tmpl) for i, n in enumerate(rows)]
    X = vq_synth.make_x(specs[0], 71, batch)
    dX, ws = torch.from_numpy(X).cuda(), torch.zeros(vq.vq_workspace_bytes(fmt, batch), dtype=torch.uint8, device="cuda")
    members, keep = [], []
    for i, spec in enumerate(specs):
        L = draw(spec, 70, i)
        dY = torch.full((batch, spec.N), float("nan"), dtype=torch.float16, device="cuda")
        members.append((torch.from_numpy(L.idx).cuda(), torch.from_numpy(L.cb).cuda(), torch.from_numpy(L.scale).cuda(), dY, spec.N))
        keep.append((spec, L, dY))
    torch.cuda.synchronize()
    vq.vq_gemm_small_batch_grouped(fmt, members, dX, batch, ws)
    torch.cuda.synchronize()
    for spec, L, dY in keep:
        Y, A = orc.gemm(oracle_fmt(spec), L.idx, L.cb, L.scale, X, threads=8)
        assert_outputs_close(dY.cpu().numpy(), Y, A, spec.name)


@pytest.mark.parametrize("spec,batch", [
    (_spec("row_fp16_long", 7424, 14336, 2, 4, 1, 256, False), 16),
    (_spec("row_i8_long", 9728, 11008, 2, 4, 1, 256, True), 16),
    (_spec("warp6_i4_long", 14784, 7168, 2, 6, 96, 256, 2), 10),
], ids=lambda v: v.name if hasattr(v, "name") else None)
def test_every_launch_reads_its_indices_before_they_are_replaced(spec, batch):
    """Launches in a row, all rows of all of them bit-identical: the index bytes of a unit are read before their stage is refilled
    (where a table changes with every unit, the warps wait for global memory between the two)."""
    import torch
    L = draw(spec, 63)
    dev = DeviceLayer(spec, L)
    X = vq_synth.make_x(spec, 64, batch)
    dX = torch.from_numpy(X).cuda()
    Ys = torch.empty((60, batch, spec.N), dtype=torch.float16, device="cuda")
    torch.cuda.synchronize()
    for Y in Ys:
        vq.vq_gemm_small_batch(dev.fmt, dev.idx, dev.cb, dev.scale, dX, Y, batch, dev.ws)
    torch.cuda.synchronize()
    same = (Ys.view(torch.int16) == Ys[0].view(torch.int16)).flatten(1).all(1)
    assert bool(same.all()), f"{int((~same).sum())} of {len(Ys)} launches differ from the first"
    rows = _rows(spec.N)
    Y, A = orc.gemm(oracle_fmt(spec), L.idx, L.cb, L.scale, X, rows=rows, threads=8)
    assert_outputs_close(Ys[0].cpu().numpy()[:, rows], Y, A, spec.name)
