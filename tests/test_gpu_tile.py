"""The tcgen05 kernel (vq_tile.cu) against the oracle: at sizes near where it takes over from the other kernels, at the edges of its
tiles and with more tiles than CTAs; every table kind, codebook type and batch class."""
import numpy as np
import pytest

import vq_synth
from oracle import vq_oracle as orc
from tests.helpers import DeviceLayer, assert_outputs_close, draw, kernels_launched, oracle_fmt

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
        for impl in (vq.VQ_IMPL_TILE, vq.VQ_IMPL_AUTO):
            Yg = dev.gemm(X, impl)
            assert_outputs_close(Yg[:, rows], Y, A, f"{spec.name} batch {batch} impl {impl}")
            assert np.isfinite(Yg.astype(np.float32)).all()
            assert np.array_equal(dev.gemm(X, impl).view(np.uint16), Yg.view(np.uint16))   # bit-identical, whoever draws the last ticket
    assert vq.vq_device_wait_failures() == 0


def test_tile_kernel_group_of_ragged_layers():
    import torch
    rows, K, batch = (3328, 416, 96), 3328, 5
    tmpl = dict(K=K, d=2, b=6, Br=32, Bc=128, int8=2)
    fmt = vq.VQFormat(sum(rows), K, 2, 6, 32, 128, vq.VQ_CB_INT4_G128)
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
    names = kernels_launched(lambda: vq.vq_gemm_small_batch_grouped(fmt, members, dX, batch, ws))
    assert len(names) == 1 and "tile_kernel" in names[0], names
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
        vq.vq_gemm_small_batch_impl(dev.fmt, dev.idx, dev.cb, dev.scale, dX, Y, batch, dev.ws, vq.VQ_IMPL_TILE)
    torch.cuda.synchronize()
    same = (Ys.view(torch.int16) == Ys[0].view(torch.int16)).flatten(1).all(1)
    assert bool(same.all()), f"{int((~same).sum())} of {len(Ys)} launches differ from the first"
    rows = _rows(spec.N)
    Y, A = orc.gemm(oracle_fmt(spec), L.idx, L.cb, L.scale, X, rows=rows, threads=8)
    assert_outputs_close(Ys[0].cpu().numpy()[:, rows], Y, A, spec.name)


KINDS = {   # d, b, Br, Bc, codebook type; every instantiation of the kernel
    "row_fp16": (2, 4, 1, 256, False), "row4_i8": (2, 4, 4, 512, True),
    "cta6_fp16": (2, 6, 128, 128, False), "cta6_i8": (2, 6, 256, 256, True), "cta6_i4": (2, 6, 128, 128, 2),
    "cta5_i8": (2, 5, 128, 256, True), "cta5_i4": (2, 5, 256, 256, 2),
    "cta_4d_fp16": (4, 8, 128, 128, False), "cta_4d_i8": (4, 8, 256, 256, True),
    "warp6_fp16": (2, 6, 32, 128, False), "warp6_i8": (2, 6, 96, 256, True), "warp6_i4": (2, 6, 64, 128, 2),
    "warp5_i8": (2, 5, 32, 256, True), "warp5_i4": (2, 5, 32, 256, 2),
    "warp5_4": (2, 5, 4, 256, False), "warp5_8": (2, 5, 8, 256, True), "warp5_16": (2, 5, 16, 256, True),
}


def _forced(spec, batches, seed):
    L = draw(spec, seed)
    dev = DeviceLayer(spec, L)
    for batch in batches:
        X = vq_synth.make_x(spec, seed + 1, batch)
        Y, A = orc.gemm(oracle_fmt(spec), L.idx, L.cb, L.scale, X, threads=8)
        assert_outputs_close(dev.gemm(X, vq.VQ_IMPL_TILE), Y, A, f"{spec.name} {spec.N} x {spec.K} batch {batch}")
    assert vq.vq_device_wait_failures() == 0


@pytest.mark.parametrize("kind", KINDS)
def test_tile_kernel_edges(kind):
    """One unit of columns, an odd number of units, a tile that is not full, one row (block) more than a tile."""
    d, b, Br, Bc, cb = KINDS[kind]
    for blocks, cols in ((1, 1), (1, 5), (max(1, 96 // Br), 2), (128 // Br + 1, 3)):
        _forced(_spec(kind, Br * blocks, Bc * cols, d, b, Br, Bc, cb), (9, 16) if d == 2 and b == 4 else (1, 8, 9, 16), 65)


@pytest.mark.parametrize("rows", [75776, 75776 + 256, 2 * 75776 + 1280])
@pytest.mark.parametrize("kind", ["row_fp16", "row4_i8", "cta6_i8", "cta_4d_fp16", "warp6_i4", "warp5_8"])
def test_tile_kernel_whole_tiles(kind, rows):
    """More tiles than CTAs (one per SM, 148): whole tiles per CTA, without tiles left over and with some (an output layer)."""
    d, b, Br, Bc, cb = KINDS[kind]
    rows = rows // Br * Br
    _forced(_spec(kind, rows, Bc * (1 if rows < 80000 else 2), d, b, Br, Bc, cb), (11,), 67)


def test_tile_kernel_refuses_what_it_does_not_cover():
    spec = _spec("row", 64, 512, 2, 4, 1, 512, True)
    dev = DeviceLayer(spec, draw(spec, 69))
    for what, batch in ((dev, 8), (DeviceLayer(_spec("b3", 64, 512, 2, 3, 1, 512, True), draw(_spec("b3", 64, 512, 2, 3, 1, 512, True), 69)), 9)):
        with pytest.raises(vq.VQError) as e:
            what.gemm(vq_synth.make_x(what.spec, 70, batch), vq.VQ_IMPL_TILE)
        assert e.value.code == 7


@pytest.mark.parametrize("spec,batch", [
    (_spec("70b_qkv_gate", 20480, 8192, 2, 4, 1, 2048, True), 16),
    (_spec("7b_gate", 22016, 4096, 2, 6, 128, 128, False), 16),
    (_spec("13b_gate", 27648, 5120, 4, 8, 256, 512, False), 8),
    (_spec("8b_gate", 28672, 4096, 2, 6, 32, 256, True), 1),
    (_spec("8b_gate_5", 28672, 4096, 2, 5, 4, 256, True), 3),
], ids=lambda v: v.name if hasattr(v, "name") else None)
def test_large_layers_are_sent_to_the_tile_kernel(spec, batch):
    import torch
    info = vq.vq_pack_info(vq.VQFormat(spec.N, spec.K, spec.d, spec.b, spec.Br, spec.Bc, int(spec.int8)))
    idx = torch.zeros(info.index_bytes, dtype=torch.uint8, device="cuda")
    cb = torch.zeros(info.codebook_bytes, dtype=torch.uint8, device="cuda")
    sc = torch.zeros(max(info.scale_bytes, 16), dtype=torch.uint8, device="cuda") if spec.int8 else None
    fmt = vq.VQFormat(spec.N, spec.K, spec.d, spec.b, spec.Br, spec.Bc, int(spec.int8))
    X, Y = (torch.zeros((batch, n), dtype=torch.float16, device="cuda") for n in (spec.K, spec.N))
    ws = torch.zeros(vq.vq_workspace_bytes(fmt, batch), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    vq.vq_gemm_small_batch(fmt, idx, cb, sc, X, Y, batch, ws)
    names = kernels_launched(lambda: vq.vq_gemm_small_batch(fmt, idx, cb, sc, X, Y, batch, ws))
    assert len(names) == 1 and "tile_kernel" in names[0], names
