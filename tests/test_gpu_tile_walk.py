"""The tcgen05 kernel's walk: pieces of tiles that meet in the workspace, whole tiles beside them, units that do not divide among
the four groups of decoding warps; row tables below batch 9; block-wise normalisation."""
import numpy as np
import pytest

import vq_synth
from oracle import vq_oracle as orc
from tests.helpers import DeviceLayer, assert_outputs_close, draw, guarded, assert_guards_intact, kernels_launched, oracle_fmt

vq = pytest.importorskip("paper_2402_15319_b200")
pytestmark = pytest.mark.gpu


def _spec(name, N, K, d, b, Br, Bc, cb):
    return vq_synth.LayerSpec(name, N=N, K=K, d=d, b=b, Br=Br, Bc=Bc, int8=cb)


def _rows(N):
    edge = [r for t in (0, 128, N // 128 * 128, N) for r in range(t - 12, t + 12) if 0 <= r < N]
    return np.unique(np.concatenate([edge, np.random.default_rng(5).integers(0, N, 64)])).astype(np.int32)


@pytest.mark.parametrize("spec,batches", [
    # one CTA per tile, several pieces a tile of equal length, pieces that cross tiles (148 CTAs)
    (_spec("equal_pieces", 4096, 4096, 2, 6, 128, 128, False), (1, 9)),
    (_spec("crossing", 5120, 5120, 4, 8, 256, 512, False), (8, 16)),
    (_spec("crossing_i4", 3328, 9088, 2, 6, 32, 128, 2), (5, 13)),
    # 1, 2, 3, 5 units: some groups of warps have none
    (_spec("units1", 256, 128, 2, 6, 128, 128, True), (1, 16)),
    (_spec("units3", 384, 384, 2, 6, 32, 128, False), (4, 12)),
    (_spec("units5", 200, 1280, 2, 5, 4, 256, True), (3, 9)),
    # whole tiles and a left-over tile shared by eight CTAs, by one
    (_spec("whole_and_shared", 149 * 128, 2048, 2, 6, 128, 128, False), (2, 16)),
    (_spec("whole_only", 296 * 128, 512, 2, 4, 1, 512, True), (11,)),
], ids=lambda v: v.name if hasattr(v, "name") else None)
def test_pieces(spec, batches):
    L = draw(spec, 91)
    dev = DeviceLayer(spec, L)
    rows = _rows(spec.N)
    for batch in batches:
        X = vq_synth.make_x(spec, 92, batch)
        Y, A = orc.gemm(oracle_fmt(spec), L.idx, L.cb, L.scale, X, rows=rows, threads=8)
        first = dev.gemm(X, vq.VQ_IMPL_TILE)
        assert_outputs_close(first[:, rows], Y, A, f"{spec.name} batch {batch}")
        for _ in range(3):
            assert np.array_equal(dev.gemm(X, vq.VQ_IMPL_TILE).view(np.uint16), first.view(np.uint16))
    assert vq.vq_device_wait_failures() == 0


@pytest.mark.parametrize("spec,batches", [
    # sums of many short tiles, read while the next ones are multiplied: 1, 2, 3 and 4 units a tile (quads without any), 3 or 4 tiles a CTA
    (_spec("units1", 444 * 128 - 32, 128, 2, 6, 32, 128, 2), (1, 16)),
    (_spec("units2", 500 * 128, 256, 2, 6, 128, 128, True), (7, 16)),
    (_spec("units3", 450 * 128 - 96, 384, 2, 6, 32, 128, False), (4, 13)),
    (_spec("units4_4d", 444 * 128, 512, 4, 8, 128, 128, False), (9, 16)),
    (_spec("units2_5b", 592 * 128 - 4, 512, 2, 5, 4, 256, True), (5, 12)),
    # a tile and a quarter per CTA: pieces that cross left-over tiles, whose shares are added beside the whole ones
    (_spec("crossing_beside", 185 * 128, 2816, 2, 6, 128, 128, True), (3, 16)),
    (_spec("crossing_beside_w", 185 * 128 - 64, 2816, 2, 6, 32, 256, False), (1, 10)),
], ids=lambda v: v.name if hasattr(v, "name") else None)
def test_sums_of_every_tile(spec, batches):
    L = draw(spec, 98)
    dev = DeviceLayer(spec, L)
    for batch in batches:
        X = vq_synth.make_x(spec, 99, batch)
        Y, A = orc.gemm(oracle_fmt(spec), L.idx, L.cb, L.scale, X, threads=8)
        first = dev.gemm(X, vq.VQ_IMPL_TILE)
        assert_outputs_close(first, Y, A, f"{spec.name} batch {batch}")
        for _ in range(3):
            assert np.array_equal(dev.gemm(X, vq.VQ_IMPL_TILE).view(np.uint16), first.view(np.uint16))
    assert vq.vq_device_wait_failures() == 0


@pytest.mark.parametrize("cb,bc", [(True, 2048), (False, 1024)])
def test_row_tables_at_batch_8(cb, bc):
    import torch
    spec = _spec("rows", 57344, 4096, 2, 4, 1, bc, cb)
    L = draw(spec, 93)
    dev = DeviceLayer(spec, L)
    X = vq_synth.make_x(spec, 94, 8)
    dX, Y = torch.from_numpy(X).cuda(), torch.empty((8, spec.N), dtype=torch.float16, device="cuda")
    names = kernels_launched(lambda: vq.vq_gemm_small_batch(dev.fmt, dev.idx, dev.cb, dev.scale, dX, Y, 8, dev.ws))
    assert len(names) == 1 and "tile_kernel" in names[0], names
    rows = _rows(spec.N)
    ref, A = orc.gemm(oracle_fmt(spec), L.idx, L.cb, L.scale, X, rows=rows, threads=8)
    assert_outputs_close(dev.gemm(X)[:, rows], ref, A, spec.name)
    assert vq.vq_device_wait_failures() == 0


@pytest.mark.parametrize("spec", [
    _spec("warp_i8", 13344, 4096, 2, 6, 32, 256, True),
    _spec("warp_fp16_odd", 19072, 3328, 2, 6, 64, 128, False),
    _spec("cta_fp16", 14336, 4096, 2, 6, 128, 128, False),
    _spec("two_tiles_a_cta", 22016, 2048, 2, 6, 256, 256, True),
], ids=lambda v: v.name)
@pytest.mark.parametrize("cols", [16, 32, 64])
def test_normalised(spec, cols):
    import torch
    L = draw(spec, 95)
    dev = DeviceLayer(spec, L)
    codes, lut = vq_synth.make_norm(spec, cols, seed=96)
    dc, dl = torch.from_numpy(codes).cuda(), torch.from_numpy(lut).cuda()
    for batch in (1, 8, 9, 16):
        X = vq_synth.make_x(spec, 97, batch)
        dX = torch.from_numpy(X).cuda()
        dY, raw = guarded((batch, spec.N), torch.float16, "cuda")
        torch.cuda.synchronize()
        vq.vq_gemm_small_batch_normalized(dev.fmt, dev.idx, dev.cb, dev.scale, dc, dl, cols, dX, dY, batch)
        torch.cuda.synchronize()
        assert_guards_intact(raw, spec.name)
        if batch in (1, 9):
            W, _ = orc.normalized_decode(oracle_fmt(spec), L.idx, L.cb, L.scale, codes, lut, cols)
            rows = _rows(spec.N)
            Wr = W[rows].astype(np.float64)
            ref, A = X.astype(np.float64) @ Wr.T, np.abs(X.astype(np.float64)) @ np.abs(Wr).T
            assert_outputs_close(dY.cpu().numpy()[:, rows], ref, A, f"{spec.name} {cols} batch {batch}")
        assert np.isfinite(dY.float().cpu().numpy()).all()
    assert vq.vq_device_wait_failures() == 0


def _normalised_rows(spec, L, codes, lut, cols, r0, n):
    """Rows r0 .. r0 + n - 1 of the normalised weights, in binary64 (whole codebook blocks)."""
    part = vq_synth.LayerSpec("part", N=n, K=spec.K, d=spec.d, b=spec.b, Br=spec.Br, Bc=spec.Bc, int8=spec.int8)
    across = spec.K // spec.Bc
    blocks = slice(r0 // spec.Br * across, (r0 + n) // spec.Br * across)
    W, _ = orc.normalized_decode(oracle_fmt(part), L.idx[r0:r0 + n], L.cb.reshape(spec.n_blocks, -1)[blocks],
                                 None if L.scale is None else L.scale[blocks], codes[r0:r0 + n], lut[blocks], cols)
    return W.astype(np.float64)


@pytest.mark.parametrize("spec,kernel", [
    (_spec("warp_i8", 16384, 4096, 2, 6, 32, 256, True), "tile_kernel"),
    (_spec("warp_fp16_odd", 18880, 3456, 2, 6, 32, 128, False), "tile_kernel"),
    (_spec("warp64_fp16_7_units", 18944, 896, 2, 6, 64, 128, False), "tile_kernel"),
    (_spec("cta_fp16", 16384, 4096, 2, 6, 128, 128, False), "tile_kernel"),
    (_spec("two_tiles_a_cta", 37888, 2048, 2, 6, 256, 256, True), "tile_kernel"),
    (_spec("one_tile_too_many", 19072, 3328, 2, 6, 64, 128, False), "warptab_kernel"),   # 149 tiles on 148 SMs
], ids=lambda v: v.name if hasattr(v, "name") else v)
@pytest.mark.parametrize("cols", [16, 32, 64])
def test_normalised_in_the_kernel_it_claims(spec, kernel, cols):
    import torch
    L = draw(spec, 95)
    dev = DeviceLayer(spec, L)
    codes, lut = vq_synth.make_norm(spec, cols, seed=96)
    dc, dl = torch.from_numpy(codes).cuda(), torch.from_numpy(lut).cuda()
    parts = [(r0, _normalised_rows(spec, L, codes, lut, cols, r0, 512)) for r0 in (0, (spec.N - 512) // 2 // 256 * 256, spec.N - 512)]
    for batch in (1, 8, 9, 16):
        X = vq_synth.make_x(spec, 97, batch)
        dX = torch.from_numpy(X).cuda()
        dY, raw = guarded((batch, spec.N), torch.float16, "cuda")
        torch.cuda.synchronize()
        call = lambda: vq.vq_gemm_small_batch_normalized(dev.fmt, dev.idx, dev.cb, dev.scale, dc, dl, cols, dX, dY, batch)  # noqa: E731
        names = kernels_launched(call)
        assert len(names) == 1 and kernel in names[0], names
        call()
        torch.cuda.synchronize()
        assert_guards_intact(raw, spec.name)
        Y, X64 = dY.cpu().numpy(), X.astype(np.float64)
        assert np.isfinite(Y.astype(np.float32)).all()
        for r0, W in parts:
            assert_outputs_close(Y[:, r0:r0 + 512], X64 @ W.T, np.abs(X64) @ np.abs(W).T, f"{spec.name} {cols} batch {batch} rows from {r0}")
    assert vq.vq_device_wait_failures() == 0
