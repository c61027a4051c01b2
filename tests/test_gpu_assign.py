"""vq_assign_indices' two-pass kernel where its ranking cannot decide: exact ties, near ties, weights of zero or of either
sign, values out of range.  Byte for byte the oracle's stream."""
import numpy as np
import pytest

import vq_synth
from oracle import vq_oracle as orc
from tests.helpers import DeviceLayer, draw, oracle_fmt

vq = pytest.importorskip("paper_2402_15319_b200")
pytestmark = pytest.mark.gpu

SPECS = [
    vq_synth.LayerSpec("d1b4", N=40, K=512, d=1, b=4, Br=1, Bc=256, int8=True),
    vq_synth.LayerSpec("d2b4", N=36, K=1024, d=2, b=4, Br=4, Bc=512, int8=False),
    vq_synth.LayerSpec("d2b6", N=64, K=512, d=2, b=6, Br=32, Bc=128, int8=False),
    vq_synth.LayerSpec("d2b8", N=64, K=512, d=2, b=8, Br=64, Bc=256, int8=True),
    vq_synth.LayerSpec("d1b6", N=40, K=512, d=1, b=6, Br=8, Bc=256, int8=False),
    vq_synth.LayerSpec("d4b6", N=64, K=1024, d=4, b=6, Br=32, Bc=512, int8=False),
    vq_synth.LayerSpec("d4b5", N=36, K=1024, d=4, b=5, Br=4, Bc=256, int8=False),
    vq_synth.LayerSpec("d4b8", N=64, K=1024, d=4, b=8, Br=64, Bc=512, int8=True),
]


def _ties(spec, L, W, h):
    L.cb[:, 1::2] = L.cb[:, ::2]                     # every entry twice: the lower index wins
    return W, h


def _near(spec, L, W, h):
    W[:] = (np.float32(0.02) * np.sign(W.astype(np.float32))).astype(np.float16)   # few distinct vectors, many equal distances
    return W, h


def _small(spec, L, W, h):
    W[::2] = np.float16(6e-8) * np.sign(W[::2])      # subnormal inputs
    return W, h * np.float32(1e-36)


def _large(spec, L, W, h):
    W[::3] = np.float16(6e4)                         # all distances of a row within a few roundings
    return W, h * np.float32(1e18)


def _overflow(spec, L, W, h):
    W[::3] = np.float16(6e4)
    return W, h * np.float32(1e30)


def _special(spec, L, W, h):
    W[0, ::5], W[1, ::7], W[2, ::3] = np.nan, np.inf, -np.inf
    h = h.copy()
    h[::4], h[1::8], h[2::16] = 0.0, -1.0, np.inf
    h[3::64] = np.nan
    return W, h


def _far(spec, L, W, h):
    L.cb[:, 3] = 100 if spec.int8 else 1.0           # one centroid of every block far outside
    return W, h


def _dead(spec, L, W, h):
    """First weights of zero, entries that differ in their first value alone, values that repeat."""
    h = h.copy()
    h[::8 * spec.d] = 0.0
    L.cb[:, 1::3, 1:] = L.cb[:, :1, 1:]
    L.cb[:, 5::8] = L.cb[:, 2:3]
    return W, h


def _assign(f, W, cb, scale, h):
    """The oracle's sequence; a distance that is no number is never the smaller one (index 0 if none is)."""
    C = cb.reshape(f.n_blocks, f.entries, f.d).astype(np.float32)
    if scale is not None:
        C = C * scale.astype(np.float32).reshape(-1, 1, 1)
    x = W.astype(np.float32).reshape(f.N, f.K // f.d, f.d)
    D = np.ones(f.K, np.float32) if h is None else h
    D = D.reshape(f.K // f.d, f.d)
    I = np.empty((f.N, f.K // f.d), np.uint8)
    blk_col = np.arange(f.K // f.d) * f.d // f.Bc
    with np.errstate(all="ignore"):
        for n in range(f.N):
            c = C[(n // f.Br) * (f.K // f.Bc) + blk_col]                 # [vectors, entries, d]
            diff = x[n][:, None, :] - c
            term = D[:, None, :] * (diff * diff)
            acc = term[..., 0]
            for t in range(1, f.d):
                acc = acc + term[..., t]
            I[n] = np.argmin(np.where(np.isnan(acc), np.float32(np.inf), acc), axis=1)
    if np.isfinite(W.astype(np.float32)).all() and np.isfinite(D).all():
        assert np.array_equal(I, orc.assign(f, W, cb, scale, h))
    return I


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("change", [_ties, _near, _small, _large, _overflow, _special, _far, _dead], ids=lambda f: f.__name__[1:])
@pytest.mark.parametrize("spec", SPECS, ids=lambda s: s.name)
def test_undecided_rankings(spec, change, weighted):
    import torch
    f, L = oracle_fmt(spec), draw(spec, 91)
    W = (0.05 * vq_synth.normal(91, 40, spec.N * spec.K)).astype(np.float16).reshape(spec.N, spec.K)
    h = (0.25 + 2.0 * vq_synth.uniform01(91, 41, spec.K)).astype(np.float32)
    W, h = change(spec, L, W, h)
    h = h.astype(np.float32) if weighted else None
    want = orc.pack(f, _assign(f, W, L.cb, L.scale, h))
    dev = DeviceLayer(spec, L)
    d_idx = torch.full((spec.N, f.stride), 0x5A, dtype=torch.uint8, device="cuda")
    vq.vq_assign_indices(dev.fmt, torch.from_numpy(W).cuda(), dev.cb, dev.scale, None if h is None else torch.from_numpy(h).cuda(), d_idx)
    torch.cuda.synchronize()
    got = d_idx.cpu().numpy()
    assert np.array_equal(got, want), f"{np.count_nonzero(got != want)} of {got.size} bytes differ"
