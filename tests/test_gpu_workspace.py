"""One workspace serves calls of any format, height and batch in turn."""
import numpy as np
import pytest

import vq_synth
from tests.helpers import DeviceLayer, draw

vq = pytest.importorskip("paper_2402_15319_b200")
pytestmark = pytest.mark.gpu


def test_one_workspace_for_calls_of_different_heights():
    """A call with few rows leaves the counters of one with many rows alone (they share the start of the workspace)."""
    import torch
    layers = [vq_synth.LayerSpec("tall", N=18500, K=4096, d=2, b=4, Br=1, Bc=2048, int8=True), vq_synth.LayerSpec("short", N=256, K=8192, d=2, b=6, Br=128, Bc=128, int8=False)]
    devs = [DeviceLayer(s, draw(s, 81)) for s in layers]
    Xs = [vq_synth.make_x(s, 82, 16) for s in layers]
    impl = {"tall": vq.VQ_IMPL_TILE, "short": vq.VQ_IMPL_STREAM}
    alone = [d.gemm(X, impl[s.name]) for s, d, X in zip(layers, devs, Xs)]
    shared = torch.zeros_like(devs[0].ws)
    for d in devs:
        d.ws = shared
    for _ in range(3):
        for s, d, X, Y in zip(layers, devs, Xs, alone):
            assert np.array_equal(d.gemm(X, impl[s.name]).view(np.uint16), Y.view(np.uint16)), s.name


@pytest.mark.parametrize("spec", [
    vq_synth.LayerSpec("block", N=2048, K=4096, d=2, b=6, Br=128, Bc=128, int8=False),
    vq_synth.LayerSpec("block_warp", N=1024, K=4096, d=2, b=6, Br=32, Bc=256, int8=True),
    vq_synth.LayerSpec("block_4d", N=1024, K=4096, d=4, b=8, Br=256, Bc=512, int8=False),
    vq_synth.LayerSpec("row", N=1024, K=4096, d=2, b=4, Br=1, Bc=1024, int8=False),
    vq_synth.LayerSpec("row_1d", N=1024, K=4096, d=1, b=4, Br=1, Bc=2048, int8=True),
], ids=lambda s: s.name)
@pytest.mark.parametrize("members", [1, 2])
def test_host_calls_in_a_row_see_their_own_activations(spec, members):
    """Pinned-host calls enqueued one after the other on one workspace: a kernel is resident before the activations of its call
    replace those of the call before, at the same address."""
    import torch
    calls, batch = 24, 2
    dev = DeviceLayer(spec, draw(spec, 83))
    X = [torch.from_numpy(vq_synth.make_x(spec, 84 + i, batch)).pin_memory() for i in range(calls)]
    total = vq.VQFormat(*[getattr(dev.fmt, f) * (members if f == "n_rows" else 1) for f in
                          ("n_rows", "k_cols", "vq_dim", "index_bits", "block_rows", "block_cols")], dev.fmt.cb_type)
    ws = torch.zeros(vq.vq_workspace_bytes_grouped_host(total, members, batch), dtype=torch.uint8, device="cuda")

    def outputs():
        return [torch.zeros((batch, spec.N), dtype=torch.float16).pin_memory() for _ in range(members)]

    def call(x, ys):
        if members == 1:
            vq.vq_gemm_small_batch_host(dev.fmt, dev.idx, dev.cb, dev.scale, x, ys[0], batch, ws)
        else:
            vq.vq_gemm_small_batch_grouped_host(total, [(dev.idx, dev.cb, dev.scale, y, spec.N) for y in ys], x, batch, ws)

    alone = []
    for x in X:
        alone.append(outputs())
        call(x, alone[-1])
        torch.cuda.synchronize()
    for _ in range(4):
        got = [outputs() for _ in X]
        for x, ys in zip(X, got):
            call(x, ys)
        torch.cuda.synchronize()
        for i, (a, g) in enumerate(zip(alone, got)):
            for p, q in zip(a, g):
                assert torch.equal(p.view(torch.int16), q.view(torch.int16)), f"{spec.name} call {i}"
