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
    impl = {"tall": vq.VQ_IMPL_AUTO, "short": vq.VQ_IMPL_STREAM}
    alone = [d.gemm(X, impl[s.name]) for s, d, X in zip(layers, devs, Xs)]
    shared = torch.zeros_like(devs[0].ws)
    for d in devs:
        d.ws = shared
    for _ in range(3):
        for s, d, X, Y in zip(layers, devs, Xs, alone):
            assert np.array_equal(d.gemm(X, impl[s.name]).view(np.uint16), Y.view(np.uint16)), s.name
