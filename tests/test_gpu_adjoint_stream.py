"""An adjoint object made on a side stream: its tables are there before the
kernel that orders the backward's synapses reads them."""
import numpy as np
import pytest

from test_gpu_adjoint import _params, _setup, snn  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batched", ["0", "1"])
def test_created_on_a_side_stream(snn, monkeypatch, batched):
    import torch
    monkeypatch.setenv("SNN_ADJ_BATCHED", batched)
    grads = []
    for stream in (torch.cuda.default_stream(), torch.cuda.Stream()):
        with torch.cuda.stream(stream):
            a, onet, cfg, g, rt = _setup(snn, M=26000, K=100, T=40, ckpt=20, seed=61)
            G, lam, target = _params(a.n_pop, seed=4)
            r = a.forward(G, lam)
            grads.append(a.backward(2 * (r.astype(np.float64) - target) / a.n_pop))
            a.close()
    assert np.abs(grads[0][0]).max() > 0
    # the same order of the same sums but for the float64 additions at the end
    assert np.allclose(grads[0][0], grads[1][0], rtol=1e-9, atol=1e-15)
    assert np.allclose(grads[0][1], grads[1][1], rtol=1e-9, atol=1e-15)
