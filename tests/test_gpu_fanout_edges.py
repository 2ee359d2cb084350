"""snn_deliver_spikes at the edges of its split: out-degrees from 0 to over a
lane batch of several warps, one spike (shared by eight warps) up to more
spikes than warps, an id out of range among valid ones; planted and reordered
networks, against a brute-force fan-out."""
import numpy as np
import pytest

import synth
from test_gpu_fanout import _brute, snn  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reordered", [False, True])
@pytest.mark.parametrize("n", [1, 5, 607, 9001])
def test_degrees_and_spike_counts(snn, n, reordered):
    import torch
    rng = np.random.default_rng(n)
    M, P = 1201, 4
    deg = rng.choice([0, 1, 31, 33, 255, 257, 700], M)
    edges = [(i, int(t), int(w), int(d)) for i in range(M)
             for t, w, d in zip(rng.integers(0, M, deg[i]), rng.integers(-200, 60, deg[i]), rng.integers(1, 9, deg[i]))]
    g = synth.make_edges(M, edges)
    net = snn.Network.from_synth(g)
    part = (rng.permutation(M) % P if reordered else np.arange(M) * P // M).astype(np.int32)
    rt = snn.Routing(net, part, P, 2)
    sim = snn.Sim(net, rt, snn.sim_params(g.cfg.dyn), device="cuda:0")
    ids = rng.integers(0, M, n).astype(np.int32)
    out = torch.zeros((8, M), dtype=torch.int32, device="cuda:0")
    try:
        l1, l2, ev = sim.deliver_spikes(torch.from_numpy(ids).to("cuda:0"), out)
        assert n < M
        assert ev == int(deg[ids].sum())
        assert l1 == sum(len({int(part[t]) // 2 for t in g.tgt[g.syn_ptr[i]:g.syn_ptr[i + 1]]}) for i in ids)
        assert l2 == sum(len({int(part[t]) for t in g.tgt[g.syn_ptr[i]:g.syn_ptr[i + 1]]}) for i in ids)
    except snn.SnnError as e:  # more entries than every neuron spiking once needs
        assert n > M and e.code == snn.SNN_E_CAPACITY
    assert np.array_equal(out.cpu().numpy(), _brute(g, ids, 8))
    bad = torch.tensor([3, M, 5], dtype=torch.int32, device="cuda:0")
    out.zero_()
    with pytest.raises(snn.SnnError):
        sim.deliver_spikes(bad, out)
    assert np.array_equal(out.cpu().numpy(), _brute(g, np.array([3, 5]), 8))
