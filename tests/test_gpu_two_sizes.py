"""Objects of different sizes in one process: the larger one, made first, runs
after the smaller one was made, as it does alone (the dynamic shared memory a
kernel may use is a limit of the function, shared by all objects)."""
import numpy as np
import pytest

import synth
from test_gpu_adjoint import _params, snn  # noqa: F401

pytestmark = pytest.mark.gpu


def _make(snn, M):
    cfg = synth.NetConfig(name="two", M=M, P=4, n_vn=2, K=20, uniform_all=True, dmax=4, seed=M,
                          dyn=synth.Dynamics(drive_lambda=1.1, w_ext=96, drive_seed=5))
    g = synth.make_network(cfg)
    net = snn.Network.from_synth(g)
    part, _ = snn.snn_partition(net, 4, "planted")
    return g, cfg, net, snn.Routing(net, part, 4, 2)


@pytest.mark.parametrize("delivery", ["0", "1", "3"])
def test_sims(snn, monkeypatch, delivery):
    monkeypatch.setenv("SNN_RESIDENT", "0")
    monkeypatch.setenv("SNN_DELIVERY", delivery)

    def make(M):
        g, cfg, net, rt = _make(snn, M)
        return snn.Sim(net, rt, snn.sim_params(cfg.dyn, raster_cap=M * 20, raster_steps=40), device="cuda:0")

    alone = make(60000)
    alone.step(40)
    want, raster = alone.read_state(), alone.read_raster(0, 40)
    alone.close()
    big = make(60000)
    small = make(1024)
    small.step(40)
    small.read_raster(0, 40)
    big.step(40)
    assert big.sync_status() == 0
    got, r2 = big.read_state(), big.read_raster(0, 40)
    assert np.array_equal(want[0].view(np.uint32), got[0].view(np.uint32)) and np.array_equal(want[1], got[1])
    assert np.array_equal(raster[0], r2[0]) and np.array_equal(raster[1], r2[1])


@pytest.mark.parametrize("batched", ["0", "1"])
def test_adjoints(snn, monkeypatch, batched):
    monkeypatch.setenv("SNN_ADJ_BATCHED", batched)
    G, lam, target = _params(4, seed=3)

    def make(M):
        g, cfg, net, rt = _make(snn, M)
        return snn.Adjoint(net, g.is_exc, rt, snn.sim_params(cfg.dyn, raster_cap=M * 30),
                           snn.adjoint_params(T=30, ckpt_every=10), device="cuda:0")

    def grads(a):
        r = a.forward(G, lam)
        return a.backward(2 * (r - target) / 4)

    alone = make(20000)
    want = grads(alone)
    alone.close()
    big = make(20000)
    small = make(1024)
    grads(small)
    got = grads(big)
    for w, x in zip(want, got):
        assert np.allclose(w, x, rtol=1e-12, atol=0)


def test_threads_read_one_sim(snn):
    """State, counters and raster of one sim read by several threads at once."""
    import threading
    g, cfg, net, rt = _make(snn, 20000)
    sim = snn.Sim(net, rt, snn.sim_params(cfg.dyn, raster_cap=20000 * 20, raster_steps=40), device="cuda:0")
    sim.step(40)
    want = sim.read_state()[0], sim.read_counts(), sim.read_raster(0, 40)[0]
    bad = []

    def read(k):
        for _ in range(100):
            if k % 3 == 0 and not np.array_equal(sim.read_state()[0], want[0]):
                bad.append("state")
            if k % 3 == 1 and sim.read_counts() != want[1]:
                bad.append("counts")
            if k % 3 == 2 and not np.array_equal(sim.read_raster(0, 40)[0], want[2]):
                bad.append("raster")

    ts = [threading.Thread(target=read, args=(k,)) for k in range(6)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad
