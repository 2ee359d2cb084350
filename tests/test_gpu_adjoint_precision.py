"""The gradients' error against 64 bits where roundings could add up: two
weights only, and gains for which weight times gain, rounded to float32, is
too large by nearly half a unit in the last place for every synapse.  Products
rounded like that once for all steps shift the gradients by 3.5e-7; rounded
term by term (the gain times the adjoint, then the weight) the errors differ
in sign and leave 2.2e-8 (both from a float32 model of the backward).  The
bound lies between."""
import numpy as np
import pytest

import oracle
import oracle.adjoint as adj
import synth
from test_gpu_adjoint import snn  # noqa: F401

pytestmark = pytest.mark.gpu

WEIGHTS = (81, -83)


def _gains(n_pop):
    G = np.empty((n_pop, n_pop), np.float32)
    for a in range(n_pop):
        for b in range(n_pop):
            w = WEIGHTS[b % 2]
            x = np.float32(1.1 + 0.05 * a + 0.03 * b) + np.arange(4000, dtype=np.float32) * np.float32(2 ** -23)
            exact = w * x.astype(np.float64)
            G[a, b] = x[np.argmax(((np.float32(w) * x).astype(np.float64) - exact) / exact)]
    return G


@pytest.fixture(scope="module")
def case():
    M, P, n_vn, T = 16384, 4, 2, 300
    cfg = synth.NetConfig(name="adjp", M=M, P=P, n_vn=n_vn, K=64, uniform_all=True, dmax=8, seed=5,
                          dyn=synth.Dynamics(w_ext=89, drive_seed=4000))
    g = synth.make_network(cfg)
    g.w[:] = np.where(np.repeat(g.is_exc, np.diff(g.syn_ptr)) != 0, *WEIGHTS)
    net = adj.from_synth(g, cfg.dyn, oracle.partition_planted(M, P), oracle.group_contiguous(P, n_vn),
                         oracle.alpha32(cfg.dyn.dt_ms, cfg.dyn.tau_ms))
    G, lam = _gains(2 * n_vn), np.full(2 * n_vn, 0.85, np.float32)
    tr = adj.forward_fp32(net, G, lam, T)
    grates = T * net.pop_sizes() * 2.0 ** -20  # (a neuron's share of it is a power of two: no rounding there)
    return cfg, g, G, lam, T, grates, adj.backward(net, G, lam, tr, grates)


@pytest.mark.parametrize("batched", ["0", "1"])
def test_roundings_do_not_add_up(snn, monkeypatch, case, batched):
    monkeypatch.setenv("SNN_ADJ_BATCHED", batched)
    cfg, g, G, lam, T, grates, (oG, olam) = case
    net = snn.Network.from_synth(g)
    part, _ = snn.snn_partition(net, cfg.P, "planted")
    rt = snn.Routing(net, part, cfg.P, cfg.n_vn, "contiguous")
    a = snn.Adjoint(net, g.is_exc, rt, snn.sim_params(cfg.dyn, raster_cap=0),
                    snn.adjoint_params(T=T, ckpt_every=50), device="cuda:0")
    a.forward(G, lam)
    dG, dlam = a.backward(grates)
    err = max(np.abs(dG - oG).max(), np.abs(dlam - olam).max()) / max(np.abs(oG).max(), np.abs(olam).max())
    print("gradient error against 64 bits: %.3g" % err)
    assert err <= 1e-7
