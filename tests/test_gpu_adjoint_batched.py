"""The batched backward of the adjoint (several steps gathered at once; chosen
for large networks) at the sizes where it has edges, against the float64
oracle on the same trajectory: each delay class alone and mixed, segments
shorter than a batch, partitions of odd sizes, and a partition larger than the
parts of it that are staged.  Relative error at most 1e-5, as the adjoint's
other tests."""
import numpy as np
import pytest

import oracle
import synth
from oracle import adjoint as adj
from test_gpu_adjoint import _params, snn  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,P,n_vn,K,dmax,T,ckpt", [
    (1203, 3, 1, 40, 1, 40, 40), (1203, 3, 3, 40, 2, 41, 5), (2048, 4, 2, 40, 3, 60, 1), (2047, 4, 4, 60, 16, 64, 7),
    (2048, 4, 2, 40, 8, 62, 20), (17003, 1, 1, 24, 5, 20, 20)])
def test_batched_gradients_against_float64_oracle(snn, monkeypatch, M, P, n_vn, K, dmax, T, ckpt):
    cfg = synth.NetConfig(name="adjb", M=M, P=P, n_vn=n_vn, K=K, uniform_all=True, dmax=dmax, seed=M + dmax,
                          dyn=synth.Dynamics(w_ext=89, drive_seed=4000))
    g = synth.make_network(cfg)
    net = snn.Network.from_synth(g)
    part, _ = snn.snn_partition(net, P, "planted")
    rt = snn.Routing(net, part, P, n_vn, "contiguous")
    onet = adj.from_synth(g, cfg.dyn, oracle.partition_planted(M, P), oracle.group_contiguous(P, n_vn),
                          oracle.alpha32(cfg.dyn.dt_ms, cfg.dyn.tau_ms))
    G, lam, target = _params(2 * n_vn, seed=3)
    tr = adj.forward_fp32(onet, G, lam, T)
    grates = 2 * (tr.rates - target) / (2 * n_vn)
    oG, olam = adj.backward(onet, G, lam, tr, grates)
    scale = max(np.abs(oG).max(), np.abs(olam).max())
    assert scale > 0
    for batched in ("1", "0"):
        monkeypatch.setenv("SNN_ADJ_BATCHED", batched)
        a = snn.Adjoint(net, g.is_exc, rt, snn.sim_params(cfg.dyn, raster_cap=M * T),
                        snn.adjoint_params(T=T, ckpt_every=ckpt), device="cuda:0")
        assert np.allclose(a.forward(G, lam), tr.rates, rtol=1e-6, atol=0)
        for _ in range(2):  # a second backward starts clean
            dG, dlam = a.backward(grates)
        assert max(np.abs(dG - oG).max(), np.abs(dlam - olam).max()) / scale <= 1e-5
        a.close()
