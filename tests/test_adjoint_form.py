"""Which form of the adjoint's backward a network takes (told by its workspace):
the batched one from 25,000 neurons on, but with many synapses per neuron and
few delays only from the size on where it is the faster one."""
import ctypes

import pytest

import paper_2205_07125_gb300 as snn
import synth


@pytest.mark.parametrize("M,K,dmax,batched", [
    (24000, 10, 8, False), (26000, 20, 8, True), (26000, 50, 1, True), (30000, 150, 1, False), (30000, 150, 3, False),
    (30000, 150, 4, True), (42000, 150, 1, True), (26000, 300, 8, False), (29000, 300, 8, True)])
def test_form_by_size_synapses_and_delays(monkeypatch, M, K, dmax, batched):
    cfg = synth.NetConfig(name="form", M=M, P=4, n_vn=2, K=K, uniform_all=True, dmax=dmax, seed=1)
    g = synth.make_network(cfg)
    net = snn.Network.from_synth(g)
    part, _ = snn.snn_partition(net, 4, "planted")
    rt = snn.Routing(net, part, 4, 2)
    assert rt.info()["max_delay"] == dmax
    prm, ap = snn.sim_params(cfg.dyn), snn.adjoint_params(T=10, ckpt_every=5)
    size = {}
    for form in ("0", "1", None):
        if form is None:
            monkeypatch.delenv("SNN_ADJ_BATCHED", raising=False)
        else:
            monkeypatch.setenv("SNN_ADJ_BATCHED", form)
        nb = ctypes.c_size_t(0)
        assert snn._lib.snn_adjoint_workspace_bytes(rt.h, ctypes.byref(prm), ctypes.byref(ap), ctypes.byref(nb)) == 0
        size[form] = nb.value
    assert size["0"] != size["1"]
    assert size[None] == size["1" if batched else "0"]
