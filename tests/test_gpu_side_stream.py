"""A sim on a side stream (not ordered with the legacy stream): its tables, a
restored state and the autotuner's restored state are there before the kernels
that read them."""
import numpy as np
import pytest

import synth
from test_gpu_parity import _compare, _run_pair, snn  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("delivery,resident", [("0", "1"), ("0", "0"), ("1", "0"), ("2", "1"), ("3", "0")])
def test_restore_and_autotune_on_a_side_stream(snn, monkeypatch, delivery, resident):
    import torch
    monkeypatch.setenv("SNN_DELIVERY", delivery)
    monkeypatch.setenv("SNN_RESIDENT", resident)
    cfg = synth.SCALE.scaled(M=1 << 15, P=16, n_vn=4, K=100, n_part=70, n_vn_t=20, n_remote=10, seed=57)
    g = synth.make_network(cfg)
    with torch.cuda.stream(torch.cuda.Stream()):
        sim, o, rec, _ = _run_pair(snn, g, cfg, 60, cfg.P, cfg.n_vn)
        sim.step(20)
        sim.autotune(10)
        sim.step(40)
        _compare(sim, o, 60, rec)
        blob = sim.save_state()
        sim.step(25)
        V, ref, t = sim.read_state()
        for _ in range(3):
            sim.load_state(blob)
            sim.step(25)
            V2, ref2, t2 = sim.read_state()
            assert t2 == t == 85
            assert np.array_equal(V.view(np.uint32), V2.view(np.uint32)) and np.array_equal(ref, ref2)
        sim.reset(reupload=True)
        sim.step(85)
        assert np.array_equal(sim.read_state()[0].view(np.uint32), V.view(np.uint32))
    assert sim.sync_status() == 0
