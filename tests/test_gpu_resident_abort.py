"""Waits of the resident kernel that run out while blocks have more spikes
than a message holds: every block leaves with an error, and a reset sim steps
on with the right results."""
import pytest

import synth
from test_gpu_parity import _compare, _run_pair, snn  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lists", [1, 4096])
@pytest.mark.parametrize("blocks", [2, 8, 24])
def test_given_up_volley_ends_with_an_error(snn, monkeypatch, blocks, lists):
    for k in ("SNN_PERSIST", "SNN_PERSIST_SMEM", "SNN_PERSIST_DEFER", "SNN_DELIVERY", "SNN_BAR_GROUPS",
              "SNN_PERSIST_BLOCKS_PER_SM", "SNN_RESIDENT"):
        monkeypatch.delenv(k, raising=False)
    monkeypatch.setenv("SNN_RESIDENT_BLOCKS", str(blocks))
    monkeypatch.setenv("SNN_RESIDENT_LIST", str(lists))
    monkeypatch.setenv("SNN_BARRIER_LIMIT_NS", "20000000")
    monkeypatch.setenv("SNN_TEST_SKIP_BARRIER", "1")
    cfg = synth.NetConfig(name="burst", M=3001, P=4, n_vn=2, K=50, uniform_all=True, dmax=4, seed=77,
                          dyn=synth.Dynamics(drive_lambda=0.5, w_ext=200))
    g = synth.make_network(cfg)
    g.v0[:] = -45.0  # every neuron spikes in the first step, whose messages block 0 does not publish
    sim, o, rec, _ = _run_pair(snn, g, cfg, 50, 4, 2)
    sim.step(50)
    assert sim.sync_status() == -8
    assert sim.read_state()[2] == 0
    sim.reset()
    sim.step(50)
    assert sim.sync_status() == 0
    c, _ = _compare(sim, o, 50, rec)
    assert c["spikes"] >= g.M
