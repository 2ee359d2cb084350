"""The resident kernel's spike messages tell old from new whatever the step
numbers do: resets and captured graphs repeat them, the messages' tags go on."""
import numpy as np
import pytest

import synth
from test_gpu_parity import _compare, _run_pair, snn  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _plain_env(monkeypatch):
    for k in ("SNN_PERSIST", "SNN_PERSIST_SMEM", "SNN_PERSIST_DEFER", "SNN_DELIVERY", "SNN_BAR_GROUPS",
              "SNN_PERSIST_BLOCKS_PER_SM", "SNN_RESIDENT"):
        monkeypatch.delenv(k, raising=False)


def _net():
    cfg = synth.NetConfig(name="tags", M=1500, P=4, n_vn=2, K=60, uniform_all=True, dmax=2, seed=83,
                          dyn=synth.Dynamics(drive_lambda=1.1, w_ext=150, drive_seed=9))
    return cfg, synth.make_network(cfg)


def test_single_steps_from_rest_past_the_tags_16_bits(snn, monkeypatch):
    """65,534 times one step from rest, then 40 steps: with tags that count on
    the second of them has tag 65,536, whose 16 bits in the message words are
    those of words that were never written."""
    monkeypatch.setenv("SNN_RESIDENT_BLOCKS", "9")  # (messages in global memory, kept between launches)
    cfg, g = _net()
    sim, o, rec, _ = _run_pair(snn, g, cfg, 40, cfg.P, cfg.n_vn)
    for _ in range(65534):
        sim.step(1)
        sim.reset()
    sim.step(40)
    assert sim.sync_status() == 0
    c, _ = _compare(sim, o, 40, rec)
    assert c["spikes"] > 100


def test_restored_state_after_a_launch_that_gave_up(snn, monkeypatch):
    """A launch of 65,536 steps gives up in its first step (block 0 is silent:
    test switch); the first step after it, of a restored state, has the same 16
    bits in its tag as the messages that the others left."""
    monkeypatch.setenv("SNN_RESIDENT_BLOCKS", "9")
    cfg, g = _net()
    sim, o, rec, rt = _run_pair(snn, g, cfg, 60, cfg.P, cfg.n_vn)
    sim.step(25)
    blob = sim.save_state()
    sim.step(35)
    V, ref, t = sim.read_state()
    monkeypatch.setenv("SNN_BARRIER_LIMIT_NS", "20000000")
    monkeypatch.setenv("SNN_TEST_SKIP_BARRIER", "1")
    late = snn.Sim(sim.net, rt, sim.params, device="cuda:0")
    late.step(65536)
    assert late.sync_status() == -8
    late.load_state(blob)
    late.step(35)
    assert late.sync_status() == 0
    V2, ref2, t2 = late.read_state()
    assert t2 == t == 60
    assert np.array_equal(V.view(np.uint32), V2.view(np.uint32)) and np.array_equal(ref, ref2)


@pytest.mark.parametrize("blocks", [1, 4, 9])
def test_captured_steps_replay(snn, monkeypatch, blocks):
    """A CUDA graph that holds a call of three steps, replayed between calls
    that are not captured."""
    import torch
    monkeypatch.setenv("SNN_RESIDENT_BLOCKS", str(blocks))
    monkeypatch.setenv("SNN_RESIDENT_LIST", "1")
    cfg, g = _net()
    g.v0[::3] = -45.0
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        sim, o, rec, _ = _run_pair(snn, g, cfg, 132, cfg.P, cfg.n_vn)
        sim.step(2)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            sim.step(3)
        for _ in range(20):
            graph.replay()
        sim.step(10)
        for _ in range(20):
            graph.replay()
    assert sim.sync_status() == 0
    c, _ = _compare(sim, o, 132, rec)
    assert c["spikes"] > 1000
