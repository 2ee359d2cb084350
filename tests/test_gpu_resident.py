"""GPU parity of the resident step kernel (the whole network on the chip, one
exchange of the blocks' spikes per step) against the CPU oracle, at the sizes
where its parts have edges: one block, a cluster, many blocks; neuron counts
that are no multiple of 4 or of the blocks; the smallest and largest delay;
lists of one entry, so that everything past them takes its way round; every
neuron spiking at once; networks too large for it, which other kernels step."""
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


@pytest.mark.parametrize("blocks", [1, 2, 7, 8, 152])
@pytest.mark.parametrize("lists", [1, 40, 4096])
@pytest.mark.parametrize("M,P,n_vn,dmax", [(4096, 4, 2, 1), (5003, 5, 5, 16), (1021, 6, 3, 3)])
def test_blocks_lists_and_odd_sizes(snn, monkeypatch, blocks, lists, M, P, n_vn, dmax):
    monkeypatch.setenv("SNN_RESIDENT_BLOCKS", str(blocks))
    monkeypatch.setenv("SNN_RESIDENT_LIST", str(lists))
    cfg = synth.NetConfig(name="res", M=M, P=P, n_vn=n_vn, K=90, uniform_all=True, dmax=dmax, seed=31 + M,
                          dyn=synth.Dynamics(drive_lambda=1.1, w_ext=96, drive_seed=5))
    g = synth.make_network(cfg)
    sim, o, rec, _ = _run_pair(snn, g, cfg, 160, P, n_vn, "greedy" if M == 5003 else "planted")
    assert sim.launches(10) == 1
    for part in (1, 2, 157):  # the state crosses launches
        sim.step(part)
    assert sim.sync_status() == 0
    c, _ = _compare(sim, o, 160, rec)
    assert c["spikes"] > 100


@pytest.mark.parametrize("lists", [1, 4096])
@pytest.mark.parametrize("blocks", [1, 4, 60])
def test_every_neuron_spikes_at_once(snn, monkeypatch, blocks, lists):
    monkeypatch.setenv("SNN_RESIDENT_BLOCKS", str(blocks))
    monkeypatch.setenv("SNN_RESIDENT_LIST", str(lists))
    M = 3001
    cfg = synth.NetConfig(name="burst", M=M, P=4, n_vn=2, K=50, uniform_all=True, dmax=4, seed=77,
                          dyn=synth.Dynamics(drive_lambda=0.5, w_ext=200))
    g = synth.make_network(cfg)
    g.v0[:] = -45.0
    sim, o, rec, _ = _run_pair(snn, g, cfg, 50, 4, 2)
    sim.step(50)
    assert sim.sync_status() == 0
    c, _ = _compare(sim, o, 50, rec)
    assert c["spikes"] >= M


@pytest.mark.parametrize("blocks", [2, 8, 24])
def test_wait_for_a_silent_block_is_bounded(snn, monkeypatch, blocks):
    """Block 0 does not publish its first step (test switch): every block's
    wait runs out, the host reads SNN_E_TIMEOUT, and a reset sim steps on."""
    monkeypatch.setenv("SNN_RESIDENT_BLOCKS", str(blocks))
    monkeypatch.setenv("SNN_BARRIER_LIMIT_NS", "20000000")
    monkeypatch.setenv("SNN_TEST_SKIP_BARRIER", "1")
    cfg = synth.TINY
    g = synth.make_network(cfg)
    sim, o, rec, _ = _run_pair(snn, g, cfg, 60, 4, 2)
    sim.step(50)
    assert sim.sync_status() == -8
    assert sim.read_state()[2] == 0
    sim.reset()
    sim.step(60)
    assert sim.sync_status() == 0
    _compare(sim, o, 60, rec)


def test_small_workspace_and_switch_take_the_other_kernels(snn, monkeypatch):
    """Without room for its tables, or switched off, the network runs on the
    persistent kernel with shared-memory state, with the same results."""
    cfg = synth.SCALE.scaled(M=1 << 14, P=16, n_vn=4, K=200, n_part=140, n_vn_t=40, n_remote=20, seed=53)
    g = synth.make_network(cfg)
    monkeypatch.setenv("SNN_RESIDENT", "0")
    sim, o, rec, rt = _run_pair(snn, g, cfg, 120, cfg.P, cfg.n_vn)
    small = sim.workspace_bytes
    sim.step(120)
    _compare(sim, o, 120, rec)
    monkeypatch.delenv("SNN_RESIDENT")
    import ctypes
    import torch
    nb = ctypes.c_size_t(0)
    prm = sim.params
    assert snn._lib.snn_sim_workspace_bytes(rt.h, ctypes.byref(prm), ctypes.byref(nb)) == 0
    assert nb.value > small
    ws = torch.empty(small, dtype=torch.uint8, device="cuda:0")
    h = ctypes.c_void_p()
    rc = snn._lib.snn_sim_create(ctypes.byref(sim.net.s), rt.h, ctypes.byref(prm), ws.data_ptr(), small,
                                 torch.cuda.current_stream().cuda_stream, ctypes.byref(h))
    assert rc == 0
    assert snn._lib.snn_step(h, 120) == 0 and snn._lib.snn_sync_status(h) == 0
    V = np.empty(g.M, np.float32)
    assert snn._lib.snn_read_state(h, V.ctypes.data, None, None) == 0
    assert np.array_equal(V.view(np.uint32), o.V.view(np.uint32))
    snn._lib.snn_sim_destroy(h)
