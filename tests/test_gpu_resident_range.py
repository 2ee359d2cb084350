"""The calls and networks that the resident kernel leaves to the persistent
one: short calls of larger networks, and firing above its line.  Whichever
kernel runs, the results are the oracle's, and the choice follows the firing."""
import numpy as np
import pytest

import synth
from test_gpu_parity import _compare, _run_pair, snn  # noqa: F401

pytestmark = pytest.mark.gpu
RESIDENT = 3001


@pytest.fixture(autouse=True)
def _plain_env(monkeypatch):
    for k in ("SNN_PERSIST", "SNN_PERSIST_SMEM", "SNN_PERSIST_DEFER", "SNN_DELIVERY", "SNN_BAR_GROUPS",
              "SNN_PERSIST_BLOCKS_PER_SM", "SNN_RESIDENT"):
        monkeypatch.delenv(k, raising=False)


def _cfg(M, w_ext, K=30, lam=0.8):
    return synth.NetConfig(name="range", M=M, P=4, n_vn=2, K=K, uniform_all=True, dmax=8, seed=3,
                           dyn=synth.Dynamics(drive_lambda=lam, w_ext=w_ext, drive_seed=6))


@pytest.mark.parametrize("M", [1 << 15, 30001])
def test_short_and_long_calls_in_turn(snn, M):
    cfg = _cfg(M, 96)
    g = synth.make_network(cfg)
    sim, o, rec, _ = _run_pair(snn, g, cfg, 200, 4, 2)
    assert sim.kernel(1) != RESIDENT and sim.kernel(100) == RESIDENT
    for _ in range(10):
        for part in (1, 8, 1, 10):
            sim.step(part)
    assert sim.sync_status() == 0
    _compare(sim, o, 200, rec)


@pytest.mark.parametrize("M", [1 << 15, 30001])
def test_firing_above_the_line_takes_the_other_kernel(snn, M):
    """About 350 Hz: within a long call, and in the calls after a short one."""
    cfg = _cfg(M, 3000)
    g = synth.make_network(cfg)
    T = 2300
    sim, o, rec, _ = _run_pair(snn, g, cfg, T, 4, 2, cur_every=500)
    assert sim.kernel(100) == RESIDENT
    sim.step(100)
    assert sim.sync_status() == 0 and sim.kernel(100) != RESIDENT
    sim.step(50)
    sim.reset()
    sim.step(T)  # (the firing of the run before)
    assert sim.sync_status() == 0
    _compare(sim, o, T, rec)
    fresh = snn.Sim(sim.net, sim.routing, sim.params, device="cuda:0")
    assert fresh.launches(T) == 1 + 2 * 3
    fresh.step(T)
    assert fresh.sync_status() == 0 and fresh.kernel(100) != RESIDENT
    assert all(np.array_equal(a, b) for a, b in zip(fresh.read_raster(0, T), sim.read_raster(0, T)))
    assert all(np.array_equal(a, b) for a, b in zip(fresh.read_hashes(0, T), sim.read_hashes(0, T)))
    assert fresh.read_counts() == sim.read_counts()


def test_back_below_the_line(snn):
    """A volley takes the next call off the resident kernel, the quiet after it back."""
    cfg = _cfg(1 << 15, 96, lam=0.2)
    g = synth.make_network(cfg)
    g.v0[:] = -45.0
    sim, o, rec, _ = _run_pair(snn, g, cfg, 60, 4, 2)
    seen = []
    for _ in range(6):
        seen.append(sim.kernel(10) == RESIDENT)
        sim.step(10)
        assert sim.sync_status() == 0
    assert seen == [True, False, True, True, True, True]
    _compare(sim, o, 60, rec)


def test_given_up_call_of_several_launches_stops(snn, monkeypatch):
    """A wait that runs out in the first launch of a long call: none of the
    others steps on, and a reset sim does."""
    monkeypatch.setenv("SNN_BARRIER_LIMIT_NS", "20000000")
    monkeypatch.setenv("SNN_TEST_SKIP_BARRIER", "1")
    cfg = _cfg(1 << 15, 96)
    g = synth.make_network(cfg)
    sim, o, rec, _ = _run_pair(snn, g, cfg, 1100, 4, 2, cur_every=300)
    sim.step(1100)
    assert sim.sync_status() == -8
    assert sim.read_state()[2] == 0
    sim.reset()
    sim.step(1100)
    assert sim.sync_status() == 0
    _compare(sim, o, 1100, rec)


def test_forced(snn, monkeypatch):
    monkeypatch.setenv("SNN_RESIDENT", "1")
    cfg = _cfg(1 << 15, 3000)
    g = synth.make_network(cfg)
    sim, o, rec, _ = _run_pair(snn, g, cfg, 90, 4, 2)
    for part in (1, 9, 80):
        assert sim.kernel(part) == RESIDENT
        sim.step(part)
    assert sim.sync_status() == 0
    _compare(sim, o, 90, rec)
