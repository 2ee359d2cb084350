"""Each step kernel by name: the parity tests again on the persistent kernel
with the delay ring (networks of their sizes run on the resident kernel
otherwise), and the resident kernel in the shapes that only large networks
take by themselves: two to four quads of neurons per thread, messages of eight
words, without records."""
import numpy as np
import pytest

import synth
import test_gpu_batch as batch
import test_gpu_parity as parity
from test_gpu_batch import test_batch_of_one_equals_plain_sim, test_batch_uneven_networks  # noqa: F401
from test_gpu_parity import (_run_pair, snn, test_barrier_wait_is_bounded, test_capacity_overflow_is_reported,  # noqa: F401
                             test_checkpoint_resume_bit_exact, test_degenerate_networks,
                             test_locality_delays_several_tiles, test_ragged_sizes_and_uneven_partitions,
                             test_raster_of_wide_steps, test_relay_policies_counts_and_currents,
                             test_reset_replays_identically, test_step_in_chunks_equals_one_call,
                             test_tiny_full_run, test_tiny_greedy_partition_and_grouping)

pytestmark = pytest.mark.gpu
_VARS = ("SNN_PERSIST", "SNN_PERSIST_SMEM", "SNN_PERSIST_DEFER", "SNN_DELIVERY", "SNN_BAR_GROUPS",
         "SNN_PERSIST_BLOCKS_PER_SM", "SNN_RESIDENT", "SNN_RESIDENT_BLOCKS", "SNN_RESIDENT_THREADS",
         "SNN_RESIDENT_LIST")


@pytest.fixture(autouse=True)
def _persistent_ring(request, snn, monkeypatch):
    """The tests of the other modules: every step on k_persist with the delay ring."""
    for k in _VARS:
        monkeypatch.delenv(k, raising=False)
    if request.function.__module__ in (parity.__name__, batch.__name__):
        monkeypatch.setenv("SNN_RESIDENT", "0")
        step = snn.Sim.step

        def checked(sim, T):
            assert 0 < sim.kernel(T) < 1000 and sim.kernel(T) % 100 > 0
            step(sim, T)
        monkeypatch.setattr(snn.Sim, "step", checked)


@pytest.fixture
def path():
    return "persistent"


@pytest.mark.parametrize("records", [False, True])
@pytest.mark.parametrize("M,P,n_vn,dmax,blocks,threads,mapping", [
    (6001, 5, 5, 3, 2, 384, "greedy"), (6001, 5, 5, 3, 2, 384, "planted"), (12000, 4, 2, 4, 2, 512, "planted"),
    (12002, 4, 2, 2, 2, 512, "greedy"), (4001, 3, 3, 8, 3, 384, "planted"), (5003, 5, 5, 16, 2, 1024, "planted")])
def test_resident_shapes_of_large_networks(snn, monkeypatch, M, P, n_vn, dmax, blocks, threads, mapping, records):
    monkeypatch.setenv("SNN_RESIDENT", "1")
    monkeypatch.setenv("SNN_RESIDENT_BLOCKS", str(blocks))
    monkeypatch.setenv("SNN_RESIDENT_THREADS", str(threads))
    cfg = synth.NetConfig(name="resq", M=M, P=P, n_vn=n_vn, K=70, uniform_all=True, dmax=dmax, seed=17 + M,
                          dyn=synth.Dynamics(drive_lambda=1.1, w_ext=96, drive_seed=5))
    g = synth.make_network(cfg)
    T = 130
    sim, o, rec, rt = _run_pair(snn, g, cfg, T, P, n_vn, mapping)
    if not records:
        sim.close()
        prm = snn.sim_params(cfg.dyn, raster_cap=max(4096, M * T // 10), raster_steps=T)
        sim = snn.Sim(sim.net, rt, prm, device="cuda:0")
    assert sim.kernel(1) == 3001
    for part in (1, 2, 127):
        sim.step(part)
    assert sim.sync_status() == 0
    if records:
        parity._compare(sim, o, T, rec)
        return
    r = o.run(T)
    ids, off = sim.read_raster(0, T)
    assert np.array_equal(off, r["raster_off"]) and np.array_equal(ids, r["raster_ids"])
    V, ref, t = sim.read_state()
    assert t == T and np.array_equal(V.view(np.uint32), o.V.view(np.uint32)) and np.array_equal(ref, o.ref)
    assert len(ids) > 100
