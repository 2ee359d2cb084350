"""The device partitioner's rounds at the edges of its selection: bins of equal
or no gain that hold more keys than a round's list, gains over many powers of
two, rounds of the largest size, neuron counts around the blocks' shares, and
odd and even numbers of iterations (two run side by side).  Labels and
objective equal the oracle's."""
import numpy as np
import pytest

import synth
from test_gpu_partition import _both, snn  # noqa: F401

pytestmark = pytest.mark.gpu


def _net(kind, M):
    rng = np.random.default_rng(M)
    if kind == "star":  # neuron 0 shares one synapse with every other: equal gains
        pairs = [(0, j) for j in range(1, M)] + [(j, (j % (M - 1)) + 1) for j in range(1, M)]
    elif kind == "sparse":  # most neurons share no synapse with a part: gains of 0
        pairs = [(i, (i + 1) % M) for i in range(0, M, 3)]
    else:  # out-degrees of 1 to some hundreds, repeated synapses: gains over many powers of two
        deg = np.minimum((rng.pareto(0.7, M) + 1).astype(int), 300)
        pairs = [(i, int(j)) for i in range(M) for j in np.repeat(rng.integers(0, M, deg[i]), 1 + i % 2)]
    return synth.make_edges(M, [(a, b, 1, 1) for a, b in pairs])


@pytest.mark.parametrize("iters", [1, 3, 4])
@pytest.mark.parametrize("kind,M", [("star", 5000), ("sparse", 7001), ("wide", 1217), ("wide", 4864)])
def test_rounds_equal_oracle(snn, kind, M, iters):
    g = _net(kind, M)
    for batch, grow in [(2048, 0), (2048, 2), (65, 0)]:
        _both(snn, g, 3, batch, grow, iters, 5)


@pytest.mark.parametrize("M", [2, 75, 76, 77, 151, 153, 2049])
def test_small_shares(snn, M):
    g = _net("sparse", M) if M < 4 else _net("wide", M)
    _both(snn, g, 2, 2048, 2, 2, 9)
