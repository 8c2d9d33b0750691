"""Bond dimensions of single circuits of a large batch, those copied together with the status words and those copied
apart from them (more than 512 KB of later circuits in between): each circuit's own, and a failed circuit is reported
whichever circuit is read."""
import numpy as np
import pytest

from synth import brickwork_circuit

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_06672_gb300.build import build_library
    build_library()
    import paper_2511_06672_gb300 as G
    return G


def test_dims_and_status_of_a_large_batch(G):
    from paper_2511_06672_gb300 import _native as N
    d, n, batch = 2, 40, 3500
    runs = {0: 1, 1: 2, 200: 3, 302: 4, 303: 5, 304: 6, 3498: 7, 3499: 8}   # circuit: seed; the others stay |0...0>
    ops, begin = [], [0]
    for c in range(batch):
        if c in runs:
            gates = brickwork_circuit(n, d, 6, 4, runs[c])
            ops.append(G.ops_from_gates(gates, d, disentangle_after_t=False))
        begin.append(begin[-1] + (len(ops[-1]) if c in runs else 0))
    sim = G.Simulator([n] * batch, d, chi_max=4, cluster_size=1)
    sim.run(np.concatenate(ops), begin)
    for c, seed in runs.items():
        alone = G.Simulator(n, d, chi_max=4, cluster_size=1)
        alone.run(G.ops_from_gates(brickwork_circuit(n, d, 6, 4, seed), d, disentangle_after_t=False))
        want = alone.bond_dims()
        assert sim.bond_dims(c) == want and max(want) > 1
        alone.close()
    assert sim.bond_dims(2) == [1] * (n - 1)
    # a replay list that ends after one visit fails circuit 303, the only one that runs
    sim.reset()
    sim.set_replay([(0, 0)], circuit=303)
    again = G.ops_from_gates(brickwork_circuit(n, d, 6, 4, runs[303]), d)
    sim.run(again, [0] * 304 + [len(again)] * (batch - 303))
    for c in (0, 303, 3499):
        with pytest.raises(G.GcampsError) as ei:
            sim.bond_dims(c)
        assert ei.value.code == N.EINVAL
    sim.close()
