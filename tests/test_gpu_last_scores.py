"""gcamps_get_last_scores after a run: the scores of the last visit are the class search's, whatever decided earlier
visits.  The identity's exact entropy is among them and every evaluated vn is the von Neumann entropy of its class,
also where classes that make theta a product across the bond tie for the best."""
import numpy as np
import pytest

from oracle.gcamps import GCAMPS, entropy_from_singular_values, renyi2_from_singular_values
from synth import brickwork_circuit

pytestmark = pytest.mark.gpu

TOL = 1e-10   # the bar of the scoring parity tests


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_06672_gb300.build import build_library
    build_library()
    import paper_2511_06672_gb300 as G
    return G


@pytest.mark.parametrize("d,n,t,seed,csize,precision", [(2, 6, 5, 1, 8, 0), (2, 8, 9, 2, 4, 0), (3, 5, 4, 3, 16, 0),
                                                        (3, 6, 6, 4, 8, 0), (3, 5, 4, 3, 8, 1)])
def test_last_visit_has_the_search_scores(G, d, n, t, seed, csize, precision):
    gates = brickwork_circuit(n, d, t, t, seed)
    ops = G.ops_from_gates(gates, d)
    sim = G.Simulator(n, d, chi_max=d ** (n // 2), cluster_size=csize, precision=precision)
    ref = GCAMPS(2, d, chi_max=d)
    products = 0
    begin = 0
    # a launch per disentangling, each stopped after one to three visits: many end at a visit that applies a class
    for i, end in enumerate(np.nonzero(ops["kind"] == G.OP_DISENTANGLE)[0]):
        ops[end]["q1"] = 1 + i % 3
        sim.run(ops[begin: end + 1])
        sim.sync()
        begin = int(end) + 1
        if not sim.decisions():
            continue
        s2, vn, evaluated = sim.last_scores()
        assert evaluated[0]
        svs = ref.schmidt_values(np.asarray(sim.last_theta()))
        want = np.array([entropy_from_singular_values(v) for v in svs])
        want2 = np.array([renyi2_from_singular_values(v) for v in svs])
        products += int(want.min() < 1e-10)
        tol = TOL if not precision else 1e-4
        for k in np.nonzero(evaluated)[0]:
            assert abs(vn[k] - want[k]) < tol and abs(s2[k] - want2[k]) < tol
        # whatever is not evaluated does not beat the best of the evaluated ones
        assert vn[evaluated].min() <= want.min() + tol
    assert products > 0
    sim.close()
