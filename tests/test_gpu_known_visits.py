"""Bond visits whose decision is known without exact entropies (bonds of dimension 1, clean bonds, product classes)
decide as the oracle's full SVD search does, for tie tolerances with and without the purity test, for every score
kind, with the clusters that take each estimate path, and where truncation changes the state between visits."""
import pytest

from oracle.gcamps import GCAMPS
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


@pytest.mark.parametrize("d,n,t,seed,tie_tol,kind,csize,chi", [
    (3, 7, 8, 3, 1e-10, 0, 1, 27), (3, 7, 8, 3, 1e-10, 0, 16, 27), (2, 9, 11, 5, 1e-10, 0, 2, 16),
    (2, 9, 11, 5, 1e-12, 0, 8, 16),   # purity bound above half the tolerance: no purity test
    (2, 9, 11, 5, 1e-3, 0, 8, 16),    # tolerance above the screen's list threshold
    (3, 6, 7, 2, 1e-10, 1, 8, 27), (3, 6, 7, 2, 1e-10, 2, 8, 27),
    (2, 10, 14, 4, 1e-10, 0, 8, 3),   # chi_max truncates: no bond stays clean
    (2, 8, 8, 1, 1e-10, 0, 8, 1),
])
def test_decisions_match_full_search(G, d, n, t, seed, tie_tol, kind, csize, chi):
    gates = brickwork_circuit(n, d, t, t, seed)
    sim = G.Simulator(n, d, chi_max=chi, tie_tol=tie_tol, score_kind=kind, cluster_size=csize)
    sim.run(G.ops_from_gates(gates, d))
    sim.sync()
    ref = GCAMPS(n, d, chi_max=chi, cutoff=1e-12, tie_tol=tie_tol, score_kind=kind)
    for gt in gates:
        ref.apply_gate(gt)
        if not hasattr(gt, "sp_index"):
            ref.disentangle()
    assert sim.decisions() == ref.decisions
    assert sim.bond_dims() == ref.mps.bond_dims()
    assert sim.stats()["candidates_scored"] == ref.candidates_scored
    # the last visit is scored whatever is known about it
    s2, vn, evaluated = sim.last_scores()
    shape_ok = sim.last_theta() is not None
    assert evaluated.any() and shape_ok
    sim.close()
