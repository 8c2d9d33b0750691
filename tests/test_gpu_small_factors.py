"""The factorisations that keep their matrix in shared memory, through circuits whose bonds take their edge sizes:
without truncation the state is the dense one, and with the bond dimensions of the oracle.  Dimensions 2 and 3, bonds
on both sides of the limits (23 columns, 1024 entries, one warp against several, odd and even column counts)."""
import numpy as np
import pytest

from oracle import statevector as sv
from oracle.gcamps import GCAMPS
from synth import brickwork_circuit

pytestmark = pytest.mark.gpu

# the state's relative error per step is a few hundred roundings (2^-53) of a factor of norm 1; a hundred steps of
# both sweeps stay far below this
TOL = 1e-11


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_06672_gb300.build import build_library
    build_library()
    import paper_2511_06672_gb300 as G
    return G


@pytest.mark.parametrize("d,n,t,seed", [(2, 4, 3, 1), (2, 9, 6, 2), (2, 12, 9, 3), (3, 3, 2, 4), (3, 6, 4, 5),
                                        (3, 7, 5, 6), (3, 8, 4, 7)])
@pytest.mark.parametrize("disentangle", [False, True])
def test_states_and_bonds(G, d, n, t, seed, disentangle):
    gates = brickwork_circuit(n, d, max(t, 3), t, seed)
    chi = d ** (n // 2)
    sim = G.Simulator(n, d, chi_max=chi, cluster_size=4)
    sim.run(G.ops_from_gates(gates, d, disentangle_after_t=disentangle))
    sim.sync()
    ref = GCAMPS(n, d, chi_max=chi, cutoff=1e-12)
    for gt in gates:
        ref.apply_gate(gt)
        if disentangle and not hasattr(gt, "sp_index"):
            ref.disentangle()
    assert sim.bond_dims() == ref.mps.bond_dims()
    err, _ = sv.same_up_to_phase(sim.statevector(), sv.run(gates, n, d))
    assert err < TOL
    for b in range(n - 1):
        got = sim.schmidt_values(b)
        assert abs(float(np.sum(got ** 2)) - 1.0) < TOL and np.all(np.diff(got) <= 0)
    sim.close()
