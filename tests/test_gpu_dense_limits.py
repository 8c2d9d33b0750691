"""The dense readout at its largest registers, 2^20 and 3^12 entries, and one site below: the state is the dense
simulation's up to one phase, and amplitudes are entries of it.  One more site is refused."""
import numpy as np
import pytest

from oracle import statevector as sv
from synth import brickwork_circuit

pytestmark = pytest.mark.gpu

# a few hundred Fourier passes of unit norm at a few roundings (2^-53) each
TOL = 1e-12


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_06672_gb300.build import build_library
    build_library()
    import paper_2511_06672_gb300 as G
    return G


@pytest.mark.parametrize("d,n,layers,t", [(2, 19, 5, 3), (2, 20, 6, 3), (3, 11, 5, 2), (3, 12, 6, 2)])
def test_largest_registers(G, d, n, layers, t):
    gates = brickwork_circuit(n, d, layers, t, n)
    sim = G.Simulator(n, d, chi_max=d ** t, cluster_size=4)
    sim.run(G.ops_from_gates(gates, d, disentangle_after_t=False))
    psi = sim.statevector()
    assert sim.stats()["discarded_weight"] < 1e-20
    err, _ = sv.same_up_to_phase(psi, sv.run(gates, n, d).reshape(-1))
    assert err < TOL
    for y in (0, d ** n - 1, int(np.argmax(np.abs(psi)))):
        assert sim.amplitude([(y // d ** (n - 1 - j)) % d for j in range(n)]) == psi[y]
    sim.close()


@pytest.mark.parametrize("d,n", [(2, 21), (3, 13)])
def test_a_larger_register_is_refused(G, d, n):
    sim = G.Simulator(n, d, chi_max=2)
    with pytest.raises(G.GcampsError) as ei:
        sim.statevector()
    assert ei.value.code == 1   # GCAMPS_EINVAL
    with pytest.raises(G.GcampsError):
        sim.amplitude([0] * n)
    sim.close()
