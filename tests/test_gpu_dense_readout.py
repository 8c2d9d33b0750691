"""The dense readout through C's word of elementary gates: on registers of both dimensions, from the smallest to sizes
whose passes leave CTAs without work, with every kind of gate in the word, the state vector is the dense simulation's
up to one phase, amplitudes are entries of it, and its phase is the documented one: that of <C 0|v>, v the hashed
vector, so that C|y> = prod_j D_j^{y_j} C|0> holds between handles."""
import numpy as np
import pytest

from oracle import statevector as sv
from synth import brickwork_circuit

pytestmark = pytest.mark.gpu

# a hundred Fourier passes of unit norm at a few roundings (2^-53) each
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


@pytest.mark.parametrize("d,n,layers,t", [(2, 2, 0, 0), (2, 2, 3, 2), (3, 2, 4, 2), (2, 5, 9, 3), (3, 5, 6, 4), (2, 13, 6, 2),
                                          (3, 8, 5, 2)])
def test_state_phase_and_amplitudes(G, d, n, layers, t):
    gates = brickwork_circuit(n, d, layers, t, 40 + n) if layers else []
    sim = G.Simulator(n, d, chi_max=d ** (n // 2))
    if gates:
        sim.run(G.ops_from_gates(gates, d, disentangle_after_t=False))
    psi = sim.statevector()
    ref = sv.run(gates, n, d).reshape(-1)
    err, _ = sv.same_up_to_phase(psi, ref)
    assert err < TOL
    # the phase: C|0> from the Cliffords alone, on a handle of its own
    c0 = sv.run([g for g in gates if hasattr(g, "sp_index")], n, d).reshape(-1)
    with np.errstate(over="ignore"):
        def part(k):
            z = np.arange(d ** n, dtype=np.uint64) * np.uint64(2) + np.uint64(k) + np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            return ((z ^ (z >> np.uint64(31))) >> np.uint64(11)).astype(np.float64) / 2.0 ** 53 - 0.5
        ph = np.vdot(c0, part(1) + 1j * part(2))
    assert np.max(np.abs(psi - ref * (ph / abs(ph)))) < TOL
    rng = np.random.default_rng(n)
    for y in rng.integers(d ** n, size=3):
        digits = [(int(y) // d ** (n - 1 - j)) % d for j in range(n)]
        assert sim.amplitude(digits) == psi[y]
    sim.close()
