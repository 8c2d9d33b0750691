"""Phase gradients of observables that are not zero: Z strings evolved through a circuit's Cliffords, against the
oracle's dense gradient.  Both dimensions, with and without disentangling, bonds whose transfer matrices fit shared
memory and bonds beyond it; for d = 3 O = (W + W^dag) / 2 changes the norm of the state it is applied to."""
import numpy as np
import pytest

from oracle import statevector as sv
from oracle.tableau import Tableau
from oracle.weyl import Weyl
from synth import param_phase_circuit

pytestmark = pytest.mark.gpu

VALUE_TOL, GRAD_TOL = 1e-10, 1e-9   # the bars of the gradient tests


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_06672_gb300.build import build_library
    build_library()
    import paper_2511_06672_gb300 as G
    return G


def _evolved(gates, n, d):
    """Exponents (x, z) of C Z_q C^dag, C the circuit's Cliffords."""
    t = Tableau(n, d)
    for g in gates:
        if hasattr(g, "sp_index"):
            t.apply_gate(sv.gate_unitary(g, d), [g.q0, g.q1])
    return [(r.x.astype(np.int32), r.z.astype(np.int32)) for r in t.rows[:n]]


def _run(G, d, n, layers, ngates, seed, disentangle):
    gates, _ = param_phase_circuit(n, d, layers, ngates, seed)
    sim = G.Simulator(n, d, chi_max=d ** (n // 2), cutoff=1e-14, snapshot_entries=1 << 20, snapshot_max_gates=ngates)
    sim.run(G.ops_from_gates(gates, d, disentangle_after_t=disentangle))
    sim.sync()
    return gates, sim


@pytest.mark.parametrize("d,n,layers,ngates,seed", [(3, 4, 6, 5, 2), (3, 6, 6, 8, 2), (3, 7, 6, 5, 1), (2, 6, 6, 8, 4),
                                                    (2, 11, 8, 9, 1)])
@pytest.mark.parametrize("disentangle", [True, False])
def test_gradient_of_evolved_strings(G, d, n, layers, ngates, seed, disentangle):
    gates, sim = _run(G, d, n, layers, ngates, seed, disentangle)
    # states without disentangling leave the shared-memory transfer (200 entries of E) at these sizes
    assert disentangle or n < 7 or max(sim.bond_dims()) ** 2 > 200
    largest = 0.0
    for x, z in _evolved(gates, n, d):
        if d == 2 and int(np.sum(x * z)) % 2:
            continue
        val, grad = sim.expect_gradient(x, z)
        rval, rgrad = sv.observable_and_phase_gradient(gates, n, d, Weyl(0, x, z, d))
        rgrad = np.array(rgrad)
        largest = max(largest, float(np.max(np.abs(rgrad))))
        assert abs(val - rval) < VALUE_TOL
        assert np.max(np.abs(grad - rgrad)) < GRAD_TOL
    assert largest > 0.1
    sim.close()


@pytest.mark.parametrize("n,layers,ngates,seed", [(6, 6, 8, 3), (11, 8, 9, 2)])
def test_strings_with_an_odd_number_of_y_factors_have_gradient_zero(G, n, layers, ngates, seed):
    """For d = 2 such a string (phase 1) is anti-Hermitian: Re <W>, the mean of (W + W^dag) / 2 = 0, is 0 for every
    phase."""
    gates, sim = _run(G, 2, n, layers, ngates, seed, True)
    odd = [(x, z) for x, z in _evolved(gates, n, 2) if int(np.sum(x * z)) % 2]
    assert odd
    for x, z in odd:
        val, grad = sim.expect_gradient(x, z)
        assert abs(val) < VALUE_TOL
        assert np.max(np.abs(grad)) < GRAD_TOL
    sim.close()
