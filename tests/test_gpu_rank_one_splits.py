"""Splits after a class that makes theta nearly a product: what is left beside the product lies below, around and above
the residual up to which the factors are taken from one column (1e-14 of the norm, and never above the cutoff), and
below and above the cutoff.  Bond dimensions are the oracle's and the state is the dense one but for what the cutoff
drops."""
import pytest

from oracle import statevector as sv
from oracle.gcamps import GCAMPS
from synth import Diag, brickwork_circuit

pytestmark = pytest.mark.gpu

# a few hundred roundings (2^-53) of a state of norm 1
TOL = 1e-13


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_06672_gb300.build import build_library
    build_library()
    import paper_2511_06672_gb300 as G
    return G


def _circuit(d, n, seed, eps):
    """Three phase gates, the last two by angles of order eps: the class that undoes the first leaves them."""
    gates = brickwork_circuit(n, d, 6, 3, seed)
    at = [i for i, g in enumerate(gates) if not hasattr(g, "sp_index")]
    for i, a in zip(at, (1.1, eps, 0.7 * eps)):
        gates[i] = Diag(gates[i].site, (0.0, a) if d == 2 else (0.0, a, -0.6 * a), gates[i].param)
    return gates[: at[2] + 1]


# left: the ratio of the second to the first singular value after the first visit, for eps = 1
@pytest.mark.parametrize("d,n,seed,left", [(2, 2, 20, 0.4456), (2, 2, 34, 0.6103), (3, 2, 3, 0.6752), (2, 3, 4, 0.1588)])
@pytest.mark.parametrize("ratio,cutoff", [(0.0, 1e-12), (3e-15, 1e-12), (3e-14, 1e-12), (3e-13, 1e-12), (3e-12, 1e-12),
                                          (3e-9, 1e-12), (3e-14, 1e-15)])
def test_split_of_a_near_product(G, d, n, seed, left, ratio, cutoff):
    gates = _circuit(d, n, seed, ratio / left)
    sim = G.Simulator(n, d, chi_max=d ** (n // 2), cutoff=cutoff, max_sweeps=1)
    ref = GCAMPS(n, d, chi_max=d ** (n // 2), cutoff=cutoff, max_sweeps=1)
    for g in gates:
        ref.apply_gate(g)
    ref.disentangle()
    assert ref.decisions[0][1] != 0 and (ref.mps.bond_dims()[ref.decisions[0][0]] > 1) == (ratio > cutoff)
    sim.run(G.ops_from_gates(gates, d, disentangle_after_t=False))
    sim.disentangle()
    assert sim.decisions() == ref.decisions and sim.bond_dims() == ref.mps.bond_dims()
    err, _ = sv.same_up_to_phase(sim.statevector(), sv.run(gates, n, d).reshape(-1))
    assert err < TOL + (3.0 * ratio if ratio < cutoff else 0.0)
    sim.close()
