"""<W> and overlaps on both sides of the limits of their shared-memory routes, against a plain contraction of the
library's own site tensors (fetched one by one): states of two sites, odd and even lengths, bonds of 11 and 12 (the
halves' limit), chains below and above 8192 entries, overlaps of states with different bonds below and above 200.  The
strings are chosen as C P C^dag for a short P, so their values are not zero."""
import numpy as np
import pytest

from oracle.weyl import Weyl, tau
from synth import param_phase_circuit

pytestmark = pytest.mark.gpu

# a chain of n steps, each a few dozen roundings (2^-53) of transfer matrices of norm 1
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


def _rows(exps, phase, n, d):
    return [Weyl(p, e[:n], e[n:], d) for e, p in zip(exps, phase)]


def _product(rows, x, z, n, d):
    """prod_q rows(X_q)^x_q rows(Z_q)^z_q: what the tableau of rows makes of W(x, z)."""
    out = Weyl.identity(n, d)
    for q in range(n):
        out = out * rows[n + q] ** int(x[q]) * rows[q] ** int(z[q])
    return out


def _contract(bra, ket, ops=None):
    """<bra| (x)_j ops[j] |ket> of two lists of (chi_l, d, chi_r) tensors."""
    e = np.ones((1, 1), dtype=complex)
    for j, (a, b) in enumerate(zip(bra, ket)):
        if ops is not None and ops[j] is not None:
            b = np.einsum("st,atb->asb", ops[j], b)
        t = np.tensordot(e, b, axes=(1, 0))                  # (a, s, d)
        e = np.tensordot(a.conj(), t, axes=((0, 1), (0, 1)))
    return complex(e[0, 0])


def _sites(sim, n):
    return [np.asarray(sim.site(j)) for j in range(n)]


def _state(G, d, n, chi, t, layers, seed, cutoff=1e-12):
    """Truncated to chi without disentangling: bonds fill up to the limit."""
    sim = G.Simulator(n, d, chi_max=chi, cutoff=cutoff, cluster_size=4)
    gates, _ = param_phase_circuit(n, d, layers, t, seed)
    sim.run(G.ops_from_gates(gates, d, disentangle_after_t=False))
    sim.sync()
    return sim


def _strings(sites, d, n):
    """The four strings of largest |<P>| among those on one site and some on two and three, the last ones at random."""
    rng = np.random.default_rng(n)
    found = []
    for k in range(n * (d * d - 1) + 2 * n):
        px, pz = np.zeros(n, dtype=int), np.zeros(n, dtype=int)
        one = k < n * (d * d - 1)
        for q in [k % n] if one else rng.choice(n, size=min(n, 2 + k % 2), replace=False):
            v = 1 + k // n if one else int(rng.integers(1, d * d))
            px[q], pz[q] = v // d, v % d
        p = Weyl(0, px, pz, d)
        found.append((abs(_contract(sites, sites, _matrices(p, n))), k, px, pz))
    found.sort(key=lambda f: (-f[0], f[1]))
    assert found[0][0] > 1e-3
    return [f[2:] for f in found[:4] + found[-2:]]


def _matrices(p, n):
    return [p.local_matrix(j) if p.x[j] or p.z[j] else None for j in range(n)]


def _staged(dims, d):
    """The rule of the staged route of <W>."""
    full = [1] + list(dims) + [1]
    sites = [a * d * b for a, b in zip(full[:-1], full[1:])]
    return sum(sites) <= 8192 and max(b * b for b in full) <= 128 and max(sites) <= 384


@pytest.mark.parametrize("d,n,chi,t,layers,staged", [
    (2, 2, 2, 2, 8, True), (3, 2, 3, 2, 8, True), (3, 3, 3, 3, 8, True), (2, 7, 8, 6, 8, True), (2, 12, 12, 14, 8, False),
    (3, 9, 11, 8, 8, True), (3, 9, 12, 8, 8, False), (3, 34, 11, 20, 16, True), (3, 40, 11, 24, 16, False),
    (2, 40, 11, 40, 16, True), (2, 44, 11, 48, 16, False)])
def test_expectation_values(G, d, n, chi, t, layers, staged):
    sim = _state(G, d, n, chi, t, layers, 7 * n + chi)
    assert _staged(sim.bond_dims(), d) == staged, sim.bond_dims()
    fwd, inv = _rows(*sim.tableau(), n, d), _rows(*sim.inverse_tableau(), n, d)
    sites = _sites(sim, n)
    for px, pz in _strings(sites, d, n):
        w = _product(fwd, px, pz, n, d)
        p = _product(inv, w.x, w.z, n, d)                    # C^dag W C, phase included
        assert np.array_equal(p.x, px) and np.array_equal(p.z, pz)
        want = tau(d) ** p.r * _contract(sites, sites, _matrices(p, n))
        got = sim.expect_weyl(w.x.astype(np.int32), w.z.astype(np.int32))
        assert abs(got - want) < TOL
    sim.close()


def _shared(ba, bk, d):
    """The rule of the overlap's shared-memory route."""
    a, k = [1] + list(ba) + [1], [1] + list(bk) + [1]
    return all(a[j + 1] * k[j + 1] <= 200 and a[j] * d * k[j + 1] <= 824 for j in range(len(a) - 1))


# one circuit truncated with two cutoffs: bonds of the bra times those of the ket around 200
@pytest.mark.parametrize("d,n,t,cut_a,cut_b,shared", [
    (2, 2, 2, 1e-12, 1e-12, True), (3, 3, 3, 1e-12, 1e-12, True), (3, 7, 6, 0.1, 0.1, True), (3, 7, 6, 0.06, 0.21, True),
    (3, 7, 6, 0.21, 0.06, True), (3, 7, 6, 0.02, 0.21, False), (3, 7, 6, 0.21, 0.02, False), (3, 7, 6, 1e-12, 1e-12, False)])
def test_overlaps_of_different_bonds(G, d, n, t, cut_a, cut_b, shared):
    a, b = (_state(G, d, n, d ** (n // 2), t, 8, 5, cutoff=c) for c in (cut_a, cut_b))
    da, db = a.bond_dims(), b.bond_dims()
    assert _shared(da, db, d) == shared, (da, db)
    want = _contract(_sites(a, n), _sites(b, n))
    got = a.overlap(b)
    assert abs(got - want) < TOL and abs(want) > 1e-3
    a.close()
    b.close()
