"""Clifford gates taken several at a time (runs of gates on disjoint qudits) leave the tableaux of the oracle's dense
conjugation, gate by gate: lists of one- and two-qudit gates in any qudit order, with shared and disjoint neighbours,
longer than one window of gates, split by T gates, and a layer as wide as the largest register."""
import numpy as np
import pytest

from oracle import clifford
from oracle.gcamps import GCAMPS
from synth import sp4_order

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


def _gates(rng, d, n, count, layer):
    one = [clifford.H_gate(d), clifford.S_gate(d)]
    for i in range(count):
        if rng.random() < 0.3:
            yield (int(rng.integers(n)),), clifford.images_by_conjugation(one[rng.integers(2)], 1, d)
        else:
            q = (2 * i % (n - 1), 2 * i % (n - 1) + 1) if layer else tuple(int(v) for v in rng.choice(n, 2, replace=False))
            shift = tuple(int(v) for v in rng.integers(d, size=4))
            yield q, clifford.random_gate_images(int(rng.integers(sp4_order(d))), shift, d)


def _op(G, q, imgs):
    op = np.zeros((), dtype=G.OP_DTYPE)
    op["kind"], op["q0"], op["q1"] = G.OP_CLIFFORD, q[0], q[1] if len(q) == 2 else -1
    flat = []
    for w in imgs:
        for a in range(len(q)):
            flat += [int(w.x[a]), int(w.z[a])]
        flat.append(int(w.r))
    op["img"][: len(flat)] = flat
    return op


@pytest.mark.parametrize("d,n,count,layer", [(2, 2, 12, False), (3, 2, 12, False), (3, 9, 90, False),
                                             (2, 33, 80, False), (3, 64, 32, True), (2, 128, 140, True)])
def test_lists_match_gate_by_gate(G, d, n, count, layer):
    rng = np.random.default_rng(100 * d + n)
    ref = GCAMPS(n, d, chi_max=4)
    ops = []
    for q, imgs in _gates(rng, d, n, count, layer):
        ref.apply_clifford(list(q), imgs)
        ops.append(_op(G, q, imgs))
    sim = G.Simulator(n, d, chi_max=4)
    sim.run(np.array(ops, dtype=G.OP_DTYPE))
    sim.sync()
    e, p = sim.tableau()
    re_, rp = ref.tab.exps_phase()
    assert np.array_equal(e, re_) and np.array_equal(p, rp)
    assert sim.stats()["clifford_gates"] == count
    ie, ip = sim.inverse_tableau()
    rows = ref.tab.inverse_rows() if n <= 9 else []
    for k, w in enumerate(rows):
        assert np.array_equal(ie[k], np.concatenate([w.x, w.z])) and ip[k] == w.r
    sim.close()
