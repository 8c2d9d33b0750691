"""Clifford lists longer than the window of gates that is taken at once (256), and inverse rows at every size: the
forward tableau is that of the images' products, and conjugating each inverse row by it gives back the generator, phase included.  The
dense list gives two qudits inverse rows with exponents 2 on nearly every site of the widest register before they take
part in gates, so the sums z(row) . x(row) that are packed three to a word come near their largest value, 4 x 128."""
import numpy as np
import pytest

from oracle import clifford
from oracle.weyl import Weyl
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


def _random_two(rng, d, q):
    shift = tuple(int(v) for v in rng.integers(d, size=4))
    return q, clifford.random_gate_images(int(rng.integers(sp4_order(d))), shift, d)


def _named(G, d, gate, q):
    """(sites, images) of a named gate, its images as the library states them (pinned on the CPU)."""
    img, step = G.named_images(d, gate), 5 if len(q) == 2 else 3
    rows = np.asarray(img).reshape(-1, step)
    return q, [Weyl(r[-1], r[0:-1:2], r[1:-1:2], d) for r in rows]


def _random_list(G, rng, d, n, count):
    return [_random_two(rng, d, tuple(int(v) for v in rng.choice(n, 2, replace=False))) for _ in range(count)]


def _dense_list(G, rng, d, n, count):
    """First gates that make every Z an X Z, then SUMs onto qudits 0 and 1, so that C^dag Z_0 C and C^dag Z_1 C have
    exponents d - 1 nearly everywhere; then gates on those two."""
    out = []
    for q in range(n):   # C^dag Z C = (S^dag)^(d-1) X S^(d-1) = X Z up to a phase
        out += [_named(G, d, G.GATE_S, (q,))] * (d - 1) + [_named(G, d, G.GATE_H, (q,))]
    for t in (0, 1):
        for q in range(2, n):
            out += [_named(G, d, G.GATE_SUM, (q, t))] * (d - 1)
    return out + [_random_two(rng, d, (0, 1)) for _ in range(count)]


def _op(G, q, imgs):
    op = np.zeros((), dtype=G.OP_DTYPE)
    op["kind"], op["q0"], op["q1"] = G.OP_CLIFFORD, q[0], q[1] if len(q) == 2 else -1
    flat = [int(v) for w in imgs for v in [e for a in range(len(q)) for e in (w.x[a], w.z[a])] + [w.r]]
    op["img"][: len(flat)] = flat
    return op


def _conjugate(rows, q, imgs, d):
    """Every row's factors on the sites q replaced by the product of the generators' images."""
    k, seen = len(q), {}
    for row in rows:
        key = tuple(int(v) for s in q for v in (row.x[s], row.z[s]))
        if key not in seen:
            seen[key] = Weyl.identity(k, d)
            for img, power in zip(imgs, key):
                seen[key] = seen[key] * img ** power
        w = seen[key]
        row.r = (row.r + w.r) % (2 * d)
        row.x[list(q)], row.z[list(q)] = w.x, w.z


def _dots(exps, rows, n):
    e = exps[list(rows)].astype(int)
    return int((e[:, n:] @ e[:, :n].T).max())


@pytest.mark.parametrize("d,n,count,build", [(2, 11, 600, _random_list), (3, 12, 513, _random_list), (3, 40, 257, _random_list),
                                             (2, 128, 300, _random_list), (3, 128, 6, _dense_list), (2, 128, 6, _dense_list)])
def test_long_and_dense_lists(G, d, n, count, build):
    gates = build(G, np.random.default_rng(1000 * d + n), d, n, count)
    ref = [Weyl.single(n, d, k % n, "Z" if k < n else "X") for k in range(2 * n)]
    for q, imgs in gates:
        _conjugate(ref, q, imgs, d)
    sim = G.Simulator(n, d, chi_max=4)
    sim.run(np.array([_op(G, q, imgs) for q, imgs in gates], dtype=G.OP_DTYPE))
    sim.sync()
    e, p = sim.tableau()
    assert np.array_equal(e, [np.concatenate([r.x, r.z]) for r in ref]) and np.array_equal(p, [r.r for r in ref])
    ie, ip = sim.inverse_tableau()
    fwd = [Weyl(ph, row[:n], row[n:], d) for row, ph in zip(e, p)]
    for k in range(2 * n):
        back = Weyl(ip[k], np.zeros(n), np.zeros(n), d)
        for q in range(n):
            if ie[k][q]:
                back = back * fwd[n + q] ** int(ie[k][q])
            if ie[k][n + q]:
                back = back * fwd[q] ** int(ie[k][n + q])
        assert back == Weyl.single(n, d, k % n, "Z" if k < n else "X")
    if build is _dense_list:
        # the rows that the gates on the two qudits multiply
        before = G.Simulator(n, d, chi_max=4)
        before.run(np.array([_op(G, q, imgs) for q, imgs in gates[:-count]], dtype=G.OP_DTYPE))
        assert _dots(before.inverse_tableau()[0], (0, 1, n, n + 1), n) >= (d - 1) ** 2 * (n - 2)
        before.close()
    sim.close()
