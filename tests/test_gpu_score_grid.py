"""gcamps_score_theta on a grid of one CTA per class and, for tensors past its limit, on the engine's cluster: scores
against the oracle's SVD entropies on both sides of every boundary (warp or CTA a class at 10 rows, chunks of the long
side, wide and tall, the 6561-entry limit), and the choice and evaluation count of the cluster's pruning."""
import numpy as np
import pytest

from oracle.gcamps import GCAMPS

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


@pytest.mark.parametrize("d,cl,cr", [(2, 1, 1), (2, 1, 40), (2, 4, 5), (2, 5, 4), (2, 16, 17), (2, 17, 16), (2, 31, 33),
                                     (3, 1, 1), (3, 3, 27), (3, 27, 3), (3, 3, 11), (3, 11, 10), (3, 27, 27),
                                     (3, 27, 28), (3, 9, 81)])
@pytest.mark.parametrize("kind", [0, 1, 2])
def test_scores_and_choice(G, d, cl, cr, kind):
    rng = np.random.default_rng(10000 * d + 100 * cl + cr)
    shape = (cl * d, d * cr)
    r = max(1, min(shape) // 2)
    th = (rng.standard_normal((shape[0], r)) + 1j * rng.standard_normal((shape[0], r))) @ (
        rng.standard_normal((r, shape[1])) + 1j * rng.standard_normal((r, shape[1])))
    th = (th / np.linalg.norm(th)).reshape(cl, d, d, cr)
    sim = G.Simulator(12, d, chi_max=81, cluster_size=4, score_kind=kind)
    ref = GCAMPS(2, d, chi_max=81, cutoff=1e-12, score_kind=kind)
    s2, vn, choice, evaluated = sim.score_theta(th)
    svs = ref.schmidt_values(th)
    p = [v ** 2 / np.sum(v ** 2) for v in svs]
    assert np.max(np.abs(s2 + np.log([np.sum(q * q) for q in p]))) <= TOL
    assert np.max(np.abs(vn + [np.sum(q[q > 0] * np.log(q[q > 0])) for q in p])) <= TOL
    assert choice == ref.choose(ref.score_keys(th))
    assert 1 <= evaluated <= len(svs)
    sim.close()
