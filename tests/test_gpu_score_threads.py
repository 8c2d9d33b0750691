"""Class scores from several host threads at once, each with its own handle and its own tensor shape: every call
succeeds, and gives what the same call gives alone."""
import threading

import numpy as np
import pytest

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


# two shapes that need different amounts of shared memory, half of the threads each, for the warp-per-class and the
# CTA-per-class kernel; small, so that the calls' host parts overlap often
@pytest.mark.parametrize("d,n,shapes", [(2, 18, [(2, 200), (2, 112)]), (3, 10, [(4, 40), (4, 27)])])
def test_threads_score_different_shapes(G, d, n, shapes):
    rng = np.random.default_rng(d)
    shapes = shapes * 4
    chi = max(max(s) for s in shapes)
    sims = [G.Simulator(n, d, chi_max=chi, cluster_size=4) for _ in shapes]
    thetas = []
    for cl, cr in shapes:
        th = rng.standard_normal((cl, d, d, cr)) + 1j * rng.standard_normal((cl, d, d, cr))
        thetas.append(th / np.linalg.norm(th))
    alone = [sim.score_theta(th) for sim, th in zip(sims, thetas)]
    failures = []
    go = threading.Barrier(len(shapes))

    def work(sim, th, want):
        go.wait()
        for _ in range(3000):
            try:
                got = sim.score_theta(th)
            except G.GcampsError as ex:
                failures.append(repr(ex))
                continue
            if not (np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]) and got[2:] == want[2:]):
                failures.append("a score differs")

    threads = [threading.Thread(target=work, args=a) for a in zip(sims, thetas, alone)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, (len(failures), failures[:3])
    for sim in sims:
        sim.close()
