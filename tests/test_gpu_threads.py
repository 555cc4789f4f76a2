"""Handles of one process in several threads, each on its own stream: the kernels that they share are launched with
the shared memory, clusters and grids of either handle, in turn and at once.  Every solve gives the bits that
it gives alone."""
import threading

import numpy as np
import pytest

import qpgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import paper_2507_02470_gb300 as p
    p.build()
    return p


def side_by_side(jobs, rounds):
    """jobs: callables that solve and return arrays, the first call being the reference."""
    want = [j() for j in jobs]
    failed = []

    def work(j, w):
        try:
            for _ in range(rounds):
                for a, b in zip(j(), w):
                    assert np.array_equal(a, b)
        except BaseException as e:  # noqa: BLE001
            failed.append(e)

    ts = [threading.Thread(target=work, args=a) for a in zip(jobs, want)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not failed, failed


def solving(s, iters):
    def job():
        s.solve(tol=1e-30, max_iter=iters)
        return s.get()[:4]
    return job


SETS = {
    "clusters": ([(66, 20), (700, 200), (2500, 800)], 1, 1500),
    "cluster_and_grid": ([(2500, 800), (3000, 900)], 60, 100),
    "grids": ([(2600, 700), (20_011, 3001), (60_000, 9000)], 60, 60),
    "grids_without_rows": ([(2600, 0), (40_000, 0)], 60, 60),
}


@pytest.mark.parametrize("name", list(SETS))
def test_resident_solves_in_threads(pkg, name):
    sizes, iters, rounds = SETS[name]
    ss = [pkg.Solver(qpgen.large_cqp(n=n, m=m, seed=i)) for i, (n, m) in enumerate(sizes)]
    side_by_side([solving(s, iters) for s in ss], rounds)
    for s in ss:
        s.close()


def test_batches_in_threads(pkg):
    """Small and large factors copied to shared memory, and none: one kernel at several sizes of shared memory."""
    groups = [[40, 60, 90], [300, 350, 400], [1500, 2500], [3200, 700]]
    bs = [pkg.BatchSolver([qpgen.portfolio(10 * g + i, n=n) for i, n in enumerate(ns)], **({} if g % 2 else {"autotune": 0}))
          for g, ns in enumerate(groups)]

    def job(b):
        def run():
            b.solve(tol=1e-30, max_iter=25)
            return [v for i in range(b.count) for v in b.get(i)[:3]]
        return run
    side_by_side([job(b) for b in bs], 80)
    for b in bs:
        b.close()
