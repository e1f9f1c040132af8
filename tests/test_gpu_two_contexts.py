"""Two contexts used from two host threads at once: the kernels' shared-memory
allowance belongs to the function on the device, so a launch of one thread may
not depend on what the other asked for last.  The solves are one-cluster teams
(no launch waits for another's)."""
import threading

import numpy as np
import pytest

import oracle
from gpu_util import dev
from paper_2106_07616_gb300 import clouds, rbffd

pytestmark = pytest.mark.gpu


def both(jobs):
    """Run the jobs in threads of their own, started together; their errors."""
    gate, errors = threading.Barrier(len(jobs)), []

    def go(job):
        gate.wait()
        try:
            job()
        except rbffd.RbffdError as e:
            errors.append(str(e))

    ts = [threading.Thread(target=go, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    return errors


def test_solves_of_unlike_size_from_two_threads():
    fps = [clouds.kovasznay(64, dt=0.2), clouds.kovasznay(30, dt=0.4)]
    probs = [rbffd.Problem(rbffd.Context(0), fp, rbffd.PREC_MIXED, precond=rbffd.PRECOND_AMG)
             for fp in fps]

    def job(P, fp):
        for _ in range(60):
            P.simple_iterate(fp.dt, krylov_tol=1e-6)

    assert both([lambda P=P, fp=fp: job(P, fp) for P, fp in zip(probs, fps)]) == []
    for P in probs:
        P.close()


def test_weights_of_unlike_size_from_two_threads():
    jobs = []
    for q, degree in ((66, 6), (12, 2)):
        C = rbffd.Context(0)
        x, y = clouds.jittered_grid(15, seed=q)
        idx = np.ascontiguousarray(oracle.knn(x, y, q))
        a = dev(x), dev(y), q, dev(idx.ravel()), degree
        w = [dev(np.zeros(idx.size)) for _ in range(3)]
        jobs.append(lambda C=C, a=a, w=w: [rbffd.rbffd_weights(C, *a, *w) for _ in range(400)])
    assert both(jobs) == []
