"""Budgets: what a context holds for speed alone (the kept workspace, the dense
coarse operators, the resident solves' lists) goes back when another
allocation needs the room, and the solves then stream."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import ctx, rel_l2
from paper_2106_07616_gb300 import clouds, rbffd

pytestmark = pytest.mark.gpu
FIELDS = ("u", "v", "p")


def list_bytes(fp):
    """What a problem's lists take: its bytes with and without them."""
    full = rbffd.Problem(ctx(), fp)
    bytes_full = full.nbytes
    full.close()
    C = rbffd.Context(0, hbm_budget=bytes_full - 1)
    P = rbffd.Problem(C, fp)
    bytes_without = P.nbytes
    P.close()
    C.close()
    assert bytes_without < bytes_full
    return bytes_full - bytes_without


def keep_workspace(C, n):
    x, y = clouds.random_cloud(n, 3)
    d = [torch.as_tensor(a, device="cuda:0") for a in (x, y)]
    idx = torch.zeros((n, 12), dtype=torch.int32, device="cuda:0")
    rbffd.rbffd_build_stencils(C, *d, None, 12, idx)


@pytest.mark.parametrize("precision,precond", [
    (rbffd.PREC_FP64, rbffd.PRECOND_AMG), (rbffd.PREC_MIXED, rbffd.PRECOND_AMG_FGMRES),
    (rbffd.PREC_MIXED, rbffd.PRECOND_AMG)])
@pytest.mark.parametrize("flow", ["kovasznay", "cavity"])
def test_budget_of_exactly_the_streaming_solves(flow, precision, precond):
    fp = clouds.kovasznay(64, degree=2, q=12, dt=0.2) if flow == "kovasznay" else \
        clouds.cavity(90, degree=4, q=30, re=100.0)
    full = rbffd.Problem(ctx(), fp, precision, precond=precond)
    full.amg_info()  # uploads the hierarchy
    streaming = full.nbytes - list_bytes(fp)
    full.close()
    C = rbffd.Context(0, hbm_budget=streaming)
    keep_workspace(C, 1000)
    P = rbffd.Problem(C, fp, precision, precond=precond)
    P.simple_iterate(fp.dt, krylov_tol=1e-12, krylov_maxit=100000)
    assert P.nbytes == streaming
    O = oracle.Problem(fp, krylov_tol=1e-12, krylov_maxit=100000)
    O.simple_iterate(fp.dt)
    for k in FIELDS:
        assert rel_l2(P.get(k), O.get(k)) <= 1e-8, k
    # one byte less is refused, as before the resident solves
    D = rbffd.Context(0, hbm_budget=streaming - 1)
    with pytest.raises(rbffd.RbffdError) as e:
        Q = rbffd.Problem(D, fp, precision, precond=precond)
        Q.simple_iterate(fp.dt, krylov_tol=1e-12, krylov_maxit=100000)
    assert e.value.code == rbffd.ENOMEM
    P.close()


def test_what_cannot_fit_takes_nothing():
    """A request the budget would not hold even without them leaves the lists."""
    fp = clouds.kovasznay(64, degree=2, q=12, dt=0.2)
    C = rbffd.Context(0, hbm_budget=64 << 20)
    P = rbffd.Problem(C, fp)
    before = P.nbytes
    with pytest.raises(rbffd.RbffdError) as e:
        rbffd.Problem(C, clouds.kovasznay(250, dt=0.2))
    assert e.value.code == rbffd.ENOMEM
    assert P.nbytes == before
    P.close()


def test_captured_batch_after_its_members_gave_their_lists_back():
    """Members of a batch whose iteration is replayed from a capture lose their
    lists to a third problem: the next iterations run without them."""
    fps = [clouds.cavity(90, degree=4, q=30, re=100.0), clouds.cavity(91, degree=4, q=30, re=100.0)]
    third = clouds.kovasznay(100, dt=0.2)

    def march(C, with_third):
        probs = [rbffd.Problem(C, fp, rbffd.PREC_FP64, precond=rbffd.PRECOND_AMG) for fp in fps]
        B = rbffd.Batch(C, probs)
        B.set_autotune(False)
        for k in range(6):
            if k == 4 and with_third:
                full = sum(P.nbytes for P in probs)
                T = rbffd.Problem(C, third)
                assert sum(P.nbytes for P in probs) < full
            _, _, status = B.iterate([fp.dt for fp in fps], krylov_tol=1e-12, krylov_maxit=100000)
            assert not status.any()
        assert B.graph_stats()[0] >= 1
        return [[P.get(k) for k in FIELDS] for P in probs]

    probe = [rbffd.Problem(ctx(), fp, rbffd.PREC_FP64, precond=rbffd.PRECOND_AMG) for fp in fps]
    for P in probe:
        P.amg_info()
    held = sum(P.nbytes for P in probe)
    last = rbffd.Problem(ctx(), third)
    # a MB more than the batch's tables would need the third problem's lists
    # and a MB of the members'
    budget = held + last.nbytes - list_bytes(third) - (1 << 20)
    assert sum(list_bytes(fp) for fp in fps) > 2 << 20
    for P in (*probe, last):
        P.close()
    want = march(ctx(), False)
    got = march(rbffd.Context(0, hbm_budget=budget), True)
    for a, b in zip(got, want):
        for f, g in zip(a, b):
            assert rel_l2(f, g) <= 1e-8
