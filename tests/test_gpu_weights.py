"""The weights kernel's lanes-a-cloud variants against the oracle: counts that
leave a warp part filled, every variant and both its limits (q and the number
of clouds), q = m, and singular clouds beside regular ones
of the same warp."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import ctx, dev
from paper_2106_07616_gb300 import clouds, rbffd

pytestmark = pytest.mark.gpu


def gpu_weights(x, y, idx, degree):
    n, q = idx.shape
    w = [torch.full((n, q), np.nan, dtype=torch.float64, device="cuda:0") for _ in range(3)]
    bad = rbffd.rbffd_weights(ctx(), dev(x), dev(y), q, dev(idx.ravel()), degree, *w)
    return bad, [a.cpu().numpy() for a in w]


# (q, degree, n): 4, 8, 16 and 32 lanes by q; fewer clouds move to more lanes
@pytest.mark.parametrize("q,degree,side", [(12, 2, 99), (12, 2, 98), (12, 2, 70), (12, 2, 37),
                                           (6, 1, 101), (20, 3, 71), (24, 3, 51), (28, 3, 51),
                                           (30, 4, 21), (42, 5, 13), (3, 1, 99), (1, 0, 2)])
def test_weights_match_oracle(q, degree, side):
    """Row by row, to the parity tests' 1e-10 of the row's largest weight; where
    the oracle finds a singular cloud (three points of an edge), the same one."""
    x, y = clouds.jittered_grid(side, seed=q + side)
    idx = np.ascontiguousarray(oracle.knn(x, y, q))
    bad, got = gpu_weights(x, y, idx, degree)
    try:
        want = oracle.weights(x, y, idx, degree)
    except ValueError as e:
        assert f"(first singular {bad})" in str(e)
        return
    assert bad == -1
    for g, o in zip(got, want):
        scale = np.maximum(np.abs(o).max(axis=1, keepdims=True), 1e-300)
        err = (np.abs(g - o) / scale).max()
        assert err <= 1e-10, err


@pytest.mark.parametrize("q,degree", [(12, 2), (20, 3), (28, 3), (42, 5)])
def test_singular_clouds_leave_their_neighbours(q, degree):
    """Clouds whose points repeat are zero, the first is named, the rest are
    what they are alone."""
    n = 10007
    x, y = (a[:n].copy() for a in clouds.jittered_grid(101, seed=3))
    idx = oracle.knn(x, y, q)
    ok, regular = gpu_weights(x, y, idx, degree)
    broken = [41, 42, 5000, n - 1]
    for i in broken:
        idx[i, -1] = idx[i, 1]
    bad, got = gpu_weights(x, y, idx, degree)
    assert ok == -1
    rest = np.setdiff1d(np.arange(n), broken)
    assert bad == broken[0]
    for a, b in zip(got, regular):
        assert not a[broken].any()
        assert np.array_equal(a[rest], b[rest])


@pytest.mark.parametrize("slope", [0.0, 1.0, -1.0, 2.0, -0.25])
@pytest.mark.parametrize("q,degree", [(12, 2), (20, 3), (42, 5)])
def test_points_of_a_line_are_singular(q, degree, slope):
    """On y = slope x two columns of the polynomials are one, up to a power of
    two: singular."""
    r = np.random.Generator(np.random.PCG64(q))
    x = np.sort(r.integers(-2**20, 2**20, 3000)).astype(np.float64)  # slope x exact
    x = np.unique(x)
    y = slope * x
    bad, got = gpu_weights(x, y, oracle.knn(x, y, q), degree)
    assert bad == 0
    assert not any(a.any() for a in got)
