"""The batched launches' team plan (host only): every solve once, the caps and
the grid kept, and never slower than equal teams under the same cost."""
import numpy as np
import pytest

from paper_2106_07616_gb300 import _build, rbffd

LAT = 512.0


def equal_span(work, cap, rows, cmax):
    team, _, size, nteams = rbffd.plan_work_lists(work, cap, rows, cmax)
    t = np.zeros(nteams)
    for i, k in enumerate(team):
        t[k] += work[i] / rows[i] * (LAT + rows[i] / size)
    return t.max()


@pytest.mark.parametrize("m,lo,hi", [(1, 100, 200), (2, 144, 90000), (4, 5000, 9000),
                                     (16, 1000, 64000), (64, 1000, 64000), (256, 1000, 64000),
                                     (304, 200, 300)])
def test_plan_teams(m, lo, hi):
    _build.build()
    rng = np.random.Generator(np.random.PCG64(m))
    cmax = 304
    rows = np.exp(rng.uniform(np.log(lo), np.log(hi), m)).astype(np.int32)
    work = rows * rng.integers(20, 150, m).astype(np.float64)
    cap = np.minimum(160, np.maximum(1, rows // 60)).astype(np.int32)
    team, ctas, nctas, span = rbffd.plan_teams(work, cap, rows, cmax)
    assert team.min() == 0 and nctas <= cmax
    assert set(team) == set(range(team.max() + 1))
    per_team = [set(ctas[team == t]) for t in range(team.max() + 1)]
    assert all(len(s) == 1 for s in per_team)
    assert sum(s.pop() for s in per_team) == nctas
    assert (ctas >= 1).all() and (ctas <= cap).all()
    t = np.zeros(team.max() + 1)
    for i, k in enumerate(team):
        t[k] += work[i] / rows[i] * (LAT + rows[i] / ctas[i])
    assert span == pytest.approx(t.max(), rel=1e-12)
    assert span <= equal_span(work, cap, rows, cmax) * (1 + 1e-9)


def test_plan_teams_rejects_bad_input():
    with pytest.raises(rbffd.RbffdError):
        rbffd.plan_teams([1.0], [0], [10], 4)
    with pytest.raises(rbffd.RbffdError):
        rbffd.plan_teams([-1.0], [1], [10], 4)


def plain_search(work, cap, rows, cmax):
    """The plan's span by a search that leaves nothing out."""
    m, best = len(work), np.inf
    order = np.argsort(-work, kind="stable")
    g, gmax = 1, min(m, cmax)
    while g <= gmax:
        w, lat, most = np.zeros(g), np.zeros(g), np.full(g, 160)
        for i in order:
            k = int(np.argmin(w))
            w[k] += work[i]
            lat[k] += work[i] / rows[i] * LAT
            most[k] = min(most[k], cap[i], max(1, (rows[i] * 8 + 255) // 256))
        c, left = np.ones(g), cmax - g
        while True:
            k = int(np.argmax(lat + w / c))
            if left == 0 or c[k] >= most[k]:
                break
            c[k] += 1
            left -= 1
        best = min(best, float((lat + w / c).max()))
        g = gmax + 1 if g == gmax else min(gmax, g + max(1, g // 16))
    return best


@pytest.mark.parametrize("seed", range(12))
def test_plan_teams_leaves_out_no_shorter_plan(seed):
    """Counts of groups skipped by the bounds hold no shorter plan."""
    _build.build()
    rng = np.random.Generator(np.random.PCG64(seed))
    m, cmax = int(rng.integers(1, 60)), int(rng.choice([60, 152, 304]))
    rows = np.exp(rng.uniform(np.log(100), np.log(100 * 4 ** (1 + seed % 4)), m)).astype(np.int32)
    work = rows * rng.integers(20, 150, m).astype(np.float64)
    cap = np.minimum(160, np.maximum(1, rows // 60)).astype(np.int32)
    *_, span = rbffd.plan_teams(work, cap, rows, cmax)
    assert span == pytest.approx(plain_search(work, cap, rows, cmax), rel=1e-12)
