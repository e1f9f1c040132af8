"""The cloud search at the shapes where its cell grid and shared-memory lists
can go wrong, bit-exact against the oracle's brute force."""
import time

import numpy as np
import pytest
import torch

import oracle
from gpu_util import ctx, dev
from paper_2106_07616_gb300 import clouds, rbffd

pytestmark = pytest.mark.gpu


def blob(seed):  # most points in one cell: more candidates than the list holds
    r = np.random.Generator(np.random.PCG64(seed))
    return (np.r_[r.normal(0, 1e-4, 2000), r.uniform(-1, 1, 200)],
            np.r_[r.normal(0, 1e-4, 2000), r.uniform(-1, 1, 200)])


def line(seed):
    x = np.random.Generator(np.random.PCG64(seed)).uniform(0, 1, 700)
    return x, np.zeros(700)


def thin(seed):  # box of aspect 1000
    x, y = clouds.random_cloud(1500, seed)
    return x, 1e-3 * y


def two(seed):  # duplicates: every point twice
    x, y = clouds.random_cloud(400, seed)
    return np.r_[x, x], np.r_[y, y]


CASES = {"blob": blob, "line": line, "thin": thin, "duplicates": two,
         "lattice": lambda s: tuple(a.ravel().astype(float) for a in np.mgrid[0:23, 0:31]),
         "random": lambda s: clouds.random_cloud(3001, s)}


@pytest.mark.parametrize("q", [1, 2, 12, 42, 129])
@pytest.mark.parametrize("case", sorted(CASES))
def test_clouds_match_brute_force(case, q):
    x, y = (np.ascontiguousarray(a) for a in CASES[case](11))
    r = np.random.Generator(np.random.PCG64(q))
    for tag in (None, (r.uniform(size=x.size) < 0.2).astype(np.int8)):
        idx = torch.zeros((x.size, q), dtype=torch.int32, device="cuda:0")
        rbffd.rbffd_build_stencils(ctx(), dev(x), dev(y), None if tag is None else dev(tag), q, idx)
        assert np.array_equal(idx.cpu().numpy(), oracle.knn(x, y, q, tag)), (case, q, tag is None)


def test_graded_cloud_matches_brute_force():
    fp = clouds.cylinder(6000, h0=0.1, hmax=0.5)
    idx = torch.zeros((fp.n, 20), dtype=torch.int32, device="cuda:0")
    rbffd.rbffd_build_stencils(ctx(), dev(fp.x), dev(fp.y), dev(fp.tag), 20, idx)
    assert np.array_equal(idx.cpu().numpy(), oracle.knn(fp.x, fp.y, 20, fp.tag))


def noisy_line(n, noise, seed):
    r = np.random.Generator(np.random.PCG64(seed))
    return np.sort(r.uniform(0, 1, n)), noise * r.uniform(-1, 1, n)


def two_lines(seed):  # clusters far apart: most cells of the long axis are empty
    x, y = noisy_line(1500, 1e-15, seed)
    x[1400:] = 3.0 + 1000.0 * x[1400:]
    return x, y


LONG = {"noise_1e-15": lambda s: noisy_line(3000, 1e-15, s),
        "noise_1e-6": lambda s: noisy_line(3000, 1e-6, s),
        "noise_1e-3": lambda s: noisy_line(3000, 1e-3, s), "two_lines": two_lines}


@pytest.mark.parametrize("q", [2, 20, 129])
@pytest.mark.parametrize("upright", [False, True])
@pytest.mark.parametrize("case", sorted(LONG))
def test_boxes_longer_than_the_grid_match_brute_force(case, upright, q):
    """Aspects beyond what square cells can follow: one column or row of cells
    whose short side is far below the spacing."""
    x, y = LONG[case](5)
    if upright:
        x, y = y, x
    r = np.random.Generator(np.random.PCG64(q))
    for tag in (None, (r.uniform(size=x.size) < 0.2).astype(np.int8)):
        idx = torch.zeros((x.size, q), dtype=torch.int32, device="cuda:0")
        rbffd.rbffd_build_stencils(ctx(), dev(x), dev(y), None if tag is None else dev(tag), q, idx)
        assert np.array_equal(idx.cpu().numpy(), oracle.knn(x, y, q, tag)), (case, q, tag is None)


def test_a_long_line_takes_no_longer_than_a_square_cloud():
    """40 000 points on a line up to rounding: the search's work is that of
    40 000 points (ring by ring along the line it would be 10 000 times that)."""
    def seconds(x, y):
        idx = torch.zeros((x.size, 20), dtype=torch.int32, device="cuda:0")
        a = dev(np.ascontiguousarray(x)), dev(np.ascontiguousarray(y))
        rbffd.rbffd_build_stencils(ctx(), *a, None, 20, idx)
        t = time.perf_counter()
        rbffd.rbffd_build_stencils(ctx(), *a, None, 20, idx)
        return time.perf_counter() - t

    square = seconds(*clouds.random_cloud(40000, 3))
    for x, y in (noisy_line(40000, 1e-15, 3), noisy_line(40000, 1e-15, 3)[::-1]):
        assert seconds(x, y) < 20 * square + 0.01


@pytest.mark.parametrize("n", [262144, 263000, 600001])
def test_many_cells_match_brute_force_on_a_sample(n):
    """Around the number of cells from which the scan's tiles are summed first,
    and well above: every point's cloud holds distinct points in order, and a
    sample's clouds are the brute force's."""
    g = torch.Generator(device="cuda:0").manual_seed(n)
    x, y = (torch.rand(n, generator=g, device="cuda:0", dtype=torch.float64) for _ in range(2))
    q = 12
    idx = torch.zeros((n, q), dtype=torch.int32, device="cuda:0")
    rbffd.rbffd_build_stencils(ctx(), x, y, None, q, idx)
    c = idx.long()
    assert torch.equal(c[:, 0], torch.arange(n, device="cuda:0"))
    d2 = (x[c] - x[:, None]) ** 2 + (y[c] - y[:, None]) ** 2
    assert bool((d2[:, 1:] > d2[:, :-1]).all())
    for i in torch.randint(n, (64,), generator=g, device="cuda:0").tolist() + [0, n - 1]:
        far = (x - x[i]) ** 2 + (y - y[i]) ** 2
        assert torch.equal(torch.topk(far, q, largest=False).indices, c[i])
