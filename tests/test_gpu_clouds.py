"""The cloud search at the shapes where its cell grid and shared-memory lists
can go wrong, bit-exact against the oracle's brute force."""
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
