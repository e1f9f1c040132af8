"""The partial sums of a resident team's exchanges (host only): a CTA that has
left one exchange writes the partials of the next while a slower CTA still
reads, so consecutive exchanges of a solve may share no byte, whatever their
number of values and type.  Every sequence of exchanges the solvers can make
is walked with the slots that csrc/resident.cuh gives them."""
import os
import subprocess

import pytest

from paper_2106_07616_gb300 import _build

MAIN = """
#include "resident.cuh"
using namespace rbffd;
int main() {
  printf("sizes %zu %zu %d %d\\n", RES_SHARE_BYTES, RES_PART_BYTES, RES_MAXB, RES_CLUSTER);
  for (unsigned e = 0; e < 2; ++e)
    for (int v = 0; v <= 32; ++v) {
      for (size_t bytes = 4; bytes <= 8; bytes += 4)
        printf("grid %u %zu %d %zu\\n", e, bytes, v, res_slot(e, v, 0, bytes));
      for (int vmax = v > 0 ? v : 1; vmax <= 32; ++vmax)
        printf("cluster %u %d %d %d\\n", e, vmax, v, res_cluster_slot(e, vmax, v, 0));
    }
}
"""


@pytest.fixture(scope="module")
def table(tmp_path_factory):
    d = tmp_path_factory.mktemp("slots")
    (d / "slots.cu").write_text(MAIN)
    exe = str(d / "slots")
    cmd = ["nvcc", *_build.ARCH, "-std=c++17", "-I", os.path.join(_build.HERE, "csrc"), "-I",
           _build.INCLUDE, "-o", exe, str(d / "slots.cu")]
    subprocess.run(cmd, check=True, capture_output=True)
    out = {}
    for line in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n"):
        w = line.split()
        if w:
            out[(w[0],) if w[0] == "sizes" else (w[0], *map(int, w[1:4]))] = \
                list(map(int, w[1:] if w[0] == "sizes" else w[4:]))
    return out


# A solver: what it may do next after each of its exchanges.  (V, bytes) is an
# exchange of V values on the array named with it, BAR a barrier alone.
BAR = None


def ir(nr, pt):  # k_ir_res: residual, phases A and C, the update's barrier
    return {"start": ["R", "R0"], "R0": ["R"], "R": ["A", "undo"], "undo": ["R"], "A": ["C", "x"],
            "C": ["A", "x"], "x": ["R"]}, {
        "R0": BAR, "undo": BAR, "x": BAR, "R": (3 * nr, 8, "f64", 3 * nr),
        "A": (2 * nr, pt, "sums", 5 * nr), "C": (5 * nr, pt, "sums", 5 * nr)}


def bicg(nr, bars):  # k_bicg_res: start, (re)starts, phases A and C, `bars` barriers in the cycle
    step, what = {"start": ["i", "s"], "s": ["i"], "i": ["I"]}, {
        "s": BAR, "i": BAR, "I": (2 * nr, 8, "sums", 5 * nr), "A": (3 * nr, 8, "sums", 5 * nr),
        "C": (5 * nr, 8, "sums", 5 * nr)}
    for name, after in (("A", ["I", "C"]), ("C", ["A"])):
        first = name + "0" if bars else name
        for k in range(bars):
            step[name + str(k)] = [name + str(k + 1) if k + 1 < bars else name]
            what[name + str(k)] = BAR
        for a in after:
            step.setdefault(a, []).append(first)
    step["A"].append("i")
    step["C"].append("i")
    return step, what


def fgmres(cycle):  # k_fgmres_res: residual, restart, `cycle` barriers, two passes of D products
    step = {"start": ["T", "s"], "s": ["T"], "T": ["r"], "r": ["c0"], "x": ["T"]}
    what = {"s": BAR, "r": BAR, "x": BAR, "T": (2, 8, "f64", 2)}
    for k in range(cycle):
        step["c%d" % k] = ["c%d" % (k + 1)] if k + 1 < cycle else ["P%d" % d for d in (2, 31)]
        what["c%d" % k] = BAR
    for d in (2, 31):
        what["P%d" % d] = what["Q%d" % d] = (d, 4, "sums", 32)
        step["P%d" % d], step["Q%d" % d] = ["Q%d" % d], ["c0", "x"]
    return step, what


SOLVERS = {"ir_%d_%d" % (nr, pt): ir(nr, pt) for nr in (1, 2) for pt in (4, 8)}
SOLVERS.update({"bicg_jacobi_%d" % nr: bicg(nr, 0) for nr in (1, 2)})
SOLVERS.update({"bicg_amg_%d" % k: bicg(1, k) for k in (4, 5)})
SOLVERS.update({"fgmres_%d" % k: fgmres(k) for k in (3, 4)})


def walk(solver, span):
    """Every reachable pair of consecutive exchanges: the byte ranges they
    share.  span(exchange, parity) -> (array, begin, end)."""
    step, what = solver
    seen, todo, bad = set(), [("start", 1)], []
    while todo:
        at, parity = todo.pop()  # parity of the exchange `at`
        for nxt in step[at]:
            if at != "start" and what[at] and what[nxt]:
                a, b = span(what[at], parity), span(what[nxt], 1 - parity)
                if a[0] == b[0] and a[1] < b[2] and b[1] < a[2]:
                    bad.append((at, nxt, parity))
            if (nxt, 1 - parity) not in seen:
                seen.add((nxt, 1 - parity))
                todo.append((nxt, 1 - parity))
    return bad


@pytest.mark.parametrize("name", sorted(SOLVERS))
def test_consecutive_exchanges_share_no_slot(table, name):
    share, part, maxb, cluster = table[("sizes",)]
    assert part >= 2 * share

    def grid(ex, parity):  # the last value's CTAs end before the next value's begin
        begin, end = (table[("grid", parity, ex[1], v)][0] for v in (0, ex[0]))
        assert end - begin == ex[0] * ex[1] * maxb and 0 <= begin and end <= share
        return "part", begin, end

    def in_cluster(ex, parity):
        begin, end = (table[("cluster", parity, ex[3], v)][0] for v in (0, ex[0]))
        assert end - begin == ex[0] * cluster and end <= 2 * ex[3] * cluster
        return ex[2], begin, end

    assert walk(SOLVERS[name], grid) == []
    assert walk(SOLVERS[name], in_cluster) == []


def test_the_walk_finds_halves_that_depend_on_the_number_of_values():
    def span(ex, parity):
        return "part", parity * ex[0] * ex[1], (parity + 1) * ex[0] * ex[1]

    found = {k for k, s in SOLVERS.items() if walk(s, span)}
    assert {k for k in SOLVERS if k.startswith(("ir", "bicg_jacobi"))} <= found
