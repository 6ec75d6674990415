"""Dealing of segments (csrc/segments.h), on the CPU: every plane of every column goes to one block,
the lists are those of the plain level-by-level deal, and many columns are dealt in little time."""
import math
import os
import random
import subprocess
import time

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1802_00438_gb300", "csrc")
DRIVER = r"""
#include <cstdio>
#include "segments.h"
int main()   // stdin: nz slots fill edge tol first last nspeed cols; stdout: budget, then the segments
{
    int nz, slots, cols, uneven;
    double fill, edge, tol, first, last;
    while (std::scanf("%d %d %lf %lf %lf %lf %lf %d %d", &nz, &slots, &fill, &edge, &tol, &first, &last, &uneven,
                      &cols) == 9) {
        std::vector<double> w(cols, 1.0), speed;
        w.front() = first;
        w.back() = last;
        for (int b = 0; uneven && b < slots; b++) speed.push_back(1.0 + 0.04 * (1.0 - 2.0 * b / slots));
        std::vector<stn::Segment> out;
        stn::SegmentDealer d(nz, slots, fill, edge, w, speed);
        const double b = d.best(tol, &out);
        std::printf("%.17g %.17g %zu\n", b, d.best(tol, nullptr), out.size());
        for (const stn::Segment &q : out) std::printf("%d %d %d %d\n", q.col, q.z0, q.z1, q.block);
    }
}
"""


@pytest.fixture(scope="module")
def deal(tmp_path_factory):
    d = tmp_path_factory.mktemp("segments")
    (d / "driver.cpp").write_text(DRIVER)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, "-o", str(d / "driver"), str(d / "driver.cpp")], check=True)

    def run(*case):
        r = subprocess.run([str(d / "driver")], input=" ".join(map(repr, case)), capture_output=True, text=True,
                           check=True).stdout.split("\n")
        b, est, n = r[0].split()
        segs = [tuple(map(int, x.split())) for x in r[1:1 + int(n)]]
        return float(b), float(est), segs
    return run


def plain(nz, slots, fill, edge, first, last, uneven, cols, budget):
    """One deal, level by level, everything sorted at every level; None: the budget is too small."""
    w = [first if c == 0 and cols > 1 else last if c == cols - 1 else 1.0 for c in range(cols)]
    blocks = [[budget * (1.0 + 0.04 * (1.0 - 2.0 * b / slots)) if uneven else budget, b] for b in range(slots)]
    rest, spare, out = [(c, 0) for c in range(cols)], [], []
    while rest:
        if not blocks:
            if not spare:
                return None
            blocks, spare = sorted(spare, key=lambda b: (-b[0], b[1])), []
        if len(rest) > len(blocks):
            rest.sort(key=lambda q: (-(nz - q[1]) * w[q[0]], q[0]))
        level, rest = rest[:len(blocks)], rest[len(blocks):]
        for (c, z0), b in zip(level, blocks):
            h, fixed = nz - z0, fill + (edge if z0 == 0 else 0.0)
            take = max(1, int(min(h, math.floor((b[0] - fixed) / w[c]))))
            if take == h and take > 1 and fixed + edge + h * w[c] > b[0]:
                take = max(1, min(h - 1, math.floor((b[0] - fixed - edge) / w[c])))
            out.append((c, z0, z0 + take, b[1]))
            if take < h:
                rest.append((c, z0 + take))
            else:
                b[0] -= fixed + edge + take * w[c]
                if b[0] >= fill + 4:
                    spare.append(b)
        blocks = blocks[len(level):]
        rest.sort()
    return out


def load(segs, nz, slots, fill, edge, first, last, cols):
    w = [first if c == 0 and cols > 1 else last if c == cols - 1 else 1.0 for c in range(cols)]
    cost = [0.0] * slots
    for c, z0, z1, b in segs:
        cost[b] += fill + (edge if z0 == 0 else 0.0) + (edge if z1 == nz else 0.0) + (z1 - z0) * w[c]
    return max(cost)


def covered(segs, nz, slots, cols):
    per = [[] for _ in range(cols)]
    for c, z0, z1, b in segs:
        assert 0 <= b < slots
        per[c].append((z0, z1))
    for p in per:
        p.sort()
        assert p[0][0] == 0 and p[-1][1] == nz
        assert all(a[1] == b[0] for a, b in zip(p, p[1:])) and all(a < b for a, b in p)


def test_lists(deal):
    rng = random.Random(11)
    for _ in range(120):
        slots = int(math.exp(rng.uniform(0, math.log(300))))
        nz = int(math.exp(rng.uniform(0, math.log(600))))
        cols = rng.randint(1, min(8 * slots, 700))
        fill, edge = rng.choice([2.0, 8.0, 10.0, 12.5]), rng.choice([0.0, 12.0, 24.0])
        first, last, uneven = 1.05, rng.choice([1.05, 1.45]), rng.randint(0, 1)
        b, est, segs = deal(nz, slots, fill, edge, 0.25, first, last, uneven, cols)
        covered(segs, nz, slots, cols)
        assert est == b
        assert segs == plain(nz, slots, fill, edge, first, last, uneven, cols, b)


@pytest.mark.parametrize("nz,slots,cols,fill,edge", [(4, 152, 82919, 8.0, 0.0), (10, 1216, 100000, 10.0, 24.0),
                                                     (1, 304, 50000, 5.0, 0.0), (500, 152, 1300, 8.0, 0.0)])
def test_many_columns(deal, nz, slots, cols, fill, edge):
    """More than 8 columns per block: no bisection; within 3 % of the mean share (its last column's
    cut costs a block at most one more fill: 1 %; the budget is raised in steps of 0.25 %)."""
    t = time.perf_counter()
    b, est, segs = deal(nz, slots, fill, edge, 0.25, 1.05, 1.45, 0, cols)
    assert time.perf_counter() - t < 3.0   # 0.1 s with the driver's output; 18 s when sorted at every level
    covered(segs, nz, slots, cols)
    mean = (nz * (cols - 2 + 1.05 + 1.45) + cols * (fill + 2 * edge)) / slots
    assert abs(est - mean) <= 1e-9 * mean
    assert load(segs, nz, slots, fill, edge, 1.05, 1.45, cols) <= 1.03 * mean
