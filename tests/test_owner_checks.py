"""The tests of the owner lists in the bounds-checked build, on the CPU: every
entry that a walk along jagged rows reads passes, and offsets that leave their
slice or the lists do not."""

import os
import subprocess

import numpy as np
import pytest

from paper_1311_6811_gb300 import build as libbuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def checks(tmp_path_factory):
    d = tmp_path_factory.mktemp("owners")
    out = d / "owner_checks"
    subprocess.run([libbuild.nvcc(), *libbuild.ARCH, "-std=c++17", "-I", os.path.join(ROOT, "include"),
                    "-I", libbuild.CSRC, os.path.join(ROOT, "tests", "host", "owner_checks.cu"), "-o", str(out)],
                   check=True, capture_output=True)

    def run(rows):
        inp = d / "rows.txt"
        inp.write_text("".join("%d %d %d %d %d %d\n" % tuple(r) for r in rows))
        lines = subprocess.run([str(out), str(inp)], capture_output=True, text=True, check=True).stdout.split()
        return np.array(lines, int).reshape(-1, 2)
    return run


def _jagged_walk(counts):
    """(lane, entry) reads of a slice's lanes, entries relative to the slice."""
    reads, pos = [], 0
    for j in range(max(counts)):
        has = [l for l, n in enumerate(counts) if j < n]
        reads += [(l, pos + k) for k, l in enumerate(has)]
        pos += len(has)
    return reads


def test_every_read_of_a_jagged_walk_passes(checks):
    rng = np.random.default_rng(1)
    for high, base in ((3, 0), (60, 1000), (1, 7)):
        counts = rng.integers(0, high + 1, 32)
        counts[5] = high
        off = base + np.concatenate([[0], np.cumsum(counts)])
        total = int(off[-1]) + 50
        rows = [(off[l], off[l + 1], off[0], off[32], total, off[0] + e) for l, e in _jagged_walk(list(counts))]
        assert len(rows) == counts.sum() and (checks(rows) == 1).all()
        # each entry of the slice is read once
        assert sorted(r[5] for r in rows) == list(range(off[0], off[32]))


def test_offsets_outside_the_lists_fail(checks):
    rows = [(10, 20, 0, 100, 200, 99),    # sound
            (20, 10, 0, 100, 200, 100),   # reversed; one past the slice
            (10, 120, 0, 100, 200, 0),    # past its slice
            (10, 20, 15, 100, 200, 14),   # before its slice; the entry too
            (10, 20, 0, 100, 90, 50),     # the slice past the lists
            (0, 0, 100, 0, 200, 50)]      # a slice that ends before it starts
    got = checks(rows)
    assert got[:, 0].tolist() == [1, 0, 0, 0, 0, 0]
    assert got[:, 1].tolist() == [1, 0, 1, 0, 1, 0]
