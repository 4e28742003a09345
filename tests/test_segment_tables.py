"""The work lists of the closed-form search of the last hidden layer (host side): every segment of every row appears exactly
once, in its community, with its length and its row's normaliser; rows and split segments are covered once; slots are
contiguous per community.  Checked through a small host-only program on seeded graphs against brute force."""
import os
import subprocess

import numpy as np
import pytest

from conftest import random_graph

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2112_09335_b200", "csrc")


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    exe = tmp_path_factory.mktemp("seg") / "seg"
    subprocess.run(["g++", "-std=c++17", "-O1", "-fopenmp", "-I", CSRC, os.path.join(HERE, "segment_tables_harness.cpp"), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("n,p,m,limit,target,rows", [(1, 0.0, 1, 256, 32, 8), (60, 0.2, 3, 4, 8, 7), (300, 0.1, 7, 6, 64, 50), (3000, 0.004, 13, 256, 32, 42)])
def test_every_segment_once(harness, n, p, m, limit, target, rows):
    rng = np.random.default_rng(n)
    row_ptr, col_idx, A = random_graph(rng, n, p)
    comm = rng.integers(0, m, size=n)
    comm[:m] = np.arange(m)
    text = f"{n} {m} {limit} {target} {rows}\n" + " ".join(map(str, row_ptr)) + "\n" + " ".join(map(str, col_idx)) + "\n" + " ".join(map(str, comm)) + "\n"
    out = subprocess.run([harness], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    order = np.lexsort((np.arange(n), comm))
    full = (A + np.eye(n))[order][:, order]
    c = comm[order]
    want = {}
    for i in range(n):
        for k in np.unique(c[full[i] > 0]):
            want[(i, int(k))] = int(((full[i] > 0) & (c == k)).sum())
    got, covered, pieces, slots = {}, np.zeros(n, dtype=int), {}, {}
    for line in out:
        f = line.split()
        if not f:
            continue
        if f[0] == "seg":            # row, community, length, slot
            key = (int(f[1]), int(f[2]))
            assert key not in got and int(f[3]) <= limit
            got[key] = int(f[3])
            slots.setdefault(int(f[2]), set()).add(int(f[4]))
        elif f[0] == "rows":         # first, count, community, slot
            covered[int(f[1]):int(f[1]) + int(f[2])] += 1
            assert (c[int(f[1]):int(f[1]) + int(f[2])] == int(f[3])).all()
            slots.setdefault(int(f[3]), set()).add(int(f[4]))
        elif f[0] == "piece":        # row, community, length, slot
            key = (int(f[1]), int(f[2]))
            pieces[key] = pieces.get(key, 0) + int(f[3])
            slots.setdefault(int(f[2]), set()).add(int(f[4]))
        elif f[0] == "slots":
            ptr = list(map(int, f[1:]))
    assert (covered == 1).all()
    assert {**got, **pieces} == want and not set(got) & set(pieces)
    for k in range(m):
        assert slots[k] == set(range(ptr[k], ptr[k + 1]))
