"""The launches of a step-size search where their dispatch changes: the lane groups of the last hidden layer's search (4, 8, 16,
32 float4 per row of the output) and the segment lengths at which their walk changes, the hidden layers' sums in shared memory
and, with more communities, in global memory, sweeps with few and with many chunks, gradients with few and with many splits,
all class widths of the output rows; against the oracle."""
import numpy as np
import pytest

from conftest import dense_to_csr, tiny_problem
from paper_2112_09335_b200 import binding
from test_gpu_edge_cases import run_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("classes", [1, 4, 5, 8, 9, 16, 17, 24, 25, 32, 33, 40, 41, 48, 49, 64, 65, 96, 97, 128])
def test_output_widths(classes):
    run_pair(tiny_problem(20 + classes, n=90, widths=(6, 9, classes), n_comm=3), n_it=3)


@pytest.mark.parametrize("n_comm", [384, 385])
def test_communities_around_the_shared_memory_of_a_sweep(n_comm):
    """8 warps x 32 bytes per community are kept in shared memory up to 96 KB: 384 communities."""
    run_pair(tiny_problem(60, n=800, widths=(5, 7, 6, 5), n_comm=n_comm, p=0.01), n_it=3)


@pytest.mark.parametrize("classes", [3, 7, 16, 23, 40, 70])
@pytest.mark.parametrize("entries", [2, 4, 23, 47, 127, 300])
def test_lengths_of_segments(classes, entries):
    """The closed form walks segments of 1, 2 and 3 entries, longer ones by a group of lanes, and those of 24 entries or more
    (up to 16 columns), 48 (up to 32) or 128 by a whole warp.  Communities of `entries` fully connected nodes, one more or one
    less, and single edges between them; at 300 the rows are cut and their long segments go in pieces."""
    n_comm = 9 if entries < 100 else 4
    sizes = [max(1, entries + (m % 3) - 1) for m in range(n_comm)]
    comm = np.repeat(np.arange(n_comm), sizes)
    n = len(comm)
    rng = np.random.default_rng(entries)
    cross = np.triu(rng.random((n, n)) < 1.0 / n, 1)
    A = ((comm[:, None] == comm[None, :]) | cross | cross.T).astype(np.float64)
    np.fill_diagonal(A, 0.0)
    pr = tiny_problem(64, n=n, widths=(6, 9, classes), n_comm=n_comm)
    order = rng.permutation(n)
    row_ptr, col_idx = dense_to_csr(A[np.ix_(order, order)])
    pr.update(A=A, row_ptr=row_ptr, col_idx=col_idx, community=comm[order])
    run_pair(pr, n_it=3)


def test_many_chunks_and_a_search_of_several_sweeps():
    """More than 512 chunks of stored entries, and first step parameters so small that every search needs a second sweep."""
    run_pair(tiny_problem(61, n=2600, widths=(6, 10, 8, 4), n_comm=5, p=0.012), n_it=3, tau0=1e-3, theta0=1e-5, bt_max_trials=64)


@pytest.mark.parametrize("classes", [3, 7, 16, 23])
def test_closed_form_with_more_chunks_than_warps(classes):
    """155 k stored entries in chunks of at most 32: more than the 3,552 warps the chip holds, so narrow rows take chunks from the counter."""
    run_pair(tiny_problem(65, n=5000, widths=(6, 9, classes), n_comm=5, p=0.006), n_it=2)


@pytest.mark.parametrize("n", [900, 1100, 5000])
def test_few_and_many_splits_of_the_weight_gradient(n):
    run_pair(tiny_problem(62, n=n, widths=(33, 9, 4), n_comm=4, p=3.0 / n), n_it=2)


@pytest.mark.parametrize("width,more,fewer", [(130, 200, 130), (300, 80, 61), (520, 9, 5)])
def test_handles_with_different_shared_memory_needs(width, more, fewer):
    """The scoring of layer 1 takes 8 warps x (2 V x 512 B + 32 B per community) + 16 B per community of dynamic shared memory
    (V = 2, 4, 8 at these widths of layer 2), above 48 KB for both handles of a pair.  The limit a launch is held to belongs to
    the kernel: the handle with fewer communities, stepped in between, must not lower it for the other."""
    def steps(handles):
        for _ in range(2):
            for g in handles:
                g.step(1)
        return [[g.get_state(binding.ST_Z, 1), g.weights(2)] for g in handles]

    def make(n_comm):
        pr = tiny_problem(63, n=800, widths=(5, 6, width, 3), n_comm=n_comm, p=0.01)
        return binding.GcnAdmm(pr["n"], pr["row_ptr"], pr["col_idx"], pr["X"].astype(np.float32), pr["y"], pr["mask"], pr["widths"],
                               pr["n_comm"], pr["community"], [w.astype(np.float32) for w in pr["W"]], nu=0.05, rho=0.08, use_graph=0)
    a, b = make(more), make(fewer)
    alone = steps([a])
    a.destroy()
    alone += steps([b])
    b.destroy()
    pair = [make(more), make(fewer)]
    together = steps(pair)
    for g in pair:
        g.destroy()
    for got, want in zip(together, alone):
        assert all(np.array_equal(x, y) for x, y in zip(got, want))
