"""Device memory of a handle against what its arrays need."""
import numpy as np
import pytest

from conftest import tiny_problem
from paper_2112_09335_b200 import binding

pytestmark = pytest.mark.gpu

MB = 1 << 20


def handle(pr, **kw):
    return binding.GcnAdmm(pr["n"], pr["row_ptr"], pr["col_idx"], pr["X"].astype(np.float32), pr["y"], pr["mask"], pr["widths"],
                           pr["n_comm"], pr["community"], [w.astype(np.float32) for w in pr["W"]], **kw)


def memory_of(make, count=1):
    """Device memory that `count` handles hold, after a first round has loaded kernels and made streams."""
    import torch
    for _ in range(2):
        binding.release_idle()
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        made = [make() for _ in range(count)]
        torch.cuda.synchronize()
        used = free - torch.cuda.mem_get_info()[0]
        for g in made:
            g.destroy()
    binding.release_idle()
    return used


def test_small_handles_take_little():
    pr = tiny_problem(75, n=200, widths=(6, 9, 4), n_comm=3)
    assert memory_of(lambda: handle(pr), count=8) <= 8 * 4 * MB      # a slab of 2 MB each, and as much again for the driver


def test_depth_costs_the_state_of_a_layer_and_no_more():
    """Six layers: Z, H and P of each, U, three scratch matrices of the widest, two of the last layer's width, the weights, the
    gradient and its split sums (4 x 148 of the largest, and of the last layer for its own line of launches)."""
    n, widths = 8000, (16, 256, 256, 256, 256, 256, 8)
    pr = tiny_problem(76, n=n, widths=widths, n_comm=3, p=5.0 / n)
    ld, L = [(w + 3) // 4 * 4 for w in widths], len(widths) - 1
    rows = sum(ld[1:]) * 2 + sum(ld[:-1]) + 3 * max(ld) + 3 * ld[-1]
    weights = sum(a * b for a, b in zip(ld, ld[1:]))
    split = 4 * 148 * (256 * 256 + 256 * 8)
    arrays = 4 * (n * rows + 2 * weights + 2 * 256 * 256 + split)
    # tables of 48 k stored entries, and rounding; a matrix of 256 columns more per hidden layer would be 33 MB
    assert memory_of(lambda: handle(pr)) <= arrays + 12 * MB
