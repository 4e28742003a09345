"""The launches of a step-size search where their dispatch changes: the lane groups of the narrow output layer (4, 8, 16
float4 per row, then a whole warp) and their fall back to larger ones when the communities' sums do not fit, sweeps with few
and with many chunks, gradients with few and with many splits, all class widths of the output rows; against the oracle."""
import numpy as np
import pytest

from conftest import tiny_problem
from test_gpu_edge_cases import run_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("classes", [1, 4, 5, 8, 9, 16, 17, 24, 25, 32, 33, 40, 41, 48, 49, 64, 65, 96, 97, 128])
def test_output_widths(classes):
    run_pair(tiny_problem(20 + classes, n=90, widths=(6, 9, classes), n_comm=3), n_it=3)


@pytest.mark.parametrize("n_comm,classes", [(96, 5), (97, 5), (192, 20), (193, 20)])
def test_communities_around_the_limits_of_the_lane_groups(n_comm, classes):
    run_pair(tiny_problem(60, n=800, widths=(5, 7, classes), n_comm=n_comm, p=0.01), n_it=3)


def test_many_chunks_and_a_search_of_several_sweeps():
    """More than 512 chunks of stored entries, and first step parameters so small that every search needs a second sweep."""
    run_pair(tiny_problem(61, n=2600, widths=(6, 10, 8, 4), n_comm=5, p=0.012), n_it=3, tau0=1e-3, theta0=1e-5, bt_max_trials=64)


@pytest.mark.parametrize("n", [900, 1100, 5000])
def test_few_and_many_splits_of_the_weight_gradient(n):
    run_pair(tiny_problem(62, n=n, widths=(33, 9, 4), n_comm=4, p=3.0 / n), n_it=2)
