"""What a launch that gave up a bounded wait leaves behind.  No kernel is made to give up: the flag it would raise is written
from the host, and the searches that find it raised leave at once, which strands the counters the launches hand to each other
exactly as a wait that ran out does."""
import numpy as np
import pytest

from conftest import tiny_problem
from paper_2112_09335_b200 import binding

pytestmark = pytest.mark.gpu


def handle(pr, **kw):
    return binding.GcnAdmm(pr["n"], pr["row_ptr"], pr["col_idx"], pr["X"].astype(np.float32), pr["y"], pr["mask"], pr["widths"],
                           pr["n_comm"], pr["community"], [w.astype(np.float32) for w in pr["W"]], nu=0.05, rho=0.08, **kw)


def save(g):
    out = [(binding.ST_U, 0)]
    for l in range(1, g.L + 1):
        out += [(binding.ST_W, l), (binding.ST_Z, l), (binding.ST_TAU, l)] + ([(binding.ST_THETA, l)] if l < g.L else [])
    return {k: g.get_state(*k) for k in out}


def load(g, state):
    for k, v in state.items():
        g.set_state(*k, v)


@pytest.mark.parametrize("n,widths,n_comm,p,long_row,use_graph", [
    (300, (6, 9, 4), 3, 0.05, 0, 0),              # closed form only
    (300, (6, 9, 7, 4), 3, 0.05, 0, 0),           # scored sweeps and closed form
    (300, (6, 9, 7, 4), 3, 0.05, 0, 1),           # the same, recorded
    (2600, (6, 10, 8, 5, 4), 5, 0.012, 8, 0),     # many chunks, cut rows, two scored layers
])
def test_a_handle_goes_on_from_a_checkpoint(n, widths, n_comm, p, long_row, use_graph):
    import torch
    pr = tiny_problem(81, n=n, widths=widths, n_comm=n_comm, p=p)
    stream = torch.cuda.Stream()
    kw = dict(long_row=long_row, use_graph=use_graph, stream=stream.cuda_stream)
    g, fresh = handle(pr, **kw), handle(pr, **kw)
    try:
        g.step(3)
        checkpoint = save(g)
        g.set_state(binding.ST_PIPELINE_FLAG, 0, np.array([1], dtype=np.int32))
        g.step(2)
        for l in range(1, g.L):                    # the searches of the hidden layers left at once
            assert np.array_equal(g.get_state(binding.ST_W, l), checkpoint[(binding.ST_W, l)])
        for l in range(1, g.L - 1):
            assert np.array_equal(g.get_state(binding.ST_Z, l), checkpoint[(binding.ST_Z, l)])
        with pytest.raises(binding.GcnAdmmError) as e:
            g.decisions()
        assert e.value.code == -6
        load(g, checkpoint)
        load(fresh, checkpoint)
        g.step(3)
        fresh.step(3)
        a, b = g.decisions(), fresh.decisions()
        assert np.array_equal(a["trial_w"], b["trial_w"]) and np.array_equal(a["trial_z"], b["trial_z"])
        assert (a["trial_z"] >= -1).all()
        for k, v in save(fresh).items():           # a recorded pass may form H_1 afresh one pass earlier than another
            got = g.get_state(*k)
            assert np.array_equal(got, v) if use_graph == 0 else np.allclose(got, v, rtol=1e-3, atol=1e-5 * np.abs(v).max()), k
    finally:
        g.destroy()
        fresh.destroy()
