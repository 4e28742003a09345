"""Host buffers of every size class (read and written inside the permuting kernel, staged in one part, staged in several,
page-locked), device memory that comes back to later handles, and handles made and destroyed by several threads."""
import threading

import numpy as np
import pytest

from conftest import tiny_problem
from paper_2112_09335_b200 import binding

pytestmark = pytest.mark.gpu


def handle(pr, **kw):
    return binding.GcnAdmm(pr["n"], pr["row_ptr"], pr["col_idx"], pr["X"].astype(np.float32), pr["y"], pr["mask"], pr["widths"],
                           pr["n_comm"], pr["community"], [w.astype(np.float32) for w in pr["W"]], nu=0.05, rho=0.08, **kw)


@pytest.mark.parametrize("n,width", [(70, 3), (3000, 21), (3000, 22), (3000, 349), (3000, 350), (3000, 1053)])
@pytest.mark.parametrize("pinned", [False, True])
def test_state_round_trip(n, width, pinned):
    """Z_1 of n x width floats: 840 bytes, either side of 256 KB, either side of a 4 MB part, and three parts and a bit."""
    import torch
    pr = tiny_problem(70, n=n, widths=(5, width, 3), n_comm=4, p=3.0 / n)
    g = handle(pr)
    try:
        rng = np.random.default_rng(width)
        z = rng.standard_normal((n, width)).astype(np.float32)
        w = rng.standard_normal((5, width)).astype(np.float32)
        if pinned:
            z, w = (torch.from_numpy(a).pin_memory().numpy() for a in (z, w))
        for _ in range(2):
            g.set_state(binding.ST_Z, 1, z)
            g.set_state(binding.ST_W, 1, w)
            g.set_state(binding.ST_THETA, 1, np.arange(1.0, 5.0))
            assert np.array_equal(g.get_state(binding.ST_Z, 1), z)
            assert np.array_equal(g.weights(1), w)
            assert np.array_equal(g.get_state(binding.ST_THETA, 1), np.arange(1.0, 5.0))
        logits, labels = g.predict()
        assert np.array_equal(labels, logits.argmax(axis=1))
    finally:
        g.destroy()


def test_handles_on_recycled_memory_and_from_threads():
    """Handles of other sizes leave their contents in the slabs later ones are cut from: results must not depend on it."""
    small, big = tiny_problem(71, n=300, widths=(7, 11, 4), n_comm=3), tiny_problem(72, n=900, widths=(7, 30, 9, 5), n_comm=5, p=0.02)

    def run(pr):
        g = handle(pr)
        try:
            g.step(4)
            return [g.weights(l) for l in range(1, len(pr["widths"]))] + [g.get_state(binding.ST_U)]
        finally:
            g.destroy()
    want = {id(p): run(p) for p in (small, big)}
    bad = []

    def work():
        for p in (big, small, small, big):
            if not all(np.array_equal(a, b) for a, b in zip(run(p), want[id(p)])):
                bad.append(p["n"])
    threads = [threading.Thread(target=work) for _ in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_idle_memory_goes_back_on_request():
    """A destroyed handle's slab stays with the process until release_idle(); a live handle keeps its own."""
    import torch
    small, big = tiny_problem(73, n=300, widths=(7, 11, 4), n_comm=3), tiny_problem(74, n=5000, widths=(7, 4000, 4), n_comm=3, p=6e-4)

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    for pr in (big, small):                         # kernels and the streams of two handles are loaded and made
        g = handle(pr)
        g.step(2)
        g.destroy()
    binding.release_idle()
    before = free()
    live = handle(small)
    live.step(2)
    want = live.get_state(binding.ST_U)
    g = handle(big)
    g.step(2)
    g.destroy()
    slab = 5000 * 4000 * 4 * 5                       # a good part of it: Z_1, H_1 and three scratch matrices
    assert free() < before - slab
    binding.release_idle()
    assert free() > before - (32 << 20)              # the live handle's own slab and what the driver rounds up
    assert np.array_equal(live.get_state(binding.ST_U), want)
    live.step(1)
    assert np.isfinite(live.objective()).all()
    live.destroy()


@pytest.mark.parametrize("n,classes", [(70, 3), (1598, 40), (1599, 40), (30000, 35), (40000, 104)])   # either side of 256 KB together, one part and a bit, five
@pytest.mark.parametrize("pinned", [False, True])
def test_predictions_together_and_apart(n, classes, pinned):
    """Labels and logits in one call, either alone, into pageable and page-locked memory: the same values."""
    import torch
    pr = tiny_problem(73, n=min(n, 2000), widths=(5, 6, classes), n_comm=4, p=0.002)
    if n > 2000:                                    # a ring: a dense adjacency of that size would not fit
        pr["n"] = n
        pr["row_ptr"] = np.arange(0, 2 * n + 1, 2, dtype=np.int64)
        i = np.arange(n)
        pr["col_idx"] = np.sort(np.stack([(i - 1) % n, (i + 1) % n], 1), 1).reshape(-1).astype(np.int32)
        rng = np.random.default_rng(1)
        pr["X"], pr["y"], pr["community"] = rng.standard_normal((n, 5)), rng.integers(0, classes, n), rng.integers(0, 4, n)
        pr["mask"] = (rng.random(n) < 0.3).astype(np.uint8)
    g = handle(pr)
    try:
        lib = binding.load()
        def buf(shape, dt):
            t = torch.full(shape, -1, dtype=dt)
            return (t.pin_memory() if pinned else t).numpy()
        logits, labels = buf((n, classes), torch.float32), buf((n,), torch.int32)
        assert lib.gcn_admm_predict(g._h, binding._ptr(logits), binding._ptr(labels)) == 0
        assert np.array_equal(labels, logits.argmax(axis=1))
        only = buf((n, classes), torch.float32), buf((n,), torch.int32)
        assert lib.gcn_admm_predict(g._h, binding._ptr(only[0]), None) == 0 and lib.gcn_admm_predict(g._h, None, binding._ptr(only[1])) == 0
        assert np.array_equal(only[0], logits) and np.array_equal(only[1], labels)
        assert abs(g.objective()[5] - (labels == pr["y"])[pr["mask"] != 0].mean()) < 1e-12
    finally:
        g.destroy()
