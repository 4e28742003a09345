"""Gradient and T of a hidden Z block in one launch (narrow next layers): the Z update against the oracle from a perturbed state, at
the edges of its forms' widths, for both searches that follow, with ragged row blocks and communities."""
import numpy as np
import pytest

from conftest import tiny_problem
from oracle import gcn_admm_oracle as orc
from paper_2112_09335_b200 import binding
from parity_utils import push_state, relerr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,widths", [(333, (9, h, c)) for h, c in [(6, 1), (18, 4), (33, 5), (40, 8), (7, 9), (130, 12), (16, 13), (70, 16), (31, 17),
                                                                   (36, 24), (20, 25), (129, 32), (12, 33), (65, 48), (257, 47)]]
                         + [(97, (9, 21, 16, 3)), (200, (9, 260, 29, 40)), (31, (5, 1024, 10))])
def test_z_update(n, widths):
    pr = tiny_problem(seed=n + widths[-1], n=n, widths=widths, n_comm=5, p=min(0.2, 12.0 / n))
    ws = [(0.5 * w).astype(np.float32) for w in pr["W"]]
    X = pr["X"].astype(np.float32)
    g = binding.GcnAdmm(n, pr["row_ptr"], pr["col_idx"], X, pr["y"], pr["mask"], widths, 5, pr["community"], ws, nu=0.7, rho=0.9)
    o = orc.OracleADMM(n, pr["row_ptr"], pr["col_idx"], X, pr["y"], pr["mask"], list(widths), orc.Params(nu=0.7, rho=0.9), 5, pr["community"], ws)
    try:
        rng = np.random.default_rng(n)
        L, M = len(widths) - 1, 5
        Z = [None] + [o.Z[l] + 0.1 * rng.standard_normal(o.Z[l].shape) for l in range(1, L + 1)]
        push_state(g, o, Z=Z, U=0.1 * rng.standard_normal(o.U.shape), W=[None] + [w.astype(np.float64) for w in ws],
                   tau=[None] + [0.37] * L, theta=[None] + [[0.23] * M for _ in range(1, L)])
        o.forced_tol = 1e-4
        for l in range(1, L):
            push_state(g, o, Z=Z, theta=[None] + [[0.23] * M for _ in range(1, L)])
            g.step_block(binding.PHASE_Z, l)
            trials = g.decisions()["trial_z"][0, l - 1]
            got = g.get_state(binding.ST_Z, l)
            for m in range(M):
                want, _, rec = o.update_Z(l, m, o.W, forced=int(trials[m]))
                assert rec["ok"], (l, m, rec)               # the accepted trial passes in fp64, the one before it fails
                # a step is G / theta: fp32 sums of at most 48 and 1024 products, 1e-5 as for every single block
                assert relerr(got[o.V[m]], want) <= 1e-5, (l, m)
    finally:
        g.destroy()
