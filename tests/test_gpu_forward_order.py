"""Problem 1's forward pass in both orders of product and propagation (the narrow next layer's product first on graphs of many
entries per row, the propagation first otherwise) and with H_1 kept or formed again; against the oracle's."""
import numpy as np
import pytest

from conftest import tiny_problem
from oracle import gcn_admm_oracle as orc
from paper_2112_09335_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p,widths", [
    (60, 0.02, (6, 40, 3)),            # few entries per row: propagation first
    (60, 0.30, (6, 40, 3)),            # product first
    (600, 0.05, (9, 130, 3)),          # the same on the tensor cores
    (60, 0.30, (6, 40, 3, 2)),         # both in one pass: 40 -> 4 padded columns, then 4 -> 4
    (60, 0.30, (6, 8, 80, 8, 5)),      # wider, narrower, about equal
    (60, 0.30, (6, 80, 20, 4)),        # product first twice
])
def test_logits_in_both_orders(n, p, widths):
    pr = tiny_problem(7, n=n, widths=widths, n_comm=3, p=p)
    w32 = [w.astype(np.float32) for w in pr["W"]]
    x32 = pr["X"].astype(np.float32)
    g = binding.GcnAdmm(n, pr["row_ptr"], pr["col_idx"], x32, pr["y"], pr["mask"], pr["widths"], 3, pr["community"], w32)
    o = orc.OracleADMM(n, pr["row_ptr"], pr["col_idx"], x32, pr["y"], pr["mask"], pr["widths"], orc.Params(), 3,
                       pr["community"], w32)
    try:
        for fresh in (True, False):
            if not fresh:
                w1 = (w32[0] * 0.5).astype(np.float32)
                g.set_state(binding.ST_W, 1, w1)
                o.W[1] = w1.astype(np.float64)
            want, _ = o.predict()
            logits, labels = g.predict()
            assert np.abs(logits - want).max() <= 5e-6 * np.abs(want).max()
            assert np.array_equal(labels, np.argmax(logits, axis=1))
            assert g.objective()[5] == np.mean((labels == pr["y"])[pr["mask"] != 0])
    finally:
        g.destroy()
