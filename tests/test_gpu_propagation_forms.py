"""The forms of the propagation kernels: every lane split (columns per row x sets of entries), vectors of one, two and
four floats, rows in the caller's order, cut and uncut long rows, against the oracle's A~ X."""
import numpy as np
import pytest

from oracle import gcn_admm_oracle as orc
from paper_2112_09335_b200 import binding, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=[(0, 1.0, 4), (2, 1.0, 0), (3, 0.4, 0)], ids=["1000 rows cut", "19717 rows", "67737 rows"])
def case(request):
    index, scale, long_row = request.param          # few rows, tens of thousands, and past the lines of the dispatch rule
    wl = inputs.make_workload(index, scale=scale)
    g = binding.GcnAdmm(wl.n, wl.row_ptr, wl.col_idx, wl.X, wl.y, wl.train_mask, wl.widths, wl.n_comm, wl.community,
                        wl.w_init, long_row=long_row)
    yield wl, g, orc.normalized_adjacency(wl.n, wl.row_ptr, wl.col_idx)
    g.destroy()


@pytest.mark.parametrize("width", [1, 3, 4, 8, 9, 16, 18, 32, 33, 64, 66, 127, 128, 130, 257, 260])
@pytest.mark.parametrize("shift", [0, 1])
def test_device_propagation(case, width, shift):
    """`shift` moves both matrices off the 16-byte boundary their width would allow."""
    import torch
    wl, g, At = case
    x = np.random.default_rng(width).standard_normal((wl.n, width)).astype(np.float32)
    buf = torch.zeros(2, wl.n * width + 4, device="cuda")
    buf[0, shift:shift + wl.n * width] = torch.from_numpy(x).cuda().reshape(-1)
    src, dst = buf[0, shift:].data_ptr(), buf[1, shift:].data_ptr()
    want = At @ x.astype(np.float64)
    scale = abs(At) @ np.abs(x.astype(np.float64)) + 1e-30
    torch.cuda.synchronize()
    for _ in range(2):                              # the counters of the cut rows are left ready for the next call
        buf[1] = -7.0
        torch.cuda.synchronize()
        g.propagate(src, width, dst)
        got = buf[1, shift:shift + wl.n * width].reshape(wl.n, width).cpu().numpy()
        assert np.max(np.abs(got - want) / scale) < 1e-6
        assert float(buf[1, shift + wl.n * width]) == -7.0


@pytest.mark.parametrize("width", [20, 21, 30, 35, 36, 42, 47, 48, 49])
def test_lane_splits_of_narrow_operands(case, width):
    """Two and three vectors per lane, whole and ragged; rows of vectors of one, two and four floats."""
    import torch
    wl, g, At = case
    x = np.random.default_rng(width).standard_normal((wl.n, width)).astype(np.float32)
    src, dst = torch.from_numpy(x).cuda(), torch.full((wl.n, width), -7.0, device="cuda")
    torch.cuda.synchronize()
    g.propagate(src.data_ptr(), width, dst.data_ptr())
    want = At @ x.astype(np.float64)
    scale = abs(At) @ np.abs(x.astype(np.float64)) + 1e-30
    assert np.max(np.abs(dst.cpu().numpy() - want) / scale) < 1e-6
