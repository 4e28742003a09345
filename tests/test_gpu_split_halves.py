"""The product by split halves (rows of A scaled to a common exponent, columns of B likewise, each element a pair of fp16 numbers)
at the edges of its tiles, column groups and K chunks, over the fp32 range, and on values no scale can hold."""
import pytest

from paper_2112_09335_b200 import binding, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def handle():
    wl = inputs.make_workload(0)
    g = binding.GcnAdmm(wl.n, wl.row_ptr, wl.col_idx, wl.X, wl.y, wl.train_mask, wl.widths, wl.n_comm, wl.community, wl.w_init)
    yield g
    g.destroy()


def product(g, a, b, tensor_cores=1):
    import torch
    c = torch.full((a.shape[0], b.shape[1]), float("nan"), device="cuda")
    torch.cuda.synchronize()
    g.dense_product(a.data_ptr(), b.data_ptr(), c.data_ptr(), a.shape[0], b.shape[1], a.shape[1], tensor_cores)
    return c


def bound(k):
    """Relative to sum |a||b|: both operands to 2^-23, the dropped product of the low parts 2^-24, and an accumulator that is rounded
    toward zero (2^-23) at each of ceil(k / 16) matrix instructions and once at the end."""
    return (2.5 + -(-k // 16) + 1) * 2.0 ** -23


@pytest.mark.parametrize("m", [16384, 16385, 19071])                                   # whole tiles, one row more, a tile less one row
@pytest.mark.parametrize("n,k", [(1, 32), (16, 33), (17, 63), (33, 64), (49, 65), (65, 96), (97, 40), (129, 47), (193, 128), (257, 100), (8, 2048), (40, 8), (256, 11), (64, 31)])
def test_edges(handle, m, n, k):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(m + n + k)
    a = torch.randn(m, k, generator=gen, device="cuda")
    b = torch.randn(k, n, generator=gen, device="cuda")
    got = product(handle, a, b).double()
    want, size = a.double() @ b.double(), a.double().abs() @ b.double().abs()
    assert float(((got - want).abs() / size).max()) < bound(k)


def test_scales(handle):
    """Rows between 2^-60 and 2^60, columns between 2^-50 and 2^50, some of either zero: the error is relative to each element's own terms."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(5)
    m, n, k = 16500, 130, 100
    a = torch.randn(m, k, generator=gen, device="cuda") * torch.exp2(torch.randint(-60, 61, (m, 1), generator=gen, device="cuda").float())
    b = torch.randn(k, n, generator=gen, device="cuda") * torch.exp2(torch.randint(-50, 51, (1, n), generator=gen, device="cuda").float())
    a[::97] = 0
    b[:, ::13] = 0
    got = product(handle, a, b).double()
    want, size = a.double() @ b.double(), a.double().abs() @ b.double().abs()
    assert bool((got[size == 0] == 0).all())
    assert float(((got - want).abs() / size)[size > 0].max()) < bound(k)


@pytest.mark.parametrize("spread", [20, 28])
def test_elements_far_below_the_largest_of_their_row(handle, spread):
    """A row and a column whose largest elements meet zeros: the sum of what is left, `spread` bits below them, is as good as any other."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(spread)
    m, n, k = 16400, 48, 64
    a = torch.randn(m, k, generator=gen, device="cuda").clamp(-2, 2)
    b = torch.randn(k, n, generator=gen, device="cuda")
    a[:, 0], b[0] = 2.0 ** (spread + 1), 0.0
    got = product(handle, a, b).double()
    want, size = a.double() @ b.double(), a.double().abs() @ b.double().abs()
    # the elements of A that are smallest of all may be off by 2^-51 of the row's largest
    floor = 2.0 ** (spread + 1 - 51) * b.double().abs().sum(0)
    assert bool(((got - want).abs() <= bound(k) * size + floor).all())


@pytest.mark.parametrize("spread", [0, 20, 26, 27, 28, 30, 34, 60, 100])
def test_each_element_by_itself(handle, spread):
    """Every column of B picks one element of each row of A, `spread` bits below the row's largest: no sum hides how it is held.  By halves
    to 2^-23 down to 27 bits below, then, in rows that are formed again, by TF32 pairs to 2^-21; and half a unit (2^-24) for the sum of the pair."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(spread)
    m, n, k = 16400, 48, 64
    a = (1 + torch.rand(m, k, generator=gen, device="cuda")) * 2.0 ** -spread
    a[:, ::3] *= -1
    a[:, 0] = 1
    b = torch.zeros(k, n, device="cuda")
    b[torch.arange(1, n + 1), torch.arange(n)] = 1
    want = a[:, 1:n + 1].double()
    off = float(((product(handle, a, b).double() - want).abs() / want.abs()).max())
    assert off <= (2.0 ** -23 if spread <= 27 else 2.0 ** -21) + 2.0 ** -24


@pytest.mark.parametrize("n,k", [(8, 2048), (100, 767), (256, 256), (40, 32)])
def test_errors_of_random_signs_do_not_add_up(handle, n, k):
    """Root mean squares, against that of the result: after j of J matrix instructions a sum of random signs has grown to sqrt(j / J) of it,
    and each cuts off 2^-23 of what is there (2/3 J + 1 of them in all); the pairs' errors, 2.5 x 2^-23 a term, have random signs too."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(k)
    a = torch.randn(16384, k, generator=gen, device="cuda")
    b = torch.randn(k, n, generator=gen, device="cuda")
    want = a.double() @ b.double()
    off = float((product(handle, a, b).double() - want).norm() / want.norm())
    assert off < (2 / 3 * -(-k // 16) + 1 + 2.5 + 1) * 2.0 ** -23


def test_values_without_a_scale_stay_in_their_row(handle):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(7)
    m, n, k = 16384, 40, 64
    a = torch.randn(m, k, generator=gen, device="cuda")
    b = torch.randn(k, n, generator=gen, device="cuda")
    clean = product(handle, a, b)
    a[5, 3], a[700, 9] = float("inf"), float("nan")
    got = product(handle, a, b)
    assert not bool(torch.isfinite(got[5]).any()) and not bool(torch.isfinite(got[700]).any())
    keep = torch.ones(m, dtype=torch.bool, device="cuda")
    keep[5] = keep[700] = False
    assert torch.equal(got[keep], clean[keep])


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_a_weight_without_a_scale_stays_in_its_column(bad):
    """The columns of a layer's weights share one scale: that of the finite ones."""
    import numpy as np
    wl = inputs.make_workload(3, scale=0.05)
    assert wl.n >= 4096
    w = [np.array(x, dtype=np.float32) for x in wl.w_init]
    r = int(np.argmin(np.abs(w[-1][:, 2])))          # not the element the scale comes from
    logits = []
    for value in (w[-1][r, 2], bad):
        w[-1][r, 2] = value
        g = binding.GcnAdmm(wl.n, wl.row_ptr, wl.col_idx, wl.X, wl.y, wl.train_mask, wl.widths, wl.n_comm, wl.community, w, tensor_cores=2)
        try:
            logits.append(g.predict()[0])
        finally:
            g.destroy()
    clean, got = logits
    others = [c for c in range(clean.shape[1]) if c != 2]
    assert np.isfinite(clean).all() and not np.isfinite(got[:, 2]).any()
    assert np.array_equal(got[:, others], clean[:, others])


def test_partial_sums_far_above_their_gradient():
    """64 splits of 256 rows hold 1.1e37 each in the rows of half of the features, of one sign in one half of the nodes and of the other
    in the rest: their magnitudes add up to more than the largest float, what is left of the gradient is 7e30.  One W block, against fp32 FMA."""
    import numpy as np
    n, hidden, classes = 16384, 64, 8
    X = np.ones((n, 16), dtype=np.float32)
    X[:, :8] = 1e8
    X[n // 2:, :8] *= -1
    rng = np.random.default_rng(0)
    W1 = np.zeros((16, hidden), dtype=np.float32)
    W1[8:] = rng.uniform(0.5, 1.0, (8, hidden)) / 8
    W2 = rng.standard_normal((hidden, classes)).astype(np.float32)
    Z1 = np.broadcast_to(-4.3e26 * (1 + np.arange(hidden) / hidden), (n, hidden)).astype(np.float32)
    found = []
    for tensor_cores in (0, 1):
        g = binding.GcnAdmm(n, np.zeros(n + 1, np.int64), np.zeros(0, np.int32), X, np.zeros(n, np.int32), np.zeros(n, np.uint8), [16, hidden, classes],
                            2, np.arange(n, dtype=np.int32) // (n // 2), [W1, W2], nu=1.0, rho=1.0, tau0=2e34, tensor_cores=tensor_cores)
        try:
            g.set_state(binding.ST_Z, 1, Z1)
            g.step_block(binding.PHASE_W, 1)
            d = g.decisions()
            found.append((d["trial_w"][0, 0], d["q_w"][0, 0], g.get_state(binding.ST_W, 1), g.predict()[0]))
        finally:
            g.destroy()
    (trial, q, w, logits), (trial_tc, q_tc, w_tc, logits_tc) = found
    assert trial == 0 and np.abs(w - W1).max() > 1e-4                       # the block moves
    assert trial_tc == trial and abs(q_tc - q) < 1e-4 * abs(q)
    assert np.abs(w_tc - w).max() < 1e-6 and np.abs(logits_tc - logits).max() < 1e-5 * np.abs(logits).max()
