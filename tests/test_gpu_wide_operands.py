"""Products whose operands span more of the fp32 range than a pair of fp16 numbers under one scale holds: by themselves, at the edges of
tiles, column groups and K chunks, and where training and inference form them (features that nobody scaled, units near dead)."""
import numpy as np
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
    """Relative to sum |a||b|, by TF32 pairs: both operands to 2^-21, the dropped product of the low parts 2^-22, and an accumulator
    that is rounded toward zero (2^-23) at each of ceil(k / 8) matrix instructions and once at the end."""
    return (8 + 2 + -(-k // 8) + 1) * 2.0 ** -23


def worst(got, a, b):
    want, size = a.double() @ b.double(), a.double().abs() @ b.double().abs()
    return float(((got.double() - want).abs() / size).max())


@pytest.mark.parametrize("where", ["both", "rows of A", "B"])
@pytest.mark.parametrize("m,n,k", [(16384, 1, 32), (16385, 16, 33), (19071, 17, 8), (16511, 33, 64), (20001, 49, 65), (16384, 65, 96), (16500, 97, 40),
                                   (33001, 129, 47), (16385, 193, 128), (19000, 257, 100), (16384, 8, 2048), (40000, 256, 256)])
def test_range(handle, m, n, k, where):
    """Column j of A is larger by 2^s_j, row j of B smaller by as much, s_j between -60 and 60, so that every term counts; or one operand
    with the other level, where the largest terms alone do."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(m + n + k)
    a = torch.randn(m, k, generator=gen, device="cuda")
    b = torch.randn(k, n, generator=gen, device="cuda")
    s = torch.exp2(torch.randint(-60, 61, (k,), generator=gen, device="cuda").float())
    if where != "B":
        a = a * s
    if where != "rows of A":
        b = b / s[:, None]
    assert worst(product(handle, a, b), a, b) < bound(k)


@pytest.mark.parametrize("below", [26, 27, 28, 29, 30, 34, 50, 100])
@pytest.mark.parametrize("n,k", [(48, 64), (256, 40)])
def test_a_few_rows_leave_the_others_as_they_are(handle, n, k, below):
    """Rows whose largest element meets zeros, the rest 2^below under it; every other row has the bits it has without them."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(below)
    m = 16400
    a = torch.rand(m, k, generator=gen, device="cuda") + 0.5
    b = torch.randn(k, n, generator=gen, device="cuda")
    b[0] = 0
    clean = product(handle, a, b)
    rows = torch.tensor([0, 127, 128, 9000, m - 1], device="cuda")
    a[rows, 0] = 2.0 ** below
    got = product(handle, a, b)
    others = torch.ones(m, dtype=torch.bool, device="cuda")
    others[rows] = False
    assert torch.equal(got[others], clean[others])
    assert worst(got[rows], a[rows], b) < bound(k)


def test_an_infinite_row_beside_one_of_wide_range(handle):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(3)
    m, n, k = 16384, 40, 64
    a = torch.randn(m, k, generator=gen, device="cuda")
    b = torch.randn(k, n, generator=gen, device="cuda")
    a[6, 3], a[7, 0], b[0] = float("inf"), 2.0 ** 70, 0.0
    got = product(handle, a, b)
    assert not bool(torch.isfinite(got[6]).any())
    keep = torch.arange(m, device="cuda") != 6
    assert worst(got[keep], a[keep], b) < bound(k)


def test_more_row_tiles_per_block_than_marks(handle):
    """148 blocks of 2,048 row tiles each and two tiles more, with wide rows in the first, the last marked alone, and the tiles that share a mark."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(4)
    tiles, k, n = 148 * 2048 + 2, 8, 1
    m = tiles * 128 - 5
    a = torch.randn(m, k, generator=gen, device="cuda")
    b = torch.randn(k, n, generator=gen, device="cuda")
    b[0] = 0
    for tile in (0, 148 * 2046, 148 * 2047, 148 * 2048, 148 * 2048 + 1):
        a[tile * 128 + 17, 0] = 2.0 ** 60
    got = product(handle, a, b)
    for at in range(0, m, 1 << 22):
        assert worst(got[at:at + (1 << 22)], a[at:at + (1 << 22)], b) < bound(k)


# ---- where the trainer forms them: nodes without edges, so that every propagation is the identity -------------------

N, C0, C1, C2 = 16384, 32, 64, 64


def trainer(X, W1, W2, **params):
    return binding.GcnAdmm(N, np.zeros(N + 1, np.int64), np.zeros(0, np.int32), X, np.zeros(N, np.int32), np.zeros(N, np.uint8), [C0, C1, C2], 2,
                           np.arange(N, dtype=np.int32) // (N // 2), [W1, W2], **params)


def forward(X, W1, W2):
    """Logits in fp64 and the size that an error is held against: |relu(X W1)| with |X||W1| in the place of the sums, times |W2|."""
    X, W1, W2 = (np.asarray(v, dtype=np.float64) for v in (X, W1, W2))
    return np.maximum(X @ W1, 0) @ W2, np.abs(X) @ np.abs(W1) @ np.abs(W2)


def problem(seed=0):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((N, C0))
    W1 = rng.uniform(-1, 1, (C0, C1)) * np.sqrt(6.0 / (C0 + C1))
    W2 = rng.uniform(-1, 1, (C1, C2)) * np.sqrt(6.0 / (C1 + C2))
    return rng, X, W1, W2


def f32(*arrays):
    return [np.ascontiguousarray(a, dtype=np.float32) for a in arrays]


SPREADS = [30, 38, 50]
# two products, each within bound(64) < 2.3e-6 of its own sizes, and a ReLU between them that passes errors on as they are
FORWARD = 5e-6


@pytest.mark.parametrize("spread", SPREADS)
def test_predictions_from_features_nobody_scaled(spread):
    """A feature 2^spread larger than the others, with weights as much smaller."""
    _, X, W1, W2 = problem()
    X[:, 0] *= 2.0 ** spread
    W1[0] *= 2.0 ** -spread
    X, W1, W2 = f32(X, W1, W2)
    g = trainer(X, W1, W2)
    try:
        got = g.predict()[0].astype(np.float64)
    finally:
        g.destroy()
    want, size = forward(X, W1, W2)
    assert np.max(np.abs(got - want) / size) < FORWARD


@pytest.mark.parametrize("spread", SPREADS)
@pytest.mark.parametrize("loaded", [False, True])
def test_predictions_with_units_near_dead(spread, loaded):
    """Hidden units whose incoming weights are 2^-spread of the others' and whose outgoing ones 2^spread; at create and by set_state."""
    _, X, W1, W2 = problem(1)
    W1[:, ::7] *= 2.0 ** -spread
    W2[::7] *= 2.0 ** spread
    X, W1, W2 = f32(X, W1, W2)
    g = trainer(X, np.zeros_like(W1) if loaded else W1, np.zeros_like(W2) if loaded else W2)
    try:
        if loaded:
            g.set_state(binding.ST_W, 1, W1)
            g.set_state(binding.ST_W, 2, W2)
        got = g.predict()[0].astype(np.float64)
    finally:
        g.destroy()
    want, size = forward(X, W1, W2)
    assert np.max(np.abs(got - want) / size) < FORWARD


@pytest.mark.parametrize("at", [0, 255, 148 * 256 - 1, 148 * 256, 200 * 256 - 1])
def test_one_large_weight_anywhere(at):
    """The scale of a layer's weights comes from one element of 51,200 (148 blocks of 256 look at them), 2^30 above the others."""
    rng = np.random.default_rng(6)
    X, W1, W2 = rng.standard_normal((N, 200)), rng.uniform(-1, 1, (200, 256)), rng.uniform(-1, 1, (256, 16))
    W1.flat[at] = 2.0 ** 30
    X[:, at // 256] *= 2.0 ** -30
    X, W1, W2 = f32(X, W1, W2)
    g = binding.GcnAdmm(N, np.zeros(N + 1, np.int64), np.zeros(0, np.int32), X, np.zeros(N, np.int32), np.zeros(N, np.uint8), [200, 256, 16], 2,
                        np.arange(N, dtype=np.int32) // (N // 2), [W1, W2])
    try:
        got = g.predict()[0].astype(np.float64)
    finally:
        g.destroy()
    want, size = forward(X, W1, W2)
    assert np.max(np.abs(got - want) / size) < bound(200) + bound(256)


@pytest.mark.parametrize("spread", SPREADS)
def test_weight_step_with_units_near_dead(spread):
    """Gradient columns and weight columns 2^-spread of the others: the W_1 block moves H_1 by the product with the gradient and leaves images
    of the moved weights.  The logits of both, H_1 as it was moved and as it is formed anew, against fp64 with the moved weights."""
    rng, X, W1, W2 = problem(2)
    unit = np.where(np.arange(C1) % 7 == 0, 2.0 ** -spread, 1.0)
    Z1 = np.maximum(X @ (W1 + 0.5 * rng.uniform(-1, 1, W1.shape) * np.sqrt(6.0 / (C0 + C1))), 0) * unit
    X, W1, W2, Z1 = f32(X, W1 * unit, W2 / unit[:, None], Z1)
    g = trainer(X, W1, W2, nu=1.0, rho=1.0, tau0=4e4)
    try:
        g.set_state(binding.ST_Z, 1, Z1)
        g.step_block(binding.PHASE_W, 1)
        assert g.decisions()["trial_w"][0, 0] >= 0
        W = g.get_state(binding.ST_W, 1)
        moved = g.predict()[0].astype(np.float64)
        g.set_state(binding.ST_Z, 1, Z1)                       # H_1 has to be formed anew
        anew = g.predict()[0].astype(np.float64)
    finally:
        g.destroy()
    assert np.abs((W - W1) / unit).max(axis=0).min() > 1e-3       # every unit moves
    want, size = forward(X, W, W2)
    assert np.max(np.abs(anew - want) / size) < FORWARD
    assert np.max(np.abs(moved - want) / size) < FORWARD + bound(C0) + 2.0 ** -22   # the product with the gradient, and H - D / tau in fp32


@pytest.mark.parametrize("spread", SPREADS)
def test_hidden_gradient_with_weights_of_wide_range(spread):
    """Rows of W_2 2^-spread of the others: their columns of G = S W_2^T, seen in Z_1 that starts from zero there, against fp32 FMA."""
    rng, X, W1, W2 = problem(3)
    dead = np.arange(C1) % 7 == 0
    W2[dead] *= 2.0 ** -spread
    Z1 = np.maximum(X @ W1, 0)
    Z1[:, dead] = 0
    X, W1, W2, Z1 = f32(X, W1, W2, Z1)
    Z2 = rng.standard_normal((N, C2)).astype(np.float32)
    found = []
    for tensor_cores in (0, 1):
        g = trainer(X, W1, W2, nu=1e-30, rho=1.0, theta0=64.0, tensor_cores=tensor_cores)
        try:
            g.set_state(binding.ST_Z, 1, Z1)
            g.set_state(binding.ST_Z, 2, Z2)
            g.step_block(binding.PHASE_Z, 1)
            found.append((g.decisions()["trial_z"][0, 0], g.get_state(binding.ST_Z, 1).astype(np.float64)))
        finally:
            g.destroy()
    (trial, z), (trial_tc, z_tc) = found
    assert (trial >= 0).all() and (trial_tc == trial).all()
    moved, error = z[:, dead] - Z1[:, dead], z_tc[:, dead] - z[:, dead]
    # sums of 64 products; in S both sides form H_2 - Z_2, from sums of 64 products as well: ten times the bound of one of them
    assert np.abs(moved).max() > 0 and np.linalg.norm(error) < 10 * bound(C2) * np.linalg.norm(moved)


def test_a_weight_step_leaves_no_mark_of_the_weights_before_it():
    """Weights of wide range are loaded and moved to where they are not; logits from the images the move left have the bits of those from
    images of the same weights loaded anew."""
    rng, X, W1, W2 = problem(4)
    moved = W1 + 0.5 * rng.uniform(-1, 1, W1.shape) * np.sqrt(6.0 / (C0 + C1))
    W1[:, ::7] *= 2.0 ** -40
    Z1 = np.maximum(X @ moved, 0)
    X, W1, W2, Z1 = f32(X, W1, W2, Z1)
    g = trainer(X, W1, W2, nu=1.0, rho=1.0, tau0=4e4)
    try:
        g.set_state(binding.ST_Z, 1, Z1)
        g.step_block(binding.PHASE_W, 1)
        assert g.decisions()["trial_w"][0, 0] >= 0
        W = g.get_state(binding.ST_W, 1)
        assert np.abs(W).min() > 2.0 ** -18 * np.abs(W).max()          # no element small under either scale
        g.set_state(binding.ST_Z, 1, Z1)                               # H_1 has to be formed anew
        after_step = g.predict()[0]
        g.set_state(binding.ST_W, 1, W)
        after_load = g.predict()[0]
    finally:
        g.destroy()
    assert np.array_equal(after_step, after_load)


@pytest.mark.parametrize("n", [600, 5000, 20000])
def test_a_gradient_beside_a_far_larger_one(n):
    """Layer widths that are no multiples of four: what a W block decides does not depend on the gradient, 2^40 times as large, that another
    layer's block has formed before it."""
    rng = np.random.default_rng(5)
    widths = [9, 21, 16, 3]
    X = rng.standard_normal((n, 9)).astype(np.float32)
    W = f32(*(rng.uniform(-1, 1, (a, b)) for a, b in zip(widths, widths[1:])))
    Z1 = np.maximum(X @ W[0], 0) + 0.1 * rng.standard_normal((n, 21))
    Z2 = 2.0 ** 40 * rng.standard_normal((n, 16))
    found = []
    for first in (None, 2):
        g = binding.GcnAdmm(n, np.zeros(n + 1, np.int64), np.zeros(0, np.int32), X, np.zeros(n, np.int32), np.zeros(n, np.uint8), widths, 2,
                            np.arange(n, dtype=np.int32) // ((n + 1) // 2), W, tensor_cores=2)
        try:
            g.set_state(binding.ST_Z, 1, Z1.astype(np.float32))
            g.set_state(binding.ST_Z, 2, Z2.astype(np.float32))
            if first is not None:
                g.step_block(binding.PHASE_W, first)
            g.step_block(binding.PHASE_W, 1)
            d = g.decisions()
            found.append((d["trial_w"][0, 0], d["q_w"][0, 0], g.get_state(binding.ST_W, 1)))
        finally:
            g.destroy()
    (trial, q, w), (trial_after, q_after, w_after) = found
    assert trial >= 0 and trial_after == trial and q_after == q and np.array_equal(w_after, w)
