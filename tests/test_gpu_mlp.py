"""GPU damping network (BF16 tensor-core forward, backward and Adam through
the C ABI) against the FP64 reference network.

Tolerances come from the arithmetic: the GPU rounds weights and
activations to BF16 (unit roundoff 2^-8 = 3.9e-3) and accumulates in FP32,
so each layer carries a relative error of a few 2^-8.  Outputs lie in
(0, 0.9): |y_gpu - y_ref| <= 0.02 everywhere and <= 0.002 on average.
Gradient blocks, in relative norm: a model of the rounding (FP64 products of
BF16-rounded operands) differs from the exact gradient by up to 4% for W1
(its operands X and dz1 are both rounded and its sums cancel), 1.6% b1,
1.4% W2, 0.9% b2, 0.4% W3, 0.3% b3; the bounds below are about twice that.
A transposed or shifted weight, a dropped ReLU mask or a wrong sign moves
the results by far more.

Device buffers are kept referenced for as long as a kernel may read them:
a temporary tensor's memory returns to the caching allocator at once."""
import numpy as np
import pytest

from oracle import mlp
from paper_2003_03134_gb300 import build, gbp

pytestmark = pytest.mark.gpu

BLOCKS = [("W1", 0, 1024, 0.08), ("b1", 1024, 1088, 0.04), ("W2", 1088, 5184, 0.03), ("b2", 5184, 5248, 0.02),
          ("W3", 5248, 5312, 0.01), ("b3", 5312, 5313, 0.01)]


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    gbp.lib()
    return t


def _params(seed):
    """Reference initialisation with a stronger output layer, so that the
    predictions spread over (0, 0.9) and every layer's gradient matters."""
    p = mlp.unpack(mlp.init_params(seed))
    rng = np.random.default_rng(seed + 100)
    p["W3"] = rng.normal(0.0, 0.5, 64)
    p["b1"] = rng.normal(0.0, 0.1, 64)
    p["b2"] = rng.normal(0.0, 0.1, 64)
    return mlp.pack(p).astype(np.float32).astype(np.float64)


def _data(seed, n):
    rng = np.random.default_rng(seed)
    X = rng.normal(size=(n, 16)).astype(np.float32)
    t = rng.uniform(0.0, 0.9, n).astype(np.float32)
    return X, t


def _dev(torch, a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("n", [1, 31, 128, 1000, 4099])
def test_forward_matches_reference(torch, n):
    p = _params(0)
    X, _ = _data(n, n)
    net = gbp.DampingNet(p)
    Xd = _dev(torch, X)
    yd = torch.full((n,), -1.0, dtype=torch.float32, device="cuda")
    net.forward(Xd.data_ptr(), n, yd.data_ptr())
    torch.cuda.synchronize()
    y = yd.cpu().numpy().astype(np.float64)
    ref, _ = mlp.forward(p, X.astype(np.float64))
    err = np.abs(y - ref)
    assert err.max() <= 0.02, err.max()
    if n >= 100:   # the average is only meaningful over many rows
        assert err.mean() <= 0.002, err.mean()
    assert ((y > 0) & (y < 0.9)).all()
    net.close()


@pytest.mark.parametrize("n,seed", [(128, 1), (777, 2), (5000, 3)])
def test_gradient_matches_reference(torch, n, seed):
    p = _params(seed)
    X, t = _data(seed + 50, n)
    net = gbp.DampingNet(p)
    Xd, td = _dev(torch, X), _dev(torch, t)
    loss, g = net.gradient(Xd.data_ptr(), td.data_ptr(), n)
    rloss, rg = mlp.loss_and_grad(p, X.astype(np.float64), t.astype(np.float64))
    assert abs(loss - rloss) <= 0.01 * rloss
    for name, a, b, tol in BLOCKS:
        num = np.linalg.norm(g[a:b] - rg[a:b])
        den = np.linalg.norm(rg[a:b])
        assert num <= tol * den, (name, num, den)
    net.close()


def test_gradient_is_reproducible(torch):
    p = _params(4)
    X, t = _data(9, 3000)
    Xd, td = _dev(torch, X), _dev(torch, t)
    net = gbp.DampingNet(p)
    l1, g1 = net.gradient(Xd.data_ptr(), td.data_ptr(), 3000)
    l2, g2 = net.gradient(Xd.data_ptr(), td.data_ptr(), 3000)
    assert l1 == l2
    np.testing.assert_array_equal(g1, g2)
    net.close()


def test_first_adam_step_matches_reference(torch):
    """Adam's first step moves each parameter by lr * g / (|g| + eps), i.e.
    by +-lr wherever the gradient is clearly non-zero."""
    p = _params(5)
    X, t = _data(11, 2048)
    lr = 1e-3
    net = gbp.DampingNet(p)
    Xd, td = _dev(torch, X), _dev(torch, t)
    net.train_step(Xd.data_ptr(), td.data_ptr(), 2048, lr)
    p1 = net.params.astype(np.float64)
    _, rg = mlp.loss_and_grad(p, X.astype(np.float64), t.astype(np.float64))
    rp1, _, _ = mlp.adam_step(p, rg, np.zeros_like(p), np.zeros_like(p), 1, lr)
    d, rd = p1 - p, rp1 - p
    assert np.abs(d - rd).max() <= 2.0 * lr * (1 + 1e-3)
    clear = np.abs(rg) > 1e-3 * np.abs(rg).max()
    agree = np.abs(d[clear] - rd[clear]) <= 1e-2 * lr
    assert agree.mean() >= 0.95, agree.mean()
    net.close()


def test_training_fits_a_teacher_network(torch):
    """Regression onto a teacher network's outputs: the loss falls by more
    than 10x in 600 Adam steps on minibatches given by index."""
    teacher = _params(6)
    X, _ = _data(13, 16384)
    t, _ = mlp.forward(teacher, X.astype(np.float64))
    t = t.astype(np.float32)
    Xd, td = _dev(torch, X), _dev(torch, t)
    net = gbp.DampingNet(mlp.init_params(7))
    loss0, _ = net.gradient(Xd.data_ptr(), td.data_ptr(), 16384)
    gen = torch.Generator(device="cpu").manual_seed(0)
    for _ in range(600):
        idx = torch.randint(0, 16384, (512,), generator=gen, dtype=torch.int32).cuda()
        net.train_step(Xd.data_ptr(), td.data_ptr(), 512, 3e-3, idx_ptr=idx.data_ptr())
    loss1, _ = net.gradient(Xd.data_ptr(), td.data_ptr(), 16384)
    assert loss1 < loss0 / 10, (loss0, loss1)
    net.close()


def test_indexed_minibatch_equals_gathered_rows(torch):
    p = _params(8)
    X, t = _data(15, 1000)
    idx = np.random.default_rng(3).permutation(1000)[:300].astype(np.int32)
    a = gbp.DampingNet(p)
    b = gbp.DampingNet(p)
    Xd, td, idxd = _dev(torch, X), _dev(torch, t), _dev(torch, idx)
    Xg, tg = _dev(torch, X[idx]), _dev(torch, t[idx])
    la = a.train_step(Xd.data_ptr(), td.data_ptr(), 300, 1e-3, idx_ptr=idxd.data_ptr(), want_loss=True)
    lb = b.train_step(Xg.data_ptr(), tg.data_ptr(), 300, 1e-3, want_loss=True)
    assert la == lb
    np.testing.assert_array_equal(a.params, b.params)
    a.close()
    b.close()


def test_invalid_arguments(torch):
    p = mlp.init_params(0).astype(np.float32)
    bad = p.copy()
    bad[17] = np.nan
    with pytest.raises(gbp.GBPError):
        gbp.DampingNet(bad)
    net = gbp.DampingNet(p)
    X, t = _data(0, 4)
    Xd, td = _dev(torch, X), _dev(torch, t)
    with pytest.raises(gbp.GBPError):
        net.gradient(Xd.data_ptr(), td.data_ptr(), 0)
    with pytest.raises(gbp.GBPError):
        net.train_step(Xd.data_ptr(), td.data_ptr(), 4, 0.0)
    with pytest.raises(gbp.GBPError):
        net.set_params(bad)
    net.forward(Xd.data_ptr(), 0, td.data_ptr())   # empty batch is a no-op
    np.testing.assert_array_equal(net.params, p)
    net.close()


@pytest.mark.parametrize("n", [1, 15, 16, 17, 63, 65, 29184 - 1, 29184 + 17])
@pytest.mark.parametrize("offset", [0, 1])
def test_forward_rows_do_not_depend_on_their_place(torch, n, offset):
    """Row counts around the 16-row tile and around one tile per resident warp (152 SMs x 12 warps x 16 rows),
    rows aligned to 8 bytes or to a float only: each row's prediction is bitwise the one it gets in another
    place of another call, and rows past the end are not written."""
    p = _params(1)
    X, _ = _data(n, n)
    net = gbp.DampingNet(p)
    buf = torch.zeros(n * 16 + 1, dtype=torch.float32, device="cuda")
    buf[offset:offset + n * 16] = _dev(torch, X).reshape(-1)
    y = torch.full((n + 16,), -1.0, dtype=torch.float32, device="cuda")
    net.forward(buf[offset:].data_ptr(), n, y.data_ptr())
    perm = torch.randperm(n, generator=torch.Generator().manual_seed(n)).cuda()
    Xp = _dev(torch, X)[perm].contiguous()
    yp = torch.empty(n, dtype=torch.float32, device="cuda")
    net.forward(Xp.data_ptr(), n, yp.data_ptr())
    torch.cuda.synchronize()
    assert torch.equal(y[:n][perm], yp)
    assert bool((y[n:] == -1.0).all())
    ref, _ = mlp.forward(p, X.astype(np.float64))
    assert np.abs(y[:n].cpu().numpy() - ref).max() <= 0.02


# One wave of mlp_grad_kernel's warps takes 2048 x 32 rows; more go in groups of 128 a warp.
WAVE_ROWS = 2048 * 32


@pytest.mark.parametrize("n", [WAVE_ROWS, WAVE_ROWS + 1, WAVE_ROWS + 97])
def test_gradient_and_step_around_one_wave_of_rows(torch, n):
    """Both sides of the switch from a warp per 32 rows to a warp per 128, the last group one row, a group and a
    row: the gradient against the reference, twice the same bits; an Adam step moves every parameter by what its
    gradient says, and the packed weights are the new ones."""
    p = _params(9)
    X, t = _data(17, n)
    Xd, td = _dev(torch, X), _dev(torch, t)
    net = gbp.DampingNet(p)
    loss, g = net.gradient(Xd.data_ptr(), td.data_ptr(), n)
    loss2, g2 = net.gradient(Xd.data_ptr(), td.data_ptr(), n)
    assert loss == loss2
    np.testing.assert_array_equal(g, g2)
    rl, rg = mlp.loss_and_grad(p, X.astype(np.float64), t.astype(np.float64))
    assert abs(loss - rl) <= 0.01 * rl
    for name, a, b, tol in BLOCKS:
        assert np.linalg.norm(g[a:b] - rg[a:b]) <= tol * np.linalg.norm(rg[a:b]), name
    lr = 1e-3
    net.train_step(Xd.data_ptr(), td.data_ptr(), n, lr)
    w0, w1 = p.astype(np.float32).astype(np.float64), net.params.astype(np.float64)
    step = lr * g / (np.abs(g) + 1e-8)
    # powf may be 4 ulp (2.4e-7) off, which 1 - 0.999^1 = 1e-3 amplifies to 2.4e-4 in the second moment, half of it
    # in its root; the other roundings are below 1e-6; the new weight rounds once
    assert (np.abs(w1 - (w0 - step)) <= 1.5e-4 * lr + 2.0 ** -24 * np.abs(w1)).all()
    other = gbp.DampingNet(w1)
    y, yo = (torch.empty(1000, dtype=torch.float32, device="cuda") for _ in range(2))
    net.forward(Xd.data_ptr(), 1000, y.data_ptr())
    other.forward(Xd.data_ptr(), 1000, yo.data_ptr())
    torch.cuda.synchronize()
    assert torch.equal(y, yo)
    net.close()
    other.close()


def test_grouped_rows_add_up_as_single_ones_do(torch):
    """Rows whose output is saturated at their target have a gradient of exactly zero.  As many of them behind one
    wave of rows halve the batch's weights, and nothing else: the grouped gradient of all is, bit for bit, half the
    ungrouped one of the wave."""
    p = _params(10)
    X, t = _data(19, WAVE_ROWS)
    rng = np.random.default_rng(20)
    big = (200.0 * rng.normal(size=(4096, 16))).astype(np.float32)
    y, _ = mlp.forward(p, big.astype(np.float64))
    big = big[y == y.max()]   # 1 / (1 + exp(-z)) rounds to 1 in 64 bits: z > 36
    assert len(big) > 500 and abs(y.max() - 0.9) < 1e-15
    fill = big[np.arange(WAVE_ROWS) % len(big)]
    net = gbp.DampingNet(p)
    Xa, ta = _dev(torch, X), _dev(torch, t)
    Xb = _dev(torch, np.concatenate([X, fill]))
    tb = _dev(torch, np.concatenate([t, np.full(WAVE_ROWS, 0.9, np.float32)]))
    la, ga = net.gradient(Xa.data_ptr(), ta.data_ptr(), WAVE_ROWS)
    lb, gb = net.gradient(Xb.data_ptr(), tb.data_ptr(), 2 * WAVE_ROWS)
    assert lb == 0.5 * la
    np.testing.assert_array_equal(gb, np.float32(0.5) * ga)
    net.close()
