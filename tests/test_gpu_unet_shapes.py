"""The U-Net's tensor-core kernels at the edges of their tiles: widths whose
channels fill their storage or leave odd offsets in the concatenations, row
counts that leave partial tiles and several chunks of the weight gradients,
and buffers shared by batches of different grids.

Sparse weights of +-1, inputs of 0 and 1 and output errors of -1, 0 and 1
keep every activation a small integer and every gradient a small integer
times one BF16 number, so every rounding of the device is exact and the
comparison with PyTorch (FP32, CPU) needs no tolerance for the order of the
sums: 1e-6, the rounding of the reference's own scale factors."""
import numpy as np
import pytest

from test_gpu_unet import F, _GradBF16

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_01600_gb300 import lbms
    lbms.load()
    return lbms


def _sparse_params(shapes, seed):
    """A +-1 entry per output channel (at a random tap), the input channels
    taken in turn so that none feeds many outputs; biases 0 or 1."""
    rng = np.random.default_rng(seed)
    out = []
    for sh in shapes:
        a = np.zeros(sh, dtype=np.float32)
        if len(sh) == 1:
            a[:] = rng.integers(0, 2, sh)
        elif sh[2] == 2:         # transposed [ci][co][2][2][2]: one input channel per output and child
            ci = rng.permutation(sh[0])
            for co in range(sh[1]):
                for t in range(8):
                    a[ci[(co + t) % sh[0]], co, t >> 2, (t >> 1) & 1, t & 1] = rng.choice([-1.0, 1.0, 1.0, 1.0])
        else:
            ci = rng.permutation(sh[1])
            for co in range(sh[0]):
                a[(co, ci[co % sh[1]]) + tuple(rng.integers(0, sh[2], 3))] = rng.choice([-1.0, 1.0, 1.0, 1.0])
        out.append(a)
    return out


def _inputs(B, Z, Y, X, seed):
    rng = np.random.default_rng(seed)
    m = (rng.random((B, 1, Z, Y, X)) < 0.6).astype(np.float32)
    return np.concatenate([rng.integers(0, 2, (B, 16, Z, Y, X)).astype(np.float32) * m, m], axis=1)


def _reference(params, x, seed):
    """Targets, output, loss and gradients; asserts that BF16 holds every value."""
    p = [torch.tensor(a, requires_grad=True) for a in params]
    W, b = p[0::2], p[1::2]
    kept = []

    def keep(h):
        assert torch.equal(h.detach().bfloat16().float(), h.detach())
        h.retain_grad()
        kept.append(h)
        return h

    def conv(h, i):
        return keep(F.relu(F.conv3d(h, W[i], b[i], padding=1)))

    e1 = conv(conv(torch.tensor(x), 0), 1)
    e2 = conv(conv(F.max_pool3d(e1, 2), 2), 3)
    e3 = conv(conv(F.max_pool3d(e2, 2), 4), 5)
    d2 = conv(conv(torch.cat([keep(F.conv_transpose3d(e3, W[6], b[6], stride=2)), e2], 1), 7), 8)
    d1 = conv(conv(torch.cat([keep(F.conv_transpose3d(d2, W[9], b[9], stride=2)), e1], 1), 10), 11)
    # the head's bias gradient sums the output gradient before its BF16 rounding
    y = _GradBF16.apply(F.conv3d(d1, W[12])) + b[12].reshape(1, 3, 1, 1, 1)
    m = torch.tensor(x[:, 16:17])
    t = y.detach() - torch.tensor(np.random.default_rng(seed).integers(-1, 2, y.shape).astype(np.float32))
    loss = (((y - t) * m) ** 2).sum() / (3.0 * m.sum())
    loss.backward()
    for h in kept:   # exact in BF16 where the ReLU lets it through
        g = h.grad * (h.detach() != 0)
        assert torch.equal(g.bfloat16().float(), g)
    return t.numpy(), y.detach().numpy(), float(loss.detach()), [q.grad.numpy() for q in p]


def _check(net, params, x, seed):
    t, y, lref, grads = _reference(params, x, seed)
    assert np.array_equal(net.forward(x), y)
    assert net.train_batch(x, t, lr=0.0) == pytest.approx(lref, rel=1e-6)
    for i, (g, r) in enumerate(zip(net.get(1), grads)):
        assert np.abs(g - r).max() <= 1e-6 * np.abs(r).max(), i




@pytest.mark.parametrize("width", [5, 14, 31, 32])
def test_widths(L, width):
    net = L.UNet(width=width, max_voxels=2 * 12 * 16 * 20, seed=1)
    params = _sparse_params(net.shapes(), 100 + width)
    net.set(params)
    _check(net, params, _inputs(2, 12, 16, 20, 200 + width), width)
    net.close()


def test_several_chunks_and_changing_grids(L):
    """26 x 26 x 40 rows: two chunks of rows at full resolution; then a smaller
    grid in the same buffers, then the first again."""
    net = L.UNet(width=28, max_voxels=24 * 24 * 36, seed=2)
    params = _sparse_params(net.shapes(), 7)
    net.set(params)
    for k, (Z, Y, X) in enumerate([(24, 24, 36), (8, 12, 16), (24, 24, 36)]):
        _check(net, params, _inputs(1, Z, Y, X, 300 + k), k)
    net.close()


@pytest.mark.parametrize("copies", [4, 32])
def test_copies_of_a_volume(L, copies):
    """The gradients of a batch of equal volumes are those of the volume: the
    scale divides by a power of two, the sums are exact.  One volume has 8
    chunks of rows at full resolution; 4 copies have 32 (three windows a CTA of
    the weight gradients instead of one), 32 copies also at half resolution."""
    Z, Y, X = 40, 40, 64
    net = L.UNet(width=28, max_voxels=copies * Z * Y * X, seed=4)
    params = _sparse_params(net.shapes(), 17)
    net.set(params)
    x = _inputs(1, Z, Y, X, 400)
    y = net.forward(x)
    rng = np.random.default_rng(5)
    d = np.zeros(y.shape, dtype=np.float32)
    d.reshape(-1)[rng.choice(d.size, 64, replace=False)] = rng.choice([-1.0, 1.0], 64)
    loss = net.train_batch(x, y - d, lr=0.0)
    one = net.get(1)
    many_loss = net.train_batch(np.repeat(x, copies, 0), np.repeat(y - d, copies, 0), lr=0.0)
    assert many_loss == pytest.approx(loss, rel=1e-12)
    for i, (g, r) in enumerate(zip(net.get(1), one)):
        assert np.abs(r).max() > 0
        # the head's bias gradient sums FP32 values before their rounding to BF16
        assert np.allclose(g, r, rtol=1e-6, atol=0) if i == 25 else np.array_equal(g, r), i
    net.close()
