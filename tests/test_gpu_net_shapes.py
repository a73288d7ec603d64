"""The pointwise network's tensor-core kernels at the edges of their tiles:
row counts that leave half a 128-row tile and split the weight gradients in
one to sixteen chunks, widths of one, several and half-filled column tiles.

Every input of a layer feeds one of its units, with weight +-1, inputs and
output errors are small integers: activations are integers below 256 and
gradients integers below 2^16 times the BF16 value of the loss gradient's
scale, so that every rounding and every order of the sums is exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_01600_gb300 import lbms
    lbms.load()
    return lbms


@pytest.mark.parametrize("width,depth,rows", [(64, 1, 64), (64, 2, 192), (128, 1, 320), (192, 3, 1088), (704, 3, 8256),
                                              (128, 2, 32768), (2048, 1, 128)])
def test_exact_integers(L, width, depth, rows):
    rng = np.random.default_rng(width + rows)
    net = L.Net(width=width, depth=depth, seed=1)
    net.set_gemm("tcgen05")
    dims = [L.Net.FEATURES] + [width] * depth + [3]
    layers = []
    for i, o in zip(dims[:-1], dims[1:]):
        W = np.zeros((o, i))
        W[rng.integers(0, o, i), np.arange(i)] = rng.choice([-1.0, 1.0, 1.0], i)
        layers.append((W, rng.integers(0, 2, o).astype(np.float64)))
    net.set(layers)
    x = rng.integers(0, 2, (rows, L.Net.FEATURES)).astype(np.float64)

    act = [x]
    for W, b in layers[:-1]:
        act.append(np.maximum(act[-1] @ W.T + b, 0.0))
        assert act[-1].max() < 256
    y = act[-1] @ layers[-1][0].T + layers[-1][1]
    d = rng.choice([-1.0, 1.0], (rows, 3)) * (rng.random((rows, 3)) < min(0.5, 400.0 / rows))
    scale = np.float32(2.0) / np.float32(3 * rows)
    unit = float(torch.tensor(scale).to(torch.bfloat16).double())

    bits = L.to_bf16_bits(x.astype(np.float32))
    assert np.array_equal(net.forward(bits), y)
    loss = net.train_batch(bits, (y - d).astype(np.float32))
    assert loss == pytest.approx((d * d).sum() / (3 * rows), rel=1e-12)
    got = net.get(1)
    D = d
    for l in range(depth, -1, -1):
        gW, gb = got[l]
        assert (np.abs(D).T @ act[l]).max() < 2 ** 16
        assert np.array_equal(gW, unit * (D.T @ act[l]))
        if l == depth:      # summed before their rounding to BF16: FP32 sums of `rows` terms
            assert np.all(np.abs(gb - float(scale) * D.sum(0)) <= rows * 2.0 ** -24 * float(scale) * np.abs(D).sum(0))
        else:
            assert np.array_equal(gb, unit * D.sum(0))
        D = (D @ layers[l][0]) * (act[l] > 0)
