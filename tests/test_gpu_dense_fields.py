"""Conversions between the caller's dense grid and the device: the feature
windows at extents below the largest window (periodic wraps more than once)
and reading and restarting fields on both sides of the size from which the
device converts them."""
import numpy as np
import pytest

from test_gpu_net import _reference_features
from workloads import cases

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_01600_gb300 import lbms
    lbms.load()
    return lbms


@pytest.mark.parametrize("shape", [(3, 5, 20), (7, 6, 17), (8, 1, 24), (1, 4, 33)])
def test_feature_windows_on_small_extents(L, shape):
    case = cases.open_channel(shape[2], shape[1], shape[0], current_A_cm2=0.8)
    case.solid[:, :, 5:9] = np.random.default_rng(3).random(case.solid[:, :, 5:9].shape) < 0.4
    s = L.Solver.from_case(case)
    s.set_bc(case.x_in, case.current_A_cm2)
    net = L.Net(width=64, depth=1, seed=1)
    got = net.features(s, case.n_fluid)
    ref = _reference_features(case)
    # one BF16 rounding (2^-8) of an FP32 value
    assert np.all(np.abs(got[:, :16] - ref[:, :16]) <= 2.0 ** -8 * np.abs(ref[:, :16]) + 1e-6)
    net.close()
    s.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("shape", [(16, 31, 33), (16, 32, 32), (25, 27, 41)])   # 16,368, 16,384 and 27,675 cells
def test_fields_round_trip(L, precision, shape):
    c = cases.porous(shape, radius=2, porosity=0.5, seed=5, current_A_cm2=1.0)
    s = L.Solver.from_case(c, precision=precision)
    s.set_bc(c.x_in, c.current_A_cm2)
    X = np.random.default_rng(6).random((3,) + c.shape)
    s.set_fields(X)
    got = s.fields()
    f = ~c.solid
    # exact in FP64; a double-float pair keeps 48 bits
    assert np.all(np.abs(got - X)[:, f] <= (0.0 if precision == "fp64" else 2.0 ** -48))
    assert np.all(got[:, c.solid] == 0.0)
    s.close()
