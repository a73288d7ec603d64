"""A product of the pointwise network whose wait ran out: the prediction made
from it is an error, and the handle keeps its state."""
import numpy as np
import pytest

from workloads import cases

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_01600_gb300 import lbms
    lbms.load()
    return lbms


def test_warm_start_after_a_wait_that_ran_out(L):
    c = cases.porous((12, 14, 30), radius=2, porosity=0.5, seed=9, current_A_cm2=1.0)
    s = L.Solver.from_case(c)
    s.set_bc(c.x_in, c.current_A_cm2)
    s.step(30)
    before = s.fields()
    net = L.Net(width=64, depth=1, seed=1)
    assert L.load().lbms_internal_net_timeout(net._h) == 0
    with pytest.raises(L.LbmsError) as e:
        net.warm_start(s)
    assert e.value.status == L.LBMS_ECUDA and "timed out" in str(e.value)
    assert np.array_equal(s.fields(), before) and s.info().steps == 30
    X = net.warm_start(s)                # reported once
    assert np.abs(s.fields() - X).max() <= 2.0 ** -48 and s.info().steps == 0   # a double-float pair
    net.close()
    s.close()
