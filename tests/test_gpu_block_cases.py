"""The step of one block per case on batches of many small cases, where FP64
takes it, and of 3-D cases of more than 128 cells, against a forced variant."""
import pytest

from test_gpu_step_small import PRECISIONS, _box, _same

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_01600_gb300 import lbms
    lbms.load()
    return lbms


@pytest.mark.parametrize("precision,tol", PRECISIONS)
@pytest.mark.parametrize("dim,fluid,count", [(2, 61, 80), (3, 64, 160), (2, 120, 120), (3, 128, 152), (3, 300, 60)])
def test_many_cases(L, precision, tol, dim, fluid, count):
    boxes = [_box(dim, fluid), _box(dim, fluid - 9)]
    _same(L, [boxes[k % 2] for k in range(count)], precision, tol, (33, 2))
