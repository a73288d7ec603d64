"""The FP64 coupling of the small handles' steps (one reciprocal for all
quotients) against the general one, on states whose mixture denominators,
determinants and reacting denominators change sign: the clamps of tau must
fall on the same side."""
import numpy as np
import pytest

from test_gpu_step_small import _box

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1809_01600_gb300 import lbms
    lbms.load()
    return lbms


def _field(c, kind):
    rng = np.random.default_rng(11)
    X = np.empty((3,) + c.shape)
    X[0] = 0.5 + 0.1 * rng.random(c.shape)
    X[1] = 0.1 + 0.1 * rng.random(c.shape)
    at = rng.random(c.shape) < 0.3
    if kind == "mixture":          # the inert species' denominator, both signs of its numerator
        X[0][at] = 0.1 * rng.random(at.sum()) - 0.05
        X[1][at] = 0.1 * rng.random(at.sum()) - 0.05
    elif kind == "reacting":       # sums that the reacting species divide by
        X[0][at] = -1.5 * rng.random(at.sum())
    X[2] = 1.0 - X[0] - X[1]
    if kind == "empty":            # no gas at all in some cells
        X[:, at] = 0.0
    return X


# Each step rounds differently by a few ulp of O(1) values (1e-15); four steps,
# velocities bounded by 0.1
@pytest.mark.parametrize("coupling", ["ms", "tau_only"])
@pytest.mark.parametrize("kind", ["mixture", "reacting", "empty"])
@pytest.mark.parametrize("dim,fluid", [(2, 60), (2, 300), (2, 900), (3, 120), (3, 300), (3, 900)])
def test_signs_of_the_denominators(L, dim, fluid, kind, coupling):
    c = _box(dim, fluid)
    out = []
    for variant in (0, 1):
        s = L.Solver.from_case(c, precision="fp64", coupling=coupling, step_variant=variant)
        s.set_bc(c.x_in, c.current_A_cm2)
        s.set_fields(_field(c, kind))
        got = []
        for _ in range(4):
            s.step(1)
            got.append(s.fields())
        out.append(got)
        s.close()
    for a, r in zip(*out):
        assert np.isfinite(r).all()
        assert np.abs(a - r).max() <= 1e-12 * max(1.0, np.abs(r).max())
