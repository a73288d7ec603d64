"""The steps of handles that do not fill the GPU (a block per case in shared
memory; one overlapped launch a step) against a forced step-kernel variant, at
the edges of their sizes: 64, 65, 128, 129, 320 and 321 fluid cells, and around
the size from which the tiled step takes over."""
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


def _box(dim, fluid, periodic=False):
    """A box with exactly `fluid` fluid cells, inlet and outlet planes fluid."""
    nz, ny = (5, 4) if dim == 3 else (1, 7)
    nx = fluid // (ny * nz) + 3
    c = cases.open_channel(nx, ny, nz, current_A_cm2=1.0)
    inner = [(z, y, x) for x in range(1, nx - 1) for y in range(ny) for z in range(nz)]
    rng = np.random.default_rng(fluid)
    for k in rng.permutation(len(inner))[:c.solid.size - fluid]:
        c.solid[inner[k]] = True
    assert c.n_fluid == fluid and c.dim == dim
    return c.with_(periodic_x=periodic)


def _same(L, cs, precision, tol, steps):
    out = []
    for variant in (0, 1):
        b = L.Batch.from_cases(cs, precision=precision, step_variant=variant)
        for k, c in enumerate(cs):
            b.set_bc(c.x_in, 0.0 if c.periodic_x else c.current_A_cm2, case=k)
            rng = np.random.default_rng(k)
            X = np.empty((3,) + c.shape)
            X[0] = 0.45 + 0.1 * rng.random(c.shape)
            X[1] = 0.12 + 0.05 * rng.random(c.shape)
            X[2] = 1.0 - X[0] - X[1]
            b.set_fields(k, X)
        for n in steps:
            b.step(n)
        assert b.info().steps == sum(steps)
        out.append(([b.fields(k, u=True, tau=True) for k in range(len(cs))], b.residuals(sum(steps))))
        b.close()
    for a, r in zip(out[0][0], out[1][0]):
        assert np.abs(a[0] - r[0]).max() <= tol
        assert np.abs(a[2] - r[2]).max() <= 1e3 * tol
    assert np.allclose(out[0][1], out[1][1], rtol=1e-3 if precision == "fp16" else 1e-5)


# the bounds of test_gpu_step_tile.py; FP64 divides once for five quotients
# (a few ulp, 1e-15, a step)
PRECISIONS = [("fp64", 1e-12), ("fp32", 1e-7), ("fp16", 5e-6)]


@pytest.mark.parametrize("precision,tol", PRECISIONS)
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("fluid", [64, 65, 128, 129, 320, 321])
def test_sizes(L, precision, tol, dim, fluid):
    _same(L, [_box(dim, fluid)], precision, tol, (33, 1, 2))


@pytest.mark.parametrize("precision,tol", PRECISIONS)
def test_batches_and_periodic_boxes(L, precision, tol):
    _same(L, [_box(2, 61), _box(2, 300), _box(2, 100, periodic=True)], precision, tol, (40,))
    _same(L, [_box(3, 61), _box(3, 900), _box(3, 500, periodic=True)], precision, tol, (40, 1))
    _same(L, [_box(2, 700), _box(2, 330)], precision, tol, (1, 35))


@pytest.mark.parametrize("precision,tol", PRECISIONS)
@pytest.mark.parametrize("fluid", [38848, 38849])     # 38,848 and 38,912 cells of storage: small; 38,913 on: tiled
def test_around_the_tiled_step(L, precision, tol, fluid):
    _same(L, [_box(2, fluid)], precision, tol, (35,))
    _same(L, [_box(2, fluid + 64)], precision, tol, (35,))
