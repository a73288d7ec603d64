"""The default time step of anodes that fill the GPU (one thread per cell,
tiled populations, packed arithmetic, overlapped launches) against a forced
step-kernel variant with rows of populations, and against the oracle."""
import numpy as np
import pytest

from oracle import Oracle
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


def _cases(kind):
    if kind == "3d":           # odd extents, rows over one 16-voxel window, a last tile that is not full
        return [cases.porous((41, 53, 67), radius=2, porosity=0.5, seed=301, current_A_cm2=1.5)]
    if kind == "2d":
        return [cases.porous((301, 403), radius=3, porosity=0.6, seed=302, current_A_cm2=1.0)]
    if kind == "batch":        # uneven cases, padding cells between them, a strip one voxel high
        return [cases.porous((37, 40, 48), radius=2, porosity=0.5, seed=303, current_A_cm2=1.5),
                cases.porous((3, 5, 17), radius=1, porosity=0.7, seed=304, current_A_cm2=0.5),
                cases.porous((29, 31, 50), radius=2, porosity=0.55, seed=305, current_A_cm2=1.0)]
    # periodic in x: the sources come from the 32-bit table
    return [cases.open_channel(40, 38, 36).with_(periodic_x=True)]


def _start(c, seed):
    rng = np.random.default_rng(seed)
    X = np.empty((3,) + c.shape)
    X[0] = 0.45 + 0.1 * rng.random(c.shape)
    X[1] = 0.12 + 0.05 * rng.random(c.shape)
    X[2] = 1.0 - X[0] - X[1]
    return X


# FP64: FMA contraction only.  FP32: one FP32 rounding (6e-8) of a population
# of size w |dX| <= 1e-2 a link and step, 40 steps.  FP16 storage: a flipped
# half-precision rounding, 2^-11 of the same.
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-13), ("fp32", 1e-7), ("fp16", 5e-6)])
@pytest.mark.parametrize("kind", ["3d", "2d", "batch", "periodic"])
def test_default_step_equals_a_forced_variant(L, kind, precision, tol):
    cs = _cases(kind)
    out = []
    for variant in (0, 1):
        b = L.Batch.from_cases(cs, precision=precision, step_variant=variant)
        for k, c in enumerate(cs):
            b.set_bc(c.x_in, 0.0 if c.periodic_x else c.current_A_cm2, case=k)
            b.set_fields(k, _start(c, k))
        i = b.info()
        assert i.threads_per_cell == (1 if variant == 0 else 3)
        assert i.neighbour_bits == (32 if variant == 1 or kind == "periodic" else 1)
        b.step(39)                                   # a graph of 32 and single steps
        b.step(1)
        out.append(([b.fields(k, u=True, tau=True) for k in range(len(cs))], b.residuals(40),
                    None if kind == "periodic" else b.overpotentials()[0]))
        b.close()
    for a, r in zip(out[0][0], out[1][0]):
        assert np.abs(a[0] - r[0]).max() <= tol
        assert np.abs(a[2] - r[2]).max() <= 1e3 * tol
    assert np.allclose(out[0][1], out[1][1], rtol=1e-3 if precision == "fp16" else 1e-5)
    if kind != "periodic":
        assert np.allclose(out[0][2], out[1][2], rtol=1e3 * tol)


def test_default_step_against_the_oracle_with_flux_balance(L):
    c = cases.porous((41, 53, 67), radius=2, porosity=0.5, seed=301, current_A_cm2=1.5)
    s = L.Solver.from_case(c, precision="fp64")
    s.set_bc(c.x_in, c.current_A_cm2)
    assert s.info().threads_per_cell == 1 and s.info().neighbour_bits == 1
    o = Oracle(c)
    s.step(35)
    o.step(35)
    f = ~c.solid
    assert np.abs(s.fields() - o.X)[:, f].max() <= 1e-11
    flux, totals = s.boundary_flux()
    assert np.allclose(flux, o.plane_flux()[:, 0], rtol=1e-8, atol=1e-12)
    assert np.allclose(totals, o.total(), rtol=1e-11)
    s.close()
