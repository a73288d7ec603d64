"""lbms_get_info names the step that a handle takes: cells per block, blocks
per SM, neighbour lookup and threads per cell, on both sides of the sizes
between which the step changes."""
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


def _info(L, cs, precision, **kw):
    b = L.Batch.from_cases(cs, precision=precision, **kw)
    for k, c in enumerate(cs):                 # a forced variant takes effect with the boundary data
        b.set_bc(c.x_in, 0.0 if c.periodic_x else c.current_A_cm2, case=k)
    i = b.info()
    b.close()
    return i.tile_cells, i.tile_min_blocks, i.neighbour_bits, i.threads_per_cell


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("fluid,want", [(64, (64, 1, 32, 3)), (65, (128, 1, 32, 3)), (128, (128, 1, 32, 3)),
                                        (129, (320, 1, 32, 3)), (320, (320, 1, 32, 3)), (321, (32, 4, 1, 3))])
def test_small_handles(L, precision, fluid, want):
    assert _info(L, [_box(2, fluid)], precision) == want


def test_periodic_boxes_read_the_table(L):
    assert _info(L, [_box(2, 700, periodic=True)], "fp32") == (32, 4, 32, 3)
    assert _info(L, [_box(2, 700), _box(2, 700, periodic=True)], "fp32") == (32, 4, 32, 3)


@pytest.mark.parametrize("precision,blocks", [("fp32", 10), ("fp16", 10)])
def test_around_the_tiled_step(L, precision, blocks):
    assert _info(L, [_box(3, 38912)], precision) == (32, 4, 1, 3)
    assert _info(L, [_box(3, 38913)], precision) == (64, blocks, 1, 1)


def test_forced_variants(L):
    assert _info(L, [_box(2, 64)], "fp32", step_variant=1) == (32, 8, 32, 3)
    assert _info(L, [_box(2, 64)], "fp32", step_variant=9) == (64, 8, 1, 1)


# a block per case while it gives no SM more FP64 warps than the launches do,
# and in 3-D FP32 / FP16 from 128 cells on only with enough cases
@pytest.mark.parametrize("dim,precision,fluid,cases_,want", [
    (2, "fp64", 64, 1, 32), (2, "fp64", 64, 76, 32), (2, "fp64", 64, 77, 64), (3, "fp64", 60, 152, 64),
    (3, "fp64", 60, 153, 32), (2, "fp64", 60, 229, 64), (2, "fp64", 60, 320, 32), (2, "fp64", 128, 114, 32),
    (2, "fp64", 128, 115, 128), (3, "fp64", 120, 153, 32), (2, "fp64", 300, 1, 32), (3, "fp64", 300, 100, 32),
    (3, "fp32", 128, 1, 128), (3, "fp32", 129, 1, 32), (3, "fp32", 300, 56, 32), (3, "fp32", 300, 57, 320),
    (3, "fp16", 300, 56, 32), (3, "fp16", 300, 57, 320), (2, "fp32", 300, 1, 320), (2, "fp16", 320, 300, 320)])
def test_a_block_per_case_where_it_pays(L, dim, precision, fluid, cases_, want):
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the counts are for 152 SMs")
    assert _info(L, [_box(dim, fluid)] * cases_, precision)[0] == want


def _channel(nx, ny, nz, fluid):
    """A channel with `fluid` fluid cells, end planes fluid."""
    import numpy as np
    from workloads import cases
    c = cases.open_channel(nx, ny, nz, current_A_cm2=1.0)
    inner = c.solid[:, :, 1:-1]
    drop = np.random.default_rng(fluid).permutation(inner.size)[:c.solid.size - fluid]
    z, y, x = np.unravel_index(drop, inner.shape)
    inner[z, y, x] = True
    assert c.n_fluid == fluid
    return c


# cells per block, threads per cell: launches of 32 cells (three threads each),
# tiles of 64, or halves of them where a second wave of tiles would be short
FP64 = [((300, 220, 1), 58368, (32, 3)), ((300, 220, 1), 58369, (64, 1)), ((400, 220, 1), 77824, (64, 1)),
        ((400, 220, 1), 77825, (32, 3)), ((400, 220, 1), 87552, (32, 3)), ((400, 220, 1), 87553, (64, 1)),
        ((60, 40, 32), 53504, (32, 3)), ((60, 40, 32), 53505, (64, 1)), ((60, 40, 32), 58368, (64, 1)),
        ((60, 40, 32), 58369, (32, 1)), ((60, 40, 32), 72960, (32, 1)), ((60, 40, 32), 72961, (64, 1))]


@pytest.mark.parametrize("shape,fluid,want", FP64)
def test_fp64_by_size(L, shape, fluid, want):
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the sizes are for 152 SMs")
    cells, _, bits, threads = _info(L, [_channel(*shape, fluid)], "fp64")
    assert (cells, threads) == want and bits == 1


@pytest.mark.parametrize("shape,fluid", [((300, 220, 1), 50001), ((400, 220, 1), 80001), ((60, 40, 32), 50001),
                                         ((60, 40, 32), 58369), ((60, 40, 32), 66001), ((60, 40, 32), 72960)])
@pytest.mark.parametrize("periodic", [False, True])
def test_fp64_steps_against_a_forced_variant(L, shape, fluid, periodic):
    from test_gpu_step_small import _same
    _same(L, [_channel(*shape, fluid).with_(periodic_x=periodic)], "fp64", 1e-12, (33, 2))
