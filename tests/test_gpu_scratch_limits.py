"""Device scratch at its limits: conversions of dense fields fall back to the
host when no memory is left for them, and a refused allocation leaves nothing
behind that a later call reports."""
import numpy as np
import pytest

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


def _tube(nx, ny, nz):
    """A grid that is solid but for its end planes and a tube of one voxel:
    a large dense grid with few fluid cells."""
    c = cases.open_channel(nx, ny, nz, current_A_cm2=0.5)
    c.solid[:, :, 1:-1] = True
    c.solid[nz // 2, ny // 2, :] = False
    return c


def _field(c):
    x = np.linspace(0.0, 1.0, c.shape[2])
    X = np.empty((3,) + c.shape)
    X[0] = 0.5 + 0.1 * x
    X[1] = 0.2 - 0.1 * x * x
    X[2] = 1.0 - X[0] - X[1]
    return X


class _Full:
    """Holds all device memory but `left` bytes."""

    def __init__(self, left):
        self.left = left

    def __enter__(self):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        self.hog = torch.empty(free - self.left, dtype=torch.uint8, device="cuda")
        assert torch.cuda.mem_get_info()[0] <= self.left

    def __exit__(self, *a):
        del self.hog
        torch.cuda.empty_cache()


def _use(s, c, X):
    s.set_bc(c.x_in, c.current_A_cm2)
    s.set_fields(X)
    back = s.fields()
    s.step(5)
    r = s.residual(5)
    return back, s.fields(), r


def test_fields_convert_on_the_host_when_the_device_is_full(L):
    c = _tube(2048, 64, 64)                          # 8.4 M voxels: 201 MB for three species
    X = _field(c)
    want = _use(L.Solver.from_case(c, torch_allocator=False), c, X)
    s = L.Solver.from_case(c, torch_allocator=False)
    with _Full(100 << 20):
        got = _use(s, c, X)
        s.set_fields(X)                              # refused once, not asked for again
        s.step(1)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]) and got[2] == want[2]
    f = ~c.solid
    assert np.abs(got[0] - X)[:, f].max() <= 2.0 ** -48 and np.all(got[0][:, c.solid] == 0.0)
    s.close()


def test_a_refused_allocation_is_not_repeated(L, monkeypatch):
    c = _tube(64, 32, 32)
    X = _field(c)
    want = _use(L.Solver.from_case(c), c, X)
    s = L.Solver.from_case(c)
    asked = []
    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", lambda size, *a: asked.append(size) or 0)
    got = _use(s, c, X)
    assert len(asked) == 1
    monkeypatch.undo()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]) and got[2] == want[2]
    s.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_one_species_at_a_time(L, precision):
    c = _tube(2048, 72, 77)                          # 11.4 M voxels: three species pass 256 MB
    X = _field(c)
    s = L.Solver.from_case(c, precision=precision)
    held = s.info().device_bytes
    s.set_bc(c.x_in, c.current_A_cm2)
    s.set_fields(X)
    got = s.fields()
    assert s.info().device_bytes == held             # given back after each call
    assert np.abs(got - X)[:, ~c.solid].max() <= (0.0 if precision == "fp64" else 2.0 ** -48)
    assert np.all(got[:, c.solid] == 0.0)
    s.close()


def test_training_goes_on_after_a_batch_that_did_not_fit(L):
    net = L.UNet(width=8, max_voxels=128 ** 3, seed=3)
    rng = np.random.default_rng(1)
    net.set([rng.standard_normal(p.shape).astype(np.float32) for p in net.get(0)])
    small = rng.random((1, 17, 8, 8, 8), dtype=np.float32)
    want = net.forward(small)                        # a forward pass adds in one order: equal bits
    with _Full(600 << 20):                           # the layout of 128^3 voxels takes 2.5 GB
        with pytest.raises(L.LbmsError) as e:
            net.forward(np.zeros((1, 17, 128, 128, 128), np.float32))
        assert e.value.status == L.LBMS_ENOMEM
        assert np.array_equal(net.forward(small), want)
    assert np.array_equal(net.forward(small), want)
    net.close()


def test_what_a_handle_keeps(L):
    c = _tube(256, 64, 64)                           # 1.05 M voxels: 25 MB for three species
    s = L.Solver.from_case(c)
    held = s.info().device_bytes
    for _ in range(2):
        s.set_bc(c.x_in, c.current_A_cm2)
        s.set_fields(_field(c))
        s.fields()
    assert s.info().device_bytes - held == 24 * c.solid.size <= 256 << 20
    s.close()


def test_what_a_network_keeps(L):
    net = L.Net(width=64, depth=1, seed=1)
    s = []
    for shape, most in (((256, 64, 64), 64 << 20), ((2048, 96, 80), 512 << 20)):   # 45 MB and 680 MB of working memory
        c = _tube(*shape)
        s.append(L.Solver.from_case(c, torch_allocator=False))
        s[-1].set_bc(c.x_in, c.current_A_cm2)
        s[-1].fields()                               # the handle's own room, kernels loaded
        net.features(s[0], int((~_tube(256, 64, 64).solid).sum()))
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        for _ in range(2):
            X = net.warm_start(s[-1])
        assert free - torch.cuda.mem_get_info()[0] <= (2 << 20) + (0 if shape[0] == 2048 else most)
        assert np.abs(X.sum(0)[~c.solid] - 1.0).max() <= 1e-12
        del X
    for h in s:
        h.close()
    net.close()
