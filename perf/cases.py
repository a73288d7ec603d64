"""What the performance of this framework is measured on: the calls a user's
program makes through the Python binding, over the sizes that its own
configurations, tests and benchmark use.

* ``kind = "lbm"``: a handle with boundary data and a state; one pass is
  ``steps`` time steps watched by a residual every 100 steps (the loop of a
  run to steady state) and the mole fractions of every case read back.
* ``kind = "unet"``: one optimiser step of the 3-D U-Net warm start on its
  training volumes, and the gradients.
* ``kind = "net"``: one optimiser step of the pointwise warm-start network on
  the caller's rows, and the gradients.
* ``kind = "start"``: the U-Net's prediction for an anode, which becomes the
  handle's state.

Mole fractions come back in the handle's own precision (the binding hands
out FP64 arrays; FP32 and FP16-storage handles compute in FP32).
"""
import math

import numpy as np
import torch

from paper_1809_01600_gb300 import lbms

CHECK = 100          # steps between two residual checks (the library's default)
UNET_WIDTH = 28      # the default U-Net: 1.05M parameters
PERIODIC_Q = {2: 9, 3: 19}


def listed():
    return [
        # The homogenised set-up of the paper's Section 4.2: 15 one-dimensional
        # 64-node strips (3 currents x 5 dilutions) in one batch.  The smallest
        # call: 960 cells, nothing but the latency of a step.
        _lbm("strips_15x64_fp32", dim=2, nx=64, ny=1, nz=1, cases=15, radius=0, porosity=1.0, precision="fp32",
             steps=2000),
        # The small resolved 2-D anode in FP64, the precision of reference runs.
        _lbm("anode2d_96x48_fp64", dim=2, nx=96, ny=48, nz=1, cases=1, radius=4, porosity=0.45, precision="fp64",
             steps=1000),
        # A sweep of uneven 2-D anodes in one batch.
        _lbm("sweep2d_8x1000x500_fp32", dim=2, nx=1000, ny=500, nz=1, cases=8, radius=4, porosity=0.50,
             precision="fp32", steps=1000, uneven=True),
        # One small 3-D anode of odd extents: a fraction of the GPU, every step a launch.
        _lbm("anode3d_61x37x29_fp32", dim=3, nx=61, ny=37, nz=29, cases=1, radius=3, porosity=0.40, precision="fp32",
             steps=1000),
        # Steady states for training a warm start: many anodes of one grid in one batch.
        _lbm("batch3d_48x64x32x32_fp32", dim=3, nx=64, ny=32, nz=32, cases=48, radius=3, porosity=0.42,
             precision="fp32", steps=500),
        # A held-out anode of the warm-start grid, run in the chosen form (FP16 storage).
        _lbm("anode3d_96x96x96_fp16", dim=3, nx=96, ny=96, nz=96, cases=1, radius=3, porosity=0.42, precision="fp16",
             steps=1000),
        # The headline anode in both of its forms.
        _lbm("anode3d_256x128x128_fp32", dim=3, nx=256, ny=128, nz=128, cases=1, radius=3, porosity=0.40,
             precision="fp32", steps=1000),
        _lbm("anode3d_256x128x128_fp16", dim=3, nx=256, ny=128, nz=128, cases=1, radius=3, porosity=0.40,
             precision="fp16", steps=1000),
        # Training the U-Net on volumes of the two training grids.
        dict(name="unet_train_8x64x32x32", kind="unet", batch=8, nx=64, ny=32, nz=32),
        dict(name="unet_train_4x96x96x96", kind="unet", batch=4, nx=96, ny=96, nz=96),
        # Training the pointwise network at its default width and batch.
        dict(name="net_train_8192x704", kind="net", rows=8192, width=704, depth=3),
        # A start predicted for a held-out anode whose extents are not multiples of four.
        dict(name="start_95x90x86", kind="start", nx=95, ny=90, nz=86, radius=3, porosity=0.42),
    ]


def draw(rng):
    def span(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    what = rng.choice(["strips", "anode2d", "sweep2d", "anode3d", "anode3d", "batch3d", "unet", "net", "start"])
    if what == "strips":
        return _lbm(None, dim=2, nx=span(17, 129), ny=1, nz=1, cases=span(1, 32), radius=0, porosity=1.0,
                    precision=rng.choice(["fp64", "fp32", "fp16"]), steps=100 * span(5, 30))
    if what == "anode2d":
        return _lbm(None, dim=2, nx=span(48, 400), ny=span(24, 200), nz=1, cases=1, radius=rng.randint(2, 5),
                    porosity=round(rng.uniform(0.45, 0.6), 3), precision=rng.choice(["fp64", "fp32", "fp16"]),
                    steps=100 * span(4, 15))
    if what == "sweep2d":
        return _lbm(None, dim=2, nx=span(128, 1000), ny=span(64, 500), nz=1, cases=span(2, 8),
                    radius=rng.randint(2, 6), porosity=round(rng.uniform(0.45, 0.55), 3),
                    precision=rng.choice(["fp32", "fp16"]), steps=100 * span(2, 10), uneven=True)
    if what == "anode3d":
        n = span(20, 160)
        return _lbm(None, dim=3, nx=max(16, int(n * rng.uniform(0.8, 1.4))), ny=max(12, int(n * rng.uniform(0.6, 1.0))),
                    nz=max(11, int(n * rng.uniform(0.6, 1.0))), cases=1, radius=rng.randint(2, 4),
                    porosity=round(rng.uniform(0.35, 0.5), 3), precision=rng.choice(["fp32", "fp16", "fp32", "fp64"]),
                    steps=100 * span(1, 4))
    if what == "batch3d":
        return _lbm(None, dim=3, nx=span(24, 72), ny=span(16, 40), nz=span(16, 40), cases=span(4, 40),
                    radius=rng.randint(2, 4), porosity=round(rng.uniform(0.35, 0.5), 3),
                    precision=rng.choice(["fp32", "fp16"]), steps=100 * span(1, 4), uneven=rng.random() < 0.5)
    if what == "unet":
        return dict(kind="unet", batch=rng.randint(1, 8), nx=4 * rng.randint(4, 18), ny=4 * rng.randint(3, 12),
                    nz=4 * rng.randint(3, 12))
    if what == "net":
        return dict(kind="net", rows=64 * span(4, 256), width=64 * span(2, 14), depth=rng.randint(1, 4))
    return dict(kind="start", nx=span(30, 100), ny=span(20, 90), nz=span(20, 90), radius=rng.randint(2, 4),
                porosity=round(rng.uniform(0.35, 0.5), 3))


def _lbm(name, **kw):
    c = dict(kind="lbm", uneven=False)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def _grids(case):
    """(nz, ny, nx) of every anode of the case; an uneven batch shrinks to half the extents."""
    out = []
    for k in range(case.get("cases", 1)):
        f = 1.0 - 0.5 * k / case["cases"] if case.get("uneven") else 1.0
        out.append(tuple(1 if n == 1 else max(8, int(n * f)) for n in (case["nz"], case["ny"], case["nx"])))
    return out


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + 17)


def _shifts(a, dim):
    """The face neighbours' values of a boolean field [..., z, y, x]: y and z periodic, x not."""
    n = torch.zeros_like(a)
    n[..., 1:] |= a[..., :-1]
    n[..., :-1] |= a[..., 1:]
    n |= torch.roll(a, 1, -2) | torch.roll(a, -1, -2)
    if dim == 3:
        n |= torch.roll(a, 1, -3) | torch.roll(a, -1, -3)
    return n


def _masks(count, grid, dim, radius, porosity, gen):
    """`count` solid masks of overlapping balls on one grid (inlet and outlet
    planes fluid, fluid that the inlet does not reach solid), as numpy."""
    nz, ny, nx = grid
    if radius == 0:
        return [np.zeros(grid, dtype=bool) for _ in range(count)]
    r = torch.arange(-radius, radius + 1)
    offs = [(z, y, x) for z in (r.tolist() if dim == 3 else [0]) for y in r.tolist() for x in r.tolist()
            if x * x + y * y + z * z <= radius * radius]
    while True:
        p = -math.log(porosity) / len(offs)
        c = torch.rand((count, nz, ny, nx), generator=gen, device="cuda") < p
        c = torch.nn.functional.pad(c, (radius, radius))
        solid = torch.zeros_like(c)
        for z, y, x in offs:
            solid |= torch.roll(c, (z, y, x), (1, 2, 3))
        fluid = ~solid[..., radius:radius + nx]
        fluid[..., 0] = True
        fluid[..., -1] = True
        seen = torch.zeros_like(fluid)
        seen[..., 0] = True
        have = -1
        while True:
            for _ in range(24):
                seen |= _shifts(seen, dim) & fluid
            now = int(seen.sum())
            if now == have:
                break
            have = now
        if bool(seen[..., -1].all()):
            return list((~seen).cpu().numpy())
        porosity = min(0.95, porosity + 0.03)


def _points(count, gen):
    """(inlet mole fractions, current) of every anode: H2:H2O = 4:1, Ar the balance."""
    u = torch.rand((count, 2), generator=gen, device="cuda").cpu().numpy()
    out = []
    for a, b in u:
        xh = 0.45 + 0.30 * float(a)
        out.append(((xh, xh / 4.0, 1.0 - 1.25 * xh), 0.25 + 0.75 * float(b)))
    return out


def _state(grid, x_in, gen):
    """A field on its way to the steady state: H2 falls towards the outlet
    and H2O rises, with a transverse ripple."""
    nz, ny, nx = grid
    a = torch.rand(4, generator=gen, device="cuda", dtype=torch.float64)
    x = torch.arange(nx, device="cuda", dtype=torch.float64) / max(nx - 1, 1)
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None] / ny
    z = torch.arange(nz, device="cuda", dtype=torch.float64)[:, None, None] / nz
    drop = (0.04 + 0.08 * a[0]) * x * (1.0 + 0.3 * torch.sin(2 * math.pi * (y + a[1])) * torch.cos(2 * math.pi * (z + a[2])))
    drop = drop.expand(nz, ny, nx)
    return torch.stack([x_in[0] - drop, x_in[1] + 0.9 * drop, x_in[2] + 0.1 * drop])


def _inputs(case, seed):
    gen = _gen(seed)
    grids = _grids(case)
    if case.get("uneven"):
        masks = [_masks(1, g, case["dim"], case["radius"], case["porosity"], gen)[0] for g in grids]
    else:
        masks = _masks(len(grids), grids[0], case["dim"], case["radius"], case["porosity"], gen)
    points = _points(len(grids), gen)
    fields = [_state(g, p[0], gen) for g, p in zip(grids, points)]
    return grids, masks, points, fields


def _handle(case, masks, points, fields):
    dim, prec = case["dim"], case["precision"]
    if len(masks) == 1:
        h = lbms.Solver(masks[0], dim=dim, precision=prec)
        h.set_bc(*points[0])
        h.set_fields(fields[0].cpu().numpy())
    else:
        h = lbms.Batch(masks, dim=dim, precision=prec)
        for k, (x_in, current) in enumerate(points):
            h.set_bc(x_in, current, case=k)
        for k, X in enumerate(fields):
            h.set_fields(k, X.cpu().numpy())
    return h


def _unet_shapes(w):
    out = []
    for ci, co in ((17, w), (w, w), (w, 2 * w), (2 * w, 2 * w), (2 * w, 4 * w), (4 * w, 4 * w)):
        out += [(co, ci, 3, 3, 3), (co,)]
    out += [(4 * w, 2 * w, 2, 2, 2), (2 * w,), (2 * w, 4 * w, 3, 3, 3), (2 * w,), (2 * w, 2 * w, 3, 3, 3), (2 * w,)]
    out += [(2 * w, w, 2, 2, 2), (w,), (w, 2 * w, 3, 3, 3), (w,), (w, w, 3, 3, 3), (w,), (3, w, 1, 1, 1), (3,)]
    return out


def _unet_params(gen):
    """Weights of the size a trained network has: He-uniform, a smaller head, small biases."""
    out = []
    for sh in _unet_shapes(UNET_WIDTH):
        if len(sh) == 1:
            out.append((0.05 * torch.randn(sh, generator=gen, device="cuda")).cpu().numpy())
            continue
        fan = sh[0] if sh[2] == 2 else int(np.prod(sh[1:]))
        a = math.sqrt(6.0 / fan) * (0.3 if sh[2] == 1 else 1.0)
        out.append((a * (2.0 * torch.rand(sh, generator=gen, device="cuda") - 1.0)).cpu().numpy())
    return out


def _volumes(case, seed):
    """Training volumes [B, 17, Z, Y, X] (feature columns on fluid voxels, the
    fluid mask) and targets [B, 3, Z, Y, X], and the network's weights."""
    gen = _gen(seed)
    B, Z, Y, X = case["batch"], case["nz"], case["ny"], case["nx"]
    m = (torch.rand((B, 1, Z, Y, X), generator=gen, device="cuda") < 0.45).float()
    f = torch.rand((B, 16, Z, Y, X), generator=gen, device="cuda") * m
    x = torch.cat([f, m], 1)
    t = (4.0 * torch.nn.functional.avg_pool3d(f[:, 0:3], 3, stride=1, padding=1) + f[:, 3:6] * f[:, 6:7] - 1.0) * m
    return x, t, _unet_params(gen)


def _rows(case, seed):
    """Feature rows (BF16 bit patterns), targets and the network's layers."""
    gen = _gen(seed)
    x = torch.zeros((case["rows"], 64), device="cuda")
    x[:, :16] = 2.0 * torch.rand((case["rows"], 16), generator=gen, device="cuda") - 1.0
    x = x.to(torch.bfloat16)
    t = torch.randn((case["rows"], 3), generator=gen, device="cuda")
    dims = [64] + [case["width"]] * case["depth"] + [3]
    layers = []
    for i, o in zip(dims[:-1], dims[1:]):
        W = math.sqrt(2.0 / (16 if i == 64 else i)) * torch.randn((o, i), generator=gen, device="cuda")
        layers.append((W, 0.1 * torch.randn(o, generator=gen, device="cuda")))
    return x, t, layers


def _start_inputs(case, seed):
    gen = _gen(seed)
    grid = (case["nz"], case["ny"], case["nx"])
    mask = _masks(1, grid, 3, case["radius"], case["porosity"], gen)[0]
    return mask, _points(1, gen)[0], _unet_params(gen)


# -------------------------------------------------------------- the passes
def prepare(case, seed):
    kind = case["kind"]
    if kind == "lbm":
        _, masks, points, fields = _inputs(case, seed)
        return dict(case=case, h=_handle(case, masks, points, fields))
    if kind == "unet":
        x, t, params = _volumes(case, seed)
        net = lbms.UNet(width=UNET_WIDTH, max_voxels=case["batch"] * case["nx"] * case["ny"] * case["nz"], seed=3)
        net.set(params)
        x, t = x.cpu().numpy(), t.cpu().numpy()
        for k in range(case["batch"]):
            net.add_volume(x[k], t[k])
        return dict(case=case, net=net)
    if kind == "net":
        x, t, layers = _rows(case, seed)
        net = lbms.Net(width=case["width"], depth=case["depth"], seed=3)
        net.set([(W.cpu().numpy(), b.cpu().numpy()) for W, b in layers])
        return dict(case=case, net=net, x=x.view(torch.uint16).cpu().numpy(), t=t.cpu().numpy())
    mask, (x_in, current), params = _start_inputs(case, seed)
    net = lbms.UNet(width=UNET_WIDTH, max_voxels=(case["nx"] + 3) * (case["ny"] + 3) * (case["nz"] + 3), seed=3)
    net.set(params)
    h = lbms.Solver(mask, dim=3, precision="fp16")
    h.set_bc(x_in, current)
    return dict(case=case, net=net, h=h)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "lbm":
        h, n = state["h"], case.get("cases", 1)
        for _ in range(case["steps"] // CHECK):
            h.step(CHECK)
            h.residual(CHECK) if n == 1 else h.residuals(CHECK)
        fields = [h.fields()] if n == 1 else [h.fields(k) for k in range(n)]
        if not case["uneven"] and n > 1:
            fields = [np.stack(fields)]
        if case["precision"] == "fp64":
            return fields
        return [torch.from_numpy(X).float() for X in fields]
    if kind == "unet":
        # a fine-tuning rate: the network goes on from trained weights
        loss = state["net"].train(1, max_batch=case["batch"], lr=1e-5)
        return [loss] + state["net"].get(1)
    if kind == "net":
        loss = state["net"].train_batch(state["x"], state["t"], lr=1e-5)
        return [loss] + [g for layer in state["net"].get(1) for g in layer]
    return torch.from_numpy(state["net"].warm_start(state["h"])).float()


def work(case):
    kind = case["kind"]
    if kind == "lbm":
        q, dim = PERIODIC_Q[case["dim"]], case["dim"]
        cells = sum(z * y * x for z, y, x in _grids(case))
        fluid = cells * case["porosity"]
        word, xw = {"fp64": (8, 8), "fp32": (4, 4), "fp16": (2, 4)}[case["precision"]]
        out = 3 * cells * (8 if case["precision"] == "fp64" else 4)
        # every population and mole fraction read once and written once a step
        return {"bytes": case["steps"] * fluid * 3 * 2 * (q * word + xw) + out,
                "flops": case["steps"] * fluid * 3 * (8 * q + 20 * dim + 40)}
    if kind == "net":
        w, d, r = case["width"], case["depth"], case["rows"]
        macs = 16 * w + (d - 1) * w * w + 3 * w
        return {"bytes": r * (32 + 12) + 4 * 8 * macs, "flops": 6 * r * macs}
    w = UNET_WIDTH
    if kind == "unet":
        vox = case["batch"] * case["nx"] * case["ny"] * case["nz"]
    else:
        vox = math.prod((n + 3) // 4 * 4 for n in (case["nx"], case["ny"], case["nz"]))
    # multiply-adds a voxel of the finest level: 3x3x3 convolutions, transposed convolutions, head
    macs = 27 * (17 * w + w * w + 2 * w * w + w * w) + 3 * w
    macs += 27 * (2 * w * w + 4 * w * w + 8 * w * w + 4 * w * w) / 8 + 2 * w * w
    macs += 27 * (8 * w * w + 16 * w * w) / 64 + 8 * w * w / 8
    params = sum(int(np.prod(s)) for s in _unet_shapes(w))
    if kind == "unet":
        return {"bytes": vox * (17 * 2 + 16) + params * 4 * 8, "flops": 6 * vox * macs}
    return {"bytes": vox * (17 * 2 + 3 * 4) + params * 2, "flops": 2 * vox * macs}


# ------------------------------------------------------------ 64-bit values
def exact(case, seed):
    kind = case["kind"]
    if kind == "lbm":
        grids, masks, points, fields = _inputs(case, seed)
        out = [_exact_lbm(case, m, p, f).cpu().numpy() for m, p, f in zip(masks, points, fields)]
        return [np.stack(out)] if not case["uneven"] and len(out) > 1 else out
    if kind == "unet":
        if case["batch"] * case["nx"] * case["ny"] * case["nz"] > 1200000:
            return None
        return _exact_unet_step(case, seed)
    if kind == "net":
        return _exact_net_step(case, seed)
    return _exact_start(case, seed)


GAS_M, GAS_V = (2.016, 18.015, 39.948), (6.12, 13.1, 16.2)    # kg/kmol and Fuller volumes (Table 1)
R_GAS, FARADAY = 8.3145, 96485.0


def _scaling(nx, current, T=1073.0, p=101325.0, pore=1e-6, length=2e-3):
    """Lattice diffusivities and the outlet flux (Eqs. 39-42), and D_ij / C_t in SI units."""
    D = np.zeros((3, 3))
    for i in range(3):
        for j in range(3):
            if i != j:
                D[i, j] = 1e-4 * 0.00143 * T ** 1.75 * math.sqrt(1 / GAS_M[i] + 1 / GAS_M[j]) / (
                    p / 1e5 * (GAS_V[i] ** (1 / 3) + GAS_V[j] ** (1 / 3)) ** 2)
    K = [pore / 3 * math.sqrt(8 * R_GAS * T / (math.pi * m / 1000)) for m in GAS_M]
    E = np.zeros((3, 3))
    for i in range(3):
        for j in range(3):
            if i != j:
                E[i, j] = 0.5 * (1 / (1 / D[i, j] + 1 / K[i]) + 1 / (1 / D[i, j] + 1 / K[j]))
    dx = length / (nx - 1)
    dt = dx * dx / (6 * min(E[0, 1], E[0, 2], E[1, 2]))
    ct = p / (R_GAS * T)
    N = np.array([1.0, -1.0, 0.0]) * current * 1e4 / (2 * FARADAY)
    return E * dt / dx ** 2, N * dt / (ct * dx), E, ct, N, dx


def _links(dim):
    if dim == 2:
        e = [(x, y, 0) for x in (-1, 0, 1) for y in (-1, 0, 1)]
        w = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}
    else:
        e = [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1) if abs(x) + abs(y) + abs(z) <= 2]
        w = {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
    return e, [w[sum(c * c for c in v)] for v in e]


def _exact_lbm(case, mask, point, X0):
    """The method on the fluid cells, in FP64: pull streaming with half-way
    bounce-back, the Dirichlet inlet (Eq. 36), the flux outlet (Eq. 39), the
    lagged central gradient, the Maxwell-Stefan coupling and BGK."""
    dim = case["dim"]
    (x_in, current), steps = point, case["steps"] // CHECK * CHECK
    nz, ny, nx = mask.shape
    D, q, *_ = _scaling(nx, current)
    e, w = _links(dim)
    Q = len(e)
    opp = [e.index((-a, -b, -c)) for a, b, c in e]
    solid = torch.from_numpy(mask).cuda()
    cell = (~solid).reshape(-1).nonzero().reshape(-1)
    n = cell.numel()
    index = torch.full((solid.numel(),), -1, dtype=torch.int64, device="cuda")
    index[cell] = torch.arange(n, device="cuda")
    x, y, z = cell % nx, (cell // nx) % ny, cell // (nx * ny)
    me = torch.arange(n, device="cuda")
    take, near = [], {}
    for k, (a, b, c) in enumerate(e):
        xs = x - a
        inside = (xs >= 0) & (xs < nx)
        src = index[(((z - c) % nz) * ny + (y - b) % ny) * nx + xs.clamp(0, nx - 1)]
        src = torch.where(inside, src, torch.full_like(src, -1))
        take.append(torch.where(src >= 0, k * n + src, opp[k] * n + me))
        near[(-a, -b, -c)] = (torch.where(src >= 0, src, me), inside)   # the neighbour at x - e_k
    take = torch.stack(take)
    W = torch.tensor(w, dtype=torch.float64, device="cuda")[None, :, None]
    at_in = (x == 0).nonzero().reshape(-1)
    at_out = (x == nx - 1).nonzero().reshape(-1)
    w_out = sum(wk for wk, v in zip(w, e) if v[0] == 1)
    xin = torch.tensor(x_in, dtype=torch.float64, device="cuda")
    qt = torch.tensor(q, dtype=torch.float64, device="cuda")
    X = X0.reshape(3, -1)[:, cell].contiguous()
    f = W * X[:, None, :]
    axes = [(1, 0, 0), (0, 1, 0), (0, 0, 1)][:dim]
    ev = torch.tensor(e, dtype=torch.float64, device="cuda")[:, :dim]
    inc = [k for k in range(Q) if e[k][0] == 1]
    out = [k for k in range(Q) if e[k][0] == -1]
    D12, D13, D23 = D[0, 1], D[0, 2], D[1, 2]
    for _ in range(steps):
        P = f.reshape(3, Q * n)[:, take]
        for k in out:
            P[:, k, at_out] -= (w[opp[k]] / w_out) * qt[:, None]
        for k in inc:
            P[:, k, at_in] = (w[k] + w[opp[k]]) * xin[:, None] - P[:, opp[k], at_in]
        g = []
        for ax in axes:
            (ip, hp), (im, hm) = near[ax], near[tuple(-v for v in ax)]
            dp, dm = X[:, ip] - X, X - X[:, im]
            both = (hp & hm).double() * 0.5
            g.append(dp * torch.where(hp & hm, both, hp.double()) + dm * torch.where(hp & hm, both, (hm & ~hp).double()))
        g = torch.stack(g, 1)
        X = P.sum(1)
        X1, X2, X3 = X
        b11, b12 = X1 / D13 + X2 / D12 + X3 / D13, -X1 * (1 / D12 - 1 / D13)
        b21, b22 = -X2 * (1 / D12 - 1 / D23), X2 / D23 + X1 / D12 + X3 / D23
        det = b11 * b22 - b12 * b21
        j1 = -(b22 * g[0] - b12 * g[1]) / det
        j2 = -(b11 * g[1] - b21 * g[0]) / det
        j3 = (-g[2] + X3 * (j1 / D13 + j2 / D23)) / (X1 / D13 + X2 / D23)
        J = torch.stack([j1, j2, j3])
        # Eq. 24 with the reaction's flux ratios; the mixture value for the inert species
        d1 = 1 / ((X2 + X1) / D12 + X3 / D13)
        d2 = 1 / ((X1 + X2) / D12 + X3 / D23)
        d3 = (X1 + X2 + 1e-12) / (X1 / D13 + X2 / D23 + 0.5e-12 * (1 / D13 + 1 / D23))
        tau = (3 * torch.stack([d1, d2, d3]) + 0.5).clamp(1.0, 5.0)
        v = (J + ((tau - 0.5) / 3)[:, None] * g) * (X / (X * X + 1e-24))[:, None]
        s = (v * v).sum(1, keepdim=True)
        v = v * torch.where(s > 0.01, 0.1 / s.clamp_min(1e-300).sqrt(), torch.ones_like(s))
        e_v = torch.einsum("kd,sdn->skn", ev, v)
        f = P + (W * X[:, None, :] * (1 + 3 * e_v) - P) / tau[:, None]
    full = torch.zeros((3, solid.numel()), dtype=torch.float64, device="cuda")
    full[:, cell] = X
    return full.reshape(3, nz, ny, nx)


def _conv64(h, W, b):
    """3x3x3 convolution with zero padding as 27 matrix products (FP64)."""
    B, C, Z, Y, X = h.shape
    p = torch.nn.functional.pad(h.permute(0, 2, 3, 4, 1), (0, 0, 1, 1, 1, 1, 1, 1))
    out = b.reshape(1, 1, 1, 1, -1).expand(B, Z, Y, X, W.shape[0])
    for dz in range(3):
        for dy in range(3):
            for dx in range(3):
                out = out + p[:, dz:dz + Z, dy:dy + Y, dx:dx + X] @ W[:, :, dz, dy, dx].T
    return torch.relu(out.permute(0, 4, 1, 2, 3))


def _unet64(p, x):
    F = torch.nn.functional
    W, b = p[0::2], p[1::2]

    def conv(h, i):
        return _conv64(h, W[i], b[i])

    def up(h, i):   # stride 2: the eight children of a voxel do not overlap
        B, _, Z, Y, X = h.shape
        o = torch.einsum("bczyx,cokjl->bozkyjxl", h, W[i]).reshape(B, W[i].shape[1], 2 * Z, 2 * Y, 2 * X)
        return o + b[i].reshape(1, -1, 1, 1, 1)

    e1 = conv(conv(x, 0), 1)
    e2 = conv(conv(F.max_pool3d(e1, 2), 2), 3)
    e3 = conv(conv(F.max_pool3d(e2, 2), 4), 5)
    d2 = conv(conv(torch.cat([up(e3, 6), e2], 1), 7), 8)
    d1 = conv(conv(torch.cat([up(d2, 9), e1], 1), 10), 11)
    return torch.einsum("bczyx,oc->bozyx", d1, W[12].reshape(3, -1)) + b[12].reshape(1, -1, 1, 1, 1)


def _splitmix(x):
    """SplitMix64 (Steele, Lea, Flood 2014), which draws the training volumes."""
    m = (1 << 64) - 1
    x = (x + 0x9E3779B97F4A7C15) & m
    x = ((x ^ (x >> 30)) * 0xBF58476D1CE4E5B9) & m
    x = ((x ^ (x >> 27)) * 0x94D049BB133111EB) & m
    return x ^ (x >> 31)


def _exact_unet_step(case, seed):
    x, t, params = _volumes(case, seed)
    key = _splitmix(3 ^ 0x5A5A5A5A)    # the first step of the network made with seed 3
    pick = [_splitmix(key + i) % case["batch"] for i in range(case["batch"])]
    x, t = x[pick].double(), t[pick].double()
    p = [torch.tensor(a, dtype=torch.float64, device="cuda", requires_grad=True) for a in params]
    m = x[:, 16:17]
    loss = (((_unet64(p, x) - t) * m) ** 2).sum() / (3.0 * m.sum())
    grads = torch.autograd.grad(loss, p)
    return [float(loss.detach())] + [g.cpu().numpy() for g in grads]


def _exact_net_step(case, seed):
    x, t, layers = _rows(case, seed)
    p = [a.double().requires_grad_() for layer in layers for a in layer]
    h = x.double()
    for l in range(0, len(p), 2):
        h = h @ p[l].T + p[l + 1]
        if l + 2 < len(p):
            h = torch.relu(h)
    loss = ((h - t.double()) ** 2).mean()
    grads = torch.autograd.grad(loss, p)
    return [float(loss.detach())] + [g.cpu().numpy() for g in grads]


def _profile(nx, x_in, current):
    """Eq. 19 with the fluxes held at their outlet values, integrated from the inlet (RK4, 16 substeps a node)."""
    _, _, E, ct, N, dx = _scaling(nx, current)

    def rhs(X):
        return np.array([sum((X[i] * N[j] - X[j] * N[i]) / (ct * E[i, j]) for j in range(3) if j != i)
                         for i in range(3)])

    X, h, out = np.array(x_in), dx / 16, []
    for j in range(nx):
        out.append(X)
        for _ in range(16):
            k1 = rhs(X)
            k2 = rhs(X + 0.5 * h * k1)
            k3 = rhs(X + 0.5 * h * k2)
            k4 = rhs(X + h * k3)
            X = X + h / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
    return np.stack(out, 1)


def _exact_start(case, seed):
    """The documented feature columns (include/lbms_net.h), the network and
    the clamped, renormalised prediction, in FP64."""
    mask, (x_in, current), params = _start_inputs(case, seed)
    nz, ny, nx = mask.shape
    fluid = torch.from_numpy(~mask).cuda().double()
    prof = torch.from_numpy(_profile(nx, x_in, current)).cuda()
    xr = torch.arange(nx, device="cuda", dtype=torch.float64) / (nx - 1)
    phi = fluid.mean((0, 1)).clamp_min(1.0 / (ny * nz))
    res = torch.cat([phi.new_zeros(1), torch.cumsum(0.5 * (1 / phi[:-1] + 1 / phi[1:]), 0)])

    def box(a, h):
        for axis in (1, 0):
            a = sum(torch.roll(a, d, axis) for d in range(-h, h + 1))
        a = torch.nn.functional.pad(a, (h, h))
        return sum(a[..., d:d + nx] for d in range(2 * h + 1))

    cols = [prof[s].expand(nz, ny, nx) for s in range(3)] + [xr.expand(nz, ny, nx)]
    cols += [box(fluid, h) / box(torch.ones_like(fluid), h) for h in (1, 3, 7)]
    one = torch.ones_like(fluid)
    cols += [0.5 * current * one] + [v * one for v in x_in] + [(0.5 * current * xr).expand(nz, ny, nx)]
    cols += [phi.expand(nz, ny, nx), (res / res[-1]).expand(nz, ny, nx), (0.25 / phi).expand(nz, ny, nx), one]
    x = torch.stack([c * fluid for c in cols] + [fluid])[None]
    x = torch.nn.functional.pad(x, (0, -nx % 4, 0, -ny % 4, 0, -nz % 4))
    with torch.no_grad():
        y = _unet64([torch.tensor(a, dtype=torch.float64, device="cuda") for a in params], x)[0, :, :nz, :ny, :nx]
    X = (prof[:, None, None, :] + y / 100.0).clamp_min(1e-6)
    return (X / X.sum(0) * fluid).cpu().numpy()
