"""What a program of this package spends its time on, as cases that can be run and timed.

A case is one call pattern at one size: a demagnetising field, a number of Runge-Kutta steps,
or a gradient through them, from the few thousand cells of a nanomagnet to the eight million
of a thick film.  ``listed`` names the cases, ``draw`` gives more of the same ranges,
``prepare`` makes what a program holds before the call (plan, state, maps), ``run`` is one
pass through the public entry points, ``work`` the bytes and operations it cannot do without,
and ``exact`` the same result in 64 bits from plain torch: Newell's tensor, FFT convolution
and the equations of motion, none of it this package's code.
"""
import math

import numpy as np
import torch

MU0 = 4e-7 * math.pi
#: mu0 g muB / hbar of the electron, m/(A s)
GAMMA = MU0 * 2.00231930436256 * 9.2740100783e-24 / 1.054571817e-34
DEV = "cuda"

#: six stacked layers of different size and thickness on one in-plane grid of 4 nm
STACK = "512x512x8@2,256x256x4@5,384x128x2@3,128x128x16@4,512x64x1@2,200x200x3@3"
STACK_MS = (8e5, 1.4e6, 4e5, 1e6, 6e5, 1.2e6)
STACK_GAPS = (1e-9, 10e-9, 2e-9, 5e-9, 3e-9)


def _case(kind, n, h, **more):
    """A case with every option at its default: FP32, open boundaries, uniform material, base terms."""
    c = dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], hx=h[0], hy=h[1], hz=h[2], precision="f32", steps=1, dt=1e-13,
             state="grains", images_x=0, images_y=0, images_z=0, maps=False, dmi="none", temperature=0.0, layers="")
    c.update(more)
    return c


def _cube(a):
    return (a, a, a)


def listed():
    return [
        # a single nanomagnet's field, the smallest call: launches and latency
        dict(_case("demag", (32, 32, 4), _cube(5e-9), state="random"), name="demag 32x32x4"),
        # the same magnet stepped in a loop, as a hysteresis or switching study does
        dict(_case("rk4", (32, 32, 4), _cube(5e-9), steps=10, state="random"), name="rk4 32x32x4 x10"),
        # standard-problem-4 film under the adaptive evaluator, at its step ceiling
        dict(_case("rkf45", (256, 64, 1), (1.953125e-9, 1.953125e-9, 3e-9), steps=10, dt=5e-14, state="texture"), name="rkf45 256x64x1 x10"),
        # ultrathin film with interfacial DMI at room temperature: skyrmion dynamics
        dict(_case("rk4", (512, 512, 1), (2e-9, 2e-9, 1e-9), steps=4, dt=5e-14, dmi="interfacial", temperature=300.0),
             name="rk4 512x512x1 dmi 300K x4"),
        # an element whose sizes are what the geometry gives: odd, not powers of two
        dict(_case("demag", (201, 147, 5), (4e-9, 4e-9, 3e-9)), name="demag 201x147x5"),
        # gradient of a loss on the final state with respect to the state and material maps
        dict(_case("adjoint", (256, 256, 8), _cube(3e-9), steps=2, state="texture", maps=True), name="adjoint 256x256x8 x2"),
        # a sample periodic in the plane, with material maps
        dict(_case("rk4", (160, 160, 20), _cube(4e-9), steps=4, images_x=2, images_y=2, maps=True), name="rk4 periodic 160x160x20 x4"),
        # double precision, for reference runs
        dict(_case("rk4", (128, 128, 16), _cube(4e-9), precision="f64"), name="rk4 f64 128x128x16"),
        # a wide element: long transforms in the plane, few planes
        dict(_case("demag", (1500, 700, 4), _cube(5e-9)), name="demag 1500x700x4"),
        # multilayer stack: the field of every layer on every other
        dict(_case("stack", (512, 512, 34), (4e-9, 4e-9, 0.0), dt=5e-14, state="random", layers=STACK), name="rk4 six-layer stack"),
        # the benchmark film of eight million cells, in FP32 and with the FP16 tensor-core stage
        dict(_case("rk4", (512, 512, 32), _cube(4e-9), steps=2), name="rk4 512x512x32 x2"),
        dict(_case("rk4", (512, 512, 32), _cube(4e-9), steps=2, precision="fp16"), name="rk4 fp16 512x512x32 x2"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["demag", "demag", "rk4", "rk4", "rk4", "rkf45", "adjoint", "stack"])
    a = rng.choice([2e-9, 3e-9, 4e-9, 5e-9])
    dt = 5e-14 if a < 3e-9 else 1e-13
    if kind == "stack":
        layers = []
        for _ in range(rng.randint(2, 6)):
            layers.append("%dx%dx%d@%d" % (_log_int(rng, 48, 512), _log_int(rng, 48, 512), rng.randint(1, 5), rng.randint(2, 5)))
        n = [[int(v) for v in l.split("@")[0].split("x")] for l in layers]
        size = (max(l[0] for l in n), max(l[1] for l in n), sum(l[2] for l in n))
        return _case("stack", size, (4e-9, 4e-9, 0.0), dt=5e-14, state="random", layers=",".join(layers))
    if kind == "adjoint":
        n = (_log_int(rng, 32, 256), _log_int(rng, 32, 256), _log_int(rng, 1, 8))
        return _case("adjoint", n, _cube(a), steps=rng.randint(1, 2), dt=dt, state="texture", maps=True)
    if kind == "rkf45":
        n = (_log_int(rng, 32, 512), _log_int(rng, 32, 512), _log_int(rng, 1, 4))
        return _case("rkf45", n, _cube(a), steps=rng.randint(2, 10), dt=dt, state="texture")
    if kind == "demag":
        while True:
            n = (_log_int(rng, 24, 1536), _log_int(rng, 24, 1024), _log_int(rng, 1, 32))
            if n[0] * n[1] * n[2] <= 8 << 20:
                break
        f64 = n[0] * n[1] * n[2] <= 1 << 20 and rng.random() < 0.25
        return _case("demag", n, _cube(a), precision="f64" if f64 else "f32", state=rng.choice(["grains", "random", "texture"]))
    option = rng.choice(["plain", "plain", "maps", "periodic", "terms", "f64", "fp16"])
    n = (_log_int(rng, 24, 512), _log_int(rng, 24, 512), rng.randint(17, 32) if option == "fp16" else _log_int(rng, 1, 32))
    c = _case("rk4", n, _cube(a), steps=rng.randint(1, 2), dt=dt, maps=option == "maps")
    if option == "periodic":
        c.update(images_x=rng.randint(1, 4), images_y=rng.randint(0, 4))
    elif option == "terms":
        c.update(dmi=rng.choice(["none", "bulk", "interfacial"]), temperature=rng.choice([0.0, 77.0, 300.0]))
    elif option == "fp16":
        c.update(precision="fp16")
    elif option == "f64" and n[0] * n[1] * n[2] <= 1 << 20:
        c.update(precision="f64", steps=1)
    return c


# ---------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7fffffff)


def _unit(v):
    return v / v.square().sum(0, keepdim=True).sqrt()


def _smooth(shape, sigma, g):
    """White noise over (ny, nx), smoothed by a periodic Gaussian of `sigma` cells, with values in [0, 1]."""
    ny, nx = shape
    w = torch.randn(ny, nx, generator=g, device=DEV, dtype=torch.float64)
    k2 = torch.fft.fftfreq(ny, device=DEV, dtype=torch.float64)[:, None] ** 2 + torch.fft.fftfreq(nx, device=DEV, dtype=torch.float64) ** 2
    s = torch.fft.ifft2(torch.fft.fft2(w) * torch.exp(-2 * (math.pi * sigma) ** 2 * k2)).real
    return (s - s.min()) / (s.max() - s.min()).clamp_min(1e-300)


def _magnetisation(case, n, g):
    """Unit vectors [3][nz][ny][nx] in FP64: independent cells, columnar Voronoi grains, or a smooth texture."""
    nx, ny, nz = n
    if case["state"] == "random":
        return _unit(torch.randn(3, nz, ny, nx, generator=g, device=DEV, dtype=torch.float64))
    if case["state"] == "texture":
        v = torch.stack([2 * _smooth((ny, nx), 6.0, g) - 1 for _ in range(3)])
        v[2] += 0.2
        return _unit(v)[:, None].expand(3, nz, ny, nx).contiguous()
    lx, ly = nx * case["hx"], ny * case["hy"]
    ns = max(4, int(round(lx * ly / 40e-9 ** 2)))
    sx, sy = (torch.rand(ns, generator=g, device=DEV, dtype=torch.float64) * l for l in (lx, ly))
    d = _unit(torch.randn(3, ns, generator=g, device=DEV, dtype=torch.float64))
    cx = (torch.arange(nx, device=DEV, dtype=torch.float64) + 0.5) * case["hx"]
    owner = torch.empty(ny, nx, device=DEV, dtype=torch.int64)
    rows = max(1, (1 << 26) // (nx * ns))
    for j in range(0, ny, rows):
        y = (torch.arange(j, min(ny, j + rows), device=DEV, dtype=torch.float64) + 0.5) * case["hy"]
        owner[j:j + rows] = ((cx[None, :, None] - sx) ** 2 + (y[:, None, None] - sy) ** 2).argmin(2)
    return d[:, owner][:, None].expand(3, nz, ny, nx).contiguous()


def _layers(case):
    """The stack's layers as [(nx, ny, nz)], cell sizes and lower corners, laterally centred, bottom-up."""
    n, hz = [], []
    for text in case["layers"].split(","):
        size, h = text.split("@")
        n.append(tuple(int(v) for v in size.split("x")))
        hz.append(float(h) * 1e-9)
    hx, hy = case["hx"], case["hy"]
    nx, ny = max(l[0] for l in n), max(l[1] for l in n)
    cells, origins, z = [], [], 0.0
    for i, l in enumerate(n):
        cells.append((hx, hy, hz[i]))
        origins.append(((nx - l[0]) // 2 * hx, (ny - l[1]) // 2 * hy, z))
        z += l[2] * hz[i] + STACK_GAPS[i % len(STACK_GAPS)]
    return n, cells, origins


def _planes(case):
    """(centre, height) of every plane of cells of the stack, layer by layer."""
    return [(o[2] + (q + 0.5) * c[2], c[2]) for l, c, o in zip(*_layers(case)) for q in range(l[2])]


def _material(case):
    """Ms, A, alpha, Ku, easy axis, applied field: Permalloy, or a perpendicular Co film where there is DMI."""
    if case["dmi"] != "none" or case["temperature"] > 0:
        return dict(Ms=5.8e5, A=1.5e-11, alpha=0.1, Ku=8e5, easy=(0.0, 0.0, 1.0), Hext=(0.0, 0.0, 2e4))
    return dict(Ms=8e5, A=1.3e-11, alpha=0.02, Ku=0.0, easy=(0.0, 0.0, 1.0), Hext=(0.0, 0.0, 0.1 / MU0))


def _inputs(case, seed):
    """What a program has before the call, rounded to the type it holds it in."""
    g = _gen(seed)
    ft = torch.float64 if case["precision"] == "f64" else torch.float32
    n = (case["nx"], case["ny"], case["nz"])
    if case["kind"] == "stack":
        layers = _layers(case)[0]
        m = torch.cat([_magnetisation(case, l, g).reshape(-1) for l in layers]).to(ft)
        ms = torch.cat([torch.full((l[0] * l[1] * l[2],), STACK_MS[i], device=DEV, dtype=ft) for i, l in enumerate(layers)])
        return dict(m=m, Ms_map=ms)
    s = dict(m=_magnetisation(case, n, g).to(ft))
    if case["maps"]:
        s["Ms_map"] = (6e5 + 4e5 * _smooth((n[1], n[0]), 2.0, g)).to(ft).expand(n[2], n[1], n[0]).contiguous()
        s["Ku_map"] = (5e5 * _smooth((n[1], n[0]), 2.0, g)).to(ft).expand(n[2], n[1], n[0]).contiguous()
    if case["kind"] == "adjoint":
        s["target"] = _magnetisation(case, n, g).to(ft)
    if case["kind"] == "demag":
        s["m"] = s["m"] * 8e5
    return s


def prepare(case, seed):
    from paper_2008_02478_gb300 import binding as b
    s = _inputs(case, seed)
    n, h = (case["nx"], case["ny"], case["nz"]), (case["hx"], case["hy"], case["hz"])
    prm = _material(case)
    prm.update({k: s[k] for k in ("Ms_map", "Ku_map") if k in s})
    if case["kind"] == "stack":
        plan = b.MultiPlan(*_layers(case))
    else:
        images = (case["images_x"], case["images_y"], case["images_z"])
        plan = b.Plan(*n, *h, fp64=case["precision"] == "f64", tc="fp16" if case["precision"] == "fp16" else None,
                      images=images if any(images) else None)
    if case["dmi"] != "none" or case["temperature"] > 0:
        plan.set_field_terms(b.FieldTerms(dmi=case["dmi"], D=3e-3 if case["dmi"] != "none" else 0.0,
                                          temperature=case["temperature"], seed=int(seed), Kc1=1e4))
    if case["kind"] == "rkf45":
        prm.update(method=b.RKF45, dt_max=case["dt"])
    s.update(case=case, plan=plan, prm=b.LLGParams(**prm), out=torch.empty_like(s["m"]))
    if case["kind"] == "adjoint":
        for k in ("m", "Ms_map", "Ku_map"):
            s[k].requires_grad_(True)
    return s


def run(state):
    case, plan, prm, m = state["case"], state["plan"], state["prm"], state["m"]
    if case["kind"] == "demag":
        return plan.apply(m, state["out"])
    if case["kind"] == "rkf45":
        dt, t = plan.llg_run_rkf45(m, prm, case["dt"], case["steps"])
        return m, dt, t
    if case["kind"] == "adjoint":
        from paper_2008_02478_gb300.autograd import trajectory
        end = trajectory(m, state["Ms_map"], state["Ku_map"], plan, prm, case["steps"], case["dt"])
        loss = (end - state["target"]).square().sum()
        return (end.detach(),) + torch.autograd.grad(loss, (m, state["Ms_map"], state["Ku_map"]))
    if case["precision"] == "f64":
        for _ in range(case["steps"]):
            plan.llg_step(m, prm, case["dt"])
    else:
        plan.llg_run_graph(m, prm, case["dt"], case["steps"])
    return m


# ---------------------------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------------------------
def _padded(n):
    return 1 if n == 1 else 1 << (2 * n - 2).bit_length()


def work(case):
    b = 8 if case["precision"] == "f64" else 4
    p = [_padded(case[k]) for k in ("nx", "ny", "nz")]
    cells, points = case["nx"] * case["ny"] * case["nz"], p[0] * p[1] * p[2]
    octant = 6 * b * (p[0] // 2 + 1) * (p[1] // 2 + 1) * (p[2] // 2 + 1)
    flops = 6 * 2.5 * points * max(1.0, math.log2(points)) + 15 * points
    if case["kind"] == "stack":
        n, cell, _ = _layers(case)
        cells = sum(l[0] * l[1] * l[2] for l in n)
        planes = case["nz"]
        at = _planes(case)
        pairs = len({(min(g, h), max(g, h), round(abs(y - z) * 1e15)) for y, g in at for z, h in at})
        plane = p[0] * p[1]
        octant = 6 * b * pairs * (p[0] // 2 + 1) * (p[1] // 2 + 1)
        flops = 6 * 2.5 * planes * plane * math.log2(plane) + 15 * planes * planes * plane
    # a field evaluation reads its kernel once, its source once, and writes one field
    evaluations = {"demag": 1, "rk4": 4, "stack": 4, "rkf45": 6, "adjoint": 8}[case["kind"]] * case["steps"]
    return {"bytes": float(evaluations * (octant + 6 * b * cells)), "flops": float(evaluations * (flops + 60 * cells))}


# ---------------------------------------------------------------------------------------------
# The same results in 64 bits
# ---------------------------------------------------------------------------------------------
def _newell_f(x, y, z):
    x, y, z = x.abs(), y.abs(), z.abs()
    x2, y2, z2 = x * x, y * y, z * z
    r = (x2 + y2 + z2).sqrt()
    t = 1e-300
    s = 0.5 * y * (z2 - x2) * torch.asinh(y / (x2 + z2).sqrt().clamp_min(t)) * (x2 + z2 > 0)
    s = s + 0.5 * z * (y2 - x2) * torch.asinh(z / (x2 + y2).sqrt().clamp_min(t)) * (x2 + y2 > 0)
    return s - x * y * z * torch.atan(y * z / (x * r).clamp_min(t)) * (x > 0) + (2 * x2 - y2 - z2) * r / 6


def _newell_g(x, y, z):
    sign = torch.sign(x) * torch.sign(y)
    x, y, z = x.abs(), y.abs(), z.abs()
    x2, y2, z2 = x * x, y * y, z * z
    r = (x2 + y2 + z2).sqrt()
    t = 1e-300
    s = x * y * z * torch.asinh(z / (x2 + y2).sqrt().clamp_min(t))
    s = s + y / 6 * (3 * z2 - y2) * torch.asinh(x / (y2 + z2).sqrt().clamp_min(t))
    s = s + x / 6 * (3 * z2 - x2) * torch.asinh(y / (x2 + z2).sqrt().clamp_min(t))
    s = s - z2 * z / 6 * torch.atan(x * y / (z * r).clamp_min(t)) - z * y2 / 2 * torch.atan(x * z / (y * r).clamp_min(t))
    return sign * (s - z * x2 / 2 * torch.atan(y * z / (x * r).clamp_min(t)) - x * y * r / 3)


def _far(i, j, x, h2):
    """d_i d_j of 1/r averaged over both boxes, to the second moments `h2` (per axis, over two)."""
    r2 = x[0] ** 2 + x[1] ** 2 + x[2] ** 2
    r2 = torch.where(r2 > 0, r2, torch.ones_like(r2))
    r = r2.sqrt()
    d = float(i == j)
    s = (3 * x[i] * x[j] / r2 - d) / (r2 * r)
    for k in range(3):
        a, c = float(i == k), float(j == k)
        s = s + h2[k] * (105 * x[i] * x[j] * x[k] ** 2 / r2 ** 2 - 15 * (d * x[k] ** 2 + 2 * a * x[j] * x[k] + 2 * c * x[i] * x[k] + x[i] * x[j]) / r2
                         + 3 * (d + 2 * a * c)) / (r2 * r2 * r)
    return s


PAIRS = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))


def _tensor(i, j, xs, ys, zs, hx, hy, a, b):
    """N_ij [z][y][x] at displacements zs, ys, xs (uniform in x and y) of a target box of height a from a source box of height b."""
    def wider(v, h):
        return torch.cat([v[:1] - h, v, v[-1:] + h])

    near = 0.0
    for dz, w in ((a + b) / 2, 1.0), ((a - b) / 2, -1.0), ((b - a) / 2, -1.0), (-(a + b) / 2, 1.0):
        p = torch.broadcast_tensors(wider(xs, hx)[None, None, :], wider(ys, hy)[None, :, None], (zs + dz)[:, None, None])
        near = near + w * (_newell_f(p[i], p[(i + 1) % 3], p[(i + 2) % 3]) if i == j else _newell_g(p[i], p[j], p[3 - i - j]))
    near = near[:, 2:] - 2 * near[:, 1:-1] + near[:, :-2]
    near = near[:, :, 2:] - 2 * near[:, :, 1:-1] + near[:, :, :-2]
    near = -near / (4 * math.pi * hx * hy * a)
    p = torch.broadcast_tensors(xs[None, None, :], ys[None, :, None], zs[:, None, None])
    far = -(hx * hy * b) / (4 * math.pi) * _far(i, j, p, (hx * hx / 12, hy * hy / 12, (a * a + b * b) / 24))
    return torch.where(p[0] ** 2 + p[1] ** 2 + p[2] ** 2 <= (40 * max(hx, hy, a, b)) ** 2, near, far)


def _span(n, h):
    return torch.arange(n, device=DEV, dtype=torch.float64) * h


def _wrapped(t, i, j, dims):
    """N_ij at displacements 0..n-1 along `dims` ((dimension, axis) pairs), laid out for circular convolution of length 2 n."""
    for d, axis in dims:
        n = t.shape[d]
        if n > 1:
            odd = -1.0 if (i == axis) != (j == axis) else 1.0
            t = torch.cat([t, torch.zeros_like(t.narrow(d, 0, 1)), odd * t.narrow(d, 1, n - 1).flip(d)], d)
    return t


def _demag(case):
    """H of M, both [3][nz][ny][nx], by FFT convolution."""
    n, h = (case["nx"], case["ny"], case["nz"]), (case["hx"], case["hy"], case["hz"])
    im = (case["images_x"], case["images_y"], case["images_z"])
    size = tuple(2 * v if v > 1 else 1 for v in n)[::-1]
    spec = []
    for i, j in PAIRS:
        t = 0.0
        for ix in range(-im[0], im[0] + 1):
            for iy in range(-im[1], im[1] + 1):
                for iz in range(-im[2], im[2] + 1):
                    s = [_span(n[k], h[k]) + v * n[k] * h[k] for k, v in enumerate((ix, iy, iz))]
                    t = t + _tensor(i, j, *s, h[0], h[1], h[2], h[2])
        spec.append(torch.fft.rfftn(_wrapped(t, i, j, ((0, 2), (1, 1), (2, 0)))))

    def field(M):
        m = torch.fft.rfftn(M, s=size, dim=(1, 2, 3))
        kxx, kyy, kzz, kxy, kxz, kyz = spec
        rows = ((kxx, kxy, kxz), (kxy, kyy, kyz), (kxz, kyz, kzz))
        out = [torch.fft.irfftn(r[0] * m[0] + r[1] * m[1] + r[2] * m[2], s=size) for r in rows]
        return -torch.stack([o[:n[2], :n[1], :n[0]] for o in out])

    return field


def _cross(a, b):
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]])


def _neighbours(m, axis, wrap, ghost):
    """The cells after and before each cell along an axis (0 x, 1 y, 2 z); `ghost(sign)` stands outside an open face."""
    d = 3 - axis
    n = m.shape[d]
    after, before = torch.roll(m, -1, d), torch.roll(m, 1, d)
    if wrap:
        return after, before
    at = torch.arange(n, device=DEV).reshape([-1 if k == d else 1 for k in range(4)])
    return torch.where(at == n - 1, ghost(1.0), after), torch.where(at == 0, ghost(-1.0), before)


def _philox_normals(cells, seed, step):
    """Three normals per cell: Philox4x32-10 of (cell, step) under the seed, then Box-Muller."""
    mask = np.uint64(0xffffffff)
    c = [np.arange(cells, dtype=np.uint64), *(np.full(cells, v, np.uint64) for v in (step & 0xffffffff, step >> 32, 0))]
    k0, k1 = seed & 0xffffffff, seed >> 32
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & mask, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & 0xffffffff, (k1 + 0xBB67AE85) & 0xffffffff
    u = [(v.astype(np.float64) + 0.5) / 2.0 ** 32 for v in c]
    ra, rb = np.sqrt(-2 * np.log(u[0])), np.sqrt(-2 * np.log(u[2]))
    g = np.stack([ra * np.cos(2 * np.pi * u[1]), ra * np.sin(2 * np.pi * u[1]), rb * np.cos(2 * np.pi * u[3])])
    return torch.from_numpy(g).to(DEV)


def _rate(case, mat, Ms, Ku, demag, noise):
    """dm/dt of a single mesh; Ms, Ku numbers or maps; `noise` a thermal field or None."""
    h = (case["hx"], case["hy"], case["hz"])
    wrap = [case["images_x"] > 0, case["images_y"] > 0, case["images_z"] > 0]
    e = torch.tensor(mat["easy"], device=DEV, dtype=torch.float64).reshape(3, 1, 1, 1)
    hext = torch.tensor(mat["Hext"], device=DEV, dtype=torch.float64).reshape(3, 1, 1, 1)
    terms = case["dmi"] != "none" or case["temperature"] > 0
    D = 3e-3 if case["dmi"] != "none" else 0.0
    z = torch.zeros(3, 1, 1, 1, device=DEV, dtype=torch.float64)

    def axis_vector(axis, sign):
        v = z.clone()
        v[axis] = sign
        return v

    def rate(m):
        H = demag(Ms * m) + hext
        lap, grad = 0.0, []
        for axis in range(3):
            def ghost(sign):
                if D == 0.0:
                    return m
                u = axis_vector(axis, sign) if case["dmi"] == "bulk" else _cross(axis_vector(2, 1.0), axis_vector(axis, sign))
                return m + h[axis] * D / (2 * mat["A"]) * _cross(u.expand_as(m), m)
            after, before = _neighbours(m, axis, wrap[axis], ghost)
            lap = lap + (after + before - 2 * m) / h[axis] ** 2
            grad.append((after - before) / (2 * h[axis]))
        H = H + 2 * mat["A"] / (MU0 * Ms) * lap
        H = H + 2 * Ku / (MU0 * Ms) * (m * e).sum(0, keepdim=True) * e
        if D:
            dx, dy, dz = grad
            w = torch.stack([dz[1] - dy[2], dx[2] - dz[0], dy[0] - dx[1]]) if case["dmi"] == "bulk" else torch.stack([-dx[2], -dy[2], dx[0] + dy[1]])
            H = H + 2 * D / (MU0 * Ms) * w
        if terms:  # cubic anisotropy of 1e4 J/m^3 along the axes
            s = m * m
            H = H - 2 * 1e4 / (MU0 * Ms) * m * (s.sum(0, keepdim=True) - s)
        if noise is not None:
            H = H + noise
        t = _cross(m, H)
        return -GAMMA / (1 + mat["alpha"] ** 2) * (t + mat["alpha"] * _cross(m, t))

    return rate


def _rk4(m, rate, dt):
    k1 = rate(m)
    k2 = rate(m + 0.5 * dt * k1)
    k3 = rate(m + 0.5 * dt * k2)
    k4 = rate(m + dt * k3)
    return _unit(m + dt / 6 * (k1 + 2 * k2 + 2 * k3 + k4))


def _fehlberg(m, rate, dt):
    a = ((), (1 / 4,), (3 / 32, 9 / 32), (1932 / 2197, -7200 / 2197, 7296 / 2197), (439 / 216, -8, 3680 / 513, -845 / 4104),
         (-8 / 27, 2, -3544 / 2565, 1859 / 4104, -11 / 40))
    k = []
    for row in a:
        k.append(rate(m + dt * sum((w * q for w, q in zip(row, k)), torch.zeros_like(m))))
    return _unit(m + dt * (25 / 216 * k[0] + 1408 / 2565 * k[2] + 2197 / 4104 * k[3] - k[4] / 5))


def _exact_stack(case, s):
    n, cells, origins = _layers(case)
    hx, hy = case["hx"], case["hy"]
    nx, ny, planes = case["nx"], case["ny"], case["nz"]
    size = (2 * ny if ny > 1 else 1, 2 * nx if nx > 1 else 1)
    at, spectra = _planes(case), {}

    def spectrum(p, q):
        """The kernel of plane q's field on plane p; xz and yz are odd along x or y, their spectra imaginary."""
        a, b, dz = at[p][1], at[q][1], at[p][0] - at[q][0]
        key = (a, b, round(abs(dz) * 1e15))
        if key not in spectra:
            zs = torch.tensor([abs(dz)], device=DEV, dtype=torch.float64)
            t = [_wrapped(_tensor(i, j, _span(nx, hx), _span(ny, hy), zs, hx, hy, a, b)[0], i, j, ((0, 1), (1, 0))) for i, j in PAIRS]
            k = torch.fft.rfft2(torch.stack(t))
            spectra[key] = k[:4].real.contiguous(), k[4:].imag.contiguous()
        real, imag = spectra[key]
        return (*real, *((1j if dz >= 0 else -1j) * imag))

    m = s["m"].double()
    split = [l[0] * l[1] * l[2] for l in n]
    off = [int(round(o[0] / hx)) for o in origins], [int(round(o[1] / hy)) for o in origins]

    def parts(v):
        return [w.reshape(3, l[2], l[1], l[0]) for w, l in zip(torch.split(v, [3 * c for c in split]), n)]

    mat = _material(case)
    own = [_rate(dict(case, hz=c[2]), mat, STACK_MS[i], 0.0, lambda M: 0.0, None) for i, c in enumerate(cells)]

    def rate(v):
        layers = parts(v)
        frame = torch.zeros(planes, 3, ny, nx, device=DEV, dtype=torch.float64)
        p = 0
        for i, l in enumerate(n):
            x, y = off[0][i], off[1][i]
            frame[p:p + l[2], :, y:y + l[1], x:x + l[0]] = STACK_MS[i] * layers[i].transpose(0, 1)
            p += l[2]
        F = torch.fft.rfft2(frame, s=size)
        H = torch.empty_like(frame)
        for t in range(planes):
            acc = torch.zeros_like(F[0])
            for q in range(planes):
                kxx, kyy, kzz, kxy, kxz, kyz = spectrum(t, q)
                a, b, c = F[q]
                acc[0] -= kxx * a + kxy * b + kxz * c
                acc[1] -= kxy * a + kyy * b + kyz * c
                acc[2] -= kxz * a + kyz * b + kzz * c
            H[t] = torch.fft.irfft2(acc, s=size)[:, :ny, :nx]
        out, p = [], 0
        for i, l in enumerate(n):
            x, y = off[0][i], off[1][i]
            mi = layers[i]
            h = H[p:p + l[2], :, y:y + l[1], x:x + l[0]].transpose(0, 1)
            t = _cross(mi, h)
            out.append((own[i](mi) - GAMMA / (1 + mat["alpha"] ** 2) * (t + mat["alpha"] * _cross(mi, t))).reshape(-1))
            p += l[2]
        return torch.cat(out)

    k1 = rate(m)
    k2 = rate(m + 0.5 * case["dt"] * k1)
    k3 = rate(m + 0.5 * case["dt"] * k2)
    k4 = rate(m + case["dt"] * k3)
    v = m + case["dt"] / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
    return torch.cat([_unit(w).reshape(-1) for w in parts(v)])


def exact(case, seed):
    s = _inputs(case, seed)
    if case["kind"] == "stack":
        return _exact_stack(case, s)
    demag = _demag(case)
    m = s["m"].double()
    if case["kind"] == "demag":
        return demag(m)
    mat = _material(case)
    Ms, Ku = (s[k].double() if k in s else v for k, v in (("Ms_map", mat["Ms"]), ("Ku_map", mat["Ku"])))
    dt = case["dt"]
    if case["kind"] == "adjoint":
        leaf = [v.clone().requires_grad_(True) for v in (m, Ms, Ku)]
        rate = _rate(case, mat, leaf[1], leaf[2], demag, None)
        end = leaf[0]
        for _ in range(case["steps"]):
            end = _rk4(end, rate, dt)
        return (end.detach(),) + torch.autograd.grad((end - s["target"].double()).square().sum(), leaf)
    cells = m[0].numel()
    for step in range(case["steps"]):
        noise = None
        if case["temperature"] > 0:
            sigma = math.sqrt(2 * mat["alpha"] * 1.380649e-23 * case["temperature"] / (GAMMA * MU0 * mat["Ms"] * case["hx"] * case["hy"] * case["hz"] * dt))
            noise = sigma * _philox_normals(cells, int(seed), step).reshape(m.shape)
        rate = _rate(case, mat, Ms, Ku, demag, noise)
        m = (_fehlberg if case["kind"] == "rkf45" else _rk4)(m, rate, dt)
    return (m, dt, dt * case["steps"]) if case["kind"] == "rkf45" else m
