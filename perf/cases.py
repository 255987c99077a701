"""The calls a user of this library makes, over the sizes and options it is used with.

A case is one entry point at one size: the operator apply (the inner step of every iteration), whole
solves (frequency sweeps, refinement, ports), and the convolution layers of the learned
preconditioner, forward and backward.  ``listed()`` names the reference points, ``draw()`` gives more
of the same ranges.  Geometries follow the families of structures the library is written for: an empty
cavity, a layered dielectric with conductor blocks and an absorber, a stripline box, a package with
traces and vias, and a random inhomogeneous (magnetic, lossy) grid.  ``exact()`` computes every result
in 64 bits from the definitions, with torch alone.
"""
import math

import numpy as np
import torch

from paper_1705_08849_gb300 import fit

MU0 = 4.0e-7 * math.pi
C0 = 299792458.0
EPS0 = 1.0 / (MU0 * C0 * C0)
ETA0 = MU0 * C0


def listed():
    return [
        # A closed cavity of 16^3 cells: the smallest grid in use, where a call is all latency.
        dict(name="apply_cavity16", kind="apply", geom="cavity", nx=16, ny=16, nz=16, nb=1, prec="c64", ghz=5.0),
        # The benchmark workload: one operator apply of the layered 128^3 grid in single precision.
        dict(name="apply_layered128", kind="apply", geom="layered", nx=128, ny=128, nz=128, nb=1, prec="c64", ghz=3.0),
        # A grid as a mesher leaves it: three different odd sizes, magnetic and lossy cells, PEC cells.
        dict(name="apply_ragged", kind="apply", geom="random", nx=149, ny=107, nz=83, nb=1, prec="c64", ghz=4.0),
        # The largest structure: an IC package of 37.7 million unknowns.
        dict(name="apply_package256", kind="apply", geom="package", nx=256, ny=256, nz=192, nb=1, prec="c64", ghz=10.0),
        # A frequency sweep's apply: eight systems that share one stripline geometry.
        dict(name="apply_sweep96x8", kind="apply", geom="stripline", nx=96, ny=96, nz=96, nb=8, prec="c64", ghz=2.0),
        # The double-precision apply of refinement residuals and of plain complex128 solves.
        dict(name="apply_c128_96", kind="apply", geom="stripline", nx=96, ny=96, nz=96, nb=1, prec="c128", ghz=6.0),
        # The solver of choice: COCG with Jacobi, single precision inside double-precision refinement.
        dict(name="solve_cocg128", kind="solve", geom="lossy", nx=128, ny=128, nz=128, nb=1, ghz=3.0, method="cocg",
             precision="mixed", precond="jacobi"),
        # The robust fallback: restarted flexible GMRES(30) with Jacobi.
        dict(name="solve_fgmres64", kind="solve", geom="random", nx=64, ny=64, nz=64, nb=1, ghz=6.0, method="fgmres",
             precision="mixed", precond="jacobi"),
        # A frequency sweep of a small part in one batched solve with the library's default method.
        dict(name="solve_sweep40x8", kind="solve", geom="random", nx=40, ny=36, nz=28, nb=8, ghz=5.0, method="bicgstab",
             precision="mixed", precond="none"),
        # Impedance matrices of a two-port at two frequencies, in double precision throughout.
        dict(name="ports_c128", kind="ports", geom="lossy", nx=48, ny=40, nz=32, nb=2, ghz=5.0, method="cocg",
             precision="c128", precond="jacobi"),
        # The layer the learned preconditioner spends most of its inference in: 16 -> 16 at 128^3.
        dict(name="conv_16_16_128", kind="conv", nx=128, ny=128, nz=128, cin=16, cout=16, relu=True),
        # Training at 64^3: the skip convolution's data and weight gradients.
        dict(name="conv_grad_32_16_64", kind="conv_grad", nx=64, ny=64, nz=64, cin=32, cout=16),
    ]


CONV_SHAPES = ((16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (64, 32), (32, 16))


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["apply"] * 6 + ["solve"] * 3 + ["ports"] + ["conv"] * 2 + ["conv_grad"])
    if kind == "apply":
        # 4e3 .. 1.2e7 cells times systems, any aspect ratio, odd sizes as often as even ones
        cells = math.exp(rng.uniform(math.log(4e3), math.log(1.2e7)))
        nb = rng.choice([1, 1, 1, 2, 3, 4, 8, 16])
        prec = rng.choice(["c64", "c64", "c64", "c128"])
        if prec == "c128":
            cells /= 4
        edge = max(8.0, cells / nb) ** (1 / 3)
        nx, ny, nz = (max(6, min(320, int(round(edge * math.exp(rng.uniform(-0.5, 0.5)))))) for _ in range(3))
        while nx * ny * nz * nb > 12_500_000:
            nz = max(6, nz * 3 // 4)
        return dict(kind=kind, geom=rng.choice(["cavity", "layered", "random", "package", "stripline"]), nx=nx, ny=ny,
                    nz=nz, nb=nb, prec=prec, ghz=round(rng.uniform(1.0, 20.0), 2))
    if kind in ("solve", "ports"):
        nx, ny, nz = (_log_int(rng, 16, 56) for _ in range(3))
        method, precision, precond = rng.choice([
            ("cocg", "mixed", "jacobi"), ("cocg", "mixed", "jacobi"), ("cocg", "c128", "jacobi"),
            ("fgmres", "mixed", "jacobi"), ("bicgstab", "mixed", "none")])
        geom = "random" if method in ("bicgstab", "fgmres") else rng.choice(["random", "lossy"])
        return dict(kind=kind, geom=geom, nx=nx, ny=ny, nz=nz, nb=rng.choice([1, 2, 4]) if kind == "solve" else 2,
                    ghz=round(rng.uniform(4.0, 8.0), 2), method=method, precision=precision, precond=precond)
    cin, cout = rng.choice(CONV_SHAPES)
    top = 128 if max(cin, cout) <= 32 else 64  # the wide layers are the network's coarse levels
    nx, ny, nz = (_log_int(rng, 16, top) for _ in range(3))
    if kind == "conv":
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, cin=cin, cout=cout, relu=rng.random() < 0.7)
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, cin=cin, cout=cout)


# ---- geometries ---------------------------------------------------------------------------------------


def _absorber(nx, ny, nz, h, depth=8):
    """Graded conductivity next to all six walls (quadratic profile, reflection 1e-6)."""
    depth = max(1, min(depth, min(nx, ny, nz) // 4))
    smax = -3.0 * math.log(1e-6) / (2.0 * ETA0 * depth * h)

    def layer(n):
        i = np.arange(n)
        d = depth - 1 - np.minimum(i, n - 1 - i)
        return np.where(d >= 0, d, -1)

    d = np.maximum(np.maximum(layer(nz)[:, None, None], layer(ny)[None, :, None]), layer(nx)[None, None, :])
    return np.where(d >= 0, smax * ((d + 0.5) / depth) ** 2, 0.0).astype(np.float32)


def _geometry(case, seed):
    """Cell widths and per-cell materials (arrays [nz, ny, nx]) of the case's structure."""
    rng = np.random.Generator(np.random.PCG64(seed))
    nx, ny, nz, geom = case["nx"], case["ny"], case["nz"], case["geom"]
    shape = (nz, ny, nx)
    eps, sig, imu = np.ones(shape, np.float32), np.zeros(shape, np.float32), np.ones(shape, np.float32)
    pec = np.zeros(shape, np.uint8)
    h = {"cavity": 1e-3, "stripline": 0.5e-3, "package": 0.1e-3}.get(geom, 1e-3)
    dx, dy, dz = (np.full(n, h) for n in (nx, ny, nz))

    def layers(count, choices):
        for z in np.array_split(np.arange(nz), min(count, nz)):
            eps[z] = rng.choice(np.array(choices, np.float32))

    if geom in ("layered", "lossy"):
        dx, dy, dz = (rng.uniform(0.8e-3, 1.2e-3, n) for n in (nx, ny, nz))
        layers(8, (1.0, 2.2, 3.5, 4.4, 9.8))
        sig[:] = _absorber(nx, ny, nz, h)
        if geom == "layered":  # conductor blocks inside the absorber-free interior
            for _ in range(20):
                size = [int(rng.integers(2, max(3, n // 8) + 1)) for n in (nz, ny, nx)]
                at = [int(rng.integers(n // 8, max(n // 8 + 1, n - n // 8 - s))) for n, s in zip((nz, ny, nx), size)]
                sig[at[0]:at[0] + size[0], at[1]:at[1] + size[1], at[2]:at[2] + size[2]] = 5.8e7
        else:  # every layer a lossy dielectric
            for z in np.array_split(np.arange(nz), min(8, nz)):
                sig[z] = np.maximum(sig[z], np.float32(rng.uniform(0.2, 2.0)))
    elif geom == "stripline":  # two ground planes, two strips at different heights, no losses
        layers(4, (3.0, 4.4))
        pec[0] = pec[-1] = 1
        yc, m = ny // 2, max(1, nx // 12)
        for k in (3 * nz // 8, 5 * nz // 8):
            pec[k, max(0, yc - 3):yc + 3, m:max(m + 1, nx - m)] = 1
    elif geom == "package":  # traces along x or y on the layers' top planes, vias between layers
        nl = min(6, nz)
        layers(nl, (3.5, 4.4, 11.9))
        sig[:] = _absorber(nx, ny, nz, h)
        lz = nz // nl
        for t in range(max(4, 400 * nx * ny // 65536)):
            k = (t % nl) * lz + lz - 1
            length = int(rng.integers(max(2, nx // 16), max(4, nx // 2)))
            x0, y0 = int(rng.integers(0, nx)), int(rng.integers(0, ny))
            if rng.integers(0, 2):
                pec[k, y0:y0 + 2, x0:x0 + length] = 1
            else:
                pec[k, y0:y0 + length, x0:x0 + 2] = 1
            if t % 2:
                pec[max(0, k - lz):k + 1, y0, x0] = 1
    elif geom == "random":
        dx, dy, dz = (rng.uniform(0.5e-3, 1.5e-3, n) for n in (nx, ny, nz))
        eps = rng.uniform(1.0, 10.0, shape).astype(np.float32)
        sig = rng.uniform(0.0, 5.0, shape).astype(np.float32)
        imu = rng.uniform(0.5, 1.5, shape).astype(np.float32)
        pec = (rng.random(shape) < 0.03).astype(np.uint8)
    return dict(dx=dx, dy=dy, dz=dz, eps=eps, sig=sig, imu=imu, pec=pec)


def _omega(case):
    return 2.0 * math.pi * 1e9 * case["ghz"] * (1.0 + 0.08 * np.arange(case["nb"]))


def _masked(m):
    """uint8 [nz, ny, nx, 3]: edges in a low wall plane or touching a PEC cell."""
    p = np.pad(m["pec"], ((1, 0), (1, 0), (1, 0)))
    out = np.empty(m["pec"].shape + (3,), np.uint8)
    out[..., 0] = p[1:, 1:, 1:] | p[1:, :-1, 1:] | p[:-1, 1:, 1:] | p[:-1, :-1, 1:]
    out[..., 1] = p[1:, 1:, 1:] | p[1:, 1:, :-1] | p[:-1, 1:, 1:] | p[:-1, 1:, :-1]
    out[..., 2] = p[1:, 1:, 1:] | p[1:, 1:, :-1] | p[1:, :-1, 1:] | p[1:, :-1, :-1]
    out[0, :, :, 0] = out[:, 0, :, 0] = 1
    out[0, :, :, 1] = out[:, :, 0, 1] = 1
    out[:, 0, :, 2] = out[:, :, 0, 2] = 1
    return out


def _sources(case, m, seed):
    """[nb, n_e] right-hand sides -j w j of 64 impressed edge currents each (complex128, host)."""
    rng = np.random.Generator(np.random.PCG64(seed + 1))
    free = np.flatnonzero(_masked(m).reshape(-1) == 0)
    b = np.zeros((case["nb"], 3 * case["nx"] * case["ny"] * case["nz"]), np.complex128)
    for f, w in enumerate(_omega(case)):
        at = rng.choice(free, min(64, free.size), replace=False)
        b[f, at] = -1j * w * (rng.standard_normal(at.size) + 1j * rng.standard_normal(at.size)) / math.sqrt(2.0)
    return b


def _ports(case):
    """Two columns of z-edges at different places, one cell away from the walls and further."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]

    def column(i, j, k0, k1):
        return [3 * (i + nx * (j + ny * k)) + 2 for k in range(k0, k1)], [1.0] * (k1 - k0)

    return [column(nx // 3, ny // 3, nz // 4, nz // 4 + 3), column(2 * nx // 3, ny // 2, nz // 3, nz // 3 + 4)]


# ---- inputs and passes --------------------------------------------------------------------------------


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _apply_input(case, seed):
    dt = torch.complex64 if case["prec"] == "c64" else torch.complex128
    return torch.randn(case["nb"], 3 * case["nx"] * case["ny"] * case["nz"], dtype=dt, device="cuda", generator=_gen(seed))


def _conv_inputs(case, seed):
    g = _gen(seed)
    n = case["nx"] * case["ny"] * case["nz"]
    cin, cout = case["cin"], case["cout"]
    w = torch.randn(27, cout, cin, device="cuda", generator=g) * math.sqrt(2.0 / (27 * cin))
    x = torch.randn(n, cin, device="cuda", generator=g).relu_().to(torch.bfloat16)  # a ReLU layer's output
    bias = torch.randn(cout, device="cuda", generator=g) * 0.1
    dout = torch.randn(n, cout, device="cuda", generator=g).to(torch.bfloat16)
    return x, w, bias, dout


def prepare(case, seed):
    s = dict(case=case)
    if case["kind"] in ("conv", "conv_grad"):
        x, w, bias, dout = _conv_inputs(case, seed)
        s.update(x=x, w=w, bias=bias, dout=dout)
        if case["kind"] == "conv":
            s["out"] = torch.empty_like(dout)
        else:
            s.update(din=torch.empty_like(x), dw=torch.empty_like(w), db=torch.empty_like(bias))
        return s
    m = _geometry(case, seed)
    g = fit.Grid(case["nx"], case["ny"], case["nz"], m["dx"], m["dy"], m["dz"])
    fit.fit_set_materials(g.h, m["eps"], m["sig"], m["imu"], m["pec"])
    s.update(grid=g, omega=_omega(case))
    if case["kind"] == "apply":
        s["x"] = _apply_input(case, seed)
        s["y"] = torch.empty_like(s["x"])
    elif case["kind"] == "solve":
        s["b"] = torch.from_numpy(_sources(case, m, seed)).cuda()
        s["x"] = torch.empty_like(s["b"])
    else:
        s["ports"] = _ports(case)
    return s


def _solver(case):
    return dict(method=dict(bicgstab=fit.FIT_BICGSTAB, fgmres=fit.FIT_FGMRES, cocg=fit.FIT_COCG)[case["method"]],
                precision=dict(mixed=fit.FIT_SOLVE_MIXED, c128=fit.FIT_SOLVE_C128)[case["precision"]],
                precond=dict(none=fit.FIT_PC_NONE, jacobi=fit.FIT_PC_JACOBI)[case["precond"]],
                max_iter=60000, max_outer=2000)


TOL = 1e-10  # relative residual of the solves


def run(s):
    case = s["case"]
    if case["kind"] == "apply":
        s["grid"].apply(s["omega"], s["x"], s["y"], fit.FIT_C64 if case["prec"] == "c64" else fit.FIT_C128)
        return s["y"]
    if case["kind"] == "solve":
        s["grid"].solve(s["omega"], s["b"], s["x"], TOL, **_solver(case))
        return s["x"]
    if case["kind"] == "ports":
        _, z, _ = fit.fit_z_parameters(s["grid"].h, s["omega"], s["ports"], TOL, **_solver(case))
        return z
    dims = case["nx"], case["ny"], case["nz"], case["cin"], case["cout"]
    if case["kind"] == "conv":
        fit.fit_unet_conv3(*dims, s["x"], s["w"], s["bias"], case["relu"], s["out"])
        return s["out"]
    fit.fit_unet_conv3_dgrad(*dims, s["dout"], s["w"], s["din"])
    fit.fit_unet_conv3_wgrad(*dims, s["x"], s["dout"], s["dw"], s["db"])
    return dict(din=s["din"], dw=s["dw"], db=s["db"])


def work(case):
    """Bytes and operations of one pass: inputs read once, outputs written once; a solve moves, per
    iteration, its operator's coefficients and its recurrence's vectors once."""
    cells = case["nx"] * case["ny"] * case["nz"]
    ne = 3 * cells
    if case["kind"] == "apply":
        value, coef = (8, 4) if case["prec"] == "c64" else (16, 8)
        return dict(bytes=ne * (2 * value * case["nb"] + 3 * coef), flops=90.0 * cells * case["nb"])
    if case["kind"] in ("solve", "ports"):
        value, coef = (8, 4) if case["precision"] == "mixed" else (16, 8)
        systems = case["nb"] * (2 if case["kind"] == "ports" else 1)
        its = 12.0 * cells ** (1 / 3) * (2 if case["method"] == "fgmres" else 1)  # about what these grids take
        # COCG: r, p, d read and written, D^-1 read; BiCGStab: two applies, r, p, v, d; FGMRES(30): w and
        # on average 15 basis vectors
        vectors = dict(cocg=7, bicgstab=12, fgmres=18)[case["method"]]
        return dict(bytes=its * ne * (vectors * value * systems + 3 * coef), flops=its * systems * ne * (30 + 8.0 * vectors))
    taps = 2.0 * 27 * case["cin"] * case["cout"]
    weights = 4 * 27 * case["cin"] * case["cout"]
    if case["kind"] == "conv":
        return dict(bytes=2 * cells * (case["cin"] + case["cout"]) + weights, flops=taps * cells)
    return dict(bytes=4 * cells * (case["cin"] + case["cout"]) + 2 * weights, flops=2 * taps * cells)


# ---- the same results in 64 bits ----------------------------------------------------------------------


class _Operator:
    """y = C^T M_nu C x - w^2 M_eps x + j w M_kappa x on the unmasked edges, y = x on the others."""

    def __init__(self, m):
        dx, dy, dz = (torch.from_numpy(m[k]).cuda() for k in ("dx", "dy", "dz"))
        eps, sig, imu = (torch.from_numpy(m[k]).cuda().double() for k in ("eps", "sig", "imu"))
        wx, wy, wz = dx[None, None, :], dy[None, :, None], dz[:, None, None]

        def low(t, axis):  # the value of the neighbour below, zero beyond the wall
            return torch.cat([torch.zeros_like(t.narrow(axis, 0, 1)), t.narrow(axis, 0, t.shape[axis] - 1)], axis)

        def over(t, a, b, area):  # sum of the four cells around an edge, each with a quarter of its area
            q = 0.25 * t * area
            q = q + low(q, a)
            return q + low(q, b)

        def edges(t):
            return torch.stack([over(t, 1, 0, wy * wz) / wx, over(t, 2, 0, wx * wz) / wy, over(t, 2, 1, wx * wy) / wz], -1)

        def facet(axis, width, area):
            half = 0.5 * width * imu
            return (half + low(half, axis)) / (MU0 * area)

        self.me, self.mk = EPS0 * edges(eps), edges(sig)
        self.nu = torch.stack([facet(2, wx, wy * wz), facet(1, wy, wx * wz), facet(0, wz, wx * wy)], -1)
        self.mask = torch.from_numpy(_masked(m)).cuda().bool()
        self.shape = self.me.shape

    def diagonal(self, w):
        def low(t, axis):
            return torch.cat([torch.zeros_like(t.narrow(axis, 0, 1)), t.narrow(axis, 0, t.shape[axis] - 1)], axis)

        nx, ny, nz = self.nu.unbind(-1)
        s = torch.stack([ny + low(ny, 0) + nz + low(nz, 1), nx + low(nx, 0) + nz + low(nz, 2),
                         nx + low(nx, 1) + ny + low(ny, 2)], -1)
        return torch.where(self.mask, torch.ones_like(s) + 0j, torch.complex(s - w * w * self.me, w * self.mk)).reshape(-1)

    def __call__(self, w, x):
        x = x.reshape(self.shape)
        e = x.masked_fill(self.mask, 0)

        def up(t, axis):
            return torch.cat([t.narrow(axis, 1, t.shape[axis] - 1), torch.zeros_like(t.narrow(axis, 0, 1))], axis)

        def low(t, axis):
            return torch.cat([torch.zeros_like(t.narrow(axis, 0, 1)), t.narrow(axis, 0, t.shape[axis] - 1)], axis)

        ex, ey, ez = e.unbind(-1)
        hx = self.nu[..., 0] * (ey - up(ey, 0) + up(ez, 1) - ez)
        hy = self.nu[..., 1] * (ez - up(ez, 2) + up(ex, 0) - ex)
        hz = self.nu[..., 2] * (ex - up(ex, 1) + up(ey, 2) - ey)
        y = torch.stack([low(hy, 0) - hy + hz - low(hz, 1), low(hz, 2) - hz + hx - low(hx, 0),
                         low(hx, 1) - hx + hy - low(hy, 2)], -1)
        y += torch.complex(-w * w * self.me, w * self.mk) * e
        return torch.where(self.mask, x, y).reshape(-1)

    def solve(self, w, b):
        """COCG with the diagonal, restarted from the true residual until that is at 1e-13."""
        dinv = 1.0 / self.diagonal(w)
        x, nb = torch.zeros_like(b), float(torch.linalg.vector_norm(b))
        for _ in range(6):
            r = b - self(w, x)
            if float(torch.linalg.vector_norm(r)) <= 1e-13 * nb:
                break
            p = dinv * r
            rho = (r * p).sum()
            for it in range(20000):
                q = self(w, p)
                alpha = rho / (p * q).sum()
                x += alpha * p
                r -= alpha * q
                if it % 20 == 19 and float(torch.linalg.vector_norm(r)) <= 3e-14 * nb:
                    break
                z = dinv * r
                new = (r * z).sum()
                p = z + (new / rho) * p
                rho = new
        return x


def exact(case, seed):
    if case["kind"] in ("conv", "conv_grad"):
        return _exact_conv(case, seed)
    m = _geometry(case, seed)
    a = _Operator(m)
    omega = [float(w) for w in _omega(case)]
    if case["kind"] == "apply":
        x = _apply_input(case, seed)
        return torch.stack([a(w, x[f].to(torch.complex128)) for f, w in enumerate(omega)])
    if case["kind"] == "solve":
        b = torch.from_numpy(_sources(case, m, seed)).cuda()
        return torch.stack([a.solve(w, b[f]) for f, w in enumerate(omega)])
    ports = [torch.tensor(edges, device="cuda") for edges, _ in _ports(case)]
    z = np.zeros((len(omega), len(ports), len(ports)), np.complex128)
    for f, w in enumerate(omega):
        for j, pj in enumerate(ports):
            b = torch.zeros(a.mask.numel(), dtype=torch.complex128, device="cuda")
            b[pj] = -1j * w
            x = a.solve(w, b.masked_fill(a.mask.reshape(-1), 0))
            for i, pi in enumerate(ports):
                z[f, i, j] = complex(-x[pi].sum())
    return z


def _exact_conv(case, seed):
    x, w, bias, dout = _conv_inputs(case, seed)
    nx, ny, nz, cin, cout = case["nx"], case["ny"], case["nz"], case["cin"], case["cout"]
    w = w.to(torch.bfloat16).double()  # the layer's weights enter as their bf16 rounding

    def haloed(t):
        return torch.nn.functional.pad(t.double().reshape(nz, ny, nx, -1), (0, 0, 1, 1, 1, 1, 1, 1))

    def window(t, dz, dy, dx):
        return t[dz:dz + nz, dy:dy + ny, dx:dx + nx].reshape(nx * ny * nz, -1)

    taps = [(t // 9, (t // 3) % 3, t % 3) for t in range(27)]
    if case["kind"] == "conv":
        xp = haloed(x)
        y = bias.double().repeat(nx * ny * nz, 1)
        for t, tap in enumerate(taps):
            y.addmm_(window(xp, *tap), w[t].t())
        return y.relu_() if case["relu"] else y
    xp, dp = haloed(x), haloed(dout)
    din = torch.zeros(nx * ny * nz, cin, dtype=torch.float64, device="cuda")
    dw = torch.empty(27, cout, cin, dtype=torch.float64, device="cuda")
    for t, (dz, dy, dx) in enumerate(taps):
        din.addmm_(window(dp, 2 - dz, 2 - dy, 2 - dx), w[t])
        dw[t] = dout.double().t() @ window(xp, dz, dy, dx)
    return dict(din=din, dw=dw, db=dout.double().sum(0))
