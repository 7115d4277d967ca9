"""Performance cases of the library: calls that users make, over the sizes they make them at.

Every case is one call of the public binding (paper_2606_06247_gb300.binding) on device tensors: the line and
plane operators, the divergence, the projection, the pressure solve and the time step, in the three precisions,
on channels (x periodic), boxes (walls all round) and 3D channels.  The sizes are those of the repository's
workloads (64^2 channel, 161^2 dipole box, 256^2 cavity batch, 512^2 serving slots, 4096 lines of 512, planes of
1024^2, 64^3 channel) and odd ones between them.

A case is a dict: kind, nx, ny, nz (1: 2D), walls (1: x has walls too), batch, cont (continuation points), family,
prec, and per kind: ops ("DX+DY"), refine, scheme, steps, slots (instances in use of a serving batch), lid, tuned.
"""
import decimal
import functools
import math

import numpy as np
import torch

from paper_2606_06247_gb300 import binding

D = 5           # matching points per wall
H_OVER_DX = 1.3  # smoothing length of every workload
LINE_MODES = 32  # modes of the band-limited line and plane inputs
RK3 = ((8 / 15, 8 / 15, 0.0), (2 / 15, 5 / 12, -17 / 60), (1 / 3, 3 / 4, -5 / 12))  # (a, g, z) of each substep
FOP = ((1.0, 1.0, 0.0),)


def _case(name, kind, nx, ny, nz=1, walls=0, batch=1, cont=25, family="G4", prec="f64", **more):
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, walls=walls, batch=batch, cont=cont, family=family, prec=prec, **more)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: wall-normal derivatives of one 64^2 field, where launch and latency are all there is
        _case("lines64_f64", "line_op", 64, 64, ops="W+DY+LAP"),
        # the line microbenchmark at the default continuation (extended length 537 = 3 * 179: chirp-z)
        _case("lines512_f32", "line_op", 4096, 512, prec="f32", ops="DY+LAP"),
        # the plane microbenchmark: first derivatives and Laplacian of a batch of large periodic planes
        _case("planes1024_f32", "spectral_op", 1024, 1024, batch=64, cont=26, prec="f32", ops="DX+DY+LAP"),
        # post-processing of a walled box in double precision (the dipole's odd size; extended length 186 = 2 * 3 * 31)
        _case("box161_ops_f64", "spectral_op", 161, 161, walls=1, batch=8, ops="W+DX+DY+LAP"),
        # divergence check of a batch of cavity velocities (extended length 281: prime)
        _case("box256_div_f32x2", "spectral_div", 256, 256, walls=1, batch=32, family="G8", prec="f32x2"),
        # projection of a ragged channel batch on the extended grid
        _case("channel_project_f32x2", "spectral_project", 200, 127, batch=12, prec="f32x2"),
        # pressure solves: the cavity batch in FP32 pairs, and a large channel in FP32 with one FP64-residual sweep
        _case("ppe_box256_f32x2", "ppe_solve", 256, 256, walls=1, batch=32, family="G8", prec="f32x2"),
        _case("ppe_channel512_f32", "ppe_solve", 512, 512, batch=4, prec="f32", refine=1),
        # one small solve: ten first-order projection steps of the 64^2 channel in double precision
        _case("step_channel64_f64", "step", 64, 64, scheme="fop", steps=10),
        # the headline batch: one RK3 step of 32 lid cavities of 256^2 in FP32 pairs, launch shape autotuned
        _case("step_cavity256_f32x2", "step", 256, 256, walls=1, batch=32, family="G8", prec="f32x2", scheme="rk3", steps=1,
              lid=1.0, tuned=True),
        # serving: a size class of 8 slots, 5 of them in use, per-slot viscosity and time step
        _case("step_slots512_f32x2", "step", 512, 512, walls=1, batch=8, cont=28, family="G8", prec="f32x2", scheme="rk3", steps=1,
              slots=5),
        # 3D channel requests: two 64^3 channels (extended length 90)
        _case("step_channel3d64_f32x2", "step", 64, 64, nz=64, batch=2, cont=26, prec="f32x2", scheme="rk3", steps=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# Instances of a drawn case: at most this many nodes in all, which keeps it below the largest listed case.
_NODES = {("line_op", "f32"): 1 << 23, ("spectral_op", "f32"): 1 << 24, ("ppe_solve", "f32"): 1 << 21, ("step", "f64"): 1 << 16,
          ("step", "f32x2"): 1 << 20}


def draw(rng):
    kind = rng.choice(["line_op", "spectral_op", "spectral_op", "spectral_div", "spectral_project", "ppe_solve", "step", "step"])
    prec = rng.choice(["f64", "f32x2"] if kind in ("spectral_div", "spectral_project", "step") else ["f64", "f32x2", "f32"])
    walls = rng.randint(0, 1) if prec != "f32" else 0  # FP32 on walled boxes is not at equal accuracy: users take pairs
    top = 1024 if prec == "f32" else 400
    ny = _log(rng, 40, top)
    nx = 2 * _log(rng, 20, top // 2) + rng.randint(0, 1)
    nodes = _NODES.get((kind, prec), 1 << 19)
    if kind == "line_op":
        nx, walls = _log(rng, 64, max(64, min(8192, nodes // ny))), 0
    batch = max(1, min(_log(rng, 1, 64), nodes // (nx * ny)))
    c = _case(None, kind, nx, ny, walls=walls, batch=batch, cont=rng.choice([25, 25, rng.randint(20, 32)]),
              family=rng.choice(["G4", "G8"]), prec=prec)
    if kind in ("line_op", "spectral_op"):
        names = ["W", "DY", "LAP"] + (["DX"] if kind == "spectral_op" else [])
        got = rng.sample(names, rng.randint(1, len(names)))
        c["ops"] = "+".join(o for o in ("W", "DX", "DY", "LAP") if o in got)
    elif kind == "ppe_solve" and prec == "f32":
        c["refine"] = rng.randint(0, 1)
    elif kind == "step":
        c["scheme"] = rng.choice(["fop", "rk3"])
        c["steps"] = rng.randint(1, 3) if nodes >= 8 * nx * ny * batch else 1
        if not walls and rng.random() < 0.3 and prec == "f32x2":
            n = rng.randint(24, 80)
            c.update(nx=n, ny=_log(rng, 40, 96), nz=rng.randint(24, 80), batch=rng.randint(1, 2))
    return c


# ---------------------------------------------------------------------------
# inputs

_DEV = "cuda" if torch.cuda.is_available() else "cpu"


def _lengths(c):
    """(lx, ly, lz): unit walls, an isotropic lattice."""
    dy = 1.0 / (c["ny"] - 1)
    return (c["nx"] - 1 if c["walls"] else c["nx"]) * dy, 1.0, c["nz"] * dy if c["nz"] > 1 else 0.0


def _gen(seed):
    g = torch.Generator(device=_DEV)
    g.manual_seed(seed)
    return g


def _axis(n, closed):
    return torch.arange(n, dtype=torch.float64, device=_DEV) / (n - 1 if closed else n)


def _fields(c, seed, count, modes=8):
    """`count` smooth fields [batch][nx](nz)[ny]: low trigonometric modes in x (and z), cosines times a polynomial in
    y; not periodic across the walls."""
    g = _gen(seed)
    B, nx, nz, ny = c["batch"], c["nx"], c["nz"], c["ny"]
    x, y, z = _axis(nx, c["walls"]), _axis(ny, True), _axis(nz, False)
    out = []
    for _ in range(count):
        rnd = lambda *s: torch.rand(s, generator=g, dtype=torch.float64, device=_DEV)  # noqa: E731
        kx = torch.floor(rnd(B, modes) * 6)
        ky = rnd(B, modes) * 6
        kz = torch.floor(rnd(B, modes) * 4) if nz > 1 else torch.zeros(B, modes, dtype=torch.float64, device=_DEV)
        if c["walls"]:
            kx = kx + rnd(B, modes)
        a = (2 * rnd(B, modes) - 1) / (1 + kx + ky)
        cx = torch.cos(2 * math.pi * (kx[..., None] * x + rnd(B, modes, 1)))
        cy = torch.cos(2 * math.pi * (ky[..., None] * y / 2 + rnd(B, modes, 1))) * a[..., None]
        if nz > 1:
            cz = torch.cos(2 * math.pi * (kz[..., None] * z + rnd(B, modes, 1)))
            f = torch.einsum("bmx,bmz,bmy->bxzy", cx, cz, cy)
        else:
            f = torch.einsum("bmx,bmy->bxy", cx, cy)
        out.append(f.contiguous())
    return out


def _banded(c, seed):
    """Band-limited lines or planes plus a degree-4 polynomial in y (the microbenchmarks' inputs)."""
    g = _gen(seed)
    B, nx, ny, m = c["batch"], c["nx"], c["ny"], LINE_MODES
    x, y = _axis(nx, c["walls"]), _axis(ny, True)
    powers = torch.stack([y ** i for i in range(5)])
    nrm = lambda *s: torch.randn(s, generator=g, dtype=torch.float64, device=_DEV)  # noqa: E731
    if c["kind"] == "line_op":
        k = torch.arange(1, m + 1, dtype=torch.float64, device=_DEV)
        t = 2 * math.pi * k[:, None] * y
        f = (nrm(B, nx, m) / k) @ torch.cos(t) + (nrm(B, nx, m) / k) @ torch.sin(t) + nrm(B, nx, 5) @ powers
    else:
        kx, ky = (torch.randint(0, m, (B, m), generator=g, device=_DEV).double() for _ in range(2))
        cx = torch.cos(2 * math.pi * (kx[..., None] * x + torch.rand((B, m, 1), generator=g, dtype=torch.float64, device=_DEV)))
        cy = torch.cos(2 * math.pi * ky[..., None] * y) * (nrm(B, m) / (1 + torch.hypot(kx, ky)))[..., None]
        f = cx.transpose(1, 2) @ cy + (nrm(B, 5) @ powers)[:, None, :]
    return f.contiguous()


def _velocity(c, seed):
    """Velocity components of a developed flow: smooth, no slip on the walls (the lid's speed on y = Ly)."""
    nc = 3 if c["nz"] > 1 else 2
    y = _axis(c["ny"], True)
    mask = (16 * (y * (1 - y)) ** 2)
    if c["walls"]:
        x = _axis(c["nx"], True)
        mask = (16 * (x * (1 - x)) ** 2)[:, None] * mask
    vel = [(0.3 * f * mask).contiguous() for f in _fields(c, seed, nc)]
    if c.get("lid"):
        vel[0][:, 1:-1, -1] = c["lid"]
    return vel


def _step_options(c, seed):
    """(keyword arguments of isph_step, the same as plain numbers for the check)."""
    B = c["batch"]
    force = (0.0, 0.0, 0.0) if c["walls"] else (0.08, 0.0, 0.0)
    dy = 1.0 / (c["ny"] - 1)
    nu = 1e-3 if c["walls"] else 1e-2
    dt = min(1e-3, 0.25 * dy * dy / nu)
    plain = dict(nu=[nu] * B, dt=[dt] * B, force=force, lid=c.get("lid", 0.0), active=[True] * B)
    kw = dict(nu=nu, dt=dt, force=force, u_top=c.get("lid", 0.0), scheme=c["scheme"])
    if "slots" in c:
        r = np.random.default_rng(seed)
        plain["nu"] = [float(v) for v in np.exp(r.uniform(math.log(2e-4), math.log(2e-3), B))]
        plain["dt"] = [min(1e-3, 0.25 * dy * dy / v) for v in plain["nu"]]
        used = r.permutation(B) < c["slots"]
        plain["active"] = [bool(v) for v in used]
        dev = lambda v, t: torch.tensor(v, dtype=t, device=_DEV)  # noqa: E731
        kw.update(nu_inst=dev(plain["nu"], torch.float64), dt_inst=dev(plain["dt"], torch.float64),
                  active=dev(plain["active"], torch.uint8))
    return kw, plain


def _inputs(c, seed):
    k = c["kind"]
    if k == "step":
        return _velocity(c, seed)
    if k in ("spectral_div", "spectral_project"):
        fs = _fields(c, seed, 2)
    elif k == "ppe_solve":
        fs = _fields(c, seed, 1)
    else:
        fs = [_banded(c, seed) if c["prec"] == "f32" else _fields(c, seed, 1)[0]] if k != "line_op" else [_banded(c, seed)]
    return [f.float() if c["prec"] == "f32" else f for f in fs]


_TUNED = {}  # launch shapes by case, as the autotuner's cache file keeps them


def prepare(case, seed):
    c = case
    lx, ly, lz = _lengths(c)
    ctx = binding.Context(c["nx"], c["ny"], lx, ly, x_walls=bool(c["walls"]), batch=c["batch"], n_match=D, n_cont=c["cont"],
                          family=c["family"], h_over_dx=H_OVER_DX, prec=c["prec"], refine=c.get("refine", 0), nz=c["nz"], lz=lz)
    s = dict(case=c, ctx=ctx, ins=_inputs(c, seed))
    like = s["ins"][0]
    if c["kind"] == "step":
        n = len(s["ins"])
        s["F"] = [torch.zeros_like(like) for _ in range(n)]
        s["p"] = torch.zeros_like(like)
        s["kw"], _ = _step_options(c, seed)
        if n == 3:
            s["kw"].update(w=s["ins"][2], fw=s["F"][2])
        if c.get("tuned"):
            key = str(sorted(c.items()))
            if key not in _TUNED:
                o = s["kw"]
                ctx.autotune(steps=2, nu=o["nu"], dt=o["dt"], u_top=o["u_top"], scheme=o["scheme"])
                _TUNED[key] = ctx.tune_state()
            ctx.apply_tune_state(_TUNED[key])
    else:
        s["outs"] = [torch.empty_like(like) for _ in range({"spectral_project": 2}.get(c["kind"], 1) if "ops" not in c
                                                           else len(c["ops"].split("+")))]
    return s


def run(state):
    s = state
    c, ctx, ins = s["case"], s["ctx"], s["ins"]
    k = c["kind"]
    if k == "line_op":
        ctx.line_op(ins[0], c["ops"].split("+"), s["outs"])
    elif k == "spectral_op":
        ctx.spectral_op(ins[0], c["ops"].split("+"), s["outs"])
    elif k == "spectral_div":
        ctx.spectral_div(ins[0], ins[1], s["outs"][0])
    elif k == "spectral_project":
        ctx.spectral_project(ins[0], ins[1], s["outs"][0], s["outs"][1])
    elif k == "ppe_solve":
        ctx.ppe_solve(ins[0], s["outs"][0])
    else:
        ctx.isph_step(ins[0], ins[1], s["p"], s["F"][0], s["F"][1], c["steps"], **s["kw"])
        return {"vel": list(ins), "p": s["p"], "F": list(s["F"])}
    return list(s["outs"])


# ---------------------------------------------------------------------------
# work


def work(case):
    """Fields read and written once, and 5 n log2 n flops per transformed complex line of n points (real lines in pairs)."""
    c = case
    nx, ny, nz, B = c["nx"], c["ny"], c["nz"], c["batch"]
    my, mx = ny + c["cont"], nx + (c["cont"] if c["walls"] else 0)
    hy, ncol = my // 2 + 1, nx * nz
    el = 4 if c["prec"] == "f32" else 8
    field = float(B) * ncol * ny * el
    fl = lambda n: 5.0 * n * math.log2(n)  # noqa: E731
    ycol, xrow = B * ncol / 2 * fl(my), B * hy * nz * fl(mx) + (B * hy * nx * fl(nz) if nz > 1 else 0.0)
    dct = B * ncol / 2 * fl(2 * (ny - 1))
    ppe = 2 * dct + B * ny * nz * fl(2 * (nx - 1) if c["walls"] else nx) + (B * ny * nx * fl(nz) if nz > 1 else 0.0)
    k = c["kind"]
    if k == "line_op":
        n = len(c["ops"].split("+"))
        return dict(bytes=(1 + n) * field, flops=(1 + n) * ycol)
    if k == "spectral_op":
        n = len(c["ops"].split("+"))
        return dict(bytes=(1 + n) * field, flops=(1 + n) * (ycol + xrow))
    if k == "spectral_div":
        return dict(bytes=3 * field, flops=3 * (ycol + xrow))
    if k == "spectral_project":
        return dict(bytes=4 * field, flops=4 * (ycol + xrow))
    if k == "ppe_solve":
        return dict(bytes=2 * field, flops=ppe * (1 + 3 * c.get("refine", 0)))
    nc = 3 if nz > 1 else 2
    share = c.get("slots", B) / B
    sub = (3 if c["scheme"] == "rk3" else 1) * c["steps"]
    lines = nc * (nc + 1) + 1 + nc + 2 * nc + 1  # inverse: gradients and Laplacians, div, grad; forward: u*, u, phi
    # velocity and F read and written, p written, per call; the transforms of every substep
    return dict(bytes=share * (4 * nc + 1) * field, flops=share * sub * (lines * (ycol + xrow) + ppe))


# ---------------------------------------------------------------------------
# the same results in plain 64-bit torch


@functools.lru_cache(maxsize=None)
def _gram_table(C):
    """FC(Gram) continuation table [C][2 D] to 60 digits, rounded to 64 bits: the degree D-1 polynomial of the wall
    data and zero, fitted by trigonometric modes of period T = 2 (2 D + C - 2), K = T // 4, 20 points per interval."""
    with decimal.localcontext() as ctx:
        ctx.prec = 60
        Dc = decimal.Decimal
        T, over = 2 * (2 * D + C - 2), 20
        K, per = T // 4, 20 * T
        # cos and sin of 2 pi j / per by rotation from Taylor values of the first angle
        pi = Dc("3.14159265358979323846264338327950288419716939937510582097494459230781640628620899862803482534211706798")
        th = 2 * pi / per
        s1 = c1 = Dc(0)
        term = Dc(1)
        for i in range(60):
            if i % 2 == 0:
                c1 += term if i % 4 == 0 else -term
            else:
                s1 += term if i % 4 == 1 else -term
            term = term * th / (i + 1)
        cs, sn = [Dc(1)], [Dc(0)]
        for _ in range(per - 1):
            a, b = cs[-1], sn[-1]
            cs.append(a * c1 - b * s1)
            sn.append(b * c1 + a * s1)

        def row(U):
            r = [Dc(1)]
            for k in range(1, K + 1):
                r += [cs[k * U % per], sn[k * U % per]]
            return r

        n1 = (D - 1) * over + 1
        A, B = [], []
        for i in range(2 * n1):
            U = i if i < n1 else over * (D + C) + i - n1
            A.append(row(U))
            b = [Dc(0)] * D
            if i < n1:
                u = Dc(U) / over
                for a in range(D):
                    v = Dc(1)
                    for q in range(D):
                        if q != a:
                            v = v * (u - q) / (a - q)
                    b[a] = v
            B.append(b)
        # least squares by modified Gram-Schmidt on [A | B]
        n = 2 * K + 1
        cols = [list(col) for col in zip(*A)] + [list(col) for col in zip(*B)]
        R = [[Dc(0)] * (n + D) for _ in range(n)]
        for j in range(n):
            q = cols[j]
            nrm = sum(v * v for v in q).sqrt()
            q = cols[j] = [v / nrm for v in q]
            R[j][j] = nrm
            for i in range(j + 1, n + D):
                w = cols[i]
                d = sum(x * y for x, y in zip(q, w))
                R[j][i] = d
                cols[i] = [y - d * x for x, y in zip(q, w)]
        X = [[Dc(0)] * D for _ in range(n)]
        for a in range(D):
            for i in range(n - 1, -1, -1):
                X[i][a] = (R[i][n + a] - sum(R[i][j] * X[j][a] for j in range(i + 1, n))) / R[i][i]
        Er = [[float(sum(p * X[j][a] for j, p in enumerate(row(over * (D + i))))) for a in range(D)] for i in range(C)]
    E = np.zeros((C, 2 * D))
    E[:, :D] = Er
    E[:, D:] = E[::-1, :D][:, ::-1]
    return E


class _Exact:
    """The method's operators on one grid in 64-bit torch: FC extension, FFT, symbols, inverse FFT, truncation."""

    def __init__(self, c):
        self.c = c
        self.d3 = c["nz"] > 1
        lx, ly, lz = _lengths(c)
        nx, ny, nz, C = c["nx"], c["ny"], c["nz"], c["cont"]
        self.E = torch.tensor(_gram_table(C), device=_DEV)
        self.my, self.mx = ny + C, nx + (C if c["walls"] else 0)
        dx, dy = (lx / (nx - 1) if c["walls"] else lx / nx), ly / (ny - 1)
        f64 = dict(dtype=torch.float64, device=_DEV)

        def freq(m, d):
            k = torch.arange(m, **f64)
            k = torch.where(2 * k > m, k - m, k)
            w = k * (2 * math.pi / (m * d))
            return w, torch.where(2 * k == m, torch.zeros_like(w), w)  # and without its Nyquist entry

        shape = lambda v, ax: v.reshape([-1 if a == ax else 1 for a in range(4 if self.d3 else 3)])  # noqa: E731
        kx, kx0 = (shape(v, 1) for v in freq(self.mx, dx))
        ky, ky0 = (shape(v[: self.my // 2 + 1], 3 if self.d3 else 2) for v in freq(self.my, dy))
        kz, kz0 = (shape(v, 2) for v in freq(nz, lz / nz)) if self.d3 else (torch.zeros_like(kx), torch.zeros_like(kx))
        self.h = H_OVER_DX * dx
        self.kx0, self.ky0 = kx0, ky0
        k2 = kx ** 2 + ky ** 2 + kz ** 2
        self.W = self.what(k2)
        self.sym = {"W": self.W + 0j, "DX": 1j * kx0 * self.W, "DY": 1j * ky0 * self.W, "DZ": 1j * kz0 * self.W, "LAP": -k2 * self.W + 0j}
        self.ky, self.kyl, self.kyl0 = ky, ky.flatten(), ky0.flatten()
        # pressure eigenvalues
        lam = lambda n, per, L: (torch.where(2 * torch.arange(n, **f64) > n, torch.arange(n, **f64) - n, torch.arange(n, **f64)) * 2 if per  # noqa: E731
                                 else torch.arange(n, **f64)) * math.pi / L
        l2 = shape(lam(nx, not c["walls"], lx), 1) ** 2 + shape(lam(ny, False, ly), 3 if self.d3 else 2) ** 2
        if self.d3:
            l2 = l2 + shape(lam(nz, True, lz), 2) ** 2
        self.lam2 = l2

    def what(self, k2):
        s = k2 * self.h ** 2 / 4
        t = torch.ones_like(s)
        tot = torch.ones_like(s)
        for m in range(1, {"G2": 1, "G4": 2, "G6": 3, "G8": 4, "G10": 5}[self.c["family"]]):
            t = t * s / m
            tot = tot + t
        return torch.exp(-s) * tot

    def ext(self, f, dim):
        n = f.shape[dim]
        f = f.movedim(dim, -1)
        b = torch.cat([f[..., n - D:], f[..., :D]], -1)
        return torch.cat([f, b @ self.E.T.to(f.dtype)], -1).movedim(-1, dim)

    def fwd(self, f):
        F = torch.fft.rfft(self.ext(f, -1), dim=-1)
        if self.c["walls"]:
            F = self.ext(F, 1)
        return torch.fft.fftn(F, dim=(1, 2)) if self.d3 else torch.fft.fft(F, dim=1)

    def inv(self, F):
        F = torch.fft.ifftn(F, dim=(1, 2)) if self.d3 else torch.fft.ifft(F, dim=1)
        return torch.fft.irfft(F[:, : self.c["nx"]], n=self.my, dim=-1)[..., : self.c["ny"]].contiguous()

    def div(self, comps):
        return self.inv(sum(self.sym[o] * self.fwd(f) for o, f in zip(("DX", "DY") if not self.d3 else ("DX", "DY", "DZ"), comps)))

    def project(self, fx, fy):
        U, V = self.fwd(fx), self.fwd(fy)
        g2 = self.kx0 ** 2 + self.ky0 ** 2
        q = (self.kx0 * U + self.ky0 * V) / torch.where(g2 > 0, g2, torch.ones_like(g2))
        return [self.inv(U - self.kx0 * q), self.inv(V - self.ky0 * q)]

    def lines(self, f, ops):
        F = torch.fft.rfft(self.ext(f, -1), dim=-1)
        W = self.what(self.kyl ** 2)
        s = {"W": W + 0j, "DY": 1j * self.kyl0 * W, "LAP": -self.kyl ** 2 * W + 0j, "DX": 0j * W}
        return [torch.fft.irfft(F * s[o], n=self.my, dim=-1)[..., : self.c["ny"]].contiguous() for o in ops]

    def ppe(self, rhs):
        def dct(f, dim):  # sum with even extension: its own inverse up to 2 (n - 1)
            f = f.movedim(dim, -1)
            n = f.shape[-1]
            e = torch.cat([f, f[..., 1 : n - 1].flip(-1)], -1)
            r = torch.fft.fft(e, dim=-1)[..., :n]
            return (r if f.is_complex() else r.real).movedim(-1, dim)

        c = self.c
        B = dct(rhs, -1)
        per = (1, 2) if self.d3 else (1,)
        B = dct(B, 1) if c["walls"] else torch.fft.fftn(B, dim=per)
        l2 = self.lam2.clone()
        l2.view(-1)[0] = 1.0
        P = -B / l2
        P[(slice(None),) + (0,) * (P.dim() - 1)] = 0
        P = dct(P, 1) / (2 * (c["nx"] - 1)) if c["walls"] else torch.fft.ifftn(P, dim=per).real
        return (dct(P, -1) / (2 * (c["ny"] - 1))).contiguous()

    def step(self, vel, o):
        c = self.c
        nc = len(vel)
        ax = ("DX", "DY", "DZ")[:nc]
        col = lambda v: torch.tensor(v, dtype=torch.float64, device=_DEV).reshape([-1] + [1] * (vel[0].dim() - 1))  # noqa: E731
        nu, dt = col(o["nu"]), col(o["dt"])
        fr = [o["force"][0], o["force"][1], o["force"][2]]

        def walls(v, comp):
            v = v.clone()
            v[..., 0] = 0.0
            v[..., -1] = o["lid"] if comp == 0 else 0.0
            if c["walls"]:
                v[:, 0] = 0.0
                v[:, -1] = 0.0
            return v

        F = [torch.zeros_like(v) for v in vel]
        p = torch.zeros_like(vel[0])
        for _ in range(c["steps"]):
            for a, g, z in RK3 if c["scheme"] == "rk3" else FOP:
                star, new = [], []
                for q in range(nc):
                    S = self.fwd(vel[q])
                    n = sum(vel[t] * self.inv(self.sym[ax[t]] * S) for t in range(nc)) - nu * self.inv(self.sym["LAP"] * S)
                    star.append(walls(vel[q] + dt * (-g * n - z * F[q] + a * fr[q]), q))
                    new.append(n)
                F = new
                p = self.ppe(self.div(star) / (a * dt))
                P = self.fwd(p)
                vel = [walls(star[q] - a * dt * self.inv(self.sym[ax[q]] * P), q) for q in range(nc)]
        return vel, p, F


def exact(case, seed):
    c = case
    X = _Exact(c)
    ins = [f.double() for f in _inputs(c, seed)]
    k = c["kind"]
    if k == "line_op":
        return X.lines(ins[0], c["ops"].split("+"))
    if k == "spectral_op":
        F = [X.fwd(f) for f in ins[0].split(8)]
        return [torch.cat([X.inv(X.sym[o] * f) for f in F]) for o in c["ops"].split("+")]
    if k == "spectral_div":
        return [X.div(ins)]
    if k == "spectral_project":
        return X.project(*ins)
    if k == "ppe_solve":
        return [X.ppe(ins[0])]
    o = _step_options(c, seed)[1]
    vel, p, F = X.step(ins, o)
    on = torch.tensor(o["active"], device=_DEV).reshape([-1] + [1] * (p.dim() - 1))
    keep = lambda new, old: torch.where(on, new, old)  # noqa: E731  (empty slots are left as they were)
    zero = torch.zeros_like(p)
    return {"vel": [keep(v, u) for v, u in zip(vel, ins)], "p": keep(p, zero), "F": [keep(f, zero) for f in F]}
