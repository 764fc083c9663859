"""The work whose speed is measured: what users of the library have it do,
through its public entry points, at the sizes its configurations, tests and
benchmark name.

A case is a dict of plain values.  ``kind`` selects the program:

  run2d     initialise a 2D lattice, advance it, read the moments
  monitor   the same on a small lattice in short calls, the FP64 diagnostics
            read after each (a run that is watched while it goes)
  run3d     the 3D lattice (D3Q27 + D3Q7)
  ensemble  several lattices of uneven sizes advanced together (host fields
            in, host moments out, as that interface has it)
  adjoint   one training step: forward, loss, and the gradients of the
            initial fields, C_S and the relaxation times

Fields that a program hands over or reads back are device tensors except
where ``host`` says that they are numpy arrays.  ``exact`` restates the model
in plain 64-bit torch.
"""
import math

import numpy as np
import torch

from paper_1607_08675_gb300 import lbmhd as L
from paper_1607_08675_gb300.autograd import rollout

BYTES_OF = {"fp64": 8, "fp32": 4, "fp32_dev": 4, "fp16_dev": 2, "ff": 8}

# relaxation rates of the decaying-turbulence runs (tau = 0.51 needs the
# energy-flux and bulk moments damped harder than the tied rates)
TURB = dict(tau_nu=0.51, tau_eta=0.51, C_S=0.1, s5=1.2, s6=1.2, s7=1.3, s8=1.3)
VORTEX = dict(tau_nu=0.6, tau_eta=0.6, C_S=0.1)


def listed():
    return [
        # the smallest production run: the 64^2 Orszag-Tang vortex in FP64,
        # host arrays in and out, 200 steps (latency of small launches)
        dict(name="vortex64_fp64", kind="run2d", nx=64, ny=64, prec="fp64", les=1, flow="vortex",
             steps=200, host=True),
        # a small FP32 run watched closely: ten times 20 steps + diagnostics
        dict(name="monitor256_fp32", kind="monitor", nx=256, ny=256, prec="fp32", les=1,
             flow="turb", steps=20, reads=10),
        # the 1024^2 decaying-turbulence configuration in its two precisions
        dict(name="turb1024_fp32", kind="run2d", nx=1024, ny=1024, prec="fp32", les=1, flow="turb",
             steps=200, host=False),
        dict(name="turb1024_fp64", kind="run2d", nx=1024, ny=1024, prec="fp64", les=1, flow="turb",
             steps=60, host=False),
        # the headline lattice, FP32 and FP16-deviation storage
        dict(name="turb8192_fp32", kind="run2d", nx=8192, ny=8192, prec="fp32", les=1, flow="turb",
             steps=100, host=False),
        dict(name="turb8192_fp16", kind="run2d", nx=8192, ny=8192, prec="fp16_dev", les=1,
             flow="turb", steps=100, host=False),
        # odd sizes, FP32 deviations, no closure (direct simulation)
        dict(name="dns1999x1201_dev", kind="run2d", nx=1999, ny=1201, prec="fp32_dev", les=0,
             flow="vortex", steps=100, host=False),
        # the paper's own kinetic LES (filtered equilibria)
        dict(name="kinetic4096_fp32", kind="run2d", nx=4096, ny=4096, prec="fp32", les=2,
             flow="turb", steps=40, host=False),
        # 3D: local rates at the benchmark's size, and the kinetic LES at a
        # ragged one
        dict(name="cube256_fp32", kind="run3d", nx=256, ny=256, nz=256, prec="fp32", les=1,
             steps=30),
        dict(name="box200x168x144_kinetic", kind="run3d", nx=200, ny=168, nz=144, prec="fp32",
             les=2, steps=30),
        # a small ensemble of uneven lattices, 1000 steps, autotuned once
        dict(name="ensemble8_fp32", kind="ensemble", runs=8, smallest=128, sizes=3, prec="fp32",
             steps=1000),
        # the gradient configuration: 512^2 vortex, 500 steps, checkpoints
        # every 50
        dict(name="adjoint512_fp32", kind="adjoint", nx=512, ny=512, prec="fp32", steps=500,
             every=50),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run2d", "run2d", "run2d", "monitor", "run3d", "ensemble", "adjoint"])
    if kind in ("run2d", "monitor"):
        prec = rng.choice(["fp32", "fp32", "fp32_dev", "fp16_dev", "fp64", "ff"])
        les = rng.choice([0, 1, 1, 1, 2, 3])
        slow = {"fp64": 20.0, "ff": 4.0}.get(prec, 1.0)
        side = 8192 if kind == "run2d" else 512
        while True:
            nx, ny = _log_int(rng, 40, side), _log_int(rng, 40, side)
            if rng.random() < 0.5:  # half of them with aligned rows
                nx = max(40, nx // 8 * 8)
            steps = _log_int(rng, 5, 300)
            if nx * ny * steps * slow <= 3e9:
                break
        flow = "vortex" if les == 0 else rng.choice(["turb", "vortex"])
        case = dict(kind=kind, nx=nx, ny=ny, prec=prec, les=les, flow=flow, steps=steps)
        if kind == "monitor":
            return dict(case, steps=min(steps, 40), reads=rng.randint(2, 10))
        return dict(case, host=nx * ny < 40000 and rng.random() < 0.5)
    if kind == "run3d":
        prec = rng.choice(["fp32", "fp32", "fp16_dev", "ff", "fp64"])
        slow = {"fp64": 20.0, "ff": 8.0}.get(prec, 1.0)
        while True:
            nx, ny, nz = (_log_int(rng, 20, 320) for _ in range(3))
            steps = _log_int(rng, 4, 60)
            if nx * ny * nz * steps * slow <= 6e8:
                break
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, prec=prec, les=rng.choice([0, 1, 1, 2, 3]),
                    steps=steps)
    if kind == "ensemble":
        return dict(kind=kind, runs=rng.randint(4, 12), smallest=rng.choice([64, 96, 128]),
                    sizes=rng.choice([2, 3]), prec=rng.choice(["fp32", "fp32", "fp32_dev", "fp16_dev"]),
                    steps=_log_int(rng, 100, 1000))
    nx, ny = _log_int(rng, 96, 640), _log_int(rng, 96, 640)
    return dict(kind=kind, nx=nx, ny=ny, prec=rng.choice(["fp32", "fp32", "fp32_dev", "ff"]),
                steps=_log_int(rng, 60, 400), every=rng.choice([20, 50]))


# ---- inputs ---------------------------------------------------------------


def _params(case):
    p = dict(TURB if case.get("flow") == "turb" else VORTEX)
    if case["kind"] == "run3d":
        p = dict(tau_nu=0.55, tau_eta=0.55, C_S=0.1)
    p["les"] = case.get("les", 1)
    if p["les"] >= 2:  # the closures that filter take a filter width of two nodes
        p["delta"] = 2.0
    return p


def _curl(a):
    return (0.5 * (torch.roll(a, -1, 0) - torch.roll(a, 1, 0)),
            -0.5 * (torch.roll(a, -1, 1) - torch.roll(a, 1, 1)))


def _band2(nx, ny, gen):
    """Equal-amplitude random-phase modes 4 <= |n| <= 8 of a periodic field."""
    spec = torch.zeros(ny, nx // 2 + 1, dtype=torch.complex128)
    for my in range(-8, 9):
        for mx in range(0, 9):
            if (mx or my > 0) and 16 <= mx * mx + my * my <= 64:
                ph = torch.rand((), generator=gen, dtype=torch.float64).item() * 2 * math.pi
                spec[my % ny, mx] += complex(math.cos(ph), math.sin(ph))
    return torch.fft.irfft2(spec.cuda(), s=(ny, nx))


def _fields2(nx, ny, flow, seed):
    """(rho, ux, uy, bx, by), FP64 device tensors of shape (ny, nx)."""
    gen = torch.Generator().manual_seed(seed)
    if flow == "turb":
        out = []
        for _ in range(2):
            v = _curl(_band2(nx, ny, gen))
            s = 0.04 / torch.sqrt((v[0] ** 2 + v[1] ** 2).mean())
            out += [v[0] * s, v[1] * s]
        return [torch.ones_like(out[0]), *out]
    x = (torch.arange(nx, dtype=torch.float64, device="cuda") * (2 * math.pi / nx)).expand(ny, nx)
    y = (torch.arange(ny, dtype=torch.float64, device="cuda") * (2 * math.pi / ny))[:, None].expand(ny, nx)
    dev = torch.Generator("cuda").manual_seed(seed)
    noise = lambda: torch.rand(ny, nx, generator=dev, dtype=torch.float64, device="cuda") * 2 - 1
    db = _curl(noise())
    db = [c * (1e-4 / torch.sqrt(db[0] ** 2 + db[1] ** 2).max()) for c in db]
    out = [-0.05 * torch.sin(y) + 1e-4 * noise(), 0.05 * torch.sin(x) + 1e-4 * noise(),
           -0.05 * torch.sin(y) + db[0], 0.05 * torch.sin(2 * x) + db[1]]
    return [torch.ones_like(out[0]), *[t.contiguous() for t in out]]


def _fields3(nx, ny, nz, seed):
    """(rho, ux, uy, uz, bx, by, bz), FP64 device tensors of shape (nz, ny, nx)."""
    gen = torch.Generator().manual_seed(seed)
    d = lambda a, ax: 0.5 * (torch.roll(a, -1, ax) - torch.roll(a, 1, ax))
    out = []
    for _ in range(2):
        pot = []
        for _ in range(3):
            spec = torch.zeros(nz, ny, nx // 2 + 1, dtype=torch.complex128)
            for kz in range(-4, 5):
                for ky in range(-4, 5):
                    for kx in range(0, 5):
                        if 4 <= kx * kx + ky * ky + kz * kz <= 16:
                            ph = torch.rand((), generator=gen, dtype=torch.float64).item() * 2 * math.pi
                            spec[kz % nz, ky % ny, kx] += complex(math.cos(ph), math.sin(ph))
            pot.append(torch.fft.irfftn(spec.cuda(), s=(nz, ny, nx)))
        v = [d(pot[2], 1) - d(pot[1], 0), d(pot[0], 0) - d(pot[2], 2), d(pot[1], 2) - d(pot[0], 1)]
        s = 0.04 / torch.sqrt((v[0] ** 2 + v[1] ** 2 + v[2] ** 2).mean())
        out += [(c * s).contiguous() for c in v]
    return [torch.ones_like(out[0]), *out]


def _runs(case, seed):
    """Sizes and parameters of an ensemble's runs."""
    g = np.random.default_rng(1000 + case["runs"] * 7 + case["smallest"])  # sizes are the case's
    n = [case["smallest"] << int(k) for k in g.integers(0, case["sizes"], case["runs"])]
    n[0], n[-1] = case["smallest"], case["smallest"] << (case["sizes"] - 1)
    g = np.random.default_rng(seed)
    cs, tau = g.uniform(0.05, 0.2, len(n)), g.uniform(0.51, 0.7, len(n))
    return n, cs, tau


class _Held:
    """A handle that is destroyed with the state that holds it."""

    def __init__(self, h, destroy):
        self.h, self.destroy = h, destroy

    def __del__(self):
        self.destroy(self.h)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("run2d", "monitor"):
        fields = _fields2(case["nx"], case["ny"], case["flow"], seed)
        h = L.lbmhd_create(case["nx"], case["ny"], L.lbmhd_params_default(precision=case["prec"], **_params(case)))
        s["held"] = _Held(h, L.lbmhd_destroy)
        s["fields"] = [t.cpu().numpy() for t in fields] if case.get("host") else fields
        if kind == "run2d" and not case["host"]:
            s["out"] = [torch.empty_like(t) for t in fields]
    elif kind == "run3d":
        fields = _fields3(case["nx"], case["ny"], case["nz"], seed)
        h = L.lbmhd3_create(case["nx"], case["ny"], case["nz"],
                            L.lbmhd_params_default(precision=case["prec"], **_params(case)))
        s.update(held=_Held(h, L.lbmhd3_destroy), fields=fields, out=[torch.empty_like(t) for t in fields])
    elif kind == "ensemble":
        n, cs, tau = _runs(case, seed)
        rates = {k: TURB[k] for k in ("s5", "s6", "s7", "s8")}
        b = L.lbmhd_batch_create(n, n, tau, tau, cs, L.lbmhd_params_default(precision=case["prec"], **rates))
        L.lbmhd_batch_autotune(b, None, 8)
        s["held"] = _Held(b, L.lbmhd_batch_destroy)
        s["fields"] = [[t.cpu().numpy() for t in _fields2(m, m, "turb", seed + 31 * r)] for r, m in enumerate(n)]
    else:
        f = _fields2(case["nx"], case["ny"], "vortex", seed)
        s["leaves"] = [t.requires_grad_() for t in f]
        s["scalars"] = [torch.tensor(v, dtype=torch.float64, requires_grad=True) for v in (0.1, 0.6, 0.6)]
        s["target"] = [t.detach() * 0.9 for t in f[1:]]
    torch.cuda.synchronize()  # the library's stream does not wait for torch's
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "run2d":
        h = s["held"].h
        if case["host"]:
            L.lbmhd_init(h, *s["fields"])
            L.lbmhd_step(h, case["steps"])
            return {"moments": L.lbmhd_moments(h), "state": L.lbmhd_get_state(h)}
        L.lbmhd_init_device(h, *s["fields"])
        L.lbmhd_step(h, case["steps"])
        L.lbmhd_moments_device(h, *s["out"])
        return {"moments": s["out"]}
    if kind == "monitor":
        h = s["held"].h
        L.lbmhd_init_device(h, *s["fields"])
        rows = []
        for _ in range(case["reads"]):
            L.lbmhd_step(h, case["steps"])
            d = L.lbmhd_diagnostics(h)
            rows.append([d[k] for k in L.DIAG_KEYS])
        a = np.array(rows)
        return {"sums": a[:, :5], "means": a[:, 5:], "moments": L.lbmhd_moments(h)}
    if kind == "run3d":
        h = s["held"].h
        L.lbmhd3_init_device(h, *s["fields"])
        L.lbmhd3_step(h, case["steps"])
        L.lbmhd3_moments_device(h, *s["out"])
        return {"moments": s["out"]}
    if kind == "ensemble":
        b = s["held"].h
        for r, f in enumerate(s["fields"]):
            L.lbmhd_batch_init(b, r, *f)
        L.lbmhd_batch_step(b, case["steps"])
        return [L.lbmhd_batch_moments(b, r) for r in range(b.nruns)]
    out = rollout(*s["leaves"], *s["scalars"], case["steps"], case["every"], case["prec"])
    loss = 0.5 * sum(((a - t) ** 2).sum() for a, t in zip(out[1:], s["target"]))
    grads = torch.autograd.grad(loss, [*s["leaves"], *s["scalars"]])
    return {"loss": loss.detach(), "final": [t.detach() for t in out], "grads": grads}


# operations of one node update as the model states it: moments, relaxation
# and magnetic update (2D), with the local rates and the filters of the closures
_FLOPS2 = {0: 190, 1: 215, 2: 300, 3: 270}
_FLOPS3 = {0: 720, 1: 780, 2: 900, 3: 860}


def work(case):
    kind = case["kind"]
    if kind == "ensemble":
        n, _, _ = _runs(case, 0)
        nodes = sum(m * m for m in n)
        return {"bytes": 80 * nodes, "flops": nodes * case["steps"] * _FLOPS2[1]}
    if kind == "run3d":
        nodes = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 112 * nodes, "flops": nodes * case["steps"] * _FLOPS3[case["les"]]}
    nodes = case["nx"] * case["ny"]
    if kind == "adjoint":  # forward, and a reverse sweep of about twice its operations
        return {"bytes": 8 * 19 * nodes, "flops": nodes * case["steps"] * 3 * _FLOPS2[1]}
    steps = case["steps"] * case.get("reads", 1)
    out = 80 + (152 if case.get("host") else 0)
    return {"bytes": out * nodes, "flops": nodes * steps * _FLOPS2[case["les"]]}


# ---- the model in plain 64-bit torch ---------------------------------------

_C = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_W = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
_M = [[1, 1, 1, 1, 1, 1, 1, 1, 1], [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1],
      [0, 0, 0, 0, 0, 1, -1, 1, -1], [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, -2, 0, 2, 0, 1, -1, -1, 1],
      [0, 0, -2, 0, 2, 1, 1, -1, -1], [4, -5, -5, -5, -5, 4, 4, 4, 4], [4, 0, 0, 0, 0, -1, -1, -1, -1]]


def _start2(rho, ux, uy, bx, by):
    f = []
    for (cx, cy), w in zip(_C, _W):
        cu, cb = cx * ux + cy * uy, cx * bx + cy * by
        f.append(w * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + uy * uy))
                 + 4.5 * w * (0.5 * (bx * bx + by * by) * (cx * cx + cy * cy) - cb * cb))
    g = []
    for k, (cx, cy) in enumerate(_C[:5]):
        w = 1 / 6 if k else 1 / 3
        cu, cb = cx * ux + cy * uy, cx * bx + cy * by
        g += [w * (bx + 3 * (cu * bx - cb * ux)), w * (by + 3 * (cu * by - cb * uy))]
    return torch.stack(f), torch.stack(g)


def _step2(f, g, p, cs, tn, te):
    f = torch.stack([torch.roll(f[i], (c[1], c[0]), (0, 1)) for i, c in enumerate(_C)])
    g = torch.cat([torch.roll(g[2 * k:2 * k + 2], (c[1], c[0]), (1, 2)) for k, c in enumerate(_C[:5])])
    T = torch.tensor(_M, dtype=torch.float64, device=f.device)
    les, d2 = p["les"], p.get("delta", 1.0) ** 2
    m = torch.tensordot(T, f, 1)
    rho, jx, jy = m[0], m[1], m[2]
    bx, by = g[0::2].sum(0), g[1::2].sum(0)
    m3, m4, k7 = jx * jy / rho - bx * by, (jx * jx - jy * jy) / rho - bx * bx + by * by, 0.0
    e = (jx * by - jy * bx) / rho
    if les >= 2:
        dx = lambda a: 0.5 * (torch.roll(a, -1, 1) - torch.roll(a, 1, 1))
        dy = lambda a: 0.5 * (torch.roll(a, -1, 0) - torch.roll(a, 1, 0))
    if les == 2:
        fld = [rho, jx, jy, bx, by]
        gx, gy = [dx(a) for a in fld], [dy(a) for a in fld]
        dot = lambda a, b: gx[a] * gx[b] + gy[a] * gy[b]
        rat = lambda a, b: (dot(a, b) - (fld[a] * dot(0, b) + fld[b] * dot(0, a)
                                         - fld[a] * fld[b] * dot(0, 0) / rho) / rho) / (12 * rho)
        rxx, ryy = rat(1, 1), rat(2, 2)
        m3 = m3 + d2 * (rat(1, 2) - dot(3, 4) / 12)
        m4 = m4 + d2 * (rxx - ryy - (dot(3, 3) - dot(4, 4)) / 12)
        k7 = -3 * d2 * (rxx + ryy)
        e = e + d2 * (rat(1, 4) - rat(2, 3))
    j2 = (jx * jx + jy * jy) / rho
    n = [m[3] - m3, m[4] - m4, m[5] + jx, m[6] + jy, m[7] + 3 * j2 - k7, m[8] - (5 / 3 * rho - 3 * j2 + k7)]
    taue, taum = tn, te
    if les == 1:
        q = torch.sqrt(n[1] ** 2 + 4 * n[0] ** 2)
        jm = torch.abs(g[3] - g[7] - g[4] + g[8] - 2 * e)
        taue = 0.5 * (tn + torch.sqrt(tn * tn + 18 * cs * d2 * q / rho))
        taum = 0.5 * (te + torch.sqrt(te * te + 36 * cs * d2 * jm))
    if les == 3:
        ux, uy = jx / rho, jy / rho
        uxx, uxy, uyx, uyy = dx(ux), dy(ux), dx(uy), dy(uy)
        bxx, bxy, byx, byy = dx(bx), dy(bx), dx(by), dy(by)
        ss = uxx * bxx + uyy * byy + 0.5 * (uxy + uyx) * (bxy + byx)
        jw = (byx - bxy) * (uyx - uxy)
        taue = tn + 3 * cs * d2 * torch.sqrt(ss.abs())
        taum = torch.clamp(te + 3 * cs * d2 * torch.sign(jw) * torch.sqrt(jw.abs()), min=0.5)
    snu = 1 / taue
    r = [snu, snu, p.get("s5") or 1 / tn, p.get("s6") or 1 / tn, p.get("s7") or snu, p.get("s8") or snu]
    back = (T / (T * T).sum(1, keepdim=True)).t()[:, 3:].contiguous()
    f = f - torch.tensordot(back, torch.stack([a * b for a, b in zip(r, n)]), 1)
    eq = [bx / 3, by / 3, bx / 6, by / 6 + e / 2, bx / 6 - e / 2, by / 6, bx / 6, by / 6 - e / 2, bx / 6 + e / 2, by / 6]
    return f, g - (g - torch.stack(eq)) / taum


def _moments2(f, g):
    rho = f.sum(0)
    T = torch.tensor(_M[1:3], dtype=torch.float64, device=f.device)
    j = torch.tensordot(T, f, 1)
    return [rho, j[0] / rho, j[1] / rho, g[0::2].sum(0), g[1::2].sum(0)]


def _exact2(case, fields, p, steps):
    f, g = _start2(*fields)
    for _ in range(steps):
        f, g = _step2(f, g, p, p["C_S"], p["tau_nu"], p["tau_eta"])
    return f, g


def _diag(rho, ux, uy, bx, by):
    dx = lambda a: 0.5 * (torch.roll(a, -1, 1) - torch.roll(a, 1, 1))
    dy = lambda a: 0.5 * (torch.roll(a, -1, 0) - torch.roll(a, 1, 0))
    w, j, div = dx(uy) - dy(ux), dx(by) - dy(bx), dx(bx) + dy(by)
    sums = [rho.sum(), (rho * ux).sum(), (rho * uy).sum(), bx.sum(), by.sum()]
    means = [(rho * (ux * ux + uy * uy)).mean() / 2, (bx * bx + by * by).mean() / 2, (w * w).mean() / 2,
             (ux * bx + uy * by).mean(), div.abs().max(), torch.sqrt((div * div).mean()), (j * j).mean() / 2]
    return [float(v) for v in sums], [float(v) for v in means]


def _c3():
    v, w = (0, 1, -1), (2 / 3, 1 / 6, 1 / 6)
    c = [(v[i % 3], v[i // 3 % 3], v[i // 9]) for i in range(27)]
    return c, [w[i % 3] * w[i // 3 % 3] * w[i // 9] for i in range(27)]


_AXES = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]


def _geq3(u, b, extra=None):
    out = []
    for q in range(6):
        a, sg = q // 2, 1 - 2 * (q % 2)
        for k in range(3):
            t = u[a] * b[k] - b[a] * u[k]
            if extra is not None:
                t = t + extra[a][k]
            out.append((b[k] + 3 * sg * t) / 6)
    return out


def _exact3(case, fields, p, steps):
    """BGK on D3Q27 with the six-axis magnetic populations."""
    cs, ws = _c3()
    rho, u, b = fields[0], list(fields[1:4]), list(fields[4:7])
    dot = lambda x, y: x[0] * y[0] + x[1] * y[1] + x[2] * y[2]

    def feq(rho, u, b, R=None, P=None):
        uu, bb = dot(u, u), dot(b, b)
        trR = trP = 0.0
        if R is not None:
            trR, trP = R[0][0] + R[1][1] + R[2][2], P[0][0] + P[1][1] + P[2][2]
        for c, w in zip(cs, ws):
            ax = [a for a in range(3) if c[a]]
            cu = sum((c[a] * u[a] for a in ax), torch.zeros_like(rho))
            cb = sum((c[a] * b[a] for a in ax), torch.zeros_like(rho))
            t = rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu) + 4.5 * (bb * (0.5 * len(ax) - 1 / 6) - cb * cb)
            if R is not None:
                q = sum((c[a] * c[k] * (R[a][k] - P[a][k]) for a in ax for k in ax), torch.zeros_like(rho))
                t = t + 4.5 * q - 1.5 * trR + 4.5 * trP * (0.5 * len(ax) - 1 / 6)
            yield w * t

    f, g = list(feq(rho, u, b)), _geq3(u, b)
    d2, les, tn, te, C = p.get("delta", 1.0) ** 2, p["les"], p["tau_nu"], p["tau_eta"], p["C_S"]
    grad = lambda a: [0.5 * (torch.roll(a, -1, 2 - k) - torch.roll(a, 1, 2 - k)) for k in range(3)]
    for _ in range(steps):
        f = [torch.roll(x, (c[2], c[1], c[0]), (0, 1, 2)) for x, c in zip(f, cs)]
        g = [torch.roll(x, _AXES[i // 3][::-1], (0, 1, 2)) for i, x in enumerate(g)]
        rho = sum(f[1:], f[0].clone())
        j = [sum(x if c[a] > 0 else -x for x, c in zip(f, cs) if c[a]) for a in range(3)]
        b = [g[a] + g[3 + a] + g[6 + a] + g[9 + a] + g[12 + a] + g[15 + a] for a in range(3)]
        u = [x / rho for x in j]
        R = P = E = None
        taue, taum = tn, te
        if les == 2:
            gr, gj, gb = grad(rho), [grad(x) for x in j], [grad(x) for x in b]
            rt = lambda X, gX, Y, gY: d2 * (dot(gX, gY) - (X * dot(gr, gY) + Y * dot(gr, gX)
                                                           - X * Y * dot(gr, gr) / rho) / rho) / (12 * rho)
            R = [[rt(j[a], gj[a], j[k], gj[k]) for k in range(3)] for a in range(3)]
            P = [[d2 * dot(gb[a], gb[k]) / 12 for k in range(3)] for a in range(3)]
            X = [[rt(j[a], gj[a], b[k], gb[k]) for k in range(3)] for a in range(3)]
            E = [[X[a][k] - X[k][a] for k in range(3)] for a in range(3)]
        if les == 3:
            gu, gb = [grad(x) for x in u], [grad(x) for x in b]
            ss = sum(0.25 * (gu[a][k] + gu[k][a]) * (gb[a][k] + gb[k][a]) for a in range(3) for k in range(3))
            om = [gu[2][1] - gu[1][2], gu[0][2] - gu[2][0], gu[1][0] - gu[0][1]]
            jc = [gb[2][1] - gb[1][2], gb[0][2] - gb[2][0], gb[1][0] - gb[0][1]]
            jw = dot(om, jc)
            taue = tn + 3 * C * d2 * torch.sqrt(ss.abs())
            taum = torch.clamp(te + 3 * C * d2 * torch.sign(jw) * torch.sqrt(jw.abs()), min=0.5)
        if les == 1:
            bb, s = dot(b, b), {}
            for a in range(3):
                for k in range(a, 3):
                    s[a, k] = sum(x if c[a] * c[k] > 0 else -x for x, c in zip(f, cs) if c[a] * c[k]) \
                        - j[a] * u[k] + b[a] * b[k]
                s[a, a] = s[a, a] - rho / 3 - bb / 2
            tr = (s[0, 0] + s[1, 1] + s[2, 2]) / 3
            pp = sum((s[a, a] - tr) ** 2 for a in range(3)) + 2 * (s[0, 1] ** 2 + s[0, 2] ** 2 + s[1, 2] ** 2)
            n = lambda a, k: g[6 * a + k] - g[6 * a + 3 + k] - (u[a] * b[k] - b[a] * u[k])
            ax = [n(1, 2) - n(2, 1), n(2, 0) - n(0, 2), n(0, 1) - n(1, 0)]
            taue = 0.5 * (tn + torch.sqrt(tn * tn + 18 * C * d2 * torch.sqrt(2 * pp) / rho))
            taum = 0.5 * (te + torch.sqrt(te * te + 36 * C * d2 * torch.sqrt(dot(ax, ax))))
        f = [x - (x - q) / taue for x, q in zip(f, feq(rho, u, b, R, P))]
        g = [x - (x - q) / taum for x, q in zip(g, _geq3(u, b, E))]
    rho = sum(f[1:], f[0].clone())
    return [rho, *[sum(x if c[a] > 0 else -x for x, c in zip(f, cs) if c[a]) / rho for a in range(3)],
            *[sum(g[3 * q + a] for q in range(6)) for a in range(3)]]


def _exact_adjoint(case, fields, target):
    """Forward, loss and gradients by autograd over stretches of 10 steps."""
    p = dict(VORTEX, les=1)
    leaves = [t.clone().requires_grad_() for t in fields]
    th = [torch.tensor(p[k], dtype=torch.float64, device="cuda", requires_grad=True)
          for k in ("C_S", "tau_nu", "tau_eta")]

    def go(f, g, n):
        for _ in range(n):
            f, g = _step2(f, g, p, *th)
        return f, g

    cuts = [min(10, case["steps"] - i) for i in range(0, case["steps"], 10)]
    with torch.no_grad():
        kept = [_start2(*leaves)]
        for n in cuts:
            kept.append(go(*kept[-1], n))
    last = [t.detach().requires_grad_() for t in kept[-1]]
    out = _moments2(*last)
    loss = 0.5 * sum(((a - t) ** 2).sum() for a, t in zip(out[1:], target))
    lam = torch.autograd.grad(loss, last)
    dth = [torch.zeros_like(t) for t in th]
    for n, st in zip(reversed(cuts), reversed(kept[:-1])):
        st = [t.detach().requires_grad_() for t in st]
        res = torch.autograd.grad(go(*st, n), [*st, *th], lam)
        lam = res[:2]
        dth = [a + c for a, c in zip(dth, res[2:])]
    d0 = torch.autograd.grad(_start2(*leaves), leaves, lam)
    return {"loss": loss.detach(), "final": [t.detach() for t in out],
            "grads": (*d0, *[t.cpu() for t in dth])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "adjoint":
        f = _fields2(case["nx"], case["ny"], "vortex", seed)
        return _exact_adjoint(case, f, [t * 0.9 for t in f[1:]])
    with torch.no_grad():
        if kind == "ensemble":
            n, cs, tau = _runs(case, seed)
            if sum(n) * case["steps"] > 3.2e6:  # launch-bound here: too long
                return None
            out = []
            for r, m in enumerate(n):
                p = dict(TURB, les=1, C_S=float(cs[r]), tau_nu=float(tau[r]), tau_eta=float(tau[r]))
                out.append([t.cpu() for t in _moments2(*_exact2(case, _fields2(m, m, "turb", seed + 31 * r), p, case["steps"]))])
            return out
        p = _params(case)
        if kind == "run3d":
            fields = _fields3(case["nx"], case["ny"], case["nz"], seed)
            return {"moments": _exact3(case, fields, p, case["steps"])}
        fields = _fields2(case["nx"], case["ny"], case["flow"], seed)
        if kind == "monitor":
            f, g = _start2(*fields)
            sums, means = [], []
            for _ in range(case["reads"]):
                for _ in range(case["steps"]):
                    f, g = _step2(f, g, p, p["C_S"], p["tau_nu"], p["tau_eta"])
                a, b = _diag(*_moments2(f, g))
                sums.append(a)
                means.append(b)
            return {"sums": np.array(sums), "means": np.array(means), "moments": [t.cpu() for t in _moments2(f, g)]}
        f, g = _exact2(case, fields, p, case["steps"])
        out = {"moments": _moments2(f, g)}
        if case["host"]:
            out["moments"] = [t.cpu() for t in out["moments"]]
            out["state"] = torch.cat([f, g]).cpu()
        return out
