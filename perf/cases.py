"""Timed workloads of the solver: what its users call, over the range of sizes they call it with.

Every case goes through the ctypes binding (``paper_2502_06296_gb300.chanfs``) as a simulation code
or a serving program does: a plan (or a group, or a server) is made once and kept, right-hand sides
are new, and a pass is one call, or the few calls of one time step.  Sizes come from this
repository's benchmark and tests: the 32^3 box, the 512 x 384 x 384 channel, the 1024 x 768 x 512
precision run, the 3456 x 3072 x 30 box, the ensemble and serving menus, and ragged 2^a 3^b sizes
with odd plane counts.
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2502_06296_gb300 import chanfs

# lengths of the channel (12.8 x 6.4 x 2) unless a case names others
LX, LY = 12.8, 6.4
CHANNEL_C = 0.5 * (1.0 / 5200.0) * 1e-4  # alpha nu dt of the channel step


def listed():
    return [
        # the smallest call: one pressure solve of a test box; launches and latency
        dict(name="poisson_32", kind="poisson", nx=32, ny=32, nz=32, beta=0.0, bc=0, ybc=0),
        # the pressure solve of the channel step (the headline workload's first half)
        dict(name="poisson_channel", kind="poisson", nx=512, ny=384, nz=384, beta=1.8, bc=0, ybc=0),
        # the three implicit-diffusion solves of the channel step: u, v centred, w at faces
        dict(name="helmholtz_channel", kind="helmholtz", nx=512, ny=384, nz=384, beta=1.8,
             c=CHANNEL_C),
        # a pressure solve on a ragged grid: 3-smooth x and y, odd plane count, Dirichlet z walls
        dict(name="poisson_ragged", kind="poisson", nx=216, ny=162, nz=77, beta=1.5, bc=1, ybc=0),
        # a duct: walls in y as well (cosine transforms), medium size
        dict(name="poisson_ywalls", kind="poisson", nx=384, ny=256, nz=192, beta=1.6, bc=0, ybc=1),
        # the paper's per-GPU machine: long lines in x and y, few planes; the largest FP64 call (its
        # y tiles need the tuner's choice)
        dict(name="poisson_thin", kind="poisson", nx=3456, ny=3072, nz=30, beta=1.8, bc=0, ybc=0,
             tuned=True),
        # fully implicit diffusion (Eq. 8) on a medium channel, face-located velocity
        dict(name="helmholtz3d", kind="helmholtz3d", nx=256, ny=192, nz=192, beta=1.8, c=1e-4, loc=1),
        # transforms on their own, there and back, for spectra and filters
        dict(name="spectral", kind="spectral", nx=256, ny=256, nz=129, beta=0.0),
        # the pressure solve in FP32 with FP64 refinement, the precision workload
        dict(name="refined_large", kind="refined", nx=1024, ny=768, nz=512, beta=0.0, bc=0),
        # 16 boxes of the ensemble solved together: one grouped Poisson and one grouped Helmholtz
        dict(name="ensemble", kind="ensemble", boxes=16, seed0=2502064),
        # the channel step from and to pinned host memory, as a host-side code calls it
        dict(name="batch_host", kind="batch_host", nx=512, ny=384, nz=192, beta=1.8, c=CHANNEL_C),
        # a burst of requests from six runs through the server, one Poisson to three Helmholtz
        dict(name="serve_burst", kind="serve", runs=6, requests=24, seed0=2502065),
    ]


def _smooth(lo, hi, even):
    got = [2**a * 3**b for a in range(13) for b in range(8)]
    return sorted(n for n in got if lo <= n <= hi and (not even or n % 2 == 0))


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _near(rng, lo, hi, even=False, step=1):
    """A 2^a 3^b size, spread over the logarithm of [lo, hi]."""
    x = _log(rng, lo, hi)
    menu = [n for n in _smooth(lo, hi, even) if n % step == 0]
    return min(menu, key=lambda n: abs(math.log(n / x)))


def draw(rng: random.Random):
    kind = rng.choice(["poisson", "poisson", "helmholtz", "refined", "helmholtz3d", "ywalls", "spectral",
                       "ensemble", "serve", "batch_host"])
    if kind == "ensemble":
        return dict(kind=kind, boxes=rng.randint(2, 24), seed0=rng.randrange(1 << 30))
    if kind == "serve":
        return dict(kind=kind, runs=rng.randint(2, 8), requests=rng.randint(4, 32),
                    seed0=rng.randrange(1 << 30))
    most = 6e7 if kind != "batch_host" else 2.5e7
    while True:
        nx = _near(rng, 32, 1024, even=True, step=4 if kind == "refined" else 2)
        ny = _near(rng, 24, 768)
        nz = int(round(_log(rng, 16, 512)))
        if nx * ny * nz <= most:
            break
    case = dict(kind="poisson" if kind == "ywalls" else kind, nx=nx, ny=ny, nz=nz,
                beta=rng.choice([0.0, round(rng.uniform(1.2, 2.2), 3)]))
    if kind in ("poisson", "refined"):
        case.update(bc=rng.randint(0, 1))
    if kind == "poisson":
        case.update(ybc=0)
    if kind == "ywalls":
        case.update(bc=rng.randint(0, 1), ybc=rng.randint(1, 2))
    if kind in ("helmholtz", "helmholtz3d", "batch_host"):
        case.update(c=_log(rng, 1e-8, 1e-4))
    if kind == "helmholtz3d":
        case.update(loc=rng.randint(0, 1))
    return case


# --- inputs ------------------------------------------------------------------------------------


def _dz(nz, beta):
    """Cell widths on a channel of height 2: uniform (beta 0) or tanh-clustered at the walls."""
    if beta == 0.0:
        return np.full(nz, 2.0 / nz)
    k = np.arange(nz + 1, dtype=np.float64)
    return np.diff(np.tanh(beta * (2.0 * k / nz - 1.0)) / math.tanh(beta))


def _normal(seed, nz, ny, nx):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn((nz, ny, nx), generator=g, device="cuda", dtype=torch.float64)


def _rhs(case, seed, box=None):
    """N(0,1), less its volume-weighted mean where the walls leave the constants in the null space."""
    d = box or case
    f = _normal(seed, d["nz"], d["ny"], d["nx"])
    if d.get("bc", 0) == 0 and d.get("ybc", 0) != 2:
        w = torch.from_numpy(_dz(d["nz"], d["beta"])).cuda()
        f -= (f.mean(dim=(1, 2)) * w).sum() / w.sum()
    return f


def _box(rng, menu_x, menu_y, menu_z):
    return dict(nx=rng.choice(menu_x), ny=rng.choice(menu_y), nz=rng.choice(menu_z), bc=0,
                beta=rng.uniform(1.2, 2.2), c=1e-6 * 100.0 ** rng.random())


def _ensemble(case):
    rng = random.Random(case["seed0"])
    return [_box(rng, (128, 192, 256, 384), (96, 128, 192), (64, 96, 128, 192))
            for _ in range(case["boxes"])]


def _serving(case):
    """Runs of the serving menu's smaller sizes, and (run, kind, loc) per request."""
    rng = random.Random(case["seed0"])
    menu = (64, 96, 128, 192, 256)
    runs = [_box(rng, menu, menu, menu) for _ in range(case["runs"])]
    return runs, [(rng.randrange(len(runs)), int(rng.random() >= 0.25), int(rng.random() >= 2 / 3))
                  for _ in range(case["requests"])]


def _plan(d, dtype=chanfs.F64):
    return chanfs.Plan(d["nx"], d["ny"], d["nz"], LX, LY, _dz(d["nz"], d["beta"]), d.get("bc", 0),
                       dtype, d.get("ybc", 0))


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind)
    if kind == "ensemble":
        boxes = _ensemble(case)
        plans = [_plan(b, chanfs.F32_REFINED) for b in boxes]
        for p in plans:
            p.autotune()
        s.update(plans=plans, group=chanfs.Group(plans), cs=[b["c"] for b in boxes],
                 f=[_rhs(case, seed * 1000 + i, b) for i, b in enumerate(boxes)],
                 r=[_normal(seed * 1000 + 500 + i, b["nz"], b["ny"], b["nx"]) for i, b in enumerate(boxes)])
        s.update(p=[torch.empty_like(f) for f in s["f"]], u=[torch.empty_like(f) for f in s["f"]])
    elif kind == "serve":
        runs, reqs = _serving(case)
        server = chanfs.Server(40 << 30, workers=4, max_batch=16, slots_per_run=2)
        ids = [server.add_run(b["nx"], b["ny"], b["nz"], LX, LY, _dz(b["nz"], b["beta"])) for b in runs]
        jobs = []
        for i, (r, k, loc) in enumerate(reqs):
            b = runs[r]
            f = _rhs(case, seed * 1000 + i, b) if k == 0 else _normal(seed * 1000 + i, b["nz"], b["ny"], b["nx"])
            jobs.append((ids[r], k, f, torch.empty_like(f), b["c"], loc))
        torch.cuda.synchronize()
        warm = [server.submit(r, k, f, o, c, loc) for r, k, f, o, c, loc in jobs]  # plans made resident
        for t in warm:
            server.wait(t)
        for j in jobs:
            j[3].zero_()
        s.update(server=server, jobs=jobs)
    elif kind == "batch_host":
        s.update(plan=_plan(case), c=case["c"])
        ins = [_rhs(case, seed * 10)] + [_normal(seed * 10 + i, case["nz"], case["ny"], case["nx"]) for i in (1, 2, 3)]
        s["ins"] = [torch.empty(f.shape, dtype=f.dtype, pin_memory=True).copy_(f) for f in ins]
        s["outs"] = [torch.empty(f.shape, dtype=f.dtype, pin_memory=True) for f in ins]
    else:
        plan = _plan(case, chanfs.F32_REFINED if kind == "refined" else chanfs.F64)
        if case.get("tuned"):
            plan.autotune()
        s.update(plan=plan, c=case.get("c", 0.0), loc=case.get("loc", 0))
        if kind == "helmholtz":
            s["f"] = [_normal(seed * 10 + i, case["nz"], case["ny"], case["nx"]) for i in range(3)]
            for loc in (0, 1):
                plan.helmholtz_prepare(case["c"], loc)
        else:
            s["f"] = [_rhs(case, seed * 10)] if kind in ("poisson", "refined") else \
                [_normal(seed * 10, case["nz"], case["ny"], case["nx"])]
            if kind == "helmholtz3d":
                plan.helmholtz3d_prepare(case["c"], case["loc"])
        s["out"] = [torch.empty_like(f) for f in s["f"]]
        if kind == "spectral":
            s["out"].append(torch.empty_like(s["f"][0]))
    return s


def run(s):
    kind = s["kind"]
    if kind == "ensemble":
        s["group"].poisson_solve(s["f"], s["p"])
        s["group"].helmholtz_solve(s["cs"], s["r"], None, s["u"])
        return s["p"] + s["u"]
    if kind == "serve":
        tickets = [s["server"].submit(r, k, f, o, c, loc) for r, k, f, o, c, loc in s["jobs"]]
        status = [s["server"].wait(t)[0] for t in tickets]
        return [j[3] for j in s["jobs"]] + [np.array(status)]
    if kind == "batch_host":
        i, o, c = s["ins"], s["outs"], s["c"]
        s["plan"].solve_batch_host([(chanfs.REQ_POISSON, 0.0, 0, i[0], o[0]),
                                    (chanfs.REQ_HELMHOLTZ, c, chanfs.CENTER, i[1], o[1]),
                                    (chanfs.REQ_HELMHOLTZ, c, chanfs.CENTER, i[2], o[2]),
                                    (chanfs.REQ_HELMHOLTZ, c, chanfs.FACE, i[3], o[3])])
        return o
    plan, f, out = s["plan"], s["f"], s["out"]
    if kind in ("poisson", "refined"):
        plan.poisson_solve(f[0], out[0])
    elif kind == "helmholtz":
        plan.helmholtz_solve(s["c"], f[0], chanfs.CENTER, out[0])
        plan.helmholtz_solve(s["c"], f[1], chanfs.CENTER, out[1])
        plan.helmholtz_solve(s["c"], f[2], chanfs.FACE, out[2])
    elif kind == "helmholtz3d":
        plan.helmholtz3d_solve(s["c"], f[0], s["loc"], out[0])
    else:
        plan.spectral_forward(f[0], out[0])
        plan.spectral_inverse(out[0], out[1])
    return list(out)


# --- the least work ----------------------------------------------------------------------------


def _transform_flops(d):
    """x and y transforms both ways: 5 N log2 N per complex transform, half for a real one."""
    n = d["nx"] * d["ny"] * d["nz"]
    return 5.0 * n * (math.log2(d["nx"]) + math.log2(d["ny"]))


def work(case):
    kind = case["kind"]
    if kind == "ensemble":
        n = [(b, b["nx"] * b["ny"] * b["nz"]) for b in _ensemble(case)]
        return dict(bytes=sum(32.0 * k for _, k in n), flops=sum(_transform_flops(b) + 10.0 * k for b, k in n))
    if kind == "serve":
        runs, reqs = _serving(case)
        size = lambda r: runs[r]["nx"] * runs[r]["ny"] * runs[r]["nz"]
        return dict(bytes=sum(16.0 * size(r) for r, _, _ in reqs),
                    flops=sum(5.0 * size(r) + (_transform_flops(runs[r]) if k == 0 else 0.0) for r, k, _ in reqs))
    n = case["nx"] * case["ny"] * case["nz"]
    if kind == "batch_host":
        return dict(bytes=64.0 * n, flops=_transform_flops(case) + 20.0 * n)
    if kind == "helmholtz":
        return dict(bytes=48.0 * n, flops=15.0 * n)
    if kind == "spectral":
        return dict(bytes=24.0 * n, flops=_transform_flops(case))
    return dict(bytes=16.0 * n, flops=_transform_flops(case) + 5.0 * n)


# --- what the calls return, in plain torch in 64 bits ------------------------------------------


def _z_rows(dz, bc, loc):
    """Rows (a, b, c) of the flux-form z operator; bc 0 Neumann, 1 Dirichlet; loc 1: interior faces."""
    nz = len(dz)
    dzc = 0.5 * (dz[:-1] + dz[1:])
    if loc:
        lower, upper, width = 1.0 / dz[:-1], 1.0 / dz[1:], dzc
        a, c = lower / width, upper / width
        b = -(a + c)
        a[0] = c[-1] = 0.0
        return a, b, c
    a, c = np.zeros(nz), np.zeros(nz)
    a[1:], c[:-1] = 1.0 / (dzc * dz[1:]), 1.0 / (dzc * dz[:-1])
    b = -(a + c)
    if bc:
        b[0] -= 2.0 / (dz[0] * dz[0])
        b[-1] -= 2.0 / (dz[-1] * dz[-1])
    return a, b, c


def _thomas(a, diag, c, d, shift=0.0):
    """(a, diag + shift, c) x = d along the first axis of d, in place; `shift` broadcasts over a plane."""
    n = len(a)
    cp = []
    piv = shift + diag[0]
    for k in range(n):
        if k:
            piv = shift + diag[k] - a[k] * cp[k - 1]
            d[k] -= a[k] * d[k - 1]
        cp.append(c[k] / piv)
        d[k] /= piv
    for k in range(n - 2, -1, -1):
        d[k] -= cp[k] * d[k + 1]
    return d


def _exact_helmholtz(rhs, dz, c, loc):
    a, b, e = _z_rows(dz, 1, loc)
    n = len(a)
    u = rhs.clone()
    _thomas(-c * a, 1.0 - c * b, -c * e, u[:n])
    if loc:
        u[-1] = 0.0
    return u


def _y_vectors(ny, ybc):
    """Orthonormal eigenvectors (rows) of the y stencil between walls."""
    j = torch.arange(ny, dtype=torch.float64, device="cuda")
    k = j[:, None]
    if ybc == 1:
        q = torch.cos(math.pi * k * (j + 0.5) / ny) * math.sqrt(2.0 / ny)
        q[0] *= math.sqrt(0.5)
    else:
        q = torch.sin(math.pi * (k + 1) * (j + 0.5) / ny) * math.sqrt(2.0 / ny)
        q[-1] *= math.sqrt(0.5)
    return q


def _exact_3d(f, case, rows, scale, const, null):
    """(const + scale L) p = f by transforms along x and y and a sweep along z."""
    nz, ny, nx = f.shape
    ybc = case.get("ybc", 0)
    dx, dy = LX / nx, LY / ny
    kx = torch.arange(nx // 2 + 1, dtype=torch.float64, device="cuda")
    ky = torch.arange(ny, dtype=torch.float64, device="cuda")
    lx = 2.0 * (torch.cos(2.0 * math.pi * kx / nx) - 1.0) / dx**2
    th = {0: 2.0 * math.pi * ky / ny, 1: math.pi * ky / ny, 2: math.pi * (ky + 1) / ny}[ybc]
    ly = 2.0 * (torch.cos(th) - 1.0) / dy**2
    q = _y_vectors(ny, ybc) if ybc else None
    s = torch.fft.rfft(torch.matmul(q, f), dim=2) if ybc else torch.fft.rfft2(f)
    a, b, c = rows
    n = len(a)
    col = None
    if null:  # the constants: project the mean out, pin, and take the weighted mean off again
        dz = _dz(nz, case["beta"])
        g = s[:, 0, 0].real.cpu().numpy().copy()
        g -= (g * dz).sum() / dz.sum()
        p, flux = np.zeros(nz), 0.0
        for k in range(nz - 1):
            flux += g[k] * dz[k]
            p[k + 1] = p[k] + flux * 0.5 * (dz[k] + dz[k + 1])
        col = p - (p * dz).sum() / dz.sum()
    lam = scale * (lx[None, :] + ly[:, None])
    if null:
        lam[0, 0] = -1.0
    _thomas(scale * a, const + scale * b, scale * c, s[:n], lam)
    if null:
        s[:, 0, 0] = torch.from_numpy(col).cuda().to(s.dtype)
    if n < nz:
        s[n:] = 0.0
    if ybc:
        return torch.matmul(q.T, torch.fft.irfft(s, n=nx, dim=2))
    return torch.fft.irfft2(s, s=(ny, nx))


def _exact_poisson(f, case):
    null = case.get("bc", 0) == 0 and case.get("ybc", 0) != 2
    return _exact_3d(f, case, _z_rows(_dz(case["nz"], case["beta"]), case.get("bc", 0), 0), 1.0, 0.0, null)


def _exact_packed(f):
    """Packed real spectrum along x (X_0 and X_{nx/2} share the first pair), then the complex transform along
    y, the first pair's column packed once more the same way."""
    nz, ny, nx = f.shape
    m = nx // 2
    x = torch.fft.fft(torch.fft.rfft(f, dim=2), dim=1)
    first, last = x[:, :, 0], x[:, :, m]
    k = torch.arange(ny, device="cuda")
    col = torch.where(2 * k < ny, first, torch.roll(torch.flip(last, [1]), 1, 1))
    own = (2 * k) % ny == 0
    col = torch.where(own, torch.complex(first.real, last.real), col)
    x = x[:, :, :m].clone()
    x[:, :, 0] = col
    return torch.view_as_real(x).reshape(nz, ny, nx)


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        boxes = _ensemble(case)
        p = [_exact_poisson(_rhs(case, seed * 1000 + i, b), b) for i, b in enumerate(boxes)]
        return p + [_exact_helmholtz(_normal(seed * 1000 + 500 + i, b["nz"], b["ny"], b["nx"]), _dz(b["nz"], b["beta"]),
                                     b["c"], 0) for i, b in enumerate(boxes)]
    if kind == "serve":
        runs, reqs = _serving(case)
        got = []
        for i, (r, k, loc) in enumerate(reqs):
            b = runs[r]
            got.append(_exact_poisson(_rhs(case, seed * 1000 + i, b), b) if k == 0 else
                       _exact_helmholtz(_normal(seed * 1000 + i, b["nz"], b["ny"], b["nx"]), _dz(b["nz"], b["beta"]),
                                        b["c"], loc))
        return got + [None]
    shape = (case["nz"], case["ny"], case["nx"])
    dz = _dz(case["nz"], case["beta"])
    if kind in ("poisson", "refined"):
        return [_exact_poisson(_rhs(case, seed * 10), case)]
    if kind == "helmholtz":
        return [_exact_helmholtz(_normal(seed * 10 + i, *shape), dz, case["c"], int(i == 2)) for i in range(3)]
    if kind == "batch_host":
        return [_exact_poisson(_rhs(case, seed * 10), case)] + \
            [_exact_helmholtz(_normal(seed * 10 + i, *shape), dz, case["c"], int(i == 3)) for i in (1, 2, 3)]
    f = _normal(seed * 10, *shape)
    if kind == "spectral":
        return [_exact_packed(f), f]
    return [_exact_3d(f, case, _z_rows(dz, 1, case["loc"]), -case["c"], 1.0, False)]
